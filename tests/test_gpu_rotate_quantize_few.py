"""GPU parity of the rotate+quantise kernel of few tokens (a quarter of an MX group a lane): the ends of its range of rows and tasks,
half-empty last K steps, rotations inside, at and above the group, with and without the gated producer, against the CPU oracle.  Codes
bit for bit, the tiled scales byte by byte, padding included."""
import numpy as np
import pytest

import oracle
from gpu_util import Guarded, kernels_of
from paper_2511_04214_b200 import synth
from test_gpu_rotate_quantize_decode import tiled

pytestmark = pytest.mark.gpu
TASKS = 148 * 16               # a row's K steps of 256 channels are its tasks: one for each warp of one CTA an SM


@pytest.mark.parametrize("M,K,block,gated", [
    (1, 32, 16, True), (3, 288, 32, True), (16, 14336, 32, True), (63, 1088, 64, True), (128, 4608, 128, True), (37, 16384, 2, True),
    (1, 128, 128, True), (65, 256, 8, False), (65, 9216, 32, False), (100, 1088, 64, False), (128, 4608, 128, False), (127, 4640, 32, False),
    (128, 4864, 32, False), (129, 256, 32, False), (38, 16384, 32, True),      # the last three beyond its tasks or rows
])
@pytest.mark.parametrize("signs", [False, True])
def test_codes_and_every_byte_of_the_tiled_scales(M, K, block, gated, signs):
    from paper_2511_04214_b200 import binding as bro
    x, up = synth.activations(M, K, seed=M + K), synth.weights(M, K, seed=M, std=1.0)
    x[0, :32] = 0                                          # a group of zeros
    s = synth.rotation_signs(K, seed=K) if signs else None
    sb, sd = (synth.bf16_bits(s), s.cuda()) if signs else (None, None)
    codes, scales = Guarded(bro.codes_bytes(M, K)), Guarded(bro.scales_bytes(M, K, bro.LAYOUT_GEMM))
    xd, ud = x.cuda(), up.cuda()
    if gated:
        want = oracle.swiglu_rotate_quantize_mxfp4(synth.bf16_bits(x), synth.bf16_bits(up), block, sb)
        call = lambda: bro.swiglu_rotate_quantize_mxfp4(xd, ud, block, codes.view, scales.view, bro.LAYOUT_GEMM, signs=sd)  # noqa: E731
    else:
        want = oracle.rotate_quantize_mxfp4(synth.bf16_bits(x), block, sb)
        call = lambda: bro.rotate_quantize_mxfp4(xd, block, codes.view, scales.view, bro.LAYOUT_GEMM, signs=sd)  # noqa: E731
    (name,) = kernels_of(call)
    assert ("rotate_quantize_few_kernel" in name) == (M <= 128 and M * -(-K // 256) <= TASKS)
    codes.view.fill_(0xA5), scales.view.fill_(0xA5)
    call()
    assert bro.last_device_status() == 0
    codes.check(), scales.check()
    assert np.array_equal(codes.numpy().reshape(M, K // 2), want[0])
    assert np.array_equal(scales.numpy(), tiled(want[1]))
