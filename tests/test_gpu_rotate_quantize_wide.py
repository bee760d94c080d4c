"""GPU parity of the rotate+quantise kernel whose lanes own 64 channels (blocks 32, 64, 128, K a multiple of 64) where its tiles and
stores can go wrong — codes and their scale bytes, by the flag that asks for it — and of the statistics of the same small tensors,
which the register-streaming kernel computes at these sizes, against the CPU oracle.  (The statistics of large tensors, which
the first kernel computes, are in test_gpu_large_forms.py.)"""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import Guarded
from paper_2511_04214_b200 import synth
from test_gpu_quant_error import check, reference
from test_gpu_rotate_quantize import run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bro():
    from paper_2511_04214_b200 import binding
    return binding


def device_copy(x, pad):
    """x on the device, rows `pad` elements apart from each other, the gaps holding large values."""
    if pad == 0:
        return x.cuda()
    buf = torch.full((x.shape[0], x.shape[1] + pad), 3.0e4, dtype=torch.bfloat16, device="cuda")
    buf[:, :x.shape[1]] = x.cuda()
    return buf[:, :x.shape[1]]


def all_outputs(bro, x, xd, block, signs, flags):
    M, K = x.shape
    sb = None if signs is None else synth.bf16_bits(signs)
    sd = None if signs is None else signs.cuda()
    rc, rs = oracle.rotate_quantize_mxfp4(synth.bf16_bits(x), block, sb)
    for layout in (0, 1):
        for shift in (0, 16):              # codes on 32 bytes and between
            codes, scales = Guarded(M * K // 2 + shift), Guarded(bro.scales_bytes(M, K, layout))
            bro.rotate_quantize_mxfp4(xd, block, codes.view[shift:], scales.view, layout, flags=flags, signs=sd)
            codes.check(), scales.check()
            assert np.array_equal(codes.numpy()[shift:].reshape(M, K // 2), rc)
            if layout == 0:
                assert np.array_equal(scales.numpy().reshape(M, K // 32), rs)
    if signs is None:
        gc, gs = run_gpu(bro, xd, block, 1, flags)          # (the padding of the tiled scales too)
        assert np.array_equal(gc, rc) and np.array_equal(gs, rs)
    for shift in (0, 1):                   # scale bytes on a word and between
        out = Guarded(M * (K // 32) + shift)
        bro.group_scale_bytes(xd, block, out.view[shift:].view(M, K // 32), signs=sd)
        out.check()
        assert np.array_equal(out.numpy()[shift:].reshape(M, K // 32), rs)
    mse = Guarded(M * (K // 32) * 4)
    bro.group_quant_error(xd, block, mse.view.view(torch.float32).view(M, K // 32), sd)
    mse.check()
    check(mse.view.view(torch.float32).view(M, K // 32).cpu().numpy().astype(np.float64), reference(x, block, signs))
    assert bro.last_device_status() == 0


@pytest.mark.parametrize("M,K,block", [(M, K, b) for M, K in [(1, 64), (15, 192), (16, 128), (17, 320), (129, 1088), (127, 2176), (3, 14336)]
                                       for b in (32, 64, 128) if K % b == 0])
@pytest.mark.parametrize("signs", [False, True])
def test_tiles_of_16_rows_and_128_channels(bro, M, K, block, signs):
    """Rows around the tile's 16 and the scale block's 128, K that ends inside a tile and inside a scale block, rows with gaps."""
    x = synth.activations(M, K, seed=M + K)
    s = synth.rotation_signs(K, seed=3) if signs else None
    all_outputs(bro, x, device_copy(x, 8 if signs else 0), block, s, bro.FLAG_RQ_TMA_RING)


@pytest.mark.parametrize("block", [32, 64, 128])
def test_values_at_the_ends_of_the_range_as_in_the_direct_kernel(bro, block):
    """Infinities, NaN, negative zeros, bf16 subnormals and maxima beyond the one-multiply range, in one of the two groups of a lane, in
    both, in every lane position: the same bytes as the register-streaming kernel."""
    M, K = 70, 512
    gen = torch.Generator().manual_seed(block)
    x = torch.randn(M, K, generator=gen)
    rows = torch.arange(M)
    for i, v in enumerate((float("inf"), float("-inf"), float("nan"), 3.0e38, 1.0e-40, -0.0)):
        x[rows, (rows * 37 + i * 64) % K] = v
    x[::5, :64] *= 1.0e-38
    x[1::5, 32:96] *= 1.0e30
    x[2::5] = -0.0
    x[3::5, 64:] = 0.0
    xd = x.to(torch.bfloat16).cuda()
    out = []
    for flags in (bro.FLAG_RQ_DIRECT, bro.FLAG_RQ_TMA_RING):
        codes, scales = bro.alloc_codes(M, K), bro.alloc_scales(M, K, bro.LAYOUT_GEMM)
        bro.rotate_quantize_mxfp4(xd, block, codes, scales, flags=flags)
        out.append((codes, scales))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
