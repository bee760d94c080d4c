"""GPU parity of the direct rotate+quantise kernels where the tiled scales are mostly padding: up to 64 rows the tasks are dealt out
over the CTAs and the padding rows are cleared, beyond that they are quantised as zeros.  Codes against the CPU oracle, the tiled
scales byte by byte, padding included, for the plain and the gated form."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import Guarded
from paper_2511_04214_b200 import synth

pytestmark = pytest.mark.gpu
DIRECT = 2


def tiled(canonical):
    """[M, K / 32] scale bytes in 512-byte blocks of 128 rows x 4 groups, K in 256s, zeros where there is no row or group."""
    M, G = canonical.shape
    full = np.zeros(((M + 127) // 128 * 128, (G + 7) // 8 * 8), np.uint8)
    full[:M, :G] = canonical
    t = full.reshape(full.shape[0] // 128, 4, 32, full.shape[1] // 4, 4)      # row block, row / 32, row % 32, group / 4, group % 4
    return t.transpose(0, 3, 2, 1, 4).reshape(-1)


@pytest.mark.parametrize("M,K,block", [(M, K, b) for M in (1, 31, 64, 65, 192) for K in (32, 1088, 4160, 9216) for b in (16, 32, 64, 128)
                                       if K % b == 0])
def test_codes_and_every_byte_of_the_tiled_scales(M, K, block):
    from paper_2511_04214_b200 import binding as bro
    x, up = synth.activations(M, K, seed=M + K), synth.weights(M, K, seed=M, std=1.0)
    for signs in (None, synth.rotation_signs(K, seed=K)):
        sb, sd = (None, None) if signs is None else (synth.bf16_bits(signs), signs.cuda())
        for gated in (False, True):
            codes, scales = Guarded(bro.codes_bytes(M, K)), Guarded(bro.scales_bytes(M, K, bro.LAYOUT_GEMM))
            scales.view.fill_(0xA5)
            if gated:
                rc, rs = oracle.swiglu_rotate_quantize_mxfp4(synth.bf16_bits(x), synth.bf16_bits(up), block, sb)
                bro.swiglu_rotate_quantize_mxfp4(x.cuda(), up.cuda(), block, codes.view, scales.view, bro.LAYOUT_GEMM, signs=sd)
            else:
                rc, rs = oracle.rotate_quantize_mxfp4(synth.bf16_bits(x), block, sb)
                bro.rotate_quantize_mxfp4(x.cuda(), block, codes.view, scales.view, bro.LAYOUT_GEMM, flags=DIRECT, signs=sd)
            assert bro.last_device_status() == 0
            codes.check(), scales.check()
            assert np.array_equal(codes.numpy().reshape(M, K // 2), rc)
            assert np.array_equal(scales.numpy(), tiled(rs))
