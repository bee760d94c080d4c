"""GPU parity of the GEMM for problems of few output tiles (one wave of 128- or 256-row weight tiles, K split over
the CTAs of a cluster): the edges of its tiles and of its plan, against the CPU oracle and the persistent kernel."""
import pytest
import torch

from gpu_util import Guarded
from test_gpu_gemm import quantized_pair, run_case, upload_operand

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bro():
    from paper_2511_04214_b200 import binding
    return binding


@pytest.mark.parametrize("M,K,N", [
    (1, 256, 1),              # one K step, one column
    (3, 2048, 129),           # two row blocks' worth of columns, odd N
    (16, 4128, 130),          # ragged K (half-empty last step), clusters
    (17, 3840, 1000),         # 15 steps over the cluster: parts of unequal length
    (33, 8192, 250),          # 64 token columns, most of a cluster's tokens in the first ranks
    (128, 12288, 192),        # 128 tokens split over the cluster
    (130, 2048, 264),         # a second token tile with two tokens
    (257, 10240, 136),        # three token tiles, split, the last with one token
    (20, 512, 19001),         # more than one wave of 128-row tiles: 256-row tiles, ragged last row block
    (64, 256, 18945),         # the same with one column in the last tile
])
def test_splitk_shapes(bro, M, K, N):
    _, _, ac, asc, wc, wsc = quantized_pair(M, N, K, seed=3)
    run_case(bro, ac, asc, wc, wsc)


@pytest.mark.parametrize("M,K,N", [(5, 14336, 512), (100, 14336, 384), (48, 1024, 20000)])
def test_splitk_same_result_as_persistent_kernel(bro, M, K, N):
    """fp32 sums of few-bit products: a different order of the K steps moves the last bits at most
    (2^-20 of the largest magnitude of a row leaves room for 16 roundings)."""
    _, _, ac, asc, wc, wsc = quantized_pair(M, N, K, seed=4)
    a_c, a_s = upload_operand(ac, asc)
    w_c, w_s = upload_operand(wc, wsc)
    out = []
    for flags in (0, 0, bro.FLAG_GEMM_SINGLE):
        buf = Guarded(M * N * 4, fill=0x7F)
        y = buf.view.view(torch.float32).view(M, N)
        bro.gemm_mxfp4(a_c, a_s, w_c, w_s, M, N, K, y, flags=flags)
        assert bro.last_device_status() == 0
        buf.check()
        out.append(y.clone())
    assert torch.equal(out[0], out[1])            # parts are added in rank order: run after run the same bits
    top = out[2].abs().amax(1, keepdim=True)
    assert ((out[0] - out[2]).abs() <= top * 2.0 ** -20).all()
