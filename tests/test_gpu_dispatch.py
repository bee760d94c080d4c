"""Which kernels a call launches, where a rule on its sizes has to hold at more than one entry point."""
import pytest
import torch

from gpu_util import kernels_of

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bro():
    from paper_2511_04214_b200 import binding
    return binding


@pytest.mark.parametrize("M,K,N,block", [(2048, 2048, 1024, 32), (1000, 2048, 2048, 64), (1500, 4096, 1000, 128)])
def test_the_layer_without_a_workspace_launches_what_the_layer_does(bro, M, K, N, block):
    """In front of a GEMM the line between the rotate+quantise kernels lies elsewhere than alone, whoever provides the buffers."""
    x = torch.randn(M, K, device="cuda").to(torch.bfloat16)
    wc, ws = bro.alloc_codes(N, K), bro.alloc_scales(N, K, bro.LAYOUT_GEMM)
    bro.pack_weights(torch.randn(N, K, device="cuda").to(torch.bfloat16), block, wc, ws)
    work = bro.alloc_workspace(bro.linear_workspace_bytes(M, N, K))
    y = torch.empty(M, N, dtype=torch.bfloat16, device="cuda")
    layer = kernels_of(lambda: bro.linear(x, block, wc, ws, N, y, work))
    assert len(layer) == 2
    assert kernels_of(lambda: bro.linear_static(x, block, wc, ws, N, y)) == layer


@pytest.mark.parametrize("block", [16, 32, 64, 128])
def test_plain_blocks_stay_in_registers(bro, block):
    """The register-streaming kernel stands at the registers that three CTAs an SM leave it; what only a few tokens need is not in the
    kernel that everything else takes, or it spills."""
    LOCAL_SIZE_BYTES = 3
    x = torch.randn(100, 1024, device="cuda").to(torch.bfloat16)
    codes, scales = bro.alloc_codes(100, 1024), bro.alloc_scales(100, 1024, bro.LAYOUT_GEMM)
    kernels = kernels_of(lambda: bro.rotate_quantize_mxfp4(x, block, codes, scales, flags=bro.FLAG_RQ_DIRECT), LOCAL_SIZE_BYTES)
    assert [("rotate_quantize_direct_kernel" in name, local) for name, local in kernels] == [(True, 0)]
