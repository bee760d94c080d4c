"""The GEMM of two CTAs per tile where the library picks it by the length of a row of codes, and its early weight loads and final
stores inside the whole layer: the same bits as the single-CTA kernel, which adds up K in the same order."""
import pytest
import torch

from gpu_util import Guarded

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bro():
    from paper_2511_04214_b200 import binding
    return binding


def operands(bro, M, K, N, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn(M, K, generator=gen, device="cuda").to(torch.bfloat16)
    w = torch.randn(N, K, generator=gen, device="cuda").to(torch.bfloat16)
    wc, ws = bro.alloc_codes(N, K), bro.alloc_scales(N, K, bro.LAYOUT_GEMM)
    bro.pack_weights(w, 32, wc, ws)
    return x, w, wc, ws


@pytest.mark.parametrize("M,K,N", [
    (129, 4384, 2048),        # one row beyond the single-CTA kernel's tile, few tiles: half-width units only
    (257, 2080, 8200),        # a second pair of row tiles with one row, ragged last column tile
    (777, 4384, 6004),        # a last round of half-width units
    (1000, 1056, 3001),       # five steps: the whole ring at once, odd N
    (300, 96, 20000),         # one step, several rounds
    (1300, 32, 300),          # a single group
])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_rows_of_codes_between_sectors(bro, M, K, N, dtype):
    x, _, wc, ws = operands(bro, M, K, N, M + K)
    ac, asc = bro.alloc_codes(M, K), bro.alloc_scales(M, K, bro.LAYOUT_GEMM)
    bro.rotate_quantize_mxfp4(x, 32, ac, asc)
    ld = (N + 7) // 8 * 8
    out = []
    for flags in (0, bro.FLAG_GEMM_PAIR, bro.FLAG_GEMM_SINGLE):
        buf = Guarded(M * ld * dtype.itemsize, fill=0x7F)
        y = buf.view.view(dtype).view(M, ld)
        bro.gemm_mxfp4(ac, asc, wc, ws, M, N, K, y[:, :N], flags=flags)
        assert bro.last_device_status() == 0
        buf.check()
        out.append(y.clone())
    assert torch.equal(out[0], out[2]) and torch.equal(out[1], out[2])


@pytest.mark.parametrize("M,K,N", [(130, 256, 296), (300, 1024, 520), (257, 1280, 4096), (600, 1568, 9000), (2100, 2048, 5000)])
def test_layer_with_early_weight_loads(bro, M, K, N):
    """Fewer steps than the ring, as many, more; one unit a pair and several.  The weights are packed right in front of the layer, over
    others, and the layer is called twice in a row."""
    x, w, wc, ws = operands(bro, M, K, N, N)
    want = []
    ac, asc = bro.alloc_codes(M, K), bro.alloc_scales(M, K, bro.LAYOUT_GEMM)
    bro.rotate_quantize_mxfp4(x, 32, ac, asc)
    weights = [w, -w.flip(0)]
    for v in weights:
        bro.pack_weights(v, 32, wc, ws)
        y = torch.empty(M, N, dtype=torch.bfloat16, device="cuda")
        bro.gemm_mxfp4(ac, asc, wc, ws, M, N, K, y, flags=bro.FLAG_GEMM_SINGLE)
        want.append(y)
    work = bro.alloc_workspace(bro.linear_workspace_bytes(M, N, K))
    torch.cuda.synchronize()
    got = []
    for i in range(6):
        bro.pack_weights(weights[i % 2], 32, wc, ws)
        for _ in range(2):
            got.append(torch.empty(M, N, dtype=torch.bfloat16, device="cuda"))
            bro.linear(x, 32, wc, ws, N, got[-1], work, flags=bro.FLAG_GEMM_PAIR)
    assert bro.last_device_status() == 0
    for i, y in enumerate(got):
        assert torch.equal(y, want[i // 2 % 2]), i
