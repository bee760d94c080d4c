"""The scale statistics on rows without gaps (read as one row, whole lines at a time) against the same values in rows with gaps, and
the outlier threshold wherever it can lie in the histogram."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bro():
    from paper_2511_04214_b200 import binding
    return binding


@pytest.mark.parametrize("M,K", [(1, 32), (1, 992), (3, 64), (7, 1056), (33, 4096), (1000, 3008), (5000, 32), (16385, 1024), (5590, 3008),
                                 (1, 16777216 + 32), (524289, 32)])
def test_scale_bytes_without_a_rotation(bro, M, K):
    """Last warps with one to 32 groups, rows that end inside a warp's 32 (read as one row from 2^24 elements)."""
    gen = torch.Generator().manual_seed(M + K)
    x = (torch.randn(M, K, generator=gen) * torch.exp2(torch.randint(-130, 120, (M, K // 32, 1), generator=gen).float()).expand(
        M, K // 32, 32).reshape(M, K)).to(torch.bfloat16)
    x[0, 0] = float("inf")
    x[-1, -1] = -0.0
    want = ((x.view(torch.int16).int() & 0x7FFF).view(M, K // 32, 32).amax(2) >> 7).sub(2).clamp(min=0).to(torch.uint8)
    buf = torch.full((M, K + 8), 3.0e38, dtype=torch.bfloat16, device="cuda")
    buf[:, :K] = x.cuda()
    for xd in (x.cuda(), buf[:, :K]):
        out = torch.full((M, K // 32), 0xEE, dtype=torch.uint8, device="cuda")
        bro.group_scale_bytes(xd, 1, out)
        assert torch.equal(out.cpu(), want)


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 31, 32, 33, 127, 128, 129, 1023, 1024, 1025, 2048, 32000, 32768])
@pytest.mark.parametrize("repeat", [1, 40])
def test_outlier_threshold_at_every_place_of_the_histogram(bro, k, repeat):
    """Every magnitude pattern the same number of times: the k-th largest is known, at the edges of a lane's four patterns, of a
    chunk of 128, of a segment of 1024, at both ends."""
    patterns = torch.arange(32768, dtype=torch.int32).repeat(repeat)
    gen = torch.Generator().manual_seed(k)
    bits = patterns[torch.randperm(patterns.numel(), generator=gen)]
    bits = torch.where(torch.rand(bits.numel(), generator=gen) < 0.5, bits, bits - 32768).to(torch.int16)
    K = 1024
    x = bits.view(-1, K).view(torch.bfloat16).cuda()
    M, n = x.shape[0], bits.numel()
    top_ppm = max(1, min(1000000, k * repeat * 1000000 // n))
    kk = max(1, -(-n * top_ppm // 1000000))
    t = 32767 - (kk - 1) // repeat
    mask = torch.full((M, K // 32), 0xEE, dtype=torch.uint8, device="cuda")
    info = torch.zeros(4, dtype=torch.int32, device="cuda")
    ws = torch.full((bro.outlier_workspace_bytes(),), 0xAB, dtype=torch.uint8, device="cuda")
    bro.outlier_groups(x, mask, info, ws, top_ppm=top_ppm)
    assert info.tolist() == [t, 0, kk, 0]
    want = ((x.view(torch.int16).int() & 0x7FFF).view(M, K // 32, 32).amax(2) >= t).to(torch.uint8)
    assert torch.equal(mask, want)


@pytest.mark.parametrize("M", [64, 2500])
def test_statistics_back_to_back_on_two_streams(bro, M):
    """A scan starts before its histogram is clear, a count before its output is: two passes over different tensors, interleaved on two
    streams with buffers of their own, give what each gives alone."""
    K = 2048
    gen = torch.Generator(device="cuda").manual_seed(M)
    lanes = []
    for _ in range(2):
        u8 = lambda: torch.zeros(M, K // 32, dtype=torch.uint8, device="cuda")  # noqa: E731
        lanes.append({"stream": torch.cuda.Stream(), "x": [torch.randn(M, K, generator=gen, device="cuda").mul_(3 ** i).to(torch.bfloat16) for i in range(3)],
                      "mask": u8(), "a": u8(), "b": u8(), "info": torch.zeros(4, dtype=torch.int32, device="cuda"),
                      "ws": torch.empty(bro.outlier_workspace_bytes(), dtype=torch.uint8, device="cuda"),
                      "counts": torch.zeros(2, 3, dtype=torch.int64, device="cuda"), "hist": torch.zeros(2, 256, dtype=torch.int64, device="cuda")})

    def one(s, i, stream):
        bro.outlier_groups(s["x"][i], s["mask"], s["info"], s["ws"], stream=stream)
        bro.group_scale_bytes(s["x"][i], 1, s["a"], stream=stream)
        bro.group_scale_bytes(s["x"][i], 128, s["b"], stream=stream)
        bro.scale_inflation(s["a"], s["b"], s["mask"], s["counts"], stream=stream)
        bro.scale_histogram(s["b"], s["mask"], s["hist"], stream=stream)
        with torch.cuda.stream(stream):
            return [s[k].clone() for k in ("mask", "info", "a", "b", "counts", "hist")]

    want = []
    for s in lanes:
        want.append([])
        for i in range(3):
            want[-1].append(one(s, i, torch.cuda.current_stream()))
            torch.cuda.synchronize()
    got = [[], []]
    for r in range(9):
        for j, s in enumerate(lanes):
            got[j].append(one(s, r % 3, s["stream"]))
    torch.cuda.synchronize()
    for j in range(2):
        for r, g in enumerate(got[j]):
            for p, q in zip(g, want[j][r % 3]):
                assert torch.equal(p, q), (j, r)
