"""The binding's two ways into the library, the call module and ctypes: the same outputs, the same errors, for plain arguments and for
those that the call module leaves to the general way."""
import threading

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bro():
    from paper_2511_04214_b200 import binding
    return binding


class Nothing:
    """In the place of the call module: every call goes the general way."""

    def __getattr__(self, name):
        return lambda *args: -1


class Sub(torch.Tensor):
    pass


def outcome(f, outputs):
    """What f leaves in the tensors, or the error that it raises."""
    for t in outputs:
        t.view(torch.uint8).fill_(0x5A) if t.is_contiguous() else t.zero_()
    try:
        f()
        torch.cuda.synchronize()
    except Exception as e:          # noqa: BLE001
        return (type(e).__name__, str(e))
    return [t.clone() for t in outputs]


def cases(bro):
    gen = torch.Generator(device="cuda").manual_seed(0)
    M, K, N = 33, 512, 264
    full = torch.randn(M, K + 8, generator=gen, device="cuda").to(torch.bfloat16)
    x, flat, one = full[:, :K], full[:, :K].contiguous(), full[:1, :K]
    signs = (1 - 2 * torch.randint(0, 2, (K,), generator=gen, device="cuda")).to(torch.bfloat16)
    w = torch.randn(N, K, generator=gen, device="cuda").to(torch.bfloat16)
    wc, ws = bro.alloc_codes(N, K), bro.alloc_scales(N, K, 1)
    bro.pack_weights(w, 32, wc, ws)
    ac, asc = bro.alloc_codes(M, K), bro.alloc_scales(M, K, 1)
    bro.rotate_quantize_mxfp4(x, 32, ac, asc)
    c, s, c2, s2 = torch.empty_like(ac), torch.empty_like(asc), torch.empty_like(wc), torch.empty_like(ws)
    y, yf = torch.empty(M, N, dtype=torch.bfloat16, device="cuda"), torch.empty(M, N, device="cuda")
    work, small = bro.alloc_workspace(bro.linear_workspace_bytes(M, N, K)), bro.alloc_workspace(64)
    deq, mse = torch.empty(M, K, device="cuda"), torch.empty(M, K // 32, device="cuda")
    rows = torch.empty(8 * M, dtype=torch.uint8, device="cuda")
    a, b, mask = (torch.empty(M, K // 32, dtype=torch.uint8, device="cuda") for _ in range(3))
    bro.group_scale_bytes(x, 1, a)
    info, ows = torch.empty(4, dtype=torch.int32, device="cuda"), torch.empty(bro.outlier_workspace_bytes(), dtype=torch.uint8, device="cuda")
    hist, counts = torch.empty(2, 256, dtype=torch.int64, device="cuda"), torch.empty(2, 3, dtype=torch.int64, device="cuda")
    flags = torch.zeros_like(a)
    st = torch.cuda.current_stream()
    L = lambda f, *out: (f, out)  # noqa: E731
    yield L(lambda: bro.rotate_quantize_mxfp4(x, 32, c, s), c, s)
    yield L(lambda: bro.rotate_quantize_mxfp4(one, 128, c[:1], s), c[:1], s)
    yield L(lambda: bro.rotate_quantize_mxfp4(x, 64, c, s, 0, signs=signs, stream=st), c)
    yield L(lambda: bro.rotate_quantize_mxfp4(x.as_subclass(Sub), 32, c, s), c, s)
    yield L(lambda: bro.rotate_quantize_mxfp4(x.float(), 32, c, s))                    # another type
    yield L(lambda: bro.rotate_quantize_mxfp4(x[0], 32, c, s))                         # a vector
    yield L(lambda: bro.rotate_quantize_mxfp4(full[:, ::2], 32, c, s))                 # columns with gaps
    yield L(lambda: bro.rotate_quantize_mxfp4(x, 24, c, s))                            # no such block
    yield L(lambda: bro.rotate_quantize_mxfp4(x, 32, None, s))
    yield L(lambda: bro.rotate_quantize_mxfp4(x, 1 << 40, c, s))
    yield L(lambda: bro.rotate_quantize_mxfp4(x, 32.0, c, s))
    yield L(lambda: bro.rotate_quantize_mxfp4(x, 32, c, s, stream=7))
    yield L(lambda: bro.pack_weights(w, 64, c2, s2), c2, s2)
    yield L(lambda: bro.pack_weights_rs(w, 64, signs, c2, s2), c2, s2)
    yield L(lambda: bro.pack_weights_rs(w, 64, signs[:256], c2, s2))
    yield L(lambda: bro.pack_weights_rs(w, 64, None, c2, s2))
    yield L(lambda: bro.gemm_mxfp4(ac, asc, wc, ws, M, N, K, y), y)
    yield L(lambda: bro.gemm_mxfp4(ac, asc, wc, ws, M, N, K, yf, small), yf)
    yield L(lambda: bro.gemm_mxfp4(ac, asc, wc, ws, M, N, K, y.half()))
    yield L(lambda: bro.gemm_mxfp4(ac, asc, wc, ws, M, N, K, yf.t()))
    yield L(lambda: bro.gemm_mxfp4(ac, asc, wc, ws, 1, N, K, y[:1]), y[:1])
    yield L(lambda: bro.linear(x, 32, wc, ws, N, y, work), y)
    yield L(lambda: bro.linear(one, 32, wc, ws, N, y[:1], work, stream=st), y[:1])
    yield L(lambda: bro.linear(x[:0], 32, wc, ws, N, y[:0], work))
    yield L(lambda: bro.linear(x, 32, wc, ws, N, y, small))
    yield L(lambda: bro.linear(x, 32, wc, ws, N, yf, work))
    yield L(lambda: bro.linear(x, 32, wc, ws, N, y, None))
    yield L(lambda: bro.linear(x, 32, wc, ws, N, y, work, signs=signs))
    yield L(lambda: bro.linear_rs(x, 32, signs, wc, ws, N, y, work), y)
    yield L(lambda: bro.linear_rs(x, 32, signs.float(), wc, ws, N, y, work))
    yield L(lambda: bro.swiglu_linear(x, flat, 32, wc, ws, N, y, work), y)
    yield L(lambda: bro.swiglu_linear(x, flat, 32, wc, ws, N, y, work, signs=signs), y)
    yield L(lambda: bro.swiglu_linear(x, flat[:, :256], 32, wc, ws, N, y, work))
    yield L(lambda: bro.swiglu_linear(x, flat, 0, wc, ws, N, y, work))
    yield L(lambda: bro.swiglu_rotate_quantize_mxfp4(x, flat, 64, c, s, signs=signs), c, s)
    yield L(lambda: bro.swiglu_rotate_quantize_mxfp4(x, full[:, 1:K + 1], 64, c, s))
    yield L(lambda: bro.group_quant_error(x, 32, mse), mse)
    yield L(lambda: bro.group_quant_error(x, 128, mse, signs, fmt="bint4"), mse)
    yield L(lambda: bro.group_quant_error(x, 32, mse.t()))
    yield L(lambda: bro.group_quant_error(x, 32, mse, fmt="fp8"))
    yield L(lambda: bro.group_quant_error(x, 32, mse, fmt="int4_row_sym"))
    yield L(lambda: bro.rotate_fake_quantize(x, 32, deq, "bfp4", signs), deq)
    yield L(lambda: bro.rotate_fake_quantize(x, 1, deq, "int4_row_asym", workspace=rows), deq)
    yield L(lambda: bro.rotate_fake_quantize(x, 1, deq, "int4_row_asym"))
    yield L(lambda: bro.rotate_fake_quantize(x, 1, deq[:, :256]))
    yield L(lambda: bro.group_scale_bytes(x, 64, b), b)
    yield L(lambda: bro.group_scale_bytes(x, 0, b, signs), b)
    yield L(lambda: bro.group_scale_bytes(x, 64, b[:, :8]))
    yield L(lambda: bro.outlier_groups(x, mask, info, ows, 20000), mask, info)
    yield L(lambda: bro.outlier_groups(flat, mask, info, ows), mask, info)
    yield L(lambda: bro.outlier_groups(x, mask, info[:3], ows))
    yield L(lambda: bro.outlier_groups(x, mask, info, ows[:64]))
    yield L(lambda: bro.scale_histogram(a, flags, hist), hist)
    yield L(lambda: bro.scale_histogram(a, flags, hist[:1]))
    yield L(lambda: bro.scale_inflation(a, flags, flags, counts), counts)
    yield L(lambda: bro.scale_inflation(a[:4], flags, flags, counts))


def test_both_ways_agree(bro, monkeypatch):
    call = bro._call
    for i, (f, out) in enumerate(cases(bro)):
        monkeypatch.setattr(bro, "_call", call)
        fast = outcome(f, out)
        monkeypatch.setattr(bro, "_call", Nothing())
        general = outcome(f, out)
        assert type(fast) is type(general) and len(fast) == len(general), (i, fast, general)
        if isinstance(fast, tuple):
            assert fast == general, i
        else:
            assert all(torch.equal(p, q) for p, q in zip(fast, general)), i


def test_current_stream_and_threads(bro):
    """Each thread's current stream is the one that its calls go to."""
    M, K = 64, 1024
    xs = [torch.randn(M, K, device="cuda").to(torch.bfloat16) for _ in range(4)]
    want = []
    for x in xs:
        c, s = bro.alloc_codes(M, K), bro.alloc_scales(M, K, 1)
        bro.rotate_quantize_mxfp4(x, 32, c, s)
        want.append((c, s))
    torch.cuda.synchronize()
    got = [None] * 4

    def work(i):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            c, s = bro.alloc_codes(M, K), bro.alloc_scales(M, K, 1)
            for j in range(200):
                bro.rotate_quantize_mxfp4(xs[(i + j) % 4], 32, c, s)
            bro.rotate_quantize_mxfp4(xs[i], 32, c, s)
            stream.synchronize()
            got[i] = (c, s)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for p, q in zip(got, want):
        assert torch.equal(p[0], q[0]) and torch.equal(p[1], q[1])
