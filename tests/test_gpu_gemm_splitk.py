"""GPU parity of the GEMM for problems of few output tiles (one wave of 128- or 256-row weight tiles, K split over
the CTAs of a cluster): the edges of its tiles and of its plan, against the CPU oracle and the persistent kernel."""
import ctypes

import pytest
import torch

from gpu_util import Guarded
from test_gpu_gemm import quantized_pair, run_case, upload_operand

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bro():
    from paper_2511_04214_b200 import binding
    return binding


def launches(call):
    """How many graph nodes a call becomes: 1 for the layer in one kernel, 2 for rotate + quantise and the GEMM."""
    call()                                            # (loads the kernels outside the capture)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        call()
    n = ctypes.c_size_t(0)
    assert ctypes.CDLL("libcuda.so.1").cuGraphGetNodes(ctypes.c_void_p(graph.raw_cuda_graph()), None, ctypes.byref(n)) == 0
    return n.value


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


@pytest.mark.parametrize("M,K,N,block", [
    (1, 8192, 19000, 32),     # 256-row tiles: a ring of 6 stages, 32 steps, one task a step
    (2, 4096, 1000, 64),      # clusters, rotation across lanes
    (5, 4128, 264, 32),       # K not a multiple of 256: half of the last step is padding
    (16, 2176, 136, 128),
    (31, 1024, 392, 2),       # rotations inside the group
    (33, 2048, 392, 32),      # 9 warp tasks a step for 16 warps, clusters
    (64, 256, 264, 16),       # as many tasks as warps, one step
    (64, 2048, 264, 128),
])
@pytest.mark.parametrize("signs", [False, True])
def test_layer_of_few_tokens_same_bytes_as_two_kernels(bro, M, K, N, block, signs):
    """bro.linear with few tokens quantises inside the GEMM: codes and scales left in the workspace (padding
    included) are those of rotate_quantize_mxfp4, the output is that of gemm_mxfp4 up to the order of fp32 sums
    (bf16: one ulp, 2^-8 of the row's largest magnitude at most)."""
    gen = torch.Generator(device="cuda").manual_seed(M + K)
    x = torch.randn(M, K + 8, generator=gen, device="cuda").to(torch.bfloat16)[:, :K]
    w = torch.randn(N, K, generator=gen, device="cuda").to(torch.bfloat16)
    s = (1 - 2 * torch.randint(0, 2, (K,), generator=gen, device="cuda")).to(torch.bfloat16) if signs else None
    wc, wsc = bro.alloc_codes(N, K), bro.alloc_scales(N, K, bro.LAYOUT_GEMM)
    bro.pack_weights_rs(w, block, s, wc, wsc) if signs else bro.pack_weights(w, block, wc, wsc)
    nbytes = bro.linear_workspace_bytes(M, N, K)
    ws = Guarded(nbytes + 1024, fill=0x7F)
    off = (-ws.view.data_ptr()) % 1024
    work = ws.view[off:off + nbytes]
    ldy = (N + 7) // 8 * 8
    out = Guarded(M * ldy * 2, fill=0x7F)
    y = out.view.view(torch.bfloat16).view(M, ldy)[:, :N]
    layer = (lambda: bro.linear_rs(x, block, s, wc, wsc, N, y, work)) if signs else (lambda: bro.linear(x, block, wc, wsc, N, y, work))
    assert launches(layer) == 1
    out.view.fill_(0x7F)
    ws.view.fill_(0x7F)
    layer()
    assert bro.last_device_status() == 0
    ws.check()
    out.check()
    ac, asc = bro.alloc_codes(M, K), bro.alloc_scales(M, K, bro.LAYOUT_GEMM)
    bro.rotate_quantize_mxfp4(x, block, ac, asc, signs=s)
    assert torch.equal(work[:ac.numel()], ac.flatten())
    at = (ac.numel() + 1023) // 1024 * 1024
    assert torch.equal(work[at:at + asc.numel()], asc)
    ref = torch.empty(M, N if N % 8 == 0 else ldy, dtype=torch.bfloat16, device="cuda")[:, :N]
    bro.gemm_mxfp4(ac, asc, wc, wsc, M, N, K, ref, flags=bro.FLAG_GEMM_SINGLE)
    top = ref.float().abs().amax(1, keepdim=True)
    assert ((y.float() - ref.float()).abs() <= top * 2.0 ** -8).all()


@pytest.mark.parametrize("M,K,N,shift", [
    (16, 2048, 2048, 0),       # y is x
    (16, 2048, 2048, 8),       # y starts 8 elements into x, in rows of the same stride
    (3, 1024, 1000, 0),        # fewer columns than x has
    (1, 4096, 4096, 0),
])
@pytest.mark.parametrize("signs", [False, True])
def test_layer_of_few_tokens_in_place(bro, M, K, N, shift, signs):
    """y over x: the layer is rotate + quantise and then the GEMM, so all of x has been read when y is written.  The same
    bits as the two calls give with an output of its own (the GEMM is the same kernel)."""
    gen = torch.Generator(device="cuda").manual_seed(M + K + shift)
    ld = K + 16
    buf = torch.randn(M, ld, generator=gen, device="cuda").to(torch.bfloat16)
    x, y = buf[:, :K], buf[:, shift:shift + N]
    w = torch.randn(N, K, generator=gen, device="cuda").to(torch.bfloat16)
    s = (1 - 2 * torch.randint(0, 2, (K,), generator=gen, device="cuda")).to(torch.bfloat16) if signs else None
    wc, wsc = bro.alloc_codes(N, K), bro.alloc_scales(N, K, bro.LAYOUT_GEMM)
    bro.pack_weights_rs(w, 32, s, wc, wsc) if signs else bro.pack_weights(w, 32, wc, wsc)
    ac, asc = bro.alloc_codes(M, K), bro.alloc_scales(M, K, bro.LAYOUT_GEMM)
    bro.rotate_quantize_mxfp4(x, 32, ac, asc, signs=s)
    want = torch.empty(M, N, dtype=torch.bfloat16, device="cuda")
    bro.gemm_mxfp4(ac, asc, wc, wsc, M, N, K, want)
    around = buf.clone()
    work = bro.alloc_workspace(bro.linear_workspace_bytes(M, N, K))
    bro.linear_rs(x, 32, s, wc, wsc, N, y, work) if signs else bro.linear(x, 32, wc, wsc, N, y, work)
    assert bro.last_device_status() == 0
    assert torch.equal(y, want)
    around[:, shift:shift + N] = want
    assert torch.equal(buf, around)


@pytest.mark.parametrize("M,K,N", [(65, 2048, 264), (128, 256, 1000), (64, 512, 4096), (130, 2048, 264), (64, 8192, 19000)])
def test_layer_of_more_tokens_keeps_two_kernels(bro, M, K, N):
    x = torch.randn(M, K, device="cuda").to(torch.bfloat16)
    wc, wsc = bro.alloc_codes(N, K), bro.alloc_scales(N, K, bro.LAYOUT_GEMM)
    bro.pack_weights(torch.randn(N, K, device="cuda").to(torch.bfloat16), 32, wc, wsc)
    y, work = torch.empty(M, N, dtype=torch.bfloat16, device="cuda"), bro.alloc_workspace(bro.linear_workspace_bytes(M, N, K))
    assert launches(lambda: bro.linear(x, 32, wc, wsc, N, y, work)) == 2


@pytest.mark.parametrize("M,K,N", [(2, 4096, 4096), (16, 2048, 19000)])
def test_layer_right_behind_the_packing_of_its_weights(bro, M, K, N):
    """The one-kernel layer draws its first weight tiles into L2 while the kernel before it may still be writing them: new
    weights packed into the same buffers just before every call, on two streams with buffers of their own, must be
    the ones that the layer multiplies."""
    gen = torch.Generator(device="cuda").manual_seed(K)
    x = torch.randn(M, K, generator=gen, device="cuda").to(torch.bfloat16)
    ws = [torch.randn(N, K, generator=gen, device="cuda").to(torch.bfloat16) for _ in range(3)]
    want = []
    for w in ws:
        wc, wsc = bro.alloc_codes(N, K), bro.alloc_scales(N, K, bro.LAYOUT_GEMM)
        bro.pack_weights(w, 32, wc, wsc)
        torch.cuda.synchronize()
        y, work = torch.empty(M, N, dtype=torch.bfloat16, device="cuda"), bro.alloc_workspace(bro.linear_workspace_bytes(M, N, K))
        bro.linear(x, 32, wc, wsc, N, y, work)
        want.append(y)
    torch.cuda.synchronize()
    lanes = []
    for _ in range(2):
        lanes.append((torch.cuda.Stream(), bro.alloc_codes(N, K), bro.alloc_scales(N, K, bro.LAYOUT_GEMM),
                      bro.alloc_workspace(bro.linear_workspace_bytes(M, N, K)),
                      [torch.empty(M, N, dtype=torch.bfloat16, device="cuda") for _ in range(12)]))
    torch.cuda.synchronize()
    for i in range(12):
        for stream, wc, wsc, work, ys in lanes:
            bro.pack_weights(ws[i % 3], 32, wc, wsc, stream=stream)
            bro.linear(x, 32, wc, wsc, N, ys[i], work, stream=stream)
    torch.cuda.synchronize()
    assert bro.last_device_status() == 0
    for _, _, _, _, ys in lanes:
        for i, y in enumerate(ys):
            assert torch.equal(y, want[i % 3]), i
