"""Helpers shared by the GPU parity tests (not a test module)."""
import ctypes

import numpy as np
import torch

from paper_2511_04214_b200 import synth


def gemm_scale_index(rows: int, K: int) -> np.ndarray:
    """Byte offset of every (row, group) in the tensor-core scale layout, as an int64 array
    [rows, K/32] (the documented formula, vectorised)."""
    r = np.arange(rows, dtype=np.int64)[:, None]
    g = np.arange(K // 32, dtype=np.int64)[None, :]
    kb = 2 * ((K + 255) // 256)
    return ((r // 128) * kb + g // 4) * 512 + (r % 32) * 16 + ((r % 128) // 32) * 4 + (g % 4)


def to_canonical(scales_gemm: np.ndarray, rows: int, K: int) -> np.ndarray:
    return scales_gemm[gemm_scale_index(rows, K)]


def to_gemm_layout(scales_canon: np.ndarray, rows: int, K: int) -> np.ndarray:
    kb = 2 * ((K + 255) // 256)
    out = np.zeros(((rows + 127) // 128) * kb * 512, dtype=np.uint8)
    out[gemm_scale_index(rows, K)] = scales_canon
    return out


class Guarded:
    """A device byte buffer with poisoned guard bands before and after the payload."""
    PAD = 256

    def __init__(self, nbytes: int, fill: int = 0xA5):
        self.nbytes = nbytes
        self.fill = fill
        self.raw = torch.full((nbytes + 2 * self.PAD,), fill, dtype=torch.uint8, device="cuda")
        assert self.raw.data_ptr() % 256 == 0
        self.view = self.raw[self.PAD:self.PAD + nbytes]

    def check(self):
        head = self.raw[:self.PAD].cpu().numpy()
        tail = self.raw[self.PAD + self.nbytes:].cpu().numpy()
        assert (head == self.fill).all(), "write before the start of an output buffer"
        assert (tail == self.fill).all(), "write past the end of an output buffer"

    def numpy(self):
        return self.view.cpu().numpy()


def x_from_bits(bits: np.ndarray) -> torch.Tensor:
    return synth.bits_to_bf16(bits).cuda()


class _KernelNode(ctypes.Structure):
    """CUDA_KERNEL_NODE_PARAMS of the driver API."""
    _fields_ = [("func", ctypes.c_void_p), ("grid", ctypes.c_uint * 3), ("block", ctypes.c_uint * 3), ("smem", ctypes.c_uint),
                ("params", ctypes.c_void_p), ("extra", ctypes.c_void_p), ("kern", ctypes.c_void_p), ("ctx", ctypes.c_void_p)]


def kernels_of(f, attribute=None):
    """Names (as the compiler writes them) of the kernels that f() launches, from a captured call; with the number of an attribute
    (CUfunction_attribute), pairs of the name and its value."""
    f()                                    # (a first launch sets the kernel up, which a capture does not take)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        f()
    cuda, raw, n = ctypes.CDLL("libcuda.so.1"), ctypes.c_void_p(graph.raw_cuda_graph()), ctypes.c_size_t(0)
    assert cuda.cuGraphGetNodes(raw, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert cuda.cuGraphGetNodes(raw, nodes, ctypes.byref(n)) == 0
    names = []
    for node in nodes:
        kind, params, name = ctypes.c_int(-1), _KernelNode(), ctypes.c_char_p()
        assert cuda.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        if kind.value != 0:                # CU_GRAPH_NODE_TYPE_KERNEL
            continue
        assert cuda.cuGraphKernelNodeGetParams_v2(ctypes.c_void_p(node), ctypes.byref(params)) == 0
        func = ctypes.c_void_p(params.func)
        if not params.func:
            assert cuda.cuKernelGetFunction(ctypes.byref(func), ctypes.c_void_p(params.kern)) == 0
        assert cuda.cuFuncGetName(ctypes.byref(name), func) == 0
        value = ctypes.c_int(0)
        if attribute is not None:
            assert cuda.cuFuncGetAttribute(ctypes.byref(value), ctypes.c_int(attribute), func) == 0
        names.append(name.value.decode() if attribute is None else (name.value.decode(), value.value))
    return names
