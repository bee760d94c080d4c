"""GPU parity of the kernels that a call takes for its size alone, at sizes that take them: the kernel whose lanes own 64 channels
(blocks 32, 64, 128), the one of the full-dimension rotation, and those on either side of their lines.  Each test names the kernel
and looks that the call launches it.  The tensors are large, so the oracle works out sampled rows."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import Guarded, kernels_of, to_canonical
from paper_2511_04214_b200 import synth
from test_gpu_quant_error import reference

pytestmark = pytest.mark.gpu

WIDE, GLOBAL, FEW, SHUFFLES = ("rotate_quantize_wide_kernel", "rotate_quantize_global_wide_kernel", "rotate_quantize_global_few_kernel",
                               "rotate_quantize_global_kernel")
CODES, BYTES, ERROR = range(3)


@pytest.fixture(scope="module")
def bro():
    from paper_2511_04214_b200 import binding
    return binding


class Large:
    """A tensor on the device, rows `pad` elements apart (large values between them), and the rows that the oracle looks at."""

    def __init__(self, M, K, pad, signs):
        gen = torch.Generator(device="cuda").manual_seed(M + K)
        buf = torch.full((M, K + pad), 3.0e4, dtype=torch.bfloat16, device="cuda")
        self.x = buf[:, :K]
        self.x.copy_(torch.randn(M, K, generator=gen, device="cuda") * torch.exp2(
            torch.randint(-6, 7, (M, 1), generator=gen, device="cuda").float()))
        self.x[:, ::97] *= 30.0
        rng = np.random.default_rng(M)
        self.rows = np.unique(np.r_[0:min(M, 20), max(0, M - 20):M, rng.integers(0, M, 60)])
        self.sample = self.x[torch.from_numpy(self.rows).cuda()].cpu()
        self.signs = synth.rotation_signs(K, seed=3) if signs else None
        self.sign_bits = synth.bf16_bits(self.signs) if signs else None
        self.device_signs = self.signs.cuda() if signs else None


def launches(f, kernel):
    names = kernels_of(f)
    assert len(names) == 1 and kernel in names[0], names


def compare(bro, t, block, what, kernel, layout=0):
    M, K = t.x.shape
    rc, rs = oracle.rotate_quantize_mxfp4(synth.bf16_bits(t.sample), block, t.sign_bits)
    if what == CODES:
        codes, scales = Guarded(bro.codes_bytes(M, K)), Guarded(bro.scales_bytes(M, K, layout))
        launches(lambda: bro.rotate_quantize_mxfp4(t.x, block, codes.view, scales.view, layout, signs=t.device_signs), kernel)
        codes.check(), scales.check()
        s = scales.numpy()
        s = to_canonical(s, M, K) if layout else s.reshape(M, K // 32)
        assert np.array_equal(codes.numpy().reshape(M, K // 2)[t.rows], rc) and np.array_equal(s[t.rows], rs)
        if layout:                         # (the padding rows read as zero)
            last = scales.numpy().reshape(-1, 2 * ((K + 255) // 256), 32, 4, 4)[-1].transpose(2, 1, 0, 3).reshape(128, -1)
            assert not last[(M - 1) % 128 + 1:].any()
    elif what == BYTES:
        for shift in (0, 1):               # on a word and between
            out = Guarded(M * (K // 32) + shift)
            launches(lambda: bro.group_scale_bytes(t.x, block, out.view[shift:].view(M, K // 32), signs=t.device_signs), kernel)
            out.check()
            assert np.array_equal(out.numpy()[shift:].reshape(M, K // 32)[t.rows], rs)
    else:
        mse = Guarded(M * (K // 32) * 4)
        launches(lambda: bro.group_quant_error(t.x, block, mse.view.view(torch.float32).view(M, K // 32), t.device_signs), kernel)
        mse.check()
        got = mse.view.view(torch.float32).view(M, K // 32).cpu().numpy().astype(np.float64)[t.rows]
        ref = reference(t.sample, block, t.signs)
        # (32 squares in fp32, each with a few roundings, as in the tests of the small sizes)
        assert np.all(np.abs(got - ref) <= 1e-5 * ref + 1e-37)
    assert bro.last_device_status() == 0


@pytest.mark.parametrize("signs,pad", [(False, 0), (True, 8)])
@pytest.mark.parametrize("M,K,block", [(603, 1088, 64), (600, 1152, 128), (403, 4096, 64), (1187, 2176, 128)])
def test_64_channels_a_lane(bro, M, K, block, signs, pad):
    """Row tiles with rows missing, K that ends inside a tile of 128 channels, every output."""
    t = Large(M, K, pad, signs)
    for what in (CODES, BYTES, ERROR):
        compare(bro, t, block, what, WIDE)


@pytest.mark.parametrize("signs,pad", [(False, 0), (True, 8)])
def test_64_channels_a_lane_block_32(bro, signs, pad):
    """The error of a block of 32 from 2^25 elements, its codes at K with lanes to save."""
    t = Large(15889, 2112, pad, signs)
    compare(bro, t, 32, ERROR, WIDE)
    compare(bro, t, 32, CODES, WIDE, 1)


@pytest.mark.parametrize("signs,pad", [(False, 0), (True, 8)])
@pytest.mark.parametrize("what,M,K,kernel", [
    (CODES, 741, 2048, GLOBAL), (CODES, 740, 2048, FEW), (CODES, 149, 4096, GLOBAL), (CODES, 148, 4096, FEW), (CODES, 1, 2048, FEW),
    (CODES, 65537, 256, GLOBAL), (CODES, 1500, 256, SHUFFLES), (CODES, 2049, 512, GLOBAL), (CODES, 2048, 512, SHUFFLES), (CODES, 131, 1024, GLOBAL),
    (BYTES, 65537, 256, GLOBAL), (BYTES, 8193, 512, GLOBAL), (BYTES, 2049, 1024, GLOBAL), (BYTES, 2048, 1024, SHUFFLES),
    (ERROR, 8195, 256, GLOBAL), (ERROR, 4099, 512, GLOBAL), (ERROR, 2049, 1024, GLOBAL), (ERROR, 8192, 256, SHUFFLES)])
def test_full_dimension_on_either_side_of_the_lines(bro, what, M, K, kernel, signs, pad):
    t = Large(M, K, pad, signs)
    compare(bro, t, 0, what, kernel)
    if what == CODES:
        compare(bro, t, 0, what, kernel, 1)


@pytest.mark.parametrize("K", [8192, 32768])
def test_padding_of_one_row_of_the_full_dimension(bro, K):
    """More CTAs than rows, those that only clear."""
    t = Large(1, K, 0, True)
    compare(bro, t, 0, CODES, GLOBAL, 1)


def extremes(M, K):
    """Infinities, NaN, negative zeros, subnormals and maxima beyond the one-multiply range: in one group beside a usual one, in both."""
    gen = torch.Generator(device="cuda").manual_seed(K)
    x = torch.randn(M, K, generator=gen, device="cuda")
    rows = torch.arange(M, device="cuda")
    for i, v in enumerate((float("inf"), float("-inf"), float("nan"), 3.0e38, 1.0e-40, -0.0)):
        some = rows[rows % 7 == i]
        x[some, (some * 37 + i * 64) % K] = v
    x[::5, :64] *= 1.0e-38
    x[1::5, 32:96] *= 1.0e30
    x[2::35] = -0.0
    x[3::35, 64:] = 0.0
    return x.to(torch.bfloat16)


@pytest.mark.parametrize("M,K,block", [(603, 1088, 64), (600, 1152, 128), (16400, 2048, 32), (8200, 256, 0), (5000, 512, 0), (2100, 1024, 0),
                                       (1100, 2048, 0)])
def test_values_at_the_ends_of_the_range(bro, M, K, block):
    """The statistics of a large tensor against those of its rows in small calls, which other kernels compute — bytes the same, errors
    the same where they are no number or infinite, else up to the order of their 32 fp32 additions (31 roundings of each sum at
    most, 62 * 2^-24) — and its codes and scale bytes against each other."""
    x = extremes(M, K)
    full = [torch.empty(M, K // 32, dtype=dt, device="cuda") for dt in (torch.uint8, torch.float32)]
    launches(lambda: bro.group_quant_error(x, block, full[1]), GLOBAL if block == 0 else WIDE)
    bro.group_scale_bytes(x, block, full[0])
    codes, scales = bro.alloc_codes(M, K), bro.alloc_scales(M, K, 0)
    bro.rotate_quantize_mxfp4(x, block, codes, scales, 0)
    assert torch.equal(scales.view(M, K // 32), full[0])
    step = 70
    if K > 1024 and block == 0:            # (no other kernel: compare with single rows)
        step = 1
    for first in sorted({min(i * step, M - step) for i in (*range(12), M)}):
        part = x[first:first + step].contiguous()
        b, e = torch.empty_like(full[0][:step]), torch.empty_like(full[1][:step])
        bro.group_scale_bytes(part, block, b)
        bro.group_quant_error(part, block, e)
        assert torch.equal(b, full[0][first:first + step])
        g = full[1][first:first + step]
        assert torch.equal(torch.isnan(g), torch.isnan(e)) and torch.equal(torch.isinf(g), torch.isinf(e))
        ok = torch.isfinite(g)
        assert torch.all((g[ok] - e[ok]).abs() <= 62 * 2.0 ** -24 * e[ok])
        c, s = bro.alloc_codes(step, K), bro.alloc_scales(step, K, 0)
        flags = 0 if block == 0 else bro.FLAG_RQ_DIRECT
        bro.rotate_quantize_mxfp4(part, block, c, s, 0, flags=flags)
        assert torch.equal(c, codes[first:first + step]) and torch.equal(s.view(step, -1), b)
    assert bro.last_device_status() == 0
