"""GPU parity of the full-dimension rotation of few rows, every row length, in all three outputs — codes, scale bytes, MXFP4 error —
against the CPU oracle.  (Which kernel computes which at which size, and those that only many rows reach: test_gpu_large_forms.py.)"""
import pytest

from paper_2511_04214_b200 import synth
from test_gpu_rotate_quantize_wide import all_outputs, device_copy

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bro():
    from paper_2511_04214_b200 import binding
    return binding


@pytest.mark.parametrize("M,K", [(1, 256), (7, 256), (9, 512), (130, 512), (3, 1024), (131, 1024), (5, 2048), (129, 2048), (2, 4096), (150, 4096),
                                 (1, 8192), (130, 8192), (3, 16384), (2, 32768)])
@pytest.mark.parametrize("signs", [False, True])
def test_full_dimension_units(bro, M, K, signs):
    """Several rows at a time (the last ones missing), one row in a warp, in several warps; rows with gaps."""
    x = synth.activations(M, K, seed=M + K)
    s = synth.rotation_signs(K, seed=3) if signs else None
    all_outputs(bro, x, device_copy(x, 8 if signs else 0), 0, s, 0)
