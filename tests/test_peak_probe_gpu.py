"""The FMA rates that rooflines are stated against: an SM issues 128 FP32 FMAs and 2 FP64 FMAs per clock, so their
ratio is 64 at equal clocks; 66 leaves 3 % for the launches (it falls where the FP32 chains are throttled)."""
import pytest

from paper_1807_02718_gb300 import fh as F

pytestmark = pytest.mark.gpu


def test_fp64_rate_is_the_pipes():
    ratio = F.fh_probe_fma_peak(0, False, 16384) / F.fh_probe_fma_peak(0, True, 4096)
    assert ratio < 66.0, ratio
