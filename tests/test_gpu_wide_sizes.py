"""The wide-patch sweep at the edges of its tiles (one row of 256 / G pixels a CTA, walked last to
first by the transpose): one pixel more or less than whole tiles, one tile only, and the class
counts on both sides of each lane count, against the same one-step oracle comparison and
tolerances as the other wide-patch sizes."""
import pytest

from tests.test_gpu_wide_patch import B, test_wide_sweep_step as _step  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W,K,M,sp,prec", [
    (15, 15, 9, 3, 1, "fp32"), (12, 17, 9, 5, 1, "fp32"), (13, 33, 16, 4, "inf", "fp32"),
    (10, 16, 17, 4, 2, "fp32"), (11, 23, 32, 3, 1, "fp32"), (10, 65, 4, 4, 1, "fp32"),
    (11, 31, 8, 3, 1, "fp32"), (13, 15, 17, 3, 1, "fp64")])
def test_wide_sweep_tile_edges(B, H, W, K, M, sp, prec):  # noqa: F811
    _step(B, H, W, K, M, sp, prec)
