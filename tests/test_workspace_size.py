"""Device bytes of a context (no GPU): what is not live at the same time shares
memory, so a pixel takes 504 bytes for d <= 16 and 952 for d <= 32 in either
precision, plus a fixed part (padding to 128 rows of two arrays, alignment)."""
import pytest

import paper_2007_14283_gb300 as ms
from paper_2007_14283_gb300 import build


@pytest.fixture(scope="module", autouse=True)
def lib():
    build.build()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("dim,per_pixel", [(1, 505), (16, 505), (17, 953), (32, 953)])
def test_bytes_per_pixel(dim, per_pixel, precision):
    cfg = ms.ms_config_default(dim=dim, precision=precision)
    for n in (0, 1, 127, 128, 129, 5000, 262144, (1 << 24) - 1):
        assert ms.ms_workspace_bytes(cfg, n) <= per_pixel * n + 2 * 128 * 256 + 32 * 512
