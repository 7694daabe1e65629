"""Sorts on both sides of the length up to which a pass is one launch."""
import numpy as np
import pytest

from paper_2503_00308_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
SHORT = 64 * 512   # items of a short sort at most; its blocks take 512


@pytest.fixture(scope="module")
def arlib():
    from paper_2503_00308_gb300 import _build, ar
    _build.build()
    assert torch.cuda.is_available()
    return ar


@pytest.mark.parametrize("tile", [8, 16])
@pytest.mark.parametrize("n", [256, 257, SHORT // 4, SHORT // 4 + 1, SHORT // 2, SHORT // 2 + 1])
def test_short_and_long_sorts_agree(arlib, n, tile):
    """Two events per Gaussian and cell: two cells in one batch sort twice the
    events of one, so that either, or only one cell's, is short; the bounds are equal."""
    sc = synth.object_scene(n, 5 + n, mean_sd=0.25, logscale_mu=-3.0, logscale_sd=0.1, opacity_mu=1.0)
    cam = synth.look_camera(120, 90, 90.0, centre=(0, 0, -4))
    lo, hi = synth.cell_grid([0.004, 0.002, 0.004, 0.0, 0.002, 0.0], [1, 1, 2, 1, 1, 1])
    s = arlib.Scene(sc)
    a, b = (torch.full((2, 90, 120, 3), -7.0, device="cuda") for _ in range(2))
    s.render(cam, lo, hi, a, b, tile=tile)
    assert arlib.ar_last_render_stats(s.handle)["n_records"] == 2 * n   # every Gaussian has its events
    for c in range(2):
        a1, b1 = (torch.full_like(t[:1], -7.0) for t in (a, b))
        s.render(cam, lo[c:c + 1], hi[c:c + 1], a1, b1, tile=tile)
        assert torch.equal(a[c], a1[0]) and torch.equal(b[c], b1[0])
    s.close()
