"""Long radix sorts, whose tiles hold 2048 items, around the edge of a tile and
with more cells than one digit counts."""
import numpy as np
import pytest

from paper_2503_00308_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
SHORT, TILE = 64 * 512, 2048   # items of a short sort at most; of a long one's tile


@pytest.fixture(scope="module")
def arlib():
    from paper_2503_00308_gb300 import _build, ar
    _build.build()
    assert torch.cuda.is_available()
    return ar


@pytest.mark.parametrize("n,cells", [
    (17 * TILE // 4 - 1, 2), (17 * TILE // 4, 2), (17 * TILE // 4 + 1, 2),   # a pair of each cell less, none, one more
    (65, 256), (64, 257), (60, 300),                                         # one cell digit, and two
])
@pytest.mark.parametrize("shift", [0, 2])
def test_long_sorts_agree_with_the_short_sorts_of_the_cells(arlib, n, cells, shift):
    """The events of the batch (and of (cell, tile) entries as many at least) make a
    long sort, those of a cell by itself a short one: the bounds are equal."""
    sc = synth.object_scene(n, 5 + n, mean_sd=0.25, logscale_mu=-3.0, logscale_sd=0.1, opacity_mu=1.0)
    cam = synth.look_camera(45, 35, 40.0, centre=(0, 0, -4))
    lo, hi = synth.cell_grid([0.01, 0.0, 0.004, 0.0, 0.0, 0.0], [cells, 1, 1, 1, 1, 1])
    s = arlib.Scene(sc)
    arlib.ar_debug_set_prefix(s.handle, shift)
    a, b = (torch.full((cells, 35, 45, 3), -7.0, device="cuda") for _ in range(2))
    s.render(cam, lo, hi, a, b, tile=16)
    assert arlib.ar_last_render_stats(s.handle)["n_records"] == cells * n   # every pair has its two events
    assert 2 * n <= SHORT < 2 * n * cells
    for c in sorted({0, 1, cells // 2, cells - 1}):
        a1, b1 = (torch.full_like(t[:1], -7.0) for t in (a, b))
        s.render(cam, lo[c:c + 1], hi[c:c + 1], a1, b1, tile=16)
        assert torch.equal(a[c], a1[0]) and torch.equal(b[c], b1[0])
    s.close()
