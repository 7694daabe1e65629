"""Events and tile entries counted and written by blocks: both sides of the
number of blocks up to which a block adds up the counts itself, cells that begin
inside a block, and several cells in one."""
import numpy as np
import pytest

from paper_2503_00308_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def arlib():
    from paper_2503_00308_gb300 import _build, ar
    _build.build()
    assert torch.cuda.is_available()
    return ar


# events by blocks of 2048 pairs, entries by blocks of 256 events, 2048 of either at most
@pytest.mark.parametrize("n,cells", [
    (3, 1500),          # many cells to a block
    (2047, 3), (2049, 2),
    (32_768, 8), (32_769, 8),      # 524288 events in the batch, and more
    (299_593, 14), (299_594, 14),  # 4194302 pairs, and 4194316
])
@pytest.mark.parametrize("shift", [0, 2])
def test_a_batch_gives_the_bounds_of_its_cells(arlib, n, cells, shift):
    sc = synth.object_scene(n, n, mean_sd=0.25, logscale_mu=-3.0 if n < 100_000 else -6.0, logscale_sd=0.1, opacity_mu=1.0)
    cam = synth.look_camera(45, 35, 40.0, centre=(0, 0, -4))
    lo, hi = synth.cell_grid([0.01, 0.0, 0.004, 0.0, 0.0, 0.0], [cells, 1, 1, 1, 1, 1])
    s = arlib.Scene(sc)
    arlib.ar_debug_set_prefix(s.handle, shift)
    a, b = (torch.full((cells, 35, 45, 3), -7.0, device="cuda") for _ in range(2))
    s.render(cam, lo, hi, a, b, tile=16)
    for c in sorted({0, 1, cells // 2, cells - 1}):
        a1, b1 = (torch.full_like(t[:1], -7.0) for t in (a, b))
        s.render(cam, lo[c:c + 1], hi[c:c + 1], a1, b1, tile=16)
        assert torch.equal(a[c], a1[0]) and torch.equal(b[c], b1[0])
    s.close()
