"""Images of less than three tiles a side are swept by whole tiles, larger ones by
halves where the segments are many."""
import numpy as np
import pytest

from paper_2503_00308_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
SEGMENTS, ENTRIES = 152, 64   # of a batch that may be swept by halves: with a side of 48 pixels or more


@pytest.fixture(scope="module")
def arlib():
    from paper_2503_00308_gb300 import _build, ar
    _build.build()
    assert torch.cuda.is_available()
    return ar


@pytest.mark.parametrize("size,cells", [((47, 47), 20), ((48, 33), 26), ((31, 48), 26), ((20, 20), 40)])
@pytest.mark.parametrize("move", ["x", "xyz_yaw", "6dof"])
def test_a_batch_gives_the_bounds_of_its_cells(arlib, size, cells, move):
    """A cell by itself, a few segments, is swept by whole tiles: the bounds are equal."""
    sc = synth.object_scene(3000, 11)
    cam = synth.look_camera(*size, 1.1 * size[0])
    on = {"x": (1, 0, 0, 0, 0, 0), "xyz_yaw": (1, 1, 1, 0, 1, 0), "6dof": (1, 1, 1, 1, 1, 1)}[move]
    lo, hi = synth.cell_grid(np.array(on) * np.array([0.02] * 3 + [0.008] * 3), [cells, 1, 1, 1, 1, 1])
    tiles = -(-size[0] // 16) * -(-size[1] // 16)
    s = arlib.Scene(sc)
    a, b = (torch.full((cells, size[1], size[0], 3), -7.0, device="cuda") for _ in range(2))
    s.render(cam, lo, hi, a, b, tile=16)
    st = arlib.ar_last_render_stats(s.handle)
    assert cells * tiles >= SEGMENTS > tiles and 2 * st["n_entries"] >= ENTRIES * cells * tiles
    for c in (0, 1, cells - 1):
        a1, b1 = (torch.full_like(t[:1], -7.0) for t in (a, b))
        s.render(cam, lo[c:c + 1], hi[c:c + 1], a1, b1, tile=16)
        assert torch.equal(a[c], a1[0]) and torch.equal(b[c], b1[0])
    s.close()
