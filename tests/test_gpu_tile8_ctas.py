"""The sweep at tile 8: fewer segments run four CTAs per SM, more run six."""
import numpy as np
import pytest

from paper_2503_00308_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
SIX = 4256   # segments from which six run


@pytest.fixture(scope="module")
def arlib():
    from paper_2503_00308_gb300 import _build, ar
    _build.build()
    assert torch.cuda.is_available()
    return ar


@pytest.mark.parametrize("rel", [False, True])
@pytest.mark.parametrize("move", ["x", "xyz_yaw", "6dof"])
@pytest.mark.parametrize("size,cells", [((64, 56), 76), ((61, 50), 75), ((400, 304), 3)])
def test_both_give_the_same_bounds(arlib, rel, move, size, cells):
    """A batch of cells at the line or above it, one less below it or a cell by itself: the
    bounds are equal."""
    tiles = -(-size[0] // 8) * -(-size[1] // 8)
    sc = synth.object_scene(3000, 11)
    cam = synth.look_camera(*size, 1.1 * size[0])
    on = {"x": (1, 0, 0, 0, 0, 0), "xyz_yaw": (1, 1, 1, 0, 1, 0), "6dof": (1, 1, 1, 1, 1, 1)}[move]
    lo, hi = synth.cell_grid(np.array(on) * np.array([0.05] * 3 + [0.01] * 3), [cells, 1, 1, 1, 1, 1])
    s = arlib.Scene(sc)
    if rel:
        arlib.ar_scene_set_blend(s.handle, arlib.AR_BLEND_RELATIONAL)

    def render(c0, c1):
        a, b = (torch.full((c1 - c0, size[1], size[0], 3), -7.0, device="cuda") for _ in range(2))
        s.render(cam, lo[c0:c1], hi[c0:c1], a, b, tile=8)
        return a, b

    a, b = render(0, cells)
    assert (cells - 1) * tiles < SIX and (cells * tiles >= SIX) == (size != (61, 50))
    a1, b1 = render(0, cells - 1)
    assert torch.equal(a[:-1], a1) and torch.equal(b[:-1], b1)
    a1, b1 = render(cells - 1, cells)
    assert torch.equal(a[-1:], a1) and torch.equal(b[-1:], b1)
    s.close()
