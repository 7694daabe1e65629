"""The sweep of a tile by halves, taken with many segments of long lists,
against whole tiles."""
import numpy as np
import pytest

from paper_2503_00308_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
SEGMENTS, ENTRIES = 152, 64   # halves with at least this many segments and entries per segment


@pytest.fixture(scope="module")
def arlib():
    from paper_2503_00308_gb300 import _build, ar
    _build.build()
    assert torch.cuda.is_available()
    return ar


@pytest.mark.parametrize("rel", [False, True])
@pytest.mark.parametrize("move", ["x", "xyz_yaw", "6dof"])
@pytest.mark.parametrize("n,size,scale,sat", [
    (6000, (161, 119), 1.0, 0.0),      # ragged edges: the last halves hold 7 rows, the last tiles one column
    (20_000, (176, 72), 0.05, 0.0),    # narrow cells; the last row of tiles has an empty second half
    (40_000, (150, 100), 0.2, 0.05),   # faint: pixels stop late, sweeps go on in a wider window
])
def test_halves_give_the_bounds_of_whole_tiles(arlib, rel, move, n, size, scale, sat):
    """Four cells in one batch are swept by halves, each by itself by whole
    tiles: a pixel's sweep does not depend on the others, so the bounds are equal."""
    sc = synth.object_scene(n, 11)
    if sat:
        sc.opacity[:] = np.float32(sat)
    cam = synth.look_camera(*size, 1.1 * size[0])
    on = {"x": (1, 0, 0, 0, 0, 0), "xyz_yaw": (1, 1, 1, 0, 1, 0), "6dof": (1, 1, 1, 1, 1, 1)}[move]
    lo, hi = synth.cell_grid(scale * np.array(on) * np.array([0.02] * 3 + [0.008] * 3), [4, 1, 1, 1, 1, 1])
    tiles = -(-size[0] // 16) * -(-size[1] // 16)
    s = arlib.Scene(sc)
    if rel:
        arlib.ar_scene_set_blend(s.handle, arlib.AR_BLEND_RELATIONAL)
    a, b = (torch.full((4, size[1], size[0], 3), -7.0, device="cuda") for _ in range(2))
    s.render(cam, lo, hi, a, b, tile=16)
    st = arlib.ar_last_render_stats(s.handle)
    assert 4 * tiles >= SEGMENTS > tiles and 2 * st["n_entries"] >= ENTRIES * 4 * tiles
    for c in range(4):
        a1, b1 = (torch.full_like(t[:1], -7.0) for t in (a, b))
        s.render(cam, lo[c:c + 1], hi[c:c + 1], a1, b1, tile=16)
        assert torch.equal(a[c], a1[0]) and torch.equal(b[c], b1[0])
    s.close()
