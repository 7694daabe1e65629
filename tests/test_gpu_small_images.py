"""A batch of few segments, where tiles would be swept by halves, is swept by whole tiles
in low images whose middle row lies near the edge of tiles and in relational sweeps of
small screen boxes at six pose variables; a batch of more segments is not."""
import numpy as np
import pytest

from paper_2503_00308_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
# of a batch that may be swept by halves; below EDGE not with H < 96 and H % 32 < 6 or > 26,
# below SMALL_REL not the relational one of small boxes at six pose variables
SEGMENTS, ENTRIES, EDGE, SMALL_REL = 152, 64, 1216, 2280


@pytest.fixture(scope="module")
def arlib():
    from paper_2503_00308_gb300 import _build, ar
    _build.build()
    assert torch.cuda.is_available()
    return ar


@pytest.mark.parametrize("size,cells", [((47, 26), 26), ((47, 27), 26), ((33, 37), 20), ((31, 38), 26), ((60, 95), 7),
                                        ((60, 96), 7), ((33, 33), 135), ((33, 33), 136)])
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
    assert cells * tiles >= SEGMENTS > tiles and (cells * tiles >= EDGE) == (cells >= 136)
    assert 2 * st["n_entries"] >= ENTRIES * cells * tiles
    for c in (0, 1, cells - 1):
        a1, b1 = (torch.full_like(t[:1], -7.0) for t in (a, b))
        s.render(cam, lo[c:c + 1], hi[c:c + 1], a1, b1, tile=16)
        assert torch.equal(a[c], a1[0]) and torch.equal(b[c], b1[0])
    s.close()


@pytest.mark.parametrize("logscale,dense,cells", [(-4.5, False, 6), (-1.5, True, 6), (-4.5, False, 66)])
@pytest.mark.parametrize("move", ["xyz_yaw", "6dof"])
def test_relational_batches_give_the_bounds_of_their_cells(arlib, logscale, dense, cells, move):
    """Small and large boxes, and more segments; a cell by itself is swept by whole tiles."""
    sc = synth.object_scene(3000, 11, logscale_mu=logscale)
    cam = synth.look_camera(100, 77, 110.0)
    on = {"xyz_yaw": (1, 1, 1, 0, 1, 0), "6dof": (1, 1, 1, 1, 1, 1)}[move]
    lo, hi = synth.cell_grid(0.05 * np.array(on) * np.array([0.02] * 3 + [0.008] * 3), [cells, 1, 1, 1, 1, 1])
    s = arlib.Scene(sc)
    arlib.ar_scene_set_blend(s.handle, arlib.AR_BLEND_RELATIONAL)
    a, b = (torch.full((cells, 77, 100, 3), -7.0, device="cuda") for _ in range(2))
    s.render(cam, lo, hi, a, b, tile=16)
    st = arlib.ar_last_render_stats(s.handle)
    assert cells * 35 >= SEGMENTS and (cells * 35 >= SMALL_REL) == (cells == 66)
    assert 2 * st["n_entries"] >= ENTRIES * cells * 35
    assert (st["n_triples"] >= 32 * st["n_entries"]) == dense
    for c in (0, cells - 1):
        a1, b1 = (torch.full_like(t[:1], -7.0) for t in (a, b))
        s.render(cam, lo[c:c + 1], hi[c:c + 1], a1, b1, tile=16)
        assert torch.equal(a[c], a1[0]) and torch.equal(b[c], b1[0])
    s.close()
