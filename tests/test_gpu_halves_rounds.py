"""The halves of tiles over several rounds: parts that are abandoned and swept
again beside parts that are complete, with pixels listed for the FP64 sweep."""
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
@pytest.mark.parametrize("shift", [0, 3])
@pytest.mark.parametrize("threshold", [0.0, 1e-6])
def test_restarted_halves_give_the_bounds_of_whole_tiles(arlib, rel, move, shift, threshold):
    """Lists longer than the first window (512 entries) and than their depth prefix, so that
    segments restart; a cell by itself is swept by whole tiles."""
    sc = synth.cube_scene(2000, 1)
    sc.opacity[:] = np.float32(0.3)
    cam = synth.look_camera(171, 125, 171.0, centre=(0.0, 0.0, -1.5))
    on = {"x": (1, 0, 0, 0, 0, 0), "xyz_yaw": (1, 1, 1, 0, 1, 0), "6dof": (1, 1, 1, 1, 1, 1)}[move]
    lo, hi = synth.cell_grid(0.3 * np.array(on) * np.array([0.05] * 3 + [0.02] * 3), [4, 1, 1, 1, 1, 1])
    tiles = -(-cam.width // 16) * -(-cam.height // 16)

    def render(c0, c1):
        s = arlib.Scene(sc)   # (a fresh one: the first window is learned from render to render)
        arlib.ar_debug_set_prefix(s.handle, shift)
        arlib.ar_scene_set_fp64_alpha(s.handle, threshold)
        if rel:
            arlib.ar_scene_set_blend(s.handle, arlib.AR_BLEND_RELATIONAL)
        a, b = (torch.full((c1 - c0, cam.height, cam.width, 3), -7.0, device="cuda") for _ in range(2))
        s.render(cam, lo[c0:c1], hi[c0:c1], a, b, tile=16)
        st = arlib.ar_last_render_stats(s.handle)
        s.close()
        return a, b, st

    a, b, st = render(0, 4)
    assert 4 * tiles >= SEGMENTS > tiles and 2 * st["n_entries"] >= ENTRIES * 4 * tiles
    assert st["n_restarted"] > 0 and st["n_fp64_segments"] > 0
    for c in range(4):
        a1, b1, _ = render(c, c + 1)
        assert torch.equal(a[c], a1[0]) and torch.equal(b[c], b1[0])
