"""The two forms of the FP64 sweep: lanes on the evaluations of a few pixels, and
a lane per pixel where nearly every pixel is listed."""
import numpy as np
import pytest

from paper_2503_00308_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
# a lane per pixel from two work items (of 8 pixels) per resident CTA, eleven per
# SM, and four items per listed segment
SM_ITEMS, SEGMENT_ITEMS = 2 * 11, 4


@pytest.fixture(scope="module")
def arlib():
    from paper_2503_00308_gb300 import _build, ar
    _build.build()
    assert torch.cuda.is_available()
    return ar


@pytest.mark.parametrize("tile", [8, 16])
@pytest.mark.parametrize("rel", [False, True])
@pytest.mark.parametrize("move", ["x", "xyz_yaw", "6dof"])
@pytest.mark.parametrize("shift", [0, 2])
def test_both_forms_give_the_same_bounds(arlib, tile, rel, move, shift):
    """Every evaluation in FP64 (threshold 0): a batch of cells is swept with a lane per
    pixel, a cell by itself has too few items for that.  The bounds are equal."""
    sc = synth.object_scene(2000, 17, mean_sd=0.8, logscale_mu=-2.0)
    sc.opacity[:] = np.float32(0.2)
    cam = synth.look_camera(173, 141, 120.0)   # ragged: 99 tiles of 16, 396 of 8
    on = {"x": (1, 0, 0, 0, 0, 0), "xyz_yaw": (1, 1, 1, 0, 1, 0), "6dof": (1, 1, 1, 1, 1, 1)}[move]
    lo, hi = synth.cell_grid(0.1 * np.array(on) * np.array([0.02] * 3 + [0.008] * 3), [3, 1, 1, 1, 1, 1])
    most = SM_ITEMS * torch.cuda.get_device_properties(0).multi_processor_count
    tiles = -(-cam.width // tile) * -(-cam.height // tile)
    assert tiles * tile * tile // 8 < most      # a cell's items, all pixels of all tiles listed
    s = arlib.Scene(sc)
    arlib.ar_debug_set_prefix(s.handle, shift)
    if rel:
        arlib.ar_scene_set_blend(s.handle, arlib.AR_BLEND_RELATIONAL)

    def render(c0, c1):
        a, b = (torch.full((c1 - c0, cam.height, cam.width, 3), -7.0, device="cuda") for _ in range(2))
        s.render(cam, lo[c0:c1], hi[c0:c1], a, b, tile=tile)
        return a, b, arlib.ar_last_render_stats(s.handle)

    arlib.ar_scene_set_fp64_alpha(s.handle, 1e30)
    f32 = render(0, 3)
    arlib.ar_scene_set_fp64_alpha(s.handle, 0.0)
    a, b, st = render(0, 3)
    listed = int(((a != f32[0]) | (b != f32[1])).any(dim=-1).sum())   # at least these
    assert listed // 8 >= max(most, SEGMENT_ITEMS * st["n_fp64_segments"])
    for c in range(3):
        a1, b1, _ = render(c, c + 1)
        assert torch.equal(a[c], a1[0]) and torch.equal(b[c], b1[0])
    s.close()
