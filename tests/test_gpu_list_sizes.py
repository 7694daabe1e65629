"""Lists on both sides of the sizes at which the record build and the radix
sorts change their kernels."""
import numpy as np
import pytest

from paper_2503_00308_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
COOP_MAX = 20480     # records built by groups of lanes up to here, by one thread each above
TOL = 1e-4           # the parity contract


@pytest.fixture(scope="module")
def arlib():
    from paper_2503_00308_gb300 import _build, ar
    _build.build()
    assert torch.cuda.is_available()
    return ar


def render(ar, sc, cam, lo, hi, limit=0):
    s = ar.Scene(sc)
    if limit:
        ar.ar_set_workspace_limit(s.handle, limit)
    a = torch.full((lo.shape[0], cam.height, cam.width, 3), -7.0, device="cuda")
    b = torch.full_like(a, -7.0)
    s.render(cam, lo, hi, a, b, tile=16)
    st = ar.ar_last_render_stats(s.handle)
    torch.cuda.synchronize()
    s.close()
    return a, b, st


@pytest.mark.parametrize("move", ["x", "xyz_yaw", "6dof"])
def test_builders_give_the_same_records(arlib, move):
    """One batch's list is the one-thread builder's, a cell's alone the group
    builder's: the bounds and the counts of splits and fallbacks are the same.
    A camera inside a faint scene: nearly every record is built, some by
    splitting their cell, some of a high Taylor order."""
    sc = synth.box_scene(20_000, 3)
    sc.opacity[:] = np.float32(0.02)
    cam = synth.look_camera(256, 144, 180.0, centre=(0.0, 0.0, 0.0))
    on = {"x": (1, 0, 0, 0, 0, 0), "xyz_yaw": (1, 1, 1, 0, 1, 0), "6dof": (1, 1, 1, 1, 1, 1)}[move]
    hw = np.array(on) * np.array([0.05] * 3 + [0.02] * 3)
    lo, hi = synth.cell_grid(hw, [12, 1, 1, 1, 1, 1])
    a1, b1, one = render(arlib, sc, cam, lo, hi)
    a2, b2, each = render(arlib, sc, cam, lo, hi, limit=1 << 20)   # a cell per batch: at most 20000 records
    assert one["n_built"] > COOP_MAX and one["n_built"] == each["n_built"]
    assert torch.equal(a1, a2) and torch.equal(b1, b2)
    assert (one["n_split"], one["n_fallback"]) == (each["n_split"], each["n_fallback"])
    if move != "x":
        assert one["n_split"] > 0


@pytest.mark.parametrize("n", [1, 1023, 1024, 1025, 2049])
def test_sort_tile_edges(arlib, orc, n):
    """Two events per Gaussian, 2048 per tile of the radix sorts: a single tile
    (its histogram taken as the digits' totals) and more."""
    sc = synth.object_scene(n, 40 + n, mean_sd=0.3, logscale_mu=-3.5)
    cam = synth.look_camera(24, 16, 26.0, centre=(0, 0, -4))
    lo, hi = synth.cell_grid([0.01, 0.0, 0.01, 0.0, 0.004, 0.0], [1, 1, 2, 1, 1, 1])
    a, b, _ = render(arlib, sc, cam, lo, hi)
    for c in range(2):
        olo, ohi, frag = orc.render_abstract(sc, cam, lo[c], hi[c])
        e = np.maximum(np.abs(a[c].double().cpu().numpy() - olo), np.abs(b[c].double().cpu().numpy() - ohi)).max(axis=-1)
        assert e[frag == 0].max() <= TOL, (n, c, e.max())
