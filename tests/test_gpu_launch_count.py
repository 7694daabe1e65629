"""ar_render_stats.n_launches against the kernels that the CUDA profiler sees."""
import numpy as np
import pytest

from paper_2503_00308_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DIMS = {"x": (1, 0, 0, 0, 0, 0), "xyz_yaw": (1, 1, 1, 0, 1, 0), "6dof": (1, 1, 1, 1, 1, 1)}


@pytest.fixture(scope="module")
def arlib():
    from paper_2503_00308_gb300 import _build, ar
    _build.build()
    assert torch.cuda.is_available()
    return ar


def kernels(call):
    from torch.profiler import ProfilerActivity, profile
    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        call()
        torch.cuda.synchronize()
    return sum("ar::" in e.name for e in prof.events())


@pytest.fixture(scope="module")
def seen(arlib):
    """Whether the profiler works here (its first session may see nothing)."""
    w = synth.tiny64()
    s = arlib.Scene(w.scene)
    a, b = (torch.empty((1, 32, 32, 3), device="cuda") for _ in range(2))
    n = [kernels(lambda: s.render(w.camera, w.cells_lo, w.cells_hi, a, b, tile=16)) for _ in range(2)]
    s.close()
    if not n[1]:
        pytest.skip("the profiler sees no kernels")


@pytest.mark.parametrize("move,n,size,cells,tile,more", [
    ("x", 64, (32, 32), 1, 16, {}),                          # one round
    ("6dof", 3000, (120, 90), 1, 8, {}),                     # two
    ("xyz_yaw", 5000, (120, 90), 5, 16, {}),                 # three; more pairs than the group builder takes
    ("6dof", 5000, (120, 90), 5, 8, {"prefix": 2}),          # two phases of binning
    ("x", 3000, (120, 90), 4, 16, {"cull": 1}),
    ("6dof", 3000, (120, 90), 4, 16, {"fp64": 1e-6}),        # both forms of the FP64 sweep
    ("xyz_yaw", 3000, (120, 90), 6, 16, {"limit": 1 << 20}), # a batch per cell
    ("6dof", 500, (60, 40), 2, 16, {"plain": True}),
])
@pytest.mark.parametrize("graphs", [False, True])
def test_launches_are_counted(arlib, seen, move, n, size, cells, tile, more, graphs):
    sc = synth.object_scene(n, 3)
    cam = synth.look_camera(*size, 1.1 * size[0])
    lo, hi = synth.cell_grid(np.array(DIMS[move]) * np.array([0.02] * 3 + [0.008] * 3), [cells, 1, 1, 1, 1, 1])
    s = arlib.Scene(sc)
    arlib.ar_scene_set_graphs(s.handle, graphs)
    if "prefix" in more:
        arlib.ar_debug_set_prefix(s.handle, more["prefix"])
    if "cull" in more:
        arlib.ar_debug_set_cull(s.handle, more["cull"])
    if "fp64" in more:
        arlib.ar_scene_set_fp64_alpha(s.handle, more["fp64"])
    if "limit" in more:
        arlib.ar_set_workspace_limit(s.handle, more["limit"])
    a, b = (torch.empty((cells, size[1], size[0], 3), device="cuda") for _ in range(2))
    render = s.render_plain_fp64 if "plain" in more else s.render
    for _ in range(3):
        seen_now = kernels(lambda: render(cam, lo, hi, a, b, tile=tile))
        assert arlib.ar_last_render_stats(s.handle)["n_launches"] == seen_now
    s.close()
