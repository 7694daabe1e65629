"""The concrete render's pair lists (ar_render_concrete): Gaussians taken 32 at a
time, pairs beyond the cutoff dropped by an FP32 test, groups of equal depth,
against the oracle's FP64 render.

Tolerance: both sides blend in FP64 (the colour left out by the early stop is
below 1e-13), and the output is rounded to float32: half an ulp below 1 is
2^-25, doubled here."""
import numpy as np
import pytest

from paper_2503_00308_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
TOL = 2.0 ** -24


@pytest.fixture(scope="module")
def arlib():
    from paper_2503_00308_gb300 import _build, ar
    _build.build()
    assert torch.cuda.is_available()
    return ar


@pytest.mark.parametrize("n", [1, 31, 32, 33, 64, 97])
@pytest.mark.parametrize("kind", ["spread", "one_depth", "needles", "faint"])
def test_pair_lists(arlib, orc, n, kind):
    """Lists that end on, before and after a batch of 32; one group of equal
    depths (no Gaussian occludes another); covariances so narrow that the FP32
    test is off; opacities around the 1/255 cutoff."""
    sc = synth.object_scene(n, 100 + n, mean_sd=0.2, logscale_mu=-2.5)
    if kind == "one_depth":
        sc.uw[:, 2] = np.float32(0.25)
    elif kind == "needles":
        sc.logscale[:, 0] = np.float32(-1.5)
        sc.logscale[:, 1:] = np.float32(-12.0)
    elif kind == "faint":
        sc.opacity[:] = np.linspace(0.003, 0.02, n).astype(np.float32)
    cam = synth.look_camera(37, 21, 40.0, centre=(0, 0, -4))
    deltas = np.array([[0.0] * 6, [0.02, -0.01, 0.03, 0.0, 0.0, 0.0], [0.01, 0.0, 0.0, 0.004, -0.006, 0.008]])
    s = arlib.Scene(sc)
    out = torch.full((3, cam.height, cam.width, 3), -7.0, device="cuda")
    s.render_concrete(cam, deltas, out)
    torch.cuda.synchronize()
    s.close()
    for p in range(3):
        ref = np.asarray(orc.render_concrete(sc, cam, deltas[p]))
        assert np.abs(out[p].double().cpu().numpy() - ref).max() <= TOL, (kind, n, p)
