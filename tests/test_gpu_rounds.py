"""Renders that take one windowed round, two or three."""
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


@pytest.mark.parametrize("tile", [8, 16])
@pytest.mark.parametrize("n", [256, 257, 4096, 4097, 16384, 16385])
def test_the_number_of_rounds_changes_no_bound(arlib, n, tile):
    """A first render has a window of 512 entries: 512 events need one round,
    32768 at most two.  With a depth prefix forced there are always three.
    Faint, so that sweeps go past the window."""
    sc = synth.object_scene(n, 9 + n, mean_sd=0.25, logscale_mu=-1.5, logscale_sd=0.1)
    sc.opacity[:] = np.float32(0.02)
    cam = synth.look_camera(40, 24, 30.0, centre=(0, 0, -4))
    lo, hi = synth.cell_grid([0.004, 0.002, 0.004, 0.0, 0.002, 0.0], [1, 1, 1, 1, 1, 1])
    out = []
    for shift in (0, 3):
        s = arlib.Scene(sc)
        arlib.ar_debug_set_prefix(s.handle, shift)
        a, b = (torch.full((1, 24, 40, 3), -7.0, device="cuda") for _ in range(2))
        s.render(cam, lo, hi, a, b, tile=tile)
        st = arlib.ar_last_render_stats(s.handle)
        assert st["n_records"] == n
        if shift == 0 and n != 257:   # (257: no tile need have all of them)
            assert (st["n_restarted"] > 0) == (n > 256)
        out.append((a, b))
        s.close()
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
