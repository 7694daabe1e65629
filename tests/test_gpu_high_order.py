"""The last kernel of the record build finishes every pair that it is given as
one of a high Taylor order, also where MatrixInv does not hold on the cell."""
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


@pytest.mark.parametrize("dims,shift,degrees", [
    ((0, 0, 1, 0, 0, 0), 0.3, 0.0),
    ((1, 1, 1, 0, 1, 0), 0.1, 3.0),
    ((1, 1, 1, 1, 1, 1), 0.05, 2.5),
])
def test_high_order_list_leaves_no_record_unfinished(arlib, orc, dims, shift, degrees):
    """The same records, bit for bit, whether the pairs go through the build's
    own lists or all through the high-order list."""
    sc = synth.cube_scene(60, 3, half=0.3)
    cam = synth.look_camera(32, 32, 28.0, centre=(0, 0, -1.0))
    clo = -np.array(dims) * np.array([shift] * 3 + [degrees * synth.DEG] * 3)
    rec = orc.records(sc, cam, clo, -clo)
    seen = rec["valid"] > 0
    assert (seen & (rec["pieces"] > 0)).any()      # MatrixInv holds on pieces of the cell only
    gi = np.repeat(np.arange(sc.n), 4)
    px, py = np.tile([3, 16, 16, 28], sc.n), np.tile([9, 16, 17, 20], sc.n)
    out = []
    for on in (False, True):
        s = arlib.Scene(sc)
        arlib.ar_debug_set_high_order(s.handle, on)
        out.append(s.debug_alpha(cam, clo, -clo, gi, px, py, 0))
        s.close()
    assert (out[0][:, 39].astype(int) & 1).sum() >= 4 * seen.sum() * 0.9
    assert np.array_equal(out[0][:, 39], out[1][:, 39])
    for o in out:
        o[(o[:, 39].astype(int) & 4) != 0, 21:33] = 0.0   # a pair that falls back has no W
    assert np.array_equal(out[0], out[1])
