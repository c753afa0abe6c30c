"""3D FP64 grids of more rows or planes than one launch's blocks: a structure
across the border between two launches gives the bits of the same structure in
a short grid whose ends are too far away to matter (a step reaches one node)."""
import numpy as np
import pytest

from paper_2203_01462_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _case(axis, n, at):
    """A grid n nodes long along axis, the structure's centre on node `at`."""
    size = [9, 8, 8]
    size[axis] = n
    w = I.workload_3d(*size, dx=20e-9, nsteps=60, npml=0, design=(5, 4, 4), gap=(2, 2, 2), source="dipole", real="f64")
    w.update(I.pulse(800e-9, 900e12))
    for k in ("design", "gap", "src"):
        lo, hi = list(w[k + "_lo"]), list(w[k + "_hi"])
        lo[axis], hi[axis] = lo[axis] + at - n // 2, hi[axis] + at - n // 2
        w[k + "_lo"], w[k + "_hi"] = lo, hi
    return w


@pytest.mark.parametrize("axis,border", [(2, 65535), (1, 4 * 65535)])
def test_more_tiles_than_one_launch(axis, border):
    from paper_2203_01462_gb300.binding import Solver
    out = []
    for w in (_case(axis, 140, 70), _case(axis, border + 70, border)):
        s = Solver(w)
        W, g = s.evaluate(I.rho_uniform(w, 17), 5e5, 2.0)
        gh = s.gap_history()
        s.sync()
        out.append((float(W.item()), g.cpu().numpy(), gh.cpu().numpy()))
    assert np.isfinite(out[0][0]) and out[0][0] > 0
    assert out[0][0] == out[1][0]
    np.testing.assert_array_equal(out[0][1], out[1][1])
    np.testing.assert_array_equal(out[0][2], out[1][2])
