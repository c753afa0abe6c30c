"""FP64 3D half steps (one node per thread, 8 x 4-node blocks) against the
wavefront kernel (four nodes per thread): the same arithmetic with every
rounding fixed, so the same bits, at sizes that leave blocks partly empty, with
kappa above 1, a Courant number that is not a power of two, a gap and a source
in the same rows, and no absorbing layer."""
import numpy as np
import pytest

from paper_2203_01462_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,npml,design,kw", [
    ((33, 21, 29), 4, (9, 7, 6), {}),
    ((32, 20, 24), 3, (9, 7, 6), dict(pml_kappa_max=2.5, pml_alpha_max=1e3)),
    ((41, 19, 23), 4, (20, 7, 6), dict(courant=0.41, eps_s=1.7, eps_g=1.3)),
    ((17, 13, 14), 0, (5, 4, 4), dict(courant=0.37)),
])
@pytest.mark.parametrize("source", ["dipole", "sheet"])
def test_same_bits_as_the_wavefront_kernel(n, npml, design, kw, source):
    from paper_2203_01462_gb300.binding import Solver
    w = I.workload_3d(*n, dx=20e-9, nsteps=90, npml=npml, design=design, gap=(2, 2, 2), source=source, real="f64",
                      substrate=source == "sheet", **kw)
    w.update(I.pulse(800e-9, 600e12))
    rho = I.rho_uniform(w, 81)
    out = []
    for wave in (0, 2):
        s = Solver(w)
        s.set_wavefront(wave)
        W, g = s.evaluate(rho, 5e5, 2.0)
        gh = s.gap_history()
        s.sync()
        out.append((float(W.item()), g.cpu().numpy(), gh.cpu().numpy()))
    assert np.isfinite(out[0][0]) and out[0][0] > 0
    assert out[0][0] == out[1][0]
    np.testing.assert_array_equal(out[0][1], out[1][1])
    np.testing.assert_array_equal(out[0][2], out[1][2])
