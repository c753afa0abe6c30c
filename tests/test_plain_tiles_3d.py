"""3D FP32 half steps with straight code for tiles clear of everything, and the
instances without it, against the wavefront kernel (which has none): the same
arithmetic, so the same bits, on both sides of the lines between the two."""
import numpy as np
import pytest

from paper_2203_01462_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,npml,design,source,steps", [
    ((160, 48, 32), 4, (40, 12, 8), "dipole", 90),   # a quarter of the tiles are plain: plain instances
    ((160, 48, 32), 4, (90, 30, 16), "sheet", 90),   # most plain tiles hold design nodes
    ((129, 41, 27), 4, (40, 12, 8), "dipole", 90),   # ragged, a tenth: general instances
    ((160, 48, 32), 4, (40, 12, 8), "tfsf", 90),     # a small plane wave: general forward, plain adjoint
    ((128, 128, 128), 6, (40, 30, 20), "dipole", 24),   # 2^21 nodes
    ((128, 127, 128), 20, (20, 20, 20), "sheet", 24),   # just below, few plain tiles
    ((160, 152, 151), 8, (40, 30, 20), "tfsf", 24),  # 3.67e6 nodes with a plane wave: plain
    ((159, 152, 151), 8, (40, 30, 20), "tfsf", 24),  # just below: general forward
])
def test_same_bits_as_the_wavefront_kernel(n, npml, design, source, steps):
    from paper_2203_01462_gb300.binding import Solver
    w = I.workload_3d(*n, dx=20e-9, nsteps=steps, npml=npml, design=design, gap=(2, 2, 2), source=source, real="f32",
                      substrate=source == "sheet", tf_margin=1)
    w.update(I.pulse(800e-9, 900e12))
    if steps < 60 and source != "dipole":  # a source that the short run carries into the design box
        w["src_lo"][2], w["src_hi"][2] = w["design_lo"][2] - 3, w["design_lo"][2] - 2
        if source == "tfsf":
            w["tf_lo"][2] = w["design_lo"][2] - 1
    rho = I.rho_uniform(w, 82)
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
