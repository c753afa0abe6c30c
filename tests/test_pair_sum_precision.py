"""The blocked FP32 adjoint's sensitivity sums are as good as FP64 sums of the
same products.  In plane, where up to 32 steps go into one sum: against one
launch per half step, whose fields are the same bits and whose products are
added up in FP64 one by one.  Each of those N additions rounds by 2^-54 of the
running sum in the mean, so the two may differ by about sqrt(N) 2^-53 of the
gradient: 2.3e-15 in the rms over 420 steps."""
import numpy as np
import pytest

from paper_2203_01462_gb300 import inputs as I


def case(nx, ny, design):
    w = I.workload_2d_inplane(nx, ny, dx=20e-9, nsteps=420, npml=10, design=design, gap=(4, 4), real="f32",
                              material=I.SILVER, src_offset=(ny - design[1]) // 2 - 13)
    w.update(I.pulse(413e-9, 300e12))
    return w


@pytest.mark.gpu
@pytest.mark.parametrize("nx,ny,design", [(120, 250, (60, 150)), (430, 158, (250, 60))])
def test_inplane_sums(nx, ny, design):
    from paper_2203_01462_gb300.binding import Solver
    w = case(nx, ny, design)
    u = I.rho_uniform(w, 94)
    rho = 0.03 * u + (0.35 + 0.6 * u) * I.rho_bowtie(w).reshape(-1)
    out = []
    for steps in (0, 1):
        s = Solver(w)
        if steps:
            s.set_steps_per_launch(steps)
        W, g = s.evaluate(rho, 5e5, 3.0)
        s.sync()
        out.append((float(W.item()), g.cpu().numpy()))
    assert out[0][0] > 0 and out[0][0] == out[1][0]
    assert np.linalg.norm(out[0][1] - out[1][1]) <= 2.3e-15 * np.linalg.norm(out[1][1]) > 0
