"""E_z FP64 contexts of more than 450 000 nodes run temporally blocked launches
by default where the design box holds 4 % of them, and one launch per step where
it holds less; the same bits in W~ and the gap history (form 1 of the Drude
update in both), the gradient to the rounding of its FP64 sums."""
import numpy as np
import pytest

from paper_2203_01462_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,design,blocked", [((720, 640), (130, 140), False), ((720, 640), (140, 140), True),
                                              ((700, 640), (20, 20), True)])
def test_default(n, design, blocked):
    from paper_2203_01462_gb300.binding import Solver
    w = I.workload_2d(*n, dx=10e-9, nsteps=120, npml=8, design=design, gap=(3, 3), real="f64",
                      src_offset=n[1] // 2 - design[1] // 2 - 14)
    w.update(I.pulse(800e-9, 1200e12))
    rho = 0.1 * I.rho_uniform(w, 62)
    out, launches = [], []
    for steps in (0, 1):
        s = Solver(w)
        s.set_graphs(0)
        if steps:
            s.set_steps_per_launch(steps)
        s.set_design(rho)
        s.set_damping(5e5, 2.0)
        c = s.info().launches
        s.forward()
        launches.append(s.info().launches - c)
        W, g = s.evaluate(rho, 5e5, 2.0)
        gh = s.gap_history()
        s.sync()
        out.append((float(W.item()), g.cpu().numpy(), gh.cpu().numpy()))
    assert launches[1] >= w["nsteps"]
    assert launches[0] < w["nsteps"] if blocked else launches[0] == launches[1]
    assert out[0][0] > 0 and out[0][0] == out[1][0]
    np.testing.assert_array_equal(out[0][2], out[1][2])
    assert np.linalg.norm(out[0][1] - out[1][1]) <= 1e-12 * np.linalg.norm(out[1][1]) > 0
