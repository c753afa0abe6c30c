"""In-plane FP64 contexts run temporally blocked launches by default where the
design box is enough of the grid, and one launch per half step elsewhere: which
of the two, what a context holds for it, and that the fields are the same bits
on both sides of the line (the gradient to the rounding of its FP64 sums)."""
import numpy as np
import pytest

from paper_2203_01462_gb300 import inputs as I

# grid, design box, blocked: one wave of tiles; on either side of the line
CASES = [((240, 200), (20, 20), True), ((400, 350), (120, 120), False), ((400, 350), (140, 140), True)]


def _case(n, design, real="f64"):
    w = I.workload_2d_inplane(*n, dx=10e-9, nsteps=160, npml=8, design=design, gap=(4, 4), real=real,
                              src_offset=n[1] // 2 - design[1] // 2 - 14, snapshot_every=32)
    w.update(I.pulse(800e-9, 900e12))
    return w


def test_memory_of_a_context_that_never_blocks():
    """No second state: with one launch per half step as the default, a context
    holds less than the FP32 context's words twice over."""
    from paper_2203_01462_gb300.binding import workspace_bytes
    for n, design, blocked in CASES:
        double, single = workspace_bytes(_case(n, design)), workspace_bytes(_case(n, design, "f32"))
        # (FP64 accumulators do not double, so even with the same buffers it is a little less)
        assert (double > 1.97 * single) == blocked, (n, design, double / single)


@pytest.mark.gpu
@pytest.mark.parametrize("n,design,blocked", CASES)
def test_default(n, design, blocked):
    from paper_2203_01462_gb300.binding import Solver
    w = _case(n, design)
    rho = I.rho_uniform(w, 61)
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
    assert launches[1] >= 2 * w["nsteps"]
    assert launches[0] < w["nsteps"] if blocked else launches[0] == launches[1]
    assert out[0][0] > 0 and out[0][0] == out[1][0]
    np.testing.assert_array_equal(out[0][2], out[1][2])
    assert np.linalg.norm(out[0][1] - out[1][1]) <= 1e-12 * np.linalg.norm(out[1][1]) > 0
