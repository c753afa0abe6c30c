"""The FP32 sensitivity sums at strong sources.

One launch's products (E_z, up to 8 steps) or one chunk's (E in plane, up to
32) are summed in an FP32 pair before they enter the FP64 accumulator.  The
fields scale with src_amp, the products with its square: over the amplitudes
here they pass through the whole range of the pair's scaled words, the last
binades below its limit included, and every gradient entry has to stay finite
and scale with src_amp^2."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2203_01462_gb300 import inputs as I

pytestmark = pytest.mark.gpu

AMPS = [2.0 ** k for k in range(6, 27)] + [1e10, 1e16]


def evaluate(w, rho, steps=0):
    from paper_2203_01462_gb300.binding import Solver
    s = Solver(w)
    if steps:
        s.set_steps_per_launch(steps)
    g = s.evaluate(rho, 5e5, 2.0)[1].cpu().numpy()
    s.sync()
    return g


def test_ez_small_grid():
    """8 steps per launch, against the oracle at amplitude 1 (FP32 fields: 1e-3)."""
    w = I.workload_2d(96, 80, dx=20e-9, nsteps=600, npml=8, design=(40, 30), real="f32", src_offset=3)
    w.update(I.pulse(800e-9, 300e12))
    rho = I.rho_uniform(w, 91)
    ref = O.gradient(w, rho, 5e5, 2.0)["grad"].reshape(-1)
    for a in AMPS:
        g = evaluate(dict(w, src_amp=a), rho) / a ** 2
        assert np.isfinite(g).all(), a
        assert np.linalg.norm(g - ref) <= 1e-3 * np.linalg.norm(ref), a


@pytest.mark.parametrize("snap", [0, 40])
def test_inplane(snap):
    """Chunks of 32 steps, against one launch per half step, whose fields are
    the same bits and whose products go into the FP64 accumulator one by one."""
    w = I.workload_2d_inplane(91, 91, dx=20e-9, nsteps=500, npml=8, design=(40, 40), gap=(4, 4), real="f32",
                              material=I.SILVER, src_offset=3, snapshot_every=snap)
    w.update(I.pulse(800e-9, 300e12))
    rho = 0.3 * I.rho_uniform(w, 92)
    for a in AMPS:
        v = dict(w, src_amp=a)
        g, ref = evaluate(v, rho), evaluate(v, rho, 1)
        assert np.isfinite(ref).all() and np.linalg.norm(ref) > 0
        assert np.isfinite(g).all(), a
        assert np.linalg.norm(g - ref) <= 1e-12 * np.linalg.norm(ref), a


def test_ez_several_tiles_per_sm():
    """6 steps per launch, against one launch per step (the same field bits)."""
    w = I.workload_2d(600, 420, dx=20e-9, nsteps=520, npml=8, design=(300, 200), real="f32", src_offset=80)
    w.update(I.pulse(800e-9, 600e12))
    rho = 0.1 * I.rho_uniform(w, 93)
    for a in AMPS:
        v = dict(w, src_amp=a)
        g, ref = evaluate(v, rho), evaluate(v, rho, 1)
        assert np.isfinite(ref).all() and np.linalg.norm(ref) > 0
        assert np.isfinite(g).all(), a
        assert np.linalg.norm(g - ref) <= 1e-12 * np.linalg.norm(ref), a
