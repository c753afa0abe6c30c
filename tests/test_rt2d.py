"""Temporally blocked 2D E_z launches with the tile in registers (the default
on small and medium grids) against one launch per step, through the C ABI.

Both run the same per-node arithmetic in the same rounding order, so W~ and
the gap history agree bit for bit; the gradient's FP32 products of one launch
are summed as exact FP32 pairs before they enter the FP64 accumulator, which
leaves a relative error of a few 2^-47 per launch: 1e-12 L2.  The grids put
tile edges, walls, CPML, gap and source on the region's first and last rows
and columns: one node less and more than one tile, a grid smaller than a
tile, the smallest one, no CPML, kappa and alpha in the CPML, a gap too large
for the staging buffer, a design box up to the walls, run lengths and
checkpoint intervals that leave launches of every step count, runs that end
while the gap field is still a front of 1e-30, and source amplitudes whose
products leave the FP32 range."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2203_01462_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def case(nx, ny, real, **kw):
    n = kw.pop("npml", 6)
    d = kw.pop("design", (max(3, nx - 2 * n - 6), max(3, ny - 2 * n - 6)))
    w = I.workload_2d(nx, ny, dx=20e-9, nsteps=kw.pop("nsteps", 149), npml=n, design=d, gap=kw.pop("gap", (2, 1)),
                      real=real, src_offset=kw.pop("src_offset", 1), **kw)
    w.update(I.pulse(800e-9, 1200e12))
    return w


def run(w, rho, spl):
    from paper_2203_01462_gb300.binding import Solver
    s = Solver(w)
    if spl:
        s.set_steps_per_launch(spl)
    W, g = s.evaluate(rho, 5e5, 2.0)
    gh = s.gap_history()
    s.sync()
    return float(W.item()), g.cpu().numpy(), gh.cpu().numpy(), s.info().launches


CASES = [
    ("f64", dict(nx=24, ny=24)), ("f64", dict(nx=25, ny=23)), ("f64", dict(nx=49, ny=17, npml=3)),
    ("f64", dict(nx=6, ny=6, npml=1, design=(2, 2), gap=(1, 1), src_offset=0)),
    ("f64", dict(nx=61, ny=47, npml=0, src_offset=3)), ("f64", dict(nx=75, ny=70, snapshot_every=7)),
    ("f64", dict(nx=40, ny=44, pml_kappa_max=3.0, pml_alpha_max=1e3)),
    ("f32", dict(nx=700, ny=220, nsteps=230)), ("f32", dict(nx=673, ny=256, npml=10, snapshot_every=19)),
    ("f32", dict(nx=640, ny=256, npml=0, src_offset=40, filter_radius=3, nsteps=301)),
    ("f32", dict(nx=600, ny=300, npml=10, gap=(17, 17), design=(300, 60), src_offset=80, nsteps=301)),
    ("f32", dict(nx=650, ny=241, pml_kappa_max=2.0, pml_alpha_max=1e3, courant=0.25, eps_s=1.7, eps_g=1.3, nsteps=500, src_offset=90)),
    ("f32", dict(nx=601, ny=270, npml=0, design=(601, 270), src_offset=100, nsteps=301)),
    # many tiles, most of them of the background or of the design box alone
    ("f32", dict(nx=1501, ny=1420, npml=10, design=(700, 150), src_offset=610, nsteps=301, snapshot_every=50)),
]


@pytest.mark.parametrize("real,kw", CASES)
def test_blocked_equals_one_launch_per_step(real, kw):
    w = case(real=real, **kw)
    rho = 0.1 * I.rho_uniform(w, 71)
    W1, g1, h1, n1 = run(w, rho, 1)
    W, g, h, n = run(w, rho, 0)
    assert n < n1
    assert np.isfinite(W1) and W1 > 0
    assert W == W1
    np.testing.assert_array_equal(h, h1)
    assert np.linalg.norm(g - g1) <= 1e-12 * np.linalg.norm(g1)


def plane(nx, ny, real, **kw):
    n = kw.pop("npml", 6)
    d = kw.pop("design", (max(3, nx - 2 * n - 7), max(3, ny - 2 * n - 7)))
    w = I.workload_2d_inplane(nx, ny, dx=20e-9, nsteps=kw.pop("nsteps", 170), npml=n, design=d, gap=kw.pop("gap", (2, 1)),
                              real=real, material=I.SILVER, src_offset=kw.pop("src_offset", 1), **kw)
    w.update(I.pulse(800e-9, 1200e12))
    return w


PLANE = [
    ("f64", dict(nx=24, ny=25)), ("f64", dict(nx=49, ny=17, npml=3)), ("f64", dict(nx=57, ny=48, npml=0, src_offset=3)),
    ("f64", dict(nx=7, ny=7, npml=1, design=(2, 2), gap=(1, 1), src_offset=1)),
    ("f64", dict(nx=75, ny=70, snapshot_every=7)),
    ("f32", dict(nx=41, ny=37)), ("f32", dict(nx=48, ny=33, snapshot_every=33)), ("f32", dict(nx=97, ny=95, npml=0)),
    ("f32", dict(nx=130, ny=121, npml=10, gap=(24, 22), snapshot_every=45, nsteps=230)),
    ("f32", dict(nx=321, ny=60, design=(280, 41), src_offset=0)),
    ("f32", dict(nx=60, ny=61, npml=0, design=(59, 60), src_offset=10)),
]


@pytest.mark.parametrize("real,kw", PLANE)
def test_inplane_blocked_equals_one_launch_per_half_step(real, kw):
    """E in plane: the default (blocked launches, sensitivities summed from
    the records of up to 32 adjoint steps) against one launch per half step,
    with a gap record beyond the staging buffer, chunks of every length and
    a design box up to the walls."""
    w = plane(real=real, **kw)
    rho = 0.1 * I.rho_uniform(w, 73)
    W1, g1, h1, n1 = run(w, rho, 1)
    W, g, h, n = run(w, rho, 0)
    assert n < n1
    assert np.isfinite(W1) and W1 > 0
    assert W == W1
    np.testing.assert_array_equal(h, h1)
    assert np.linalg.norm(g - g1) <= 1e-12 * np.linalg.norm(g1)


def test_inplane_blocked_with_kappa():
    """kappa above 1 in the CPML: the product by 1/kappa and the sum with psi
    may be rounded together, so FP64 agreement rather than equal bits."""
    w = plane(60, 57, "f64", pml_kappa_max=3.0, pml_alpha_max=1e3)
    rho = 0.1 * I.rho_uniform(w, 74)
    W1, g1, h1, _ = run(w, rho, 1)
    W, g, h, _ = run(w, rho, 0)
    assert abs(W - W1) <= 1e-11 * W1
    assert np.max(np.abs(h - h1)) <= 1e-11 * np.max(np.abs(h1))
    assert np.linalg.norm(g - g1) <= 1e-11 * np.linalg.norm(g1)


@pytest.mark.parametrize("amp", [1e-17, 1e16])
def test_sensitivity_sum_follows_the_source_amplitude(amp):
    """The fields scale with src_amp, the gradient with its square: products
    of 1e-34 and below (or 1e32) in FP32 lose nothing against amplitude 1."""
    w = I.small_2d(nx=41, ny=37, nsteps=400, dx=20e-9, npml=6, design=(17, 15), real="f32")
    w.update(I.pulse(800e-9, 300e12))
    rho = I.rho_uniform(w, 72)
    ref = O.gradient(w, rho, 5e5, 2.0)["grad"].reshape(-1)
    g = run(dict(w, src_amp=amp), rho, 0)[1] / amp ** 2
    assert np.linalg.norm(g - ref) <= 1e-3 * np.linalg.norm(ref)
