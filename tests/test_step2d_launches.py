"""The 2D E_z step kernel of one launch per step (k_step2d, k_step2d_pair),
asked for with fdtd_set_steps_per_launch(1): grids left to the library's choice
run temporally blocked launches instead.  Its vector path against the oracle on
the cases of test_parity_2d_vector (same geometry, same tolerances), and the L2
access-policy windows, which only these launches take."""
import ctypes

import numpy as np
import pytest

import test_parity_2d_vector as V
from paper_2203_01462_gb300 import binding, inputs as I

pytestmark = pytest.mark.gpu


class OneStep(binding.Solver):
    def __init__(self, *a, **kw):
        super().__init__(*a, **kw)
        self.set_steps_per_launch(1)


@pytest.fixture
def one_step(monkeypatch):
    monkeypatch.setattr(binding, "Solver", OneStep)


@pytest.mark.parametrize("snap,material", [(0, "gold"), (64, "silver")])
def test_fp64_vector_path_matches_oracle(one_step, snap, material):
    V.test_fp64_vector_path_matches_oracle(snap, material)


@pytest.mark.parametrize("snap", [0, 64])
def test_fp32_vector_path_matches_oracle(one_step, snap):
    V.test_fp32_vector_path_matches_oracle(snap)


def test_fp32_vector_path_bowtie_silver_unfiltered(one_step):
    V.test_fp32_vector_path_bowtie_silver_unfiltered()


def test_fp64_vector_path_each_sensitivity_term(one_step):
    V.test_fp64_vector_path_each_sensitivity_term()


def test_one_launch_per_step(one_step):
    w = V.wide_case("f32", nsteps=40)
    s = V.solver(w)
    s.set_graphs(0)
    s.set_design(I.rho_uniform(w, 1))
    s.set_damping(0.0, 1.0)
    s.set_stability_guard(0)
    n0 = s.info().launches
    s.forward()
    assert s.info().launches - n0 >= 40


# ------------------------------------------------ L2 windows

_PERSISTING_L2 = 6  # cudaLimitPersistingL2CacheSize


def set_aside():
    import torch
    v = ctypes.c_size_t(0)
    rt = ctypes.CDLL("libcudart.so." + torch.version.cuda.split(".")[0])
    assert rt.cudaDeviceGetLimit(ctypes.byref(v), _PERSISTING_L2) == 0
    return v.value


@pytest.mark.parametrize("real,snap", [("f32", 0), ("f64", 8)])
@pytest.mark.parametrize("first", ["steps", "residency"])
def test_windows_change_no_result(real, snap, first):
    """Residency asked for before or after the steps per launch: set aside
    while launches take windows, given back while they are blocked."""
    w = V.wide_case(real, nsteps=260, snapshot_every=snap)
    plain, held = OneStep(w), binding.Solver(w)
    try:
        if first == "steps":
            held.set_steps_per_launch(1)
            held.set_l2_residency(0.3)
        else:
            held.set_l2_residency(0.3)
            assert set_aside() == 0  # blocked launches take no window
            held.set_steps_per_launch(1)
        assert set_aside() > 0
        for seed in (4, 5):
            rho = I.rho_uniform(w, seed)
            Wp, gp = plain.evaluate(rho, 2e5, 2.0)
            Wh, gh = held.evaluate(rho, 2e5, 2.0)
            plain.sync()
            held.sync()
            assert float(Wp.item()) > 0 and float(Wp.item()) == float(Wh.item())
            assert np.array_equal(gp.cpu().numpy(), gh.cpu().numpy())
        held.set_steps_per_launch(4)
        assert set_aside() == 0
        held.set_steps_per_launch(1)
        assert set_aside() > 0
    finally:
        held.set_l2_residency(0.0)
    assert set_aside() == 0
