"""What an in-plane context holds of the adjoint's records."""
from paper_2203_01462_gb300 import inputs as I
from paper_2203_01462_gb300.binding import workspace_bytes


def test_adjoint_records_follow_the_steps_between_checkpoints():
    """The blocked adjoint keeps records of as many steps as are summed at a
    time: at most 32, and no more than there are between two checkpoints.  A
    run of 32 steps holds 28 more slots of forward and 28 of adjoint records
    than one of 4 (and 29 more steps of gap history and source samples)."""
    w = I.workload_2d_inplane(291, 291, dx=0.5e-9, nsteps=4, npml=15, design=(200, 200), gap=(20, 20), real="f32",
                              material=I.SILVER)
    slot = 4 * 2 * 200 * 201  # bytes, without row padding
    few, many, more = (workspace_bytes(dict(w, nsteps=n)) for n in (4, 32, 60))
    assert 56 * slot <= many - few <= 1.1 * 56 * slot
    assert 28 * slot <= more - many <= 1.1 * 28 * slot
