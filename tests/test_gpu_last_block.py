"""Runs whose last block is not full: the threads beyond the last walker walk a
copy of it, which has to be read before the walker's own thread, in another warp,
writes the slice's end over it.  Slices of one step, in which hardly anything else
keeps the warps together: no invariant check fires, and every walker's bits and the
run's status are those of the run in one launch."""
import numpy as np
import pytest

from conftest import make_workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("walkers", [1, 31, 33, 96, 129, 225])
@pytest.mark.parametrize("interaction", [0, 1, 2])
def test_slices_of_one_step(walkers, interaction):
    import paper_2012_06478_gb300 as rms
    rng = np.random.default_rng(5)
    n = 150
    wl = make_workload(rng.integers(0, 3, size=(6, 5, 7)), voxel_um=0.2, D=[2.0, 1.0, 1.5], kappa=0.8,
                       T2=[50.0, np.inf, 90.0], dt=2e-3, n_steps=n, G=rng.normal(size=(1, n)), n_walkers=walkers,
                       seed=11, interaction=interaction, rec_steps=[])
    sub = rms.rms_create_substrate(wl.labels, wl.voxel_um, wl.D, T2=wl.T2, kappa=wl.kappa)
    seq = rms.rms_set_sequence(sub, wl.dt, wl.G, wl.dirs, wl.b, wl.rec_steps)
    for precision in (rms.RMS_FP64, rms.RMS_FP32):
        for flags in (0, rms.RMS_CHECKED):
            got = []
            for slice_steps in (n, 1):
                run = rms.rms_run(seq, walkers, wl.seed, precision, flags, interaction=interaction,
                                  steps_per_launch=slice_steps)
                got.append(rms.rms_read_walkers(run))  # raises where a check fired
                got[-1]["status"] = run.status  # whether a walker met the limit of draws
                run.close()
            for k in ("i", "o", "c", "A", "phase", "status"):
                np.testing.assert_array_equal(got[0][k], got[1][k], err_msg=f"{k} {precision} {flags}")
    seq.close()
    sub.close()
