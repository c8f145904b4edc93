"""Labels of next to no diffusion (step lengths below the smallest normal float):
a walker on a voxel's face still takes the faces it meets at once, in the FP32 form
as in the plain one.  Walkers put on faces and corners, 100 steps of 1e-40 voxels;
the forms round a direction differently, so that one walker in 100 may leave its
twin."""
import numpy as np
import pytest

from conftest import make_workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("step", [1e-40, 1e-25])
def test_faces_met_at_once(step):
    import paper_2012_06478_gb300 as rms
    voxel, dt, W = 0.2, 2e-3, 256
    wl = make_workload(np.zeros((5, 4, 6), int), voxel_um=voxel, D=(step * voxel) ** 2 / (6.0 * dt), dt=dt, n_steps=100,
                       n_walkers=W, seed=3)
    sub = rms.rms_create_substrate(wl.labels, wl.voxel_um, wl.D)
    seq = rms.rms_set_sequence(sub, wl.dt, wl.G, wl.dirs, wl.b, wl.rec_steps)
    first = rms.rms_run(seq, W, wl.seed, rms.RMS_FP64, step_end=1)
    state = rms.rms_read_walkers(first)
    first.close()
    state.update(step=1)
    state["o"][:] = np.random.default_rng(1).integers(0, 2, size=(W, 3))
    got = []
    for precision in (rms.RMS_FP64, rms.RMS_FP32):
        run = rms.rms_run(seq, W, wl.seed, precision, resume=state)
        got.append(rms.rms_read_walkers(run)["i"])
        run.close()
    # an axis hops between the two sides of its face, to the side of the last step's
    # direction: 7 in 8 walkers are not where they started, with a deviation of 0.02
    assert np.any(got[0] != state["i"], axis=1).mean() > 0.8
    assert np.any(got[0] != got[1], axis=1).sum() <= W // 100
    seq.close()
    sub.close()
