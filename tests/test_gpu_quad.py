"""The plain form's four-lane kernel (runs of few walkers) against the
one-thread kernel (runs of many): a run above the line between them gives every
walker the bits that runs of its parts below it give, over shapes, relaxation,
unequal D and an open axis; and the parts' moments add up."""
import numpy as np
import pytest

from conftest import make_workload

pytestmark = pytest.mark.gpu

LINE = 2 * 5 * 152 * 32  # walkers


@pytest.mark.parametrize("shapes,relax,parts", [(1, False, (33,)), (1, True, (1, 127)), (2, True, ()),
                                                (3, False, (64,)), (6, True, (31,))])
def test_few_walkers_walk_as_many_do(shapes, relax, parts):
    import paper_2012_06478_gb300 as rms
    rng = np.random.default_rng(shapes)
    lab = rng.integers(0, 4, size=(9, 7, 11))
    if shapes == 1:
        lab = np.kron(rng.integers(0, 4, size=(3, 3, 3)), np.ones((4, 4, 4), int))
    n = 41
    wl = make_workload(lab, voxel_um=0.2, D=[2.0, 1.0, 1.5, 0.7] if relax else 2.0,
                       kappa=rng.uniform(0, 2, size=(4, 4)), T2=[50.0, 70.0, 90.0, 60.0] if relax else np.inf,
                       dt=2e-3, n_steps=n, G=rng.normal(size=(shapes, n)), periodic=(1, 0, 1),
                       rec_steps=np.array([1, 8, n]), n_walkers=LINE + 33, seed=7)
    sub = rms.rms_create_substrate(wl.labels, wl.voxel_um, wl.D, T2=wl.T2, kappa=wl.kappa, periodic=(1, 0, 1))
    seq = rms.rms_set_sequence(sub, wl.dt, wl.G, wl.dirs, wl.b, wl.rec_steps)
    run = rms.rms_run(seq, wl.n_walkers, wl.seed, rms.RMS_FP64)
    _, mom, _ = rms.rms_read_signal(run)
    full = rms.rms_read_walkers(run)
    run.close()
    cuts = [0, *np.cumsum(parts), LINE, LINE + 33]
    total = np.zeros_like(mom)
    for a, b in zip(cuts, cuts[1:]):
        part = rms.rms_run(seq, int(b - a), wl.seed, rms.RMS_FP64, walker_begin=int(a))
        total += rms.rms_read_signal(part)[1]
        got = rms.rms_read_walkers(part)
        part.close()
        for k in ("i", "o", "i0", "o0", "c", "A", "phase"):
            np.testing.assert_array_equal(got[k], full[k][a:b], err_msg=f"{k} {a} {b}")
    np.testing.assert_allclose(total, mom, rtol=0, atol=1e-12 * np.abs(mom).max())
    seq.close()
    sub.close()
