"""The plain form's four-lane kernel (runs of few walkers) against the
one-thread kernel (runs of many): a run above the line between them gives every
walker the bits that runs of its parts below it give, over shapes, relaxation,
unequal D and an open axis; and the parts' moments add up.  Both, which skip the
range checks of products and quotients where a run's numbers allow it, against
the verification kernel, which checks every one; and runs whose numbers do not
allow it (weights near the largest double, a resumed offset of -0 or below the
normal numbers) against it too."""
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


@pytest.mark.parametrize("W", [LINE + 5, 700])
@pytest.mark.parametrize("case", ["plain", "weights", "offsets"])
def test_unchecked_arithmetic(W, case):
    import paper_2012_06478_gb300 as rms
    rng = np.random.default_rng(11)
    n = 30
    G = rng.normal(size=(2, n)) * (rng.random((2, n)) < 0.7)
    if case == "weights":
        G *= 1e306
    wl = make_workload(rng.integers(0, 3, size=(5, 6, 7)), voxel_um=0.2, D=[2.0, 1.0, 1.5], kappa=0.7,
                       T2=[50.0, np.inf, 90.0], dt=2e-3, n_steps=n, G=G, n_walkers=W, seed=3)
    sub = rms.rms_create_substrate(wl.labels, wl.voxel_um, wl.D, T2=wl.T2, kappa=wl.kappa)
    seq = rms.rms_set_sequence(sub, wl.dt, wl.G, wl.dirs, wl.b, wl.rec_steps)
    state = None
    if case == "offsets":
        first = rms.rms_run(seq, W, wl.seed, rms.RMS_FP64, step_end=3)
        state = rms.rms_read_walkers(first)
        state.update(step=3, moments=rms.rms_read_signal(first)[1])
        first.close()
        state["o"][::7, 0] = -0.0
        state["o"][1::7, 1] = 1e-310
    got = []
    for flags in (0, rms.RMS_TRAJ_HASH):
        run = rms.rms_run(seq, W, wl.seed, rms.RMS_FP64, flags, resume=state)
        got.append(rms.rms_read_walkers(run))
        run.close()
    for k in ("i", "o", "c", "A", "phase"):
        np.testing.assert_array_equal(got[0][k], got[1][k], err_msg=k)
    seq.close()
    sub.close()
