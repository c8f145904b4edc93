"""The FP32 read-out where its sums could go wrong: the sum of alpha over many
walkers when combinations alone fill the blocks; several groups of combinations over
tiles of ordinary, saturated and nearly saturated walkers; phases that are not
finite."""
import numpy as np
import pytest

from conftest import make_workload
from test_gpu_readout import fp32_readout_bound

pytestmark = pytest.mark.gpu


def _sequence(shapes, nd, nb, W):
    """A sequence whose third step has no gradient, and a state after its second."""
    import paper_2012_06478_gb300 as rms
    rng = np.random.default_rng([shapes, nd])
    dirs = rng.normal(size=(nd, 3))
    dirs /= np.linalg.norm(dirs, axis=1, keepdims=True)
    dt = 1e-3
    wl = make_workload(np.zeros((8, 8, 8), int), D=2.0, dt=dt, n_steps=3, G=[[1.0, -1.0, 0.0]] * shapes, dirs=dirs,
                       b=dt ** 3 * np.linspace(0.0, 6.0, nb), n_walkers=W, seed=3)
    sub = rms.rms_create_substrate(wl.labels, wl.voxel_um, wl.D)
    seq = rms.rms_set_sequence(sub, wl.dt, wl.G, wl.dirs, wl.b, wl.rec_steps)
    first = rms.rms_run(seq, W, wl.seed, rms.RMS_FP32, step_end=2)
    state = rms.rms_read_walkers(first)
    first.close()
    state.update(step=2)
    return sub, seq, wl, state


def _signal(seq, wl, state):
    import paper_2012_06478_gb300 as rms
    run = rms.rms_run(seq, wl.n_walkers, wl.seed, rms.RMS_FP32, resume=state)
    S, _, alpha = rms.rms_read_signal(run)
    run.close()
    return S, alpha


def test_sum_of_alpha():
    # a chunk adds the sums of its tiles one after another, each addition within half a
    # unit of the sum so far: over 16 384 walkers in 256 tiles that is 128 2^-53 of the
    # whole, and exp adds 2.  All walkers alike, so that the roundings add up.
    sub, seq, wl, state = _sequence(1, 512, 480, 1_000_000)
    for A in (0.375, 0.8125, 1.65625):
        state["A"][:] = A
        S, alpha = _signal(seq, wl, state)
        want = np.exp(np.longdouble(-A)) * wl.n_walkers
        assert abs(alpha - want) <= 130 * 2.0 ** -53 * want, float((alpha - want) / want) * 2.0 ** 53
        assert np.all(S[:, :, 0] == 1.0)
    seq.close()
    sub.close()


def test_groups_and_saturated_tiles():
    W = 70_003
    sub, seq, wl, state = _sequence(2, 256, 8, W)
    rng = np.random.default_rng(2)
    state["A"][:] = rng.uniform(0.0, 3.0, size=W)
    state["A"][6400:6500] = np.inf   # a whole tile and a half of saturated walkers
    state["A"][12800:12928] = 700.0  # tiles whose alphas are below 2^-900
    state["A"][20000] = -30.0        # and one far above the others
    state["phase"][:] = 0.5 * rng.normal(size=state["phase"].shape)
    S, alpha = _signal(seq, wl, state)
    import paper_2012_06478_gb300 as rms
    bs = rms.rms_sequence_bvalues(seq)
    al = np.exp(-state["A"])
    assert abs(alpha - al.sum()) <= 1e-12 * al.sum()
    assert np.all(S[:, :, 0] == 1.0)
    some = np.arange(0, 256, 5)
    for s in range(2):
        gp = state["phase"][:, s] @ wl.dirs[some].T
        for i in range(1, 8):
            q = np.sqrt(wl.b[i] / bs[s])
            want = (al[:, None] * np.exp(-1j * q * gp)).sum(0) / al.sum()
            P = q * (np.abs(state["phase"][:, s]) @ np.abs(wl.dirs[some]).T).max()
            assert np.abs(S[s, some, i] - want).max() <= fp32_readout_bound(P)
    seq.close()
    sub.close()


@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_phases_that_are_not_finite(value):
    sub, seq, wl, state = _sequence(2, 3, 4, 1000)
    state["phase"][777, 1, 1] = value
    S, alpha = _signal(seq, wl, state)
    assert alpha == 1000.0
    assert np.all(np.isfinite(S[0]))
    assert np.all(S[:, :, 0] == 1.0)
    assert np.all(np.isnan(S[1, :, 1:]))
    seq.close()
    sub.close()
