"""The plain form's read-out of many walkers and very many combinations, whose
blocks are filled by combinations alone: a chunk's sums stay as near to their
values as sums over 4096 walkers bring a signal.

1e6 walkers of 64 different phases, 131 072 combinations, against extended
precision.  A chunk of n walkers adds n / 64 sums of tiles one after another: with
half a unit's rounding each, growing sums and independent chunks, a signal of
modulus 1 is off by 0.26 n / (8 sqrt(W)) units of 2^-53 in the mean square, 1.1 of
them for chunks of 8 x 4096 walkers, the longest; the dot product and its factor add 1 each at
phases of a radian.  2 units are allowed."""
import numpy as np
import pytest

from conftest import make_workload
from test_gpu_readout_sizes import _exact, _readout

pytestmark = pytest.mark.gpu


def test_sums_over_many_walkers():
    import paper_2012_06478_gb300 as rms
    rng = np.random.default_rng(8)
    W, nd, nb = 1_000_000, 512, 256
    dirs = rng.normal(size=(nd, 3))
    dirs /= np.linalg.norm(dirs, axis=1, keepdims=True)
    dt = 1e-3
    b = dt * dt * dt * np.linspace(0.05, 6.0, nb)
    wl = make_workload(np.zeros((8, 8, 8), int), D=2.0, dt=dt, n_steps=3, G=[[1.0, -1.0, 0.0]], dirs=dirs, b=b,
                       n_walkers=W, seed=3)
    sub = rms.rms_create_substrate(wl.labels, wl.voxel_um, wl.D)
    seq = rms.rms_set_sequence(sub, wl.dt, wl.G, wl.dirs, wl.b, wl.rec_steps)
    bs = rms.rms_sequence_bvalues(seq)[0]
    first = rms.rms_run(seq, W, wl.seed, rms.RMS_FP64, step_end=2)
    state = rms.rms_read_walkers(first)
    first.close()
    kinds = 0.5 * rng.normal(size=(64, 3))
    which = rng.integers(0, 64, size=W)
    state.update(step=2, phase=kinds[which][:, None, :])
    run = rms.rms_run(seq, W, wl.seed, rms.RMS_FP64, resume=state)  # its one step has no gradient
    S, _, alpha = rms.rms_read_signal(run)
    run.close()
    seq.close()
    sub.close()
    assert alpha == W
    ld = np.longdouble
    share = np.bincount(which, minlength=64).astype(ld) / W
    gp = kinds.astype(ld) @ dirs.T.astype(ld)
    some = np.arange(0, nb, 16)
    phi = np.sqrt(b / bs)[some].astype(ld)[None, None, :] * gp[:, :, None]
    re, im = (share[:, None, None] * np.cos(phi)).sum(0), -(share[:, None, None] * np.sin(phi)).sum(0)
    off = np.sqrt(float(((S[0][:, some].real - re) ** 2 + (S[0][:, some].imag - im) ** 2).mean()))
    assert off <= 2 * 2.0 ** -53, off * 2.0 ** 53


@pytest.mark.parametrize("W,S,nd,nb", [(256, 1, 3, 2), (257, 1, 30, 11), (1000, 8, 5, 1), (3001, 1, 64, 9),
                                       (4097, 1, 130, 1), (20001, 2, 3, 4), (9999, 3, 70, 5)])
def test_groups_and_remainders_of_ordinary_walkers(W, S, nd, nb):
    """Several groups of combinations, part tiles and part chunks, with phases of a few
    radians alone: within a term's bound, the dot product's and three roundings."""
    rng = np.random.default_rng([W, nd])
    phase = rng.normal(size=(W, S, 3)) * 0.5
    A = rng.uniform(0.0, 3.0, size=W)
    dirs = rng.normal(size=(nd, 3))
    dirs /= np.linalg.norm(dirs, axis=1, keepdims=True)
    bs = rng.uniform(0.7, 1.4, size=S)
    b = np.linspace(0.5, 8.0, nb)
    got, asum = _readout(phase, A, bs, dirs, b)
    want, asum_w = _exact(phase, A, bs, dirs, b)
    P = np.sqrt(b.max() / bs.min()) * (np.abs(phase) @ np.abs(dirs).T).max()
    # the terms' bound is relative to alphas of 1 at most, the signal to their mean
    tol = (2.0 ** -51.8 + 2.0 ** -55 * P) / np.exp(-A).mean() + 5 * 2.0 ** -53 * P + 3 * 2.0 ** -53
    assert max(np.abs((got - want).real).max(), np.abs((got - want).imag).max()) <= tol
    assert abs(asum - asum_w) <= 1e-14 * asum_w


@pytest.mark.parametrize("W,S,nd,nb", [(1, 1, 1, 1), (1, 1, 512, 1), (2, 6, 64, 11), (10, 1, 400, 25), (64, 1, 3, 2),
                                       (65, 2, 90, 30), (100, 1, 30, 11), (200, 8, 16, 4), (255, 1, 130, 3)])
def test_few_walkers(W, S, nd, nb):
    """Terms in FP64, blocks of few combinations: sums of at most 64 terms a thread, 64
    threads and 4 chunks round 132 times at most, by half a unit of a sum that is
    the alphas' at most."""
    rng = np.random.default_rng([W, nd, nb])
    phase = rng.normal(size=(W, S, 3)) * 0.5
    A = rng.uniform(0.0, 3.0, size=W)
    dirs = rng.normal(size=(nd, 3))
    dirs /= np.linalg.norm(dirs, axis=1, keepdims=True)
    bs = rng.uniform(0.7, 1.4, size=S)
    b = np.linspace(0.0, 8.0, nb) if nb > 1 else np.array([2.0])
    got, asum = _readout(phase, A, bs, dirs, b)
    want, asum_w = _exact(phase, A, bs, dirs, b)
    P = np.sqrt(b.max() / bs.min()) * (np.abs(phase) @ np.abs(dirs).T).max()
    tol = (132 + 4 + 6 * P) * 2.0 ** -53
    assert max(np.abs((got - want).real).max(), np.abs((got - want).imag).max()) <= tol
    assert abs(asum - asum_w) <= 136 * 2.0 ** -53 * asum_w
    if nb > 1:
        assert np.all(got[:, :, 0] == 1.0)
