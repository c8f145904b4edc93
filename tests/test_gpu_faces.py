"""The walk through face bits (a byte per voxel: which faces lead into the same
label inside the volume; labels are looked up only at the other faces) at the
sizes where it can go wrong: axes of one, two and three voxels, odd edges,
closed and periodic, and a single label.  Both forms' production kernels against the oracle's walkers: the
plain form bit for bit, the FP32 form voxel by voxel (the runs are short
enough that its walkers stay with their twins; at most 1 in 1000 may leave)."""
import numpy as np
import pytest

from conftest import make_workload

pytestmark = pytest.mark.gpu

SHAPES = [  # nx, ny, nz, periodic, labels
    (1, 1, 1, (1, 1, 1), 1), (1, 2, 3, (1, 0, 1), 2), (2, 1, 17, (0, 1, 1), 3), (33, 1, 2, (1, 1, 0), 4),
    (31, 32, 33, (0, 0, 0), 5), (5, 64, 3, (1, 1, 1), 2), (16, 16, 16, (1, 1, 1), 1), (7, 9, 11, (1, 0, 1), 9)]


def _labels(nx, ny, nz, L, seed):
    rng = np.random.default_rng(seed)
    blocks = rng.integers(0, L, size=((nz + 2) // 3, (ny + 2) // 3, (nx + 2) // 3))
    lab = np.repeat(np.repeat(np.repeat(blocks, 3, 0), 3, 1), 3, 2)[:nz, :ny, :nx].copy()
    lab.flat[0] = L - 1
    return lab


@pytest.mark.parametrize("nx,ny,nz,periodic,L", SHAPES)
@pytest.mark.parametrize("interaction", [0, 1, 2])
def test_walkers_through_face_bits(oracle_lib, nx, ny, nz, periodic, L, interaction):
    import paper_2012_06478_gb300 as rms
    rng = np.random.default_rng(nx + 100 * ny + interaction)
    n = 120
    G = np.zeros((1, n))
    G[0, :30], G[0, 60:90] = 1.0, -1.0
    wl = make_workload(_labels(nx, ny, nz, L, nx + ny + nz), periodic=periodic, D=rng.uniform(0.8, 2.0, L),
                       kappa=rng.uniform(0.0, 1.0, (L, L)), T2=rng.uniform(20, 60, L), dt=2e-3, n_steps=n, G=G,
                       n_walkers=300, seed=3 + nx, interaction=interaction, rec_steps=np.array([50, n]))
    o = oracle_lib.run(wl)
    g = rms.simulate(wl, rms.RMS_FP64, walkers=True)
    for k in ("i", "o", "c", "A", "phase"):
        assert np.array_equal(g[k], o[k].astype(g[k].dtype)), k
    f = rms.simulate(wl, rms.RMS_FP32, walkers=True)
    assert np.any(f["i"] != o["i"], axis=1).sum() <= 0.001 * 300 + 1
    lab = wl.labels[tuple(np.mod(f["i"], [nx, ny, nz])[:, a] for a in (2, 1, 0))]
    assert np.array_equal(lab, f["c"])
