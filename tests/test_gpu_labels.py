"""The pass over a new substrate's labels takes eight voxels at a time: row lengths
around and below eight, voxel counts that are no multiple of eight, rows that end
inside a group.  Walkers against the oracle's through the face bits it leaves, and a
label out of range refused wherever it stands."""
import numpy as np
import pytest

from conftest import make_workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz", [(8, 3, 5), (9, 4, 3), (15, 2, 2), (24, 1, 7), (3, 3, 3), (1, 1, 9), (7, 1, 1),
                                      (401, 2, 3), (2, 40, 5), (16, 8, 8)])
@pytest.mark.parametrize("periodic", [(1, 1, 1), (0, 1, 0)])
def test_walkers_of_every_row_length(oracle_lib, nx, ny, nz, periodic):
    import paper_2012_06478_gb300 as rms
    rng = np.random.default_rng([nx, ny, nz])
    n = 90
    wl = make_workload(rng.integers(0, 3, size=(nz, ny, nx)) * (rng.random((nz, ny, nx)) < 0.6), periodic=periodic,
                       D=2.0, kappa=0.6, dt=2e-3, n_steps=n, G=rng.normal(size=(1, n)), n_walkers=400, seed=nx)
    o = oracle_lib.run(wl)
    g = rms.simulate(wl, rms.RMS_FP64, walkers=True)
    for k in ("i", "o", "c", "phase"):
        np.testing.assert_array_equal(g[k], o[k].astype(g[k].dtype), err_msg=k)


@pytest.mark.parametrize("shape", [(3, 3, 3), (4, 4, 4), (1, 1, 1), (2, 5, 13)])
def test_label_out_of_range(shape):
    import paper_2012_06478_gb300 as rms
    lab = np.zeros(shape, np.uint16)
    for at in sorted({0, lab.size // 2, max(lab.size - 2, 0), lab.size - 1}):
        for value, ok in ((2, False), (1, True), (65535, False)):
            lab.flat[at] = value
            if ok:
                rms.rms_create_substrate(lab, 0.2, np.ones(2)).close()
            else:
                with pytest.raises(rms.RmsError):
                    rms.rms_create_substrate(lab, 0.2, np.ones(2))
        lab.flat[at] = 0
