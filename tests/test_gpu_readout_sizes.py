"""rms_readout_noalloc over its sizes and values: tiles of 64 walkers and their
remainders, few walkers (floating-point terms), one and many combinations
groups, several threads to a combination, phases outside the fixed-point range
in some tiles, saturated walkers, and b = 0.  Against numpy with phases in
extended precision: every term is within 2^-51 + 2^-53 |phi| (fixed point, and
the FP64 dot product and sincos), a signal within that plus the roundings of
its sums, 2^-52 at most."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _readout(phase, A, bs, dirs, b):
    import torch
    from paper_2012_06478_gb300 import _lib
    t = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (phase, A, bs, dirs, b)]
    W, S, _ = phase.shape
    n = S * dirs.shape[0] * b.size
    re, im = torch.full((2, n), np.nan, dtype=torch.float64, device="cuda").unbind(0)
    asum = torch.zeros(1, dtype=torch.float64, device="cuda")
    rc = _lib.lib.rms_readout_noalloc(t[0].data_ptr(), t[1].data_ptr(), W, S, t[2].data_ptr(), dirs.shape[0],
                                      t[3].data_ptr(), b.size, t[4].data_ptr(), re.data_ptr(), im.data_ptr(),
                                      asum.data_ptr(), C.c_void_p(torch.cuda.current_stream().cuda_stream))
    torch.cuda.synchronize()
    assert rc == _lib.RMS_OK, _lib.last_error()
    return (re.cpu().numpy() + 1j * im.cpu().numpy()).reshape(S, dirs.shape[0], b.size), float(asum.item())


def _exact(phase, A, bs, dirs, b):
    ld = np.longdouble
    al = np.exp(-A.astype(ld))
    S = np.zeros((phase.shape[1], dirs.shape[0], b.size), np.complex128)
    for s in range(phase.shape[1]):
        gp = phase[:, s].astype(ld) @ dirs.T.astype(ld)
        for i in range(b.size):
            phi = ld(np.sqrt(b[i] / bs[s])) * gp
            S[s, :, i] = ((al[:, None] * np.cos(phi)).sum(0) / al.sum()).astype(float) - 1j * (
                (al[:, None] * np.sin(phi)).sum(0) / al.sum()).astype(float)
    return S, float(al.sum())


@pytest.mark.parametrize("W,S,nd,nb", [(1, 1, 1, 1), (63, 1, 3, 2), (255, 2, 2, 3), (256, 1, 3, 2), (257, 1, 30, 11),
                                       (1000, 8, 5, 1), (4097, 1, 130, 1), (3001, 1, 64, 9), (20001, 2, 3, 4)])
def test_sizes(W, S, nd, nb):
    rng = np.random.default_rng([W, nd])
    phase = rng.normal(size=(W, S, 3)) * 0.5
    A = rng.uniform(0.0, 3.0, size=W)
    dirs = rng.normal(size=(nd, 3))
    dirs /= np.linalg.norm(dirs, axis=1, keepdims=True)
    bs = rng.uniform(0.7, 1.4, size=S)
    b = np.linspace(0.0, 8.0, nb) if nb > 1 else np.array([2.0])
    if W > 500:  # tiles with small, large and mixed phases, and saturated walkers
        phase[64:128] *= 1e-6
        phase[128:192] *= 1e5
        phase[200] *= 1e7
        A[300:420] = np.inf
    got, asum = _readout(phase, A, bs, dirs, b)
    want, asum_w = _exact(phase, A, bs, dirs, b)
    al = np.exp(-A)
    P = np.sqrt(b.max() / bs.min()) * np.abs(phase).sum(axis=2).max(axis=1)
    tol = float((al * (2.0 ** -51 + 2.0 ** -51 * P)).sum() / al.sum()) + 2.0 ** -51
    assert np.abs(got - want).max() <= tol, (np.abs(got - want).max(), tol)
    assert abs(asum - asum_w) <= 1e-14 * asum_w
    if nb > 1:
        assert np.all(got[:, :, 0] == 1.0)


def test_values_that_are_not_finite():
    rng = np.random.default_rng(9)
    phase = rng.normal(size=(1000, 1, 3))
    dirs, bs, b = np.eye(3), np.ones(1), np.array([0.0, 1.0])
    A = np.zeros(1000)
    phase[777, 0, 1] = np.nan
    got, _ = _readout(phase, A, bs, dirs, b)
    assert np.isnan(got[0, 1]).all()
    got, asum = _readout(np.zeros((1000, 1, 3)), np.full(1000, np.inf), bs, dirs, b)
    assert asum == 0.0 and np.isnan(got).all()


def test_under_capture():
    import torch
    from paper_2012_06478_gb300 import _lib
    rng = np.random.default_rng(4)
    arrays = rng.normal(size=(1000, 1, 3)), rng.uniform(size=1000), np.ones(1), np.eye(3), np.array([0.0, 2.0])
    want, _ = _readout(*arrays)  # the first call, before the capture
    t = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in arrays]
    re, im = torch.zeros((2, 6), dtype=torch.float64, device="cuda").unbind(0)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        rc = _lib.lib.rms_readout_noalloc(t[0].data_ptr(), t[1].data_ptr(), 1000, 1, t[2].data_ptr(), 3, t[3].data_ptr(),
                                          2, t[4].data_ptr(), re.data_ptr(), im.data_ptr(), None,
                                          C.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert rc == _lib.RMS_OK, _lib.last_error()
    graph.replay()
    torch.cuda.synchronize()
    np.testing.assert_array_equal(re.cpu().numpy() + 1j * im.cpu().numpy(), want.ravel())
