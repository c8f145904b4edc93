"""The bound that rms.h states for one term of the plain form's read-out: one walker
of alpha 1 among saturated ones, so that S is its term, beside walkers of phases up
to P in the same 64.  Along an axis at b = b_s the dot product and its factor are
exact, and S's parts are within 2^-51.8 + 2^-55 P of those of e^{-i phi} (and the
half unit of their rounding to a double)."""
import numpy as np
import pytest

from test_gpu_readout_sizes import _readout

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P", [1.0, 4.0, 127.0, 2000.0, 3e4, 1e6])
def test_term_beside_larger_phases(P):
    rng = np.random.default_rng(int(P))
    W = 256
    worst = 0.0
    for _ in range(40):
        phase = np.zeros((W, 1, 3))
        phase[:, 0] = rng.uniform(-1.0, 1.0, size=(W, 3)) * P
        phase[::7, 0] = P
        phase[1::7, 0] = rng.uniform(-4.0, 4.0, size=(len(phase[1::7]), 3))
        A = np.full(W, np.inf)
        j = int(rng.integers(0, W))
        A[j] = 0.0
        S, asum = _readout(phase, A, np.ones(1), np.eye(3), np.ones(1))
        assert asum == 1.0
        phi = phase[j, 0].astype(np.longdouble)
        off = np.abs([S[0, :, 0].real - np.cos(phi), S[0, :, 0].imag + np.sin(phi)]).astype(float)
        worst = max(worst, off.max())
    assert worst <= 2.0 ** -51.8 + 2.0 ** -55 * P + 2.0 ** -54, np.log2(worst)
