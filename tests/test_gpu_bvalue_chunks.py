"""b_s at the edges of the chunks of 1024 steps and of the windows of 32 in which the
GPU takes the chains of additions: the oracle's sums bit for bit."""
import numpy as np
import pytest

from test_gpu_bvalue import _bvalues

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [31, 32, 33, 1023, 1024, 1025, 2079, 3073])
def test_chunk_edges(oracle_lib, N):
    import paper_2012_06478_gb300 as rms
    rng = np.random.default_rng(N)
    # random, of few bits (ties), large and small in turn, and back to zero again and again
    G = np.stack([rng.normal(size=N), np.round(rng.normal(size=N) * 8) / 8, rng.normal(size=N) * 10.0 ** rng.integers(-9, 9, N),
                  np.where(np.arange(N) % 2, -1.0, 1.0)])
    got = _bvalues(rms, G, 2e-4)
    for s in range(G.shape[0]):
        assert got[s] == oracle_lib.bvalue(np.ascontiguousarray(G[s]), 2e-4), s
