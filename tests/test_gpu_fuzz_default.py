"""The random configurations of test_gpu_fuzz through the kernels that a run without
verification flags takes: unchecked products and quotients, four lanes to a walker
up to 48 640 walkers and one thread above, relaxation decided at the launch.  Odd
slices, walker ids past 2^32, runs cut and resumed among them.  The plain FP64 form
equals the CPU oracle bit for bit, moments and signal to 1e-12."""
import os

import numpy as np
import pytest

from test_gpu_fuzz import ERR_LEAPS, random_case
from test_gpu_parity import assert_moments_close, assert_signal_close

pytestmark = pytest.mark.gpu
NT = os.cpu_count() or 1
KEYS = ("i", "o", "i0", "o0", "c", "A", "phase")


@pytest.mark.parametrize("seed,many", [(s, False) for s in range(100, 132)] + [(s, True) for s in range(200, 208)])
def test_random_configuration(oracle_lib, seed, many):
    import paper_2012_06478_gb300 as rms
    wl, ex = random_case(seed)
    if seed % 4:  # three in four: elastic collision without absorbing membranes
        wl = wl.with_(interaction=0, rho=None)
    if many:
        wl = wl.with_(n_walkers=48_640 + 77)
    kw = dict(walkers=True, walker_begin=ex["walker_begin"], steps_per_launch=ex["spl"])
    if ex["cut"]:
        part = rms.simulate(wl, rms.RMS_FP64, step_end=ex["cut"], **kw)
        state = {k: part[k] for k in KEYS}
        state.update(step=ex["cut"], moments=part["moments"])
        g = rms.simulate(wl, rms.RMS_FP64, resume=state, **kw)
    else:
        g = rms.simulate(wl, rms.RMS_FP64, **kw)
    o = oracle_lib.run(wl, ex["walker_begin"], ex["walker_begin"] + wl.n_walkers, n_threads=NT)
    assert o["err"] & ~ERR_LEAPS == 0, o["err"]
    for k in KEYS:
        np.testing.assert_array_equal(g[k], o[k].astype(g[k].dtype), err_msg=k)
    if wl.rec_steps.size:
        assert_moments_close(g["moments"], o["moments"])
    S_o, asum_o = oracle_lib.readout(o, wl)
    if asum_o > 0:
        assert_signal_close(g["S"], S_o)
    assert abs(g["alpha_sum"] - asum_o) <= 1e-12 * max(asum_o, 1e-300)
