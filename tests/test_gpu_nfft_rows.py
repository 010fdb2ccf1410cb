"""The NFFT of the mixed path with 16 and with 32 rows of N per item (the latter for
grids of 24576 values on in lockstep batches of 8 walkers on): the chains of 7 and of
8 walkers are the same for the first 7, and so must M be.

Bound: an FP32 sum of a grid point has about 32 terms of an item, 6 roundings of
2^-24 of the sum of magnitudes, which is at most some 25 times the largest |M|."""
import numpy as np
import pytest

from tests.helpers import problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_omega", [383, 384, 400])
def test_rows_per_item_leave_M(n_omega):
    import torch
    from paper_1901_01047_gb300 import walker
    c, eps, kr, G0 = problem(16, 1.0, 0.0, 4.0, 3.0, 2.0, 512)
    prob = dict(nc=16, site_sub=c.site_sub, U=4.0, beta=3.0, K=1.0, G0=G0)
    got = []
    for W in (7, 8):
        gw = walker.Walkers([prob], n_walkers=W, precision="mixed", k_sub=32, warmup_sweeps=6, n_tau_meas=16, seed=9,
                            n_omega_meas=n_omega, recompute_at_measure=True, stream=torch.cuda.current_stream().cuda_stream)
        gw.sweep(8)
        got.append(gw.measure_M()[0][:7])
        assert len({st["proposals"] for st in gw.stats()[:7]}) > 1
        gw.close()
    for a, b in zip(*got):
        assert np.abs(a).max() > 0 and np.abs(a - b).max() <= 25 * 6 * 2.0 ** -24 * np.abs(a).max()
