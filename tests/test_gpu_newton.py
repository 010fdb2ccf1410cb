"""The Newton recompute of a mixed walker whose N has drifted far: 16 sites, 30
sweeps without a recompute, then one in the window before the first measurement.

With N0 the drifted N, A = N^-1 in FP64 and R = 1 - A N0, one term N0 + N0 R
leaves N0 R^2, the two taken from max |R| = 1e-4 on leave N0 R^3.  Bound of N
against the FP64 inverse, in units of the largest entries: the rounding of N to
FP32 (2^-24, twice for the sum), the products N0 R in 3xTF32 or FP32 (2^-20 of
|N0| |R|: 2^-22 per term and the truncated sums), the residual's digits (2^-40 of
the row and column maxima per term, summed like sqrt(n)), and N0 R^3."""
import numpy as np
import pytest

from oracle import ctaux
from tests.helpers import problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("method", ["auto", "newton_df"])
def test_recompute_of_a_far_drifted_N_leaves_the_third_power(method):
    import torch
    from paper_1901_01047_gb300 import walker
    nc, U, beta, n_tau, sweeps = 16, 6.0, 6.0, 2048, 40
    c, eps, kr, G0 = problem(nc, 1.0, -0.15, U, beta, 2.85, n_tau)
    prob = dict(nc=nc, site_sub=c.site_sub, U=U, beta=beta, K=1.0, G0=G0)
    ow = ctaux.OracleWalker(nc, c.site_sub, U, beta, 1.0, G0, warmup_sweeps=sweeps - 1, n_tau_meas=16, seed=3)
    ow.enable_log(1 << 22)
    ow.sweep(sweeps)
    log = ow.log()
    N = {}
    for measure in (False, True):
        gw = walker.Walkers([prob], precision="tf32", k_sub=16, warmup_sweeps=sweeps - 1, n_tau_meas=16, seed=3,
                            recompute_every=8, recompute_method=method, stream=torch.cuda.current_stream().cuda_stream)
        gw.set_forced_decisions(0, log)
        gw.sweep(sweeps - 3)
        gw.set_recompute(0, 0, measure)
        gw.sweep(3)
        st = gw.state(0)
        N[measure] = st["N"]
        gw.close()
    site, tau, s = st["site"], st["tau"], st["s"].astype(np.float64)
    n = site.size
    gamma = np.arccosh(1.0 + U * beta * nc / 2)
    x = tau[:, None] - tau[None, :]
    sg, x = np.where(x < 0, -1.0, 1.0), np.where(x < 0, x + beta, x) * (n_tau / beta)
    i = np.clip(x.astype(int), 0, n_tau - 1)
    row = -G0[0][c.site_sub[site[:, None], site[None, :]]]
    lo, hi = np.take_along_axis(row, i[..., None], 2)[..., 0], np.take_along_axis(row, i[..., None] + 1, 2)[..., 0]
    g = sg * (lo + (x - i) * (hi - lo))
    told = []
    for sp in range(2):
        e = np.exp((1 - 2 * sp) * gamma * s)
        A = np.diag(e) - g * (e - 1.0)[None, :]
        N0 = N[False][sp]
        R = np.eye(n) - A @ N0
        D, D2 = N0 @ R, N0 @ R @ R
        digits = 2.0 ** -40 * np.sqrt(n) * np.abs(A).max(1)[:, None] * np.abs(N0).max(0)[None, :]
        bound = 2.0 ** -23 * np.abs(N0).max() + 2.0 ** -20 * (np.abs(N0) @ np.abs(R)).max() \
            + (np.abs(N0) @ digits).max() + 2 * np.abs(D2 @ R).max()
        off = np.abs(N[True][sp] - np.linalg.inv(A)).max()
        print("order %d max|R| %.1e |R| %.1e: off %.1e, bound %.1e, one term leaves %.1e"
              % (n, np.abs(R).max(), np.linalg.norm(R, 2), off, bound, np.abs(D2).max()))
        assert 1e-4 <= np.abs(R).max() < 1 and np.abs(D2).max() <= 0.5 * np.abs(D).max()
        assert off <= bound
        told.append(np.abs(D2).max() / bound)
    assert max(told) > 2  # one term alone would not pass
