"""The products of the default recompute, entry by entry: N right after it against
N0 + N0 R + N0 R^2 in FP64, N0 the drifted N, R = 1 - A N0 (16 sites, drifted by
TF32 products so that the terms are large).

Bound of an entry: the rounding of N to FP32 (2^-24, twice for the sum), 2^-21 of
(|N0| |R|) for the product (chunks of 32 terms summed in FP32, about eight
roundings of 2^-24 that count; the FP32 kernel of "newton_df" with its chain over
all n reaches 1.1 times this bound), and the residual's digits (2^-40 of the row
and column maxima per term, like sqrt(n))."""
import numpy as np
import pytest

from oracle import ctaux
from tests.helpers import problem

pytestmark = pytest.mark.gpu


def test_terms_of_the_recompute_keep_fp32():
    import torch
    from paper_1901_01047_gb300 import walker
    nc, U, beta, n_tau, sweeps = 16, 6.0, 10.0, 2048, 50
    c, eps, kr, G0 = problem(nc, 1.0, -0.15, U, beta, 2.85, n_tau)
    prob = dict(nc=nc, site_sub=c.site_sub, U=U, beta=beta, K=1.0, G0=G0)
    ow = ctaux.OracleWalker(nc, c.site_sub, U, beta, 1.0, G0, warmup_sweeps=sweeps - 1, n_tau_meas=16, seed=4)
    ow.enable_log(1 << 22)
    ow.sweep(sweeps)
    log = ow.log()
    N = {}
    for measure in (False, True):
        gw = walker.Walkers([prob], precision="tf32", k_sub=16, warmup_sweeps=sweeps - 1, n_tau_meas=16, seed=4,
                            recompute_every=4, stream=torch.cuda.current_stream().cuda_stream)
        gw.set_forced_decisions(0, log)
        gw.sweep(sweeps - 1)
        gw.set_recompute(0, 0, measure)
        gw.sweep(1)
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
    for sp in range(2):
        e = np.exp((1 - 2 * sp) * gamma * s)
        A = np.diag(e) - g * (e - 1.0)[None, :]
        N0 = N[False][sp]
        R = np.eye(n) - A @ N0
        D, D2 = N0 @ R, N0 @ R @ R
        r = np.abs(R).max()
        assert 1e-4 <= r < 1
        ref = N0 + D + (D2 if np.abs(D2).max() <= 0.5 * np.abs(D).max() else 0.0)
        digits = 2.0 ** -40 * np.sqrt(n) * np.abs(A).max(1)[:, None] * np.abs(N0).max(0)[None, :]
        prod = np.abs(N0) @ np.abs(R)
        off = np.abs(N[True][sp] - ref)
        bound = 2.0 ** -23 * np.abs(ref) + 2.0 ** -21 * prod + np.abs(N0) @ digits
        print("order %d max|R| %.1e: off / bound %.2f" % (n, r, (off / bound).max()))
        assert np.all(off <= bound)
