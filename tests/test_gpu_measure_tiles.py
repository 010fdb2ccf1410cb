"""G(tau) of one measurement against the estimator in numpy on the walker's own
N, at the edges of the product kernels: every site class (nc <= 8, 16, 36, 64
in FP32; a power of two or not, <= 16 or more in FP64), tau grids that end
inside a tile, commensurate (n_tau an even multiple) and not, orders above and
below the 256 vertices of an FP32 item.

    G(d, a) = g0(d, tau_a) + (1/Nc) sum_{r', i} g0(r' + d - r_i, tau_a - tau_i) b_i(r'),
    b_i(r') = (e^{V_i} - 1) sum_j N_ij g0(r_j - r', tau_j)

Bounds, in units of S(d, a) = the same sums of absolute values: FP64 n 2^-52 for
the sums and 4 n_tau 2^-53 for the interpolation weights (grid times up to
n_tau, one rounding each); FP32 sums of 32 terms (b, then G), the rounding of
the table, of b and of the interpolation: 80 2^-24."""
import numpy as np
import pytest

from oracle import g0 as og0
from paper_1901_01047_gb300 import inputs

pytestmark = pytest.mark.gpu


def _interp(table, d, t, beta):
    n_tau = table.shape[-1] - 1
    neg = t < 0
    x = np.where(neg, t + beta, t) * (n_tau / beta)
    k = np.clip(x.astype(int), 0, n_tau - 1)
    lo, hi = table[d, k], table[d, k + 1]
    return np.where(neg, -1.0, 1.0) * (lo + (x - k) * (hi - lo))


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("side,beta,ntm,n_tau", [(1, 3.0, 16, 512), (2, 3.0, 100, 1000), (2, 3.0, 130, 512),
                                                 (3, 3.0, 128, 512), (4, 3.0, 33, 1056), (4, 11.0, 40, 1040),
                                                 (5, 1.5, 96, 576), (6, 1.5, 129, 1032), (7, 1.5, 64, 512)])
def test_measured_G_equals_the_estimator_on_the_same_N(side, beta, ntm, n_tau, precision):
    import torch
    from paper_1901_01047_gb300 import walker
    c = inputs.make_cluster(((side, 0), (0, side)))
    nc, U = side * side, 4.0
    eps = inputs.square_dispersion(c.kpts, 1.0 if nc > 1 else 0.0, 0.0)
    G0 = og0.g0_table(eps, inputs.k_dot_r(c), U / 2, U, beta, n_tau)
    prob = dict(nc=nc, site_sub=c.site_sub, U=U, beta=beta, K=1.0, G0=G0)
    gw = walker.Walkers([prob], n_walkers=1, precision=precision, k_sub=16, warmup_sweeps=12, n_tau_meas=ntm, seed=side,
                        init_config_size=4, recompute_at_measure=True, stream=torch.cuda.current_stream().cuda_stream)
    gw.sweep(13)
    G, sign, count = gw.measure_G()
    st = gw.state(0)
    gw.close()
    assert count[0] == 1
    site, tau, s = st["site"], st["tau"], st["s"].astype(np.float64)
    gamma = np.arccosh(1.0 + U * beta * nc / 2)
    n, sub = site.size, c.site_sub
    add = np.empty((nc, nc), int)  # add[y, d] = x with sub[x, y] = d
    for x in range(nc):
        add[np.arange(nc), sub[x]] = x
    ta = (np.arange(ntm) + 0.5) * beta / ntm
    for sp in range(2):
        g0 = -G0[sp]
        em1 = np.exp((1 - 2 * sp) * gamma * s) - 1.0
        gr = _interp(g0, sub[site[None, :], np.arange(nc)[:, None]], np.broadcast_to(tau, (nc, n)), beta)  # [r', j]
        b, B = em1 * (gr @ st["N"][sp].T), np.abs(em1) * (np.abs(gr) @ np.abs(st["N"][sp]).T)
        gx = np.stack([_interp(g0, sub[x, site][None, :], ta[:, None] - tau[None, :], beta) for x in range(nc)])
        for d in range(nc):
            corr = sum(gx[add[r, d]] @ b[r] for r in range(nc)) / nc
            S = sum(np.abs(gx[add[r, d]]) @ B[r] for r in range(nc)) / nc
            ref = _interp(g0, np.full(ntm, d), ta, beta)
            tol = (80 * 2.0 ** -24 if precision == "mixed" else (n + 4 * n_tau) * 2.0 ** -52) * (S + np.abs(ref))
            assert np.all(np.abs(sign[0] * -G[0][sp, d] - (ref + corr)) <= tol)
