"""The Gauss-Jordan inverse's panels of 4 columns and of single columns (which a
walker's recompute takes from capacities of about 9000 and 40000 on, whatever its
order), the line between clusters of 16 and of 8 blocks (3 and 4 walkers), and a
matrix without an inverse on both paths of dca_fresh_N.

Bound of N: |A N - 1| <= 4 n eps |A| |N| (norms: largest row sum)."""
import numpy as np
import pytest

from tests.helpers import problem

pytestmark = pytest.mark.gpu


def _matrix(G0, sub, site, tau, s, beta, n_tau, gamma, sp):
    x = tau[:, None] - tau[None, :]
    sg, x = np.where(x < 0, -1.0, 1.0), np.where(x < 0, x + beta, x) * (n_tau / beta)
    i = np.clip(x.astype(int), 0, n_tau - 1)
    row = -G0[0][sub[site[:, None], site[None, :]]]
    lo, hi = np.take_along_axis(row, i[..., None], 2)[..., 0], np.take_along_axis(row, i[..., None] + 1, 2)[..., 0]
    e = np.exp((1 - 2 * sp) * gamma * s)
    return np.diag(e) - sg * (lo + (x - i) * (hi - lo)) * (e - 1.0)[None, :]


@pytest.mark.parametrize("capacity,walkers", [(512, 3), (512, 4), (10240, 1), (41088, 1)])
def test_recompute_with_narrow_panels_and_at_the_cluster_line(capacity, walkers):
    import torch
    from paper_1901_01047_gb300 import walker
    nc, U, beta, n_tau = 4, 4.0, 8.0, 1024
    c, eps, kr, G0 = problem(nc, 1.0, 0.0, U, beta, 1.0, n_tau)
    prob = dict(nc=nc, site_sub=c.site_sub, U=U, beta=beta, K=1.0, G0=G0)
    gw = walker.Walkers([prob], n_walkers=walkers, k_sub=16, warmup_sweeps=4, n_tau_meas=8, seed=5, capacity=capacity,
                        recompute_every=2, recompute_at_measure=True, stream=torch.cuda.current_stream().cuda_stream)
    orders = set()
    for _ in range(6):
        gw.sweep(1 if orders else 5)
        for wi in range(walkers):
            st = gw.state(wi)
            site, tau, s = st["site"], st["tau"], st["s"].astype(np.float64)
            n = site.size
            orders.add(n)
            for sp in range(2):
                A = _matrix(G0, c.site_sub, site, tau, s, beta, n_tau, np.arccosh(1.0 + U * beta * nc / 2), sp)
                bound = 4 * n * 2.0 ** -52 * np.abs(A).sum(1).max() * np.abs(st["N"][sp]).sum(1).max()
                assert np.abs(A @ st["N"][sp] - np.eye(n)).max() <= bound
    assert max(orders) > 16  # more than a panel and more rows than blocks
    gw.close()


@pytest.mark.parametrize("n", [40, 330])
def test_a_matrix_without_an_inverse_is_refused(n):
    from paper_1901_01047_gb300 import walker
    nc, U, beta, n_tau = 4, 4.0, 8.0, 64
    c, eps, kr, G0 = problem(nc, 1.0, 0.0, U, beta, 1.0, n_tau)
    rng = np.random.default_rng(n)
    conf = (rng.integers(0, nc, n).astype(np.int32), rng.random(n) * beta,
            np.where(rng.random(n) < 0.5, 1, -1).astype(np.int32))
    good = dict(nc=nc, site_sub=c.site_sub, U=U, beta=beta, K=1.0, G0=G0)
    before = walker.fresh_N(good, *conf)
    with pytest.raises(walker.WalkerError) as e:  # finite entries whose products overflow: no pivot is left
        walker.fresh_N(dict(good, G0=np.full_like(G0, 1e308)), *conf)
    assert e.value.code == -5
    after = walker.fresh_N(good, *conf)
    assert all(np.array_equal(a, b) for a, b in zip(before, after))
