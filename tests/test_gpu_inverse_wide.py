"""The inverse spread over the whole device (orders from 320 on) at the edges of
its panels of 16 columns and its update items of 8 rows and 64 columns:
|A N - 1| <= 4 n eps |A| |N| (norms: largest row sum), and the sign of det A."""
import numpy as np
import pytest

from tests.helpers import problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [319, 320, 321, 335, 336, 384, 449])
def test_inverse_spread_over_the_device(n):
    from paper_1901_01047_gb300 import walker
    nc, U, beta, n_tau = 16, 4.0, 6.0, 1024
    c, eps, kr, G0 = problem(nc, 1.0, 0.0, U, beta, 1.0, n_tau)
    prob = dict(nc=nc, site_sub=c.site_sub, U=U, beta=beta, K=1.0, G0=G0)
    rng = np.random.default_rng(n)
    site, tau = rng.integers(0, nc, n).astype(np.int32), rng.random(n) * beta
    s = np.where(rng.random(n) < 0.5, 1, -1).astype(np.int32)
    gamma = np.arccosh(1.0 + U * beta * nc / 2)
    x = tau[:, None] - tau[None, :]
    sg, x = np.where(x < 0, -1.0, 1.0), np.where(x < 0, x + beta, x) * (n_tau / beta)
    i = np.clip(x.astype(int), 0, n_tau - 1)
    row = -G0[0][c.site_sub[site[:, None], site[None, :]]]
    lo, hi = np.take_along_axis(row, i[..., None], 2)[..., 0], np.take_along_axis(row, i[..., None] + 1, 2)[..., 0]
    g = sg * (lo + (x - i) * (hi - lo))
    N = walker.fresh_N(prob, site, tau, s)
    sign = 1
    for sp in range(2):
        e = np.exp((1 - 2 * sp) * gamma * s)
        A = np.diag(e) - g * (e - 1.0)[None, :]
        bound = 4 * n * 2.0 ** -52 * np.abs(A).sum(1).max() * np.abs(N[sp]).sum(1).max()
        assert np.abs(A @ N[sp] - np.eye(n)).max() <= bound
        sign *= int(np.linalg.slogdet(A)[0])
    assert N[2] == sign
