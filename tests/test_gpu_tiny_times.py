"""N from scratch for vertices whose times differ by less than the fixed-point
words of the build resolve (2^-62 beta): g0 jumps by one at equal times, so their
order decides, and the matrix is that of g0(0+) above and -g0(beta) below the
diagonal.  Bound of N: 1e-12 times the condition number of the 4 x 4 matrix."""
import numpy as np
import pytest

from tests.helpers import problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fn", ["dca_fresh_N", "dca_fresh_N_noalloc"])
@pytest.mark.parametrize("tau", [[0.0, 1e-25, 2.0, 3.0], [1e-25, 0.0, 2.0, 3.0], [5e-324, 0.0, 1e-300, 2e-300],
                                 [0.0, 0.0, 1e-25, 1e-25], [3.0, 3.0 - 2.0 ** -51, 3.0, 0.0]])
def test_order_of_times_closer_than_the_grid_words(tau, fn):
    from paper_1901_01047_gb300 import walker
    nc, U, beta, n_tau = 4, 4.0, 4.0, 1024
    c, eps, kr, G0 = problem(nc, 1.0, 0.0, U, beta, 1.0, n_tau)
    prob = dict(nc=nc, site_sub=c.site_sub, U=U, beta=beta, K=1.0, G0=G0)
    site, tau = np.zeros(4, np.int32), np.array(tau)
    s = np.array([1, -1, 1, -1], np.int32)
    gamma = np.arccosh(1.0 + U * beta * nc / 2)
    t = tau[:, None] - tau[None, :]
    sg, x = np.where(t < 0, -1.0, 1.0), np.where(t < 0, t + beta, t) * (n_tau / beta)
    i = np.clip(x.astype(int), 0, n_tau - 1)
    row = -G0[0][c.site_sub[0, 0]]
    g = sg * (row[i] + (x - i) * (row[i + 1] - row[i]))
    N = walker.fresh_N(prob, site, tau, s, fn=fn)
    sign = 1
    for sp in range(2):
        e = np.exp((1 - 2 * sp) * gamma * s)
        A = np.diag(e) - g * (e - 1.0)[None, :]
        ref = np.linalg.inv(A)
        assert np.abs(N[sp] - ref).max() <= 1e-12 * np.linalg.cond(A) * np.abs(ref).max()
        sign *= int(np.linalg.slogdet(A)[0])
    assert N[2] == sign
