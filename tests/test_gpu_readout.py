"""Edges of the two-stage NFFT read-out and of the blocked Gauss-Jordan inverse.

The NFFT of the FP64 path and the dense DFT measure the same sums on the same
chain; the window error of the NFFT is about 1e-12 of sum |c_ij|, so 1e-10
relative to the largest value bounds both the factorisations of the transform
(L = 4 n_omega = P Q: prime cofactors, squares, P = 2) and the direct sum that
larger grids take."""
import numpy as np
import pytest

from tests.helpers import problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_omega", [8, 29, 33, 64, 1000])
def test_nfft_readout_equals_the_dense_transform(n_omega):
    import torch
    from paper_1901_01047_gb300 import walker
    c, eps, kr, G0 = problem(4, 1.0, 0.0, 4.0, 4.0, 1.0, 1024)
    prob = dict(nc=4, site_sub=c.site_sub, U=4.0, beta=4.0, K=1.0, G0=G0)
    got = []
    for method in ("nfft", "dft"):
        gw = walker.Walkers([prob], n_walkers=2, k_sub=16, warmup_sweeps=5, n_tau_meas=16, seed=11,
                            n_omega_meas=n_omega, freq_method=method, stream=torch.cuda.current_stream().cuda_stream)
        gw.sweep(8)
        got.append(np.array(gw.measure_M()[0]))
        gw.close()
    assert np.abs(got[0] - got[1]).max() < 1e-10 * np.abs(got[1]).max()


@pytest.mark.parametrize("n", [1, 2, 15, 16, 17, 31, 48, 129, 255])
def test_inverse_at_the_edges_of_its_panels(n):
    # residual of the returned inverse: |A N - 1| <= 4 n eps |A| |N| (norms: largest row sum)
    from paper_1901_01047_gb300 import walker
    nc, U, beta = 4, 4.0, 6.0
    c, eps, kr, G0 = problem(nc, 1.0, 0.0, U, beta, 1.0, 1024)
    prob = dict(nc=nc, site_sub=c.site_sub, U=U, beta=beta, K=1.0, G0=G0)
    rng = np.random.default_rng(n)
    site, tau = rng.integers(0, nc, n).astype(np.int32), rng.random(n) * beta
    s = np.where(rng.random(n) < 0.5, 1, -1).astype(np.int32)
    gamma = np.arccosh(1.0 + U * beta * nc / 2)
    x = tau[:, None] - tau[None, :]
    sg, x = np.where(x < 0, -1.0, 1.0), np.where(x < 0, x + beta, x) * (1024 / beta)
    i = np.clip(x.astype(int), 0, 1023)
    row = -G0[0][c.site_sub[site[:, None], site[None, :]]]
    lo, hi = np.take_along_axis(row, i[..., None], 2)[..., 0], np.take_along_axis(row, i[..., None] + 1, 2)[..., 0]
    g = sg * (lo + (x - i) * (hi - lo))
    for fn in ("dca_fresh_N", "dca_fresh_N_noalloc"):
        N = walker.fresh_N(prob, site, tau, s, fn=fn)
        sign = 1
        for sp in range(2):
            e = np.exp((1 - 2 * sp) * gamma * s)
            A = np.diag(e) - g * (e - 1.0)[None, :]
            bound = 4 * n * 2.0 ** -52 * np.abs(A).sum(1).max() * np.abs(N[sp]).sum(1).max()
            assert np.abs(A @ N[sp] - np.eye(n)).max() <= bound
            sign *= int(np.linalg.slogdet(A)[0])
        assert N[2] == sign
