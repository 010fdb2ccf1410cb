"""N right after a recompute of the mixed path against the FP64 inverse of
N^-1 = e^V - g0 (e^V - 1) on the walker's own vertex list, sweep by sweep, with
orders around one 32-box, one 128-tile and two tiles of the tensor-core
correction.  Bound 1e-6 of max|N|, as in tests/test_gpu_mixed.py: the FP32
rounding of N (6e-8) and what is left of the drift after one Newton step."""
import numpy as np
import pytest

from tests.helpers import problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("method", ["auto", "newton_df"])
@pytest.mark.parametrize("beta", [0.1, 0.75, 3.05, 6.2])
def test_recomputed_N_around_the_tiles_of_the_correction(beta, method):
    import torch
    from paper_1901_01047_gb300 import walker
    nc, U, n_tau = 16, 6.0, 1024
    c, eps, kr, G0 = problem(nc, 1.0, 0.0, U, beta, U / 2, n_tau)
    prob = dict(nc=nc, site_sub=c.site_sub, U=U, beta=beta, K=1.0, G0=G0)
    gw = walker.Walkers([prob], n_walkers=1, precision="mixed", k_sub=32, warmup_sweeps=20, n_tau_meas=16, seed=5,
                        recompute_every=4, recompute_at_measure=True, recompute_method=method,
                        stream=torch.cuda.current_stream().cuda_stream)
    gw.sweep(20)
    gamma = np.arccosh(1.0 + U * beta * nc / 2)
    for _ in range(6):
        gw.sweep(1)
        st = gw.state(0)
        site, tau, s = st["site"], st["tau"], st["s"].astype(np.float64)
        n = site.size
        x = tau[:, None] - tau[None, :]
        sg, x = np.where(x < 0, -1.0, 1.0), np.where(x < 0, x + beta, x) * (n_tau / beta)
        i = np.clip(x.astype(int), 0, n_tau - 1)
        row = -G0[0][c.site_sub[site[:, None], site[None, :]]]
        lo, hi = np.take_along_axis(row, i[..., None], 2)[..., 0], np.take_along_axis(row, i[..., None] + 1, 2)[..., 0]
        g = sg * (lo + (x - i) * (hi - lo))
        for sp in range(2):
            e = np.exp((1 - 2 * sp) * gamma * s)
            ref = np.linalg.inv(np.diag(e) - g * (e - 1.0)[None, :]) if n else np.zeros((0, 0))
            if n:
                assert np.abs(st["N"][sp] - ref).max() <= 1e-6 * np.abs(ref).max()
    gw.close()
