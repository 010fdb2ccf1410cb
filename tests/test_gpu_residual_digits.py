"""G of a mixed walker measured right after the default recompute (residual from
digit planes), against the FP64 walker of the same decisions: 16 sites, beta =
16, orders about 600, condition numbers of N^-1 of 1e6 to 4e7.

Bound: twice the error with N from the Gauss-Jordan inverse, which is that of N
rounded to FP32.  The digits cut N0 at 2^-40 of its column maxima; at 2^-37 they
left up to 5 times that rounding, so an eighth of it adds up to sqrt(1 + 24 / 64)
= 1.2 of it, and the rest is for another realisation of the rounding."""
import numpy as np
import pytest

from tests.helpers import problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed", [284024626524, 358348827832, 395510928486, 268098011958])
def test_G_after_the_default_recompute_is_at_the_rounding_of_N(seed):
    import torch
    from paper_1901_01047_gb300 import walker
    nc, U, beta, warm = 16, 6.0, 16.0, 24
    c, eps, kr, G0 = problem(nc, 1.0, -0.15, U, beta, U / 2, 4096)
    prob = dict(nc=nc, site_sub=c.site_sub, U=U, beta=beta, K=1.0, G0=G0)
    kw = dict(k_sub=64, warmup_sweeps=warm, n_tau_meas=256, init_config_size=250, seed=seed, duplicate_rule="update",
              stream=torch.cuda.current_stream().cuda_stream)

    def measured(gw):
        gw.sweep(warm)
        gw.set_recompute(8, 0, True)
        gw.reset_measurements()
        gw.sweep(1)
        return gw.measure_G()[0][0]

    gw = walker.Walkers([prob], log_capacity=1 << 18, recompute_every=4, **kw)
    ref = measured(gw)
    log = gw.decision_log(0)
    gw.close()
    err = {}
    for method in ("gj", "auto"):
        gw = walker.Walkers([prob], precision="mixed", recompute_method=method, recompute_every=4, **kw)
        gw.set_forced_decisions(0, log)
        err[method] = np.linalg.norm(measured(gw) - ref) / np.linalg.norm(ref)
        gw.close()
    print(err)
    assert err["auto"] <= 2 * err["gj"], err
