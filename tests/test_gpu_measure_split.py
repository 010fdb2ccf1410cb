"""G(tau) of walkers measured with the vertices of an item split (few walkers) and
whole (many): the chains of 2 and of 6 walkers are the same for the first two, and so
must G be.  16 sites, 128 tau points: 64 and 192 items, on either side of the line;
36 sites: 144 items for one walker and 288 for two.

Bound: the same FP32 products and sums of 32 terms either way; only the totals are
added in another order, double-float and FP64: 2^-40 of sums of some 100 largest |G|."""
import numpy as np
import pytest

from tests.helpers import problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nc,few,many,ntm", [(16, 2, 6, 128), (8, 2, 12, 100), (36, 1, 2, 256)])
def test_split_items_leave_G(nc, few, many, ntm):
    import torch
    from paper_1901_01047_gb300 import walker
    U, beta = 6.0, 72.0 / nc
    c, eps, kr, G0 = problem(nc, 1.0, 0.0, U, beta, U / 2, 1024)
    prob = dict(nc=nc, site_sub=c.site_sub, U=U, beta=beta, K=1.0, G0=G0)
    got = []
    for W in (few, many):
        gw = walker.Walkers([prob], n_walkers=W, precision="mixed", k_sub=64, warmup_sweeps=8, n_tau_meas=ntm, seed=2,
                            init_config_size=250, recompute_every=8, recompute_at_measure=True,
                            stream=torch.cuda.current_stream().cuda_stream)
        gw.sweep(9)
        order = gw.state(0)["site"].size
        got.append(gw.measure_G()[0][:few])
        gw.close()
    print("order", order)
    assert order > 100
    for a, b in zip(*got):
        assert np.abs(a - b).max() <= 100 * 2.0 ** -40 * np.abs(a).max()
