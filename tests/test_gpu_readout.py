"""Edges of the two-stage NFFT read-out.

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
