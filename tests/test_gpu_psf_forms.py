"""Eq. (4) fits that take each kernel of csrc/emd_psf.cu by the strips of fine
pixels a thread has -- one, two to four (both with the moments in registers),
more than four (moments in memory) -- against the FP64 oracle. The bars are
those derived for the other fits (tests/test_gpu_psf.py): core elements 1e-5
of max|h|, relative L2 1e-3, the reported loss within the Cauchy-Schwarz
bound of a model error of 4e-6 |f|."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


# 160 PSFs: one CTA each, so ceil(Kh ceil(Kh / 4) / 512) strips per thread
@pytest.mark.parametrize("K,r", [(21, 2),    # 41 x 11: one
                                 (25, 2),    # 49 x 13: two
                                 (43, 2),    # 85 x 22: four
                                 (33, 3)])   # 97 x 25: five
def test_strips_per_thread_match_the_oracle(K, r):
    from paper_2302_05804_gb300 import emd
    n, lam, iters = 160, 1e-2, 60
    rng = np.random.default_rng(K)
    f = np.stack([synth.moffat_psf(K, rng.uniform(2.0, 3.5), rng.uniform(2.5, 4.5))
                  for _ in range(n)]).astype(np.float32)
    g = synth.gaussian_kernel(r).astype(np.float32)
    h, loss = emd.emd_fit_psf(f, g, r, lam, 1e-4, iters)
    Kh = r * (K - 1) + 1
    for t in (0, n - 1):
        h0 = np.kron(f[t].astype(np.float64), np.ones((r, r)))[:Kh, :Kh] / r ** 2
        ho = oracle.psf_fit(f[t], g, r, lam, iters, 1e-4, h0)
        core = h0 >= 1e-3 * h0.max()
        assert np.abs(h[t] - ho)[core].max() <= 1e-5 * np.abs(ho).max()
        assert np.linalg.norm(h[t] - ho) <= 1e-3 * np.linalg.norm(ho)
        L = oracle.psf_loss(h[t].astype(np.float64), f[t], g, r, lam)
        dm = 4e-6 * np.linalg.norm(f[t].astype(np.float64))
        assert abs(float(loss[t]) - L) <= 2 * np.sqrt(L) * dm + dm * dm
