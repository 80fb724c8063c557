"""Heavy-tailed noise in the FFT form transforms u' z and u' y of an exposure as one
complex image, whose rounding is of the size of the larger: data far above the
model (a start 1e-4 of the sky, and of twice that on one half of the image) and
far below it, against the FP64 oracle, at the bars the FFT form has elsewhere
(relative L2 1e-5 after one iteration, 2e-5 after five)."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W,n,K,r,nu,start", [(200, 150, 5, 21, 1, 3.0, 1e-4),   # groups
                                                (200, 150, 4, 21, 1, 3.0, 300.0),
                                                (1000, 900, 3, 31, 1, 3.0, 1e-4),  # one group
                                                (90, 70, 5, 13, 2, 4.0, 1e-4),
                                                (60, 50, 3, 13, 3, 4.0, 1e-4)])
def test_data_far_from_the_model(H, W, n, K, r, nu, start):
    from paper_2302_05804_gb300 import emd
    p = synth.make_problem("hsc", H=H, W=W, n=n, K=K, r=r, mask_frac=0.03,
                           fwhm=(1.5 * r, 3.0 * r), n_points=max(3, H * W // 400), n_gal=2)
    u, y0, _, _ = oracle.prepare(p)
    g = np.random.default_rng(H + n)
    x0 = (g.uniform(0.5, 1.5, (r * H, r * W)) * start * max(np.nanmean(p.y), 1.0))
    x0[:, r * W // 2:] *= 2.0
    x0 = x0.astype(np.float32)
    xo = x0.astype(np.float64)
    d = emd.Deconvolver(H, W, n, K, r)
    try:
        d.set_frames(p.y, p.v, p.f, p.mask)
        d.set_precision(emd.EMD_PREC_FFT_FP32)
        d.set_noise(emd.EMD_NOISE_STUDENT_T, nu)
        d.set_x(x0)
        for k, bar in ((1, 1e-5), (4, 2e-5)):
            d.iterate(k)
            for _ in range(k):
                xo = oracle.em_step_student(xo, y0, u, p.f, nu, r)[0]
            x = d.x().astype(np.float64)
            assert np.linalg.norm(x - xo) <= bar * np.linalg.norm(xo)
    finally:
        d.close()
