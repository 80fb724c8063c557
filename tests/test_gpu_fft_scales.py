"""The FFT form packs two exposures into one complex transform, whose rounding is of
the size of the larger. Exposures with flux scales of their own (PSFs that sum to
1, to 3e-4, to 4000; equal signal to noise) against the FP64 oracle, at the bars the
FFT form has elsewhere (relative L2 1e-5 after one iteration, 2e-5 after five)."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

FLUX = [1.0, 3e-4, 4000.0, 1.0, 0.02, 900.0, 1.0]


@pytest.mark.parametrize("H,W,n,K,r,nu", [(200, 150, 7, 21, 1, 0.0),
                                          (1130, 1160, 3, 43, 1, 0.0),  # split launch
                                          (110, 120, 5, 21, 2, 0.0),
                                          (60, 50, 2, 13, 3, 0.0),
                                          (200, 150, 5, 21, 1, 3.0)])
def test_exposures_of_different_flux(H, W, n, K, r, nu):
    from paper_2302_05804_gb300 import emd
    p = synth.make_problem("hsc", H=H, W=W, n=n, K=K, r=r, mask_frac=0.03,
                           fwhm=(1.5 * r, 3.0 * r), n_points=max(3, H * W // 400), n_gal=2)
    c = np.array(FLUX[:n], np.float32)[:, None, None]
    y, v, f = p.y * c, p.v * c * c, p.f * c
    u, bad = oracle.weights(v, p.mask, y)
    assert bad == 0
    y0 = np.where(p.mask != 0, y.astype(np.float64), 0.0)
    g = np.random.default_rng(H + n)
    x0 = (g.uniform(0.5, 1.5, (r * H, r * W)) * max(np.nanmean(p.y), 1.0)).astype(np.float32)
    xo = x0.astype(np.float64)
    N = oracle.numerator(y0, u, f, r)
    d = emd.Deconvolver(H, W, n, K, r)
    try:
        d.set_frames(y, v, f, p.mask)
        d.set_precision(emd.EMD_PREC_FFT_FP32)
        if nu > 0:
            d.set_noise(emd.EMD_NOISE_STUDENT_T, nu)
        d.set_x(x0)
        for k, bar in ((1, 1e-5), (4, 2e-5)):
            d.iterate(k)
            if nu > 0:
                for _ in range(k):
                    xo = oracle.em_step_student(xo, y0, u, f, nu, r)[0]
            else:
                xo = oracle.em_run(xo, N, u, f, k, r)
            x = d.x().astype(np.float64)
            err = np.linalg.norm(x - xo) / np.linalg.norm(xo)
            assert err <= bar
    finally:
        d.close()
