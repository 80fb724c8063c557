"""The FFT form's pairs of exposures and exposure groups (csrc/emd_fft.cu)
against the FP64 oracle, at the bars the FFT form has elsewhere (relative L2
1e-5 after one iteration, 2e-5 after five): odd n (a pair with one exposure),
one tile with many groups, groups of unequal size, more tiles than one group
allows, r = 2 and heavy-tailed noise with groups."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

# (H, W, n, K, r, nu)
CASES = [(60, 50, 40, 15, 1, 0.0),      # one tile, one pair per group
         (200, 150, 9, 43, 1, 0.0),     # 6 tiles, odd n
         (700, 650, 11, 43, 1, 0.0),    # 72 tiles, groups of unequal size
         (1100, 900, 3, 43, 1, 0.0),    # 143 tiles, odd n, one group of two pairs
         (110, 120, 7, 21, 2, 0.0),     # r = 2, groups through the scratch
         (200, 150, 5, 21, 1, 3.0),     # heavy-tailed, groups
         (90, 70, 5, 13, 2, 4.0)]       # heavy-tailed, r = 2


@pytest.mark.parametrize("H,W,n,K,r,nu", CASES)
def test_pairs_and_groups_match_the_oracle(H, W, n, K, r, nu):
    from paper_2302_05804_gb300 import emd
    p = synth.make_problem("hsc", H=H, W=W, n=n, K=K, r=r, mask_frac=0.03,
                           fwhm=(1.5 * r, 3.0 * r), n_points=max(3, H * W // 400), n_gal=2)
    g = np.random.default_rng(H + n)
    x0 = (g.uniform(0.5, 1.5, (r * H, r * W)) * max(np.nanmean(p.y), 1.0)).astype(np.float32)
    u, y, N, _ = oracle.prepare(p)
    xo = x0.astype(np.float64)
    d = emd.Deconvolver(H, W, n, K, r)
    try:
        d.set_frames(p.y, p.v, p.f, p.mask)
        d.set_precision(emd.EMD_PREC_FFT_FP32)
        if nu > 0:
            d.set_noise(emd.EMD_NOISE_STUDENT_T, nu)
        d.set_x(x0)
        for k, bar in ((1, 1e-5), (4, 2e-5)):
            d.iterate(k)
            if nu > 0:
                for _ in range(k):
                    xo = oracle.em_step_student(xo, y, u, p.f, nu, r)[0]
            else:
                xo = oracle.em_run(xo, N, u, p.f, k, r)
            x = d.x().astype(np.float64)
            assert np.linalg.norm(x - xo) <= bar * np.linalg.norm(xo)
    finally:
        d.close()
