"""The launch forms of the FP32 direct iteration (csrc/emd_taps.cu: taps in the
constant bank; split items with grid barriers) against the CTA-pair kernel,
which evaluates every output with the same FP32 operations in the same order:
the iterates agree bit for bit. Shapes take each branch of the form rule:
the taps form on 64 x 128 and 64 x 64 tiles, with and without partial planes,
Kc mod 4 = 1 and 3, several chunks, r = 2, heavy-tailed noise (half the
exposures per chunk); the split form with both tile sizes, one exposure,
and chunks that carry Den and N' over."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

# (H, W, n, K, r, nu)
CASES = [(1300, 2600, 3, 5, 1, 0.0),    # taps, 64 x 64 tiles, partials, Kc mod 4 = 1
         (2100, 2603, 3, 7, 1, 0.0),    # taps, 64 x 128 tiles, ragged columns
         (701, 803, 9, 21, 1, 0.0),     # taps, partials, one chunk
         (1027, 1030, 11, 43, 1, 0.0),  # taps, chunks of 4, 4 and 3 exposures
         (1200, 1301, 3, 13, 2, 0.0),   # taps, r = 2
         (1300, 1300, 3, 15, 1, 3.0),   # taps, heavy-tailed, chunks of 1
         (520, 530, 9, 9, 1, 0.0),      # split, 32 x 64 tiles
         (61, 47, 1, 47, 1, 0.0),       # split, one exposure, widest PSF
         (200, 150, 5, 9, 1, 2.0),      # split, heavy-tailed, chunks of 2, 2 and 1
         (90, 70, 3, 13, 2, 4.0)]       # split, heavy-tailed, r = 2


@pytest.mark.parametrize("H,W,n,K,r,nu", CASES)
def test_launch_forms_equal_the_cta_pair_kernel(H, W, n, K, r, nu):
    from paper_2302_05804_gb300 import emd
    p = synth.make_problem("hsc", H=H, W=W, n=n, K=K, r=r, mask_frac=0.03,
                           fwhm=(1.2 * r, 2.5 * r), n_points=40, n_gal=3, seed_offset=H + K)
    g = np.random.default_rng(n)
    x0 = (g.uniform(0.5, 1.5, (r * H, r * W)) * 10.0).astype(np.float32)
    out = []
    for prec in (emd.EMD_PREC_FP32, emd.EMD_PREC_FP32_PAIR):
        d = emd.Deconvolver(H, W, n, K, r)
        try:
            d.set_frames(p.y, p.v, p.f, p.mask)
            if nu > 0:
                d.set_noise(emd.EMD_NOISE_STUDENT_T, nu)
            d.set_precision(prec)
            d.set_x(x0)
            d.iterate(1)
            one = d.x()
            d.iterate(2)
            out.append((one, d.x()))
        finally:
            d.close()
    np.testing.assert_array_equal(out[0][0], out[1][0])
    np.testing.assert_array_equal(out[0][1], out[1][1])
