"""The numerator N = sum_t F_t^T (u_t y_t) of both kernels that compute it (the
launches with the taps in their parameters; the CTA-pair kernel, for kernels
that do not fit there and for the streaming passes).

Rounding: with equal taps and data a sum of m terms grows evenly, and a chain of
m FP32 additions leaves a relative error of c sqrt(m / 3), c = 2.5e-8 the rms of one
rounding. Blocks of 4 Kc terms and their sum (Kc / 4 of them): 3.0 c to 3.2 c for
Kc = 43 and 47 (one chain of Kc^2 terms: 25 c to 27 c = 6.2e-7 to 6.8e-7). n
exposures add c sqrt(n / 3). The bar 2e-7 is 2.3 to 2.7 times that for n <= 4."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def frames(H, W, n, K, seed):
    g = np.random.default_rng(seed)
    f = g.uniform(0.9, 1.1, (n, K, K))
    f = (f / f.sum(axis=(1, 2), keepdims=True)).astype(np.float32)
    v = g.uniform(50.0, 60.0, (n, H, W)).astype(np.float32)
    y = g.uniform(10.0, 12.0, (n, H, W)).astype(np.float32)
    return y, v, f


# (H, W, n, K, r); T: tiles of 64 x 128
CASES = [(150, 170, 1, 43, 1),    # parts, 64 x 64 tiles
         (190, 140, 4, 43, 1),    # four parts
         (140, 150, 3, 23, 2),    # r = 2: two exposures a launch
         (150, 170, 2, 93, 2)]    # kernels too large for the launch: CTA pairs


@pytest.mark.parametrize("H,W,n,K,r", CASES)
def test_rounding_of_the_numerator(H, W, n, K, r):
    from paper_2302_05804_gb300 import emd
    y, v, f = frames(H, W, n, K, H + n)
    d = emd.Deconvolver(H, W, n, K, r)
    try:
        d.set_frames(y, v, f)
        N = np.empty((r * H, r * W), np.float32)
        emd.emd_get_numerator(d.ctx, N)
    finally:
        d.close()
    want = oracle.numerator(y, (np.float32(1.0) / v).astype(np.float64), f, r)
    err = np.linalg.norm(N - want) / np.linalg.norm(want)
    assert err <= 2e-7


# shapes over the rules: one and more launches, rows of pixels past 64 x 64 and
# 64 x 128 tiles, odd sides, tiles that add in place
@pytest.mark.parametrize("H,W,K,r", [(61, 47, 47, 1), (300, 257, 5, 1), (129, 131, 9, 2),
                                     (1300, 2603, 7, 1), (2497, 2049, 5, 1)])
def test_both_kernels_agree_bit_for_bit(H, W, K, r):
    """With one exposure a streaming pass is one iteration, with its numerator from
    the CTA-pair kernel."""
    from paper_2302_05804_gb300 import emd
    g = np.random.default_rng(H)
    y, v, f = frames(H, W, 1, K, H)
    y += g.normal(0.0, 20.0, y.shape).astype(np.float32)
    mask = (g.random(y.shape) > 0.05).astype(np.uint8)
    x0 = g.uniform(1.0, 2.0, (r * H, r * W)).astype(np.float32)
    d = emd.Deconvolver(H, W, 1, K, r)
    try:
        d.set_frames(y, v, f, mask)
        d.set_x(x0)
        d.iterate(1)
        a = d.x()
        d.set_x(x0)
        emd.emd_iterate_streaming(d.ctx, 1)
        b = d.x()
    finally:
        d.close()
    np.testing.assert_array_equal(a, b)


def test_many_exposures_in_order():
    """Several launches add their exposures in exposure order: the first exposures
    alone, then all of them with the rest weighing nothing, give the same bits."""
    from paper_2302_05804_gb300 import emd
    H, W, n, K = 140, 200, 11, 31
    y, v, f = frames(H, W, n, K, 5)
    out = []
    for m in (n, 7):
        mask = np.ones((n, H, W), np.uint8)
        mask[7:] = 0
        d = emd.Deconvolver(H, W, m, K, 1)
        try:
            d.set_frames(y[:m], v[:m], f[:m], mask[:m])
            N = np.empty((H, W), np.float32)
            emd.emd_get_numerator(d.ctx, N)
            out.append(N)
        finally:
            d.close()
    np.testing.assert_array_equal(out[0], out[1])
