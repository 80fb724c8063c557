"""The FFT form's update where the numerator is exactly 0: a latent pixel that
valid pixels reach gets x' = 0 (data of 0, or terms that cancel), one that none
reaches keeps its x. Every pixel against the FP64 oracle, bar 1e-4 of
max(|x|, rms x): the PSFs have no tap below 0.3 of their mean, so that Den is
nowhere below 0.3 / K^2 of its typical value and the transform's floor of
~1e-7 of it stays under 1e-4 of any pixel. Shapes: one tile, exposure groups, the
split launch (more tiles than SMs), r = 2, heavy-tailed noise."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def frames(H, W, n, K, zero_taps, seed):
    g = np.random.default_rng(seed)
    f = g.uniform(0.3, 1.0, (n, K, K))
    if zero_taps:  # an empty rim: pixels under it alone do not count
        f[:, :2] = f[:, -2:] = 0.0
        f[:, :, :2] = f[:, :, -2:] = 0.0
    f = (f / f.sum(axis=(1, 2), keepdims=True)).astype(np.float32)
    v = g.uniform(50.0, 90.0, (n, H, W)).astype(np.float32)
    y = g.uniform(5.0, 20.0, (n, H, W)).astype(np.float32)
    mask = (g.random((n, H, W)) > 0.05).astype(np.uint8)
    a, b = H // 2, W // 2
    y[:, :a, :b] = 0.0                       # valid and 0: N = 0
    mask[:, a:, b:] = 0                      # no valid pixel
    y[0, a:, :K], y[1, a:, :K] = 7.0, -7.0   # two exposures that cancel
    v[:, a:, :K], mask[:2, a:, :K], mask[2:, a:, :K] = 64.0, 1, 0
    f[1] = f[0]
    y[mask == 0] = np.nan
    return y, v, f, mask


@pytest.mark.parametrize("H,W,n,K,r,nu", [(70, 66, 3, 9, 1, 0.0),
                                          (260, 250, 9, 21, 1, 0.0),
                                          (1130, 1160, 3, 43, 1, 0.0),
                                          (150, 140, 4, 13, 2, 0.0),
                                          (150, 170, 3, 9, 1, 3.0)])
def test_zero_numerators_against_the_oracle(H, W, n, K, r, nu):
    from paper_2302_05804_gb300 import emd
    y, v, f, mask = frames(H, W, n, K, K < 40, H + K)
    u, bad = oracle.weights(v, mask, y)
    assert bad == 0
    y0 = np.where(mask != 0, y.astype(np.float64), 0.0)
    N = oracle.numerator(y0, u, f, r)
    x = np.full((r * H, r * W), 3.0)
    d = emd.Deconvolver(H, W, n, K, r)
    try:
        d.set_frames(y, v, f, mask)
        d.set_precision(emd.EMD_PREC_FFT_FP32)
        if nu > 0:
            d.set_noise(emd.EMD_NOISE_STUDENT_T, nu)
        d.set_x(x.astype(np.float32))
        d.iterate(1)
        got = d.x().astype(np.float64)
    finally:
        d.close()
    want = oracle.em_step_student(x, y0, u, f, nu, r)[0] if nu > 0 else oracle.em_step(x, N, u, f, r)
    h, w = r * (H // 2 - K), r * (W // 2 - K)
    assert h > 0 and w > 0 and (want[:h, :w] == 0.0).all()
    assert (want[-h:, -w:] == 3.0).all()
    scale = np.maximum(np.abs(want), np.sqrt(np.mean(want * want)))
    assert (np.abs(got - want) / scale).max() <= 1e-4
