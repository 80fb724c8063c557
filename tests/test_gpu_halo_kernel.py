"""The halo-exchange kernel itself (csrc/emd_halo.cu): contexts with a fixed tile
shape run it, and shapes that no launch form takes. Bit for bit against the
CTA-pair kernel, Gaussian and heavy-tailed, with ring slots reused within a launch
and the ring laid out anew when the noise model changes; and its autotuner on a
shape that starts undecided. (Contexts with EMD_TILE_AUTO run the launch forms on
the shapes of test_gpu_halo.py.)"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def problem(H, W, n, K, r):
    return synth.make_problem("hsc", H=H, W=W, n=n, K=K, r=r, mask_frac=0.05,
                              fwhm=(1.2 * r, 3.0 * r), n_points=60, n_gal=4, seed_offset=H + W + K)


def context(emd, p, shape):
    """shape: a tile shape, or None for the CTA-pair kernel."""
    d = emd.Deconvolver(p.H, p.W, p.n, p.K, p.r)
    d.set_frames(p.y, p.v, p.f, p.mask)
    if shape is None:
        d.set_precision(emd.EMD_PREC_FP32_PAIR)
    else:
        d.set_tile_shape(shape)
    d.set_x((np.random.default_rng(p.n).uniform(0.5, 1.5, (p.r * p.H, p.r * p.W)) * 10.0)
            .astype(np.float32))
    return d


# (H, W, n, K, r, nu): two tiles; ragged; K = 1; r = 2; 1056 and 2560 forward items
# on about 1000 slots; the same with two tiles a slot
CASES = [(96, 80, 3, 15, 1, 0.0), (300, 257, 5, 43, 1, 0.0), (260, 300, 4, 1, 1, 0.0),
         (200, 330, 4, 9, 2, 0.0), (1400, 90, 3, 21, 1, 2.0), (1030, 1024, 8, 43, 1, 0.0),
         (700, 650, 40, 15, 1, 0.0), (1024, 1000, 12, 25, 1, 3.0)]


@pytest.mark.parametrize("H,W,n,K,r,nu", CASES)
@pytest.mark.parametrize("shape", [1, 2, 3])
def test_bits_of_the_cta_pair_kernel(H, W, n, K, r, nu, shape):
    from paper_2302_05804_gb300 import emd
    p = problem(H, W, n, K, r)
    out = []
    for which in (shape, None):
        d = context(emd, p, which)
        try:
            if nu > 0:
                d.set_noise(emd.EMD_NOISE_STUDENT_T, nu)
            d.iterate(3)
            out.append(d.x())
        finally:
            d.close()
    np.testing.assert_array_equal(out[0], out[1])


def test_ring_is_laid_out_anew_for_each_noise_model():
    from paper_2302_05804_gb300 import emd
    p = problem(520, 400, 6, 15, 1)
    out = []
    for which in (emd.EMD_TILE_64, None):
        d = context(emd, p, which)
        try:
            for nu in (0.0, 4.0, 0.0, 2.0):
                d.set_noise(emd.EMD_NOISE_STUDENT_T if nu else emd.EMD_NOISE_GAUSSIAN, nu)
                d.iterate(2)
                out.append(d.x())
        finally:
            d.close()
    for a, b in zip(out[:4], out[4:]):
        np.testing.assert_array_equal(a, b)


def test_autotuner_on_a_shape_without_a_launch_form():
    """K = 3 (below the taps form's 5) and 512 tiles of 64 x 128 (above the split
    form's): EMD_TILE_AUTO times the kernel's tile shapes on the first iterations."""
    from paper_2302_05804_gb300 import emd
    p = problem(2047, 2040, 2, 3, 1)
    d = context(emd, p, emd.EMD_TILE_AUTO)
    try:
        assert not d.tile_shape()[1]
        seen, done = set(), 0
        while done < 16 and not d.tile_shape()[1]:
            d.iterate(1)
            seen.add(d.tile_shape()[0])
            d.x()  # waits
            done += 1
        shape, decided = d.tile_shape()
        assert decided and shape in (1, 2, 3) and len(seen) > 1
        d.iterate(1)
        got = d.x()
    finally:
        d.close()
    d = context(emd, p, None)
    try:
        d.iterate(done + 1)
        np.testing.assert_array_equal(got, d.x())
    finally:
        d.close()
    d = context(emd, p, emd.EMD_TILE_AUTO)
    try:
        assert d.tile_shape() == (shape, True)  # kept for the problem shape
    finally:
        d.close()
