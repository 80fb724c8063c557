"""Captured FP32 iterations replay on the frame set that is loaded at the replay:
weights, numerator, start and PSFs alike. Two frame sets with different PSFs; the
graph is captured with the first and replayed with the second, and must give the
bits of a context that never captured. Shapes: the launches that carry taps in
their parameters (64 x 64 tiles and parts; 64 x 128 tiles adding in place;
heavy-tailed), and the split form."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def problem(H, W, n, K, r, seed):
    return synth.make_problem("hsc", H=H, W=W, n=n, K=K, r=r, mask_frac=0.03,
                              fwhm=(1.2 * r, 2.5 * r), n_points=40, n_gal=3, seed_offset=seed)


@pytest.mark.parametrize("H,W,n,K,r,nu", [(701, 803, 9, 21, 1, 0.0), (2100, 2603, 3, 7, 1, 0.0),
                                          (1300, 1300, 3, 15, 1, 3.0), (1200, 1301, 3, 13, 2, 0.0),
                                          (128, 131, 4, 15, 1, 0.0)])
def test_replay_uses_the_new_frame_sets_psfs(H, W, n, K, r, nu):
    import torch
    from paper_2302_05804_gb300 import emd
    old, new = problem(H, W, n, K, r, 1), problem(H, W, n, K, r, 2)
    x0 = np.random.default_rng(3).uniform(5.0, 15.0, (r * H, r * W)).astype(np.float32)

    def context():
        d = emd.Deconvolver(H, W, n, K, r)
        if nu > 0:
            d.set_noise(emd.EMD_NOISE_STUDENT_T, nu)
        return d

    a, b = context(), context()
    try:
        st = torch.cuda.Stream()
        emd.emd_set_stream(a.ctx, st)
        a.set_frames(old.y, old.v, old.f, old.mask)
        a.set_x(x0)
        a.iterate(2)
        was = a.x()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=st):
            a.iterate(2)  # two: the buffers are back where they were
        a.set_x(x0)
        graph.replay()
        torch.cuda.synchronize()
        np.testing.assert_array_equal(a.x(), was)
        a.set_frames(new.y, new.v, new.f, new.mask)
        a.set_x(x0)
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        got = a.x()
        b.set_frames(new.y, new.v, new.f, new.mask)
        b.set_x(x0)
        b.iterate(2)
        np.testing.assert_array_equal(got, b.x())
    finally:
        a.close()
        b.close()
