"""Device memory of a context: what emd_create takes is what every mode needs (u,
y and the latent planes), and the FP32 direct form's work planes are bounded."""
import numpy as np
import pytest

from paper_2302_05804_gb300 import emd

# H, W, n, K, r
SHAPES = [(900, 900, 24, 43, 1), (512, 512, 33, 85, 2), (512, 512, 100, 15, 4),
          (1000, 1000, 31, 47, 8), (1000, 1000, 31, 85, 4), (128, 128, 4, 15, 1),
          (128, 131, 100, 47, 1), (4096, 4096, 33, 43, 1), (700, 650, 40, 15, 1),
          (2048, 2048, 33, 85, 2)]


def plane_bytes(H, W, n, K, r):
    """An upper bound on one plane: two more of them with each exposure."""
    return (emd.emd_ctx_bytes(H, W, n + 1, K, r) - emd.emd_ctx_bytes(H, W, n, K, r)) / 2


@pytest.mark.parametrize("H,W,n,K,r", SHAPES)
def test_context_bytes(H, W, n, K, r):
    plane = plane_bytes(H, W, n, K, r)
    base = emd.emd_ctx_bytes(H, W, n, K, r)
    # u and y, two iterates, N and Den; rounding and reductions below 1 MB
    assert 0 < base <= (2 * n + 4 * r * r) * plane + (1 << 20)


@pytest.mark.gpu
@pytest.mark.parametrize("H,W,n,K,r", [s for s in SHAPES if s[:2] != (4096, 4096)])
def test_first_iteration_takes_a_bounded_workspace(H, W, n, K, r):
    """Half of what the context holds, or 64 MB, or two exposures of r^2 + 1 planes
    (heavy-tailed noise doubles an exposure's) where that is more; nothing with
    emd_create or emd_set_frames. (cudaMalloc rounds to 2 MB, and a kernel's first
    launch may take some: 32 MB allowed for.)"""
    import torch
    g = torch.Generator(device="cuda").manual_seed(H + n)
    y = torch.rand((n, H, W), generator=g, device="cuda") + 5.0
    f = torch.rand((n, K, K), generator=g, device="cuda") / (K * K)
    v = torch.full((n, H, W), 50.0, device="cuda")
    torch.cuda.synchronize()
    free = [torch.cuda.mem_get_info()[0]]
    d = emd.Deconvolver(H, W, n, K, r)
    try:
        d.set_frames(y, v, f)
        free.append(torch.cuda.mem_get_info()[0])
        d.iterate(1)
        torch.cuda.synchronize()
        free.append(torch.cuda.mem_get_info()[0])
    finally:
        d.close()
    base = emd.emd_ctx_bytes(H, W, n, K, r)
    assert free[0] - free[1] <= base + (32 << 20)
    most = max(base / 2, 64 << 20, 2 * (1 + r * r) * plane_bytes(H, W, n, K, r))
    assert free[1] - free[2] <= most + (32 << 20)


@pytest.mark.gpu
@pytest.mark.parametrize("H,W,n,K,r,nu", [(200, 230, 100, 29, 4, 0.0),   # split, chunks of 9
                                          (200, 230, 60, 29, 4, 3.0),
                                          (1000, 1010, 17, 15, 1, 0.0)])  # taps, two chunks
def test_chunks_within_the_bound_give_the_same_bits(H, W, n, K, r, nu):
    import synth
    p = synth.make_problem("hsc", H=H, W=W, n=n, K=K, r=r, mask_frac=0.03,
                           fwhm=(1.2 * r, 2.5 * r), n_points=40, n_gal=3, seed_offset=n)
    x0 = np.random.default_rng(n).uniform(5.0, 15.0, (r * H, r * W)).astype(np.float32)
    out = []
    for prec in (emd.EMD_PREC_FP32, emd.EMD_PREC_FP32_PAIR):
        d = emd.Deconvolver(H, W, n, K, r)
        try:
            d.set_frames(p.y, p.v, p.f, p.mask)
            if nu > 0:
                d.set_noise(emd.EMD_NOISE_STUDENT_T, nu)
            d.set_precision(prec)
            d.set_x(x0)
            d.iterate(2)
            out.append(d.x())
        finally:
            d.close()
    np.testing.assert_array_equal(out[0], out[1])


@pytest.mark.gpu
@pytest.mark.parametrize("H,W,n,K,nu", [(701, 803, 9, 21, 0.0), (128, 131, 4, 15, 3.0),
                                        (900, 1000, 4, 43, 0.0), (900, 1000, 3, 43, 2.0)])
def test_first_iteration_under_capture(H, W, n, K, nu):
    """No memory is taken then: the CTA-pair kernel runs, with the same bits; the next
    uncaptured iteration runs the launch form, or the halo-exchange kernel (the last
    two shapes)."""
    import torch
    import synth
    p = synth.make_problem("hsc", H=H, W=W, n=n, K=K, r=1, mask_frac=0.03, fwhm=(1.2, 2.5),
                           n_points=40, n_gal=3)
    x0 = np.full((H, W), 8.0, np.float32)
    d = emd.Deconvolver(H, W, n, K, 1)
    try:
        st = torch.cuda.Stream()
        emd.emd_set_stream(d.ctx, st)
        d.set_frames(p.y, p.v, p.f, p.mask)
        if nu > 0:
            d.set_noise(emd.EMD_NOISE_STUDENT_T, nu)
        d.set_x(x0)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=st):
            d.iterate(2)
        graph.replay()
        torch.cuda.synchronize()
        got = d.x()
        d.set_x(x0)
        d.iterate(2)
        np.testing.assert_array_equal(got, d.x())
    finally:
        d.close()
