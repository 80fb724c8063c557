"""The performance cases of the EM multi-frame deconvolution library: what its
users call, over the range of sizes, forms and noise models that they use.

A case's "op" is one of
  iterate   a loaded frame set: start, a number of EM iterations, result
            (emd_set_x, emd_iterate, emd_get_x)
  ingest    a new frame set: upload, weights and numerator, and the
            log-likelihood of a start (emd_set_frames, emd_set_x, emd_loglik)
  batch     a continuous batch of uneven jobs, stepped until all are done
            (emd_batch_add, emd_batch_step, emd_batch_sync, emd_get_x)
  fit_psf   super-resolved PSFs by Eq. (4) (emd_fit_psf)

Inputs are synthetic frame sets of the kind the repository's workloads use:
point and extended sources of lognormal flux, elliptical Moffat PSFs, a sky
level per exposure, photon-like variance, masked bad columns and cosmic rays
(their y is NaN). They are made on the GPU from the seed alone.
"""
import math

import numpy as np
import torch

from paper_2302_05804_gb300 import emd

FORMS = {"fp32": emd.EMD_PREC_FP32, "fft": emd.EMD_PREC_FFT_FP32,
         "split_bf16": emd.EMD_PREC_SPLIT_BF16}


def _iterate(name, H, W, n, K, r, form, iters, nu=0.0):
    c = dict(op="iterate", H=H, W=W, n=n, K=K, r=r, form=form, iters=iters, nu=nu)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest job of the serving range: a cut-out around one object
        _iterate("patch_128", 128, 128, 4, 15, 1, "fp32", 50),
        # the same kind of job in the FFT form, as the server runs it; ragged
        _iterate("patch_200x150_fft", 200, 150, 9, 21, 1, "fft", 50),
        # one detector's crop with the survey's depth and PSFs, odd sides
        _iterate("crop_1021x1009", 1021, 1009, 33, 43, 1, "fp32", 2),
        # a mid-range job of the serving range in the FFT form, odd sides
        _iterate("frames_1203x1021_fft", 1203, 1021, 22, 29, 1, "fft", 10),
        # robust deconvolution (satellite trails): heavy-tailed noise, FFT form
        _iterate("student_1024_fft", 1024, 1024, 20, 31, 1, "fft", 5, 3.0),
        # tensor-core form with the precision of the split products
        _iterate("split_bf16_2048", 2048, 2048, 33, 43, 1, "split_bf16", 1),
        # two-fold super-resolution of a full frame set, FFT form
        _iterate("sr2_2048_fft", 2048, 2048, 33, 85, 2, "fft", 1),
        # the full frame set of the paper (Fig. 1) in the default form ...
        _iterate("hsc_4096", 4096, 4096, 33, 43, 1, "fp32", 1),
        # ... and in the FFT form
        _iterate("hsc_4096_fft", 4096, 4096, 33, 43, 1, "fft", 2),
        # a new frame set arrives: weights, numerator, log-likelihood
        dict(name="ingest_1024", op="ingest", H=1024, W=1024, n=33, K=43, r=1),
        # the server's inner loop: uneven jobs, leaving the batch one by one
        dict(name="batch_12_fft", op="batch", jobs=12, smin=128, smax=900, nmin=4, nmax=24,
             kmin=15, kmax=43, iters=6, form="fft"),
        # the PSFs of a full frame set on a grid twice as fine
        dict(name="fit_psf_33", op="fit_psf", n=33, K=43, r=2, iters=300),
    ]


def _log_uniform(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    op = rng.choice(["iterate"] * 8 + ["ingest", "batch", "fit_psf"])
    if op == "fit_psf":
        return dict(op=op, n=_log_uniform(rng, 2, 40), K=2 * rng.randint(7, 21) + 1,
                    r=rng.choice([2, 2, 3]), iters=_log_uniform(rng, 50, 300))
    if op == "batch":
        smin = _log_uniform(rng, 100, 300)
        return dict(op=op, jobs=rng.randint(2, 16), smin=smin, smax=_log_uniform(rng, smin, 900),
                    nmin=4, nmax=rng.randint(5, 24), kmin=15, kmax=2 * rng.randint(8, 21) + 1,
                    iters=rng.randint(2, 8), form=rng.choice(["fft", "fft", "fp32"]))
    H = _log_uniform(rng, 120, 2500)
    W = min(4096, max(96, int(H * rng.uniform(0.6, 1.6))))
    n = rng.randint(4, 40)
    K = 2 * rng.randint(7, 21) + 1
    if op == "ingest":
        return dict(op=op, H=min(H, 1500), W=min(W, 1500), n=n, K=K, r=1)
    form = rng.choice(["fp32", "fp32", "fp32", "fft", "fft", "fft", "split_bf16"])
    r = 2 if rng.random() < 0.2 else 1
    nu = 0.0
    if form != "split_bf16" and rng.random() < 0.2:
        nu = rng.choice([2.0, 3.0, 5.0])
    if r == 2:
        K = 2 * K - 1  # the fine grid's PSF
        H, W = max(64, H // 2), max(64, W // 2)
    c = _iterate(None, H, W, n, K, r, form, 1, nu)
    # iterations: as many as keep the pass far below the largest listed one,
    # and in the split form few enough for 16-bit roundings not to pile up
    per = 4.0 * n * H * W * (K + r - 1) ** 2 * (1.5 if nu else 1.0)
    if form == "fft":
        per /= 12.0
    top = 2 if form == "split_bf16" else 50
    most = max(1, min(top, int(3e12 / per)))
    while per > 3.5e12:  # larger than a full frame set: fewer exposures
        n = max(1, n // 2)
        per /= 2.0
    c["n"], c["iters"] = n, _log_uniform(rng, 1, most)
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _good(m):
    """Smallest 2^a 3^b 5^c 7^d >= m (transform sizes)."""
    while True:
        q = m
        for p in (2, 3, 5, 7):
            while q % p == 0:
                q //= p
        if q == 1:
            return m
        m += 1


def _moffat(K, fwhm, beta, e, ang):
    """K x K elliptical Moffat profile of unit sum (float64, on the GPU)."""
    h = K // 2
    a = fwhm / (2.0 * math.sqrt(2.0 ** (1.0 / beta) - 1.0))
    g = torch.arange(-h, h + 1, dtype=torch.float64, device="cuda")
    yy, xx = g[:, None], g[None, :]
    u = math.cos(ang) * xx + math.sin(ang) * yy
    v = (-math.sin(ang) * xx + math.cos(ang) * yy) / (1.0 - e)
    p = (1.0 + (u * u + v * v) / (a * a)) ** (-beta)
    return p / p.sum()


class _Conv:
    """The zero-padded "same" convolution with K x K PSFs and its transpose
    on an H x W grid, in the given type, by whole-image FFTs."""

    def __init__(self, H, W, K, dtype):
        self.H, self.W, self.K, self.h, self.dtype = H, W, K, K // 2, dtype
        self.s = (_good(H + K - 1), _good(W + K - 1))

    def spectrum(self, a):
        return torch.fft.rfft2(a.to(self.dtype), s=self.s)

    def forward(self, xs, fs):
        z = torch.fft.irfft2(xs * fs, s=self.s)
        return z[self.h:self.h + self.H, self.h:self.h + self.W]

    def adjoint(self, ws, fs):
        z = torch.fft.irfft2(ws * fs.conj(), s=self.s)
        z = torch.roll(z, (self.h, self.h), (0, 1))
        return z[:self.H, :self.W]


def _down(z, r):
    return z if r == 1 else z.reshape(z.shape[0] // r, r, z.shape[1] // r, r).sum((1, 3))


def _up(w, r):
    return w if r == 1 else w.repeat_interleave(r, 0).repeat_interleave(r, 1)


def _psfs(n, K, r, rng):
    return torch.stack([_moffat(K, r * rng.uniform(3.0, 7.0), rng.uniform(2.5, 4.5),
                                rng.uniform(0.0, 0.15), rng.uniform(0.0, math.pi))
                        for _ in range(n)]).float()


def _frames(H, W, n, K, r, seed, trails=False):
    """(y, v, f, mask) of a synthetic frame set, on the GPU."""
    rng = np.random.default_rng([seed, H, W, n, K, r])
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(rng.integers(1 << 31)))
    Hf, Wf = r * H, r * W
    count = max(8, Hf * Wf // 840)
    sky = np.zeros((2, Hf, Wf))
    for k, m in ((0, count), (1, max(2, count // 10))):  # points, extended sources
        np.add.at(sky[k], (rng.integers(0, Hf, m), rng.integers(0, Wf, m)),
                  rng.lognormal(6.0, 1.5, m))
    sky = torch.from_numpy(sky.astype(np.float32)).cuda()
    f = _psfs(n, K, r, rng)
    conv = _Conv(Hf, Wf, K, torch.float32)
    kb = min(K, 31)
    blob = _Conv(Hf, Wf, kb, torch.float32)
    x = sky[0] + blob.forward(blob.spectrum(sky[1]), blob.spectrum(_moffat(kb, 8.0, 3.0, 0.1, 0.7)))
    xs = conv.spectrum(x.clamp_min(0.0))
    y = torch.empty((n, H, W), dtype=torch.float32, device="cuda")
    v = torch.empty_like(y)
    mask = torch.empty((n, H, W), dtype=torch.uint8, device="cuda")
    for t in range(n):
        z = _down(conv.forward(xs, conv.spectrum(f[t])), r)
        v[t] = rng.uniform(50.0, 400.0) + z.clamp_min(0.0)
        y[t] = z + v[t].sqrt() * torch.randn(z.shape, generator=gen, device="cuda")
        if trails:  # a bright trail across the exposure, not masked
            a, b = int(rng.integers(0, H)), float(rng.uniform(-1.0, 1.0))
            cols = torch.arange(W, device="cuda")
            rows = (a + (b * cols).long()) % H
            y[t, rows, cols] += 5000.0
        bad = torch.rand((H, W), generator=gen, device="cuda") < 0.004
        bad = torch.nn.functional.max_pool2d(bad.float()[None, None], 3, 1, 1)[0, 0] > 0
        for j in rng.integers(0, W, max(1, W // 100)):
            bad[:, int(j)] = True
        y[t][bad] = float("nan")
        mask[t] = (~bad).to(torch.uint8)
    return y, v, f, mask


def _broadening(r):
    """Normalised Gaussian of FWHM r pixels (odd side), float32."""
    sig = r / (2.0 * math.sqrt(2.0 * math.log(2.0)))
    k = int(math.ceil(3 * sig))
    a = np.arange(-k, k + 1)
    g = np.exp(-(a[:, None] ** 2 + a[None, :] ** 2) / (2 * sig * sig))
    return torch.from_numpy((g / g.sum()).astype(np.float32)).cuda()


def _jobs(case, seed):
    """(H, W, n, K, iterations) of a batch's jobs: sides log-uniform, one of
    each end of the range among them. The shapes are the case's own; the
    seed makes their inputs."""
    rng = np.random.default_rng([case["jobs"], case["smin"], case["smax"], case["nmax"]])
    out = []
    for j in range(case["jobs"]):
        if j < 2:
            S = (case["smin"], case["smax"])[j]
        else:
            S = int(round(math.exp(rng.uniform(math.log(case["smin"]), math.log(case["smax"])))))
        K = 2 * int(rng.integers(case["kmin"] // 2, case["kmax"] // 2 + 1)) + 1
        out.append((S, S + int(rng.integers(0, 9)), int(rng.integers(case["nmin"], case["nmax"] + 1)),
                    K, case["iters"] + int(rng.integers(0, 3))))
    return out


def _fit_inputs(case, seed):
    rng = np.random.default_rng([seed, case["n"], case["K"]])
    return _psfs(case["n"], case["K"], 1, rng), _broadening(case["r"])


_LAM, _LR = 1e-3, 1e-4  # Eq. (4)'s weight and the Adam step of the repository's benchmark


class _Batch:
    """A batch and its jobs' contexts, as the server holds them."""

    def __init__(self, jobs):
        self.batch, self.jobs = emd.emd_batch_create(jobs), []

    def __del__(self):
        emd.emd_batch_destroy(self.batch)
        for d, _, _, _ in self.jobs:
            d.close()


def prepare(case, seed):
    op = case["op"]
    if op == "fit_psf":
        f, g = _fit_inputs(case, seed)
        Kh = case["r"] * (case["K"] - 1) + 1
        return dict(op=op, f=f, g=g, r=case["r"], iters=case["iters"],
                    h=torch.empty((case["n"], Kh, Kh), dtype=torch.float32, device="cuda"),
                    loss=torch.empty(case["n"], dtype=torch.float32, device="cuda"))
    if op == "batch":
        b = _Batch(case["jobs"])
        for j, (H, W, n, K, iters) in enumerate(_jobs(case, seed)):
            d = emd.Deconvolver(H, W, n, K, 1)
            d.set_frames(*_frames(H, W, n, K, 1, seed + j))
            d.set_precision(FORMS[case["form"]])
            b.jobs.append((d, iters, torch.full((H, W), 5.0, device="cuda"),
                           torch.empty((H, W), device="cuda")))
        return dict(op=op, b=b)
    H, W, n, K, r = (case[k] for k in ("H", "W", "n", "K", "r"))
    d = emd.Deconvolver(H, W, n, K, r)
    x0 = torch.full((r * H, r * W), 5.0 / (r * r), device="cuda")
    if op == "ingest":
        return dict(op=op, d=d, frames=_frames(H, W, n, K, r, seed), x0=x0,
                    num=torch.empty((r * H, r * W), device="cuda"),
                    u=torch.empty((n, H, W), device="cuda"))
    d.set_frames(*_frames(H, W, n, K, r, seed, trails=case["nu"] > 0))
    d.set_precision(FORMS[case["form"]])
    if case["nu"] > 0:
        d.set_noise(emd.EMD_NOISE_STUDENT_T, case["nu"])
    return dict(op=op, d=d, x0=x0, iters=case["iters"], out=torch.empty_like(x0))


def run(state):
    op = state["op"]
    if op == "iterate":
        d = state["d"]
        d.set_x(state["x0"])
        d.iterate(state["iters"])
        return d.x(state["out"])
    if op == "ingest":
        d = state["d"]
        d.set_frames(*state["frames"])
        d.set_x(state["x0"])
        emd.emd_get_numerator(d.ctx, state["num"])
        emd.emd_get_weights(d.ctx, state["u"])
        ll, chi2 = d.loglik()
        return {"num": state["num"], "u": state["u"], "ll": ll, "chi2": chi2}
    if op == "batch":
        b = state["b"]
        slots = []
        for d, iters, x0, _ in b.jobs:
            d.set_x(x0)
            slots.append(emd.emd_batch_add(b.batch, d.ctx, iters))
        done = 0
        while done < len(b.jobs):
            done += emd.emd_batch_step(b.batch)
        emd.emd_batch_sync(b.batch)
        out = []
        for s, (d, _, _, x) in zip(slots, b.jobs):
            out.append(d.x(x))
            emd.emd_batch_remove(b.batch, s)
        return out
    return emd.emd_fit_psf(state["f"], state["g"], state["r"], _LAM, _LR, state["iters"],
                           h_out=state["h"], loss_out=state["loss"])


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _iterate_work(H, W, n, K, r, form, iters, nu=0.0):
    lat, exp = r * r * H * W, n * H * W
    passes = 3 if nu else 2  # forward model and adjoint; heavy-tailed: two adjoints
    if form == "fft":
        # whole-image transforms: per exposure one per operator, one of x and
        # one or two of the sums, and the products
        m = (r * H + K - 1) * (r * W + K - 1)
        flops = iters * (2.5 * m * math.log2(m) * (passes * n + passes) + 4.0 * m * passes * n)
    else:
        Kc = 2 * (((K - 1) // 2 + r - 1) // r) + 1
        flops = iters * passes * 2.0 * exp * r * r * Kc * Kc
    # u (heavy-tailed: and y) and N once per iteration, x in and out
    bytes_ = 4.0 * iters * (exp * (2 if nu else 1) + 3 * lat)
    return bytes_, flops


def work(case):
    op = case["op"]
    if op == "iterate":
        b, fl = _iterate_work(*(case[k] for k in ("H", "W", "n", "K", "r", "form", "iters", "nu")))
    elif op == "ingest":
        H, W, n, K = case["H"], case["W"], case["n"], case["K"]
        # y, v, mask in; u out and the kept y; N, x; one adjoint and one forward model
        b = 4.0 * n * H * W * 4 + n * H * W + 4.0 * 3 * H * W
        fl = 4.0 * n * H * W * K * K
    elif op == "batch":
        b = fl = 0.0
        for H, W, n, K, iters in _jobs(case, 0):
            bb, ff = _iterate_work(H, W, n, K, 1, case["form"], iters)
            b, fl = b + bb, fl + ff
    else:
        n, K, r = case["n"], case["K"], case["r"]
        Kh, Kg = r * (K - 1) + 1, _broadening_side(r)
        b = 4.0 * n * (K * K + Kh * Kh)
        fl = 4.0 * n * Kh * Kh * Kg * Kg * case["iters"]
    return {"bytes": b, "flops": fl}


def _broadening_side(r):
    return 2 * int(math.ceil(3 * r / (2.0 * math.sqrt(2.0 * math.log(2.0))))) + 1


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------

def _weights(y, v, mask):
    ok = mask != 0
    u = torch.where(ok, 1.0 / v.double(), torch.zeros((), dtype=torch.float64, device="cuda"))
    return u, torch.where(ok, y, torch.zeros((), device="cuda")).double()


def _em(frames, r, nu, iters, x0):
    y, v, f, mask = frames
    n, H, W = y.shape
    conv = _Conv(r * H, r * W, f.shape[1], torch.float64)
    hold = n * conv.s[0] * (conv.s[1] // 2 + 1) * 16 < 30e9
    fs = [conv.spectrum(f[t]) for t in range(n)] if hold else None

    def spec(t):
        return fs[t] if hold else conv.spectrum(f[t])

    def adjoint(w, t):
        return conv.adjoint(conv.spectrum(_up(w, r)), spec(t))

    num = None
    x = torch.full((r * H, r * W), x0, dtype=torch.float64, device="cuda")
    for _ in range(iters):
        xs = conv.spectrum(x)
        den, nt = torch.zeros_like(x), torch.zeros_like(x)
        for t in range(n):
            u, yt = _weights(y[t], v[t], mask[t])
            z = _down(conv.forward(xs, spec(t)), r)
            if nu:
                u = u * (nu + 1.0) / (nu + u * (yt - z) ** 2)
            den += adjoint(u * z, t)
            if nu or num is None:
                nt += adjoint(u * yt, t)
        if nu or num is None:
            num = nt
        ok = den > 1e-13 * den.max()
        x = torch.where(ok, x * num.clamp_min(0.0) / torch.where(ok, den, torch.ones_like(den)), x)
    return x


def _fit(f, g, r, lam, lr, iters):
    """Projected Adam on Eq. (4) for all PSFs, returning the iterate of
    lowest loss and that loss."""
    f, g = f.double(), g.double()
    n, K, _ = f.shape
    Kh, hg = r * (K - 1) + 1, g.shape[0] // 2
    pad = r * K - Kh
    taps = [(a, b, g[a, b].item()) for a in range(2 * hg + 1) for b in range(2 * hg + 1)]

    def shifted(h, sign):
        hp = torch.nn.functional.pad(h, (hg, hg, hg, hg))
        out = torch.zeros_like(h)
        for a, b, w in taps:  # convolution (sign +1) or correlation (-1)
            i, j = (2 * hg - a, 2 * hg - b) if sign > 0 else (a, b)
            out += w * hp[:, i:i + Kh, j:j + Kh]
        return out

    h = f.repeat_interleave(r, 1).repeat_interleave(r, 2)[:, :Kh, :Kh] / (r * r)
    m, v = torch.zeros_like(h), torch.zeros_like(h)
    best, bh = None, h.clone()
    for k in range(iters + 1):
        q = torch.nn.functional.pad(shifted(h, 1), (0, pad, 0, pad))
        res = q.reshape(n, K, r, K, r).sum((2, 4)) - f
        dy, dx = h[:, 1:] - h[:, :-1], h[:, :, 1:] - h[:, :, :-1]
        loss = res.square().sum((1, 2)) + lam * (dy.square().sum((1, 2)) + dx.square().sum((1, 2)))
        if best is None:
            best = loss.clone()
        better = loss < best
        best = torch.where(better, loss, best)
        bh = torch.where(better[:, None, None], h, bh)
        if k == iters:
            break
        rep = res.repeat_interleave(r, 1).repeat_interleave(r, 2)[:, :Kh, :Kh]
        gr = 2.0 * shifted(rep, -1)
        gr[:, 1:] += 2.0 * lam * dy
        gr[:, :-1] -= 2.0 * lam * dy
        gr[:, :, 1:] += 2.0 * lam * dx
        gr[:, :, :-1] -= 2.0 * lam * dx
        m = 0.9 * m + 0.1 * gr
        v = 0.999 * v + 0.001 * gr * gr
        step = (m / (1.0 - 0.9 ** (k + 1))) / ((v / (1.0 - 0.999 ** (k + 1))).sqrt() + 1e-8)
        h = (h - lr * step).clamp_min(0.0)
    return bh, best


def exact(case, seed):
    op = case["op"]
    if op == "fit_psf":
        f, g = _fit_inputs(case, seed)
        return _fit(f, g, case["r"], _LAM, _LR, case["iters"])
    if op == "batch":
        return [_em(_frames(H, W, n, K, 1, seed + j), 1, 0.0, iters, 5.0)
                for j, (H, W, n, K, iters) in enumerate(_jobs(case, seed))]
    H, W, n, K, r = (case[k] for k in ("H", "W", "n", "K", "r"))
    if op == "iterate":
        frames = _frames(H, W, n, K, r, seed, trails=case["nu"] > 0)
        return _em(frames, r, case["nu"], case["iters"], 5.0 / (r * r))
    y, v, f, mask = _frames(H, W, n, K, r, seed)
    conv = _Conv(H, W, K, torch.float64)
    xs = conv.spectrum(torch.full((H, W), 5.0, dtype=torch.float64, device="cuda"))
    num = torch.zeros((H, W), dtype=torch.float64, device="cuda")
    us = torch.empty((n, H, W), dtype=torch.float64, device="cuda")
    chi2 = logdet = 0.0
    for t in range(n):
        u, yt = _weights(y[t], v[t], mask[t])
        us[t] = u
        fs = conv.spectrum(f[t])
        num += conv.adjoint(conv.spectrum(u * yt), fs)
        chi2 += (u * (yt - conv.forward(xs, fs)) ** 2).sum().item()
        logdet += (v[t].double()[mask[t] != 0] * (2.0 * math.pi)).log().sum().item()
    return {"num": num, "u": us, "ll": -0.5 * (chi2 + logdet), "chi2": chi2}
