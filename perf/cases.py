"""Timed cases of the deconvolution sampler: what its users run, through the
package's public entry points (``bdecon.Sampler``, ``bdecon.Server``).

Every case is seeded synthetic microscopy data of the recipes this repository
uses everywhere else (filaments and blobs, Gaussian PSF on 2 ceil(3 sigma) + 1
pixels, Poisson photons, camera scalars or sCMOS maps).  The kinds of call:

  resume       a handle in hand, a checkpointed object from the host, a segment
               of sweeps, and the segment's mean, trace and final object back --
               a chain that is run on and on in segments (exact resume).  With
               ``burn`` > 0 the checkpoint is the object after that many sweeps
               (the state a long chain spends its life in: few acceptances),
               with 0 an object near the start of a chain (many acceptances)
  advance      a handle in hand whose chains simply go on: a segment of sweeps
               of every chain, then the running mean and the traces
  job          the whole call from host buffers: create (one frame or a batch),
               sweep, the posterior mean of every frame, close
  serve        jobs of mixed sizes through the running serving loop
  uncertainty  quantile, standard-deviation and coefficient-of-variation maps
               of a finished chain's kept objects
  evaluate     the Eq. 9 log posterior and the expected image of a given object
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2411_00991_gb300 import bdecon, synth

QUANTILES = (0.05, 0.25, 0.5, 0.75, 0.95)


def _case(name, kind, H, W, sigma, L, chains=1, double=False, augmented=False, sub=1, maps=True, peak=50.0,
          sweeps=1, refresh=50, burn=0):
    return dict(name=name, kind=kind, H=H, W=W, sigma=sigma, L=L, chains=chains, double=double, augmented=augmented,
                sub=sub, maps=maps, peak=peak, sweeps=sweeps, refresh=refresh, burn=burn)


def listed():
    return [
        # a few-patch ragged region of interest, the smallest call: launches, copies and step latency
        _case("roi_24x20_L5", "resume", 20, 24, 1.0, 5, maps=False, peak=20.0, sweeps=20, burn=20),
        # the 64 x 64 camera-scalar frame deconvolved from start to end, 200 sweeps, from host buffers to the mean
        _case("job_64_L9", "job", 64, 64, 1.5, 9, maps=False, peak=20.0, sweeps=200),
        # the same frame's first sweeps in the plain double sampler (the reference chain, validation runs)
        _case("fp64_64_L9", "resume", 64, 64, 1.5, 9, double=True, maps=False, peak=20.0, sweeps=10),
        # a ragged frame in the double sampler past its first sweeps
        _case("fp64_250x203_L17", "resume", 250, 203, 1.2, 17, double=True, sweeps=3, burn=60),
        # the 512 x 512 sCMOS frame (NA 1.4 widefield) in the middle of a long chain: the interactive workload
        _case("widefield_512_L17", "resume", 512, 512, 1.2, 17, sweeps=50, burn=150),
        # the same frame in the photon-count augmented sampler
        _case("augmented_512_L17", "resume", 512, 512, 1.2, 17, augmented=True, sweeps=30, burn=60),
        # a 150 x 150 inset on an object lattice twice as fine as the camera (Nyquist lattice)
        _case("inset_150_sub2_L13", "resume", 150, 150, 2.0, 13, sub=2, sweeps=20, burn=20),
        # the 2048 x 2048 low-SNR frame, wide PSF, 4 chains: the largest single problem, state beyond L2
        _case("lowsnr_2048_L31", "advance", 2048, 2048, 4.0, 31, chains=4, peak=5.0, sweeps=2, burn=4),
        # a batch of uneven frames x 4 chains from host buffers to means (the batched production form)
        dict(name="batch_uneven_x4", kind="job", sides="128,256,384,512,512,768", sigmas="1.2,3.6,2.1,1.4,2.6,3.5",
             chains=4, double=False, sweeps=10, refresh=10, peak=40.0),
        # four single-chain jobs of mixed sizes arriving together at the serving loop
        dict(name="serve_4_jobs", kind="serve", sides="160,256,352,640", sigmas="1.1,2.4,1.6,3.1", sweeps=60,
             refresh=50, peak=50.0),
        # uncertainty maps from the 100 kept objects of a 512 x 512 chain
        _case("uncertainty_512", "uncertainty", 512, 512, 1.2, 17, sweeps=100),
        # scoring a given object of a wide-PSF frame (model checks, traces of external reconstructions)
        _case("evaluate_1024_L25", "evaluate", 1024, 1024, 4.0, 25, peak=100.0),
    ]


def _psf_side(sigma):
    return 2 * int(math.ceil(3 * sigma)) + 1


def draw(rng):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["resume"] * 4 + ["advance"] * 3 + ["job"] * 2 + ["batch"] * 2 + ["serve", "uncertainty", "evaluate"])
    budget = 8.0e9                        # window cells scored: below the largest listed case's
    if kind in ("batch", "serve"):
        n = rng.randint(2, 6)
        sides = [logint(40, 640) for _ in range(n)]
        sigmas = [round(rng.uniform(1.0, 4.0), 2) for _ in range(n)]
        chains = rng.randint(1, 4) if kind == "batch" else 1
        cells = sum(s * s * _psf_side(g) ** 2 for s, g in zip(sides, sigmas)) * chains
        sweeps = max(2, min(60, int(budget / cells)))
        c = dict(kind="job" if kind == "batch" else "serve", sides=",".join(map(str, sides)),
                 sigmas=",".join(map(str, sigmas)), sweeps=sweeps, refresh=rng.choice([10, 50]),
                 peak=round(math.exp(rng.uniform(math.log(3), math.log(200))), 1))
        if kind == "batch":
            c.update(chains=chains, double=False)
        return c
    double = kind in ("resume", "job") and rng.random() < 0.25
    augmented = kind in ("resume", "advance") and rng.random() < 0.25
    sub = 2 if kind == "resume" and rng.random() < 0.25 else 1
    hi = {"evaluate": 1400, "uncertainty": 600, "advance": 1400}.get(kind, 700)
    if sub > 1:
        hi = 300
    if double:
        hi = 220
    H = logint(400 if kind == "advance" else 20, hi)
    W = min(hi, max(20, int(round(H * rng.uniform(0.6, 1.6)))))
    sigma = round(rng.uniform(0.8, 4.0 if not double else 2.5), 2)
    L = _psf_side(sigma)
    chains = rng.randint(2, 4) if kind == "advance" else rng.choice([1, 1, 2]) if kind == "job" else 1
    cells = H * W * sub * sub * chains * L * L
    if kind == "advance":
        sweeps = max(2, min(100, int(budget / 3 / cells)))
    elif kind == "uncertainty":
        sweeps = max(10, min(120, int(budget / cells)))
    elif kind == "evaluate":
        sweeps = 1
    else:
        sweeps = max(1, min(20 if sub > 1 else 100, int((budget / 60 if double else budget / 4) / cells)))
    return dict(kind=kind, H=H, W=W, sigma=sigma, L=L, chains=chains, double=double, augmented=augmented, sub=sub,
                maps=rng.random() < 0.6, peak=round(math.exp(rng.uniform(math.log(3), math.log(200))), 1),
                sweeps=sweeps, refresh=rng.choice([10, 50]),
                burn=rng.choice([0, 20]) if sub > 1 else rng.choice([0, 20, 60]) if kind in ("resume", "advance") and not double else 0)


# ----------------------------------------------------------------- inputs --
def _truth(shape, peak, rng):
    """Filaments (one-pixel direction random walks) and blobs on background 1,
    at the density of the 512 x 512 recipe, built with array operations."""
    Hh, Ww = shape
    frac = Hh * Ww / 512.0 ** 2
    out = np.zeros(shape)
    n, length = max(1, int(round(200 * frac))), 200
    th = rng.uniform(0, 2 * math.pi, (n, 1)) + np.cumsum(rng.normal(0.0, 0.08, (n, length)), axis=1)
    y = rng.uniform(0, Hh, (n, 1)) + np.cumsum(np.sin(th), axis=1)
    x = rng.uniform(0, Ww, (n, 1)) + np.cumsum(np.cos(th), axis=1)
    keep = (np.arange(length)[None, :] < rng.uniform(20, 200, (n, 1))) & (y >= 0) & (y < Hh) & (x >= 0) & (x < Ww)
    out[y[keep].astype(int), x[keep].astype(int)] = 1.0
    for _ in range(max(1, int(round(50 * frac)))):
        cy, cx, s, a = rng.uniform(0, Hh), rng.uniform(0, Ww), rng.uniform(1.0, 3.0), rng.uniform(0.3, 1.0)
        r = int(math.ceil(4 * s))
        y0, y1, x0, x1 = max(0, int(cy) - r), min(Hh, int(cy) + r + 1), max(0, int(cx) - r), min(Ww, int(cx) + r + 1)
        gy = np.exp(-(np.arange(y0, y1) - cy) ** 2 / (2 * s * s))
        gx = np.exp(-(np.arange(x0, x1) - cx) ** 2 / (2 * s * s))
        out[y0:y1, x0:x1] += a * np.outer(gy, gx)
    return 1.0 + out * ((peak - 1.0) / out.max())


def _problem(H, W, sigma, L, seed, chains=1, augmented=False, sub=1, maps=True, peak=50.0, refresh=50, burn_in=0,
             n_samples=0):
    rng = np.random.default_rng(seed)
    R = L // 2
    truth = _truth((sub * H + 2 * R, sub * W + 2 * R), peak, rng) / (sub * sub)
    psf = synth.gaussian_psf(sigma, L)
    if maps:
        off, var = synth.scmos_maps(H, W, rng)
        gain = 2.1
    else:
        off, var, gain = 100.0, 2.56, 2.0
    image = synth.simulate_frame(truth, psf, gain, off, var, rng, subpixel=sub)
    return synth.Problem(image=image, psf=psf, gain=gain, offset=off, var=var, n_chains=chains, seed=seed, burn_in=burn_in,
                         refresh_every=refresh, n_samples=n_samples, augmented=augmented, subpixel=sub)


def _of_case(case, seed, **more):
    return _problem(case["H"], case["W"], case["sigma"], case["L"], seed, chains=case["chains"],
                    augmented=case["augmented"], sub=case["sub"], maps=case["maps"], peak=case["peak"],
                    refresh=case["refresh"], **more)


def _many(case, seed):
    """Frames of a batch or of serving jobs: sides and PSF sigmas from the case."""
    sides, sigmas = [int(v) for v in case["sides"].split(",")], [float(v) for v in case["sigmas"].split(",")]
    return [_problem(s, s, g, _psf_side(g), seed + 7919 * k, chains=case.get("chains", 1), maps=case["kind"] == "serve",
                     peak=case["peak"], refresh=case["refresh"]) for k, (s, g) in enumerate(zip(sides, sigmas))]


def _start_object(prob, seed):
    """A positive object near the frame's mean level, as a chain has it in its
    first sweeps; every value exact in float."""
    rng = np.random.default_rng(seed + 101)
    g, o, _ = prob.maps()
    level = max(0.1, float(((prob.image - o) / g).mean())) / prob.subpixel ** 2
    return (level * np.exp(0.1 * rng.standard_normal(prob.object_shape()))).astype(np.float32).astype(np.float64)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "serve":
        jobs = _many(case, seed)
        return dict(kind=kind, jobs=jobs, sweeps=case["sweeps"],
                    server=bdecon.Server(mem_budget=16 << 30, max_jobs=16, segment_sweeps=20))
    precision = bdecon.BDECON_FP64 if case["double"] else bdecon.BDECON_FP32
    if kind == "job":
        probs = _many(case, seed) if "sides" in case else [_of_case(case, seed)]
        return dict(kind=kind, probs=probs, precision=precision, sweeps=case["sweeps"])
    stream = torch.cuda.current_stream().cuda_stream
    if kind == "uncertainty":
        prob = _of_case(case, seed, n_samples=case["sweeps"])
        s = bdecon.Sampler(prob, precision=precision, max_sweeps=case["sweeps"] + 8, flags=bdecon.FLAG_SECOND_MOMENT,
                           stream=stream)
        s.sweep(case["sweeps"])
        s.sync()
        return dict(kind=kind, sampler=s)
    prob = _of_case(case, seed)
    if kind == "evaluate":
        return dict(kind=kind, sampler=bdecon.Sampler(prob, precision=precision, max_sweeps=8, stream=stream),
                    rho=_start_object(prob, seed))
    if kind == "advance":
        s = bdecon.Sampler(prob, precision=precision, max_sweeps=1 << 17, stream=stream)
        s.sweep(case["burn"])
        s.sync()
        return dict(kind=kind, sampler=s, sweeps=case["sweeps"])
    # resume: the checkpoint of a chain after `burn` sweeps (float sweeps reach it sooner), or a first object
    rho, done = _start_object(prob, seed), 0
    if case["burn"]:
        b = bdecon.Sampler(prob, precision=bdecon.BDECON_FP32, max_sweeps=case["burn"] + 8, stream=stream)
        b.sweep(case["burn"])
        rho, done = b.get_state()
        b.close()
    s = bdecon.Sampler(prob, precision=precision, max_sweeps=done + case["sweeps"] + 8, stream=stream)
    return dict(kind=kind, sampler=s, rho=rho, done=done, sweeps=case["sweeps"])


# -------------------------------------------------------------------- run --
def run(state):
    kind, s = state["kind"], state.get("sampler")
    if kind == "resume":
        s.set_state(state["rho"], state["done"])
        s.sweep(state["sweeps"])
        return dict(mean=s.posterior_mean(), trace=s.trace()[state["done"]:], rho=s.get_state()[0])
    if kind == "advance":
        s.sweep(state["sweeps"])
        n = s.problems[0].n_chains
        return dict(mean=s.posterior_mean(), trace=[s.trace(0, c)[-state["sweeps"]:] for c in range(n)],
                    accepted=[s.accept_counts(0, c)[-state["sweeps"]:] for c in range(n)])
    if kind == "job":
        s = bdecon.Sampler(state["probs"], precision=state["precision"], max_sweeps=state["sweeps"],
                           stream=torch.cuda.current_stream().cuda_stream)
        s.sweep(state["sweeps"])
        out = [s.posterior_mean(p) for p in range(len(state["probs"]))]
        out += [s.trace(p) for p in range(len(state["probs"]))]
        s.close()
        return out
    if kind == "serve":
        ids = [state["server"].submit(q, state["sweeps"]) for q in state["jobs"]]
        return [state["server"].result(i)[0] for i in ids]
    if kind == "uncertainty":
        return dict(quantiles=s.posterior_quantiles(QUANTILES), std=s.posterior_std(), cv=s.posterior_cv())
    s.set_state(state["rho"], 0)
    return dict(log_posterior=s.log_posterior(), mu=s.get_mu())


# ------------------------------------------------------------------- work --
def _update_work(H, W, L, S, sub, chains, sweeps, refresh, double, peak):
    """Operations and bytes of the sweeps: per pixel update L_c^2 window cells
    at 4 operations per photon count that matters (about 8 sigma of the photon
    posterior) + 10, and 12 per patch-spectrum entry; per sweep and pixel the
    object, expected image, its derived per-pixel values, the spectrum and the
    running mean once; per refresh the convolution."""
    Lc = (L + sub - 2) // sub + 1
    R = L // 2
    obj = (sub * H + 2 * R) * (sub * W + 2 * R) * chains
    terms = 4.0 + 2.0 * math.sqrt(min(peak, 10.0))
    flops = obj * sweeps * (Lc * Lc * (4 * terms + 10) + 12.0 * S * S)
    flops += (sweeps // refresh if refresh else 0) * chains * H * W * 2.0 * (L + sub - 1) ** 2
    return flops, obj * sweeps * 68.0 * (2 if double else 1)


def work(case):
    kind = case["kind"]
    if "sides" in case:
        flops = nbytes = 0.0
        for s, g in zip(case["sides"].split(","), case["sigmas"].split(",")):
            s, L = int(s), _psf_side(float(g))
            f, b = _update_work(s, s, L, L, 1, case.get("chains", 1), case["sweeps"], case["refresh"], False, case["peak"])
            flops, nbytes = flops + f, nbytes + b
        return dict(bytes=nbytes, flops=flops)
    H, W, L, sub = case["H"], case["W"], case["L"], case["sub"]
    obj = (sub * H + L - 1) * (sub * W + L - 1)
    if kind == "uncertainty":
        n = case["sweeps"]
        return dict(bytes=obj * (4.0 * n + 16.0 + 8.0 * (len(QUANTILES) + 2)), flops=obj * n * math.log2(max(2, n)))
    if kind == "evaluate":
        # the object in, the expected image out; the convolution, the photon sums and the patch transforms
        terms = 6.0 + 6.0 * math.sqrt(case["peak"] / 4)
        return dict(bytes=8.0 * obj + H * W * (12.0 + 8.0), flops=H * W * (2.0 * L * L + 6 * terms) + obj * 16.0 * L)
    flops, nbytes = _update_work(H, W, L, L + sub - 1, sub, case["chains"], case["sweeps"], case["refresh"], case["double"],
                                 case["peak"])
    return dict(bytes=nbytes, flops=flops)


# ------------------------------------------------------------------ exact --
class _Model:
    """The model in 64 bits with plain torch: Eq. 1-2 expected image, Eq. 6
    likelihood by a log-sum-exp over photon counts, Eq. 7-8 patch prior (all
    frequencies, without the constant log B(alpha))."""

    def __init__(self, prob, device):
        t = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=device)  # noqa: E731
        self.dev, self.S, self.L, self.R = device, prob.S, prob.L, prob.L // 2
        g, o, v = prob.maps()
        self.c, self.s2, self.var = t((prob.image.astype(np.float64) - o) / g), t(v / g ** 2), t(v)
        self.K = t(prob.psf / prob.psf.sum())
        self.Ho, self.Wo = prob.object_shape()
        self.H, self.W = prob.H, prob.W
        cap = float(self.c.max())
        self.n_phi = int(1.3 * max(cap, 1.0) + 12 * math.sqrt(max(cap, 1.0)) + 60)
        # patches by shape: top-left corners, sides, exponents alpha - 1
        self.groups = []
        S = self.S
        for i0s, ph in self._runs(self.Ho):
            for j0s, pw in self._runs(self.Wo):
                kw = torch.zeros(ph, pw, dtype=torch.float64, device=device)
                for p in range(self.L):
                    for q in range(self.L):
                        kw[(p - self.R) % ph, (q - self.R) % pw] += self.K[p, q]
                mag = torch.fft.fft2(kw).abs()
                corners = torch.tensor([(i, j) for i in i0s for j in j0s], device=device)
                self.groups.append(dict(i0=corners[:, 0], j0=corners[:, 1], ph=ph, pw=pw, a1=mag / mag.sum() - 1.0))

    def _runs(self, n):
        full = n // self.S
        out = [([k * self.S for k in range(full)], self.S)] if full else []
        return out + ([([full * self.S], n - full * self.S)] if n % self.S else [])

    def loglik(self, mu, c, s2, var):
        """log sum_phi Normal(c; phi, s2) Poisson(phi; mu) up to the Jacobian of Eq. 4, elementwise."""
        lmu = mu.log()
        m = torch.full_like(mu, -math.inf)
        acc = torch.zeros_like(mu)
        for phi in range(self.n_phi):
            lt = -(c - phi) ** 2 / (2 * s2) + phi * lmu - math.lgamma(phi + 1.0)
            n = torch.maximum(m, lt)
            acc = acc * (m - n).exp() + (lt - n).exp()
            m = n
        return m + acc.log() - mu - 0.5 * (2 * math.pi * var).log()

    def expected(self, rho):
        w = self.K.flip(0, 1)
        out = torch.zeros(self.H, self.W, dtype=torch.float64, device=self.dev)
        for p in range(self.L):
            for q in range(self.L):
                out += w[p, q] * rho[p:p + self.H, q:q + self.W]
        return out

    def prior_of(self, X, a1):
        m = X.abs()
        return (a1 * m.log()).sum((-2, -1)) + (a1.numel() - 1) * m.sum((-2, -1)).log()

    def patches(self, rho, grp):
        u, v = torch.arange(grp["ph"], device=self.dev), torch.arange(grp["pw"], device=self.dev)
        return rho[(grp["i0"][:, None, None] + u[None, :, None]), (grp["j0"][:, None, None] + v[None, None, :])]

    def log_posterior(self, rho, mu):
        tot = self.loglik(mu, self.c, self.s2, self.var).sum()
        for grp in self.groups:
            tot = tot + self.prior_of(torch.fft.fft2(self.patches(rho, grp)), grp["a1"]).sum()
        return float(tot)

    def window_loglik(self, mu, idx):
        """l(mu) of gathered cells: the photon counts as one axis, in chunks."""
        c, s2 = self.c.view(-1)[idx], self.s2.view(-1)[idx]
        phi = torch.arange(self.n_phi, dtype=torch.float64, device=self.dev)
        lt = -(c[..., None] - phi) ** 2 / (2 * s2[..., None]) + phi * mu.clamp_min(1e-300).log()[..., None] - torch.lgamma(phi + 1)
        return torch.logsumexp(lt, -1) - mu


def _philox(m, t, chain, seed):
    """Philox4x32-10 of the counters (m, t, chain, 0) under key `seed` (Salmon et al., SC'11)."""
    mask = np.uint64(0xFFFFFFFF)
    c = [m.astype(np.uint64), np.full(m.shape, t, np.uint64), np.full(m.shape, chain, np.uint64), np.zeros(m.shape, np.uint64)]
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    for _ in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & mask, (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), p0 & mask]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c


def _exact_chain(prob, rho, t0, sweeps, device):
    """The sampler's chain in 64 bits: per class one Metropolis-Hastings step
    of every patch's pixel, all of a class at once."""
    M = _Model(prob, device)
    rho = torch.as_tensor(rho, dtype=torch.float64, device=device).clone()
    mu = M.expected(rho)
    base = M.log_posterior(rho, mu)
    total, trace = torch.zeros_like(rho), []
    n = M.Ho * M.Wo
    k = torch.arange(M.L, device=device)
    for grp in M.groups:
        grp["X"] = torch.fft.fft2(M.patches(rho, grp))
        fh, fw = torch.arange(grp["ph"], device=device), torch.arange(grp["pw"], device=device)
        grp["eh"] = torch.exp(-2j * math.pi * (fh[:, None] * fh[None, :] % grp["ph"]).double() / grp["ph"])
        grp["ew"] = torch.exp(-2j * math.pi * (fw[:, None] * fw[None, :] % grp["pw"]).double() / grp["pw"])
    for t in range(t0 + 1, t0 + sweeps + 1):
        x = _philox(np.arange(n), t, 0, prob.seed)
        u = [((v >> np.uint64(9)).astype(np.float64) + 0.5) * 2.0 ** -23 for v in x[:3]]
        hz = torch.as_tensor(prob.step * np.sqrt(-2 * np.log(u[0])) * np.cos(2 * np.pi * u[1]), device=device).view(M.Ho, M.Wo)
        lu = torch.as_tensor(np.log(u[2]), device=device).view(M.Ho, M.Wo)
        gain = torch.zeros((), dtype=torch.float64, device=device)
        for a in range(M.S):
            for b in range(M.S):
                for grp in M.groups:
                    if a >= grp["ph"] or b >= grp["pw"]:
                        continue
                    i, j = grp["i0"] + a, grp["j0"] + b
                    old = rho[i, j]
                    new = old * hz[i, j].exp()
                    d = new - old
                    aa, bb = i[:, None, None] - 2 * M.R + k[None, :, None], j[:, None, None] - 2 * M.R + k[None, None, :]
                    ok = (aa >= 0) & (aa < M.H) & (bb >= 0) & (bb < M.W)
                    idx = torch.where(ok, aa * M.W + bb, 0)
                    m0 = mu.view(-1)[idx]
                    m1 = m0 + d[:, None, None] * M.K
                    dl = torch.where(ok, M.window_loglik(m1, idx) - M.window_loglik(m0, idx), 0.0).sum((1, 2))
                    X1 = grp["X"] + d[:, None, None] * (grp["eh"][:, a, None] * grp["ew"][None, :, b])
                    dp = M.prior_of(X1, grp["a1"]) - M.prior_of(grp["X"], grp["a1"])
                    bad = (ok & (m1 <= 0)).any(2).any(1)
                    acc = (lu[i, j] < dl + dp + hz[i, j]) & ~bad
                    rho[i, j] = torch.where(acc, new, old)
                    put = ok & acc[:, None, None]
                    mu.view(-1)[idx[put]] = m1[put]
                    grp["X"] = torch.where(acc[:, None, None], X1, grp["X"])
                    gain = gain + torch.where(acc, dl + dp, 0.0).sum()
        base = base + float(gain)
        trace.append(base)
        total += rho
    return (total / sweeps).cpu().numpy(), np.array(trace), rho.cpu().numpy()


def exact(case, seed):
    """64-bit values of the same inputs.  A float chain has none: it parts
    from the 64-bit chain at the first accept decision that rounding turns, and
    from there is another (equally valid) chain.  Nor has a state that the
    case reaches by sampling."""
    if case["kind"] == "evaluate":
        prob = _of_case(case, seed)
        dev = torch.device("cuda")
        M = _Model(prob, dev)
        rho = torch.as_tensor(_start_object(prob, seed), device=dev)
        mu = M.expected(rho)
        return dict(log_posterior=M.log_posterior(rho, mu), mu=mu.cpu().numpy())
    if case["kind"] == "resume" and case["double"] and not case["burn"] and not case["augmented"] and case["sub"] == 1:
        prob = _of_case(case, seed)
        cells = (case["H"] + case["L"]) * (case["W"] + case["L"]) * case["L"] ** 2 * case["sweeps"]
        steps = case["L"] ** 2 * case["sweeps"]
        if cells * (1.5 * case["peak"] + 60) > 2.0e11 or steps > 4000 or case["sweeps"] > case["refresh"]:
            return None
        mean, trace, rho = _exact_chain(prob, _start_object(prob, seed), 0, case["sweeps"], torch.device("cuda"))
        return dict(mean=mean, trace=trace, rho=rho)
    return None
