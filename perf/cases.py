"""Timed work of the framework: the calls a user's program makes, over the
range of sizes they are made with.

``listed()`` names the cases, ``draw(rng)`` gives more of the same ranges,
``prepare(case, seed)`` makes what a program has in hand before the call (the
light curves, the maps and events resident on the device, the starts of a
refinement), ``run(state)`` makes the call and returns its whole result,
``work(case)`` states the bytes and operations the call cannot do without, and
``exact(case, seed)`` computes the same result in 64 bits with torch alone.

Light curves are shaped like survey-plus-follow-up data: 8-hour nightly
windows over [-40, 40] d, denser about the peak, magnification of a binary
lens (point source, from the lens polynomial), F = Fs A + Fb with noise
sigma = 0.01 sqrt(F) + 0.002 and, where stated, 1 % outliers of 5 sigma.
Truths: u0 log-uniform in [1e-3, 0.5], alpha uniform, tE log-uniform in
[5, 80] d, Fb / Fs uniform in [0, 2].
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1511_01157_gb300 as morse

L = 2.0          # maps cover [-2, 2]^2 Einstein radii
X = 3.0          # rays cover [-3, 3]^2
GAMMA = 0.53     # limb darkening of the finite-source maps


# ------------------------------------------------------------------ cases
def listed():
    return [
        # the smallest call: a small grid through a resident 512^2 map for a
        # sparse survey light curve, as a program that looks about a
        # candidate lens makes it many times in a row
        dict(name="grid_local", kind="grid", s=1.0, q=1e-3, npix=512,
             rays=4000, n_ep=201, outliers=0.0, fp16=False, n_u0=6,
             n_alpha=24, n_t0=5, n_tE=5, top_k=16),
        # one map for one event from host buffers to fits: 500 epochs, a
        # 512^2 map of 4000^2 FP64 rays, 72 000 trajectories
        dict(name="one_map", kind="search", s=1.0, q=1e-3, npix=512,
             rays=4000, n_ep=500, outliers=0.0, deflect="fp64", n_u0=20,
             n_alpha=36, n_t0=10, n_tE=10, top_k=16),
        # the full trajectory grid of a 3000-epoch event on one resident map
        dict(name="grid_full", kind="grid", s=0.9, q=5e-4, npix=1024,
             rays=10000, n_ep=3000, outliers=0.01, fp16=False, n_u0=40,
             n_alpha=72, n_t0=25, n_tE=20, top_k=256),
        # the (s, q) search: maps built and searched one after another
        dict(name="sweep", kind="sweep", n_maps=4, npix=1024, rays=10000,
             n_ep=3000, outliers=0.01, fp16=False, n_u0=40, n_alpha=72,
             n_t0=25, n_tE=20, top_k=256),
        # the largest maps: 4096^2 of 1.6e9 rays near resonance, searched
        # through their FP16 tables; a ragged count of epochs
        dict(name="sweep_fp16_4096", kind="sweep", n_maps=2, npix=4096,
             rays=40000, n_ep=4999, outliers=0.0, fp16=True, n_u0=25,
             n_alpha=40, n_t0=20, n_tE=10, top_k=16),
        # many light curves of uneven length against a bank of maps
        dict(name="batch", kind="batch", n_events=12, len_lo=200,
             len_hi=20000, n_maps=4, npix=1024, rays=10000, n_u0=25,
             n_alpha=40, n_t0=20, n_tE=10, top_k=16),
        # a training step through the autograd function: chi^2 and gradient
        # of 4096 trajectories
        dict(name="grad", kind="grad", s=0.9, q=5e-4, npix=1024, rays=10000,
             n_ep=3000, outliers=0.01, n=4096),
        # refinement of grid minima that lie on several maps, an odd count
        dict(name="refine", kind="refine", n_maps=16, npix=1024, rays=10000,
             n_ep=3000, outliers=0.01, n=2047, iters=50),
        # peak libraries of a slice of the (s, q) grid
        dict(name="peaks", kind="peaks", n_maps=16, npix=1024, rays=10000,
             n_u0=40, n_alpha=72, sub=2, max_peaks=8, delta=0.1),
        # the search of the trajectories whose peaks come at the observed
        # peak time
        dict(name="aligned", kind="aligned", s=0.9, q=5e-4, npix=1024,
             rays=10000, n_ep=3000, outliers=0.01, n_u0=40, n_alpha=72,
             n_t0=3, n_tE=20, max_peaks=2, delta=0.1, top_k=16),
        # the point-source map of one lens by the polynomial, to host
        dict(name="map_poly", kind="poly", s=0.9, q=5e-4, npix=1024),
        # a finite-source map (a giant's radius), to host
        dict(name="finite", kind="finite", s=0.9, q=5e-4, npix=1024,
             rays=10000, rho=0.3),
    ]


def _logu(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _logi(rng, lo, hi):
    return int(round(_logu(rng, lo, hi)))


def _lens(rng):
    return dict(s=_logu(rng, 0.3, 3.0), q=_logu(rng, 1e-5, 1e-1))


def _grid_axes(rng, lo, hi):
    """Grid axes with between lo and hi trajectories in all."""
    n = _logu(rng, lo, hi)
    n_t0 = rng.randint(3, 25)
    n_tE = rng.randint(3, 20)
    lines = max(12.0, n / (n_t0 * n_tE))
    n_alpha = max(4, min(72, int(round(math.sqrt(1.8 * lines)))))
    n_u0 = max(2, min(60, int(round(lines / n_alpha))))
    return dict(n_u0=n_u0, n_alpha=n_alpha, n_t0=n_t0, n_tE=n_tE)


def draw(rng):
    kind = rng.choice(["grid", "grid", "search", "sweep", "batch", "grad",
                       "refine", "peaks", "aligned", "poly", "finite"])
    npix = rng.choice([256, 500, 512, 777, 1024, 1024])
    rays = int(round(npix * rng.uniform(7.0, 10.0)))
    out = rng.choice([0.0, 0.01])
    c = dict(kind=kind, npix=npix)
    if kind in ("grid", "search"):
        c |= _lens(rng) | dict(rays=rays, n_ep=_logi(rng, 200, 6000),
                               outliers=out) | _grid_axes(rng, 2e3, 6e5)
        c["top_k"] = rng.choice([1, 16, 50, 256])
        if kind == "grid":
            c["fp16"] = rng.random() < 0.25
        else:
            c["deflect"] = rng.choice(["fp32", "fp64"])
    elif kind == "sweep":
        c |= dict(n_maps=rng.randint(2, 6), rays=rays,
                  n_ep=_logi(rng, 300, 4000), outliers=out,
                  fp16=rng.random() < 0.25) | _grid_axes(rng, 2e4, 4e5)
        c["top_k"] = rng.choice([16, 100, 256])
    elif kind == "batch":
        c |= dict(n_events=rng.randint(3, 12), len_lo=200,
                  len_hi=_logi(rng, 2000, 20000), n_maps=rng.randint(1, 4),
                  rays=rays, top_k=16) | _grid_axes(rng, 2e4, 2e5)
    elif kind == "grad":
        c |= _lens(rng) | dict(rays=rays, n_ep=_logi(rng, 200, 8000),
                               outliers=out, n=_logi(rng, 8, 16384))
    elif kind == "refine":
        c |= dict(n_maps=rng.randint(1, 16), rays=rays,
                  n_ep=_logi(rng, 300, 4000), outliers=out,
                  n=_logi(rng, 16, 4096), iters=rng.choice([20, 40, 50]))
    elif kind == "peaks":
        c |= dict(n_maps=rng.randint(1, 16), rays=rays,
                  n_u0=rng.randint(5, 40), n_alpha=rng.randint(8, 72),
                  sub=rng.choice([1, 2, 2, 4]), max_peaks=8,
                  delta=rng.choice([0.05, 0.1, 0.2]))
    elif kind == "aligned":
        c |= _lens(rng) | dict(rays=rays, n_ep=_logi(rng, 300, 4000),
                               outliers=out, n_u0=rng.randint(10, 40),
                               n_alpha=rng.randint(16, 72),
                               n_t0=rng.randint(1, 5),
                               n_tE=rng.randint(8, 20), max_peaks=2,
                               delta=0.1, top_k=16)
    elif kind == "poly":
        c |= _lens(rng)
    else:
        c |= _lens(rng) | dict(rays=rays, rho=_logu(rng, 3e-3, 0.5))
    return c


# ------------------------------------------------- light curves and lenses
def _mag_point(s, q, y1, y2):
    """Point-source magnification of the binary lens (s, q) at the source
    positions (y1, y2): 64-bit torch tensors in, A out.  The quintic's roots
    by Aberth's iteration, images by their lens-equation residual."""
    m1, m2 = 1.0 / (1.0 + q), q / (1.0 + q)
    z1, z2 = -s * m2, s * m1
    zeta = torch.complex(y1, y2)
    zc = zeta.conj()
    one = torch.ones_like(zeta)
    # P = (z - z1)(z - z2), N = m1 (z - z2) + m2 (z - z1), ascending powers
    p = [z1 * z2, -(z1 + z2), 1.0]
    nn = [-(m1 * z2 + m2 * z1), 1.0]
    a = [(zc - z1) * p[0] + nn[0], (zc - z1) * p[1] + nn[1], (zc - z1) * p[2]]
    b = [(zc - z2) * p[0] + nn[0], (zc - z2) * p[1] + nn[1], (zc - z2) * p[2]]
    ab = [0 * one for _ in range(5)]
    for i in range(3):
        for j in range(3):
            ab[i + j] = ab[i + j] + a[i] * b[j]
    c = [0 * one for _ in range(6)]
    for i in range(5):
        c[i + 1] = c[i + 1] + ab[i]
        c[i] = c[i] - zeta * ab[i]
    w = [m1 * b[i] + m2 * a[i] for i in range(3)]
    for i in range(3):
        for j in range(3):
            c[i + j] = c[i + j] - p[i] * w[j]
    start = [zeta + 0.9 * complex(math.cos(0.4 + 1.2566 * k),
                                  math.sin(0.4 + 1.2566 * k))
             for k in range(5)]
    r = torch.stack(start)
    for _ in range(60):
        f = c[5].expand_as(r)
        d = torch.zeros_like(r)
        for k in range(4, -1, -1):
            d = d * r + f
            f = f * r + c[k]
        n = f / d
        rep = torch.zeros_like(r)
        for k in range(1, 5):
            rep = rep + 1.0 / (r - r.roll(k, 0))
        step = n / (1.0 - n * rep)
        step = torch.where(torch.isfinite(step.abs()), step,
                           torch.zeros_like(step))
        r = r - step
    rc = r.conj()
    res = (r - m1 / (rc - z1) - m2 / (rc - z2) - zeta).abs()
    img = res < 1e-7 * (1.0 + r.abs())
    k = m1 / (rc - z1) ** 2 + m2 / (rc - z2) ** 2
    amp = 1.0 / (1.0 - (k * k.conj()).real).abs()
    return torch.where(img, amp, torch.zeros_like(amp)).sum(0)


def _times(n, rng):
    """Observing times (d): 8-hour nightly windows over [-40, 40] d, more
    sites for long light curves, five times denser within 2 d of the peak."""
    sites = 1 if n <= 1200 else 3
    m = 6 * n
    w = rng.integers(0, 80, m) - 40.0
    site = rng.integers(0, sites, m)
    t = w + (site * 8.0 + 8.0 * rng.random(m)) / 24.0
    t = t[t < 40.0]
    keep = (np.abs(t) < 2.0) | (rng.random(t.size) < 0.2)
    t = t[keep]
    while t.size < n:
        t = np.concatenate([t, rng.uniform(-40.0, 40.0, n)])
    t = rng.permutation(t)[:n]
    return np.sort(t).astype(np.float32).astype(np.float64)


def _truth(rng, s, q):
    return dict(s=s, q=q, t0=0.0,
                u0=float(np.exp(rng.uniform(np.log(1e-3), np.log(0.5)))),
                alpha=float(rng.uniform(0.0, 2.0 * np.pi)),
                tE=float(np.exp(rng.uniform(np.log(5.0), np.log(80.0)))),
                Fb=float(rng.uniform(0.0, 2.0)))


def _light_curve(rng, tr, n, outliers):
    t = _times(n, rng)
    tau = (t - tr["t0"]) / tr["tE"]
    c, s = math.cos(tr["alpha"]), math.sin(tr["alpha"])
    y1 = torch.tensor(tau * c - tr["u0"] * s, device="cuda")
    y2 = torch.tensor(tau * s + tr["u0"] * c, device="cuda")
    A = _mag_point(tr["s"], tr["q"], y1, y2).cpu().numpy()
    f = A + tr["Fb"]
    sig = 0.01 * np.sqrt(f) + 0.002
    flux = f + sig * rng.standard_normal(n)
    k = int(round(outliers * n))
    if k:
        i = rng.choice(n, k, replace=False)
        flux[i] += 5.0 * sig[i] * rng.choice([-1.0, 1.0], k)
    return t, flux, sig


def _rng(seed):
    return np.random.default_rng([int(seed), 1511])


def _sq(case, rng):
    """Lenses of a case: its own, or a slice of the (s, q) range that holds
    the truth lens (near resonance for the largest maps)."""
    if "s" in case:
        return np.array([case["s"]]), np.array([case["q"]])
    n = case["n_maps"]
    if case["npix"] > 2048:
        s = np.exp(rng.uniform(np.log(0.8), np.log(1.25), n))
        q = np.exp(rng.uniform(np.log(1e-4), np.log(1e-2), n))
    else:
        s = np.exp(rng.uniform(np.log(0.3), np.log(3.0), n))
        q = np.exp(rng.uniform(np.log(1e-5), np.log(1e-1), n))
    return s, q


def _inputs(case, seed):
    """Host inputs of a case from its seed: lenses, light curves, starts."""
    rng = _rng(seed)
    kind = case["kind"]
    s, q = _sq(case, rng)
    d = dict(s=s, q=q)
    if kind == "batch":
        lens = np.exp(rng.uniform(np.log(case["len_lo"]),
                                  np.log(case["len_hi"]), case["n_events"]))
        # the longest light curve is always there: calls of another seed
        # are of the same size
        lens *= case["len_hi"] / lens.max()
        lens = np.maximum(lens.astype(int), case["len_lo"])
        d["events"] = []
        for n in lens:
            ts = float(np.exp(rng.uniform(np.log(0.3), np.log(3.0))))
            tq = float(np.exp(rng.uniform(np.log(1e-5), np.log(1e-1))))
            d["events"].append(_light_curve(rng, _truth(rng, ts, tq), int(n),
                                            0.0))
    elif "n_ep" in case:
        k = int(rng.integers(0, len(s)))
        tr = _truth(rng, float(s[k]), float(q[k]))
        d["truth"] = tr
        d["events"] = [_light_curve(rng, tr, case["n_ep"],
                                    case["outliers"])]
    if kind in ("grad", "refine"):
        n, tr = case["n"], d["truth"]
        d["theta"] = np.stack(
            [tr["t0"] + rng.uniform(-1.0, 1.0, n),
             tr["tE"] * np.exp(rng.uniform(-0.3, 0.3, n)),
             tr["u0"] * np.exp(rng.uniform(-0.5, 0.5, n)),
             tr["alpha"] + rng.uniform(-0.2, 0.2, n)], axis=1)
        d["map_of"] = rng.integers(0, len(s), n)
    if kind in ("poly", "finite"):
        # lenses near the case's own: another seed is another lens
        d["s"] = s * np.exp(rng.uniform(-0.02, 0.02))
        d["q"] = q * np.exp(rng.uniform(-0.1, 0.1))
    return d


def _u0_alpha_lines(case):
    u0 = np.exp(np.linspace(np.log(1e-3), np.log(0.5), case["n_u0"]))
    return np.array([(u, 2.0 * np.pi * k / case["n_alpha"], 0.0) for u in u0
                     for k in range(case["n_alpha"])])


def _peak_time(t, f):
    """The peak time read off a light curve: the largest running median of
    seven epochs."""
    w = np.lib.stride_tricks.sliding_window_view(f, 7)
    return float(t[3 + int(np.argmax(np.median(w, axis=1)))])


# ---------------------------------------------------------------- prepare
_CTX = None


def _context():
    """The program's context: one for the process, on a torch stream."""
    global _CTX
    if _CTX is None:
        _CTX = morse.Context(0, stream=torch.cuda.Stream())
    return _CTX


def _grid(case):
    return morse.Grid.make(case["n_u0"], case["n_alpha"], case["n_t0"],
                           case["n_tE"], 1e-3, 0.5, -2.0, 2.0, 5.0, 80.0,
                           True, True, case["top_k"])


def prepare(case, seed):
    ctx = _context()
    d = _inputs(case, seed)
    kind, st = case["kind"], dict(case=case, ctx=ctx)
    st["s"], st["q"] = d["s"], d["q"]

    def maps(deflect):
        return [ctx.build_map(s, q, L, case["npix"], case["rays"],
                              image_halfwidth=X, deflect=deflect,
                              fp16log=bool(case.get("fp16")))
                for s, q in zip(d["s"], d["q"])]

    if kind == "search":
        st["light_curve"] = d["events"][0]
    elif "events" in d:
        st["events"] = [ctx.event(*e) for e in d["events"]]
    if kind in ("grid", "batch", "grad"):
        st["maps"] = maps("fp64")
    elif kind in ("refine", "peaks", "aligned", "finite"):
        st["maps"] = maps("fp32")
    if kind in ("grid", "search", "sweep", "batch"):
        st["grid"] = _grid(case)
    if kind == "grad":
        st["theta"] = torch.tensor(d["theta"], device="cuda",
                                   requires_grad=True)
        st["chi2"] = morse.chi2_function()
    elif kind == "refine":
        f = np.zeros(case["n"], dtype=morse.FIT_DTYPE)
        f["t0"], f["tE"], f["u0"], f["alpha"] = d["theta"].T
        f["chi2"] = np.inf
        f["idx"] = np.arange(case["n"])
        st["starts"], st["map_of"] = f, d["map_of"].astype(np.int32)
    elif kind in ("peaks", "aligned"):
        st["lines"] = _u0_alpha_lines(case)
        if kind == "peaks":
            # another seed is another slice: lines turned by a few degrees
            st["lines"][:, 1] += 0.1 * _rng(seed).random()
        else:
            t, f, _ = d["events"][0]
            st["tp"] = [_peak_time(t, f)]
            n = len(st["lines"])
            st["grid"] = morse.Grid.make(
                case["max_peaks"] * n, 1, case["n_t0"], case["n_tE"], 1.0,
                1.0, -0.05, 0.05, 5.0, 80.0, False, True, case["top_k"])
    return st


# -------------------------------------------------------------------- run
def _fits(f):
    return {k: f[k] for k in ("chi2", "t0", "tE", "u0", "alpha", "Fs", "Fb",
                              "idx", "flags")}


def run(st):
    c, ctx = st["case"], st["ctx"]
    kind = c["kind"]
    if kind == "grid":
        return _fits(ctx.grid_chi2(st["events"][0], st["maps"][0],
                                   st["grid"]))
    if kind == "search":
        t, f, sig = st["light_curve"]
        return _fits(ctx.search(t, f, sig, 0.0, st["s"][0], st["q"][0], L,
                                c["npix"], c["rays"], st["grid"],
                                image_halfwidth=X, deflect=c["deflect"]))
    if kind == "sweep":
        return _fits(ctx.sweep(st["events"][0], st["s"], st["q"], L,
                               c["npix"], c["rays"], st["grid"],
                               image_halfwidth=X, deflect="fp32",
                               fp16log=c["fp16"]))
    if kind == "batch":
        return _fits(ctx.grid_chi2_batch(st["events"], st["maps"],
                                         st["grid"]))
    if kind == "grad":
        theta = st["theta"]
        chi2 = st["chi2"].apply(theta, ctx, st["events"][0], st["maps"][0])
        (g,) = torch.autograd.grad(chi2.sum(), theta)
        return {"chi2": chi2, "grad": g}
    if kind == "refine":
        return _fits(ctx.refine_batch(st["events"][0], st["maps"],
                                      st["map_of"], st["starts"],
                                      iters=c["iters"]))
    if kind == "peaks":
        n, pos, height = ctx.line_peaks_batch(
            st["maps"], st["lines"], sub=c["sub"], max_peaks=c["max_peaks"],
            delta=c["delta"])
        return {"count": n, "pos": pos, "height": height}
    if kind == "aligned":
        return _fits(ctx.peak_search(
            st["events"][0], st["maps"][0], st["grid"], st["lines"],
            tp=st["tp"], min_peaks=1, sub=2, max_peaks=c["max_peaks"],
            delta=c["delta"]))
    if kind == "poly":
        m = ctx.build_map(st["s"][0], st["q"][0], L, c["npix"], 2,
                          generator="poly")
    else:
        m = st["maps"][0].finite_source(c["rho"], GAMMA)
    A = m.values()
    m.free()
    return {"A": A}


# ------------------------------------------------------------------- work
def work(case):
    """Bytes: each map, light curve and start read once, each result written
    once.  Operations: 40 per trajectory and epoch of a grid (the position,
    the bilinear lookup, the sums), 72 with the gradient, 44 per ray, 40 per
    profile sample, 2 per kernel tap, 4000 per polynomial texel."""
    kind = case["kind"]
    tex = 4.0 * case["npix"] ** 2
    nm = case.get("n_maps", 1)
    traj = 1.0
    for k in ("n_u0", "n_alpha", "n_t0", "n_tE"):
        traj *= case.get(k, 1)
    n_ep, k = case.get("n_ep", 0), case.get("top_k", 0)
    rec = 72.0
    rays = 44.0 * case.get("rays", 0) ** 2
    if kind == "grid":
        return dict(bytes=tex + 12 * n_ep + rec * k,
                    flops=40.0 * traj * n_ep)
    if kind in ("search", "sweep"):
        return dict(bytes=nm * (tex + rec * k) + 12 * n_ep,
                    flops=nm * (rays + 40.0 * traj * n_ep))
    if kind == "batch":
        lo, hi = case["len_lo"], case["len_hi"]
        n_ep = case["n_events"] * (hi - lo) / math.log(hi / lo)
        return dict(bytes=nm * tex + 12 * n_ep +
                    rec * k * nm * case["n_events"],
                    flops=40.0 * traj * n_ep * nm)
    if kind == "grad":
        return dict(bytes=tex + 12 * n_ep + 72.0 * case["n"],
                    flops=72.0 * case["n"] * n_ep)
    if kind == "refine":
        return dict(bytes=nm * tex + 12 * n_ep + 2 * rec * case["n"],
                    flops=72.0 * case["n"] * n_ep * case["iters"])
    if kind == "peaks":
        lines = case["n_u0"] * case["n_alpha"]
        return dict(bytes=nm * tex + nm * lines *
                    (4.0 + 16.0 * case["max_peaks"]),
                    flops=40.0 * nm * lines * 1.1 * case["npix"] *
                    case["sub"])
    if kind == "aligned":
        lines = case["n_u0"] * case["n_alpha"]
        return dict(bytes=tex + 12 * n_ep + 24.0 * lines + rec * k,
                    flops=40.0 * traj * case["max_peaks"] * n_ep +
                    40.0 * lines * 2.2 * case["npix"])
    if kind == "poly":
        return dict(bytes=tex, flops=4000.0 * case["npix"] ** 2)
    px = case["rho"] * case["npix"] / (2.0 * L)
    return dict(bytes=2 * tex, flops=2.0 * math.pi * max(px, 0.6) ** 2 *
                case["npix"] ** 2)


# ------------------------------------------------------------------ exact
def _ray_map(s, q, npix, rays):
    """A of inverse ray shooting on the cell-centred ray grid, 64 bits."""
    e1, e2 = 1.0 / (1.0 + q), q / (1.0 + q)
    xa, xb = -s * e2, s * e1
    h, D = 2.0 * X / rays, 2.0 * L / npix
    x = -X + (torch.arange(rays, device="cuda", dtype=torch.float64) +
              0.5) * h
    cnt = torch.zeros(npix * npix + 1, dtype=torch.int64, device="cuda")
    step = max(1, 8_000_000 // rays)
    for r0 in range(0, rays, step):
        x2 = x[r0:r0 + step, None]
        da, db = x[None] - xa, x[None] - xb
        ra, rb = da * da + x2 * x2, db * db + x2 * x2
        y1 = x[None] - e1 * da / ra - e2 * db / rb
        y2 = x2 - e1 * x2 / ra - e2 * x2 / rb
        i, j = torch.floor((y1 + L) / D), torch.floor((y2 + L) / D)
        ok = (i >= 0) & (i < npix) & (j >= 0) & (j < npix)
        k = torch.where(ok, j * npix + i,
                        torch.full_like(i, float(npix * npix)))
        cnt += torch.bincount(k.long().reshape(-1),
                              minlength=npix * npix + 1)
    return (cnt[:-1].double() * (h * h / (D * D))).reshape(npix, npix)


def _lookup(A, y1, y2):
    """Bilinear between texel centres (clamped); the single lens outside."""
    n = A.shape[0]
    D = 2.0 * L / n
    u2 = y1 * y1 + y2 * y2
    out = (u2 + 2.0) / torch.sqrt(u2 * (u2 + 4.0))
    inside = (y1.abs() < L) & (y2.abs() < L)
    x = ((y1 + L) / D - 0.5).clamp(0, n - 1)
    y = ((y2 + L) / D - 0.5).clamp(0, n - 1)
    i, j = x.long().clamp(max=n - 2), y.long().clamp(max=n - 2)
    fx, fy = x - i, y - j
    k = j * n + i
    F = A.reshape(-1)
    m00, m10, m01, m11 = F[k], F[k + 1], F[k + n], F[k + n + 1]
    v = (m00 * (1 - fx) + m10 * fx) * (1 - fy) + (m01 * (1 - fx) +
                                                  m11 * fx) * fy
    gx = ((m10 - m00) * (1 - fy) + (m11 - m01) * fy) / D
    gy = ((m01 - m00) * (1 - fx) + (m11 - m10) * fx) / D
    return torch.where(inside, v, out), gx, gy, inside, u2


def _fit(A, F, w):
    """chi^2, Fs, Fb and residuals of F = Fs A + Fb, weighted."""
    S1 = w.sum()
    Ab, Fm = (A @ w) / S1, (w * F).sum() / S1
    a, f = A - Ab[:, None], F - Fm
    saa = (a * a) @ w
    Fs = (a @ (w * f)) / saa
    r = f[None] - Fs[:, None] * a
    return (r * r) @ w, Fs, Fm - Fs * Ab, r


def _grid_exact(A, ev, case):
    """The grid's top_k records in 64 bits."""
    t, F, sig = (torch.tensor(v, device="cuda") for v in ev)
    w = 1.0 / sig ** 2
    u0 = torch.tensor(np.exp(np.linspace(np.log(1e-3), np.log(0.5),
                                         case["n_u0"])), device="cuda")
    tE = torch.tensor(np.exp(np.linspace(np.log(5.0), np.log(80.0),
                                         case["n_tE"])), device="cuda")
    t0 = torch.linspace(-2.0, 2.0, case["n_t0"], dtype=torch.float64,
                        device="cuda")
    if case["n_t0"] == 1:
        t0 = t0[:1]
    n = case["n_u0"] * case["n_alpha"] * case["n_t0"] * case["n_tE"]
    chi, fs, fb = (torch.empty(n, dtype=torch.float64, device="cuda")
                   for _ in range(3))

    def pars(j):
        iE = j % case["n_tE"]
        j = j // case["n_tE"]
        i0 = j % case["n_t0"]
        j = j // case["n_t0"]
        return (t0[i0], tE[iE], u0[j // case["n_alpha"]],
                2.0 * math.pi * (j % case["n_alpha"]).double() /
                case["n_alpha"])
    step = max(1, 16_000_000 // t.numel())
    for a in range(0, n, step):
        j = torch.arange(a, min(a + step, n), device="cuda")
        p0, pE, pu, pa = pars(j)
        tau = (t[None] - p0[:, None]) / pE[:, None]
        c, s = torch.cos(pa)[:, None], torch.sin(pa)[:, None]
        m = _lookup(A, tau * c - pu[:, None] * s, tau * s +
                    pu[:, None] * c)[0]
        chi[j], fs[j], fb[j], _ = _fit(m, F, w)
    v, order = torch.sort(chi, stable=True)
    j = order[:case["top_k"]]
    p0, pE, pu, pa = pars(j)
    return dict(chi2=v[:case["top_k"]], t0=p0, tE=pE, u0=pu, alpha=pa,
                Fs=fs[j], Fb=fb[j])


def _records(rows, case, shape, values_only):
    """Fields of the records, laid out as run() gives them; only chi^2 where
    rounding of the map itself decides the order of near ties."""
    out = {}
    for k in ("chi2", "t0", "tE", "u0", "alpha", "Fs", "Fb"):
        out[k] = None if values_only and k != "chi2" else torch.stack(
            [r[k] for r in rows]).reshape(shape).cpu().numpy()
    out["idx"] = out["flags"] = None
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind in ("refine", "peaks", "aligned"):
        return None  # decided by the order of iterations or of near ties
    d = _inputs(case, seed)
    if kind == "poly":
        n = case["npix"]
        c = -L + (torch.arange(n, device="cuda", dtype=torch.float64) +
                  0.5) * (2.0 * L / n)
        y2, y1 = torch.meshgrid(c, c, indexing="ij")
        A = _mag_point(float(d["s"][0]), float(d["q"][0]), y1.reshape(-1),
                       y2.reshape(-1))
        return {"A": A.reshape(n, n).cpu().numpy()}
    if kind in ("grid", "search", "sweep", "batch"):
        n_ep = sum(len(e[0]) for e in d["events"])
        traj = case["n_u0"] * case["n_alpha"] * case["n_t0"] * case["n_tE"]
        if traj * n_ep * len(d["s"]) > 2.0e10:
            return None  # over about 20 seconds
    if kind == "finite":
        # the source map is the library's own 32-bit one: its values are the
        # input, made again here
        A = _ray_map(float(d["s"][0]), float(d["q"][0]), case["npix"],
                     case["rays"])
        return {"A": _finite(A, case["rho"]).cpu().numpy()}
    maps = [_ray_map(float(s), float(q), case["npix"], case["rays"])
            for s, q in zip(d["s"], d["q"])]
    if kind == "grad":
        return _grad_exact(maps[0], d, case)
    rows = [_grid_exact(A, e, case) for e in d["events"] for A in maps]
    k = case["top_k"]
    if kind == "batch":
        return _records(rows, case, (len(d["events"]), len(maps), k), False)
    if kind == "sweep":
        return _records(rows, case, (len(maps), k), True)
    # the order of near ties in a long list is a matter of rounding too
    return _records(rows, case, (k,), bool(case.get("fp16")) or k > 16 or
                    case.get("deflect") == "fp32")


def _grad_exact(A, d, case):
    t, F, sig = (torch.tensor(v, device="cuda") for v in d["events"][0])
    w = 1.0 / sig ** 2
    th = torch.tensor(d["theta"], device="cuda")
    D = []
    step = max(1, 16_000_000 // t.numel())
    for a in range(0, th.shape[0], step):
        t0, tE, u0, al = (v[:, None] for v in th[a:a + step].T)
        tau = (t[None] - t0) / tE
        c, s = torch.cos(al), torch.sin(al)
        y1, y2 = tau * c - u0 * s, tau * s + u0 * c
        m, gx, gy, inside, u2 = _lookup(A, y1, y2)
        u = torch.sqrt(u2)
        slope = -8.0 / (u2 * (u2 + 4.0) ** 1.5) / u
        gx = torch.where(inside, gx, slope * y1)
        gy = torch.where(inside, gy, slope * y2)
        chi, Fs, _, r = _fit(m, F, w)
        dt = gx * c + gy * s
        parts = [-dt / tE, -dt * tau / tE, -gx * s + gy * c,
                 -gx * y2 + gy * y1]
        D.append(torch.cat([chi[:, None]] + [
            (-2.0 * Fs * ((r * p) @ w))[:, None] for p in parts], dim=1))
    D = torch.cat(D)
    return {"chi2": D[:, 0].cpu().numpy(), "grad": D[:, 1:].cpu().numpy()}


def _finite(A, rho):
    """A convolved with a limb-darkened source of radius rho: brightness
    integrated over each texel on 8 x 8 midpoints and normalised; outside
    the map the single lens at the texel's centre."""
    n = A.shape[0]
    D = 2.0 * L / n
    R = int(math.ceil(rho / D + 0.5))
    o = (torch.arange(8, dtype=torch.float64, device="cuda") + 0.5) / 8 - 0.5
    k = torch.arange(-R, R + 1, dtype=torch.float64, device="cuda")
    p = (k[:, None] + o[None]).reshape(-1) * D
    r2 = (p[:, None] ** 2 + p[None] ** 2) / (rho * rho)
    b = torch.where(r2 < 1.0, 1.0 - GAMMA * (1.0 - 1.5 * torch.sqrt(
        (1.0 - r2).clamp(min=0.0))), torch.zeros_like(r2))
    m = 2 * R + 1
    W = b.reshape(m, 8, m, 8).sum((1, 3))
    if float(W.sum()) == 0.0:
        return A
    W = W / W.sum()
    c = -L + (torch.arange(-R, n + R, device="cuda", dtype=torch.float64) +
              0.5) * D
    u2 = c[:, None] ** 2 + c[None] ** 2
    P = (u2 + 2.0) / torch.sqrt(u2 * (u2 + 4.0))
    P[R:R + n, R:R + n] = A
    N = P.shape[0] + m
    f = torch.fft.irfft2(torch.fft.rfft2(P, s=(N, N)) *
                         torch.fft.rfft2(W, s=(N, N)), s=(N, N))
    return f[2 * R:2 * R + n, 2 * R:2 * R + n]
