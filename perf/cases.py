"""Workloads of the Wiener-filter library as its users run them, for timing and for
comparing results: single objective calls, batches, both channels, both
precisions, square, rectangular and odd maps, data synthesis, differentiation,
MAP solves and a band-power estimate.  Every input is drawn on the GPU from a seed; the exact
values come from plain torch in 64 bits.

Inputs follow the paper's three kinds of map: "cmb" (temperature, analytic C_l at 2
arcmin pixels, scan-striped noise), "density" (projected galaxy density,
k^-1.5 with a cut-off, Poisson noise) and "shear" (joint E/B, k^-1.2, B at 1% of E,
Poisson shape noise).  All have a mask of point-source-like holes and a band of rows."""
import math

import numpy as np
import torch

from paper_1810_00503_gb300 import autograd, synth, wf

M = 10  # L-BFGS memory of every solve (the library's default)

# Sizes are those of the benchmark, the tests and the paper's workloads.
CASES = [
    # One small FP64 density map: the call of a unit test, a notebook or an outer
    # optimiser on a toy problem.  All launches and host latency.
    dict(name="eval_32_fp64", op="eval", kind="density", ny=32, nx=32, C=1, B=1, precision="fp64"),
    # One CMB patch evaluated alone, as an external optimiser or sampler does it.
    dict(name="eval_1024_single", op="eval", kind="cmb", ny=1024, nx=1024, C=1, B=1, precision="mixed"),
    # The simulation batch of the CMB band powers (100 noise-bias + 20 Fisher maps).
    dict(name="eval_1024_batch", op="eval", kind="cmb", ny=1024, nx=1024, C=1, B=120, precision="mixed"),
    # Hessian-vector products of the joint E/B shear maps (curvature, Lanczos,
    # an external Newton-CG): 53 maps, the E/B band-power batch.
    dict(name="hess_eb_512", op="hess", kind="shear", ny=512, nx=512, C=2, B=53, precision="mixed"),
    # Differentiable chi^2 of a density batch, gradients to the modes and to ten band amplitudes.
    dict(name="autograd_512", op="autograd", kind="density", ny=512, nx=512, C=1, B=64, precision="mixed", bands=10),
    # Maps whose sides are not powers of two, the benchmark's size.
    dict(name="any_768", op="any", kind="cmb", ny=768, nx=768, C=1, B=64, precision="mixed"),
    # The same with odd sides, two channels and FP64: a survey's cut-out in a precise check.
    dict(name="any_375x315_eb_fp64", op="any", kind="shear", ny=375, nx=315, C=2, B=8, precision="fp64"),
    # Data synthesis of 100 simulations on a rectangular patch.
    dict(name="simulate_512x1024", op="simulate", kind="cmb", ny=512, nx=1024, C=1, B=100, precision="mixed"),
    # The batched MAP solve of the CMB simulations: the first eight iterations, in which the
    # history grows.  (Later iterates follow rounding: two of the library's own stage variants differ by
    # 1e-3 after 16 and by 1e-2 after 24, so a longer run has nothing to be compared with.)
    dict(name="solve_1024_batch", op="solve", kind="cmb", ny=1024, nx=1024, C=1, B=120, precision="mixed", iters=8),
    # One FP64 map solved: the reference-accuracy path.
    dict(name="solve_1024_fp64", op="solve", kind="cmb", ny=1024, nx=1024, C=1, B=1, precision="fp64", iters=12),
    # A heterogeneous batch: 48 maps of each of five sizes, own masks and noise, solved in shared launches.
    dict(name="solve_many_64_1024", op="solve_many", kind="density", ny=64, nx=1024, C=1, B=48, precision="mixed",
         iters=8),
    # A joint E/B band-power estimate, the leakage-bias form: 20 simulations, 2 Fisher ones a row.
    dict(name="bandpower_eb_256", op="bandpower", kind="shear", ny=256, nx=256, C=2, B=20, precision="mixed", bands=8,
         iters=10),
]


def listed():
    return [dict(c) for c in CASES]


def _smooth(lo, hi):
    """Every 7-smooth number of [lo, hi]."""
    out = []
    for n in range(lo, hi + 1):
        m = n
        for p in (2, 3, 5, 7):
            while m % p == 0:
                m //= p
        if m == 1:
            out.append(n)
    return out


def draw(rng):
    """One more case: the same operations over sides 8..1024 (square or not), one or two
    channels, both precisions, batches up to the listed pixel counts."""
    op = rng.choice(["eval", "eval", "hess", "autograd", "any", "any", "simulate", "signal", "solve", "solve",
                     "solve_many", "bandpower"])
    C = rng.choice([1, 1, 2])
    precision = rng.choice(["mixed", "mixed", "fp64"])
    if op == "any":
        sides = _smooth(12, 1024)
        ny = min(sides, key=lambda v: abs(v - math.exp(rng.uniform(math.log(12), math.log(1024)))))
        nx = min(sides, key=lambda v: abs(v - math.exp(rng.uniform(math.log(12), math.log(1024)))))
    else:
        lo = 6 if op in ("solve", "bandpower") else 3
        a = rng.randint(lo, 10)
        b = a if rng.random() < 0.6 else rng.randint(lo, 10)
        if op == "solve_many":
            a, b = rng.randint(5, 6), rng.randint(8, 10)  # the smallest and the largest side of the batch
        if op == "bandpower":
            a = b = min(a, 8)
        ny, nx = 1 << a, 1 << b
    kind = "shear" if C == 2 else rng.choice(["cmb", "density"])
    # most pixels (all maps and channels) a call of the kind gets
    most = {"eval": 120 << 20, "hess": 53 << 19, "autograd": 64 << 18, "any": 64 * 768 * 768, "simulate": 100 << 19,
            "signal": 100 << 19, "solve": 90 << 20, "solve_many": 36 << 20, "bandpower": 20 << 17}[op]
    if precision == "fp64":
        most //= 64  # the FP64 path serves single maps and small batches
    per = C * (nx * nx * 4 // 3 if op == "solve_many" else ny * nx)
    B = max(1, min(300, int(math.exp(rng.uniform(0.0, math.log(max(1.0, most / per)))))))
    case = dict(op=op, kind=kind, ny=ny, nx=nx, C=C, B=B, precision=precision)
    if op == "autograd":
        case["bands"] = rng.randint(4, 24)
    if op == "bandpower":
        case.update(B=max(2, min(B, 24)), bands=rng.randint(3, 8))
    if op in ("solve", "solve_many", "bandpower"):
        case["iters"] = rng.choice([4, 5, 6]) if precision == "mixed" else rng.choice([6, 8])
    return case


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _freqs(ny, nx):
    """Signed mode numbers of the half plane (my (ny, 1), mx (1, nx/2+1)), FP64."""
    my = torch.fft.fftfreq(ny, 1.0 / ny, device="cuda", dtype=torch.float64)[:, None]
    mx = torch.arange(nx // 2 + 1, device="cuda", dtype=torch.float64)[None]
    return my, mx


def _modulus(ny, nx):
    """|k| in units of the longer side's fundamental."""
    my, mx = _freqs(ny, nx)
    N = max(ny, nx)
    return torch.sqrt((my * (N / ny)) ** 2 + (mx * (N / nx)) ** 2)


def _rotation(ny, nx):
    """Kaiser-Squires cosine and sine per mode: 1 and 0 at k = 0, sine 0 on the
    Nyquist line of an even side."""
    my, mx = _freqs(ny, nx)
    qy, qx = my / ny, mx / nx
    k2 = qx ** 2 + qy ** 2
    one = torch.where(k2 == 0, torch.ones_like(k2), k2)
    c = torch.where(k2 == 0, torch.ones_like(k2), (qx ** 2 - qy ** 2) / one)
    s = 2 * qx * qy / one
    if ny % 2 == 0:
        s[ny // 2] = 0
    if nx % 2 == 0:
        s[:, nx // 2] = 0
    return c, s


def _apply_A(S, amp, rot, ny, nx):
    """Pixel maps of whitened spectra S (B, C, ny, nx/2+1): U^-1 R(k) sqrt(P) S."""
    a = S * amp
    if S.shape[1] == 2:
        c, s = rot
        a = torch.stack([c * a[:, 0] - s * a[:, 1], s * a[:, 0] + c * a[:, 1]], 1)
    return torch.fft.irfft2(a, s=(ny, nx), norm="ortho")


def _apply_AT(x, amp, rot):
    """sqrt(P) R(k)^T U x."""
    a = torch.fft.rfft2(x, norm="ortho")
    if x.shape[1] == 2:
        c, s = rot
        a = torch.stack([c * a[:, 0] + s * a[:, 1], -s * a[:, 0] + c * a[:, 1]], 1)
    return a * amp


def _randn(gen, *shape):
    return torch.randn(*shape, generator=gen, device="cuda", dtype=torch.float32)


def _mask(gen, B, ny, nx):
    """Observed pixels (B, ny, nx): a band of rows and smooth holes are masked, about a quarter in all."""
    k = _modulus(ny, nx)
    white = torch.fft.rfft2(_randn(gen, B, ny, nx))
    sm = torch.fft.irfft2(white * torch.exp(-0.5 * (k * (2 * math.pi * 3.0 / max(ny, nx))) ** 2).float(), s=(ny, nx))
    lim = sm.mean((1, 2), keepdim=True) + 1.2 * sm.std((1, 2), keepdim=True)
    y0 = torch.randint(0, ny, (B, 1), generator=gen, device="cuda")
    band = (torch.arange(ny, device="cuda")[None] - y0) % ny < max(1, (15 * ny) // 100)
    return ((sm <= lim) & ~band[:, :, None]).to(torch.uint8)


def _spectrum(kind, C, ny, nx):
    """P (C, ny, nx/2+1), FP64: variance of each unitary mode, 0 at k = 0."""
    k = _modulus(ny, nx)
    if kind == "cmb":
        pix = 2.0 / 60.0 * math.pi / 180.0
        ell = 2 * math.pi * k / (max(ny, nx) * pix)
        P = torch.from_numpy(synth.cmb_cl(ell.cpu().numpy()) / (pix * pix)).cuda()[None]
    else:
        safe = torch.where(k == 0, torch.ones_like(k), k)
        P1 = safe ** -1.2 if kind == "shear" else safe ** -1.5 * torch.exp(-((4.0 * k / max(ny, nx)) ** 2))
        P1 = torch.where(k == 0, torch.zeros_like(k), P1)
        P = torch.stack([P1, 0.01 * P1][:C])
    return P


def _variance(gen, kind, B, C, ny, nx):
    """Noise variance per pixel (B, C, ny, nx), FP32."""
    if kind == "cmb":  # scan stripes, +-5% per row
        y = torch.arange(ny, device="cuda", dtype=torch.float32)
        v = 9.0 * (0.5 + 1.25 * (1.0 + torch.sin(16 * math.pi * y / ny)))
        v = v * (1.0 + 0.05 * (2 * torch.rand(B, ny, generator=gen, device="cuda") - 1))
        return v[:, None, :, None].expand(B, C, ny, nx).contiguous()
    mean, num = (10.0, 0.09) if kind == "shear" else (20.0, 1.0)
    n = torch.poisson(torch.full((B, 1, ny, nx), mean, device="cuda"), generator=gen).clamp_(min=1)
    return (num / n).expand(B, C, ny, nx).contiguous()


def _maps(gen, kind, B, C, ny, nx, precision, shared):
    """d, mask, Ninv, P of B maps in the input type; shared: one mask and one noise level map for all
    (simulations of one survey)."""
    dt = torch.float64 if precision == "fp64" else torch.float32
    nb = 1 if shared else B
    mask = _mask(gen, nb, ny, nx)
    var = _variance(gen, kind, nb, C, ny, nx)
    obs = mask[:, None] != 0
    P = _spectrum(kind, C, ny, nx)
    if kind != "cmb":  # signal-to-noise 1 per pixel
        w = torch.full((nx // 2 + 1,), 2.0, device="cuda", dtype=torch.float64)
        w[0] = 1.0
        if nx % 2 == 0:
            w[-1] = 1.0
        P = P * (float(var.mean()) / (float((P * w).sum()) / (C * ny * nx)))
    P = P.to(dt).contiguous()
    rot = _rotation(ny, nx)
    amp, rot = P.sqrt(), tuple(r.to(dt) for r in rot)
    Ninv = torch.where(obs, 1.0 / var, torch.zeros_like(var)).to(dt).expand(B, C, ny, nx).contiguous()
    mask = mask.expand(B, ny, nx).contiguous()
    d = torch.empty(B, C, ny, nx, dtype=dt, device="cuda")
    step = max(1, (1 << 25) // (C * ny * nx))
    for i in range(0, B, step):  # d = M (A z + n), a group of maps at a time
        j = min(B, i + step)
        z = torch.fft.rfft2(_randn(gen, j - i, C, ny, nx).to(dt), norm="ortho")
        noise = _randn(gen, j - i, C, ny, nx).to(dt) * (var[:1] if shared else var[i:j]).sqrt().to(dt)
        d[i:j] = (_apply_A(z, amp, rot, ny, nx) + noise) * mask[i:j, None]
    return d, mask, Ninv, P


def _state(gen, B, C, ny, nx, precision):
    """Whitened modes of white fields (B, C, ny, nx/2+1)."""
    dt = torch.float64 if precision == "fp64" else torch.float32
    return torch.fft.rfft2(_randn(gen, B, C, ny, nx).to(dt), norm="ortho")


def _bands(n_bands, C, ny, nx):
    """Log-spaced bands of |k| from 1 to the Nyquist mode (C, ny, nx/2+1), channel c's ids after channel c-1's."""
    k = _modulus(ny, nx)
    edges = torch.logspace(0, math.log10(max(ny, nx) / 2), n_bands + 1, device="cuda", dtype=torch.float64)
    ids = torch.bucketize(k, edges, right=True) - 1
    ids = torch.where((k >= 1) & (ids < n_bands), ids, torch.full_like(ids, -1))
    return torch.stack([torch.where(ids >= 0, ids + c * n_bands, ids) for c in range(C)]).to(torch.int16).contiguous()


def _sides(c):
    """Sides of a heterogeneous batch: powers of two from the smallest to the largest."""
    n, out = c["ny"], []
    while n <= c["nx"]:
        out.append(n)
        n *= 2
    return out


def _inputs(c, seed):
    gen = torch.Generator("cuda").manual_seed(int(seed))
    op, ny, nx, C, B, prec = c["op"], c["ny"], c["nx"], c["C"], c["B"], c["precision"]
    if op == "solve_many":
        return {"sets": [_maps(gen, c["kind"], B, C, n, n, prec, False) for n in _sides(c)]}
    dt = torch.float64 if prec == "fp64" else torch.float32
    one = op == "bandpower"
    x = dict(zip(("d", "mask", "Ninv", "P"),
                 _maps(gen, c["kind"], 1 if one else B, C, ny, nx, prec, op in ("eval", "hess", "solve", "simulate"))))
    if op in ("eval", "hess", "autograd", "any", "signal"):
        x["s"] = _state(gen, B, C, ny, nx, prec)
    if op == "autograd":
        x["band"] = _bands(c["bands"], C, ny, nx)
        x["logq"] = 0.2 * _randn(gen, c["bands"] * C)
    if op in ("simulate", "bandpower"):
        sig = torch.where(x["Ninv"] > 0, x["Ninv"].clamp(min=1e-30).rsqrt(), torch.zeros_like(x["Ninv"]))
        x["z"] = _randn(gen, B, C, ny, nx).to(dt)
        x["noise"] = _randn(gen, B, C, ny, nx).to(dt) * sig
    if one:
        nf = 2 if B > 2 else 1
        x["band"] = _bands(c["bands"], C, ny, nx)
        x["u"] = _randn(gen, c["bands"] + (1 if C == 2 else 0), nf, C, ny, nx).to(dt)
    return x


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def _opts(c):
    """A fixed budget of iterations (no convergence test ends a solve earlier)."""
    return dict(max_iter=c["iters"], gtol_rel=0.0, lbfgs_m=M)


def prepare(case, seed):
    c, x = dict(case), _inputs(case, seed)
    op = c["op"]
    if op == "solve_many":
        c["problems"] = [wf.Problem(*s, precision=c["precision"], lbfgs_m=M) for s in x["sets"]]
        return c
    if op in ("any", "bandpower"):
        c.update(x)
        return c
    P = x.pop("P")
    c["problem"] = wf.Problem(x.pop("d"), x.pop("mask"), x.pop("Ninv"), P, precision=c["precision"], lbfgs_m=M)
    c.update(x)
    return c


def _sum(c, t):
    """chi^2 beside the fields it belongs to: the mixed path's sums carry the accuracy of its FP32
    fields, and go on in that type."""
    return t.float() if c["precision"] == "mixed" else t


def run(c):
    op = c["op"]
    if op == "eval":
        chi2, grad = c["problem"].eval(c["s"])
        return {"chi2": _sum(c, chi2), "grad": grad}
    if op == "hess":
        return {"hv": c["problem"].hess_vec(c["s"])}
    if op == "any":
        chi2, grad = wf.eval_any(c["s"], c["mask"], c["Ninv"], c["P"], d=c["d"])
        return {"chi2": _sum(c, chi2), "grad": grad}
    if op == "signal":
        return {"x": c["problem"].signal_map(c["s"])}
    if op == "simulate":
        return {"d": c["problem"].simulate(c["z"], c["noise"])}
    if op == "autograd":
        s, logq = c["s"].detach().requires_grad_(), c["logq"].detach().requires_grad_()
        chi2 = autograd.chi2(s, logq.double().exp(), c["problem"], c["band"])
        gs, gq = torch.autograd.grad(chi2.sum(), (s, logq))
        return {"chi2": _sum(c, chi2.detach()), "ds": gs, "dlogq": gq}
    if op == "solve":
        r = c["problem"].solve(**_opts(c))
        return {"s": r.s, "chi2": [e["chi2"] for e in r.stats[:8]], "iters": [e["iters"] for e in r.stats[:8]]}
    if op == "solve_many":
        rs = wf.solve_many(c["problems"], max_iter=c["iters"], gtol_rel=0.0, lbfgs_m=M)
        return {"s": [r.s for r in rs], "chi2": [r.stats[0]["chi2"] for r in rs]}
    eb = c["C"] == 2
    est, _ = wf.bandpower_estimate(c["d"][0], c["mask"][0], c["Ninv"][0], c["P"], c["band"], c["bands"] * c["C"],
                                   c["z"], c["noise"], c["u"], precision=c["precision"],
                                   leak_split=c["bands"] if eb else 0, **_opts(c))
    if c["precision"] == "mixed":  # as _sum; the rest of the estimate is small differences of these
        return {k: est[k].astype(np.float32) for k in ("theta_fid", "E_maps", "bias")}
    return {k: est[k] for k in ("theta_fid", "E_maps", "bias", "fisher", "cov_E", "theta_hat")}


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
def _pass(ny, nx, C, B, elt, maps=2):
    """Bytes and flops of one operator pass: the modes in, the modes out, `maps` pixel maps, the power
    table; two real 2-D transforms and the per-mode and per-pixel steps."""
    npix, nsp = C * ny * nx, C * ny * (nx // 2 + 1)
    return B * elt * (4 * nsp + maps * npix) + elt * nsp, B * npix * (5.0 * math.log2(ny * nx) + 20.0)


def _solve(ny, nx, C, B, elt, iters):
    """Bytes and flops of a MAP solve: each iteration reads the stored pairs and the weights once, reads
    and writes the gradient, and writes a new pair."""
    v, by, fl = float(B) * elt * C * ny * nx, 0.0, 0.0
    for k in range(iters):
        np_ = min(k, M)
        by += (2 * np_ + 2 + 2 + 1) * v
        fl += B * C * ny * nx * (5.0 * math.log2(ny * nx) + 20.0 + 12.0 * np_)
    return by + 3 * v, fl


def work(case):
    c = case
    ny, nx, C, B, elt = c["ny"], c["nx"], c["C"], c["B"], 8 if c["precision"] == "fp64" else 4
    npix, nsp = C * ny * nx, C * ny * (nx // 2 + 1)
    if c["op"] == "solve":
        by, fl = _solve(ny, nx, C, B, elt, c["iters"])
    elif c["op"] == "solve_many":
        got = [_solve(n, n, C, B, elt, c["iters"]) for n in _sides(c)]
        by, fl = sum(g[0] for g in got), sum(g[1] for g in got)
    elif c["op"] == "bandpower":
        nf = 2 if B > 2 else 1
        nF = (c["bands"] + (1 if C == 2 else 0)) * nf
        by, fl = _solve(ny, nx, C, 1 + B + nF, elt, c["iters"])
        by += elt * npix * (2.0 * B + nF)
    elif c["op"] == "simulate":
        by, fl = B * elt * 4.0 * npix + elt * nsp, B * npix * (5.0 * math.log2(ny * nx) + 10.0)
    elif c["op"] == "signal":
        by, fl = B * elt * (2.0 * nsp + npix) + elt * nsp, B * npix * (2.5 * math.log2(ny * nx) + 5.0)
    else:
        by, fl = _pass(ny, nx, C, B, elt, 1 if c["op"] == "hess" else 2)
        if c["op"] == "any":
            by += B * ny * nx  # the mask
        if c["op"] == "autograd":
            by += 2 * nsp  # the band table
    return {"bytes": by, "flops": fl}


# ---------------------------------------------------------------------------
# Exact values: plain torch, 64 bits
# ---------------------------------------------------------------------------
class _Op:
    """chi^2 of a group of maps in FP64 (complex128 half planes)."""

    def __init__(self, d, mask, Ninv, P):
        self.ny, self.nx = Ninv.shape[-2:]
        self.d = d.double()
        self.W = Ninv.double() * (mask[:, None] != 0)
        self.amp = P.double().sqrt()
        self.rot = _rotation(self.ny, self.nx)
        self.w = torch.full((self.nx // 2 + 1,), 2.0, device="cuda", dtype=torch.float64)
        self.w[0] = 1.0
        if self.nx % 2 == 0:
            self.w[-1] = 1.0

    def dot(self, a, b):
        """Full-plane inner product of two half-plane spectra, per map."""
        return ((a.real * b.real + a.imag * b.imag) * self.w).sum((1, 2, 3))

    def A(self, s):
        return _apply_A(s, self.amp, self.rot, self.ny, self.nx)

    def chi2_grad(self, s):
        r = self.d - self.A(s)
        chi2 = self.dot(s, s) + (r * r * self.W).sum((1, 2, 3))
        return chi2, 2 * (s - _apply_AT(self.W * r, self.amp, self.rot))

    def hess(self, v):
        return 2 * (v + _apply_AT(self.W * self.A(v), self.amp, self.rot))

    def lbfgs(self, iters, m=M):
        """`iters` L-BFGS iterations from 0 with the exact step along each direction (two-loop
        recursion, H0 = (s.y / y.y) I)."""
        col = lambda t: t.view(-1, 1, 1, 1)  # noqa: E731
        s = torch.zeros(self.d.shape[:-1] + (self.nx // 2 + 1,), dtype=torch.complex128, device="cuda")
        _, g = self.chi2_grad(s)
        S, Y = [], []
        for _ in range(iters):
            r, al = g.clone(), []
            for a, b in zip(reversed(S), reversed(Y)):
                al.append(self.dot(a, r) / self.dot(a, b))
                r -= col(al[-1]) * b
            if S:
                r *= col(self.dot(S[-1], Y[-1]) / self.dot(Y[-1], Y[-1]))
            for a, b, t in zip(S, Y, reversed(al)):
                r += col(t - self.dot(b, r) / self.dot(a, b)) * a
            q = self.hess(r)  # p = -r
            step = self.dot(g, r) / self.dot(r, q)
            S.append(-col(step) * r)
            Y.append(-col(step) * q)
            s = s + S[-1]
            g = g + Y[-1]
            if len(S) > m:
                S.pop(0)
                Y.pop(0)
        return s


def _groups(B, per):
    """Ranges of maps whose FP64 work fits comfortably."""
    step = max(1, (1 << 24) // per)
    return [(i, min(B, i + step)) for i in range(0, B, step)]


def _theta(P, band, nb, w):
    """Mean of P over the full-plane modes of each band."""
    out = []
    for l in range(nb):
        sel = (band == l).double() * w
        out.append((P.double() * sel).sum() / sel.sum())
    return torch.stack(out)


def _exact_bandpower(c, x):
    """The estimator of the simulations (leakage-bias form for two channels)."""
    C, nb, B = c["C"], c["bands"] * c["C"], c["B"]
    L = c["bands"] if C == 2 else 0
    band, mask, Ninv, P = x["band"].long(), x["mask"], x["Ninv"], x["P"]
    ny, nx = Ninv.shape[-2:]
    rot = _rotation(ny, nx)
    obs = (mask[0] != 0) & (Ninv[0] > 0)
    op0 = _Op(x["d"], mask, Ninv, P)
    theta = _theta(P, band, nb, op0.w)
    sig = lambda z, pw: _apply_A(torch.fft.rfft2(z.double(), norm="ortho"), pw.double().sqrt(), rot, ny, nx)  # noqa: E731
    dj = (sig(x["z"], P) + x["noise"].double()) * obs
    data = [x["d"].double(), dj]
    nf, rows = x["u"].shape[1], x["u"].shape[0]
    for k in range(rows):
        keep = (band == k) if not L or k < L else (band >= L)
        data.append((sig(x["u"][k], P.double() * keep) + dj[:nf]) * obs)
    E = []
    for i, j in _groups(len(torch.cat(data)), C * ny * nx):
        d = torch.cat(data)[i:j]
        op = _Op(d, mask.expand(j - i, ny, nx), Ninv.expand(j - i, C, ny, nx), P)
        p2 = op.lbfgs(c["iters"]).abs().square() * op.w
        E.append(torch.stack([(p2 * (band == l)).sum((1, 2, 3)) / (2 * theta[l]) for l in range(nb)], 1))
    E = torch.cat(E)
    Ej = E[1:1 + B]
    bias = Ej.mean(0)
    F = torch.zeros(nb, nb, device="cuda", dtype=torch.float64)
    for lp in range(nb):
        k = L if L and lp >= L else lp
        col = (E[1 + B + k * nf:1 + B + (k + 1) * nf] - Ej[:nf]).mean(0) / theta[lp]
        F[:, lp] = col
    if L:  # E block whole, B bands their diagonal
        full = F.clone()
        F = torch.diag(full.diagonal())
        F[:L, :L] = full[:L, :L]
    covE = (Ej.T @ Ej - B * torch.outer(bias, bias)) / (B - 1)
    hat = theta + torch.linalg.solve(F, E[0] - bias)
    return {"theta_fid": theta, "E_maps": E, "bias": bias, "fisher": F, "cov_E": covE, "theta_hat": hat}


def exact(case, seed):
    c, x = case, _inputs(case, seed)
    op, C, B, ny, nx = c["op"], c["C"], c["B"], c["ny"], c["nx"]
    if op == "solve_many":
        s, chi2 = [], []
        for d, mask, Ninv, P in x["sets"]:
            parts = []
            for i, j in _groups(B, d[0].numel()):
                o = _Op(d[i:j], mask[i:j], Ninv[i:j], P)
                parts.append(o.lbfgs(c["iters"]))
                if i == 0:
                    chi2.append(float(o.chi2_grad(parts[0])[0][0]))
            s.append(torch.cat(parts))
        return {"s": s, "chi2": chi2}
    if op == "bandpower":
        return _exact_bandpower(c, x)
    out = {}
    if op == "autograd":
        q = x["logq"].double().exp()
        band = x["band"].long()
        x["P"] = x["P"].double() * torch.where(band >= 0, q[band.clamp(min=0)], torch.ones_like(x["P"].double()))
    for i, j in _groups(B, C * ny * nx):
        o = _Op(x["d"][i:j], x["mask"][i:j], x["Ninv"][i:j], x["P"])
        s = x["s"][i:j].to(torch.complex128) if "s" in x else None
        if op in ("eval", "any"):
            got = dict(zip(("chi2", "grad"), o.chi2_grad(s)))
        elif op == "hess":
            got = {"hv": o.hess(s)}
        elif op == "signal":
            got = {"x": o.A(s)}
        elif op == "simulate":
            z = torch.fft.rfft2(x["z"][i:j].double(), norm="ortho")
            got = {"d": (o.A(z) + x["noise"][i:j].double()) * (o.W > 0)}
        elif op == "autograd":
            chi2, g = o.chi2_grad(s)
            a = s - g / 2  # sqrt(P) R^T U W (d - x)
            t = -(a.real * s.real + a.imag * s.imag) * o.w
            dl = torch.stack([(t * (band == l)).sum() for l in range(q.numel())])
            got = {"chi2": chi2, "ds": g * o.w, "dlogq": dl[None]}
        else:
            got = {"s": o.lbfgs(c["iters"])}
            got["chi2"] = o.chi2_grad(got["s"])[0]
        for k, v in got.items():
            out.setdefault(k, []).append(v)
    out = {k: torch.cat(v) for k, v in out.items()}
    if op == "autograd":
        out["dlogq"] = out["dlogq"].sum(0)
    if op == "solve":
        out["chi2"] = [float(v) for v in out["chi2"][:8]]
    return out
