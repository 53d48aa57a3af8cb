"""What a user of this framework has it do, as cases that can be timed and checked.

Each case goes through the public entry points of paper_1609_06041_gb300: the
operators A and A^T (alone, and through autograd), the ramp filter D, whole
reconstructions (low-dose and few-view, one slice and a mixed batch), and the
differentiable unrolled form with its backward pass.  Everything is float32,
the one data type of the library.  Inputs are random-ellipse phantoms with
their analytic line integrals, and transmission Poisson noise for low-dose
data, drawn from the seed alone.  Launch shapes are the library's own choice
(no tuning call), as in a program that just calls it.

exact() evaluates the same mathematics in float64 with plain torch, from the
definitions in the library's header.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1609_06041_gb300 as P

GOLDEN = (math.sqrt(5.0) - 1.0) / 2.0
LANCZOS_STEPS = 12   # the library's default depth of the step-size setup


def bins_for(n):
    """Detector bins that cover the image diagonal, as the mixed batch takes them."""
    return int(math.ceil(1.44 * n))


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # one projection of the smallest configured image: a call whose launches are all its time
        {"name": "project_64", "kind": "project", "n": 64, "views": 90, "bins": 95, "batch": 1, "angles": "uniform"},
        # A and A^T of the low-dose configuration, as a user's own iteration calls them
        {"name": "project_512", "kind": "project", "n": 512, "views": 720, "bins": 736, "batch": 1,
         "angles": "uniform"},
        {"name": "backproject_512", "kind": "backproject", "n": 512, "views": 720, "bins": 736, "batch": 1,
         "angles": "uniform"},
        # the gradient of a data term in a training loop: A forward, A^T backward, a batch of slices on the odd
        # detector that covers a 384 image's diagonal
        {"name": "autograd_384", "kind": "autograd", "n": 384, "views": 90, "bins": 553, "batch": 4,
         "angles": "uniform"},
        # a golden-angle scan (irregular angles, an odd number of views) of an image with a ragged side
        {"name": "autograd_golden_250", "kind": "autograd", "n": 250, "views": 233, "bins": 361, "batch": 1,
         "angles": "golden"},
        # the largest operators: a high-resolution slice
        {"name": "autograd_1024", "kind": "autograd", "n": 1024, "views": 720, "bins": 1475, "batch": 1,
         "angles": "uniform"},
        # FBP filtering of a stack of low-dose sinograms
        {"name": "filter_736", "kind": "filter", "views": 720, "bins": 736, "batch": 4},
        # whole reconstructions, step sizes estimated in the call: the smallest configured one, ...
        {"name": "solve_lowdose_64", "kind": "solve", "n": 64, "views": 90, "bins": 95, "mode": "lowdose",
         "precond": 1, "iters": 20, "beta": 0.01, "i0": 1e4, "ellipses": 10},
        # ... the few-view configuration (its iterations are launches and latency), ...
        {"name": "solve_fewview_512", "kind": "solve", "n": 512, "views": 32, "bins": 736, "mode": "fewview",
         "precond": 3, "iters": 100, "beta": 0.0, "i0": 0.0, "ellipses": 20},
        # ... and the low-dose configuration, the framework's headline
        {"name": "solve_lowdose_512", "kind": "solve", "n": 512, "views": 720, "bins": 736, "mode": "lowdose",
         "precond": 1, "iters": 30, "beta": 0.005, "i0": 5e3, "ellipses": 20},
        # a study's slices of mixed shapes and modes in one call
        {"name": "batched_12", "kind": "batched", "count": 12, "mix": 0, "iters": 30},
        # one training step of the unrolled reconstructor (learned taps and beta), its configured batch
        {"name": "unrolled_256", "kind": "unrolled", "n": 256, "views": 180, "bins": 368, "batch": 16, "iters": 10,
         "half": 128},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["project", "backproject", "autograd", "autograd", "filter", "solve", "solve", "batched",
                       "unrolled"])
    if kind in ("project", "backproject", "autograd"):
        while True:
            n, views, batch = _log_int(rng, 64, 1024), _log_int(rng, 30, 720), rng.choice([1, 1, 2, 4])
            if n * n * views * batch <= 1024 * 1024 * 720:
                break
        if rng.random() < 0.5:
            n = max(64, n // 32 * 32)   # image sides are more often round than not
        bins = rng.choice([bins_for(n), n, n + n // 2 + 1])
        return {"kind": kind, "n": n, "views": views, "bins": bins, "batch": batch,
                "angles": rng.choice(["uniform", "uniform", "golden"])}
    if kind == "filter":
        return {"kind": kind, "views": _log_int(rng, 30, 720), "bins": _log_int(rng, 95, 1475),
                "batch": rng.choice([1, 2, 4])}
    if kind == "solve":
        n = rng.choice([_log_int(rng, 64, 512), _log_int(rng, 64, 512) // 32 * 32])
        n = max(64, n)
        views, bins = _log_int(rng, 30, 720), bins_for(n)
        low = views * bins > n * n
        return {"kind": kind, "n": n, "views": views, "bins": bins, "mode": "lowdose" if low else "fewview",
                "precond": rng.choice([1, 1, 2]) if low else rng.choice([1, 3]),
                "iters": rng.randint(10, 30) if low else rng.randint(10, 100),
                "beta": 0.005 if low else 0.0, "i0": 5e3 if low else 0.0, "ellipses": rng.randint(10, 20)}
    if kind == "batched":
        return {"kind": kind, "count": rng.randint(3, 10), "mix": rng.randint(1, 1000), "iters": rng.randint(10, 30)}
    n = _log_int(rng, 64, 256) // 2 * 2
    return {"kind": kind, "n": n, "views": _log_int(rng, 30, 180), "bins": bins_for(n), "batch": rng.randint(1, 16),
            "iters": rng.randint(3, 10), "half": rng.choice([32, 64])}


def _mixed(case):
    """Slice shapes of a mixed batch: (n, views, bins, mode); low-dose where the sinogram has the more samples."""
    r = np.random.default_rng(case["mix"])
    out = []
    for _ in range(case["count"]):
        n, v = int(r.choice([256, 384, 512])), int(r.choice([32, 90, 360, 720]))
        b = bins_for(n)
        out.append((n, v, b, "lowdose" if v * b > n * n else "fewview"))
    return out


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _angles(case):
    if case.get("angles", "uniform") == "golden":
        return np.mod(np.arange(case["views"]) * (math.pi * GOLDEN), math.pi)
    return None


def _theta(views, angles):
    t = np.arange(views) * (math.pi / views) if angles is None else angles
    return torch.tensor(t, dtype=torch.float64, device="cuda")


def _ellipses(n, count, r):
    R = n / 2.0
    rad, ang = 0.6 * R * np.sqrt(r.uniform(size=count)), 2 * math.pi * r.uniform(size=count)
    return np.stack([rad * np.cos(ang), rad * np.sin(ang), r.uniform(0.05 * R, 0.3 * R, count),
                     r.uniform(0.05 * R, 0.3 * R, count), r.uniform(0.0, math.pi, count),
                     r.uniform(0.05, 0.4, count)], axis=1)


def _phantom(n, ell):
    c = torch.arange(n, dtype=torch.float64, device="cuda") - (n - 1) / 2.0
    img = torch.zeros(n, n, dtype=torch.float64, device="cuda")
    for cx, cy, a, b, phi, val in ell:
        dx, dy = c[None, :] - cx, c[:, None] - cy
        u, v = (dx * math.cos(phi) + dy * math.sin(phi)) / a, (dy * math.cos(phi) - dx * math.sin(phi)) / b
        img += val * (u * u + v * v <= 1.0)
    return img


def _integrals(views, bins, angles, ell):
    t = _theta(views, angles)[:, None]
    s = (torch.arange(bins, dtype=torch.float64, device="cuda") - (bins - 1) / 2.0)[None, :]
    out = torch.zeros(views, bins, dtype=torch.float64, device="cuda")
    for cx, cy, a, b, phi, val in ell:
        q = (a * torch.cos(t - phi)) ** 2 + (b * torch.sin(t - phi)) ** 2
        off = s - (cx * torch.cos(t) + cy * torch.sin(t))
        out += (2.0 * a * b * val) * torch.sqrt(torch.clamp(q - off * off, min=0.0)) / q
    return out


def _scan(n, views, bins, mode, i0, count, r, gen):
    """(b, w) of one slice: Poisson counts over unit-range attenuation, or noiseless line integrals (w None)."""
    p = _integrals(views, bins, None, _ellipses(n, count, r))
    if mode == "fewview":
        return p.float(), None
    counts = torch.clamp(torch.poisson(i0 * torch.exp(-p * (2.0 / n)), generator=gen), min=1.0)
    return (-torch.log(counts / i0)).float(), counts.float()


def _ramp_taps64(bins, views, mode, tau, kappa):
    """Centred taps t[k], |k| < bins, of D (float64): the smoothed ramp, or the pure ramp with kappa = 0."""
    per = 1
    while per < 2 * bins:
        per *= 2
    k = torch.arange(per, device="cuda")
    w = (2 * math.pi / per) * torch.minimum(k, per - k).double()
    h = w / (2.0 * views * tau + kappa * w)
    t = torch.fft.ifft(h).real[:bins]
    return torch.cat([t.flip(0)[:-1], t])


def _case_inputs(case, seed):
    """The arrays of a case, from the seed alone (shared by prepare and exact)."""
    r = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    kind = case["kind"]
    if kind in ("project", "backproject", "autograd"):
        n, v, b, batch, ang = case["n"], case["views"], case["bins"], case["batch"], _angles(case)
        ells = [_ellipses(n, 12, r) for _ in range(batch)]
        d = {}
        if kind != "backproject":
            d["img"] = torch.stack([_phantom(n, e) for e in ells]).float()
        if kind != "project":   # a residual: what A^T is applied to
            d["sino"] = torch.stack([(2.0 / n) * _integrals(v, b, ang, e) for e in ells]).float()
            d["sino"] += 0.05 * torch.randn(d["sino"].shape, generator=gen, device="cuda")
        if batch == 1:
            d = {k: t[0].contiguous() for k, t in d.items()}
        return d
    if kind == "filter":
        v, b = case["views"], case["bins"]
        sino = torch.stack([0.01 * _integrals(v, b, None, _ellipses(b / 1.44, 12, r)) for _ in range(case["batch"])])
        sino = sino.float() + 0.02 * torch.randn(sino.shape, generator=gen, device="cuda")
        return {"sino": sino, "taps": _ramp_taps64(b, v, 0, math.pi * 1e-3 / (2 * v), 1e-3).float()}
    if kind == "solve":
        b, w = _scan(case["n"], case["views"], case["bins"], case["mode"], case["i0"], case["ellipses"], r, gen)
        return {"b": b, "w": w}
    if kind == "batched":
        return {"slices": [_scan(n, v, b, m, 5e3, 10, r, gen) for n, v, b, m in _mixed(case)]}
    # unrolled: low-dose slices of one geometry, their phantoms as targets
    n, v, b = case["n"], case["views"], case["bins"]
    bs, ws, xt = [], [], []
    for _ in range(case["batch"]):
        e = _ellipses(n, 10, r)
        p = _integrals(v, b, None, e) * (2.0 / n)
        counts = torch.clamp(torch.poisson(1e4 * torch.exp(-p), generator=gen), min=1.0)
        bs.append((-torch.log(counts / 1e4)).float())
        ws.append(counts.float())
        xt.append((_phantom(n, e) * (2.0 / n)).float())
    kappa = 2e-4   # about the mean of 1 / w
    tau = math.pi * kappa / (2 * v)
    taps = _ramp_taps64(b, v, 0, tau, kappa).float()
    return {"b": torch.stack(bs), "w": torch.stack(ws), "target": torch.stack(xt), "taps": taps, "tau": tau,
            "sigma": 0.9 / (1.6 + 0.4 * n / v), "beta": 0.01}   # inside the step rule's bound


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------
def _params(case, mode):
    low = mode == "lowdose"
    return P.PDTVParams(mode=P.CT_LOWDOSE if low else P.CT_FEWVIEW, iters=case["iters"], tv_iters=10,
                        precond=case.get("precond", 1), beta=case.get("beta", 0.005) if low else 0.0)


def prepare(case, seed):
    d = _case_inputs(case, seed)
    kind = case["kind"]
    s = {"kind": kind}
    if kind == "batched":
        slices = []
        for (n, v, b, m), (bb, ww) in zip(_mixed(case), d["slices"]):
            slices.append((P.Geometry(n, v, b), bb, ww, _params(case, m)))
        s["solve"] = P.BatchedSolve(slices)
        return s
    s["g"] = P.Geometry(case.get("n", 64), case["views"], case["bins"], angles=_angles(case))
    s.update(d)
    if kind == "autograd":
        s["img"].requires_grad_(True)
    elif kind == "solve":
        s["params"] = _params(case, case["mode"])
        s["ws"] = P.workspace_for(s["g"], s["params"])
        s["x"] = torch.empty(case["n"], case["n"], device="cuda")
    elif kind == "unrolled":
        s["model"] = P.UnrolledReconstructor(s["g"], d["taps"], d["beta"], d["tau"], d["sigma"], iters=case["iters"],
                                             tv_iters=10, half=min(case["half"], case["bins"]))
    return s


def run(s):
    kind = s["kind"]
    if kind == "project":
        return P.ct_project(s["g"], s["img"])
    if kind == "backproject":
        return P.ct_backproject(s["g"], s["sino"])
    if kind == "autograd":
        y = P.project(s["g"], s["img"])
        (grad,) = torch.autograd.grad(y, s["img"], s["sino"])
        return y.detach(), grad
    if kind == "filter":
        return P.ct_ramp_filter(s["g"], s["taps"], s["sino"])
    if kind == "solve":
        return P.ct_pdtv_solve(s["g"], s["b"], s["w"], s["params"], x_out=s["x"], workspace=s["ws"], report=False)[0]
    if kind == "batched":
        return s["solve"].run()[0]
    m = s["model"]
    m.zero_grad(set_to_none=True)
    x = m(s["b"], s["w"])
    loss = ((x - s["target"]) ** 2).mean()
    loss.backward()
    return [x.detach(), loss.detach(), m.taps_half.grad, m.log_beta.grad]


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------
def _nnz(n, v):
    return 2.0 * n * n * v * (2.0 * math.sqrt(2.0) / math.pi)   # two pixels per crossed line


def _filter_flops(v, b):
    per = 1
    while per < 2 * b:
        per *= 2
    return v * (5.0 * per * math.log2(per) + 3.0 * per)   # a real view's two transforms


def _solve_work(n, v, b, low, iters):
    one = 4.0 * _nnz(n, v) + (2 if low else 1) * _filter_flops(v, b) + 10 * 25.0 * n * n
    norms = LANCZOS_STEPS * (4.0 * _nnz(n, v) + (2 if low else 1) * _filter_flops(v, b))
    return 4.0 * ((2 if low else 1) * v * b + n * n), iters * one + norms


def work(case):
    kind = case["kind"]
    if kind in ("project", "backproject", "autograd"):
        n, v, b, k = case["n"], case["views"], case["bins"], case["batch"] * (2 if kind == "autograd" else 1)
        return {"bytes": 4.0 * k * (n * n + v * b), "flops": 2.0 * k * _nnz(n, v)}
    if kind == "filter":
        return {"bytes": 8.0 * case["batch"] * case["views"] * case["bins"],
                "flops": case["batch"] * _filter_flops(case["views"], case["bins"])}
    if kind == "solve":
        by, fl = _solve_work(case["n"], case["views"], case["bins"], case["mode"] == "lowdose", case["iters"])
        return {"bytes": by, "flops": fl}
    if kind == "batched":
        w = [_solve_work(n, v, b, m == "lowdose", case["iters"]) for n, v, b, m in _mixed(case)]
        return {"bytes": sum(x[0] for x in w), "flops": sum(x[1] for x in w)}
    n, v, b, k, s = case["n"], case["views"], case["bins"], case["iters"], case["batch"]
    fwd = 4.0 * _nnz(n, v) + 2 * _filter_flops(v, b) + 10 * 25.0 * n * n
    corr = 2 * 2.0 * v * b * (2 * min(case["half"], b) - 1)   # the two tap correlations of a step
    return {"bytes": 4.0 * s * (2 * v * b + 2 * n * n), "flops": s * k * (2 * fwd + corr)}


# ---------------------------------------------------------------------------
# float64 values
# ---------------------------------------------------------------------------
class _Ops:
    """A, A^T (Joseph, parallel beam) and D in float64, matrix-free, a few views at a time."""

    def __init__(self, n, v, b, angles=None):
        self.n, self.v, self.b = n, v, b
        self.t = _theta(v, angles)
        c, s = torch.cos(self.t), torch.sin(self.t)
        k = torch.arange(v, device="cuda")
        self.rows = (4 * k <= v) | (4 * k >= 3 * v) if angles is None else c.abs() >= s.abs()
        self.c, self.s = c, s
        self.a = torch.where(self.rows, 1 / c, 1 / s)
        self.m = torch.where(self.rows, -s / c, -c / s)
        self.chunk = max(1, (1 << 25) // (n * max(n, b)))

    def project(self, img):
        n, b, h = self.n, self.b, (self.n - 1) / 2.0
        dp = (torch.arange(b, device="cuda").double() - (b - 1) / 2.0)[None, :, None]
        sp = (torch.arange(n, device="cuda").double() - h)[None, None, :]
        line = torch.arange(n, device="cuda")[None, None, :] * (n + 4)
        out = torch.zeros(self.v, b, dtype=torch.float64, device="cuda")
        for rows in (True, False):
            flat = torch.nn.functional.pad(img if rows else img.t(), (2, 2)).reshape(-1).contiguous()
            ids = torch.nonzero(self.rows == rows)[:, 0]
            for i in range(0, len(ids), self.chunk):
                v = ids[i:i + self.chunk]
                u = h + dp * self.a[v][:, None, None] + sp * self.m[v][:, None, None]
                u = u.clamp(-1.5, n + 0.5)
                f = torch.floor(u)
                at = line + f.long() + 2
                f = u - f
                y = ((1 - f) * flat[at] + f * flat[at + 1]).sum(2)
                out[v] = y * self.a[v].abs()[:, None]
        return out

    def backproject(self, sino):
        n, b, h = self.n, self.b, (self.n - 1) / 2.0
        x = (torch.arange(n, device="cuda").double() - h)
        pad = torch.nn.functional.pad(sino, (2, 2))
        out = torch.zeros(n, n, dtype=torch.float64, device="cuda")
        for i in range(0, self.v, self.chunk):
            c, s = self.c[i:i + self.chunk, None, None], self.s[i:i + self.chunk, None, None]
            e = x[None, None, :] * c + x[None, :, None] * s + (b - 1) / 2.0
            e = e.clamp(-1.5, b + 0.5)
            d = torch.floor(e)
            at = d.long() + 2 + (torch.arange(len(c), device="cuda") * (b + 4))[:, None, None]
            a = self.a[i:i + self.chunk].abs()[:, None, None]
            f = e - d
            flat = pad[i:i + self.chunk].reshape(-1)
            out += (a * ((1 - f * a).clamp(min=0) * flat[at] + (1 - (1 - f) * a).clamp(min=0) * flat[at + 1])).sum(0)
        return out


def _conv64(taps, y):
    """The linear convolution of each view with centred taps."""
    half, b = (taps.numel() + 1) // 2, y.shape[-1]
    m = 2 * b + taps.numel()
    f = torch.fft.irfft(torch.fft.rfft(taps, n=m) * torch.fft.rfft(y, n=m), n=m)
    return f[..., half - 1:half - 1 + b]


class _A(torch.autograd.Function):
    @staticmethod
    def forward(ctx, x, ops):
        ctx.ops = ops
        return torch.stack([ops.project(i) for i in x])

    @staticmethod
    def backward(ctx, g):
        return torch.stack([ctx.ops.backproject(i) for i in g]), None


class _AT(torch.autograd.Function):
    @staticmethod
    def forward(ctx, y, ops):
        ctx.ops = ops
        return torch.stack([ops.backproject(i) for i in y])

    @staticmethod
    def backward(ctx, g):
        return torch.stack([ctx.ops.project(i) for i in g]), None


def _prox64(z, px, py, lam, steps):
    """The TV prox by projected gradient on the dual field; image in the last two axes."""
    pad = torch.nn.functional.pad

    def div(px, py):
        a, c = px[..., :, :-1], py[..., :-1, :]
        return pad(a, (0, 1)) - pad(a, (1, 0)) + pad(c, (0, 0, 0, 1)) - pad(c, (0, 0, 1, 0))

    for _ in range(steps):
        x = torch.relu(z + lam * div(px, py))
        qx = px + pad(x[..., :, 1:] - x[..., :, :-1], (0, 1)) / (8 * lam)
        qy = py + pad(x[..., 1:, :] - x[..., :-1, :], (0, 0, 0, 1)) / (8 * lam)
        nrm = torch.sqrt((qx * qx + qy * qy).clamp(min=1.0))
        px, py = qx / nrm, qy / nrm
    return torch.relu(z + lam * div(px, py)), px, py


def _lanczos64(op, shape):
    """The library's norm estimate: the Ritz value of a fixed-depth Lanczos run from a hashed +-1 start, plus its
    residual norm."""
    count = int(np.prod(shape))
    i = np.arange(count, dtype=np.uint64)
    x = (i * 2654435761 + 12345) & 0xFFFFFFFF
    x ^= x >> 16
    x = (x * 0x7FEB352D) & 0xFFFFFFFF
    x ^= x >> 15
    x = (x * 0x846CA68B) & 0xFFFFFFFF
    x ^= x >> 16
    q = torch.tensor(np.where(x & 1, 1.0, -1.0), device="cuda").reshape(shape) / math.sqrt(count)
    prev, alpha, beta = torch.zeros_like(q), [], []
    for j in range(LANCZOS_STEPS):
        w = op(q) - (beta[-1] if beta else 0.0) * prev
        alpha.append(float((w * q).sum()))
        w = w - alpha[-1] * q
        beta.append(float(torch.sqrt((w * w).sum())))
        prev, q = q, w / beta[-1]
    val, vec = np.linalg.eigh(np.diag(alpha) + np.diag(beta[:-1], 1) + np.diag(beta[:-1], -1))
    return val[-1] + beta[-1] * abs(vec[-1, -1])


def _solve64(n, v, b, mode, precond, iters, beta, bb, ww):
    ops, low = _Ops(n, v, b), mode == "lowdose"
    bb = bb.double()
    winv = 1.0 / ww.double() if low else None
    if low:
        kappa = float(winv.mean())
        tau = math.pi * kappa / (2 * v)
    else:
        tau, kappa = 0.01, 0.0
        if precond == 3:
            kappa = tau * (2.0 / 3.0) * (n * n / b) * float(ops.a.abs().mean())
    if precond == 2:
        per = 1
        while per < 2 * b:
            per *= 2
        k = torch.arange(per, device="cuda")
        w = (2 * math.pi / per) * torch.minimum(k, per - k).double()
        den = (2.0 * v * tau + kappa * w) ** 2
        lo, hi = (torch.fft.ifft(h).real[:b] for h in (2.0 * v * tau * w / den, kappa * w * w / den))
        lo, hi = (torch.cat([t.flip(0)[:-1], t]) for t in (lo, hi))
        sv = torch.sqrt(kappa / winv)

        def D(y):
            return _conv64(lo, y) + sv * _conv64(hi, sv * y)
    else:
        taps = _ramp_taps64(b, v, mode, tau, kappa)

        def D(y):
            return _conv64(taps, y)
    bound = 1.0 / (tau * _lanczos64(lambda x: ops.backproject(D(ops.project(x))), (n, n)))
    if low:
        sw = torch.sqrt(winv)
        bound = min(bound, 2.0 / _lanczos64(lambda y: sw * D(sw * y), (v, b)))
    sigma, lam = 0.95 * bound, tau * beta if low else tau
    x = torch.zeros(n, n, dtype=torch.float64, device="cuda")
    px, py, mu = torch.zeros_like(x), torch.zeros_like(x), torch.zeros_like(bb)
    mubar = -sigma * D(bb)
    for _ in range(iters):
        x, px, py = _prox64(x - tau * ops.backproject(mubar), px, py, lam, 10)
        res = ops.project(x) - bb
        if low:
            res = res - winv * mu
        new = mu + sigma * D(res)
        mubar = 2 * new - mu
        if low:
            mubar = mubar - sigma * D(winv * (new - mu))
        mu = new
    return x


def _unrolled64(case, d):
    ops = _Ops(case["n"], case["views"], case["bins"])
    half, b = min(case["half"], case["bins"]), d["b"].double()
    winv, tau, sigma = 1.0 / d["w"].double(), d["tau"], d["sigma"]
    h0 = (d["taps"].numel() + 1) // 2
    th = d["taps"][h0 - 1:h0 - 1 + half].double().requires_grad_(True)
    # the module keeps log beta in float32
    lb = torch.tensor(float(d["beta"])).log().cuda().double().requires_grad_(True)
    taps, lam = torch.cat([th.flip(0)[:-1], th]), tau * lb.exp()
    x = torch.zeros_like(d["target"], dtype=torch.float64)
    px, py, mu = torch.zeros_like(x), torch.zeros_like(x), torch.zeros_like(b)
    mubar = -sigma * _conv64(taps, b)
    for _ in range(case["iters"]):
        x, px, py = _prox64(x - tau * _AT.apply(mubar, ops), px, py, lam, 10)
        new = mu + sigma * _conv64(taps, _A.apply(x, ops) - b - winv * mu)
        mubar = 2 * new - mu - sigma * _conv64(taps, winv * (new - mu))
        mu = new
    loss = ((x - d["target"].double()) ** 2).mean()
    loss.backward()
    return [x.detach(), loss.detach(), th.grad, lb.grad]


def exact(case, seed):
    d = _case_inputs(case, seed)
    kind = case["kind"]
    if kind in ("project", "backproject", "autograd"):
        ops, k = _Ops(case["n"], case["views"], case["bins"], _angles(case)), case["batch"]

        def each(f, t):
            return f(t.double()) if k == 1 else torch.stack([f(i.double()) for i in t])

        if kind == "project":
            return each(ops.project, d["img"])
        if kind == "backproject":
            return each(ops.backproject, d["sino"])
        return each(ops.project, d["img"]), each(ops.backproject, d["sino"])
    if kind == "filter":
        return _conv64(d["taps"].double(), d["sino"].double())
    if kind == "solve":
        return _solve64(case["n"], case["views"], case["bins"], case["mode"], case["precond"], case["iters"],
                        case["beta"], d["b"], d["w"])
    if kind == "batched":   # the slices that about fifteen seconds are enough for
        out, left = [], 2.2e8 * 80
        for (n, v, b, m), (bb, ww) in zip(_mixed(case), d["slices"]):
            left -= float(n) * max(n, b) * v * (case["iters"] + LANCZOS_STEPS)
            out.append(_solve64(n, v, b, m, 1, case["iters"], 0.005 if m == "lowdose" else 0.0, bb, ww)
                       if left > 0 else None)
        return out
    return _unrolled64(case, d)
