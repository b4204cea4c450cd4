"""Performance cases of the library: the calls that its users make, on the
sizes of this repository's workloads, tests and benchmark.

Each case names a kind of call (products, CGLS solves, a batch of solves, a
gradient of the regularised cost, a product without the stored matrix or in
double precision, the building of a plan), the geometry, the slice count,
the storage precision and the plan flags that a user of that precision and
slice count sets.  The inputs are seeded phantoms (sums of ellipses) and
their exact line integrals with measurement noise.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2009_07226_gb300 import autograd, inputs, xct

FLAGS = ("few_slices", "narrow_tiles", "paired_rows", "keep_f64")


def _case(kind, n, m, nd, S, storage, flags="", iters=0, name=None):
    c = dict(kind=kind, n=n, m=m, nd=nd, S=S, storage=storage, flags=flags, iters=iters)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # One small slice solved alone (the 128^2 2D workload): launches and
        # latency are all of it.  Solves here run the iterations in which
        # CGLS iterates are not yet dominated by its rounding sensitivity.
        _case("cgls", 128, 180, 128, 1, "f32", iters=5, name="cgls_128_f32_1"),
        # The batched 3D workload, 512^2 x 768 angles x 64 slices, in mixed
        # precision: its two products, as one calls them from an outer loop
        # (a projection to compare with data, a back projection of residuals),
        # and its solve.
        _case("project", 512, 768, 512, 64, "f16", "paired_rows", name="project_512_f16_64"),
        _case("backproject", 512, 768, 512, 64, "f16", "paired_rows", name="backproject_512_f16_64"),
        _case("cgls", 512, 768, 512, 64, "f16", "paired_rows", iters=5, name="cgls_512_f16_64"),
        # The same operator in single precision, the library's default
        # storage: a solve of an odd number of slices.
        _case("cgls", 512, 768, 512, 27, "f32", iters=3, name="cgls_512_f32_27"),
        # A few slices of it (a quick look at part of a volume).
        _case("project", 512, 768, 512, 3, "f16", "few_slices", name="project_512_f16_3"),
        # The largest geometry: 1536^2 x 1024 angles x 32 slices.
        _case("project", 1536, 1024, 1536, 32, "f16", "narrow_tiles", name="project_1536_f16_32"),
        # One step of the TV-regularised reconstruction, forward and backward
        # through the autograd functions (1024^2 x 720 x 16, bfloat16).
        _case("gradient", 1024, 720, 1024, 16, "bf16", "narrow_tiles", name="gradient_1024_bf16_16"),
        # Jobs of uneven geometry and slice count solved together.
        _case("batch", 384, 576, 384, 20, "f16", "paired_rows", iters=3, name="batch_384_f16"),
        # The double-precision form on a few slices (a check of a reconstruction).
        _case("project_f64", 256, 384, 256, 4, "f32", "keep_f64", name="project_256_f64_4"),
        # Without the stored matrix (a grid visited once, or too large to store).
        _case("project_matfree", 256, 384, 256, 24, "f32", name="matfree_256_24"),
        # A new geometry: the plan is built, used once and released.
        _case("plan", 256, 384, 256, 1, "f32", name="plan_256_f32"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("project", "project", "backproject", "backproject", "cgls", "cgls", "gradient",
                       "batch", "project_f64", "project_matfree", "plan"))
    n = _log_int(rng, 96, 1100)
    S = _log_int(rng, 1, 100)
    if kind in ("project_f64", "project_matfree", "plan"):
        n, S = _log_int(rng, 64, 320), _log_int(rng, 1, 32)
    if kind in ("batch", "gradient"):
        n, S = _log_int(rng, 96, 640), _log_int(rng, 2, 32)
    m = max(2, int(n * rng.uniform(0.7, 1.5)))
    nd = max(2, int(n * rng.uniform(0.9, 1.1)))
    storage = rng.choice(("f16", "f16", "f16", "f32", "f32", "bf16"))
    flags = ""
    if kind == "project_f64":
        storage, flags = "f32", "keep_f64"
    elif kind == "project_matfree":
        storage = "f32"
    elif storage != "f32":
        # the flag that the documentation gives for the slice count, or none
        fit = "few_slices" if S <= 8 else "narrow_tiles" if S <= 32 else "paired_rows"
        flags = rng.choice((fit, fit, ""))
        if fit == "paired_rows" and (n - nd) % 2:
            flags = ""   # rays along grid lines meet a pixel twice there, which such a plan refuses
    iters = rng.randint(1, 3 if storage != "f32" else 4) if kind in ("cgls", "batch") else 0
    if storage == "bf16" and iters:
        storage = "f16"   # bfloat16 serves gradients and products
    return _case(kind, n, m, nd, S, storage, flags, iters)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _ellipses(rng, S, count=12):
    """[S, count, 6] (cx, cy, a, b, phi, rho): the ellipses drift from slice
    to slice as the cuts of a volume do."""
    base = np.stack([inputs.random_ellipses(rng, count, (0.0, 1.0))])
    e = np.repeat(base, S, axis=0)
    z = (np.arange(S) + 0.5) / S
    e[:, :, 2:4] *= np.sqrt(1.0 - 0.8 * (z[:, None, None] - rng.uniform(0.2, 0.8, size=(1, count, 1))) ** 2)
    e[:, :, 5] *= 0.75 + 0.5 * z[:, None]
    return torch.tensor(e, dtype=torch.float64, device="cuda")


def _images(ell, n):
    c = (torch.arange(n, device="cuda", dtype=torch.float32) - n / 2 + 0.5) * (2.0 / n)
    img = torch.zeros((ell.shape[0], n, n), device="cuda")
    e = ell.float()
    for s in range(ell.shape[0]):
        for k in range(ell.shape[1]):
            cx, cy, a, b, phi, rho = e[s, k].unbind()
            dx, dy = (c - cx)[None, :], (c - cy)[:, None]
            u = (dx * torch.cos(phi) + dy * torch.sin(phi)) / a
            v = (dy * torch.cos(phi) - dx * torch.sin(phi)) / b
            img[s] += rho * (u * u + v * v <= 1.0)
    return img


def _sinograms(ell, n, m, nd, gen):
    """Exact line integrals of the ellipses, with 1 % noise."""
    th = torch.arange(m, device="cuda", dtype=torch.float32) * (math.pi / m)
    t = torch.arange(nd, device="cuda", dtype=torch.float32) - 0.5 * (nd - 1)
    out = torch.zeros((ell.shape[0], m, nd), device="cuda")
    e = ell.float()
    h = n / 2.0
    for s in range(ell.shape[0]):
        for k in range(ell.shape[1]):
            cx, cy, a, b, phi, rho = e[s, k].unbind()
            sig2 = ((a * h * torch.cos(th - phi)) ** 2 + (b * h * torch.sin(th - phi)) ** 2)[:, None]
            tau = t[None, :] - h * (cx * torch.cos(th) + cy * torch.sin(th))[:, None]
            out[s] += 2 * rho * a * b * h * h * torch.sqrt((sig2 - tau * tau).clamp_min(0.0)) / sig2
        out[s] += 0.01 * out[s].square().mean().sqrt() * torch.randn((m, nd), device="cuda", generator=gen)
    return out


def _plan(case, n, m, nd):
    f = {k: k in case["flags"].split(",") for k in FLAGS}
    return xct.Plan(n, m, nd, case["storage"], cos_sin=inputs.angle_table(m), **f)


def _jobs(case):
    """(n, m, nd, S) of a batch's jobs: three geometries, four jobs."""
    n, m, nd, S = case["n"], case["m"], case["nd"], case["S"]
    half = (max(16, n // 2), max(16, m // 2), max(16, nd // 2))
    more = (max(16, 2 * n // 3), max(16, 2 * m // 3), max(16, 2 * nd // 3))
    return [(n, m, nd, S), (*half, max(1, S // 2)), (*more, S + 3), (*half, max(1, S // 3))]


def _data(case, seed):
    """The inputs of a case, from its seed alone."""
    n, m, nd, S, kind = (case[k] for k in ("n", "m", "nd", "S", "kind"))
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    if kind == "batch":
        return [_sinograms(_ellipses(rng, s), a, b, c, gen) for a, b, c, s in _jobs(case)]
    ell = _ellipses(rng, S)
    if kind in ("project", "plan", "project_matfree"):
        return _images(ell, n)
    if kind == "project_f64":
        return _images(ell, n).double()
    y = _sinograms(ell, n, m, nd, gen)
    if kind == "gradient":   # some way into a reconstruction: a blurred, scaled image
        x = torch.nn.functional.avg_pool2d(_images(ell, n)[:, None], 5, 1, 2)[:, 0] * 0.8
        return x, y
    return y


def prepare(case, seed):
    st = dict(case=case, data=_data(case, seed))
    if case["kind"] == "batch":
        shared = {}
        for a, b, c, _ in _jobs(case):
            if (a, b, c) not in shared:
                shared[a, b, c] = _plan(case, a, b, c)
        st["plans"] = [shared[j[:3]] for j in _jobs(case)]
    elif case["kind"] != "plan":
        st["plan"] = _plan(case, case["n"], case["m"], case["nd"])
    return st


def run(state):
    case, d = state["case"], state["data"]
    kind = case["kind"]
    if kind == "project":
        return state["plan"].project(d)
    if kind == "backproject":
        return state["plan"].backproject(d)
    if kind == "cgls":
        return state["plan"].cgls(d, case["iters"], resid=True)
    if kind == "project_f64":
        return state["plan"].project_f64(d)
    if kind == "gradient":
        x = d[0].detach().requires_grad_(True)
        loss = autograd.datafit(x, d[1], state["plan"]) + autograd.tv(x, 1e-3, 1e-3)
        (g,) = torch.autograd.grad(loss, x)
        return loss.detach(), g
    if kind == "batch":
        xs = [torch.empty((y.shape[0], p.n, p.n), device="cuda") for p, y in zip(state["plans"], d)]
        xct.xct_cgls_batch([(p.handle, y, x, y.shape[0]) for p, y, x in zip(state["plans"], d, xs)],
                           case["iters"])
        return xs
    if kind == "project_matfree":
        p = state["plan"]
        y = torch.empty((case["S"], p.m, p.nd), device="cuda")
        xct.xct_project_matfree(p.handle, d, y, case["S"])
        return y
    with _plan(case, case["n"], case["m"], case["nd"]) as plan:
        return plan.project(d)


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------

def _nnz(n, m, nd):
    """About the entries of A: a ray crosses 4 / pi pixels per unit of its
    length on average over the angles; a detector narrower than the grid's
    diagonal misses a part of it."""
    return int(4.0 / math.pi * m * n * n * min(1.0, nd / (1.08 * n)) ** 0.5)


def _product_bytes(case, n, m, nd, S):
    e = {"f32": 8, "f16": 4, "bf16": 4}[case["storage"]]
    return _nnz(n, m, nd) * e + (S * n * n + S * m * nd) * 4


def work(case):
    n, m, nd, S, kind = (case[k] for k in ("n", "m", "nd", "S", "kind"))
    nz = _nnz(n, m, nd)
    vec = 4 * S * (n * n + m * nd)
    prod = _product_bytes(case, n, m, nd, S)
    if kind in ("project", "backproject"):
        return {"bytes": prod, "flops": 2 * nz * S}
    if kind == "cgls":
        k = 2 * case["iters"] + 1
        return {"bytes": k * prod, "flops": 2 * nz * S * k}
    if kind == "gradient":
        return {"bytes": 2 * prod + vec, "flops": 4 * nz * S}
    if kind == "batch":
        k = 2 * case["iters"] + 1
        return {"bytes": sum(k * _product_bytes(case, *j) for j in _jobs(case)),
                "flops": sum(2 * _nnz(*j[:3]) * j[3] * k for j in _jobs(case))}
    if kind == "project_f64":
        return {"bytes": 12 * nz + 2 * vec, "flops": 2 * nz * S}
    if kind == "project_matfree":
        return {"bytes": vec, "flops": 2 * nz * S + 8 * nz}
    # a plan: A and its transpose are written once each, read once for the product
    return {"bytes": 3 * nz * 8 + vec, "flops": 16 * nz + 2 * nz * S}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------

class _Exact:
    """A as a float64 sparse matrix from a plain Siddon trace in torch."""

    def __init__(self, n, m, nd):
        dev = "cuda"
        cs = torch.tensor(inputs.angle_table(m), device=dev)
        t = torch.arange(nd, device=dev, dtype=torch.float64) - 0.5 * (nd - 1)
        planes = torch.arange(n + 1, device=dev, dtype=torch.float64) - n / 2
        self.n, self.m, self.nd = n, m, nd
        self.parts = []
        inf = torch.tensor(math.inf, device=dev, dtype=torch.float64)
        step = max(1, int(6e7 / ((2 * n + 2) * nd)))
        for k0 in range(0, m, step):
            c, s = cs[k0:k0 + step, 0:1], cs[k0:k0 + step, 1:2]
            px, py = (t * c).reshape(-1, 1), (t * s).reshape(-1, 1)
            dx = (-s).expand(-1, nd).reshape(-1, 1)
            dy = c.expand(-1, nd).reshape(-1, 1)
            ax, ay = (planes - px) / dx, (planes - py) / dy
            flat_x, flat_y = dx == 0, dy == 0
            inside = ~((flat_x & (px.abs() > n / 2)) | (flat_y & (py.abs() > n / 2)))
            lo = torch.maximum(torch.where(flat_x, -inf, ax.amin(1, True)), torch.where(flat_y, -inf, ay.amin(1, True)))
            hi = torch.minimum(torch.where(flat_x, inf, ax.amax(1, True)), torch.where(flat_y, inf, ay.amax(1, True)))
            hi = torch.where(inside & (hi > lo), hi, lo)
            a = torch.cat([torch.where(flat_x, lo, ax), torch.where(flat_y, lo, ay)], 1)
            a = torch.minimum(torch.maximum(a, lo), hi).sort(1).values
            ln, mid = a[:, 1:] - a[:, :-1], 0.5 * (a[:, 1:] + a[:, :-1])
            keep = ln >= 1e-9
            ix = (px + mid * dx + n / 2).floor().clamp(0, n - 1)
            iy = (py + mid * dy + n / 2).floor().clamp(0, n - 1)
            col = (iy * n + ix)[keep].to(torch.int32)
            crow = torch.zeros(keep.shape[0] + 1, dtype=torch.int32, device=dev)
            crow[1:] = keep.sum(1).cumsum(0).to(torch.int32)
            self.parts.append((k0 * nd, crow, col, ln[keep]))

    def _mats(self):
        for r0, crow, col, val in self.parts:
            yield r0, torch.sparse_csr_tensor(crow, col, val, (crow.numel() - 1, self.n * self.n))

    def project(self, x):
        """[S, n, n] float64 -> [S, m, nd]"""
        X = x.reshape(x.shape[0], -1).t().contiguous()
        y = torch.cat([a @ X for _, a in self._mats()])
        return y.t().reshape(-1, self.m, self.nd)

    def backproject(self, y):
        Y = y.reshape(y.shape[0], -1).t().contiguous()
        x = torch.zeros((self.n * self.n, Y.shape[1]), dtype=torch.float64, device="cuda")
        for r0, crow, col, val in self.parts:
            # the transpose's rows, from a sort of the entries by column
            rows = torch.repeat_interleave(torch.arange(crow.numel() - 1, device="cuda", dtype=torch.int32),
                                           (crow[1:] - crow[:-1]).long())
            col_s, at = col.sort(stable=True)
            tcrow = torch.zeros(self.n * self.n + 1, dtype=torch.int32, device="cuda")
            tcrow[1:] = torch.bincount(col_s, minlength=self.n * self.n).cumsum(0).to(torch.int32)
            t = torch.sparse_csr_tensor(tcrow, rows[at], val[at], (self.n * self.n, crow.numel() - 1))
            x += t @ Y[r0:r0 + crow.numel() - 1]
        return x.t().reshape(-1, self.n, self.n)

    def cgls(self, y, iters):
        dot = lambda v: v.reshape(v.shape[0], -1).square().sum(1)  # noqa: E731
        x = torch.zeros((y.shape[0], self.n, self.n), dtype=torch.float64, device="cuda")
        r = y.clone()
        s = self.backproject(r)
        p, gamma = s.clone(), dot(s)
        log = [torch.stack([dot(r).sqrt(), gamma.sqrt()], 1)]
        for _ in range(iters):
            q = self.project(p)
            alpha = (gamma / dot(q))[:, None, None]
            x += alpha * p
            r -= alpha * q
            s = self.backproject(r)
            new = dot(s)
            p = s + (new / gamma)[:, None, None] * p
            gamma = new
            log.append(torch.stack([dot(r).sqrt(), gamma.sqrt()], 1))
        return x, torch.stack(log)


def exact(case, seed):
    n, m, nd, S, kind = (case[k] for k in ("n", "m", "nd", "S", "kind"))
    if _nnz(n, m, nd) * max(S, 8) * (2 * case["iters"] + 1) > 2.5e11:
        return None
    d = _data(case, seed)
    if kind == "batch":
        return [_Exact(*j[:3]).cgls(y.double(), case["iters"])[0] for j, y in zip(_jobs(case), d)]
    A = _Exact(n, m, nd)
    if kind in ("project", "plan", "project_f64", "project_matfree"):
        return A.project(d.double())
    if kind == "backproject":
        return A.backproject(d.double())
    if kind == "cgls":
        return A.cgls(d.double(), case["iters"])
    x, y = d[0].double(), d[1].double()
    r = A.project(x) - y
    eps, lam = 1e-3, 1e-3
    dx = torch.zeros_like(x)
    dy = torch.zeros_like(x)
    dx[:, :, :-1] = x[:, :, 1:] - x[:, :, :-1]
    dy[:, :-1, :] = x[:, 1:, :] - x[:, :-1, :]
    q = torch.sqrt(dx * dx + dy * dy + eps * eps)
    g = A.backproject(r) - lam * (dx + dy) / q
    g[:, :, 1:] += lam * (dx / q)[:, :, :-1]
    g[:, 1:, :] += lam * (dy / q)[:, :-1, :]
    return 0.5 * r.square().sum() + lam * q.sum(), g
