"""The work that users of this framework have it do, as cases that can be timed and compared.

A case is one call sequence of a program built on the public entry points: a solve of problem (7)
(class probabilities in, hidden field and trace out), the z-update operator alone (with a handle
and without one), a batch of uneven images, a solve behind the MLR class model, and the
gradient of an unrolled solve. Sizes are those of the repository's own workloads (64 x 64,
145 x 145, 256 x 256, 610 x 340, 2048 x 2048, the uneven batch, the patch-size sweep) and generic
ones between them. Inputs are drawn on the GPU with the distributions of those workloads: Voronoi
label maps, noisy logits, softmax.
"""
import math
import random

import numpy as np
import torch

from paper_1504_07028_gb300 import binding as B
from paper_1504_07028_gb300.autograd import UnrolledSegSalsa

DEV = "cuda"


def _solve(name, H, W, K, M, sp, iters, trace=0, precision="fp32", g4="affine", sigma=None, lam=1.5):
    return {"name": name, "kind": "solve", "H": H, "W": W, "K": K, "M": M, "p": sp, "iters": iters,
            "trace": trace, "precision": precision, "g4": g4, "lam": lam,
            "sigma": sigma if sigma is not None else max(1, M) / 2.0}


def _grad(name, H, W, K, iters, every, precision, M=1, sp="1", lam=2.0):
    return {"name": name, "kind": "grad", "H": H, "W": W, "K": K, "M": M, "p": sp, "iters": iters,
            "every": every, "precision": precision, "sigma": max(1, M) / 2.0, "lam": lam}


def listed():
    return [
        # the z-update operator of one scene for a caller without a handle: the smallest call,
        # asynchronous on the caller's stream
        {"name": "zupdate_static_145x145_k16", "kind": "static", "H": 145, "W": 145, "K": 16},
        # an interactive solve of a small crop: launches and latency count
        _solve("solve_64x64_k4", 64, 64, 4, 1, "1", 200, lam=2.0),
        # the same crop in double precision (the reference runs of a study)
        _solve("solve_64x64_k4_fp64", 64, 64, 4, 1, "1", 200, precision="fp64", lam=2.0),
        # the shape of the Indian Pines subscene, traced, as an experiment logs it
        _solve("solve_145x145_k16", 145, 145, 16, 1, "1", 300, trace=10),
        # its variants: the spectral norm prior with g4 on the probability simplex
        _solve("solve_145x145_k16_inf_simplex", 145, 145, 16, 1, "inf", 100, g4="simplex"),
        # one solve of the patch-size study: 9 x 9 patch
        _solve("solve_145x145_k16_9x9", 145, 145, 16, 4, "1", 100),
        # the shape of a university scene: MLR class model from 103 bands, 5 x 5 patch
        {"name": "mlr_610x340_d103_k9_5x5", "kind": "mlr", "H": 610, "W": 340, "K": 9, "d": 103, "M": 2,
         "p": "1", "iters": 200, "sigma": 1.0, "lam": 1.5},
        # learning the prior from crops: an unrolled network of five iterations, single precision
        # (a solve is piecewise smooth: over many iterations of a large field some entry sits
        # within a rounding error of a switch, and single-precision gradients of the same
        # accuracy then differ there)
        _grad("grad_64x64_k4_unroll5", 64, 64, 4, 5, 5, "fp32"),
        # the gradient of a whole scene's solve, in the precision it is checked in
        _grad("grad_256x256_k8_fp64", 256, 256, 8, 20, 10, "fp64"),
        # a serving batch of uneven images (sizes and class counts drawn from `sizes`)
        {"name": "batch_16_uneven", "kind": "batch", "images": 16, "sizes": 5000, "lo": 96, "hi": 512,
         "iters": 100},
        # a large image with a 5 x 5 patch
        _solve("solve_1024x1024_k16_5x5", 1024, 1024, 16, 2, "1", 50, sigma=1.0),
        # the largest scene, traced
        _solve("solve_2048x2048_k16", 2048, 2048, 16, 1, "1", 100, trace=10, lam=2.0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Another case of the same ranges: sizes over their logarithm, every option in use."""
    kind = rng.choice(["static", "linear", "solve", "solve", "solve", "solve", "mlr", "grad", "batch"])
    if kind == "static":
        K = rng.randint(2, 20)
        while True:
            H, W = _log(rng, 24, 700), _log(rng, 24, 700)
            if H * (W // 2 + 1) * K <= 2 << 20:
                return {"kind": kind, "H": H, "W": W, "K": K}
    if kind == "linear":
        return {"kind": kind, "H": _log(rng, 32, 1500), "W": _log(rng, 32, 1500), "K": rng.randint(2, 20),
                "precision": rng.choice(["fp32", "fp32", "fp32", "fp64"])}
    if kind == "solve":
        M = rng.choice([0, 1, 1, 1, 1, 2, 2, 3, 4, 5])
        precision = "fp64" if rng.random() < 0.15 else "fp32"
        top = 200 if precision == "fp64" or M > 2 else 1200
        c = _solve("", _log(rng, 40, top), _log(rng, 40, top), rng.randint(2, 20), M,
                   rng.choice(["1", "1", "2", "inf"]), rng.randint(20, 60), trace=rng.choice([0, 10]),
                   precision=precision, g4=rng.choice(["affine", "affine", "affine", "simplex"]),
                   lam=rng.choice([1.0, 1.5, 2.0]))
        del c["name"]
        return c
    if kind == "mlr":
        return {"kind": kind, "H": _log(rng, 100, 700), "W": _log(rng, 100, 700), "K": rng.randint(4, 16),
                "d": rng.randint(20, 224), "M": rng.choice([1, 2]), "p": rng.choice(["1", "2"]),
                "iters": rng.randint(20, 60), "sigma": 1.0, "lam": 1.5}
    if kind == "grad":
        fp64 = rng.random() < 0.5
        top = 256 if fp64 else 72
        c = _grad("", _log(rng, 24, top), _log(rng, 24, top), rng.randint(3, 8), rng.randint(5, 20) if fp64 else 5,
                  rng.choice([5, 10]), "fp64" if fp64 else "fp32", rng.choice([0, 1, 1, 2] if fp64 else [0, 1, 1]),
                  rng.choice(["1", "2"]),
                  rng.choice([1.0, 2.0]))
        del c["name"]
        return c
    return {"kind": "batch", "images": rng.randint(3, 10), "sizes": rng.randint(0, 10 ** 6), "lo": 96,
            "hi": rng.choice([256, 512]), "iters": rng.randint(20, 60)}


# --------------------------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _labels(g, H, W, K, S):
    """Voronoi label map: S seed points, each pixel takes its nearest one, seed j carries j mod K."""
    pts = torch.rand(S, 2, generator=g, device=DEV) * torch.tensor([H, W], device=DEV, dtype=torch.float32)
    ys = torch.arange(H, device=DEV, dtype=torch.float32) + 0.5
    xs = torch.arange(W, device=DEV, dtype=torch.float32) + 0.5
    best = torch.full((H, W), float("inf"), device=DEV)
    arg = torch.zeros(H, W, device=DEV, dtype=torch.long)
    for j in range(S):
        d = (ys[:, None] - pts[j, 0]) ** 2 + (xs[None, :] - pts[j, 1]) ** 2
        arg = torch.where(d < best, torch.full_like(arg, j), arg)
        best = torch.minimum(d, best)
    return arg % K


def _logits(seed, H, W, K, dtype=torch.float32):
    """(K, H, W) logits 3 onehot(y) + N(0, 1), and the labels y."""
    g = _gen(seed)
    y = _labels(g, H, W, K, min(64, 4 * K))
    lg = torch.randn(K, H, W, generator=g, device=DEV, dtype=dtype)
    return lg.scatter_add_(0, y[None], torch.full((1, H, W), 3.0, device=DEV, dtype=dtype)), y


def _dtype(case):
    return torch.float64 if case.get("precision") == "fp64" else torch.float32


def _probs(case, seed):
    return torch.softmax(_logits(seed, case["H"], case["W"], case["K"], _dtype(case))[0], 0)


def _spectra(case, seed):
    """BF16 spectra (H, W, d) around class means and MLR weights (K, d) with an expected margin
    of about 2."""
    g = _gen(seed)
    H, W, K, d = case["H"], case["W"], case["K"], case["d"]
    y = _labels(g, H, W, K, min(64, 4 * K))
    mu = torch.rand(K, d, generator=g, device=DEV)
    x = mu[y] + 0.05 * torch.randn(H, W, d, generator=g, device=DEV)
    w = (24.0 / d) * (mu - mu.mean(0)) + torch.randn(K, d, generator=g, device=DEV) / math.sqrt(d)
    return x.bfloat16(), w.bfloat16()


def _sizes(case):
    r = random.Random(case["sizes"])
    return [(r.randint(case["lo"], case["hi"]), r.randint(case["lo"], case["hi"]), r.choice([4, 8, 16]))
            for _ in range(case["images"])]


def _rhs(case, seed):
    g = _gen(seed)
    return torch.randn(case["H"], case["W"], case["K"], generator=g, device=DEV, dtype=_dtype(case))


def _image(case, H, W, K):
    return dict(H=H, W=W, K=K, M=1, p="1", iters=case["iters"], sigma=0.5, lam=2.0)


def _params(c):
    p = c.get("p", "1")
    return B.make_params(c["H"], c["W"], c["K"], M=c.get("M", 1), sigma=c.get("sigma", 0.5),
                         lam=c.get("lam", 1.5), mu=1.0, schatten_p="inf" if p == "inf" else int(p),
                         precision=c.get("precision", "fp32"))


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case, "kind": kind}
    if kind in ("static", "linear"):
        st["rhs"] = _rhs(case, seed)
        st["z"] = torch.empty_like(st["rhs"])
        if kind == "linear":
            st["s"] = B.Solver(_params(case))
        return st
    if kind == "batch":
        images = [_image(case, *s) for s in _sizes(case)]
        st["b"] = B.Batch([_params(c) for c in images])
        st["p"] = [_probs(c, seed + 7919 * i) for i, c in enumerate(images)]
        st["z"] = [torch.empty_like(p) for p in st["p"]]
        return st
    st["s"] = B.Solver(_params(case))
    if kind == "solve":
        st["s"].set_g4(case["g4"])
        st["p"] = _probs(case, seed)
        st["z"] = torch.empty_like(st["p"])
    elif kind == "mlr":
        st["x"], st["w"] = _spectra(case, seed)
        st["z"] = torch.empty(case["K"], case["H"], case["W"], device=DEV)
    else:
        st["log_p"], st["cot"], st["lam"], st["omega"] = _grad_inputs(case, seed)
    return st


def _grad_inputs(case, seed):
    logits, y = _logits(seed, case["H"], case["W"], case["K"], _dtype(case))
    # the loss is the expected count of wrong pixels, sum_i 1 - z_i[y_i]
    cot = torch.zeros_like(logits).scatter_(0, y[None], -1.0)
    return (torch.log_softmax(logits, 0).requires_grad_(), cot,
            torch.tensor(case["lam"], dtype=logits.dtype, device=DEV, requires_grad=True),
            torch.tensor(_omega(case), dtype=logits.dtype, device=DEV, requires_grad=True))


def run(state):
    case, kind = state["case"], state["kind"]
    if kind == "static":
        rc = B.segsalsa_str_linear_solve_static(state["rhs"], state["z"])
        if rc != B.SEGSALSA_OK:
            raise RuntimeError("linear_solve_static: %d" % rc)
        return state["z"]
    if kind == "linear":
        return state["s"].linear_solve(state["rhs"], state["z"])
    if kind == "batch":
        b = state["b"]
        for i, p in enumerate(state["p"]):
            b.image(i).set_probs(p)
        b.solve(case["iters"])
        for i, z in enumerate(state["z"]):
            b.image(i).get_z(z)
        return state["z"]
    s = state["s"]
    if kind == "grad":
        lp, lam, om = state["log_p"], state["lam"], state["omega"]
        z = UnrolledSegSalsa.apply(lp, lam, om, s, case["iters"], case["every"])
        g = torch.autograd.grad(z, (lp, lam, om), state["cot"])
        return {"z": z, "log_p": g[0], "lam": g[1], "omega": g[2]}
    if kind == "mlr":
        s.set_spectra(state["x"], state["w"])
        s.solve(case["iters"])
        return {"z": s.get_z(state["z"])}
    s.set_probs(state["p"])
    trace = s.solve(case["iters"], trace_every=case["trace"])
    out = {"z": s.get_z(state["z"])}
    if trace is not None:
        # the log keeps the rows in the precision of the solve
        out["trace"] = trace.astype(s.dtype)
    return out


# ------------------------------------------------------------------------------ work model
def _iteration(H, W, K, M, size):
    """Bytes and operations of one SALSA iteration: the prior's dual (L pairs), d3 and the
    right-hand side read and written, p read, z read and written; per shift and class two
    differences, the Gram sums, the prox, the dual and J^T, and the z-update's two transforms."""
    L = (2 * M + 1) ** 2
    n = float(H) * W * K
    return size * n * (4 * L + 7), n * (28 * L + 40 + 10 * math.log2(max(2, W)))


def work(case):
    kind, size = case["kind"], 8 if case.get("precision") == "fp64" else 4
    if kind == "batch":
        each = [_iteration(H, W, K, 1, 4) for H, W, K in _sizes(case)]
        return {"bytes": case["iters"] * sum(e[0] for e in each), "flops": case["iters"] * sum(e[1] for e in each)}
    n = float(case["H"]) * case["W"] * case["K"]
    if kind in ("static", "linear"):
        return {"bytes": 2 * size * n, "flops": n * (10 * math.log2(max(2, case["W"])) + 8)}
    b, f = _iteration(case["H"], case["W"], case["K"], case["M"], size)
    if kind == "grad":  # the forward pass, its recomputation, and a unit of about the same size
        return {"bytes": 3 * case["iters"] * b, "flops": 4 * case["iters"] * f}
    extra = 2 * n * case["d"] if kind == "mlr" else 0.0
    more = 2.0 * case["H"] * case["W"] * case["d"] if kind == "mlr" else 0.0
    return {"bytes": case["iters"] * b + 2 * size * n + more, "flops": case["iters"] * f + extra}


# --------------------------------------------------------- the same results in 64 bits (torch)
def _omega(c):
    M, s = c.get("M", 1), c.get("sigma", 0.5)
    g = np.array([math.exp(-(dy * dy + dx * dx) / (2 * s * s))
                  for dy in range(-M, M + 1) for dx in range(-M, M + 1)])
    return np.sqrt(g / g.sum())


def _operator_inverse(rhs, c):
    """(3 I + c (D_h^T D_h + D_v^T D_v))^{-1} rhs over the last two axes, periodic."""
    H, W = rhs.shape[-2:]
    ky = torch.arange(H, device=rhs.device, dtype=torch.float64) * (math.pi / H)
    kx = torch.arange(W // 2 + 1, device=rhs.device, dtype=torch.float64) * (math.pi / W)
    den = 3.0 + 4.0 * c * (torch.sin(ky)[:, None] ** 2 + torch.sin(kx)[None, :] ** 2)
    return torch.fft.irfft2(torch.fft.rfft2(rhs) / den, s=(H, W))


def _shrink(a, b, c, tau, sp):
    """The symmetric matrix A of the Schatten prox u = v A from the Gram entries a, b, c."""
    if sp == "2":
        g = torch.clamp(1 - tau / torch.sqrt(a + c), min=0.0)
        return g, torch.zeros_like(g), g
    hd = 0.5 * (a - c)
    r = torch.sqrt(hd * hd + b * b)
    s1 = torch.sqrt(0.5 * (a + c) + r)
    s2 = torch.sqrt(torch.clamp(0.5 * (a + c) - r, min=1e-300))
    if sp == "1":
        g1, g2 = torch.clamp(1 - tau / s1, min=0.0), torch.clamp(1 - tau / s2, min=0.0)
    else:
        both = 0.5 * (s1 + s2 - tau)
        one = s1 - s2 >= tau
        none = s1 + s2 <= tau
        g1 = torch.where(none, 0.0, torch.where(one, 1 - tau / s1, both / s1))
        g2 = torch.where(none, 0.0, torch.where(one, 1.0, both / s2))
    kap = (g1 - g2) / (2 * r)
    m = 0.5 * (g1 + g2)
    return m + kap * hd, kap * b, m - kap * hd


def _to_simplex(v):
    s, _ = torch.sort(v, dim=0, descending=True)
    k = torch.arange(1, v.shape[0] + 1, device=v.device, dtype=v.dtype).view(-1, 1, 1)
    t = (torch.cumsum(s, 0) - 1) / k
    rho = (s > t).sum(0, keepdim=True) - 1
    return torch.clamp(v - t.gather(0, rho), min=0.0)


def _prior(z, om2, M, sp):
    gh, gv = torch.roll(z, -1, 2) - z, torch.roll(z, -1, 1) - z
    a, b, c = (gh * gh).sum(0), (gh * gv).sum(0), (gv * gv).sum(0)
    A = B_ = C = 0.0
    for j, (dy, dx) in enumerate(_shifts(M)):
        A = A + om2[j] * torch.roll(a, (-dy, -dx), (0, 1))
        B_ = B_ + om2[j] * torch.roll(b, (-dy, -dx), (0, 1))
        C = C + om2[j] * torch.roll(c, (-dy, -dx), (0, 1))
    r = torch.sqrt(0.25 * (A - C) ** 2 + B_ * B_)
    s1, s2 = torch.sqrt(0.5 * (A + C) + r), torch.sqrt(torch.clamp(0.5 * (A + C) - r, min=0.0))
    return {"1": (s1 + s2).sum(), "2": torch.sqrt(A + C).sum(), "inf": s1.sum()}[sp]


def _shifts(M):
    return [(dy, dx) for dy in range(-M, M + 1) for dx in range(-M, M + 1)]


def _iterate(p, omega, lam, c, trace=0):
    """`iters` iterations (12)-(14) from z = p / 1^T p, u = G z, d = 0 on (K, H, W) doubles;
    differentiable in p, omega and lam."""
    M, sp, iters, simplex = c["M"], c["p"], c["iters"], c.get("g4") == "simplex"
    mu, K = 1.0, p.shape[0]
    cw = (omega * omega).sum()
    z = p / p.sum(0, keepdim=True)
    d1 = d3 = d4 = torch.zeros_like(z)
    dh = [0.0] * len(_shifts(M))
    dv = list(dh)
    pp = (p * p).sum(0, keepdim=True)
    rhs, rows = None, []
    for k in range(1, iters + 1):
        logged = trace and (k % trace == 0 or k == iters)
        if k > 1:
            if omega.requires_grad:  # the operator depends on the weights: solve by its symbol
                z = _Inverse.apply(rhs, cw)
            else:
                z = _operator_inverse(rhs, float(cw))
        gh, gv = torch.roll(z, -1, 2) - z, torch.roll(z, -1, 1) - z
        a = b = cc = 0.0
        vh, vv = [], []
        for j, (dy, dx) in enumerate(_shifts(M)):
            h = omega[j] * torch.roll(gh, (-dy, -dx), (1, 2)) - dh[j]
            v = omega[j] * torch.roll(gv, (-dy, -dx), (1, 2)) - dv[j]
            vh.append(h)
            vv.append(v)
            a, b, cc = a + (h * h).sum(0), b + (h * v).sum(0), cc + (v * v).sum(0)
        A11, A12, A22 = _shrink(a, b, cc, lam / mu, sp)
        v1, v3, v4 = z - d1, z - d3, z - d4
        pv = (p * v1).sum(0, keepdim=True)
        t = 0.5 * (pv + torch.sqrt(pv * pv + 4 * pp / mu))
        n1 = p / (mu * t)
        n3 = torch.clamp(v3, min=0.0) - v3
        n4 = _to_simplex(v4) - v4 if simplex else (-(v4.sum(0, keepdim=True) - 1) / K).expand_as(v4)
        sh = sv = qh = qv = 0.0
        change = ((n1 - d1) ** 2 + (n3 - d3) ** 2 + (n4 - d4) ** 2).sum() if logged else 0.0
        for j, (dy, dx) in enumerate(_shifts(M)):
            uh, uv = vh[j] * A11 + vv[j] * A12, vh[j] * A12 + vv[j] * A22
            nh, nv = uh - vh[j], uv - vv[j]
            vh[j] = vv[j] = None
            sh = sh + torch.roll(omega[j] * (uh + nh), (dy, dx), (1, 2))
            sv = sv + torch.roll(omega[j] * (uv + nv), (dy, dx), (1, 2))
            if logged:
                change = change + ((nh - dh[j]) ** 2 + (nv - dv[j]) ** 2).sum()
                qh = qh + torch.roll(omega[j] * nh, (dy, dx), (1, 2))
                qv = qv + torch.roll(omega[j] * nv, (dy, dx), (1, 2))
            dh[j], dv[j] = nh, nv
        back = torch.roll(sh, 1, 2) - sh + torch.roll(sv, 1, 1) - sv
        rhs = (v1 + 2 * n1) + (v3 + 2 * n3) + (v4 + 2 * n4) + back
        d1, d3, d4 = n1, n3, n4
        if logged:
            gtd = n1 + n3 + n4 + torch.roll(qh, 1, 2) - qh + torch.roll(qv, 1, 1) - qv
            zp = _to_simplex(z)
            obj = -torch.log((p * zp).sum(0)).sum() + lam * _prior(zp, omega * omega, M, sp)
            rows.append([float(k), math.sqrt(float(change)), mu * math.sqrt(float((gtd * gtd).sum())), float(obj),
                         float(z.min()), float((z.sum(0) - 1).abs().max())])
    return z, np.array(rows)


class _Inverse(torch.autograd.Function):
    """A(c)^{-1} rhs with the gradients for rhs and c: z = A^{-1} r, dr = A^{-1} dz,
    dc = -<dr, (D_h^T D_h + D_v^T D_v) z>."""

    @staticmethod
    def forward(ctx, rhs, c):
        z = _operator_inverse(rhs, float(c))
        ctx.save_for_backward(z)
        ctx.c = float(c)
        return z

    @staticmethod
    def backward(ctx, zbar):
        (z,) = ctx.saved_tensors
        r = _operator_inverse(zbar, ctx.c)
        dc = sum(((torch.roll(r, -1, a) - r) * (torch.roll(z, -1, a) - z)).sum() for a in (1, 2))
        return r, -dc


def exact(case, seed):
    kind = case["kind"]
    if kind in ("static", "linear"):
        z = _operator_inverse(_rhs(case, seed).double().permute(2, 0, 1).contiguous(), 1.0)
        return z.permute(1, 2, 0).contiguous()
    if kind == "batch":
        out = []
        for i, s in enumerate(_sizes(case)):
            c = _image(case, *s)
            om = torch.tensor(_omega(c), device=DEV)
            with torch.no_grad():
                out.append(_iterate(_probs(c, seed + 7919 * i).double(), om, c["lam"], c)[0])
        return out
    om = torch.tensor(_omega(case), device=DEV)
    if kind == "grad":
        lp, cot, lam, om = (t.detach().double() for t in _grad_inputs(case, seed))
        for t in (lp, lam, om):
            t.requires_grad_()
        z, _ = _iterate(torch.exp(lp), om, lam, case)
        g = torch.autograd.grad(z, (lp, lam, om), cot)
        return {"z": z.detach(), "log_p": g[0], "lam": g[1], "omega": g[2]}
    with torch.no_grad():
        if kind == "mlr":
            x, w = _spectra(case, seed)
            lg = x.double() @ w.double().T
            p = torch.softmax(lg, -1).permute(2, 0, 1).contiguous()
            return {"z": _iterate(p, om, case["lam"], case)[0]}
        z, rows = _iterate(_probs(case, seed).double(), om, case["lam"], case, trace=case["trace"])
    return {"z": z, "trace": rows} if case["trace"] else {"z": z}
