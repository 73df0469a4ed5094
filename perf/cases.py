"""Workloads whose speed this framework is judged by, one pass each through the
public calls of ``paper_1707_02244_gb300``.

Families (a case is a dict of plain values; ``family`` selects the calls):

``product``   y = A x and A^T y on a plan (cs_forward, cs_adjoint)
``static``    C x and C^T x with no plan (cs_circulant_apply_static)
``ista``      one ISTA solve from x = 0 (cs_ista)
``recover``   step size by power iteration, then an ISTA solve with its
              convergence record (cs_opnorm2, cs_ista)
``admm``      one ADMM solve from the zero state (cs_admm)
``deblur2d``  ISTA and ADMM on a blurred, subsampled star field (cs_plan_2d)
``batch``     ISTA and ADMM on many instances of uneven size in one call
``grad``      gradient of unrolled ISTA (cs_grad)
``grad_admm`` gradient of unrolled ADMM (cs_grad_admm)

Inputs follow the recipes of the tests and the benchmark: c ~ N(0, 1/m), a
sparse signal x*, y = A x* + noise, formed in 64 bits and rounded once.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1707_02244_gb300 as cs

F64 = torch.float64


def _lg(n):
    return math.log2(n)


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # one product each way on a small plan: the latency of a single call
        {"name": "product_n1024", "family": "product", "n": 1024, "m": 307},
        # a product inside code that may not allocate, at the largest length
        {"name": "static_n16384", "family": "static", "n": 16384},
        # plain 1D ISTA of the small configuration, with the convergence
        # record that the call returns by default
        {"name": "ista_n4096", "family": "ista", "n": 4096, "m": 1024, "k": 64, "noise": 0.0, "lam": 1e-3,
         "iters": 500, "stats": True},
        # ADMM at a size of the paper's sweep: m = n/2, k = n/10
        {"name": "admm_n32768", "family": "admm", "n": 1 << 15, "m": 1 << 14, "k": 3277, "noise": 1e-3, "lam": 1e-3,
         "rho": 1.0, "iters": 200, "stats": True},
        # a VGA-sized signal with an odd number of rows, from the step size to
        # the solution
        {"name": "recover_n262144", "family": "recover", "n": 1 << 18, "m": 87381, "k": 1311, "noise": 1e-3,
         "lam": 5e-3, "power": 50, "iters": 100},
        # the large 1D instance, ISTA
        {"name": "ista_n4194304", "family": "ista", "n": 1 << 22, "m": 1 << 20, "k": 20971, "noise": 1e-4,
         "lam": 5e-3, "iters": 100, "stats": False},
        # the large 1D instance, ADMM
        {"name": "admm_n4194304", "family": "admm", "n": 1 << 22, "m": 1 << 20, "k": 20971, "noise": 1e-4,
         "lam": 5e-3, "rho": 1.0, "iters": 100, "stats": False},
        # compressed deblurring of a 4096 x 4096 star field, a third of the
        # pixels kept
        {"name": "deblur2d_4096x4096", "family": "deblur2d", "n0": 4096, "n1": 4096, "m": 5592405, "k": 20000,
         "iters": 10},
        # many independent instances, 7-smooth lengths between 2^12 and 2^20
        {"name": "batch_smooth_96", "family": "batch", "count": 96, "lg_lo": 12.0, "lg_hi": 20.0, "snap": "smooth",
         "size_seed": 17, "iters": 20},
        # many independent instances, power-of-two lengths
        {"name": "batch_pow2_256", "family": "batch", "count": 256, "lg_lo": 8.0, "lg_hi": 17.0, "snap": "pow2",
         "size_seed": 18, "iters": 50},
        # calibration by gradient descent: unrolled ISTA of the large
        # differentiable configuration, checkpoints every 25 steps
        {"name": "grad_n1048576", "family": "grad", "n": 1 << 20, "m": 1 << 18, "k": 655, "lam": 0.5, "T": 75,
         "K": 25},
        # the same through ADMM, at a middle size and an odd number of rows
        {"name": "grad_admm_n262144", "family": "grad_admm", "n": 1 << 18, "m": 65537, "k": 163, "lam": 0.5,
         "rho": 1.0, "T": 60, "K": 25},
    ]


def _log_uniform(rng, lo, hi):
    return 2.0 ** rng.uniform(_lg(lo), _lg(hi))


def _pow2(rng, lg_lo, lg_hi):
    return 1 << rng.randint(lg_lo, lg_hi)


def _rows_kept(rng, n):
    """m/n between 1/5 and 1/2, odd values among them."""
    return max(1, int(n * rng.uniform(0.2, 0.5)))


def draw(rng):
    family = rng.choice(["product", "static", "ista", "ista", "recover", "admm", "admm", "deblur2d", "batch", "batch",
                         "grad", "grad_admm"])
    if family == "product":
        n = _pow2(rng, 6, 22)
        return {"family": family, "n": n, "m": _rows_kept(rng, n)}
    if family == "static":
        return {"family": family, "n": _pow2(rng, 6, 14)}
    if family in ("ista", "recover", "admm"):
        n = _pow2(rng, 8, 22)
        m = _rows_kept(rng, n)
        c = {"family": family, "n": n, "m": m, "k": max(1, int(n * rng.uniform(0.005, 0.02))),
             "noise": rng.choice([0.0, 1e-4, 1e-3]), "lam": rng.choice([1e-3, 5e-3]), "iters": rng.randint(20, 100)}
        if family == "admm":
            c["rho"] = rng.choice([0.5, 1.0, 2.0])
        if family == "recover":
            c["power"] = rng.randint(20, 50)
        else:
            c["stats"] = rng.random() < 0.5
        return c
    if family == "deblur2d":
        n0, n1 = _pow2(rng, 5, 12), _pow2(rng, 5, 12)
        n = n0 * n1
        return {"family": family, "n0": n0, "n1": n1, "m": max(1, int(n * rng.uniform(0.25, 0.5))),
                "k": max(1, n // 839), "iters": rng.randint(4, 10)}
    if family == "batch":
        snap = rng.choice(["smooth", "pow2"])
        lo = rng.uniform(8.0, 13.0) if snap == "pow2" else rng.uniform(10.0, 13.0)
        hi = lo + rng.uniform(2.0, 20.0 - lo)
        # the total length is held near the listed cases'
        count = max(4, min(256, int(2.0 ** (23.5 - hi) * rng.uniform(1.0, 4.0))))
        return {"family": family, "count": count, "lg_lo": round(lo, 2), "lg_hi": round(hi, 2), "snap": snap,
                "size_seed": rng.randint(1, 1 << 20), "iters": rng.randint(10, 20)}
    n = _pow2(rng, 12, 20 if family == "grad" else 18)
    T = rng.randint(20, 60)
    c = {"family": family, "n": n, "m": max(1, int(n * rng.uniform(0.22, 0.3))), "k": max(1, n // 1600), "lam": 0.5,
         "T": T, "K": rng.randint(max(1, T // 4), T)}
    if family == "grad_admm":
        c["rho"] = 1.0
    return c


# ---------------------------------------------------------------- the inputs

def _device():
    return torch.device("cuda", torch.cuda.current_device())


def _gen(seed):
    g = torch.Generator(device=_device())
    g.manual_seed(int(seed))
    return g


def _normal(g, n):
    return torch.randn(n, generator=g, device=_device(), dtype=F64)


def _pick(g, n, m):
    """m distinct indices below n, in draw order."""
    return torch.randperm(n, generator=g, device=_device())[:m]


def _instance(case, g, bounded=False):
    """c, rows, y (64-bit tensors) of one 1D instance.  `bounded`: amplitudes
    +-[1, 2] instead of N(0, 1)."""
    n, m, k = case["n"], case["m"], min(case.get("k", 1), case["n"])
    c = _normal(g, n) / math.sqrt(m)
    rows = _pick(g, n, m)
    x = torch.zeros(n, device=_device(), dtype=F64)
    amp = _normal(g, k)
    if bounded:
        amp = torch.sign(amp) * (1.0 + torch.rand(k, generator=g, device=_device(), dtype=F64))
    x[_pick(g, n, k)] = amp
    y = _fwd(torch.fft.rfft(c), rows, x)
    if case.get("noise", 0.0) > 0.0:
        y = y + case["noise"] * _normal(g, m)
    return c, rows, y.float()


def _lipschitz(c):
    """max |c^|^2 >= ||A||^2: 1 over it is a valid ISTA step."""
    return float(torch.fft.rfft(c).abs().square().max())


def _f32(v):
    return float(np.float32(v))


def _sizes(case):
    """n and m of a batch's instances, from the case alone."""
    g = np.random.Generator(np.random.PCG64(case["size_seed"]))
    lg = g.uniform(case["lg_lo"], case["lg_hi"], case["count"])
    if case["snap"] == "pow2":
        n = (2.0 ** np.round(lg)).astype(np.int64)
    else:
        top = 1 << 20
        v = sorted(a * b * c * d for a in (2 ** i for i in range(21)) for b in (3 ** i for i in range(13) if a * 3 ** i <= top)
                   for c in (5 ** i for i in range(9) if a * b * 5 ** i <= top)
                   for d in (7 ** i for i in range(8) if a * b * c * 7 ** i <= top))
        v = np.array(v, dtype=np.int64)
        n = np.array([v[np.argmin(np.abs(v - min(2.0 ** u, top)))] for u in lg], dtype=np.int64)
    return n, np.maximum(1, (n * g.uniform(0.2, 0.5, case["count"])).astype(np.int64))


def _batch_inputs(case, seed):
    g = _gen(seed)
    ns, ms = _sizes(case)
    out = []
    for n, m in zip(ns.tolist(), ms.tolist()):
        c, rows, y = _instance({"n": n, "m": m, "k": max(1, round(0.01 * n)), "noise": 1e-3}, g)
        out.append((c, rows, y, 1.0 / _lipschitz(c)))
    return ns, ms, out


def _psf(n0, n1):
    """15 x 15 Gaussian of 2.5 pixels, sum 1, as the generating array
    c2[d] = psf[-d] (the PSF is symmetric)."""
    d = torch.arange(-7, 8, dtype=F64)
    w = torch.exp(-d * d / (2 * 2.5 ** 2))
    w = w / w.sum()
    c2 = torch.zeros(n0, n1, dtype=F64)
    i = torch.arange(-7, 8)
    c2.index_put_(((i % n0)[:, None].expand(15, 15), (i % n1)[None, :].expand(15, 15)), torch.outer(w, w),
                  accumulate=True)
    return c2


def _deblur_inputs(case, seed):
    g = _gen(seed)
    n0, n1, m, k = case["n0"], case["n1"], case["m"], case["k"]
    c2 = _psf(n0, n1).to(_device())
    x = torch.zeros(n0 * n1, device=_device(), dtype=F64)
    x[_pick(g, n0 * n1, k)] = torch.exp(_normal(g, k))   # log-normal flux
    pix = _pick(g, n0 * n1, m)
    h = torch.fft.rfft2(c2)
    y = _fwd(h, pix, x.view(n0, n1)) + 1e-3 * _normal(g, m)
    lam = 3e-3 * float(c2.norm()) * math.sqrt(m / (n0 * n1))
    # 1 / max |h|^2 = 1: a valid ISTA step; sigma = rho = 1e-3 for ADMM
    return c2, pix, y.float(), _f32(lam), _f32(1.0 / float(h.abs().square().max())), 1e-3


def _host(t):
    return t.cpu().numpy()


def prepare(case, seed):
    s = {"case": case}
    family = case["family"]
    stream = torch.cuda.current_stream()
    if family == "product":
        g = _gen(seed)
        c, rows, _ = _instance(case, g)
        s["plan"] = cs.cs_plan(case["n"], case["m"], _host(rows), _host(c), stream)
        s["x"] = _normal(g, case["n"]).float()
        s["r"] = _normal(g, case["m"]).float()
        s["y"] = torch.empty(case["m"], device=_device())
        s["g"] = torch.empty(case["n"], device=_device())
    elif family == "static":
        g = _gen(seed)
        n = case["n"]
        s["c"] = _normal(g, n) / math.sqrt(n)
        s["x"] = _normal(g, n).float()
        s["y"] = torch.empty(n, device=_device())
        s["yt"] = torch.empty(n, device=_device())
    elif family in ("ista", "recover", "admm"):
        c, rows, s["y"] = _instance(case, _gen(seed))
        s["plan"] = cs.cs_plan(case["n"], case["m"], _host(rows), _host(c), stream)
        s["tau"] = _f32(1.0 / _lipschitz(c))
    elif family == "deblur2d":
        c2, pix, s["y"], s["lam"], s["tau"], s["rho"] = _deblur_inputs(case, seed)
        s["plan"] = cs.cs_plan_2d(case["n0"], case["n1"], case["m"], _host(pix), _host(c2), stream)
    elif family == "batch":
        ns, ms, inst = _batch_inputs(case, seed)
        s["y"] = torch.cat([i[2] for i in inst])
        s["tau"] = np.array([i[3] for i in inst], dtype=np.float32)
        s["n"] = int(ns.sum())
        s["plan"] = cs.cs_batch_plan(ns, ms, np.concatenate([_host(i[1]) for i in inst]),
                                     np.concatenate([_host(i[0]) for i in inst]), stream)
    else:
        # Few, clearly nonzero entries and a threshold above the crosstalk:
        # the support is identified, so the gradient (of a soft threshold,
        # which has a kink) is a smooth function of the inputs.
        g = _gen(seed)
        c, rows, s["y"] = _instance(case, g, bounded=True)
        s["plan"] = cs.cs_plan(case["n"], case["m"], _host(rows), _host(c), stream)
        s["tau"] = _f32(1.0 / _lipschitz(c))
        # the gradient that arrives from the loss on the last iterate
        s["gz"] = _normal(g, case["n"]).float()
        s["gx"] = _normal(g, case["n"]).float()
    return s


# ------------------------------------------------------------------ one pass

def run(s):
    case = s["case"]
    family = case["family"]
    if family == "product":
        cs.cs_forward(s["plan"], s["x"], s["y"])
        cs.cs_adjoint(s["plan"], s["r"], s["g"])
        return [s["y"], s["g"]]
    if family == "static":
        stream = torch.cuda.current_stream()
        cs.cs_circulant_apply_static(case["n"], s["c"], s["x"], s["y"], False, stream)
        cs.cs_circulant_apply_static(case["n"], s["c"], s["x"], s["yt"], True, stream)
        return [s["y"], s["yt"]]
    if family == "ista":
        x = torch.zeros(case["n"], device=_device())
        st = cs.cs_ista(s["plan"], s["y"], case["lam"], s["tau"], case["iters"], x, stats=case["stats"])
        return [x, st["objective"]] if st else [x]
    if family == "recover":
        L = cs.cs_opnorm2(s["plan"], case["power"])
        x = torch.zeros(case["n"], device=_device())
        # 1.05: the power iteration's estimate is from below
        st = cs.cs_ista(s["plan"], s["y"], case["lam"], 1.0 / (1.05 * L), case["iters"], x)
        return [L, x, st["objective"]]
    if family == "admm":
        z = torch.empty(case["n"], device=_device())
        st = cs.cs_admm(s["plan"], s["y"], case["lam"], case["rho"], case["iters"], z, stats=case["stats"])
        return [z, st["objective"]] if st else [z]
    if family == "deblur2d":
        n = case["n0"] * case["n1"]
        x = torch.zeros(n, device=_device())
        cs.cs_ista(s["plan"], s["y"], s["lam"], s["tau"], case["iters"], x, stats=False)
        z = torch.empty(n, device=_device())
        cs.cs_admm(s["plan"], s["y"], s["lam"], s["rho"], case["iters"], z, stats=False)
        return [x, z]
    if family == "batch":
        x = torch.zeros(s["n"], device=_device())
        cs.cs_batch_ista(s["plan"], s["y"], 1e-3, s["tau"], case["iters"], x)
        z = torch.empty(s["n"], device=_device())
        cs.cs_batch_admm(s["plan"], s["y"], 1e-3, 1.0, case["iters"], z)
        return [x, z]
    dc = torch.empty(case["n"], device=_device())
    dl = torch.empty(1, device=_device())
    dy = torch.empty(case["m"], device=_device())
    if family == "grad":
        cs.cs_grad(s["plan"], s["y"], case["lam"], s["tau"], case["T"], case["K"], s["gx"], dc, dl, dy)
    else:
        cs.cs_grad_admm(s["plan"], s["y"], case["lam"], case["rho"], case["rho"], 1.0, 1.0, case["T"], case["K"],
                        s["gz"], dc, dl, dy, gx_T=s["gx"])
    return [dc, dl, dy]


# --------------------------------------------------- what a pass cannot avoid

def _fft_flops(n):
    """One real transform of length n."""
    return 2.5 * n * _lg(n)


def _solve_work(n, m, iters):
    # four real transforms an iteration and the element-wise steps
    return {"bytes": 4.0 * (2 * n + m) + 4.0 * n + n / 8.0, "flops": iters * (4 * _fft_flops(n) + 20.0 * n)}


def work(case):
    family = case["family"]
    if family == "product":
        n, m = case["n"], case["m"]
        return {"bytes": 2 * 4.0 * (n + m) + 4.0 * n + 4.0 * m, "flops": 4 * _fft_flops(n) + 12.0 * n}
    if family == "static":
        n = case["n"]
        return {"bytes": 2 * 4.0 * n + 4.0 * n + 8.0 * n, "flops": 6 * _fft_flops(n) + 12.0 * n}
    if family in ("ista", "admm"):
        return _solve_work(case["n"], case["m"], case["iters"])
    if family == "recover":
        return _solve_work(case["n"], case["m"], case["iters"] + case["power"])
    if family == "deblur2d":
        w = _solve_work(case["n0"] * case["n1"], case["m"], case["iters"])
        return {k: 2 * v for k, v in w.items()}
    if family == "batch":
        ns, ms = _sizes(case)
        w = [_solve_work(int(n), int(m), case["iters"]) for n, m in zip(ns, ms)]
        return {k: 2 * sum(x[k] for x in w) for k in ("bytes", "flops")}
    # forward and reverse steps of four real transforms each, and the two
    # correlations of a reverse step
    n, m = case["n"], case["m"]
    return {"bytes": 4.0 * (4 * n + 2 * m), "flops": case["T"] * (8 * _fft_flops(n) + 50.0 * n)}


# ----------------------------------------------------------- in 64 bits

def _fft(x):
    return torch.fft.rfft2(x) if x.dim() == 2 else torch.fft.rfft(x)


def _ifft(X, shape):
    return torch.fft.irfft2(X, s=shape) if len(shape) == 2 else torch.fft.irfft(X, n=shape[0])


def _fwd(h, rows, x):
    """(C x)[rows], C[i][j] = c[(j - i) mod n], h = DFT(c)."""
    return _ifft(h.conj() * _fft(x), tuple(x.shape)).reshape(-1)[rows]


def _adj(h, rows, r, shape):
    """C^T P^T r."""
    n = math.prod(shape)
    u = torch.zeros(n, device=r.device, dtype=F64).index_copy(0, rows, r)
    return _ifft(h * _fft(u.view(shape)), tuple(shape))


def _soft(u, g):
    return torch.sign(u) * torch.clamp(u.abs() - g, min=0.0)


def _ista64(h, rows, y, lam, tau, iters, shape):
    """x(T) and the objective at x(T-1), as cs_ista reports it."""
    x = torch.zeros(shape, device=y.device, dtype=F64)
    y = y.double()
    obj = None
    for t in range(iters):
        r = y - _fwd(h, rows, x)
        if t == iters - 1:
            obj = 0.5 * r.square().sum() + lam * x.abs().sum()
        x = _soft(x + tau * _adj(h, rows, r, shape), _f32(tau * lam))
    return x.reshape(-1), obj


def _admm64(h, rows, y, lam, rho, iters, shape):
    """z(T) and the objective as cs_admm reports it (sigma = rho, tau = 1)."""
    n = math.prod(shape)
    dev = y.device
    d = torch.full((n,), 1.0 / rho, device=dev, dtype=F64)
    d[rows] = 1.0 / (1.0 + rho)
    py = torch.zeros(n, device=dev, dtype=F64)
    py[rows] = y.double()
    d, py = d.view(shape), py.view(shape)
    b = 1.0 / (rho * h.abs().square() + rho)
    v = z = mu = nu = torch.zeros(shape, device=dev, dtype=F64)
    obj = None
    for t in range(iters):
        X = b * (rho * h * _fft(v) + rho * _fft(z - nu))
        x, cx = _ifft(X, tuple(shape)), _ifft(h.conj() * X, tuple(shape))
        v = d * (rho * (cx - mu) + py)
        z = _soft(x + nu, _f32(lam / rho))
        mu = mu + v - cx
        nu = nu + x - z
        v = v + mu
        if t == iters - 1:
            obj = 0.5 * (y.double() - cx.reshape(-1)[rows]).square().sum() + lam * z.abs().sum()
    return z.reshape(-1), obj


def _opnorm64(h, rows, n, iters):
    """Rayleigh quotient of A^T A after `iters` steps from the documented
    fixed start (a 32-bit hash of the index, in [-1, 1))."""
    mask32 = 0xffffffff
    v = torch.arange(n, device=_device(), dtype=torch.int64)
    v = (v * 2654435761 + 0x9e3779b9) & mask32
    v = v ^ (v >> 16)
    v = _mul32(v, 0x85ebca6b)
    v = v ^ (v >> 13)
    v = _mul32(v, 0xc2b2ae35)
    v = v ^ (v >> 16)
    u = (v.double() * (2.0 / 4294967296.0) - 1.0).float().double()
    L = 0.0
    for _ in range(iters):
        u = u / u.norm()
        w = _adj(h, rows, _fwd(h, rows, u), (n,))
        L = float(torch.dot(u, w))
        u = w
    return L


def _mul32(v, k):
    """v * k mod 2^32 for int64 tensors of values below 2^32."""
    lo, hi = v & 0xffff, v >> 16
    return (lo * k + (((hi * k) & 0xffff) << 16)) & 0xffffffff


def _grad64(case, c, rows, y, tau, gx, gz):
    n = case["n"]
    c = c.clone().requires_grad_(True)
    y = y.double().requires_grad_(True)
    lam = torch.tensor(float(np.float32(case["lam"])), device=y.device, dtype=F64, requires_grad=True)
    h = torch.fft.rfft(c)
    zero = torch.zeros(n, device=y.device, dtype=F64)
    if case["family"] == "grad":
        x = zero
        for _ in range(case["T"]):
            x = _soft(x + tau * _adj(h, rows, y - _fwd(h, rows, x), (n,)), tau * lam)
        loss = (x * gx.double()).sum()
    else:
        rho = case["rho"]
        d = torch.full((n,), 1.0 / rho, device=y.device, dtype=F64)
        d[rows] = 1.0 / (1.0 + rho)
        py = zero.index_copy(0, rows, y)
        b = 1.0 / (rho * h.abs().square() + rho)
        v = z = mu = nu = zero
        for _ in range(case["T"]):
            X = b * (rho * h * torch.fft.rfft(v) + rho * torch.fft.rfft(z - nu))
            x, cx = torch.fft.irfft(X, n=n), torch.fft.irfft(h.conj() * X, n=n)
            v = d * (rho * (cx - mu) + py)
            z = _soft(x + nu, lam / rho)
            mu = mu + v - cx
            nu = nu + x - z
            v = v + mu
        loss = (z * gz.double()).sum() + (x * gx.double()).sum()
    dc, dl, dy = torch.autograd.grad(loss, [c, lam, y])
    return [dc, dl.reshape(1), dy]


def exact(case, seed):
    family = case["family"]
    if family == "product":
        g = _gen(seed)
        c, rows, _ = _instance(case, g)
        x, r = _normal(g, case["n"]).float(), _normal(g, case["m"]).float()
        h = torch.fft.rfft(c)
        return [_fwd(h, rows, x.double()), _adj(h, rows, r.double(), (case["n"],))]
    if family == "static":
        g = _gen(seed)
        n = case["n"]
        c, x = _normal(g, n) / math.sqrt(n), _normal(g, n).float()
        h, X = torch.fft.rfft(c), torch.fft.rfft(x.double())
        return [torch.fft.irfft(h.conj() * X, n=n), torch.fft.irfft(h * X, n=n)]
    if family in ("ista", "recover", "admm"):
        c, rows, y = _instance(case, _gen(seed))
        h, lam, shape = torch.fft.rfft(c), _f32(case["lam"]), (case["n"],)
        if family == "admm":
            z, obj = _admm64(h, rows, y, lam, _f32(case["rho"]), case["iters"], shape)
            return [z, float(obj)] if case["stats"] else [z]
        if family == "recover":
            L = _opnorm64(h, rows, case["n"], case["power"])
            x, obj = _ista64(h, rows, y, lam, _f32(1.0 / (1.05 * L)), case["iters"], shape)
            return [L, x, float(obj)]
        x, obj = _ista64(h, rows, y, lam, _f32(1.0 / _lipschitz(c)), case["iters"], shape)
        return [x, float(obj)] if case["stats"] else [x]
    if family == "deblur2d":
        c2, pix, y, lam, tau, rho = _deblur_inputs(case, seed)
        h, shape = torch.fft.rfft2(c2), (case["n0"], case["n1"])
        return [_ista64(h, pix, y, lam, tau, case["iters"], shape)[0],
                _admm64(h, pix, y, lam, _f32(rho), case["iters"], shape)[0]]
    if family == "batch":
        xs, zs = [], []
        for c, rows, y, tau in _batch_inputs(case, seed)[2]:
            h, shape, lam = torch.fft.rfft(c), (c.numel(),), _f32(1e-3)
            xs.append(_ista64(h, rows, y, lam, _f32(tau), case["iters"], shape)[0])
            zs.append(_admm64(h, rows, y, lam, 1.0, case["iters"], shape)[0])
        return [torch.cat(xs), torch.cat(zs)]
    g = _gen(seed)
    c, rows, y = _instance(case, g, bounded=True)
    tau = _f32(1.0 / _lipschitz(c))
    gz = _normal(g, case["n"]).float()
    gx = _normal(g, case["n"]).float()
    return _grad64(case, c, rows, y, tau, gx, gz)
