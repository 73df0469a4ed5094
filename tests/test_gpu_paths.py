"""What the solvers do beside iterating, on each path that a length selects:
early stop by the monitor, warm starts, the power iteration, gradients in the
long shapes, image solves in every shape, and captured chunks against direct
launches.

Tolerances: a few iterations from zero within 1e-5 of the FP64 oracle and 100
iterations within 1e-5 (as test_gpu_shapes.py and test_gpu_solvers.py), the
gradient within 1e-3 (test_gpu_grad.py), a recorded NMSE within 1e-4 of the
one of the returned iterate.  Power iteration: a product has a relative error
below 1e-6, so 12 steps turn the vector by less than 2e-5 and the quotient,
which is second order in that and first order in the last product, moves by
less than 1e-5 relative.
"""
import numpy as np
import pytest

import oracle.cs_oracle as O
import synth
from gpu_util import f32, host, rel_l2, to_dev, torch_dev

pytestmark = pytest.mark.gpu

PATHS = [2048, 1 << 15, 1 << 17]   # one CTA, one cluster of CTAs, the passes


@pytest.fixture(scope="module")
def cs():
    import paper_1707_02244_gb300 as cs
    return cs


def _inst(n):
    m = n // 3 | 1
    g = synth.rng(8100 + n)
    c = synth.gaussian_c(g, n, m)
    rows = synth.draw_rows(g, n, m)
    x = synth.k_sparse(g, n, n // 100)
    chat = O.spectrum(c)
    y = (O.forward_fft(chat, rows, x) + 1e-3 * g.standard_normal(m)).astype(np.float32)
    return m, c, rows, chat, x, y, f32(0.9 / np.max(np.abs(chat) ** 2))


def _plan(cs, n, m, rows, c):
    torch, dev = torch_dev()
    return cs.cs_plan(n, m, rows, c, torch.cuda.current_stream(dev))


def _admm_ex(cs, plan, yd, lam, prm, iters, state=None):
    torch, dev = torch_dev()
    v = {k: torch.zeros(plan.n, device=dev) for k in ("x", "z", "mu", "nu", "v")}
    if state is not None:
        for k in ("z", "mu", "nu", "v"):
            v[k].copy_(state[k])
    st = cs.cs_admm_ex(plan, yd, lam, *prm, iters, state is not None, v["x"], v["z"], v["mu"], v["nu"], v["v"])
    return v, st


def _check_state(got, o, keys=("x", "z", "v")):
    for k in keys:
        assert rel_l2(host(got[k]), o[k]) <= 1e-5, k
    # mu and nu are running sums of v - C x and x - z: relative to those
    assert np.linalg.norm(host(got["mu"]) - o["mu"]) <= 1e-5 * np.linalg.norm(o["v"])
    assert np.linalg.norm(host(got["nu"]) - o["nu"]) <= 1e-5 * np.linalg.norm(o["x"])


@pytest.mark.parametrize("n", PATHS)
def test_monitor_stops_ista(cs, n):
    torch, dev = torch_dev()
    m, c, rows, _, x_true, y, tau = _inst(n)
    lam = f32(2e-3)
    _, h = O.ista_fft(c, rows, y.astype(np.float64), lam, tau, 25, history=True)
    tol = 0.5 * (O.nmse(h[20], x_true) + O.nmse(h[25], x_true))
    plan = _plan(cs, n, m, rows, c)
    xt = to_dev(x_true)
    try:
        cs.cs_set_monitor(plan, xt, float(tol), 5)
        x = torch.zeros(n, device=dev)
        st = cs.cs_ista(plan, to_dev(y), lam, tau, 5000, x)
    finally:
        plan.close()
    assert st["converged"] == 1 and st["iters_run"] == 25
    assert rel_l2(host(x), h[25]) <= 1e-5
    e = O.nmse(host(x), x_true)
    assert abs(st["nmse"] - e) <= 1e-4 * e


@pytest.mark.parametrize("n", PATHS)
def test_monitor_stops_admm(cs, n):
    """cs_admm takes no v, mu, nu: a watched solve carries them in the plan."""
    torch, dev = torch_dev()
    m, c, rows, _, x_true, y, _ = _inst(n)
    lam, y64 = f32(2e-3), y.astype(np.float64)
    o = O.admm_fft(c, rows, y64, lam, sigma=1.0, rho=1.0, iters=25, history=True)
    tol = 0.5 * (O.nmse(o["history"][19][1], x_true) + O.nmse(o["z"], x_true))
    plan = _plan(cs, n, m, rows, c)
    xt, yd = to_dev(x_true), to_dev(y)
    try:
        cs.cs_set_monitor(plan, xt, float(tol), 5)
        z = torch.empty(n, device=dev)
        st = cs.cs_admm(plan, yd, lam, 1.0, 5000, z)
        got, st2 = _admm_ex(cs, plan, yd, lam, (1.0, 1.0, 1.0, 1.0), 5000)
        cs.cs_set_monitor(plan)
        plain = torch.empty(n, device=dev)
        cs.cs_admm(plan, yd, lam, 1.0, 25, plain)
    finally:
        plan.close()
    for s in (st, st2):
        assert s["converged"] == 1 and s["iters_run"] == 25
        e = O.nmse(host(z), x_true)
        assert abs(s["nmse"] - e) <= 1e-4 * e
    assert torch.equal(z, plain) and torch.equal(z, got["z"])
    _check_state(got, o)


@pytest.mark.parametrize("n", PATHS)
def test_admm_warm_start(cs, n):
    """60 + 40 iterations through the state are 100, bit for bit."""
    m, c, rows, _, _, y, _ = _inst(n)
    lam, prm = f32(2e-3), (0.7, 1.3, 1.2, 1.2)
    plan = _plan(cs, n, m, rows, c)
    yd = to_dev(y)
    torch, _ = torch_dev()
    try:
        full, _ = _admm_ex(cs, plan, yd, lam, prm, 100)
        half, _ = _admm_ex(cs, plan, yd, lam, prm, 60)
        rest, _ = _admm_ex(cs, plan, yd, lam, prm, 40, half)
    finally:
        plan.close()
    assert all(torch.equal(full[k], rest[k]) for k in full)
    o = O.admm_fft(c, rows, y.astype(np.float64), lam, sigma=0.7, rho=1.3, tau1=1.2, tau2=1.2, iters=100)
    _check_state(full, o)


@pytest.mark.parametrize("lg", [6, 9, 12, 13, 14, 15, 16, 18, 20, 21])
def test_power_iteration(cs, lg):
    """12 steps from the fixed start (a 32-bit hash of the index in [-1, 1))."""
    n = 1 << lg
    m, c, rows, chat, _, _, _ = _inst(n)
    h = np.arange(n, dtype=np.uint32) * np.uint32(2654435761) + np.uint32(0x9e3779b9)
    for shift, mul in ((16, 0x85ebca6b), (13, 0xc2b2ae35)):
        h = (h ^ (h >> np.uint32(shift))) * np.uint32(mul)
    h ^= h >> np.uint32(16)
    w = (h.astype(np.float64) * (2.0 / 4294967296.0) - 1.0).astype(np.float32).astype(np.float64)
    for _ in range(12):
        u = w / np.linalg.norm(w)
        w = O.adjoint_fft(chat, rows, O.forward_fft(chat, rows, u))
        want = float(u @ w)
    plan = _plan(cs, n, m, rows, c)
    try:
        got = cs.cs_opnorm2(plan, 12)
    finally:
        plan.close()
    assert abs(got - want) <= 1e-5 * want


@pytest.mark.parametrize("n", [1 << 20, 1 << 21, 1 << 22])
def test_grad_long(cs, n):
    torch, dev = torch_dev()
    m, c, rows, chat, x_true, y, tau = _inst(n)
    y64 = y.astype(np.float64)
    lam = f32(0.05 * np.max(np.abs(O.adjoint_fft(chat, rows, y64))))
    xT = O.ista_fft(c, rows, y64, lam, tau, 3)
    gx = (2.0 * (xT - x_true)).astype(np.float32)
    o = O.ista_unrolled_grad_fft(c, rows, y64, lam, tau, 3, gx.astype(np.float64))
    plan = _plan(cs, n, m, rows, c)
    try:
        dc, dl, dy = (torch.empty(k, device=dev) for k in (n, 1, m))
        cs.cs_grad(plan, to_dev(y), lam, tau, 3, 2, to_dev(gx), dc, dl, dy)
        assert cs.cs_status_sync(plan) == 0
    finally:
        plan.close()
    assert rel_l2(host(dc), o["dc"]) <= 1e-3
    assert rel_l2(host(dy), o["dy"]) <= 1e-3
    assert abs(float(host(dl)[0]) - o["dlam"]) <= 1e-3 * abs(o["dlam"])


@pytest.mark.parametrize("n0,n1", [(8, 16), (32, 32), (32, 4096), (64, 128), (128, 512), (256, 64), (512, 2048),
                                   (1024, 256), (2048, 32), (2048, 1024), (4096, 16)])
def test_image_solves(cs, n0, n1):
    torch, dev = torch_dev()
    n = n0 * n1
    m = n // 3 | 1
    g = synth.rng(8300 + n0 + n1)
    c2 = g.standard_normal((n0, n1)) / np.sqrt(n)
    pix = g.permutation(n)[:m].astype(np.int64)
    chat2 = O.spectrum2d(c2)
    x = synth.k_sparse(g, n, max(1, n // 50))
    y = (O.forward2d_fft(chat2, pix, x).ravel() + 1e-3 * g.standard_normal(m)).astype(np.float32)
    y64, lam, tau = y.astype(np.float64), f32(1e-3), f32(0.9 / np.max(np.abs(chat2) ** 2))
    plan = cs.cs_plan_2d(n0, n1, m, pix, c2, torch.cuda.current_stream(dev))
    try:
        xd = torch.zeros(n, device=dev)
        cs.cs_ista(plan, to_dev(y), lam, tau, 3, xd)
        got, _ = _admm_ex(cs, plan, to_dev(y), lam, (0.7, 0.7, 1.0, 1.0), 3)
    finally:
        plan.close()
    assert rel_l2(host(xd), np.asarray(O.ista_fft2d(c2, pix, y64, lam, tau, 3)).ravel()) <= 1e-5
    o = O.admm_fft2d(c2, pix, y64, lam, sigma=f32(0.7), rho=f32(0.7), iters=3)
    _check_state(got, {k: np.asarray(v).ravel() for k, v in o.items()}, keys=("x", "z"))


@pytest.mark.parametrize("n", [1 << 17, 1 << 20])
def test_graphs_match_direct_launches(cs, n, monkeypatch):
    """At lengths that the passes serve: chunks with and without statistics,
    and the chains of the gradients."""
    torch, dev = torch_dev()
    m, c, rows, _, x_true, y, tau = _inst(n)
    lam, xt, yd = f32(2e-3), to_dev(x_true), to_dev(y)
    gx = to_dev(x_true)
    out = {}
    for mode in ("1", "0"):
        monkeypatch.setenv("CS_GRAPHS", mode)
        plan = _plan(cs, n, m, rows, c)
        res = []
        try:
            for stats in (False, True):
                x, z = torch.zeros(n, device=dev), torch.empty(n, device=dev)
                res += [x, z]
                for st in (cs.cs_ista(plan, yd, lam, tau, 37, x, stats=stats),
                           cs.cs_admm(plan, yd, lam, 1.0, 23, z, stats=stats)):
                    if st:
                        res.append(torch.tensor([st["objective"], st["rel_change"]], dtype=torch.float64))
            cs.cs_set_monitor(plan, xt, 1e-30, 7)
            x = torch.zeros(n, device=dev)
            st = cs.cs_ista(plan, yd, lam, tau, 37, x)
            res += [x, torch.tensor([st["nmse"]], dtype=torch.float64)]
            cs.cs_set_monitor(plan)
            for K in (5, 17):
                d = [torch.empty(k, device=dev) for k in (n, 1, m)]
                cs.cs_grad(plan, yd, lam, tau, 17, K, gx, *d)
                e = [torch.empty(k, device=dev) for k in (n, 1, m)]
                cs.cs_grad_admm(plan, yd, lam, 1.0, 1.0, 1.0, 1.0, 17, K, gx, *e)
                res += d + e
            torch.cuda.synchronize()
        finally:
            plan.close()
        out[mode] = res
    assert len(out["0"]) == len(out["1"])
    assert all(torch.equal(a, b) for a, b in zip(out["0"], out["1"]))
