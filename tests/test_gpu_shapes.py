"""GPU parity at every transform shape the calls choose by length: the
single-CTA solver (n <= 8192), the cluster of CTAs (2^13 .. 2^15), the radix-8
tiles (to 2^20) and the 4096-value tiles above, the batch's chain of each
length, and the static product, each against the FP64 oracle.

Tolerances.  One fp32 FFT of length N has a relative rms error below
eps32 * log2 N = 2.7e-6 at N = 2^22 with a constant well under 1/2, and a
product is two transforms: relative l2 2e-6 (as the product tests).  A few
iterations from zero add the errors of their products (4 resp. 2 transforms
an iteration, damped by tau ||A||^2 <= 1): 3 iterations within 1e-5.  The
static product is FP64 rounded once: eps32 / 2 per element of its size, 1e-7
in relative l2.
"""
import numpy as np
import pytest

import oracle.cs_oracle as O
import synth
from gpu_util import f32, host, rel_l2, to_dev, torch_dev

pytestmark = pytest.mark.gpu

LGS = list(range(6, 22))


@pytest.fixture(scope="module")
def cs():
    import paper_1707_02244_gb300 as cs
    return cs


def _inst(n, seed):
    m = max(1, n // 3) | 1
    g = synth.rng(seed)
    c = synth.gaussian_c(g, n, m)
    rows = synth.draw_rows(g, n, m)
    x = synth.k_sparse(g, n, max(1, n // 50))
    chat = O.spectrum(c)
    y = (O.forward_fft(chat, rows, x) + 1e-3 * g.standard_normal(m)).astype(np.float32)
    return m, c, rows, chat, y, f32(0.9 / np.max(np.abs(chat) ** 2)), g


@pytest.mark.parametrize("lg", LGS)
def test_every_length(cs, lg):
    torch, dev = torch_dev()
    n = 1 << lg
    m, c, rows, chat, y, tau, g = _inst(n, 4000 + lg)
    x0 = g.standard_normal(n).astype(np.float32)
    y64 = y.astype(np.float64)
    plan = cs.cs_plan(n, m, rows, c, torch.cuda.current_stream(dev))
    try:
        yd, xd = torch.empty(m, device=dev), torch.empty(n, device=dev)
        cs.cs_forward(plan, to_dev(x0), yd)
        cs.cs_adjoint(plan, to_dev(y), xd)
        assert rel_l2(host(yd), O.forward_fft(chat, rows, x0.astype(np.float64))) <= 2e-6
        assert rel_l2(host(xd), O.adjoint_fft(chat, rows, y64)) <= 2e-6
        lam = f32(1e-3)
        x = torch.zeros(n, device=dev)
        st = cs.cs_ista(plan, to_dev(y), lam, tau, 3, x)
        xo = O.ista_fft(c, rows, y64, lam, tau, 3)
        assert rel_l2(host(x), xo) <= 1e-5
        # the record: ||x_t||_1 and the residual are those of the last iteration's input
        xp = O.ista_fft(c, rows, y64, lam, tau, 2)
        obj = 0.5 * np.sum((y64 - O.forward_fft(chat, rows, xp)) ** 2) + lam * np.sum(np.abs(xp))
        assert abs(st["objective"] - obj) <= 1e-5 * obj
        z = torch.empty(n, device=dev)
        cs.cs_admm(plan, to_dev(y), lam, 0.7, 3, z)
        zo = O.admm_fft(c, rows, y64, lam, sigma=f32(0.7), rho=f32(0.7), iters=3)["z"]
        assert rel_l2(host(z), zo) <= 1e-5
        # one step at a time (a chunk of its own each) ends at the same bits
        x1 = torch.zeros(n, device=dev)
        for _ in range(3):
            cs.cs_ista(plan, to_dev(y), lam, tau, 1, x1, stats=False)
        assert torch.equal(x, x1)
        # 12 iterations of the power method from the fixed start: the Rayleigh
        # quotient is below ||A||^2 and above the first one's expectation m |c|^2 / n
        L = cs.cs_opnorm2(plan, 12)
        assert 0.0 < L <= float(np.max(np.abs(chat) ** 2)) * (1 + 1e-5)
    finally:
        plan.close()


def test_batch_of_every_length(cs):
    torch, dev = torch_dev()
    ns = np.array([1 << lg for lg in LGS for _ in range(2)], dtype=np.int64)
    inst = [_inst(int(n), 4100 + i) for i, n in enumerate(ns)]
    ms = np.array([t[0] for t in inst], dtype=np.int64)
    plan = cs.cs_batch_plan(ns, ms, np.concatenate([t[2] for t in inst]), np.concatenate([t[1] for t in inst]),
                            torch.cuda.current_stream(dev))
    try:
        y = to_dev(np.concatenate([t[4] for t in inst]))
        tau = np.array([t[5] for t in inst], dtype=np.float32)
        x, z = torch.zeros(int(ns.sum()), device=dev), torch.empty(int(ns.sum()), device=dev)
        cs.cs_batch_ista(plan, y, 1e-3, tau, 3, x)
        cs.cs_batch_admm(plan, y, 1e-3, 1.0, 3, z)
        assert cs.cs_batch_status_sync(plan) == 0
        xh, zh, o = host(x), host(z), 0
        for n, (m, c, rows, chat, yi, ti, _) in zip(ns.tolist(), inst):
            y64 = yi.astype(np.float64)
            assert rel_l2(xh[o:o + n], O.ista_fft(c, rows, y64, f32(1e-3), ti, 3)) <= 1e-5, n
            assert rel_l2(zh[o:o + n], O.admm_fft(c, rows, y64, f32(1e-3), sigma=1.0, rho=1.0, iters=3)["z"]) <= 1e-5, n
            o += n
    finally:
        plan.close()


@pytest.mark.parametrize("lg", range(6, 15))
def test_static_product_every_length(cs, lg):
    torch, dev = torch_dev()
    n = 1 << lg
    g = synth.rng(4200 + lg)
    c, x = g.standard_normal(n), g.standard_normal(n).astype(np.float32)
    cd, y = torch.from_numpy(c).to(dev), torch.empty(n, device=dev)
    for tr in (False, True):
        cs.cs_circulant_apply_static(n, cd, to_dev(x), y, tr, torch.cuda.current_stream(dev))
        assert rel_l2(host(y), O.circulant_apply_fft(O.spectrum(c), x.astype(np.float64), tr)) <= 1e-7


@pytest.mark.parametrize("n0,n1", [(8, 16), (32, 32), (32, 4096), (64, 128), (128, 512), (256, 64), (512, 2048),
                                   (1024, 256), (2048, 32), (4096, 16)])
def test_every_image_shape(cs, n0, n1):
    torch, dev = torch_dev()
    n = n0 * n1
    g = synth.rng(n0 + n1)
    c2 = g.standard_normal((n0, n1)) / np.sqrt(n)
    m = n // 3 | 1
    pix = g.permutation(n)[:m].astype(np.int64)
    chat2 = O.spectrum2d(c2)
    x, r = g.standard_normal(n).astype(np.float32), g.standard_normal(m).astype(np.float32)
    plan = cs.cs_plan_2d(n0, n1, m, pix, c2, torch.cuda.current_stream(dev))
    try:
        yd, xd = torch.empty(m, device=dev), torch.empty(n, device=dev)
        cs.cs_forward(plan, to_dev(x), yd)
        cs.cs_adjoint(plan, to_dev(r), xd)
        assert rel_l2(host(yd), O.forward2d_fft(chat2, pix, x.astype(np.float64)).ravel()) <= 2e-6
        assert rel_l2(host(xd), np.asarray(O.adjoint2d_fft(chat2, pix, r.astype(np.float64))).ravel()) <= 2e-6
    finally:
        plan.close()
