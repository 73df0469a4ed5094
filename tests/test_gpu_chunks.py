"""How a solve is cut into launches: the longest launch, check points, state
that is carried from one chunk to the next, and the record at a check point,
on each of the three solvers (one CTA, one cluster of CTAs, the passes).

Tolerances: 1e-5 against the FP64 oracle as in test_gpu_shapes.py (a few
iterations from zero); bit equality where the same kernel does the same
iterations in another number of launches.
"""
import numpy as np
import pytest

import oracle.cs_oracle as O
import synth
from gpu_util import f32, host, rel_l2, to_dev, torch_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cs():
    import paper_1707_02244_gb300 as cs
    return cs


def _plan(cs, n, seed):
    torch, dev = torch_dev()
    m = n // 3 | 1
    g = synth.rng(seed)
    c = synth.gaussian_c(g, n, m)
    rows = synth.draw_rows(g, n, m)
    x = synth.k_sparse(g, n, max(2, n // 100))
    chat = O.spectrum(c)
    y = (O.forward_fft(chat, rows, x) + 1e-3 * g.standard_normal(m)).astype(np.float32)
    plan = cs.cs_plan(n, m, rows, c, torch.cuda.current_stream(dev))
    return plan, c, rows, x, y, f32(0.9 / np.max(np.abs(chat) ** 2))


@pytest.mark.parametrize("n", [1024, 1 << 13, 1 << 14])
def test_solves_do_not_go_into_a_capture(cs, n):
    """A captured solve would leave out what the plan held at that moment (the
    spectrum of B for its rho), and answer wrongly when it is replayed after
    another one.  Refused as on the pass path; products are captured."""
    torch, dev = torch_dev()
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        plan, c, rows, _, y, tau = _plan(cs, n, 8150 + n)
        yd, x, z, p = to_dev(y), torch.zeros(n, device=dev), torch.empty(n, device=dev), torch.empty(plan.m, device=dev)
        try:
            cs.cs_admm(plan, yd, 1e-3, 1.0, 3, z, stats=False)
            cs.cs_forward(plan, z, p)
            st.synchronize()
            want_z, want_p = z.clone(), p.clone()
            for solve in (lambda: cs.cs_ista(plan, yd, 1e-3, tau, 3, x, stats=False),
                          lambda: cs.cs_admm(plan, yd, 1e-3, 2.0, 3, z, stats=False)):
                with torch.cuda.graph(torch.cuda.CUDAGraph(), stream=st):
                    p.zero_()
                    with pytest.raises(cs.CsError) as err:
                        solve()
                assert err.value.code == 3   # CS_ERR_CUDA
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=st):
                cs.cs_forward(plan, z, p)
            cs.cs_admm(plan, yd, 1e-3, 2.0, 3, z, stats=False)
            zo = O.admm_fft(c, rows, y.astype(np.float64), f32(1e-3), sigma=2.0, rho=2.0, iters=3)["z"]
            st.synchronize()
            assert rel_l2(host(z), zo) <= 1e-5
            cs.cs_admm(plan, yd, 1e-3, 1.0, 3, z, stats=False)
            g.replay()
            torch.cuda.synchronize()
            assert torch.equal(z, want_z) and torch.equal(p, want_p)
        finally:
            plan.close()


@pytest.mark.parametrize("n", [64, 4096, 1 << 13, 1 << 15, 1 << 17])
def test_profile_pass_inputs(cs, n):
    """The pass kernels that the measurement hook launches find inputs laid out:
    by the solve on the pass path, else by the hook from the buffers that the
    solve named (so that it sees, and reports, what y holds by then)."""
    torch, dev = torch_dev()
    plan, _, _, _, y, tau = _plan(cs, n, 8200 + n)
    yd = to_dev(y)
    x, z = torch.zeros(n, device=dev), torch.empty(n, device=dev)
    try:
        for solve, out, passes, one_launch in (
                (lambda o: cs.cs_ista(plan, yd, 1e-3, tau, 3, o, stats=False), x, (0, 1, 2, 3), n <= 1 << 15),
                (lambda o: cs.cs_admm(plan, yd, 1e-3, 1.0, 3, o, stats=False), z, (4, 5), n <= 1 << 15)):
            out.zero_()
            solve(out)
            want = out.clone()
            yd[0] = float("inf")
            for k in passes:
                cs.cs_profile_pass(plan, k, 2)
            assert cs.cs_status_sync(plan) == (5 if one_launch else 0)   # CS_ERR_NONFINITE
            yd.copy_(torch.from_numpy(y))
            out.zero_()
            solve(out)
            assert torch.equal(out, want) and cs.cs_status_sync(plan) == 0
    finally:
        plan.close()


def test_grad_segments_that_do_not_fit(cs):
    """K = T = 8000 at n = 2^22: 24000 vectors, 375 GiB.  The plan takes shorter
    segments, which give the same gradient."""
    torch, dev = torch_dev()
    n, T = 1 << 22, 8000
    plan, _, _, _, y, tau = _plan(cs, n, 8190)
    g = torch.Generator(device=dev)
    g.manual_seed(3)
    gx = torch.randn(n, generator=g, device=dev)
    torch.cuda.empty_cache()
    out = []
    try:
        for K in (T, 100, T):
            dc, dl, dy = (torch.empty(k, device=dev) for k in (n, 1, plan.m))
            cs.cs_grad(plan, to_dev(y), 0.05, tau, T, K, gx, dc, dl, dy)
            out.append((dc, dl, dy))
        assert cs.cs_status_sync(plan) == 0
    finally:
        plan.close()
    for got in (out[0], out[2]):
        assert all(torch.equal(a, b) for a, b in zip(got, out[1]))
    assert float(out[1][0].norm()) > 0.0


@pytest.mark.parametrize("n", [64, 1 << 13])
def test_launch_length_is_bounded(cs, n):
    """No launch runs more than 10000 iterations, whatever check_every is."""
    torch, dev = torch_dev()
    plan, _, _, x_true, y, tau = _plan(cs, n, 8100 + n)
    yd, xt = to_dev(y), to_dev(x_true)
    try:
        ref, x = torch.zeros(n, device=dev), torch.zeros(n, device=dev)
        assert cs.cs_ista(plan, yd, 1e-3, tau, 25000, ref)["launches"] == 3
        zref, z = torch.empty(n, device=dev), torch.empty(n, device=dev)
        count = cs.cs_admm(plan, yd, 1e-3, 1.0, 25000, zref)["launches"]
        cs.cs_set_monitor(plan, None, 0.0, 10 ** 9)
        assert cs.cs_ista(plan, yd, 1e-3, tau, 25000, x)["launches"] == 3
        assert torch.equal(x, ref)
        assert cs.cs_admm(plan, yd, 1e-3, 1.0, 25000, z)["launches"] == count
        assert torch.equal(z, zref)
        # watched, with a tolerance that is never met: launches end at 10000,
        # 15000, 25000 (the check points are 15000 apart)
        cs.cs_set_monitor(plan, xt, 1e-30, 15000)
        x.zero_()
        st = cs.cs_ista(plan, yd, 1e-3, tau, 25000, x)
        assert st["launches"] == 3 and st["iters_run"] == 25000 and st["converged"] == 0
        assert torch.equal(x, ref)
    finally:
        plan.close()
