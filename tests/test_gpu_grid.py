"""The cooperative X-mixer launches (13 <= n <= 20) against the oracle: every
qubit count (2 to 256 CTAs a set, one or two layouts after an exchange), odd and
even round counts (the tilings alternate), both cost types, given initial
states, the direct rotation form and per-layout factors, round counts past one
coefficient chunk, and sets of different sizes in one call."""

import numpy as np
import pytest
import torch

from qaoa_inputs import erdos_renyi, sk_couplings, uniform_angles

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qgm():
    import paper_2312_06451_gb300 as qg

    return qg


def instance(ctx, oracle_mod, n, kind):
    if kind == "u8":
        e = erdos_renyi(n, 0.5, 900 + n)
        return ctx.cost_precompute("maxcut", n, edges=e, dtype=torch.uint8), oracle_mod.cost_maxcut(n, e)
    J = sk_couplings(n, 900 + n)
    return ctx.cost_precompute("sk", n, J=J, dtype=torch.float32), oracle_mod.cost_sk(n, J.astype(np.float64))


def check(got, want, c):
    # the library's bounds: <C> to 1e-5 of max(|E|, rms C), the gradient to 1e-4 of its largest component
    sig = float(np.sqrt(np.mean(c**2)))
    assert abs(got[0] - want[0]) <= 1e-5 * max(abs(want[0]), sig)
    assert np.abs(got[1] - want[1]).max() <= 1e-4 * np.abs(want[1]).max()


def took_grid(ctx):
    return any(k.startswith("grid_") and v["launches"] for k, v in ctx.kernel_stats().items())


@pytest.mark.parametrize("kind", ["u8", "f32"])
@pytest.mark.parametrize("n,p", [(13, 1), (13, 4), (14, 3), (15, 2), (15, 35), (16, 1), (16, 3), (17, 1), (17, 4), (18, 3), (19, 2), (20, 1), (20, 2)])
def test_gradient(qgm, oracle_mod, n, p, kind):
    with qgm.Context(0) as ctx:
        cost, c = instance(ctx, oracle_mod, n, kind)
        ang = uniform_angles(p, 1000 + n + 31 * p)[0]
        if p > 2:
            ang[1] = np.pi / 2 - 1e-5  # direct form
            ang[2] = np.pi / 2 - 0.1   # per-layout factors
        ctx.set_profiling(True)
        want = oracle_mod.qaoa_gradient(n, c, ang)
        for ckpt in ("round", "pass"):
            check(ctx.gradient(cost, qgm.XMixer(n), ang, None, ckpt), want, c)
        E = ctx.expectation(cost, qgm.XMixer(n), ang)
        assert abs(E - want[0]) <= 1e-5 * max(abs(want[0]), float(np.sqrt(np.mean(c**2))))
        assert took_grid(ctx)


@pytest.mark.parametrize("n", [13, 16, 17, 20])
def test_initial_state(qgm, oracle_mod, n):
    r = np.random.default_rng(n)
    psi = r.standard_normal(1 << n) + 1j * r.standard_normal(1 << n)
    psi = (psi / np.linalg.norm(psi)).astype(np.complex64)
    ang = uniform_angles(2, 1100 + n)[0]
    with qgm.Context(0) as ctx:
        cost, c = instance(ctx, oracle_mod, n, "f32")
        got = ctx.gradient(cost, qgm.XMixer(n), ang, torch.from_numpy(psi).cuda())
    check(got, oracle_mod.qaoa_gradient(n, c, ang, psi0=psi.astype(np.complex128)), c)


def test_sizes_in_one_call(qgm, oracle_mod):
    """Sets of different sizes share a launch, next to on-chip and pass units; a second call replays the plan."""
    with qgm.Context(0) as ctx:
        jobs, want = [], []
        for n, kind, sets in ((13, "u8", 3), (16, "u8", 2), (15, "f32", 2), (17, "u8", 1), (18, "f32", 1), (11, "u8", 2), (21, "u8", 1)):
            cost, c = instance(ctx, oracle_mod, n, kind)
            a = uniform_angles(2, 1200 + n, sets)
            A = torch.from_numpy(a).cuda()
            jobs.append(dict(cost=cost, mixer=qgm.XMixer(n), angles=A, E=torch.zeros(sets, dtype=torch.float64, device="cuda"),
                             grad=torch.zeros_like(A)))
            want.append([oracle_mod.qaoa_gradient(n, c, x) + (c,) for x in a])
        call = ctx.batched_call(jobs, want_grad=True)
        for _ in range(2):
            for j in jobs:
                j["E"].zero_()
                j["grad"].zero_()
            call.run()
            torch.cuda.synchronize()
            for j, w in zip(jobs, want):
                for s, (E, g, c) in enumerate(w):
                    check((float(j["E"][s]), j["grad"][s].cpu().numpy()), (E, g), c)


@pytest.mark.parametrize("sets,grid", [(2, True), (6, True), (7, False)])
def test_waves(qgm, oracle_mod, sets, grid):
    """More sets of n = 19 (128 CTAs each) than the chip holds: up to three launches, then the passes."""
    n = 19
    with qgm.Context(0) as ctx:
        cost, c = instance(ctx, oracle_mod, n, "u8")
        a = uniform_angles(1, 1250, sets)
        A = torch.from_numpy(a).cuda()
        E, G = torch.zeros(sets, dtype=torch.float64, device="cuda"), torch.zeros_like(A)
        ctx.set_profiling(True)
        ctx.expectation_batched([dict(cost=cost, mixer=qgm.XMixer(n), angles=A, E=E, grad=G)], want_grad=True)
        torch.cuda.synchronize()
        assert took_grid(ctx) == grid or torch.cuda.get_device_properties(0).multi_processor_count != 152
        for s in range(sets):
            check((float(E[s]), G[s].cpu().numpy()), oracle_mod.qaoa_gradient(n, c, a[s]), c)


def test_passes_where_asked(qgm, oracle_mod):
    """Gradients without checkpoints, an installed schedule and a cap on the state scratch keep the pass kernels."""
    n = 17
    ang = uniform_angles(3, 1300)[0]
    with qgm.Context(0) as ctx:
        cost, c = instance(ctx, oracle_mod, n, "f32")
        want = oracle_mod.qaoa_gradient(n, c, ang)
        ctx.set_profiling(True)
        check(ctx.gradient(cost, qgm.XMixer(n), ang, None, "none"), want, c)
        ctx.set_state_limit(2 << 20)  # two vectors
        check(ctx.gradient(cost, qgm.XMixer(n), ang, None, "round"), want, c)
        ctx.set_state_limit(None)
        ctx.set_tuning(dict(n=n, cost_dtype=0, cmin=4, split=0, nbuf_bwd_contig=1, nbuf_bwd_gather=1))
        check(ctx.gradient(cost, qgm.XMixer(n), ang, None, "pass"), want, c)
        assert not took_grid(ctx)
