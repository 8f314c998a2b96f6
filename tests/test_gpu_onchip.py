"""The on-chip X-mixer kernel (n <= 12) against the oracle: every qubit count
(the padded ones below 9 included), odd and even round counts (the register
layouts alternate), a round count past one coefficient chunk (32), both cost
types, given initial states, and rounds in the direct rotation form
(|cos beta| < 2^-12) and with per-layout factors (|cos beta| < 1/4)."""

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
        e = erdos_renyi(n, 0.6, 500 + n) if n > 1 else np.zeros((0, 2), np.int32)
        return ctx.cost_precompute("maxcut", n, edges=e, dtype=torch.uint8), oracle_mod.cost_maxcut(n, e)
    J = sk_couplings(n, 500 + n)
    return ctx.cost_precompute("sk", n, J=J, dtype=torch.float32), oracle_mod.cost_sk(n, J.astype(np.float64))


def check(got, want, c):
    # the library's bounds: <C> to 1e-5 of max(|E|, rms C), the gradient to 1e-4 of its largest component
    sig = float(np.sqrt(np.mean(c**2)))
    assert abs(got[0] - want[0]) <= 1e-5 * max(abs(want[0]), sig)
    assert np.abs(got[1] - want[1]).max() <= 1e-4 * max(np.abs(want[1]).max(), 1e-3 * sig)


@pytest.mark.parametrize("kind", ["u8", "f32"])
@pytest.mark.parametrize("p", [1, 2, 3, 33])
@pytest.mark.parametrize("n", range(1, 13))
def test_gradient(qgm, oracle_mod, n, p, kind):
    with qgm.Context(0) as ctx:
        cost, c = instance(ctx, oracle_mod, n, kind)
        ang = uniform_angles(p, 600 + n + 31 * p)[0]
        if p > 2:
            ang[1] = np.pi / 2 - 1e-5  # direct form
            ang[2] = np.pi / 2 - 0.1   # per-layout factors
        want = oracle_mod.qaoa_gradient(n, c, ang)
        check(ctx.gradient(cost, qgm.XMixer(n), ang), want, c)
        E = ctx.expectation(cost, qgm.XMixer(n), ang)
        assert abs(E - want[0]) <= 1e-5 * max(abs(want[0]), float(np.sqrt(np.mean(c**2))))


@pytest.mark.parametrize("n", [3, 8, 9, 10, 11, 12])
def test_initial_state(qgm, oracle_mod, n):
    r = np.random.default_rng(n)
    psi = r.standard_normal(1 << n) + 1j * r.standard_normal(1 << n)
    psi = (psi / np.linalg.norm(psi)).astype(np.complex64)
    ang = uniform_angles(3, 700 + n)[0]
    with qgm.Context(0) as ctx:
        cost, c = instance(ctx, oracle_mod, n, "f32")
        got = ctx.gradient(cost, qgm.XMixer(n), ang, torch.from_numpy(psi).cuda())
    check(got, oracle_mod.qaoa_gradient(n, c, ang, psi0=psi.astype(np.complex128)), c)


def test_classes_in_one_call(qgm, oracle_mod):
    """Instances of every launch class and both cost types in one batched call."""
    with qgm.Context(0) as ctx:
        jobs, want = [], []
        for n in (2, 9, 10, 11, 12):
            for kind in ("u8", "f32"):
                cost, c = instance(ctx, oracle_mod, n, kind)
                a = uniform_angles(4, 800 + n, 3)
                A = torch.from_numpy(a).cuda()
                jobs.append(dict(cost=cost, mixer=qgm.XMixer(n), angles=A, E=torch.zeros(3, dtype=torch.float64, device="cuda"),
                                 grad=torch.zeros_like(A)))
                want.append((c, n, a))
        ctx.expectation_batched(jobs, want_grad=True)
        torch.cuda.synchronize()
        for j, (c, n, a) in zip(jobs, want):
            for s in range(3):
                check((float(j["E"][s]), j["grad"][s].cpu().numpy()), oracle_mod.qaoa_gradient(n, c, a[s]), c)
