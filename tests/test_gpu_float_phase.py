"""Float32 costs and many rounds: the phases e^{-i gamma C} have to be of unit
length to float32 rounding, or every round scales the whole state alike and
<C> drifts in proportion to p.

Annealing-like ramps (|<C>| about twice the rms cost, so a drift shows) against
the complex128 oracle, for every kernel family that evaluates float32 phases: on
chip (n <= 12), one launch (13..20), passes, multi-angle and the Grover mixer.
Tolerance: what is left per round is the rounding of two or three
common scale factors (2^-25 each at most, 2 ulp-parts of <C> each, signs at
random) and of the amplitudes themselves (averaged over the state), about 6e-8
a round in the rms: 5 sigma over p rounds is 3e-7 sqrt(p) of max(|<C>|, rms C),
and twice that for the gradient, whose adjoint vector goes through the rounds a
second time, relative to the larger of its largest component and the rms C.
With the hardware sine and cosine alone <C> is off by about 1.5e-7 p.
"""

import numpy as np
import pytest
import torch

from qaoa_inputs import erdos_renyi, sk_couplings

pytestmark = pytest.mark.gpu
P = 24


@pytest.fixture(scope="module")
def Q():
    import paper_2312_06451_gb300 as qg

    with qg.Context(0) as ctx:
        yield qg, ctx


def ramp(p, c, seed):
    r = np.random.default_rng(seed)
    t = (np.arange(p) + 0.5) / p
    return np.concatenate([0.6 * (1 - t) + 0.05 * r.uniform(-1, 1, p), -(0.3 + t) * r.uniform(0.8, 1.2, p) / np.std(c)])


def check(got, want, c, p):
    rms = float(np.sqrt(np.mean(c**2)))
    assert abs(got[0] - want[0]) <= 3e-7 * np.sqrt(p) * max(abs(want[0]), rms)
    assert np.abs(got[1] - want[1]).max() <= 6e-7 * np.sqrt(p) * max(np.abs(want[1]).max(), rms)


def sk(ctx, oracle_mod, n, seed):
    J = sk_couplings(n, seed)
    return ctx.cost_precompute("sk", n, J=J, dtype=torch.float32), oracle_mod.cost_sk(n, J.astype(np.float64))


@pytest.mark.parametrize("n,p", [(5, P), (9, P), (10, P), (12, P), (13, P), (15, P), (16, P), (17, P), (20, P), (21, 12)])
@pytest.mark.parametrize("seed", [1, 2])
def test_transverse_field(Q, oracle_mod, n, p, seed):
    qg, ctx = Q
    cost, c = sk(ctx, oracle_mod, n, 700 + 10 * n + seed)
    a = ramp(p, c, 40 * n + seed)
    check(ctx.gradient(cost, qg.XMixer(n), a), oracle_mod.qaoa_gradient(n, c, a), c, p)


@pytest.mark.parametrize("ckpt", ["none", "round", "pass"])
def test_passes(Q, oracle_mod, ckpt):
    qg, _ = Q
    n = 14
    with qg.Context(0) as ctx:
        ctx.set_tuning(dict(n=n, cost_dtype=0, cmin=4, split=0, nbuf_bwd_contig=1, nbuf_bwd_gather=1))
        cost, c = sk(ctx, oracle_mod, n, 731)
        a = ramp(P, c, 732)
        check(ctx.gradient(cost, qg.XMixer(n), a, None, ckpt), oracle_mod.qaoa_gradient(n, c, a), c, P)


@pytest.mark.parametrize("n", [8, 14])
def test_multi_angle(Q, oracle_mod, n):
    qg, ctx = Q
    cost, c = sk(ctx, oracle_mod, n, 740 + n)
    a = ramp(P, c, 741 + n)
    a = np.concatenate([np.repeat(a[:P], n) * np.random.default_rng(n).uniform(0.9, 1.1, P * n), a[P:]])
    check(ctx.gradient(cost, qg.XMixer(n, multi_angle=True), a), oracle_mod.qaoa_gradient_ma(n, c, a), c, P)


def test_grover(Q, oracle_mod):
    """Densest-k-subgraph costs given in float32, off the integers."""
    qg, ctx = Q
    n, k = 12, 5
    st = oracle_mod.dicke_states(n, k)
    c = (oracle_mod.cost_dks(n, erdos_renyi(n, 0.5, 750), st) * 0.37).astype(np.float32)
    cost = torch.from_numpy(c).cuda()
    c = c.astype(np.float64)
    a = ramp(P, c, 751)
    check(ctx.gradient(cost, qg.GroverMixer.dicke(n, k), a), oracle_mod.qaoa_gradient(n, c, a, mixer="grover", states=st), c, P)
