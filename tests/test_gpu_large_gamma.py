"""Integer costs at gammas of many whole turns: e^{-i gamma c} for a whole c only
depends on gamma modulo 2 pi, so the phase tables have to be as exact as the
float64 gamma / (2 pi) however large it is.

The oracle takes the reduced gammas (60-digit arithmetic).  Tolerance on <C>:
1e-6 of max(|<C>|, rms C) for the complex64 state, and the derivative by each
gamma times the rounding of gamma / (2 pi) to float64, at most 1.5 2^-53 of it
(the product and 1 / (2 pi) itself)."""

from decimal import Decimal, getcontext

import numpy as np
import pytest
import torch

from qaoa_inputs import erdos_renyi, uniform_angles

pytestmark = pytest.mark.gpu
getcontext().prec = 60
TWO_PI = 2 * Decimal("3.14159265358979323846264338327950288419716939937510582097494459")


def reduced(gamma):
    d = Decimal(float(gamma))
    return float(d - TWO_PI * (d / TWO_PI).to_integral_value())


@pytest.mark.parametrize("seed", range(5))
@pytest.mark.parametrize("n,path", [(4, "x"), (10, "x"), (12, "x"), (14, "x"), (18, "x"), (14, "passes"), (10, "ma")])
def test_whole_turns(oracle_mod, n, path, seed):
    import paper_2312_06451_gb300 as qg

    p = 3
    e = erdos_renyi(n, 0.7, 930 + n)
    c = oracle_mod.cost_maxcut(n, e)
    a = uniform_angles(p, 931 + 10 * n + seed)[0]
    a[:p] *= 0.25
    r = np.random.default_rng(932 + seed)
    a[p:] = 0.3 * a[p:] / np.std(c) + 2 * np.pi * np.rint(r.uniform(0.5e10, 1e10, p)) * np.array([1, -1, 1])
    turns = np.abs(a[p:]) / (2 * np.pi)
    low = a.copy()
    low[p:] = [reduced(x) for x in a[p:]]
    E, g = oracle_mod.qaoa_gradient(n, c, low)
    tol = 1e-6 * max(abs(E), float(np.sqrt(np.mean(c**2)))) + 2 * np.pi * 1.5 * 2.0**-53 * float(np.sum(turns * np.abs(g[p:])))
    with qg.Context(0) as ctx:
        if path == "passes":
            ctx.set_tuning(dict(n=n, cost_dtype=1, cmin=4, split=0, nbuf_bwd_contig=1, nbuf_bwd_gather=1))
        cost = ctx.cost_precompute("maxcut", n, edges=e, dtype=torch.uint8)
        if path == "ma":
            b = np.concatenate([np.repeat(a[:p], n), a[p:]])
            got = ctx.expectation(cost, qg.XMixer(n, multi_angle=True), b)
        else:
            got = ctx.expectation(cost, qg.XMixer(n), a)
    assert abs(got - E) <= tol
