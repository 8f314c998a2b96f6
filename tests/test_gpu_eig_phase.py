"""Eigenbasis mixers over many rounds: the phases of costs and eigenvalues keep
the norm, so <C> does not drift with p (two phases a round off unit length by 7e-8
each moved it by 3e-7 p).

float32 products, whose rounding is to nearest, against the oracle's power
series.  Tolerance: amplitudes and sums rounded at random, about 8e-8 a round in
the rms; 4e-7 sqrt(p) of max(|<C>|, rms C), and twice that for the gradient,
relative to the larger of its largest component and the rms C times the mixer's
largest eigenvalue."""

import numpy as np
import pytest
import torch

from qaoa_inputs import erdos_renyi

pytestmark = pytest.mark.gpu
P = 24


@pytest.mark.parametrize("dtype", [torch.uint8, torch.float32])
@pytest.mark.parametrize("form", ["dense", "blocks"])
@pytest.mark.parametrize("n,k", [(10, 3), (12, 5)])
def test_norm_kept(oracle_mod, n, k, form, dtype):
    import paper_2312_06451_gb300 as qg

    st = oracle_mod.dicke_states(n, k)
    e = erdos_renyi(n, 0.6, 950 + n)
    c = oracle_mod.cost_dks(n, e, st)
    r = np.random.default_rng(951 + n)
    t = (np.arange(P) + 0.5) / P
    a = np.concatenate([0.15 * (1 - t) + 0.02 * r.uniform(-1, 1, P), -(0.3 + t) * r.uniform(0.8, 1.2, P) / np.std(c)])
    with qg.Context(0) as ctx:
        cost = ctx.cost_precompute("dks", n, edges=e, k=k, dtype=torch.uint8)
        if dtype == torch.float32:
            c = (c * 0.37).astype(np.float32)
            cost, c = torch.from_numpy(c).cuda(), c.astype(np.float64)
        make = qg.xy_eigen_mixer if form == "dense" else qg.xy_sym_mixer
        mixer = make(ctx, "ring", n, k, precision="fp32")
        got = ctx.gradient(cost, mixer, a)
    E, g = oracle_mod.qaoa_gradient(n, c, a, mixer="ring", states=st)
    rms = float(np.sqrt(np.mean(c**2)))
    assert abs(got[0] - E) <= 4e-7 * np.sqrt(P) * max(abs(E), rms)
    assert np.abs(got[1] - g).max() <= 8e-7 * np.sqrt(P) * max(np.abs(g).max(), rms * 2 * n)
