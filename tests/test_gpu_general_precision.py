"""Sum-of-products X mixers by passes: the half rounds' rotations by pi/4 keep
the norm, so <C> does not drift with the rounds and the qubits.

Tolerance as for the other float32 states over many rounds: the common scale
factors of a round (here up to two half rounds of two passes, 2^-25 each, and the
phases' tables) and the amplitudes' own rounding, about 8e-8 a round in the rms;
4e-7 sqrt(p) of max(|<C>|, rms C) and twice that for the gradient, relative to the
larger of its largest component and the rms C times the mixer's largest
eigenvalue.  A rounded cosine of pi/4 in each of 2 n rotations a round would
shift <C> by 7e-8 n p."""

import numpy as np
import pytest
import torch

from qaoa_inputs import erdos_renyi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.uint8, torch.float32])
@pytest.mark.parametrize("n,p", [(13, 12), (14, 12), (16, 8), (17, 8), (20, 4)])
def test_norm_kept(oracle_mod, n, p, dtype):
    import paper_2312_06451_gb300 as qg

    e = erdos_renyi(n, 0.5, 940 + n)
    c = oracle_mod.cost_maxcut(n, e)
    r = np.random.default_rng(941 + n)
    t = (np.arange(p) + 0.5) / p
    mixer = qg.x_terms_mixer(n, {1: 1.0, 2: 0.1})
    d = oracle_mod.krawtchouk_weights(n, {1: 1.0, 2: 0.1})
    a = np.concatenate([0.4 * (1 - t) + 0.03 * r.uniform(-1, 1, p), -(0.3 + t) * r.uniform(0.8, 1.2, p) / np.std(c)])
    E, g = oracle_mod.qaoa_gradient_general(n, d, c, a)
    rms = float(np.sqrt(np.mean(c**2)))
    with qg.Context(0) as ctx:
        cost = ctx.cost_precompute("maxcut", n, edges=e, dtype=dtype)
        got = ctx.gradient(cost, mixer, a)
    assert abs(got[0] - E) <= 4e-7 * np.sqrt(p) * max(abs(E), rms)
    assert np.abs(got[1] - g).max() <= 8e-7 * np.sqrt(p) * max(np.abs(g).max(), rms * np.abs(d).max())
