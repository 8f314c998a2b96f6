"""Eigenbasis mixers with costs near the ends of the float32 range: costs times
2^e with gammas times 2^-e give the same phases bit for bit, so <C> and the beta
gradient are the unscaled ones times 2^e, up to the products' rounding."""

import numpy as np
import pytest
import torch

from qaoa_inputs import erdos_renyi, uniform_angles

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["dense", "blocks"])
@pytest.mark.parametrize("e", [-100, -60, 60, 100, 112, 118])
def test_scaled_costs(form, e):
    import paper_2312_06451_gb300 as qg

    n, k, p = 10, 4, 2
    with qg.Context(0) as ctx:
        cost = ctx.cost_precompute("dks", n, edges=erdos_renyi(n, 0.6, 960), k=k, dtype=torch.uint8).to(torch.float32)
        make = qg.xy_eigen_mixer if form == "dense" else qg.xy_sym_mixer
        mixer = make(ctx, "ring", n, k, precision="3xtf32")
        a = uniform_angles(p, 961)[0]
        b = a.copy()
        b[p:] = np.ldexp(a[p:], -e)
        E, g = ctx.gradient(cost, mixer, a)
        Es, gs = ctx.gradient(torch.ldexp(cost, torch.tensor(e, device="cuda")), mixer, b)
    assert abs(np.ldexp(Es, -e) - E) <= 1e-5 * abs(E)
    assert np.abs(np.ldexp(gs[:p], -e) - g[:p]).max() <= 1e-4 * np.abs(g[:p]).max()
