"""Orbit transforms whose M_r are compile-time constants (cyclic orbits of full
period 10 to 16, 18 and 20), beside lengths that read M_r (9, 17) and the
shorter orbits of the same subspaces, against the CPU oracle, which forms no
orbits.  Tolerances of the block-diagonal mixers: a gradient is about 30 (p + 1)
float32 roundings of order 6e-8 on values of order sigma_C, under
|dE| <= 1e-5 max(|E|, sigma_C) and |dg_i| <= 1e-4 max|g|.
"""

import numpy as np
import pytest
import torch

from qaoa_inputs import erdos_renyi, uniform_angles

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def Q():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import paper_2312_06451_gb300 as qg

    ctx = qg.Context(0)
    yield qg, ctx
    ctx.close()


@pytest.mark.parametrize("uniform", [True, False])
@pytest.mark.parametrize("n,k", [(9, 4), (10, 5), (11, 3), (12, 2), (12, 4), (13, 2), (14, 4), (14, 7), (15, 3), (16, 2), (16, 4), (17, 2), (18, 2), (18, 3), (20, 2)])
def test_orbit_lengths(Q, oracle_mod, n, k, uniform):
    qg, ctx = Q
    p = 3
    e = erdos_renyi(n, 0.5, 900 + n + k)
    st = oracle_mod.dicke_states(n, k)
    c = oracle_mod.cost_dks(n, e, st)
    dc = ctx.cost_precompute("dks", n, edges=e, k=k, dtype=torch.uint8)
    mixer = qg.xy_sym_mixer(ctx, "ring", n, k, precision="fp32")
    init = None
    if not uniform:
        rng = np.random.default_rng(n * 100 + k)
        init = rng.standard_normal(len(st)) + 1j * rng.standard_normal(len(st))
        init = (init / np.linalg.norm(init)).astype(np.complex64)
    ang = uniform_angles(p, 910 + n + k)[0]
    psi0 = None if init is None else init.astype(np.complex128)
    E_ref, g_ref = oracle_mod.qaoa_gradient(n, c, ang, "ring", st, psi0=psi0)
    d_init = None if init is None else torch.view_as_real(torch.from_numpy(init).cuda()).contiguous()
    E, g = ctx.gradient(dc, mixer, ang, init=d_init)
    E0 = ctx.expectation(dc, mixer, ang, init=d_init)
    scale = max(abs(E_ref), float(np.sqrt(np.mean(np.asarray(c, dtype=np.float64) ** 2))))
    assert abs(E - E_ref) <= 1e-5 * scale and abs(E0 - E_ref) <= 1e-5 * scale
    np.testing.assert_allclose(g, g_ref, rtol=0, atol=1e-4 * np.abs(g_ref).max())
