"""Cost vectors summed as integer quadratic forms (MaxCut, weighted MaxCut, SK)
against the oracle's float64 sums, bit for bit: instances smaller than a tile,
tile edges, and the sizes where a block takes 2, 4, 8 and 16 tiles; 32- and
64-bit sums, and couplings without a common grid (the float64 kernels)."""

import numpy as np
import pytest
import torch

from qaoa_inputs import erdos_renyi, sk_couplings

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2312_06451_gb300 as qg

    with qg.Context(0) as c:
        yield c


SIZES = [1, 2, 3, 5, 9, 11, 12, 13, 14, 17, 21, 22, 23, 24]


@pytest.mark.parametrize("n", SIZES)
def test_maxcut(ctx, oracle_mod, n):
    e = erdos_renyi(n, 0.6, 70 + n) if n > 1 else np.zeros((0, 2), np.int32)
    want = oracle_mod.cost_maxcut(n, e)
    for dtype in (torch.uint8, torch.float32):
        got = ctx.cost_precompute("maxcut", n, edges=e, dtype=dtype).cpu().numpy()
        assert np.array_equal(got.astype(np.float64), want)


@pytest.mark.parametrize("weights", ["random", "signed", "coarse", "spread"])
@pytest.mark.parametrize("n", [2, 7, 12, 15, 21, 22])
def test_weighted(ctx, oracle_mod, n, weights):
    e = erdos_renyi(n, 0.7, 170 + n)
    r = np.random.default_rng(n)
    w = r.random(len(e)).astype(np.float32)
    if weights == "signed":
        w = r.standard_normal(len(e)).astype(np.float32)
    elif weights == "coarse":  # multiples of 2^10: a grid above 1
        w = (1024.0 * r.integers(-5, 6, len(e))).astype(np.float32)
    elif weights == "spread":  # 80 powers of two apart: no exact integer sum
        w = (w * 2.0 ** r.integers(-40, 41, len(e))).astype(np.float32)
    want = oracle_mod.cost_maxcut(n, e, w.astype(np.float64))
    got = ctx.cost_precompute("wmaxcut", n, edges=e, weights=w, dtype=torch.float32).cpu().numpy()
    if weights == "spread":  # float64 sums of at most 2^8 terms: 2^-44 of the sum of |w|, rounded once to float32
        assert np.all(np.abs(got - want) <= 2.0**-24 * np.abs(want) + 2.0**-44 * np.abs(w.astype(np.float64)).sum())
    else:
        assert np.array_equal(got, want.astype(np.float32))


@pytest.mark.parametrize("fine", [False, True])  # 32-bit sums (the 2^-20 grid), 64-bit sums (all 24 bits of float32)
@pytest.mark.parametrize("n", [1, 2, 6, 12, 13, 16, 21, 23, 25])
def test_sk(ctx, oracle_mod, n, fine):
    J = sk_couplings(n, 270 + n)
    if fine:
        J = np.random.default_rng(n).standard_normal((n, n)).astype(np.float32)
        J = np.triu(J, 1) + np.triu(J, 1).T
    want = oracle_mod.cost_sk(n, J.astype(np.float64)).astype(np.float32)
    got = ctx.cost_precompute("sk", n, J=J, dtype=torch.float32).cpu().numpy()
    assert np.array_equal(got, want)
