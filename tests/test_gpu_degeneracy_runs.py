"""Degeneracies counted per (k-2)-set (densest k-subgraph and k-vertex cover
through the complement, set sizes 5..8, from 2^21 (k-1)-sets on) against a count
by halves, exactly: a set is its lower part, whose largest vertex is m, and its
upper part, all above m; the inside edges of all pairs of parts come from one
matrix product.  Dense, sparse, empty and complete graphs, one to four 32-bit
words of vertices."""

import math

import numpy as np
import pytest
import torch

from qaoa_inputs import erdos_renyi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2312_06451_gb300 as qg

    with qg.Context(0) as c:
        yield c


def by_halves(n, k, edges):
    A = torch.zeros(n, n, device="cuda")
    e = torch.from_numpy(np.asarray(edges, dtype=np.int64).reshape(-1, 2)).cuda()
    A[e[:, 0], e[:, 1]] = 1
    A[e[:, 1], e[:, 0]] = 1
    low, top = (k + 1) // 2, k * (k - 1) // 2 + 1
    counts = torch.zeros(top, dtype=torch.int64, device="cuda")

    def rows(lo, hi, size):
        sets = torch.combinations(torch.arange(lo, hi, device="cuda"), size)
        return torch.zeros(sets.shape[0], n, device="cuda").scatter_(1, sets, 1.0)

    for m in range(low - 1, n - (k - low)):
        P, Q = rows(0, m, low - 1), rows(m + 1, n, k - low)
        P[:, m] = 1
        ip, iq = ((P @ A) * P).sum(1) / 2, ((Q @ A) * Q).sum(1) / 2
        step = max(1, (1 << 25) // Q.shape[0])
        for i in range(0, P.shape[0], step):
            c = (P[i:i + step] @ A) @ Q.T + ip[i:i + step, None] + iq[None, :]
            counts += torch.bincount(c.reshape(-1).round().to(torch.int32), minlength=top)
    return counts.cpu().numpy()


@pytest.mark.parametrize("n,k,p_edge", [(88, 5, 0.5), (128, 5, 0.2), (100, 5, 1.0), (52, 6, 0.5), (66, 6, 0.9), (99, 6, 0.5), (60, 6, 0.0),
                                        (40, 7, 0.5), (45, 7, 0.8), (33, 8, 0.5), (34, 8, 1.0)])
def test_counts(ctx, n, k, p_edge):
    e = erdos_renyi(n, p_edge, 1500 + n + k)
    assert math.comb(n, k - 1) >= 1 << 21
    top = k * (k - 1) // 2 + 1
    got = ctx.cost_degeneracy("dks", n, edges=e, k=k, n_bins=max(top, 1)).cpu().numpy()
    want = by_halves(n, k, e)
    assert want.sum() == math.comb(n, k)
    assert np.array_equal(got, want)


@pytest.mark.parametrize("n,kk", [(54, 6), (41, 7)])
def test_cover_counts(ctx, n, kk):
    """k-vertex cover with n - k = kk: m minus the edges inside the complement."""
    e = erdos_renyi(n, 0.4, 1700 + n)
    got = ctx.cost_degeneracy("kvc", n, edges=e, k=n - kk, n_bins=len(e) + 1).cpu().numpy()
    inside = by_halves(n, kk, e)
    want = np.zeros(len(e) + 1, dtype=np.int64)
    for i, c in enumerate(inside):
        if c:
            want[len(e) - i] += c
    assert np.array_equal(got, want)
