"""qaoa_cost_precompute into outputs that are aligned for one value only (cost
vectors packed one behind the other): the values of an aligned output, and
nothing written around them."""

import ctypes

import numpy as np
import pytest
import torch

from qaoa_inputs import erdos_renyi, sk_couplings

pytestmark = pytest.mark.gpu
GUARD = 0xA5


@pytest.fixture(scope="module")
def Q():
    import paper_2312_06451_gb300 as qg

    with qg.Context(0) as ctx:
        yield qg, ctx


def precompute(qg, ctx, prob, n, dtype, offset):
    """The cost vector written `offset` bytes into a buffer, and the status."""
    size = 1 if dtype == torch.uint8 else 4
    buf = torch.full((64 + (size << n) + 64,), GUARD, dtype=torch.uint8, device="cuda")
    assert buf.data_ptr() % 16 == 0
    st = ctx._lib.qaoa_cost_precompute(ctx._h, ctypes.byref(prob), ctypes.c_void_p(buf.data_ptr() + 64 + offset),
                                       1 if dtype == torch.uint8 else 0, 1 << n)
    b = buf.cpu().numpy()
    lo, hi = 64 + offset, 64 + offset + (size << n)
    assert (b[:lo] == GUARD).all() and (b[hi:] == GUARD).all()
    return st, b[lo:hi].copy().view(np.uint8 if size == 1 else np.float32)


@pytest.mark.parametrize("n", [1, 2, 5, 12, 13, 22])
@pytest.mark.parametrize("kind,offsets", [("u8", (0, 1, 2, 3, 4, 7)), ("f32", (0, 4, 8, 12)), ("sk", (0, 4, 8)), ("wide", (0, 4, 12))])
def test_same_values(Q, n, kind, offsets):
    qg, ctx = Q
    B = qg.B
    e = np.ascontiguousarray(erdos_renyi(n, 0.6, 60 + n) if n > 1 else np.zeros((0, 2)), dtype=np.int32)
    if kind in ("u8", "f32"):
        dtype = torch.uint8 if kind == "u8" else torch.float32
        prob = B.QaoaProblem(B.QAOA_PROBLEM_MAXCUT, n, -1, len(e), e.ctypes.data_as(ctypes.c_void_p), None, None)
        want = ctx.cost_precompute("maxcut", n, edges=e, dtype=dtype)
    else:
        dtype = torch.float32
        J = sk_couplings(n, 61 + n).astype(np.float32)
        if kind == "wide":  # 64-bit sums
            J = np.ascontiguousarray(J * np.float32(1 + 2.0**-10), dtype=np.float32)
        prob = B.QaoaProblem(B.QAOA_PROBLEM_SK, n, -1, 0, None, None, J.ctypes.data_as(ctypes.c_void_p))
        want = ctx.cost_precompute("sk", n, J=J, dtype=dtype)
    want = want.cpu().numpy()
    for off in offsets:
        st, got = precompute(qg, ctx, prob, n, dtype, off)
        assert st == 0
        assert np.array_equal(got, want)


def test_float_output_off_its_grid_is_refused(Q):
    qg, ctx = Q
    J = np.ones((3, 3), dtype=np.float32)
    prob = qg.B.QaoaProblem(qg.B.QAOA_PROBLEM_SK, 3, -1, 0, None, None, J.ctypes.data_as(ctypes.c_void_p))
    st, got = precompute(qg, ctx, prob, 3, torch.float32, 2)
    assert st == qg.B.QAOA_ERR_INVALID and (got.view(np.uint8) == GUARD).all()
