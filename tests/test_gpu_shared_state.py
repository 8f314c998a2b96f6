"""State memory of calls that mix one-launch X-mixer units (13 <= n <= 20) with
units that run as passes or with the Grover mixer: neither kind takes memory
from the other, so what fits a cap on its own also fits it in a mixed call, and
calls of both kinds on one context hold one state buffer."""

import numpy as np
import pytest
import torch

from qaoa_inputs import erdos_renyi, uniform_angles

pytestmark = pytest.mark.gpu
MIB = 1 << 20


@pytest.fixture()
def Q():
    import paper_2312_06451_gb300 as qg

    with qg.Context(0) as ctx:
        ctx.set_profiling(True)
        yield qg, ctx


def took_grid(ctx):
    return any(k.startswith("grid_") and v["launches"] for k, v in ctx.kernel_stats().items())


def make(qg, ctx, oracle_mod, n, p, sets, kind="x"):
    """A batched gradient job and the oracle's values of its sets."""
    e = erdos_renyi(n, 0.4, 800 + n)
    cost, c = ctx.cost_precompute("maxcut", n, edges=e, dtype=torch.uint8), oracle_mod.cost_maxcut(n, e)
    a = uniform_angles(p, 801 + n, sets)
    a[:, p:] /= np.pi * np.std(c)
    A = torch.from_numpy(a).cuda()
    job = dict(cost=cost, mixer=qg.XMixer(n) if kind == "x" else qg.GroverMixer(1 << n), angles=A,
               E=torch.zeros(sets, dtype=torch.float64, device="cuda"), grad=torch.zeros_like(A))
    return job, [oracle_mod.qaoa_gradient(n, c, x, mixer=kind) for x in a], c


def check(made):
    torch.cuda.synchronize()
    for job, want, c in made:
        rms = float(np.sqrt(np.mean(c**2)))
        for s, (E, g) in enumerate(want):
            assert abs(float(job["E"][s]) - E) <= 1e-5 * max(abs(E), rms)
            assert np.abs(job["grad"][s].cpu().numpy() - g).max() <= 1e-4 * max(np.abs(g).max(), 1e-3 * rms)


def test_pass_unit_that_needs_the_whole_cap(Q, oracle_mod):
    """n = 20 without checkpoints takes exactly 16 MiB, next to an n = 16 gradient in one launch."""
    qg, ctx = Q
    ctx.set_state_limit(16 * MIB)
    made = [make(qg, ctx, oracle_mod, 16, 3, 1), make(qg, ctx, oracle_mod, 20, 2, 1)]
    ctx.expectation_batched([m[0] for m in made], want_grad=True)
    check(made)
    assert took_grid(ctx)


def test_grover_unit_beside(Q, oracle_mod):
    """Four n = 16 gradients in one launch would leave the Grover units less than their smallest form under this cap."""
    qg, ctx = Q
    ctx.set_state_limit(9 * MIB)
    made = [make(qg, ctx, oracle_mod, 16, 2, 4), make(qg, ctx, oracle_mod, 16, 2, 3, "grover")]
    ctx.expectation_batched([m[0] for m in made], want_grad=True)
    check(made)
    ctx.set_state_limit(None)
    assert not took_grid(ctx)
    ctx.expectation_batched([m[0] for m in made], want_grad=True)
    check(made)
    assert took_grid(ctx)


def test_refusal_stays_one(Q, oracle_mod):
    qg, ctx = Q
    made = [make(qg, ctx, oracle_mod, 15, 2, 1), make(qg, ctx, oracle_mod, 20, 2, 1)]
    ctx.set_state_limit(8 * MIB)
    with pytest.raises(qg.QAOAError, match="state scratch"):
        ctx.expectation_batched([m[0] for m in made], want_grad=True)
    ctx.set_state_limit(None)
    ctx.expectation_batched([m[0] for m in made], want_grad=True)
    check(made)


@pytest.mark.parametrize("grid_first", [True, False])
def test_one_buffer_for_both(Q, oracle_mod, grid_first):
    """96 gradients at n = 16 (288 MiB of vectors in one launch) and one at n = 23 (384 MiB with per-pass
    checkpoints), on one context in either order."""
    qg, ctx = Q
    e = erdos_renyi(23, 0.2, 820)
    big = ctx.cost_precompute("maxcut", 23, edges=e, dtype=torch.uint8)
    a = uniform_angles(2, 821)[0]
    made = [make(qg, ctx, oracle_mod, 16, 4, 2)]
    job = made[0][0]
    A = job["angles"].repeat(48, 1)
    many = dict(job, angles=A, E=torch.zeros(96, dtype=torch.float64, device="cuda"), grad=torch.zeros_like(A))

    def grid():
        ctx.expectation_batched([many], want_grad=True)
        torch.cuda.synchronize()
        job["E"].copy_(many["E"][:2])
        job["grad"].copy_(many["grad"][:2])
        check(made)
        assert torch.equal(many["E"].reshape(48, 2), many["E"][:2].expand(48, 2))

    def passes():
        return ctx.gradient(big, qg.XMixer(23), a, None, "pass")

    first, second = (grid, passes) if grid_first else (passes, grid)
    first()
    held = ctx.scratch_bytes()
    second()
    assert took_grid(ctx)
    assert ctx.scratch_bytes() <= max(held, 384 * MIB) + 32 * MIB


def test_capture(oracle_mod):
    """On-chip, one-launch (clusters and cooperative, more than one launch) and pass units of one call captured in a
    CUDA graph, replayed with other angles."""
    import paper_2312_06451_gb300 as qg

    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream), qg.Context(0, stream) as ctx:
        made = [make(qg, ctx, oracle_mod, n, 2, sets) for n, sets in ((11, 3), (13, 2), (16, 2), (17, 1), (19, 2), (20, 1), (21, 1))]
        call = ctx.batched_call([m[0] for m in made], want_grad=True)
        call.run()
        check(made)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            call.run()
        for turn in (1, 2):
            again = []
            for job, _, c in made:
                a = job["angles"].cpu().numpy() * (0.9 if turn == 1 else 1.2)
                job["angles"].copy_(torch.from_numpy(a))
                job["E"].zero_()
                job["grad"].zero_()
                again.append((job, [oracle_mod.qaoa_gradient(int(c.size).bit_length() - 1, c, x) for x in a], c))
            graph.replay()
            check(again)
