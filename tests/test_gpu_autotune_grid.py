"""Autotuning sizes that have a one-launch kernel (13 <= n <= 20): the tuned
schedule serves the calls that need passes and does not keep the others from the
one-launch kernel; nor does a tuning file written earlier.  A schedule set
without a tuning time is pinned."""

import numpy as np
import pytest
import torch

from qaoa_inputs import sk_couplings, uniform_angles

pytestmark = pytest.mark.gpu


def families(ctx, f):
    """The kernel families that f() launched."""
    before = {k: v["launches"] for k, v in ctx.kernel_stats().items()}
    f()
    return [k for k, v in ctx.kernel_stats().items() if v["launches"] > before.get(k, 0)]


@pytest.mark.parametrize("n,grad", [(13, True), (16, True), (16, False), (20, True)])
def test_autotuned_sizes_keep_the_one_launch_kernel(tmp_path, oracle_mod, n, grad):
    import paper_2312_06451_gb300 as qg

    J = sk_couplings(n, 910 + n)
    ang = uniform_angles(3, 911 + n)[0]
    c = oracle_mod.cost_sk(n, J.astype(np.float64))
    E, g = oracle_mod.qaoa_gradient(n, c, ang)
    path = str(tmp_path / "tuning.json")
    with qg.Context(0) as ctx:
        cost = ctx.cost_precompute("sk", n, J=J, dtype=torch.float32)
        ctx.set_profiling(True)
        t = ctx.autotune(cost, n, p=2, want_grad=grad)
        assert t["ms"] > 0 and ctx.get_tuning(n, 0) == t
        ctx.save_tuning(path)

        def run(ckpt="pass"):
            got = ctx.gradient(cost, qg.XMixer(n), ang, None, ckpt)
            assert abs(got[0] - E) <= 1e-5 * max(abs(E), np.sqrt(np.mean(c**2)))
            assert np.abs(got[1] - g).max() <= 1e-4 * np.abs(g).max()

        assert any(k.startswith("grid_") for k in families(ctx, run))
        assert not any(k.startswith("grid_") for k in families(ctx, lambda: run("none")))
    with qg.Context(0) as ctx:
        ctx.load_tuning(path)
        ctx.set_profiling(True)
        assert any(k.startswith("grid_") for k in families(ctx, run))
        ctx.set_tuning({k: t[k] for k in ("n", "cost_dtype", "cmin", "split", "nbuf_bwd_contig", "nbuf_bwd_gather")})
        assert not any(k.startswith("grid_") for k in families(ctx, run))
