"""Sets of 17 to 20 qubits with one cost type in one call: they share cooperative
launches (32 to 256 CTAs a set, found by a search over unequal descriptors, each
set with its own arrival counter), filled in order up to the chip's residency."""

import numpy as np
import pytest
import torch

from qaoa_inputs import erdos_renyi, sk_couplings, uniform_angles

pytestmark = pytest.mark.gpu


def launches_needed(sizes, room):
    """Launches of sets filled in order, each of at most `room` CTAs."""
    n, used = 1, 0
    for q in sizes:
        c = 1 << (q - 12)
        if used + c > room:
            n, used = n + 1, 0
        used += c
    return n


@pytest.mark.parametrize("kind", ["u8", "f32"])
@pytest.mark.parametrize("order", [(17, 18, 19, 20), (20, 17, 19, 18), (18, 19, 18, 17, 19, 20)])
def test_mixed_sizes(oracle_mod, kind, order):
    import paper_2312_06451_gb300 as qg

    room = 2 * torch.cuda.get_device_properties(0).multi_processor_count  # two CTAs an SM
    need = launches_needed(order, room)
    with qg.Context(0) as ctx:
        jobs, want = [], []
        for i, n in enumerate(order):
            if kind == "u8":
                e = erdos_renyi(n, 0.3, 970 + n + i)
                cost, c = ctx.cost_precompute("maxcut", n, edges=e, dtype=torch.uint8), oracle_mod.cost_maxcut(n, e)
            else:
                J = sk_couplings(n, 970 + n + i)
                cost, c = ctx.cost_precompute("sk", n, J=J, dtype=torch.float32), oracle_mod.cost_sk(n, J.astype(np.float64))
            a = uniform_angles(2, 971 + n + i)
            A = torch.from_numpy(a).cuda()
            jobs.append(dict(cost=cost, mixer=qg.XMixer(n), angles=A, E=torch.zeros(1, dtype=torch.float64, device="cuda"),
                             grad=torch.zeros_like(A)))
            want.append(oracle_mod.qaoa_gradient(n, c, a[0]) + (float(np.sqrt(np.mean(c**2))),))
        ctx.set_profiling(True)
        call = ctx.batched_call(jobs, want_grad=True)
        for _ in range(2):
            ctx.reset_stats()
            call.run()
            torch.cuda.synchronize()
            stats = {k: v["launches"] for k, v in ctx.kernel_stats().items() if v["launches"]}
            assert need <= 3 and stats.get("grid_grad_" + kind) == need and not any(k.startswith("xpass") for k in stats)
            for j, (E, g, rms) in zip(jobs, want):
                assert abs(float(j["E"][0]) - E) <= 1e-5 * max(abs(E), rms)
                assert np.abs(j["grad"][0].cpu().numpy() - g).max() <= 1e-4 * np.abs(g).max()
                j["E"].zero_()
                j["grad"].zero_()
