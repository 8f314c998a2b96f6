"""The work whose speed is measured: QAOA evaluations, gradients and pre-computations through the package's public calls.

Every case is one call that an angle-finding program makes over and over (or, for the pre-computations, once per instance). A state holds what such a
program has in hand before the call: a context (one per program, so one per state), the cost vector on the GPU, the mixer, the angles, and for batched
calls the prepared job list with its result buffers.

Angles are the iterates of an optimiser that starts from a smooth annealing-like schedule: a linear ramp, beta falling and gamma growing, with some
noise on every angle. The library's state vectors are complex64; the programs meant here keep their angles' optimiser in 32 bits too (the default type
of torch parameters), so <C> and the gradients, sums over complex64 states, are taken as float32. The reduced Grover path computes in float64 throughout
and its results stay float64; counts and costs come as the library writes them.
"""

import itertools
import math

import numpy as np
import torch

import paper_2312_06451_gb300 as qg


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # one <C> of the smallest everyday instance: what a gradient-free optimiser or a landscape scan calls; all latency
        {"name": "expect_maxcut12", "kind": "x", "call": "single", "grad": False, "problem": "maxcut", "n": 12, "p": 3, "sets": 1, "mixer": "x"},
        # a multistart's starting points on a toy instance, one batched gradient call: the whole state fits one SM
        {"name": "grad_maxcut10_b256", "kind": "x", "call": "batched", "grad": True, "problem": "maxcut", "n": 10, "p": 8, "sets": 256, "mixer": "x"},
        # BFGS on one weighted instance of the size that papers use: one gradient per call, host angles and results
        {"name": "grad_wmaxcut15", "kind": "x", "call": "single", "grad": True, "problem": "wmaxcut", "n": 15, "p": 6, "sets": 1, "mixer": "x"},
        # the same loop one step up, integer costs, from a warm start (a given initial state)
        {"name": "grad_maxcut19_warm", "kind": "x", "call": "single", "grad": True, "problem": "maxcut", "n": 19, "p": 5, "sets": 1, "mixer": "x", "warm": True},
        # angle finding over an ensemble: instances of uneven size, a few starting points each, in one call
        {"name": "grad_uneven_14_22", "kind": "uneven", "n_lo": 14, "n_hi": 22, "instances": 32, "sets": 2, "p": 6},
        # the largest single instance: SK couplings, float32 costs, forward and adjoint sweep
        {"name": "grad_sk28", "kind": "x", "call": "batched", "grad": True, "problem": "sk", "n": 28, "p": 8, "sets": 1, "mixer": "x"},
        # <C> alone of a few angle sets on a large 3-regular instance: forward sweeps, integer costs
        {"name": "expect_3reg24_b4", "kind": "x", "call": "batched", "grad": False, "problem": "3reg", "n": 24, "p": 10, "sets": 4, "mixer": "x"},
        # multi-angle QAOA: one angle per qubit and round
        {"name": "grad_ma_maxcut20", "kind": "x", "call": "batched", "grad": True, "problem": "maxcut", "n": 20, "p": 4, "sets": 2, "mixer": "ma"},
        # Grover mixer on a constrained (weight-k) feasible set of odd size, a few starting points
        {"name": "grad_grover_dks22_11", "kind": "grover", "n": 22, "k": 11, "p": 6, "sets": 4},
        # Grover-mixer QAOA on cost degeneracies: counting the weight-6 sets of 100 vertices, then 1024 reduced gradients
        {"name": "degeneracy_dks100_6", "kind": "degeneracy", "n": 100, "k": 6, "p": 10, "sets": 1024},
        # constrained ring mixer on the weight-k states through its stored eigendecomposition, a batch of starting points
        {"name": "grad_ring16_8_b256", "kind": "ring", "n": 16, "k": 8, "p": 6, "sets": 256},
        # the pre-computation of a cost vector, paid once per instance
        {"name": "cost_sk26", "kind": "cost", "problem": "sk", "n": 26},
    ]


def draw(rng):
    kind = rng.choice(["x_small", "x_mid", "x_large", "x_large", "ma", "terms", "uneven", "grover", "degeneracy", "ring", "cost"])

    def log_int(lo, hi):
        return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))))

    if kind == "x_small":
        n = rng.randint(6, 12)
        return {"kind": "x", "call": "batched", "grad": rng.random() < 0.7, "problem": rng.choice(["maxcut", "wmaxcut", "sk"]), "n": n, "p": rng.randint(1, 12),
                "sets": log_int(1, 1024), "mixer": "x"}
    if kind == "x_mid":
        n = rng.randint(12, 20)
        c = {"kind": "x", "call": "single", "grad": rng.random() < 0.8, "problem": rng.choice(["maxcut", "wmaxcut", "sk"]), "n": n, "p": rng.randint(2, 10),
             "sets": 1, "mixer": "x"}
        if rng.random() < 0.3:
            c["warm"] = True
        return c
    if kind == "x_large":
        n = rng.randint(20, 27)
        return {"kind": "x", "call": rng.choice(["single", "batched", "batched"]), "grad": rng.random() < 0.7, "problem": rng.choice(["maxcut", "sk"]), "n": n,
                "p": rng.randint(2, 8), "sets": 1, "mixer": "x"}
    if kind == "ma":
        return {"kind": "x", "call": "batched", "grad": True, "problem": rng.choice(["maxcut", "sk"]), "n": rng.randint(10, 22), "p": rng.randint(1, 5),
                "sets": rng.randint(1, 4), "mixer": "ma"}
    if kind == "terms":
        return {"kind": "x", "call": "batched", "grad": True, "problem": rng.choice(["maxcut", "sk"]), "n": rng.randint(11, 21), "p": rng.randint(1, 5),
                "sets": rng.randint(1, 4), "mixer": "terms"}
    if kind == "uneven":
        lo = rng.randint(12, 17)
        return {"kind": "uneven", "n_lo": lo, "n_hi": rng.randint(lo + 1, 21), "instances": rng.randint(4, 40), "sets": rng.randint(1, 4), "p": rng.randint(2, 7)}
    if kind == "grover":
        n = rng.randint(12, 25)
        return {"kind": "grover", "n": n, "k": rng.randint(3, n // 2), "p": rng.randint(1, 8), "sets": rng.randint(1, 6)}
    if kind == "degeneracy":
        return {"kind": "degeneracy", "n": rng.randint(40, 100), "k": rng.randint(4, 6), "p": rng.randint(1, 12), "sets": log_int(16, 1024)}
    if kind == "ring":
        n = rng.randint(10, 16)
        return {"kind": "ring", "n": n, "k": rng.randint(3, n // 2), "p": rng.randint(1, 6), "sets": log_int(8, 256)}
    return {"kind": "cost", "problem": rng.choice(["sk", "sk", "maxcut", "wmaxcut"]), "n": rng.randint(16, 26)}


# -------------------------------------------------------------- the instances
def _rng(seed, salt):
    return np.random.Generator(np.random.PCG64([int(seed), salt]))


def _er(r, n, prob=0.5):
    iu, ju = np.triu_indices(n, k=1)
    keep = r.random(iu.shape[0]) < prob
    keep[int(r.integers(0, iu.shape[0]))] = True  # at least one edge
    return np.stack([iu[keep], ju[keep]], axis=1).astype(np.int32)


def _reg3(r, n):
    """A simple 3-regular graph by the configuration model."""
    while True:
        q = r.permutation(np.repeat(np.arange(n), 3))
        a, b = np.minimum(q[0::2], q[1::2]), np.maximum(q[0::2], q[1::2])
        if (a != b).all() and np.unique(a * n + b).shape[0] == a.shape[0]:
            return np.stack([a, b], axis=1).astype(np.int32)


def _instance(problem, n, r):
    """What cost_precompute takes for one instance, its result type, and the scale of gamma for it (about 1 / std C)."""
    if problem == "sk":
        J = np.triu(np.rint(np.clip(r.standard_normal((n, n)), -7.9, 7.9) * 2.0**20) / 2.0**20, 1)
        return {"J": (J + J.T).astype(np.float32)}, torch.float32, 1.0 / math.sqrt(n * (n - 1) / 2)
    e = _reg3(r, n) if problem == "3reg" else _er(r, n)
    sd = 0.5 * math.sqrt(len(e))
    if problem == "wmaxcut":
        return {"edges": e, "weights": r.random(len(e)).astype(np.float32)}, torch.float32, 1.0 / (0.58 * sd)
    return {"edges": e}, torch.uint8, 1.0 / sd


def _problem_name(problem):
    return "maxcut" if problem == "3reg" else problem


def _angles(r, sets, p, scale, per=1):
    """sets x (p per + p): a noisy ramp; `per` betas in each round."""
    t = (np.arange(p) + 0.5) / p
    beta = 0.6 * (1.0 - t)[None, :, None] + 0.1 * r.uniform(-1, 1, (sets, p, per))
    gamma = scale * (0.3 + t)[None, :] * r.uniform(0.7, 1.3, (sets, p))
    return np.concatenate([beta.reshape(sets, p * per), -gamma], axis=1)


def _warm(r, dim):
    """A normalised complex64 initial state near the uniform one, on the GPU."""
    g = torch.Generator(device="cuda").manual_seed(int(r.integers(0, 2**31)))
    v = torch.complex(1.0 + 0.3 * torch.randn(dim, generator=g, device="cuda"), 0.3 * torch.randn(dim, generator=g, device="cuda"))
    return v / torch.linalg.vector_norm(v)


def _mixer_for(case):
    n = case["n"]
    if case["mixer"] == "ma":
        return qg.XMixer(n, multi_angle=True)
    if case["mixer"] == "terms":
        return qg.x_terms_mixer(n, {1: 1.0, 2: 1.0})
    return qg.XMixer(n)


_ring_mixers = {}  # a mixer's stored eigendecomposition: like the file a program keeps it in


def _ring_mixer(ctx, n, k):
    if (n, k) not in _ring_mixers:
        m = qg.xy_sym_mixer(ctx, "ring", n, k)
        _ring_mixers[n, k] = (m.V, m.lam, m.block_dims)
    return qg.EigenSymMixer(n, k, *_ring_mixers[n, k])


def _uneven(case, r):
    """(n, edges) of each instance: 3-regular graphs on even n and denser random ones on any n, in turn."""
    out = []
    for i in range(case["instances"]):
        n = int(r.integers(case["n_lo"], case["n_hi"] + 1))
        out.append((n, _reg3(r, n) if i % 2 == 0 and n % 2 == 0 else _er(r, n, 0.3)))
    return out


def _job(cost, mixer, angles, init=None):
    a = torch.from_numpy(angles).cuda()
    j = {"cost": cost, "mixer": mixer, "angles": a, "E": torch.empty(a.shape[0], dtype=torch.float64, device="cuda"), "grad": torch.empty_like(a)}
    return j if init is None else dict(j, init=init)


# ------------------------------------------------------------------- prepare
def prepare(case, seed):
    kind, ctx = case["kind"], qg.Context(0)
    s = {"kind": kind, "ctx": ctx}
    if kind == "x":
        n, p = case["n"], case["p"]
        r = _rng(seed, 1)
        inst, dtype, scale = _instance(case["problem"], n, r)
        cost = ctx.cost_precompute(_problem_name(case["problem"]), n, dtype=dtype, **inst)
        mixer = _mixer_for(case)
        angles = _angles(r, case["sets"], p, scale, n if case["mixer"] == "ma" else 1)
        init = _warm(r, 1 << n) if case.get("warm") else None
        s.update(grad=case["grad"], call=case["call"])
        if case["call"] == "single":
            s.update(cost=cost, mixer=mixer, angles=angles[0], init=init)
        else:
            s["jobs"] = [_job(cost, mixer, angles, init)]
    elif kind == "uneven":
        r = _rng(seed, 2)
        s.update(grad=True, call="batched", jobs=[])
        for n, e in _uneven(case, r):
            cost = ctx.cost_precompute("maxcut", n, edges=e, dtype=torch.uint8)
            s["jobs"].append(_job(cost, qg.XMixer(n), _angles(r, case["sets"], case["p"], 2.0 / math.sqrt(len(e)))))
    elif kind in ("grover", "ring"):
        n, k = case["n"], case["k"]
        r = _rng(seed, 3)
        e = _er(r, n)
        cost = ctx.cost_precompute("dks", n, edges=e, k=k, dtype=torch.uint8)
        mixer = qg.GroverMixer.dicke(n, k) if kind == "grover" else _ring_mixer(ctx, n, k)
        s.update(grad=True, call="batched", jobs=[_job(cost, mixer, _angles(r, case["sets"], case["p"], _dks_scale(n, k, len(e))))])
    elif kind == "degeneracy":
        r = _rng(seed, 4)
        e = _er(r, case["n"])
        s.update(n=case["n"], k=case["k"], edges=e,
                 angles=torch.from_numpy(_angles(r, case["sets"], case["p"], _dks_scale(case["n"], case["k"], len(e)))).cuda())
    else:
        inst, dtype, _ = _instance(case["problem"], case["n"], _rng(seed, 5))
        s.update(problem=_problem_name(case["problem"]), n=case["n"], inst=inst, dtype=dtype)
    if s.get("call") == "batched":
        s["prepared"] = ctx.batched_call(s["jobs"], want_grad=s["grad"])
    return s


def _dks_scale(n, k, m):
    """About 1 / std C of the densest-k-subgraph cost."""
    q = m / (n * (n - 1) / 2)
    return 1.0 / math.sqrt(max(0.25, k * (k - 1) / 2 * q * (1 - q) + 0.05))


# ----------------------------------------------------------------------- run
def run(s):
    ctx = s["ctx"]
    if s["kind"] == "degeneracy":
        counts = ctx.cost_degeneracy("dks", s["n"], edges=s["edges"], k=s["k"])
        E, g = ctx.grover_batched(counts, s["angles"])
        return {"counts": counts, "E": E, "grad": g}
    if s["kind"] == "cost":
        return {"cost": ctx.cost_precompute(s["problem"], s["n"], dtype=s["dtype"], **s["inst"])}
    if s["call"] == "single":
        if not s["grad"]:
            return {"E": np.float32(ctx.expectation(s["cost"], s["mixer"], s["angles"], s["init"]))}
        E, g = ctx.gradient(s["cost"], s["mixer"], s["angles"], s["init"])
        return {"E": np.float32(E), "grad": g.astype(np.float32)}
    s["prepared"].run()
    out = {"E": torch.cat([j["E"] for j in s["jobs"]]).float()}
    if s["grad"]:
        out["grad"] = torch.cat([j["grad"].reshape(-1) for j in s["jobs"]]).float()
    return out


# ---------------------------------------------------------------------- work
def _cost_bytes(problem):
    return 4 if problem in ("sk", "wmaxcut") else 1


def work(case):
    """Bytes: the cost vector and the angles in, <C>, the gradient, counts or costs out. Flops: per amplitude and round 6 for each qubit's rotation and 6 for the
    phase; a gradient sweeps three vectors so and takes 4 for each qubit's derivative term and the phase's."""
    kind = case["kind"]
    if kind == "x":
        n, p, S = case["n"], case["p"], case["sets"]
        na = p * (n + 1) if case["mixer"] == "ma" else 2 * p
        rot = (2 if case["mixer"] == "terms" else 1) * 6.0 * n + 6
        f = S * p * 2.0**n * ((3 * rot + 4 * (n + 1)) if case["grad"] else rot)
        return {"bytes": _cost_bytes(case["problem"]) * 2.0**n + 8.0 * S * (1 + na * (2 if case["grad"] else 1)), "flops": f}
    if kind == "uneven":
        N = [2.0**n for n in range(case["n_lo"], case["n_hi"] + 1)]
        mean = case["instances"] * sum(N) / len(N)
        n = case["n_hi"] - 1
        return {"bytes": mean + 8.0 * case["instances"] * case["sets"] * (1 + 4 * case["p"]), "flops": mean * case["sets"] * case["p"] * (3 * (6.0 * n + 6) + 4 * (n + 1))}
    if kind == "cost":
        n = case["n"]
        return {"bytes": _cost_bytes(case["problem"]) * 2.0**n, "flops": 2.0 * n * 2.0**n}
    D, p, S = float(math.comb(case["n"], case["k"])), case["p"], case["sets"]
    if kind == "grover":
        return {"bytes": D + 8.0 * S * (1 + 4 * p), "flops": S * p * D * 36.0}
    if kind == "degeneracy":
        return {"bytes": 8.0 * S * (1 + 4 * p), "flops": D}
    blocks = D * D / (case["n"] // 2 + 1)  # the mixer's eigenvectors, block by block
    return {"bytes": 4 * blocks + D + 8.0 * S * (1 + 4 * p), "flops": 6.0 * p * 2 * blocks * 2 * S}


# --------------------------------------------------------------------- exact
# The same sums in complex128 by plain torch: states are (sets, dim) arrays, the adjoint undoes each round on the state.
def _flip(v, q):
    """v[x xor 2^q]"""
    S, N = v.shape
    return v.view(S, N >> (q + 1), 2, 1 << q).flip(2).view(S, N)


class _XExact:
    def __init__(self, n, beta):  # beta: sets x p x (1 or n)
        self.n, self.beta, self.per = n, beta, beta.shape[2]

    def apply(self, v, k, sign):
        for q in range(self.n):
            b = self.beta[:, k, q if self.per > 1 else 0][:, None]
            f = _flip(v, q).mul_(-1j * sign * torch.sin(b))
            v = v.mul_(torch.cos(b).to(v.dtype)).add_(f)
            del f
        return v

    def terms(self, lam, psi, k):
        """2 Im <lam|H|psi>, one column for each beta of the round"""
        t = [_im(lam, _flip(psi, q)) for q in range(self.n)]
        return torch.stack(t, 1) if self.per > 1 else torch.stack(t, 1).sum(1, keepdim=True)


class _DiagExact:
    """A mixer W diag(d) W with W the Walsh-Hadamard transform."""

    def __init__(self, n, beta, d):
        self.n, self.beta, self.d = n, beta[:, :, 0], d

    def _wht(self, v):
        for q in range(self.n):
            w = v.view(v.shape[0], -1, 2, 1 << q)
            v = torch.stack([w[:, :, 0] + w[:, :, 1], w[:, :, 0] - w[:, :, 1]], 2).view(v.shape) * math.sqrt(0.5)
        return v

    def apply(self, v, k, sign):
        return self._wht(self._wht(v) * torch.exp(-1j * sign * self.beta[:, k, None] * self.d[None, :]))

    def terms(self, lam, psi, k):
        return _im(lam, self._wht(self._wht(psi) * self.d))[:, None]


class _GroverExact:
    def __init__(self, beta):
        self.beta = beta[:, :, 0]

    def apply(self, v, k, sign):
        return v + (torch.exp(-1j * sign * self.beta[:, k]) - 1)[:, None] * v.mean(1, keepdim=True)

    def terms(self, lam, psi, k):
        return _im(lam, psi.mean(1, keepdim=True).expand_as(psi))[:, None]


class _RingExact:
    """H = sum_i X_i X_i+1 + Y_i Y_i+1 on the weight-k states by swaps of neighbouring bits; e^{-i b H} by its power series in short steps."""

    def __init__(self, n, k, beta):
        self.beta = beta[:, :, 0]
        x = np.array(sorted(sum(1 << i for i in c) for c in itertools.combinations(range(n), k)), dtype=np.int64)
        self.idx, self.on = [], []
        for i in range(n):
            j = (i + 1) % n
            differ = ((x >> i) ^ (x >> j)) & 1
            self.idx.append(torch.from_numpy(np.searchsorted(x, np.where(differ, x ^ (1 << i) ^ (1 << j), x))).cuda())
            self.on.append(torch.from_numpy(2.0 * differ).cuda())

    def _h(self, v):
        w = torch.zeros_like(v)
        for i, on in zip(self.idx, self.on):
            w += v[:, i] * on
        return w

    def apply(self, v, k, sign):
        b = sign * self.beta[:, k, None]
        steps = max(1, int(math.ceil(float(b.abs().max()) * 8)))
        for _ in range(steps):
            term = v
            for m in range(1, 31):
                term = self._h(term) * (-1j * b / (steps * m))
                v = v + term
        return v

    def terms(self, lam, psi, k):
        return _im(lam, self._h(psi))[:, None]


def _im(a, b):
    """2 Im <a|b> of each set"""
    return torch.stack([2.0 * torch.dot(x.conj(), y).imag for x, y in zip(a, b.contiguous())])


def _sweep(C, mixer, gamma, grad, init=None):
    """(<C>, gradient) of each set: C float64 (dim), gamma sets x p."""
    S, p = gamma.shape
    N = C.shape[0]
    psi = torch.full((S, N), N**-0.5, dtype=torch.complex128, device="cuda") if init is None else init.to(torch.complex128).expand(S, N).clone()

    def phase(v, k, sign):
        for s in range(S):  # set by set: no more than one vector of phases at a time
            v[s] *= torch.polar(torch.ones_like(C), C * (-sign * float(gamma[s, k])))
        return v

    for k in range(p):
        psi = mixer.apply(phase(psi, k, 1.0), k, 1.0)
    E = torch.stack([torch.dot(C, v.real.square() + v.imag.square()) for v in psi])
    if not grad:
        return E, None
    lam = psi * C
    gb, gg = [None] * p, [None] * p
    for k in reversed(range(p)):
        gb[k] = mixer.terms(lam, psi, k)
        psi, lam = mixer.apply(psi, k, -1.0), mixer.apply(lam, k, -1.0)
        gg[k] = torch.stack([2.0 * torch.dot(x.conj() * C, y).imag for x, y in zip(lam, psi)])
        psi, lam = phase(psi, k, -1.0), phase(lam, k, -1.0)
    return E, torch.cat(gb + [torch.stack(gg, 1)], 1)


def _cut(mixer_of, C, a, p, per, grad, init=None):
    """_sweep over the angle sets, as many at a time as keep a vector of all of them under 8 GiB."""
    a = torch.from_numpy(a).cuda()
    step = max(1, (1 << 29) // C.shape[0])
    E, G = [], []
    for i in range(0, a.shape[0], step):
        b = a[i : i + step]
        e, g = _sweep(C, mixer_of(b[:, : p * per].reshape(-1, p, per)), b[:, p * per :], grad, init)
        E.append(e)
        G.append(g)
    return torch.cat(E), torch.cat(G) if grad else None


def _cost_exact(problem, n, inst):
    """The cost vector in float64"""
    x = torch.arange(1 << n, device="cuda")
    C = torch.zeros(1 << n, dtype=torch.float64, device="cuda")
    z = [(1 - 2 * ((x >> i) & 1)).to(torch.float64) for i in range(n)] if n <= 24 else None

    def spin(i):
        return z[i] if z is not None else (1 - 2 * ((x >> i) & 1)).to(torch.float64)

    if problem == "sk":
        W = torch.from_numpy(np.triu(inst["J"].astype(np.float64), 1))
    else:
        W = torch.zeros(n, n, dtype=torch.float64)
        for (u, v), w in zip(inst["edges"].tolist(), inst.get("weights", np.ones(len(inst["edges"]))).astype(np.float64).tolist()):
            W[u, v] += w
    for i in range(n):
        row = torch.zeros_like(C)
        for j in range(i + 1, n):
            if W[i, j] != 0:
                row.add_(spin(j), alpha=float(W[i, j]))
        C += spin(i) * row
    return C if problem == "sk" else 0.5 * (float(W.sum()) - C)


def _dks_exact(n, k, edges):
    x = np.array(sorted(sum(1 << i for i in c) for c in itertools.combinations(range(n), k)), dtype=np.int64) if math.comb(n, k) < 1 << 18 else _weight_k(n, k)
    x = torch.from_numpy(x).cuda()
    C = torch.zeros(x.shape[0], dtype=torch.float64, device="cuda")
    for u, v in edges.tolist():
        C += ((x >> u) & (x >> v) & 1).to(torch.float64)
    return C


def _weight_k(n, k):
    """The weight-k numbers below 2^n, ascending"""
    x = np.arange(1 << n, dtype=np.int64)
    w = np.zeros(1 << n, dtype=np.int8)
    for i in range(n):
        w += ((x >> i) & 1).astype(np.int8)
    return x[w == k]


def _counts_exact(n, k, edges):
    """How many k-sets have each number of inner edges: a set is its lower part, whose largest vertex is m, and its upper part, all above m."""
    A = torch.zeros(n, n, dtype=torch.float32, device="cuda")
    e = torch.from_numpy(edges).cuda().long()
    A[e[:, 0], e[:, 1]] = 1
    A[e[:, 1], e[:, 0]] = 1
    low, top = (k + 1) // 2, min(len(edges), k * (k - 1) // 2) + 1
    counts = torch.zeros(top, dtype=torch.int64, device="cuda")

    def indicator(lo, hi, size):
        sets = torch.combinations(torch.arange(lo, hi, device="cuda"), size) if size else torch.zeros(1, 0, dtype=torch.long, device="cuda")
        return torch.zeros(sets.shape[0], n, device="cuda").scatter_(1, sets, 1.0)

    for m in range(low - 1, n - (k - low)):
        P = indicator(0, m, low - 1)
        P[:, m] = 1
        Q = indicator(m + 1, n, k - low)
        inner_p, inner_q = ((P @ A) * P).sum(1) / 2, ((Q @ A) * Q).sum(1) / 2
        for i in range(0, P.shape[0], 2048):
            c = (P[i : i + 2048] @ A) @ Q.T + inner_p[i : i + 2048, None] + inner_q[None, :]
            counts += torch.bincount(c.reshape(-1).round().to(torch.int32), minlength=top)
    return counts


class _ReducedExact:
    """The Grover mixer on amplitudes sqrt(d_c) a_c, one for each cost value c"""

    def __init__(self, u, beta):
        self.u, self.beta = u, beta[:, :, 0]

    def apply(self, v, k, sign):
        return v + ((torch.exp(-1j * sign * self.beta[:, k]) - 1) * (v @ self.u))[:, None] * self.u

    def terms(self, lam, psi, k):
        return _im(lam, (psi @ self.u)[:, None] * self.u)[:, None]


def exact(case, seed):
    kind = case["kind"]
    if kind == "cost":
        inst, _, _ = _instance(case["problem"], case["n"], _rng(seed, 5))
        return {"cost": _cost_exact(case["problem"], case["n"], inst)}
    if kind == "x":
        n, p = case["n"], case["p"]
        r = _rng(seed, 1)
        inst, _, scale = _instance(case["problem"], n, r)
        per = n if case["mixer"] == "ma" else 1
        a = _angles(r, case["sets"], p, scale, per)
        init = _warm(r, 1 << n) if case.get("warm") else None
        C = _cost_exact(case["problem"], n, inst)
        if case["mixer"] == "terms":
            w = torch.zeros(1 << n, dtype=torch.float64, device="cuda")
            for i in range(n):
                w += ((torch.arange(1 << n, device="cuda") >> i) & 1).to(torch.float64)
            d = (n - 2 * w) + ((n - 2 * w).square() - n) / 2  # sum X_i + sum_{i<j} X_i X_j where w spins are down
            E, g = _cut(lambda b: _DiagExact(n, b, d), C, a, p, per, case["grad"], init)
        else:
            E, g = _cut(lambda b: _XExact(n, b), C, a, p, per, case["grad"], init)
        if case["call"] == "single":
            return {"E": float(E[0]), "grad": g[0]} if case["grad"] else {"E": float(E[0])}
        return {"E": E, "grad": g.reshape(-1)} if case["grad"] else {"E": E}
    if kind == "uneven":
        r = _rng(seed, 2)
        E, G = [], []
        for n, e in _uneven(case, r):
            a = _angles(r, case["sets"], case["p"], 2.0 / math.sqrt(len(e)))
            x, g = _cut(lambda b, n=n: _XExact(n, b), _cost_exact("maxcut", n, {"edges": e}), a, case["p"], 1, True)
            E.append(x)
            G.append(g.reshape(-1))
        return {"E": torch.cat(E), "grad": torch.cat(G)}
    n, k, p = case["n"], case["k"], case["p"]
    r = _rng(seed, 4 if kind == "degeneracy" else 3)
    e = _er(r, n)
    a = _angles(r, case["sets"], p, _dks_scale(n, k, len(e)))
    if kind == "degeneracy":
        counts = _counts_exact(n, k, e)
        d = counts.to(torch.float64)
        u = torch.sqrt(d / d.sum()).to(torch.complex128)
        E, g = _cut(lambda b: _ReducedExact(u, b), torch.arange(d.shape[0], dtype=torch.float64, device="cuda"), a, p, 1, True, u)
        return {"counts": counts, "E": E, "grad": g}
    C = _dks_exact(n, k, e)
    E, g = _cut((lambda b: _GroverExact(b)) if kind == "grover" else (lambda b: _RingExact(n, k, b)), C, a, p, 1, True)
    return {"E": E, "grad": g.reshape(-1)}
