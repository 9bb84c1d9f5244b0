"""Performance cases of the amplitude engine: what its users run.

Each case is one call (or training step) through the package's public entry
points, on the circuits of the repository's workloads and tests and on grids
between them.  ``listed`` names them, ``draw`` gives further cases of the same
ranges, ``prepare`` builds what a program holds before the call (plan, bound
workspace, device buffers), ``run`` is the call, ``work`` what it cannot do
without, and ``exact`` the same outputs in 64 bits.

Amplitudes and gradients are computed in FP32 (split FP16 or BF16 products
accumulated in FP32); the entry points hand them over in FP64 containers, and
``run`` keeps them as a program that stores them does, in single precision.
"""
import cmath
import itertools
import math

import numpy as np
import torch

import paper_1712_05384_gb300 as q
from paper_1712_05384_gb300 import _lib
from paper_1712_05384_gb300 import autograd as qgrad

# kind -> the call a case stands for:
#   batch    Plan.amplitudes, device bitstrings and result
#   host     Plan.amplitudes_host, host buffers in and out
#   all      Plan.eliminate, every output open (2^n amplitudes)
#   grad     one training step: autograd.amplitudes, a loss, its gradient
#   set      cross-entropy statistics of a computed set and samples from it


def _case(name, kind, rows, cols, depth, batch, **more):
    return dict(name=name, kind=kind, rows=rows, cols=cols, depth=depth, batch=batch, circuit_seed=0,
                **{"open": 0, "precision": "fp16", "autotune": False, "budget": 0, "samples": 0, **more})


def listed():
    return [
        # one amplitude of a small circuit: latency of the shortest pass
        _case("one_4x4_d12", "batch", 4, 4, 12, 1),
        # a ragged batch handed over in host memory, as a service does
        _case("host_5x5_d20_b130", "host", 5, 5, 20, 130),
        # the 5x5 depth-20 workload: a batch in one resident launch
        _case("batch_5x5_d20_b1024", "batch", 5, 5, 20, 1024),
        # the 4x4 depth-10 workload: all 2^16 amplitudes at once
        _case("all_4x4_d10", "all", 4, 4, 10, 1),
        # six outputs left open per bitstring, odd batch
        _case("open6_5x5_d20_b37", "batch", 5, 5, 20, 37, open=6),
        # the 6x6 depth-25 workload: wide batch, product-sum and GEMM steps
        _case("batch_6x6_d25_b1000", "batch", 6, 6, 25, 1000),
        # a plan cut into slices by its memory budget
        _case("sliced_5x6_d30_b16", "batch", 5, 6, 30, 16, budget=1 << 27),
        # the parametrised 6x6 depth-20 workload: forward, loss, adjoint pass
        _case("grad_6x6_d20_b256", "grad", 6, 6, 20, 256),
        # the benchmark's pass: 5x9 depth 40, four bitstrings, tuned at bind
        _case("deep_5x9_d40_b4", "batch", 5, 9, 40, 4, autotune=True),
        # the second split precision on GEMM-shaped steps
        _case("bf16_4x6_d34_b64", "batch", 4, 6, 34, 64, precision="bf16"),
        # plain complex64: GEMM-shaped steps on the FP32 cores
        _case("fp32_4x8_d40_b4", "batch", 4, 8, 40, 4, precision="fp32"),
        # cross-entropy statistics of all 2^16 amplitudes, samples drawn from them
        _case("set_65536", "set", 4, 4, 10, 65536, samples=10000),
    ]


# per kind: grids with the depths that keep a pass below the largest listed
# one, and the largest batch
_SHALLOW = [(3, 3, 8, 30), (3, 4, 8, 30), (4, 4, 8, 30), (4, 5, 8, 27), (5, 5, 8, 24), (5, 6, 8, 24), (6, 6, 10, 24)]
_DEEP = [(4, 5, 28, 36), (5, 5, 24, 30), (4, 6, 28, 35), (5, 6, 24, 30), (6, 6, 23, 26), (4, 7, 30, 36)]
_OPEN = [(3, 3, 6, 16), (3, 4, 6, 14), (4, 4, 6, 12), (4, 5, 6, 10)]
_GRAD = [(3, 3, 8, 24), (3, 4, 8, 24), (4, 4, 8, 22), (5, 5, 10, 20), (5, 6, 10, 20), (6, 6, 10, 20)]


def _log_int(rng, lo, hi):
    return min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))


def draw(rng):
    kind = rng.choice(["batch", "batch", "batch", "deep", "deep", "host", "all", "open", "sliced", "grad", "grad", "set"])
    more = {}
    table = {"all": _OPEN, "grad": _GRAD, "deep": _DEEP, "sliced": _DEEP}.get(kind, _SHALLOW)
    rows, cols, lo, hi = rng.choice(table)
    depth = rng.randint(lo, hi)
    seed = rng.randint(0, 1 << 20)
    if kind == "deep":
        batch = _log_int(rng, 2, 48)
        more["precision"] = rng.choice(["fp16", "fp16", "bf16", "fp32"])
    elif kind == "sliced":
        batch = _log_int(rng, 2, 16)
        more["budget"] = 1 << rng.randint(27, 28)
    elif kind == "open":
        batch = _log_int(rng, 1, 64)
        more["open"] = rng.randint(1, 6)
    elif kind == "grad":
        batch = _log_int(rng, 2, 256)
    elif kind == "set":
        batch = _log_int(rng, 100, 1 << 18)
        more["samples"] = _log_int(rng, 100, 100000)
    elif kind == "all":
        batch = 1
    else:
        batch = _log_int(rng, 1, 1024)
    c = _case("", kind if kind in ("host", "all", "grad", "set") else "batch", rows, cols, depth, batch, **more)
    c["circuit_seed"] = seed
    del c["name"]
    return c


def _n(case):
    return case["rows"] * case["cols"]


def _bits(case, seed):
    x = np.random.default_rng(seed).integers(0, 1 << _n(case), size=case["batch"], dtype=np.uint64)
    return x.astype(np.int64)


def _angles(case, seed, gates):
    """(theta, phi) of every parametrised gate, flat, single precision."""
    u = np.random.default_rng((seed, 1)).random((sum(g[0] == "R" for g in gates), 2))
    return torch.from_numpy((u * [math.pi, 2 * math.pi]).reshape(-1)).to(torch.float32)


def _set(case, seed):
    """Amplitudes of a Porter-Thomas distributed set, interleaved doubles."""
    z = np.random.default_rng(seed).standard_normal(2 * case["batch"])
    return torch.from_numpy(z * 2.0 ** (-_n(case) / 2) / math.sqrt(2.0))


def _circuit_seed(case, seed):
    """All outputs of a circuit: the circuit is the input."""
    return case["circuit_seed"] + (seed if case["kind"] == "all" else 0)


def _plan(case, seed=0):
    circuit = q.Circuit.grid(case["rows"], case["cols"], case["depth"], _circuit_seed(case, seed), case["kind"] == "grad")
    return q.Plan(q.Model(circuit), batch=case["batch"], output_mode=q.OUT_OPEN if case["kind"] == "all" else q.OUT_BATCH,
                  mem_budget_bytes=case["budget"], open_mask=(1 << case["open"]) - 1, precision=case["precision"],
                  autotune=case["autotune"], gradients=case["kind"] == "grad")


def prepare(case, seed):
    kind = case["kind"]
    state = {"kind": kind}
    if kind == "set":
        state.update(amps=_set(case, seed).cuda(), t=case["batch"], n=_n(case), m=case["samples"], seed=seed,
                     sums=torch.empty(4, dtype=torch.float64, device="cuda"),
                     cdf=torch.empty(case["batch"], dtype=torch.float64, device="cuda"),
                     idx=torch.empty(case["samples"], dtype=torch.int64, device="cuda"))
        return state
    plan = _plan(case, seed).bind()
    state["plan"] = plan
    if kind == "all":
        state["out"] = torch.empty(2 << _n(case), dtype=torch.float64, device="cuda")
        return state
    bits = _bits(case, seed)
    if kind == "host":
        state["bits"] = bits.astype(np.uint64)
        return state
    state["bits"] = torch.from_numpy(bits).cuda()
    if kind == "grad":
        gates = _gates(case)
        state["params"] = _angles(case, seed, gates).cuda().requires_grad_()
        state["norm"] = 2.0 ** _n(case) / case["batch"]
        return state
    state["out"] = torch.empty(2 * (case["batch"] << case["open"]), dtype=torch.float64, device="cuda")
    return state


def run(state):
    kind = state["kind"]
    if kind == "set":
        stats = _lib.xeb_stats(state["amps"], state["t"], state["n"], state["sums"])
        _lib.sample_from_set(state["amps"], state["t"], state["m"], state["seed"], state["cdf"], state["idx"])
        return {"stats": stats, "samples": state["idx"]}
    plan = state["plan"]
    if kind == "host":
        return plan.amplitudes_host(state["bits"]).astype(np.complex64)
    if kind == "all":
        return plan.eliminate(state["out"]).to(torch.float32)
    if kind == "grad":
        # linear cross entropy of the batch: its gradient is as well
        # conditioned as the amplitudes (log p amplifies rounding near zeros)
        a = qgrad.amplitudes(plan, state["params"], state["bits"])
        loss = -state["norm"] * a.abs().square().sum()
        grad, = torch.autograd.grad(loss, state["params"])
        return {"amplitudes": a.detach().to(torch.complex64), "grad": grad}
    return plan.amplitudes(state["bits"], state["out"], B=state["bits"].numel()).to(torch.float32)


def work(case):
    """Inputs read and outputs written once; the products and sums of the
    (unsliced) elimination, twice more for an adjoint pass."""
    if case["kind"] == "set":
        return {"bytes": 16 * case["batch"] + 8 * case["samples"], "flops": 8 * case["batch"]}
    flops = _plan({**case, "budget": 0, "kind": "all" if case["kind"] == "all" else "batch"}).info.flops_per_slice
    if case["kind"] == "all":
        return {"bytes": 16 << _n(case), "flops": flops}
    nbytes = 8 * case["batch"] + 16 * (case["batch"] << case["open"])
    if case["kind"] == "grad":
        n_par = 2 * sum(g[0] == "R" for g in _gates(case))
        return {"bytes": nbytes + 8 * n_par, "flops": 3 * flops}
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------ 64-bit values
def _gates(case, seed=0):
    """The seeded grid circuit as (kind, qubits): H layer, then per cycle the
    CZ pattern and, on qubits that had a CZ and have none, T once and then
    X^1/2 or Y^1/2 by the top bit of a SplitMix64 draw (R: parametrised)."""
    rows, cols = case["rows"], case["cols"]
    mask, state = (1 << 64) - 1, _circuit_seed(case, seed)

    def hz(o):
        return [(r * cols + c, r * cols + c + 1) for r in range(rows) for c in range(cols - 1) if c % 4 == (o + 2 * (r % 2)) % 4]

    def vt(o):
        return [(r * cols + c, r * cols + c + cols) for r in range(rows - 1) for c in range(cols) if r % 4 == (o + 2 * (c % 2)) % 4]

    layers = [hz(0), hz(2), vt(0), vt(2), hz(1), hz(3), vt(1), vt(3)]
    gates = [("H", (j,)) for j in range(rows * cols)]
    before, had_t = set(), set()
    for t in range(1, case["depth"]):
        pairs = layers[(t - 1) % 8]
        gates += [("CZ", p) for p in pairs]
        now = set(itertools.chain(*pairs))
        for j in sorted(before - now):
            if j not in had_t:
                had_t.add(j)
                gates.append(("T", (j,)))
            elif case["kind"] == "grad":
                gates.append(("R", (j,)))
            else:
                state = (state + 0x9E3779B97F4A7C15) & mask
                z = ((state ^ (state >> 30)) * 0xBF58476D1CE4E5B9) & mask
                z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
                gates.append(("Y" if ((z ^ (z >> 31)) >> 63) else "X", (j,)))
        before = now
    return gates


def _network(case, bits, angles, seed):
    """The circuit for a batch of bitstrings as factors (variables, tensor
    with the batch first, size 1 where it does not depend on it) and the
    variables of its open outputs, lowest qubit first."""
    dev = bits.device
    n, s = _n(case), math.sqrt(0.5)
    const = {"H": [[s, s], [s, -s]], "X": [[s, -1j * s], [-1j * s, s]], "Y": [[s, -s], [s, s]]}
    const = {k: torch.tensor(v, dtype=torch.complex128, device=dev) for k, v in const.items()}
    t_gate = torch.tensor([1, cmath.exp(0.25j * math.pi)], dtype=torch.complex128, device=dev)
    cz = torch.tensor([[1, 1], [1, -1]], dtype=torch.complex128, device=dev)
    cur, factors, ids, param = [None] * n, [], itertools.count(), 0
    for kind, qubits in _gates(case, seed):
        if kind == "T":
            if cur[qubits[0]] is not None:
                factors.append(((cur[qubits[0]],), t_gate))
        elif kind == "CZ":
            if all(cur[j] is not None for j in qubits):
                factors.append((tuple(cur[j] for j in qubits), cz))
        else:
            if kind == "R":
                th, ph = angles[2 * param] / 2, angles[2 * param + 1]
                param += 1
                c, sn = torch.cos(th) + 0j, -1j * torch.sin(th)
                u = torch.stack([torch.stack([c, sn * torch.exp(-1j * ph)]), torch.stack([sn * torch.exp(1j * ph), c])])
            else:
                u = const[kind]
            old, cur[qubits[0]] = cur[qubits[0]], next(ids)
            factors.append(((cur[qubits[0]],), u[:, 0]) if old is None else ((cur[qubits[0]], old), u))
    n_open = n if case["kind"] == "all" else case["open"]
    fixed = {cur[j]: (bits >> j) & 1 for j in range(n_open, n)}
    out = []
    for vs, t in factors:
        hit = [v in fixed for v in vs]
        if any(hit):
            t = t[tuple(fixed[v] if h else slice(None) for v, h in zip(vs, hit))]
            if hit == [False, True]:
                t = t.transpose(0, 1)
        else:
            t = t[None]
        out.append((tuple(v for v, h in zip(vs, hit) if not h), t))
    return out, [cur[j] for j in range(n_open)]


def _min_fill(scopes, keep):
    nb = {}
    for vs in scopes:
        for v in vs:
            nb.setdefault(v, set()).update(set(vs) - {v})
    order, width = [], 0
    todo = set(nb) - set(keep)
    while todo:
        def fill(v):
            ns = sorted(nb[v])
            return sum(b not in nb[a] for i, a in enumerate(ns) for b in ns[i + 1:]), len(ns), v
        v = min(todo, key=fill)
        ns = nb.pop(v)
        for a in ns:
            nb[a] |= ns - {a}
            nb[a].discard(v)
        order.append(v)
        todo.discard(v)
        width = max(width, len(ns) + 1)
    return order, max(width, len(keep))


def _times(a, b, drop=None):
    """Product of two factors, summed over `drop`."""
    vs = sorted(set(a[0]) | set(b[0]))
    at = {v: i + 1 for i, v in enumerate(vs)}
    left = tuple(v for v in vs if v != drop)
    batch = max(a[1].shape[0], b[1].shape[0])
    ts = [t.expand(batch, *t.shape[1:]) for _, t in (a, b)]
    return left, torch.einsum(ts[0], [0] + [at[v] for v in a[0]], ts[1], [0] + [at[v] for v in b[0]], [0] + [at[v] for v in left])


def _amplitudes64(case, bits, angles=None, seed=0):
    """Amplitudes (batch, 2^open) in complex128 by eliminating variable after
    variable; None where the tensors are too large for it."""
    factors, keep = _network(case, bits[:1], angles, seed)
    order, width = _min_fill([vs for vs, _ in factors], keep)
    if width > 27 or bits.numel() * 2.0 ** width > 2.0 ** 34:
        return None
    chunk = bits.numel() if angles is not None else max(1, min(bits.numel(), 1 << max(0, 27 - width)))
    parts = []
    for at in range(0, bits.numel(), chunk):
        factors, keep = _network(case, bits[at:at + chunk], angles, seed)
        for v in order:
            mine = sorted((f for f in factors if v in f[0]), key=lambda f: f[1].numel())
            factors = [f for f in factors if v not in f[0]]
            acc = mine[0] if len(mine) > 1 else ((), torch.ones(1, dtype=torch.complex128, device=bits.device))
            for f in mine[1:-1]:
                acc = _times(acc, f)
            factors.append(_times(acc, mine[-1], drop=v))
        acc = ((), torch.ones(1, dtype=torch.complex128, device=bits.device))
        for f in sorted(factors, key=lambda f: f[1].numel()):
            acc = _times(acc, f)
        t = acc[1].expand(min(chunk, bits.numel() - at), *acc[1].shape[1:])
        # result index bit i = i-th lowest open qubit: highest qubit first
        t = t.permute([0] + [1 + acc[0].index(v) for v in reversed(keep)])
        parts.append(t.reshape(t.shape[0], -1))
    return torch.cat(parts)


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if case["kind"] == "set":
        p = _set(case, seed).numpy().reshape(-1, 2)
        p = (p * p).sum(1)
        log_n, gamma = _n(case) * math.log(2.0), 0.5772156649015329
        s = -float(np.log(p).mean())
        stats = {"cross_entropy": s, "alpha": log_n + gamma - s, "mean_Np": float(p.mean() * 2.0 ** _n(case)),
                 "second_moment": float(((p * 2.0 ** _n(case)) ** 2).mean())}
        return {"stats": stats, "samples": None}
    bits = torch.from_numpy(_bits(case, seed) if case["kind"] != "all" else np.zeros(1, np.int64)).to(dev)
    if case["kind"] == "grad":
        params = _angles(case, seed, _gates(case)).to(dev).double().requires_grad_()
        a = _amplitudes64(case, bits, params)
        if a is None:
            return None
        a = a[:, 0]
        loss = -2.0 ** _n(case) / case["batch"] * (a.real.square() + a.imag.square()).sum()
        grad, = torch.autograd.grad(loss, params)
        return {"amplitudes": a.detach(), "grad": grad}
    a = _amplitudes64(case, bits, seed=seed)
    if a is None:
        return None
    if case["kind"] == "host":
        return a[:, 0].cpu().numpy()
    return torch.view_as_real(a.reshape(-1).contiguous()).reshape(-1)
