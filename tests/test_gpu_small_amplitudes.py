"""Amplitudes whose tensors lie far below the bounds of their entries, on each
executor: layers of small rotations (amplitudes down to 2^-150, where most
entries of a gate's table are tiny) and fixed-gate circuits deep enough that
several tensors shrunk by cancellation meet in one step."""
import numpy as np
import pytest

import errmeasure
import qgm_inputs as qi
from oracle import statevector as sv
from oracle import vec

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EXECS = [1, 2, 3]  # stepwise, resident, compiled resident


@pytest.fixture(scope="module")
def q():
    from paper_1712_05384_gb300 import build
    build.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1712_05384_gb300 as q
    return q


def _near_identity(rows, cols, layers, theta, seed):
    """Layers of RXY by about theta on every qubit, a CZ layer between two.
    The phases stay within 0.4 rad, so that no sum of a few paths cancels."""
    n, rng, gates = rows * cols, np.random.default_rng(seed), []
    pats = qi.cz_patterns(rows, cols)
    for t in range(layers):
        for j in range(n):
            gates.append(qi.Gate(qi.GATE_RXY, t, j, -1, theta * (0.75 + 0.5 * rng.random()), 0.4 * rng.random()))
        if t + 1 < layers:
            gates += [qi.Gate(qi.GATE_CZ, t, a, b) for a, b in pats[(2 * t) % 8] + pats[(2 * t + 1) % 8]]
    return qi.circuit_from_gates(n, gates)


@pytest.mark.parametrize("executor", EXECS)
@pytest.mark.parametrize("rows,cols,layers,theta", [(4, 4, 3, 0.1), (4, 4, 3, 0.02), (4, 4, 4, 0.002), (4, 5, 4, 0.1),
                                                    (4, 5, 4, 0.05), (5, 5, 4, 0.1), (4, 4, 6, 1e-5), (4, 5, 4, 1e-5),
                                                    (3, 4, 10, 1e-3)])
def test_small_rotations(q, rows, cols, layers, theta, executor):
    c = _near_identity(rows, cols, layers, theta, 1)
    rng = np.random.default_rng(2)
    p = q.Plan(q.Model(q.Circuit.from_gates(c.n, c.gates)), batch=4, executor=executor).bind()
    # all ones, zero, and strings of mixed weight; a batch (padded to four
    # entries) shares its tensors' scales, so each holds one string only
    for x in [(1 << c.n) - 1, 0] + [int(x) for x in rng.integers(0, 1 << c.n, 4)]:
        ref = vec.amplitude(c, x)
        a = p.amplitudes_host(np.full(4, x, dtype=np.uint64))
        assert p.status() == 0
        # FP32 products and short sums: the paper's 1e-5, on its own scale
        assert np.max(np.abs(a - ref)) < 1e-5 * abs(ref), (a, ref)


def test_tiny_rotations_stepwise(q):
    # inputs near 2^-50 each and table entries of 2^-18: in range one by one
    # with every input scaled first, not as raw products (2^-340 in all)
    c = _near_identity(4, 5, 5, 6.3e-6, 3)
    x = (1 << c.n) - 1
    p = q.Plan(q.Model(q.Circuit.from_gates(c.n, c.gates)), batch=4, executor=q.EXEC_STEPWISE).bind()
    ref = vec.amplitude(c, x)
    a = p.amplitudes_host(np.full(4, x, dtype=np.uint64))
    assert p.status() == 0
    assert np.max(np.abs(a - ref)) < 1e-5 * abs(ref), (a, ref)


@pytest.mark.parametrize("executor", EXECS)
@pytest.mark.parametrize("rows,cols,depth,seed", [(4, 4, 28, 1), (4, 4, 28, 4), (4, 5, 23, 0), (4, 4, 36, 2), (3, 4, 40, 0)])
def test_deep_circuits_of_fixed_gates(q, rows, cols, depth, seed, executor):
    c = qi.grid_circuit(rows, cols, depth, seed)
    bits = qi.bitstrings(c.n, 24, seed)
    m = q.Model(q.Circuit.grid(rows, cols, depth, seed))
    if executor != 1 and not _resident(q, m):
        pytest.skip("no resident layout")
    p = q.Plan(m, batch=len(bits), executor=executor).bind()
    a = p.amplitudes_host(bits)
    assert p.status() == 0
    e = errmeasure.measures(a, sv.amplitudes(c, bits), c.n)
    assert e["rel"] < 1e-5 and e["abs"] < 1e-5, e


def _resident(q, m):
    try:
        q.Plan(m, batch=24, executor=q.EXEC_RESIDENT)
        return True
    except Exception:
        return False
