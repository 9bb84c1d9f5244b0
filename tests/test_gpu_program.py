"""Stepwise passes run as step programs (small steps in shared launches, taken
as units by CTAs that wait for one another's tensors) against the FP64 oracle,
at the sizes where the cutting into units changes: one bitstring, batches that
fill no pair or no pass of 256 lanes, long sums over few outputs (more than 8
summed variables, split sums), several segments around large steps, slices,
open outputs, and the adjoint pass."""
import numpy as np
import pytest

import errmeasure
import qgm_inputs as qi
from oracle import statevector as sv

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-5  # the parity tests' bound for complex64


@pytest.fixture(scope="module")
def q():
    from paper_1712_05384_gb300 import build
    build.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1712_05384_gb300 as q
    return q


@pytest.mark.parametrize("rows,cols,depth,B,kw", [
    (2, 2, 6, 1, {}), (3, 3, 8, 1, {}), (3, 3, 16, 2, {}), (3, 4, 14, 5, {"max_fuse": 16}), (3, 4, 24, 3, {"max_fuse": 16}),
    (4, 4, 16, 37, {}), (4, 4, 24, 130, {"max_fuse": 12}), (4, 5, 20, 127, {"max_fuse": 1}), (3, 4, 30, 1000, {}),
    (4, 5, 24, 1024, {}), (4, 5, 24, 16, {"div": 6}), (4, 5, 28, 9, {"div": 3, "precision": "fp32"})])
def test_program_matches_state_vector(q, rows, cols, depth, B, kw):
    kw = dict(kw)
    c = qi.grid_circuit(rows, cols, depth, 2)
    m = q.Model(q.Circuit.grid(rows, cols, depth, 2))
    div = kw.pop("div", 0)
    if div:
        kw["mem_budget_bytes"] = q.Plan(m, batch=B, executor=q.EXEC_STEPWISE, **kw).info.arena_bytes // div
    p = q.Plan(m, batch=B, executor=q.EXEC_STEPWISE, **kw).bind()
    assert not div or p.info.n_slices > 1
    bits = qi.bitstrings(c.n, B, 5)
    ref = sv.amplitudes(c, bits)
    for _ in range(2):  # a second pass starts from the first one's workspace
        a = p.amplitudes_host(bits)
        assert p.status() == 0
        e = errmeasure.measures(a, ref, c.n)
        assert e["rel"] < TOL and e["abs"] < TOL, e


@pytest.mark.parametrize("B,k", [(1, 1), (5, 4), (37, 7)])
def test_program_with_open_outputs(q, B, k):
    c = qi.grid_circuit(3, 4, 16, 4)
    p = q.Plan(q.Model(q.Circuit.grid(3, 4, 16, 4)), batch=B, open_mask=(1 << k) - 1).bind()
    bits = qi.bitstrings(12, B, 1)
    a = p.amplitudes_host(bits)
    full = (bits & ~np.uint64((1 << k) - 1))[:, None] + np.arange(1 << k, dtype=np.uint64)[None, :]
    ref = sv.amplitudes(c, full.reshape(-1)).reshape(B, 1 << k)
    assert p.status() == 0 and np.max(np.abs(a - ref)) * 2.0 ** 6 < TOL


@pytest.mark.parametrize("rows,cols,depth,B", [(3, 3, 10, 1), (3, 4, 20, 6), (4, 4, 20, 3)])
def test_program_gradients(q, rows, cols, depth, B):
    # the deeper plans sum more than 8 variables into a gate's adjoint
    c = qi.grid_circuit(rows, cols, depth, 1, param=True)
    p = q.Plan(q.Model(q.Circuit.grid(rows, cols, depth, 1, True)), batch=B, gradients=True, executor=q.EXEC_STEPWISE).bind()
    bits = qi.bitstrings(c.n, B, 3)
    amps = sv.amplitudes(c, bits)
    n = 2 * len(c.param_gates)
    g_out = torch.zeros(n, dtype=torch.float64, device="cuda")
    # L = sum |a|^2 2^n: g_b = a_b 2^n (Wirtinger derivative to conj(a_b))
    w = amps * 2.0 ** c.n
    d_g = torch.from_numpy(np.ascontiguousarray(w).view(np.float64)).cuda()
    p.amplitude_grad(torch.from_numpy(bits.astype(np.int64)).cuda(), d_g, g_out)
    assert p.status() == 0
    got = g_out.cpu().numpy()
    eps, theta = 1e-5, np.array([[c.gates[g].theta, c.gates[g].phi] for g in c.param_gates])

    def loss(t):
        return 2.0 ** c.n * np.sum(np.abs(sv.amplitudes(c.with_angles(t[:, 0], t[:, 1]), bits)) ** 2)

    for i in np.unique(np.linspace(0, n - 1, 9).astype(int)):
        t = theta.copy().reshape(-1)
        t[i] += eps
        up = loss(t.reshape(-1, 2))
        t[i] -= 2 * eps
        fd = (up - loss(t.reshape(-1, 2))) / (2 * eps)
        assert abs(got[i] - fd) <= 1e-3 * max(abs(fd), 1e-2 * np.max(np.abs(got))), i


@pytest.mark.parametrize("rows,cols,depth,B,kw", [
    (4, 4, 32, 1000, {}), (4, 4, 32, 37, {"max_fuse": 16, "gemm": False}), (4, 6, 30, 4, {"order_kind": 1}),
    (4, 5, 31, 12, {"order_kind": 1, "max_fuse": 16, "gemm": False}), (5, 5, 28, 20, {"gemm": False}),
    (5, 6, 28, 16, {"gemm": False}), (6, 6, 25, 37, {}), (4, 6, 34, 6, {"order_kind": 1}), (5, 5, 20, 64, {"open_mask": 7}),
    (4, 5, 36, 33, {"precision": "fp32"})])
def test_register_tiled_steps_match_the_general_kernel(q, rows, cols, depth, B, kw):
    # a pass step by step runs every step with the kernel of its own launch,
    # small ones too: each form of tile (rows, columns, batch entries per CTA,
    # further inputs) against the same steps on the general product-sum kernel
    p = q.Plan(q.Model(q.Circuit.grid(rows, cols, depth, 1)), batch=B, executor=q.EXEC_STEPWISE, **kw).bind()
    bits = torch.from_numpy(qi.bitstrings(rows * cols, B, 2).astype(np.int64)).cuda()
    n = 2 * (B << p.n_open)
    a, b = (torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(2))
    p.profile(bits, a)
    assert p.status() == 0
    outer = {g["step"]: g["o_bout"] or g["in_bout"] for g in p.gemm_shapes()}
    p.set_tuning([{"step": s, "T": 1, "U": 2, "ps": int(s in outer and not outer[s])} for s in range(p.info.n_steps)])
    p.profile(bits, b)
    assert p.status() == 0
    # two FP32 evaluations of the same sums, each within 1e-5 of the largest
    assert torch.max(torch.abs(a - b)).item() <= 2e-5 * torch.max(torch.abs(b)).item()


@pytest.mark.parametrize("rows,cols,depth,div", [(3, 3, 8, 0), (4, 6, 30, 0), (3, 4, 20, 4)])
def test_outputs_are_written_whole(q, rows, cols, depth, div):
    # a pass of one slice stores its amplitudes over whatever the output
    # holds, launched directly (3x3) or as a graph (4x6); with slices it adds
    # to zeros; new buffers on every call, and a pass between that leaves the
    # slice counter elsewhere
    c = qi.grid_circuit(rows, cols, depth, 6)
    m = q.Model(q.Circuit.grid(rows, cols, depth, 6))
    kw = {}
    if div:
        kw["mem_budget_bytes"] = q.Plan(m, batch=7, executor=q.EXEC_STEPWISE).info.arena_bytes // div
    p = q.Plan(m, batch=7, executor=q.EXEC_STEPWISE, **kw).bind()
    bits = qi.bitstrings(c.n, 7, 3)
    ref = sv.amplitudes(c, bits)
    for B in (7, 3):
        for _ in range(2):
            out = torch.full((2 * 7,), float("nan"), dtype=torch.float64, device="cuda")
            p.amplitudes(torch.from_numpy(bits[:B].view(np.int64)).cuda(), out, B=B)
            a = torch.view_as_complex(out.view(7, 2)).cpu().numpy()
            assert p.status() == 0 and np.all(np.isnan(a[B:].real))
            e = errmeasure.measures(a[:B], ref[:B], c.n)
            assert e["rel"] < TOL and e["abs"] < TOL, e


@pytest.mark.parametrize("rows,cols,depth,B", [(3, 3, 10, 5), (4, 6, 30, 4)])
def test_wait_between_steps_gives_up(q, rows, cols, depth, B):
    # a segment whose first step never runs: the units that wait for it give
    # up after 2 ms and the launch ends with a status; the next passes (one
    # launch after another, or a graph) are whole
    c = qi.grid_circuit(rows, cols, depth, 3)
    p = q.Plan(q.Model(q.Circuit.grid(rows, cols, depth, 3)), batch=B, executor=q.EXEC_STEPWISE).bind()
    bits = qi.bitstrings(c.n, B, 4)
    before = p.amplitudes_host(bits)
    for _ in range(2):
        assert q._lib.selftest_program_timeout(p, 2_000_000) == -4
        assert p.status() == 0
        assert np.array_equal(p.amplitudes_host(bits), before) and p.status() == 0
    with pytest.raises(q.QgmError):
        q._lib.selftest_program_timeout(p, 10)  # limit out of range


@pytest.mark.parametrize("rows,cols,depth,B,budget", [(4, 4, 20, 8, 20000), (4, 5, 24, 16, 400000), (4, 5, 28, 9, 1 << 20)])
def test_passes_share_their_memory(q, rows, cols, depth, B, budget):
    # a pass in program order, one step by step (profile) and one for a fixed
    # assignment use the same memory in turn, in different layouts; the first
    # plan's budget holds only with a step to a launch
    c = qi.grid_circuit(rows, cols, depth, 2)
    bits = qi.bitstrings(c.n, B, 5)
    d_bits = torch.from_numpy(bits.astype(np.int64)).cuda()
    p = q.Plan(q.Model(q.Circuit.grid(rows, cols, depth, 2)), batch=B, mem_budget_bytes=budget, executor=q.EXEC_STEPWISE).bind()
    assert p.info.arena_bytes <= budget
    ref = sv.amplitudes(c, bits)
    for _ in range(2):
        e = errmeasure.measures(p.amplitudes_host(bits), ref, c.n)
        assert p.status() == 0 and e["rel"] < TOL and e["abs"] < TOL, e
        p.profile(d_bits, torch.empty(2 * B, dtype=torch.float64, device="cuda"))
        raw, ex = p.eliminate_fixed([int(bits[1]) >> j & 1 for j in range(c.n)])
        assert abs(raw[0] * 2.0 ** ex - ref[1]) * 2.0 ** (c.n / 2) < TOL
