"""Statistics of and samples from a computed set at the sizes where the
cluster kernels split differently: fewer amplitudes than CTAs or threads,
parts of uneven length, several scan tiles per CTA, and irregular values."""
import numpy as np
import pytest

from oracle import xeb

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def q():
    from paper_1712_05384_gb300 import build
    build.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1712_05384_gb300 as q
    return q


def _set(t, seed):
    z = np.random.default_rng(seed).standard_normal(2 * t) * 2.0 ** -10
    return z[0::2] + 1j * z[1::2]


def _device(a):
    return torch.from_numpy(np.ascontiguousarray(a).view(np.float64)).cuda()


@pytest.mark.parametrize("t", [1, 2, 7, 8, 9, 513, 1025, 8191, 32769, 65536, 100003])
def test_set_of_every_size(q, t):
    a = _set(t, t)
    d = _device(a)
    st = q._lib.xeb_stats(d, t, 20, torch.zeros(4, dtype=torch.float64, device="cuda"))
    ref = xeb.stats(a, 20)
    for k in ref:  # t roundings of 2^-53 at most, far below 1e-11 of the sums
        assert abs(st[k] - ref[k]) <= 1e-11 * max(1.0, abs(ref[k])), k
    m = 3001
    cdf = torch.zeros(t, dtype=torch.float64, device="cuda")
    idx = torch.full((m,), -1, dtype=torch.int64, device="cuda")
    q._lib.sample_from_set(d, t, m, 11, cdf, idx)
    want, _, _ = xeb.sample_from_set(a, m, 11)
    assert np.array_equal(idx.cpu().numpy(), want)
    total = np.cumsum(np.abs(a) ** 2)
    assert np.max(np.abs(cdf.cpu().numpy() - total)) <= 1e-12 * total[-1]


def test_irregular_probabilities(q):
    a = _set(5000, 3)
    a[17] = 1e-160  # p subnormal: its logarithm is taken on its own
    p = np.abs(a) ** 2
    st = q._lib.xeb_stats(_device(a), 5000, 20, torch.zeros(4, dtype=torch.float64, device="cuda"))
    want = -np.mean(np.log(a.real * a.real + a.imag * a.imag))
    assert abs(st["cross_entropy"] - want) <= 1e-11 * abs(want)
    a[40:60] = 0  # empty stretch: never drawn; log 0 makes the entropy infinite
    d = _device(a)
    st = q._lib.xeb_stats(d, 5000, 20, torch.zeros(4, dtype=torch.float64, device="cuda"))
    assert st["cross_entropy"] == np.inf
    idx = torch.zeros(20000, dtype=torch.int64, device="cuda")
    q._lib.sample_from_set(d, 5000, 20000, 5, torch.zeros(5000, dtype=torch.float64, device="cuda"), idx)
    assert np.array_equal(idx.cpu().numpy(), xeb.sample_from_set(a, 20000, 5)[0])
    a[99] = np.nan
    st = q._lib.xeb_stats(_device(a), 5000, 20, torch.zeros(4, dtype=torch.float64, device="cuda"))
    assert np.isnan(st["cross_entropy"]) and np.isnan(st["mean_Np"])


@pytest.mark.parametrize("t", [1, 2, 511, 512, 513, 1024, 1025, 5000, 131073, 300001])
def test_cumulative_sums_are_ordered(q, t):
    # never falling, and an entry of probability zero has its predecessor's
    # sum, so that no draw can find it: zeros strewn about and in stretches
    # over the ends of the kernels' chunks, values of every size
    rng = np.random.default_rng(t)
    a = _set(t, t) * 2.0 ** rng.integers(-30, 1, t)
    a[rng.random(t) < 0.4] = 0
    for s in range(0, t, 512 * 7):
        a[max(0, s - 300):s + 700] = 0
    if t > 2000:
        a[-3:] = 0
    a[t // 2] = 1e-3
    p = a.real * a.real + a.imag * a.imag
    cdf = torch.zeros(t, dtype=torch.float64, device="cuda")
    idx = torch.full((20000,), -1, dtype=torch.int64, device="cuda")
    q._lib.sample_from_set(_device(a), t, 20000, 7, cdf, idx)
    c = np.concatenate([[0.0], cdf.cpu().numpy()])
    step = np.diff(c)
    assert np.all(step >= 0) and np.all(step[p == 0] == 0)
    assert np.max(np.abs(c[1:] - np.cumsum(p))) <= 1e-12 * c[-1]
    assert np.all(p[idx.cpu().numpy()] > 0)
