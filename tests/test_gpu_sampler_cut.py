"""The accept / pick step decided in FP32 against the one decided in FP64, and the slice cut
against a sequential restatement, at the edges of their ranges."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)


def probabilities(T, b_bits, seed):
    """Porter-Thomas rows, and every row in eight of another kind."""
    import torch
    rng = np.random.default_rng(seed)
    p = rng.exponential(size=(T, 64)) * 2.0 ** -(b_bits + 6)
    kinds = [
        lambda r: r * (rng.random(64) < 0.1),                      # mostly zeros
        lambda r: np.where(np.arange(64) == 17, r, 0.0),           # one outcome
        lambda r: np.zeros(64),
        lambda r: r * 2.0 ** rng.integers(-80, 1, size=64),        # far apart
        lambda r: r * 2.0 ** -900,                                 # below FP32's range
        lambda r: r * 1e200,                                       # above it
        lambda r: np.where(rng.random(64) < 0.1, [np.inf, np.nan, -1e-3, -0.0][rng.integers(4)], r),
        lambda r: np.full(64, 2.0 ** -(b_bits + 6)),               # equal, accepted about half the time
    ]
    for i in range(0, T, 8):
        p[i] = kinds[(i // 8) % len(kinds)](p[i])
    return torch.from_numpy(p).cuda()


@pytest.mark.parametrize("T,b_bits,alpha", [(1, 6, 2.0), (9, 0, 1.5), (33, 34, 2.0), (5000, 50, 4.0), (20011, 58, 2.0),
                                            (200003, 34, 2.0)])
def test_sampler_equals_the_fp64_sampler(T, b_bits, alpha):
    import torch
    import paper_2112_15083_gb300 as P
    p = probabilities(T, b_bits, T)
    # rows that start 8 bytes off a 16-byte boundary take the FP64 kernel
    flat = torch.empty(T * 64 + 1, dtype=torch.float64, device="cuda")
    q = flat[1:].view(T, 64)
    q.copy_(p)
    assert p.data_ptr() % 16 == 0 and q.data_ptr() % 16 == 8
    for seed in (1, 2):
        a, b = (P.rejection_sample(x, b_bits, alpha, seed, t0=seed * 1000) for x in (p, q))
        assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])


@pytest.mark.parametrize("k", [0, 1, 3, 5, 6, 7, 11, 12])
@pytest.mark.parametrize("f", [1e-9, 0.3, 0.999, 2.0])
def test_slice_cut_equals_a_sequential_cut(k, f):
    import paper_2112_15083_gb300 as P
    rng = np.random.default_rng(100 * k + int(10 * f))
    R = rng.exponential(size=1 << k)
    R[rng.random(R.size) < 0.2] = 0.0  # ties, broken by index
    R /= max(R.sum(), 1e-3)
    if R.size >= 8:
        R[3], R[5] = -0.0, -1e-9
    order = np.lexsort((np.arange(R.size), -R))
    acc, n = 0.0, R.size
    for t, i in enumerate(order):
        acc += R[i]
        if acc >= f:
            n = t + 1
            break
    X, F = P.slice_cut(R, f)
    assert np.array_equal(X, order[:n]) and F == acc
    X, F = P.tn.slice_cut_noalloc(R, f)
    assert np.array_equal(X, order[:n]) and F == acc
