"""The most probable strings of a batch (spoofing) against a selection from the batch's own
amplitudes, over batch sizes below, at and above a block of the selection, and all of N."""
import numpy as np
import pytest

from paper_2112_15083_gb300 import circuits as cg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("n_open", [1, 6, 10, 11, 13, 16])
@pytest.mark.parametrize("cycles", [2, 10])  # 2: many equal and zero probabilities
def test_selection_equals_a_sort(n_open, cycles):
    import paper_2112_15083_gb300 as P
    rows, cols = 4, 5
    openq = cg.default_open_qubits(rows, cols, n_open)
    C = P.circuit_load(cg.sycamore_grid(rows, cols, cycles, seed=4).serialize())
    plan = P.plan(C, openq, n_auto_sliced=3, log2_batches=0, order_trials=16)
    slices = np.arange(1 << len(plan.sliced_edges()), dtype=np.uint64)
    pattern = 3
    a = plan.contract(slices, np.array([pattern], dtype=np.uint64)).reshape(-1)
    p = a.real * a.real + a.imag * a.imag
    base = sum(((pattern >> c) & 1) << q for c, q in enumerate(q for q in range(20) if q not in openq))
    for N in sorted({1, 2, max(1, p.size // 10), p.size - 1, p.size}):
        if N < 1:
            continue
        i = np.sort(np.lexsort((np.arange(p.size), -p))[:N])
        want = np.array([base + sum(((int(x) >> r) & 1) << q for r, q in enumerate(openq)) for x in i], dtype=np.uint64)
        bits, probs = plan.spoof(slices, pattern, N, return_probs=True)
        assert np.array_equal(bits, want) and np.array_equal(probs, p[i]), (n_open, N)
