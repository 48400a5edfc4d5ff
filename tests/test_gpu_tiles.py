"""Every complex64 kernel variant gives the bits of the fixed rules' choice: the packed tiles
(square and narrow, rows on either side, operands in place) among them.  Step k of a plan
with autotune = 2 + r runs the variant (k + r) mod count of its shape."""
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


# rows, cols, cycles, sliced legs, log2 batches, slices (None: all)
@pytest.mark.parametrize("case", [(3, 4, 8, 2, 4, None), (4, 5, 12, 6, 8, None), (4, 5, 10, 5, 3, [0, 1, 6, 7, 21]),
                                  (4, 6, 12, 8, 10, None)])
def test_every_variant_gives_the_same_bits(case):
    import paper_2112_15083_gb300 as P
    rows, cols, cycles, sliced, lb, slices = case
    C = P.circuit_load(cg.sycamore_grid(rows, cols, cycles, seed=1).serialize())
    openq = cg.default_open_qubits(rows, cols, 6)
    cb = cg.random_closed_bits((1 << lb) + 3, rows * cols - 6, seed=9)
    kw = dict(n_auto_sliced=sliced, log2_batches=lb, order_trials=16)
    plan = P.plan(C, openq, autotune=0, **kw)
    sl = np.array(range(1 << len(plan.sliced_edges())) if slices is None else slices, dtype=np.uint64)
    ref = plan.contract(sl, cb)
    seen = set()
    for r in range(13):
        p = P.plan(C, openq, autotune=2 + r, **kw)
        p.trace(True)
        got = p.contract(sl, cb)
        seen |= {s["kernel"] for s in p.trace_read() if s["launches"]}
        p.trace(False)
        assert np.array_equal(got, ref), (case, r)
    if rows * cols == 24:
        assert {128064, 64064, 128032, 64032, 32032, 256016, 128016, 256008, 256004, 16016} <= seen, sorted(seen)


# steps with a short side of up to 4 and K <= 16 whose long operand is read in place: the row
# kernels and the row products over stacked batches (kernel 6); ragged last groups
@pytest.mark.parametrize("case", [(4, 5, 11, 6, 8), (4, 5, 11, 6, 9), (4, 6, 8, 8, 8)])
def test_stacked_rows_give_the_same_bits(case):
    import paper_2112_15083_gb300 as P
    rows, cols, cycles, sliced, lb = case
    C = P.circuit_load(cg.sycamore_grid(rows, cols, cycles, seed=0).serialize())
    openq = cg.default_open_qubits(rows, cols, 6)
    cb = cg.random_closed_bits((1 << lb) + 77, rows * cols - 6, seed=9)
    cb[5:40] = cb[4]  # more batches on one stored block than a stack holds
    kw = dict(n_auto_sliced=sliced, log2_batches=lb, order_trials=16)
    plan = P.plan(C, openq, autotune=0, **kw)
    sl = np.arange(1 << len(plan.sliced_edges()), dtype=np.uint64)
    ref = plan.contract(sl, cb)
    seen = set()
    for r in range(6):
        p = P.plan(C, openq, autotune=2 + r, **kw)
        p.trace(True)
        got = p.contract(sl, cb)
        seen |= {s["kernel"] for s in p.trace_read() if s["launches"]}
        p.trace(False)
        assert np.array_equal(got, ref), (case, r)
    if lb == 8:
        assert 6 in seen, sorted(seen)
