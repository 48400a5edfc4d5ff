"""The launches of a replayed execution (tn_plan_launches, which the benchmark reports): the
traced launches where every step runs by itself, fewer where steps share launches."""
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


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("rows,cols,sliced,lb", [(3, 4, 2, 4), (4, 5, 6, 8)])
def test_replayed_launches(rows, cols, sliced, lb, prec):
    import bench
    import paper_2112_15083_gb300 as P
    C = P.circuit_load(cg.sycamore_grid(rows, cols, 8, seed=3).serialize())
    cb = cg.random_closed_bits(3 << lb, rows * cols - 6, seed=2)  # three groups: two reuse the stem
    slices = np.arange(1 << sliced, dtype=np.uint64)
    for autotune, grouped in ((3, False), (0, True)):
        plan = P.plan(C, cg.default_open_qubits(rows, cols, 6), n_auto_sliced=sliced, log2_batches=lb, order_trials=8,
                      precision=prec, autotune=autotune)
        assert plan.replayed_launches(False) == plan.replayed_launches(True) == 0
        plan.contract(slices, cb)
        plan.contract(slices, cb)
        first, later = plan.replayed_launches(False), plan.replayed_launches(True)
        plan.trace(True)
        plan.contract(slices, cb)
        trace = plan.trace_read()
        plan.trace(False)
        steps, ssum = bench.split_trace(trace)
        traced = sum(s["launches"] * bench.launches_per(s) for s in steps) + sum(s["launches"] for s in ssum)
        assert 0 < later <= first
        assert bench.replayed_launches(plan, 3, traced) == first + 2 * later
        assert (first + 2 * later < traced) if grouped else (first + 2 * later == traced)
