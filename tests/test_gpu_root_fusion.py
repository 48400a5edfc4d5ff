"""Which of the root step and the FP64 slice sum run fused: what fuse_root_sum asks for."""
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


def traced_sum(plan, slices, cb):
    """The slice sum's trace entry of one execution, and the plan's amplitudes."""
    plan.contract(slices, cb)
    plan.trace(True)
    out = plan.contract(slices, cb)
    entry = plan.trace_read()[-1]
    plan.trace(False)
    assert entry["launches"] == 1
    return entry, out


# a root with K <= 4 and 2^16 amplitudes of 64 slices
def short_root(**kw):
    import paper_2112_15083_gb300 as P
    C = P.circuit_load(cg.sycamore_grid(4, 5, 12, seed=0).serialize())
    plan = P.plan(C, cg.default_open_qubits(4, 5, 16), n_auto_sliced=6, log2_batches=0, order_trials=64,
                  hbm_budget_bytes=90e9, parallel_search=True, **kw)
    return plan, np.arange(64, dtype=np.uint64), np.array([5], dtype=np.uint64)


def test_fuse_root_sum_is_what_was_asked_for():
    kernels, outs = [], []
    for kw in ({}, {"fuse_root_sum": None}, {"fuse_root_sum": True}, {"fuse_root_sum": False}, {"fuse_root_sum": -1}):
        entry, out = traced_sum(*short_root(**kw))
        kernels.append(entry["kernel"])
        outs.append(out)
    assert kernels == [3, 3, 3, 2, 2]  # 3: one launch with the root step, 2: a launch of its own
    assert all(np.array_equal(o, outs[0]) for o in outs)
