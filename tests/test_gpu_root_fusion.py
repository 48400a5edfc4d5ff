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


# a root with few outputs for its terms runs unfused by default: the fused kernel forms an
# output's terms one after the other.  rows, cols, cycles, circuit seed, open qubits, sliced
# legs, log2 batches, order seed; the root's (log2 outputs, free patterns, K); fused
@pytest.mark.parametrize("case,shape,fused", [
    ((4, 5, 9, 24, 10, 9, 0, 673), (10, 9, 1), False),
    ((4, 4, 7, 38, 6, 8, 4, 344), (10, 8, 2), False),
    ((4, 5, 7, 73, 4, 12, 6, 931), (10, 12, 2), False),
    ((4, 6, 7, 48, 6, 4, 4, 739), (10, 4, 2), True),
    ((4, 4, 6, 49, 6, 9, 6, 139), (12, 9, 0), True),
])
def test_default_fuses_where_the_outputs_fill_the_chip(case, shape, fused):
    import paper_2112_15083_gb300 as P
    rows, cols, cycles, circuit_seed, n_open, sliced, lb, order_seed = case
    C = P.circuit_load(cg.sycamore_grid(rows, cols, cycles, seed=circuit_seed).serialize())
    openq = cg.default_open_qubits(rows, cols, n_open)
    cb = cg.random_closed_bits(1 << lb, rows * cols - n_open, seed=1)
    outs, kernels = [], []
    for fuse in (None, False, True):
        plan = P.plan(C, openq, n_auto_sliced=sliced, log2_batches=lb, order_trials=2, order_seed=order_seed,
                      fuse_root_sum=fuse)
        sl = np.arange(1 << sliced, dtype=np.uint64)
        entry, out = traced_sum(plan, sl, cb)
        root = P.tn.plan_host(
            C, openq, n_auto_sliced=sliced, log2_batches=lb, order_trials=2, order_seed=order_seed)[1][-1]
        assert (n_open + lb, sum(root[:3]) - n_open - lb, root[3]) == shape
        kernels.append(entry["kernel"])
        outs.append(out)
    assert kernels == [3 if fused else 2, 2, 3]
    assert np.array_equal(outs[0], outs[1]) and np.array_equal(outs[0], outs[2])
