"""A budget that holds a call's tensors but not the extra memory of steps that share launches:
the call runs, its steps one by one, with the same amplitudes."""
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
def test_call_fits_the_budget_of_its_tensors(prec):
    import paper_2112_15083_gb300 as P
    rows, cols, lb = 4, 6, 8
    C = P.circuit_load(cg.sycamore_grid(rows, cols, 10, seed=3).serialize())
    openq = cg.default_open_qubits(rows, cols, 6)
    cb = cg.random_closed_bits(1 << lb, rows * cols - 6, seed=2)
    kw = dict(n_auto_sliced=8, log2_batches=lb, order_trials=16, precision=prec, autotune=0)
    roomy = P.plan(C, openq, **kw)
    kw.update(n_auto_sliced=0, sliced=roomy.sliced_edges())
    slices = np.arange(256, dtype=np.uint64)
    want = roomy.contract(slices, cb)

    def tensors(plan):
        # the estimate less its slack and its buffers per group: the tensors and twice the leaves
        return plan.estimate(slices)[0] - (64 << 20) - (1 << lb) * (64 * 16 + 64)

    # the order search knows the budget: repeat until the budget is what its own plan's tensors take
    plan, budget = roomy, 0
    for _ in range(6):
        if tensors(plan) == budget:
            break
        budget = tensors(plan)
        plan = P.plan(C, openq, hbm_budget_bytes=float(budget), **kw)
    assert tensors(plan) == budget
    for _ in range(2):
        got = plan.contract(slices, cb)
        assert np.abs(got - want).max() <= (1e-4, 1e-3)[prec] * np.abs(want).max()
    with pytest.raises(P.TnError) as e:
        P.plan(C, openq, hbm_budget_bytes=budget * 0.25, **kw).contract(slices, cb)
    assert e.value.code == P.tn.TN_ENOMEM
