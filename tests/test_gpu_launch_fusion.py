"""Launches that were merged or re-ordered against the launches they replace, bit for bit:
the FP64 slice sum (tests/standalone/slice_sum.cu, against host sums), the root
step fused with it, and small steps sharing a launch."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2112_15083_gb300 import circuits as cg

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.fixture(scope="module", autouse=True)
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)


def test_slice_sum_against_host_sums(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path / "slice_sum")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-o", exe,
                    os.path.join(HERE, "standalone", "slice_sum.cu"), "-I" + os.path.join(ROOT, "include")], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr


# rows, cols, cycles, open qubits, sliced legs, log2 batches, batches, slices (None: all)
CASES = [
    (3, 4, 8, 6, 2, 4, 21, None),
    (3, 4, 8, 6, 3, 0, 3, [1, 2, 4]),
    (4, 5, 12, 6, 6, 10, 1024, None),
    (4, 5, 10, 6, 5, 8, 300, [0, 1, 2, 3, 9, 17]),
    (4, 5, 12, 14, 6, 0, 2, None),
    (4, 4, 9, 4, 0, 6, 64, None),
]


def make(case, prec, **kw):
    import paper_2112_15083_gb300 as P
    rows, cols, cycles, n_open, sliced, lb, nb, slices = case
    C = P.circuit_load(cg.sycamore_grid(rows, cols, cycles, seed=3).serialize())
    plan = P.plan(C, cg.default_open_qubits(rows, cols, n_open), n_auto_sliced=sliced, log2_batches=lb, order_trials=16,
                  precision={"c64": P.tn.PREC_C64, "bf16x2": P.tn.PREC_BF16X2, "fp16x2": P.tn.PREC_FP16X2}[prec], **kw)
    sl = np.arange(1 << len(plan.sliced_edges())) if slices is None else slices
    return plan, np.array(sl, dtype=np.uint64), cg.random_closed_bits(nb, rows * cols - n_open, seed=11)


@pytest.mark.parametrize("prec", ["c64", "bf16x2", "fp16x2"])
@pytest.mark.parametrize("case", CASES)
def test_root_fused_by_default_equals_separate_launches(case, prec):
    a, slices, cb = make(case, prec)
    b, _, _ = make(case, prec, fuse_root_sum=-1)
    for _ in range(2):  # the first execution may tune, the second replays
        assert np.array_equal(a.contract(slices, cb), b.contract(slices, cb))


@pytest.mark.parametrize("prec", ["c64", "bf16x2", "fp16x2"])
@pytest.mark.parametrize("case", CASES)
def test_grouped_small_steps_equal_single_launches(case, prec):
    plan, slices, cb = make(case, prec)
    plan.contract(slices, cb)
    grouped = plan.contract(slices, cb)
    plan.trace(True)  # a traced execution launches every step by itself
    single = plan.contract(slices, cb)
    plan.trace(False)
    assert np.array_equal(grouped, single)
    # other patterns and back: nothing of a group is kept for the next
    plan.contract(slices, cb ^ np.uint64(1))
    assert np.array_equal(plan.contract(slices, cb), single)
