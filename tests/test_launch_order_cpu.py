"""The order in which an execution's launches run (small steps share launches, ahead of their place
in the step list) against the arena that was planned in step order: when a launch reads an
operand, nothing has overwritten it, in the first execution and in a later batch group's."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2112_15083_gb300 import circuits as cg

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

# rows, cols, cycles, open qubits, sliced legs, log2 batches, slices (None: all)
CASES = [(3, 4, 8, 6, 2, 4, None), (4, 4, 9, 4, 0, 6, None), (4, 5, 10, 6, 5, 8, [0, 1, 2, 3, 9, 17]),
         (4, 5, 12, 6, 6, 10, None), (4, 5, 12, 14, 6, 0, None), (4, 6, 10, 6, 8, 12, [5, 6]), (4, 6, 8, 6, 4, 8, None)]


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2112_15083_gb300 as P
    out = str(tmp_path_factory.mktemp("order") / "liborder.so")
    subprocess.run([cxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-ffp-contract=off",
                    "-I", os.path.join(ROOT, "paper_2112_15083_gb300", "csrc"), "-I", os.path.join(ROOT, "include"),
                    os.path.join(HERE, "emulator", "launch_order.cpp"), "-o", out], check=True)
    lib = ctypes.CDLL(out)

    def run(case, prec, seed, plant=0):
        rows, cols, cycles, n_open, sliced, lb, slices = case
        o = P.tn.PlanOpts()
        P.lib().tn_plan_opts_default(ctypes.byref(o))
        o.log2_batches, o.n_auto_sliced, o.order_trials, o.precision, o.order_seed = lb, sliced, 2, prec, seed
        buf = cg.sycamore_grid(rows, cols, cycles, seed=3).serialize()
        openq = np.array(cg.default_open_qubits(rows, cols, n_open), dtype=np.int32)
        sl = np.arange(1 << sliced, dtype=np.uint64) if slices is None else np.array(slices, dtype=np.uint64)
        out = np.zeros(2, dtype=np.int64)
        vp = ctypes.c_void_p
        bad = lib.launch_order_check(buf, ctypes.c_size_t(len(buf)), openq.ctypes.data_as(vp), openq.size, ctypes.byref(o),
                                     sl.ctypes.data_as(vp), ctypes.c_int64(sl.size), plant, out.ctypes.data_as(vp))
        assert bad >= 0
        return bad, [int(x) for x in out]

    return run


@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("prec", [0, 1])
def test_no_operand_is_overwritten_before_it_is_read(check, case, prec):
    for seed in range(3):
        bad, (shared, ahead) = check(case, prec, seed)
        assert bad == 0
        assert shared > 0 and ahead > 0  # the order differs from the step list


@pytest.mark.parametrize("plant", [1, 2])
def test_planted_mistakes_fail(check, plant):
    assert any(check(case, 0, 0, plant)[0] > 0 for case in CASES)
