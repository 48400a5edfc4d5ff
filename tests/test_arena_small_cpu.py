"""The memory of the steps that share launches: their results are kept apart from every other
tensor of a call, take at most the 48 MiB that the estimates' slack covers, and can be laid
out like the other steps' where there is no room for that."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2112_15083_gb300 import circuits as cg

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    import __graft_entry__
    __graft_entry__.build()
    out = str(tmp_path_factory.mktemp("arena") / "libarena.so")
    subprocess.run([cxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-ffp-contract=off",
                    "-I", os.path.join(ROOT, "paper_2112_15083_gb300", "csrc"), "-I", os.path.join(ROOT, "include"),
                    os.path.join(HERE, "emulator", "arena_small.cpp"), "-o", out], check=True)
    return ctypes.CDLL(out)


# rows, cols, cycles, open qubits, sliced legs, log2 batches, slices (None: all)
@pytest.mark.parametrize("case", [(3, 4, 8, 6, 2, 4, None), (4, 4, 9, 4, 0, 6, None), (4, 5, 10, 6, 5, 8, [0, 1, 2, 3, 9, 17]),
                                  (4, 5, 12, 6, 6, 10, None), (4, 5, 12, 14, 6, 0, None), (4, 6, 10, 6, 8, 12, [5, 6])])
@pytest.mark.parametrize("prec", [0, 1])
def test_small_results_are_kept_apart(lib, case, prec):
    import paper_2112_15083_gb300 as P
    rows, cols, cycles, n_open, sliced, lb, slices = case
    o = P.tn.PlanOpts()
    P.lib().tn_plan_opts_default(ctypes.byref(o))
    o.log2_batches, o.n_auto_sliced, o.order_trials, o.precision = lb, sliced, 2, prec
    buf = cg.sycamore_grid(rows, cols, cycles, seed=3).serialize()
    openq = np.array(cg.default_open_qubits(rows, cols, n_open), dtype=np.int32)
    sl = np.arange(1 << sliced, dtype=np.uint64) if slices is None else np.array(slices, dtype=np.uint64)
    out = np.zeros(3, dtype=np.int64)
    vp = ctypes.c_void_p
    bad = lib.arena_small(buf, ctypes.c_size_t(len(buf)), openq.ctypes.data_as(vp), openq.size, ctypes.byref(o),
                          sl.ctypes.data_as(vp), ctypes.c_int64(sl.size), out.ctypes.data_as(vp))
    assert bad == 0
    without, with_small, n_small = (int(x) for x in out)
    assert n_small > 0 and with_small <= without + (48 << 20)
