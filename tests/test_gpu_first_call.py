"""The first call of a process, on a stream that is not ordered after the default one: what the library uploads for
it (function tables, rules, counters) has to be on the device before the kernels run."""
import os
import subprocess
import sys

import pytest

from gpu_common import gpu_context

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CODE = """
import ctypes, sys
import numpy as np, torch
import ffrg_inputs as fi
import paper_2412_13043_gb300 as ffrg
lib = ffrg.load()
wl = fi.make_finite_t(seed=5, N=3, T=0.05, n_pts=16, n_ext_p=4, n_ext_m=2, n_rad=9, n_ang=7) if sys.argv[1] == "ft" \
    else fi.make_d3(seed=5, n_pts=16, n_ext_p=4, n_rad=9, n_ang=7)
tab = torch.tensor(wl.tables, dtype=torch.float64, device="cuda")
out = torch.zeros(wl.problem.n_ext(), dtype=torch.float64, device="cuda")
ctx = ffrg.Context(0)
tabs = ctx.tables(wl.problem, wl.tables)
torch.cuda.synchronize()
s = torch.cuda.Stream()   # non-blocking
with torch.cuda.stream(s):
    if sys.argv[2] == "noalloc":
        code = lib.ffrg_rhs_noalloc(ctypes.byref(ffrg.to_problem(wl.problem)), ctypes.byref(ffrg.to_desc(wl.problem)),
                                    tab.data_ptr(), 1.1, out.data_ptr(), int(ffrg.FP64), s.cuda_stream)
        assert code == ffrg.OK
    else:
        out = ctx.rhs(wl.problem, tabs, 1.1, precision=ffrg.FP64)
s.synchronize()
first = out.cpu().numpy()
again = ctx.rhs(wl.problem, tabs, 1.1, precision=ffrg.FP64).cpu().numpy()
assert np.all(np.isfinite(first)) and np.array_equal(first, again), (first, again)
"""


@pytest.mark.parametrize("entry", ["noalloc", "rhs"])
@pytest.mark.parametrize("model", ["d3", "ft"])
def test_first_call_of_a_process(model, entry):
    gpu_context().close()   # skips without a device
    subprocess.run([sys.executable, "-c", CODE, model, entry], cwd=ROOT, check=True, timeout=300)
