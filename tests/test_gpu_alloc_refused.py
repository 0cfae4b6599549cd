"""Device memory that runs out: every allocation of a plan's creation, solves and
backward pass refused once (MADMAP_FAULT_ALLOC_FAIL_AT, a host-side refusal), in a
process of its own since the count is the process's.  A call either fails with the
out-of-memory status and works when it is made again, or does without the memory.
"""

from __future__ import annotations

import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PRELUDE = r'''
import os
import numpy as np, torch
import paper_0906_1775_gb300 as mm
from tests.gpu_helpers import cuda, host, make_plan
from tests.helpers import rel_rms, system_for, tiny_T

VAR = "MADMAP_FAULT_ALLOC_FAIL_AT"
count = 0        # the process's device allocations so far

def refuse_each(call):
    """The result of call(), after calls with its first, second, ... allocation refused."""
    global count
    k = 1
    while True:
        os.environ[VAR] = str(count + k)
        try:
            out = call()
        except mm.MadmapError as e:
            assert e.status == mm._lib.MADMAP_ERR_OOM, e
            count += k
            k += 1
            continue
        del os.environ[VAR]
        count += k - 1
        return out, k - 1

p = tiny_T(seed=170, n=60000, width=16, n_lags=64, ivls=(20000, 40000))
kw = dict(precision="mixed", rel_tol=1e-11, max_iter=300)
d = cuda(p.d[0])
'''


def _run(code):
    env = {k: v for k, v in os.environ.items() if k != "MADMAP_FAULT_ALLOC_FAIL_AT"}
    out = subprocess.run([sys.executable, "-c", PRELUDE + code], capture_output=True, text=True, env=env, cwd=ROOT,
                         timeout=300)
    assert out.returncode == 0 and "DONE" in out.stdout, out.stdout + out.stderr


@pytest.mark.parametrize("nth", [1, 9, 16, 20])
def test_a_solve_works_after_a_refused_allocation(nth):
    """In the float64 buffers, and in the float32 ones after them (20)."""
    _run(r'''
plan, n = refuse_each(lambda: make_plan(p))
assert n > 10
os.environ[VAR] = str(count + %d)
try:
    plan.solve(d, **kw)
    raise AssertionError("the allocation was not refused")
except mm.MadmapError as e:
    assert e.status == mm._lib.MADMAP_ERR_OOM, e
m, info = plan.solve(d, **kw)
m2, _ = make_plan(p).solve(d, **kw)
assert info["status"] == 0 and rel_rms(host(m), host(m2)) < 1e-8
print("DONE")
''' % nth)
