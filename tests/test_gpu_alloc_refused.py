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


def test_lag_gradient_and_noise_filters_do_without_their_buffers():
    """The transforms' buffers refused: direct sums; the noise filters' refused: the host's sums."""
    _run(r'''
def set_up():
    plan = make_plan(p)
    m, _ = plan.solve(d, **kw)
    g = torch.ones_like(m)
    plan.solve_backward(d, m, g, want_lags=False, **kw)
    return plan, m, g
(plan, m, g), n = refuse_each(set_up)
assert n > 30
os.environ[VAR] = str(count + 1)
_, gl, _ = plan.solve_backward(d, m, g, want_d=False, **kw)
count += 2                                     # the refused buffers, and the direct sums' item list
prm = np.array([[1.1, 3.0, 1.2]])
os.environ[VAR] = str(count + 1)
plan.set_noise(p.fs, prm)
del os.environ[VAR]
fresh = make_plan(p)
_, gl2, _ = fresh.solve_backward(d, m, g, want_d=False, **kw)
# a lag is an inner product of a = A lambda and a shifted r = d - A m, and each way of
# summing it in float32 is within 4e-6 |a| |r| of it (test_gpu_reg_transforms)
S = system_for(p)
lam, _ = S.pcg(host(g), rel_tol=1e-13, max_iter=1000)
scale = np.linalg.norm(S.unpoint(lam)) * np.linalg.norm(p.d[0] - S.unpoint(host(m)))
assert np.abs(host(gl) - host(gl2)).max() < 8e-6 * scale, np.abs(host(gl) - host(gl2)).max() / scale
other = make_plan(p, lags=mm.noise_filter(p.n_lags, p.fs, *prm[0])[None])
y = cuda(np.random.default_rng(0).standard_normal(p.n_samples), torch.float64)
assert rel_rms(host(plan.apply_ninv(y)), host(other.apply_ninv(y))) < 1e-12
print("DONE")
''')
