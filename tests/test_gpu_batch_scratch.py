"""Scratch of batched solves: as large as the set of tiles needs, grown by a larger
set, and none for windows that one CTA holds in every precision.

The device memory is the plan's own count (stats device_bytes, solve buffers
included).  Maps: right-hand sides that are powers of two times one timestream give
the same multiples of the oracle's map.
"""

from __future__ import annotations

import numpy as np
import pytest

from tests.gpu_helpers import cuda, host, make_plan
from tests.helpers import rel_rms, system_for, tiny_T

pytestmark = pytest.mark.gpu


def _problem(n, seed=160):
    return tiny_T(seed=seed, n=n, width=8, n_lags=65, ivls=(n // 3, n - n // 3))


def _bytes(plan):
    import paper_0906_1775_gb300 as mm
    return mm.madmap_plan_get_stats(plan._h)["device_bytes"]


def _solve(plan, p, n_rhs, **kw):
    d = cuda(p.d[0])
    scale = [2.0 ** (k % 5) for k in range(n_rhs)]
    import torch
    m, infos = plan.solve_batched(torch.stack([s * d for s in scale]), rel_tol=1e-12, max_iter=400, **kw)
    assert all(i["status"] == 0 for i in infos)
    return host(m) / np.array(scale)[:, None, None]


@pytest.mark.parametrize("fft_len, n, n_rhs", [(1 << 15, 90000, 4), (1 << 10, 20000, 16), (1 << 12, 60000, 5)])
def test_scratch_is_what_the_set_needs(fft_len, n, n_rhs):
    p = _problem(n)
    plan = make_plan(p, fft_len=fft_len)
    before = _bytes(plan)
    _solve(plan, p, n_rhs, precision="mixed")
    # both slots: every lane of the set at 16 bytes a complex element, two lanes an element
    need = plan.stats["n_segments"] * n_rhs * fft_len * 16 + (8 << 20)   # + solve vectors of 64 rows, tiles
    if fft_len == 1 << 10:
        need = 8 << 20
    assert _bytes(plan) - before < need, _bytes(plan) - before


@pytest.mark.parametrize("fft_len", [1 << 11, 1 << 12, 1 << 13, 1 << 14])
@pytest.mark.parametrize("prec, graph", [("fp64", 2), ("mixed", 2), ("mixed", 1)])
def test_sets_of_growing_size_on_one_plan(fft_len, prec, graph):
    """A larger set replaces the scratch of the smaller ones, whose captured loops must
    follow: 3, 8, 3, 17 and 8 right-hand sides in turn."""
    p = _problem(150000)
    plan = make_plan(p, fft_len=fft_len)
    x, _ = system_for(p).solve(p.d[0], rel_tol=1e-13, max_iter=400)
    for n_rhs in (3, 8, 3, 17, 8):
        for m in _solve(plan, p, n_rhs, precision=prec, use_graph=graph):
            assert rel_rms(m, x) < (1e-10 if prec == "fp64" else 1e-6), n_rhs
