"""Short windows in one CTA or in three kernels, by layout and number of windows.

One tile (two windows) on either side of each line: which way runs is read from
time_operator's launches (the second kernel has none where one does the work), and
both ways of a problem of this size match the operator of the same plan in the
other precision (float32 against double-float, float64 against double-float; each of
them is checked against the oracle elsewhere).
"""

from __future__ import annotations

import numpy as np
import pytest

from tests.gpu_helpers import host
from tests.helpers import rel_rms

pytestmark = pytest.mark.gpu

N_LAGS, W = 17, 48


def _plan(layout, M, tiles):
    import torch
    import paper_0906_1775_gb300 as mm
    n = 2 * tiles * (M - 2 * (N_LAGS - 1))
    lags = mm.noise_filter(N_LAGS, 100.0, 1.0, 3.0, 1.5)[None]
    off, filt = np.array([0, n]), np.zeros(1, np.int32)
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    if layout == "otf":
        u = np.arange((n - 1) // 8 + 2)
        x, y, a = W / 2 + 25 * np.sin(u * 0.011), W / 2 + 25 * np.cos(u * 0.0137), u * 1e-3
        bore = torch.from_numpy(np.stack([x, y, np.cos(a), np.sin(a)], 1).astype(np.float32)).cuda()
        return mm.Plan.from_boresight(bore, 8, np.array([[0.3, 0.2, 1.0, 0.0]]), n, W, W, True, off, filt, lags, fft_len=M)
    pix = torch.randint(0, W * W, (n,), generator=g, device="cuda", dtype=torch.int32)
    psi = torch.rand(n, generator=g, device="cuda") * 3.1
    kw = {}
    if layout == "ext":
        kw = dict(extra_index=(torch.arange(n, device="cuda") // 5000).to(torch.int32), n_extra=n // 5000 + 1)
    if layout == "hwp":
        kw = dict(hwp=(torch.remainder(torch.arange(n, device="cuda") * 0.013, 6.28).to(torch.float32),
                       torch.rand(n, generator=g, device="cuda"), np.zeros(1, np.int32), 1))
    return mm.Plan(pix, psi, W * W, off, filt, lags, fft_len=M, **kw)


@pytest.mark.parametrize("layout, M, points, prec", [
    ("hwp", 512, 3 << 19, "fp32"), ("hwp", 4096, 3 << 19, "fp32"), ("ext", 1024, 3 << 20, "fp32"),
    ("ext", 4096, 3 << 20, "fp32"), ("otf", 2048, 3 << 20, "fp32"), ("iqu", 256, 608 * 256, "fp64")])
def test_both_sides_of_each_line(layout, M, points, prec):
    import torch
    for tiles, three in ((points // M, False), (points // M + 1, True)):
        plan = _plan(layout, M, tiles)
        assert plan.stats["n_tiles"] == tiles
        launches = plan.time_operator(prec, reps=1)[1]
        assert (launches[1] > 0) == three, (tiles, launches)
        x = torch.randn((plan.n_obs, 3), device="cuda")
        d = torch.randn(plan.n_samples, device="cuda")
        dt = torch.float32 if prec == "fp32" else torch.float64
        tol = 2e-5 if prec == "fp32" else 1e-11
        y, ref = plan.apply_ATNA(x.to(dt), precision=prec), plan.apply_ATNA(x.to(torch.float64), precision="df64")
        assert rel_rms(host(y), host(ref)) < tol
        b, bref = plan.rhs(d, precision=prec), plan.rhs(d, precision="df64")
        assert rel_rms(host(b), host(bref)) < tol


@pytest.mark.parametrize("layout, M, tiles, prec", [
    ("iqu", 4096, 1100, "fp32"), ("ext", 512, 6200, "fp32"), ("otf", 1024, 3100, "fp32"), ("iqu", 512, 700, "fp64"),
    ("iqu", 256, 700, "df64")])
def test_layouts_that_stay_with_one_cta(layout, M, tiles, prec):
    launches = _plan(layout, M, tiles).time_operator(prec, reps=1)[1]
    assert launches[0] > 0 and launches[1] == 0


@pytest.mark.parametrize("prec, graph", [("fp64", 2), ("mixed", 2), ("mixed", 1)])
def test_a_tile_set_may_take_the_other_way(prec, graph):
    """One right-hand side below a line (float64, M = 256; float32 with half-wave-plate
    terms), three of them above it, inside the solver's captured loops."""
    import torch
    plan = _plan("hwp", 512, 2000) if prec == "mixed" else _plan("iqu", 256, 500)
    d = torch.randn(plan.n_samples, device="cuda")
    kw = dict(precision=prec, rel_tol=1e-9, max_iter=300, use_graph=graph)
    m, i = plan.solve(d, **kw)
    ms, infos = plan.solve_batched(torch.stack([d, 2 * d, 4 * d]), **kw)
    assert i["status"] == 0 and all(k["status"] == 0 for k in infos)
    for k in range(3):
        assert rel_rms(host(ms[k]), 2.0 ** k * host(m)) < 1e-6
