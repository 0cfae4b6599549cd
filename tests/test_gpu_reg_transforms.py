"""The operator by window length: one CTA per window (up to 2^12 points in
float32, 2^11 in the wider types), the register transforms (2^14 to 2^18) and
the three shared-memory kernels between and above.

Every row length N1 = M / 256 of 64 to 1024 points runs its own kernel.  Each length's
N^-1 is checked against the Eq. 15 direct sum on intervals that end inside,
at and past a window's exact part, and its operator (gather and scatter of both
paired windows, an odd number of them, flagged samples) against the oracle.

Tolerance: a float32 transform of 2^18 points and its inverse pass 36 radix-2
levels; each level and each twiddle product adds at most about two roundings
of 2^-24, and they add up as a random walk: 2^-24 * 2 * sqrt(2 * 36) = 1e-6.
"""

from __future__ import annotations

import numpy as np
import pytest

from tests.gpu_helpers import cuda, host, make_plan
from tests.helpers import lags_for, rel_rms, system_for, tiny_IQU, tiny_T

pytestmark = pytest.mark.gpu

TOL = 1e-6
# the same count of roundings at 2^-53; double-float rounds at 2^-47 and passes
# the two weights' products at that too
TOLS = {"fp32": TOL, "fp64": TOL * 2.0 ** -29 * 4, "df64": TOL * 2.0 ** -23 * 4}


@pytest.mark.parametrize("lg", range(8, 20))
def test_weighting_matches_direct_sum(lg):
    import torch
    from oracle.noise import apply_ninv_direct
    M = 1 << lg
    n_lags = 129 if lg > 9 else 33
    exact = M - 2 * (n_lags - 1)     # samples one window weighs exactly
    p = tiny_T(seed=90 + lg, n=4 * exact + 777, width=24, n_lags=n_lags, ivls=(1, 775, exact, exact + 1, 2 * exact))
    plan = make_plan(p, fft_len=M)
    assert plan.stats["fft_len"] == M
    y = np.random.default_rng(lg).standard_normal(p.n_samples).astype(np.float32)
    ref = apply_ninv_direct(y.astype(np.float64), p.interval_offsets, p.interval_filter, lags_for(p))
    w = host(plan.apply_ninv(cuda(y, torch.float32), precision="fp32"))[0]
    assert rel_rms(w, ref) < TOL, rel_rms(w, ref)
    # an interval alone: two windows share a complex transform, so a short one's
    # rounding is relative to its partner's values too (rms of the whole), and a
    # single sample carries no averaging (four standard deviations)
    whole = np.sqrt(np.mean(ref ** 2))
    for i in range(len(p.interval_filter)):
        a, b = int(p.interval_offsets[i]), int(p.interval_offsets[i + 1])
        scale = max(whole, np.sqrt(np.mean(ref[a:b] ** 2)))
        assert np.sqrt(np.mean((w[a:b] - ref[a:b]) ** 2)) < 4 * TOL * scale, i


@pytest.fixture(scope="module")
def flagged_iqu():
    p = tiny_IQU(seed=95, n_per_det=7001, n_lags=300, n_ivl_lo=200, n_ivl_hi=5000, flag_frac=0.02)
    return p, system_for(p)


@pytest.mark.parametrize("prec", ["fp32", "fp64", "df64"])
@pytest.mark.parametrize("lg", range(10, 19))
@pytest.mark.parametrize("runs", [-1, 1])
def test_operator_matches_oracle(flagged_iqu, lg, runs, prec):
    import torch
    p, S = flagged_iqu
    if runs == 1 and prec != "fp32":
        pytest.skip("run sums are float32")
    plan = make_plan(p, fft_len=1 << lg, scatter_runs=runs)
    x = np.random.default_rng(lg).standard_normal((S.n_obs, 3)).astype(np.float32)
    x[S.excised] = 0.0
    y = host(plan.apply_ATNA(cuda(x, torch.float32 if prec == "fp32" else torch.float64), precision=prec))[0]
    assert rel_rms(y, S.H(x.astype(np.float64))) < 2 * TOLS[prec]   # two weights and a sum more per sample
    b = host(plan.rhs(cuda(p.d), precision=prec))[0]
    assert rel_rms(b, S.rhs(p.d[0])) < 2 * TOLS[prec]


@pytest.mark.parametrize("width", [64, 65, 128, 129])
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_solve_around_the_cluster_kernel_s_map_sizes(width, prec):
    """4096 rows fill its smaller form, 16384 its larger one; 129 x 129 rows run the
    three vector kernels.  The same iterations give the oracle's map."""
    p = tiny_T(seed=150 + width, n=6 * width * width, width=width, n_lags=8, ivls=(2 * width * width, 4 * width * width))
    S = system_for(p)
    plan = make_plan(p)
    m, info = plan.solve(cuda(p.d[0]), precision=prec, rel_tol=1e-11, max_iter=200)
    x, _ = S.solve(p.d[0], rel_tol=1e-13, max_iter=400)
    assert info["status"] == 0 and rel_rms(host(m), x) < 1e-9
    capped, i4 = plan.solve(cuda(p.d[0]), precision=prec, rel_tol=1e-30, max_iter=4)
    assert i4["iters"] == 4 and i4["status"] == 1
    two, infos = plan.solve_batched(cuda(np.concatenate([p.d, 2 * p.d])), precision=prec, rel_tol=1e-11, max_iter=200)
    assert rel_rms(host(two[1]), 2 * x) < 1e-9 and infos[0]["status"] == 0


@pytest.mark.parametrize("stokes, rows, n_rhs, launches", [
    (1, 4096, 1, 1), (1, 4097, 1, 1), (1, 16384, 1, 1), (1, 16385, 1, 3),
    (1, 4096, 9, 1), (1, 4097, 8, 1), (1, 4097, 9, 3), (1, 12288, 9, 3), (1, 12289, 9, 1),
    (3, 4096, 1, 1), (3, 4096, 9, 1), (3, 4097, 1, 3), (3, 16384, 1, 3)])
def test_vector_kernels_of_an_iteration_by_map_and_batch_size(stokes, rows, n_rhs, launches):
    """Which maps run the cluster kernel (its one launch an iteration or the three of the
    vector kernels, beside the operator's own), and that both reach the map."""
    import torch
    import paper_0906_1775_gb300 as mm
    rng = np.random.default_rng(rows + stokes)
    pix = np.concatenate([np.arange(rows), rng.permutation(rows), rng.permutation(rows), np.arange(rows)]).astype(np.int32)
    n = pix.size
    psi = np.repeat([0.0, 0.8, 1.6, 2.4], rows).astype(np.float32) if stokes == 3 else None
    lags = np.array([[1.0, 0.2, 0.05]])
    plan = mm.Plan(cuda(pix), cuda(psi) if stokes == 3 else None, rows, [0, n], [0], lags, fft_len=1024,
                   tiles_per_chunk=100000)
    assert plan.n_obs == rows and plan.stats["n_excised"] == 0
    d = rng.standard_normal(n).astype(np.float32)
    D = cuda(np.stack([2.0 ** (k % 4) * d for k in range(n_rhs)]).astype(np.float32))
    from oracle.solver import System
    S = System(pix, psi, rows, stokes, np.array([0, n]), np.array([0]), lags)
    x, _ = S.solve(d, rel_tol=1e-13, max_iter=200)

    def solve(iters):
        kw = dict(precision="fp64", rel_tol=0.0, max_iter=iters, use_graph=0, iters_per_sync=1)
        torch.cuda.synchronize()
        before = mm.madmap_kernel_launch_count()
        m = plan.solve(D[0], **kw)[0][None] if n_rhs == 1 else plan.solve_batched(D, **kw)[0]
        return mm.madmap_kernel_launch_count() - before, host(m)

    solve(1)
    # the operator: one launch a chunk of tiles, two windows or right-hand sides a tile
    st = plan.stats
    chunks = -(-(-(-st["n_segments"] * n_rhs // 2)) // st["tiles_per_chunk"])
    assert solve(4)[0] - solve(2)[0] == 2 * (chunks + launches)
    for k, m in enumerate(solve(30)[1]):
        assert rel_rms(m, 2.0 ** (k % 4) * x) < 1e-9


@pytest.mark.parametrize("lg", [13, 14, 15, 16, 17, 18, 19])
def test_lag_gradient_matches_direct_correlation(lg):
    """The backward pass's lag correlation by windowed transforms, on intervals
    shorter than a window, ending in its first sample, and of several windows
    (their number odd, so that one window is alone), against direct sums.

    A lag is an inner product of a = A lambda and a shifted r = d - A m, both
    ways: a relative change of TOL in the norm of either (float32 inputs, one
    float32 transform) moves it by at most 4 TOL |a| |r|."""
    from oracle.adjoint import solve_backward
    n_lags = 257
    M = 1 << lg
    exact = M - 2 * (n_lags - 1) if 14 <= lg <= 18 else (1 << 14) - 2 * (n_lags - 1)
    p = tiny_T(seed=130 + lg, n=3 * exact + 1202, width=24, n_lags=n_lags, ivls=(1, 1200, exact + 1, 2 * exact))
    S = system_for(p)
    plan = make_plan(p, fft_len=M)
    d = cuda(p.d[0])
    m, _ = plan.solve(d, precision="fp64", rel_tol=1e-12, max_iter=1000)
    g = np.random.default_rng(lg).standard_normal(tuple(m.shape))
    _, gl, _ = plan.solve_backward(d, m, cuda(g), precision="fp64", rel_tol=1e-12, max_iter=1000)
    d64 = p.d[0].astype(np.float64)
    _, ogl, _ = solve_backward(S, d64, host(m), g)
    lam, _ = S.pcg(g, rel_tol=1e-13, max_iter=2000)
    scale = np.linalg.norm(S.unpoint(lam)) * np.linalg.norm(d64 - S.unpoint(host(m)))
    assert np.abs(host(gl) - ogl).max() < 4 * TOL * scale, np.abs(host(gl) - ogl).max() / scale


@pytest.mark.parametrize("lens, n_filters, transforms", [
    ((20000, 40000), 1, True),
    ((100,) * 600, 1, False),          # windows of 2^14 points for 100 samples each
    ((1000,) * 300, 300, False),       # a float64 transform for each filter's interval
    ((3000,) * 100, 3, True)])
def test_lag_gradient_by_the_cheaper_way(lens, n_filters, transforms):
    """Transforms or direct sums by their expected time: the transforms' buffers (a
    window pair's 2^15 points or more) show in the plan's device memory; the lags
    match direct sums in 64 bits within the bound above either way."""
    import paper_0906_1775_gb300 as mm
    from oracle.adjoint import solve_backward
    p = tiny_T(seed=131, n=sum(lens), width=16, n_lags=50, ivls=lens)
    p.interval_filter = np.arange(len(lens), dtype=np.int32) % n_filters
    lags = np.repeat(lags_for(p), n_filters, 0)
    S, plan = system_for(p, lags=lags), make_plan(p, lags=lags)
    d = cuda(p.d[0])
    m, _ = plan.solve(d, precision="fp64", rel_tol=1e-12, max_iter=1000)
    g = np.random.default_rng(2).standard_normal(tuple(m.shape))
    plan.solve_backward(d, m, cuda(g), precision="fp64", rel_tol=1e-12, max_iter=1000, want_lags=False)
    before = mm.madmap_plan_get_stats(plan._h)["device_bytes"]
    _, gl, _ = plan.solve_backward(d, m, cuda(g), precision="fp64", rel_tol=1e-12, max_iter=1000)
    grown = mm.madmap_plan_get_stats(plan._h)["device_bytes"] - before
    assert (grown > 8 << 15) == transforms, grown
    d64 = p.d[0].astype(np.float64)
    _, ogl, _ = solve_backward(S, d64, host(m), g)
    lam, _ = S.pcg(g, rel_tol=1e-13, max_iter=2000)
    scale = np.linalg.norm(S.unpoint(lam)) * np.linalg.norm(d64 - S.unpoint(host(m)))
    assert np.abs(host(gl) - ogl).max() < 4 * TOL * scale, np.abs(host(gl) - ogl).max() / scale


@pytest.mark.parametrize("n_lags", [64, 100, 1024])
def test_noise_filters_on_the_device_match_the_host(n_lags):
    """set_noise and noise_vjp against madmap_noise_filter and its chain rule: the
    same sums in float64 with another order, relative to the largest lag."""
    import torch
    import paper_0906_1775_gb300 as mm
    prm = np.array([[1.0, 0.1, 2.0], [0.8, 5.0, 1.3], [1.2, 0.0, 1.0]])
    p = tiny_T(seed=140, n=9000, width=8, n_lags=n_lags, ivls=(3000, 3000, 3000))
    lags = np.stack([mm.noise_filter(n_lags, 100.0, *q) for q in prm])
    args = (cuda(p.pix), None, p.n_pix, p.interval_offsets, [0, 1, 2])
    plan, ref = mm.Plan(*args, np.ones((3, 1)) * (np.arange(n_lags) == 0)), mm.Plan(*args, lags)
    plan.set_noise(100.0, prm)
    y = cuda(np.random.default_rng(0).standard_normal(p.n_samples), torch.float64)
    assert rel_rms(host(plan.apply_ninv(y)), host(ref.apply_ninv(y))) < 1e-13
    g = np.random.default_rng(1).standard_normal((3, n_lags))
    out = plan.noise_vjp(100.0, prm, cuda(g, torch.float64))
    for k in range(3):
        want = mm.madmap_noise_filter_vjp(n_lags, 100.0, *prm[k], g[k])
        assert np.allclose(out[k], want, rtol=1e-11, atol=1e-11 * np.abs(want).max())
    with pytest.raises(mm.MadmapError):
        plan.set_noise(100.0, prm * np.array([-1.0, 1.0, 1.0]))


@pytest.mark.parametrize("prec", ["fp32", "fp64", "df64"])
def test_alignment_takes_no_more_windows(prec):
    """IQU windows start at multiples of 16 samples, but not where an interval would then
    need another window: intervals of one window's most samples, of four and of 60 windows'
    exact ones, and of an odd length (several aligned windows), at odd offsets."""
    import torch
    from synth import make_flat_problem
    n_lags, M = 301, 1 << 14
    exact = M - 2 * (n_lags - 1)
    lens = [3 * exact + 777, M - (n_lags - 1), 4 * exact, 60 * exact]
    p = make_flat_problem("align", 180, 48, 1, sum(lens), 3, n_lags, det_angles_deg=[0.0], hwp_step_deg=22.5,
                          interval_lengths=lambda rng, tot: list(lens), noise=(1.0, 1.0, 1.5))
    plan, S = make_plan(p, fft_len=M), system_for(p)
    assert plan.stats["n_segments"] == 4 + 1 + 4 + 61
    x = np.random.default_rng(3).standard_normal((S.n_obs, 3)).astype(np.float32)
    x[S.excised] = 0.0
    y = host(plan.apply_ATNA(cuda(x, torch.float32 if prec == "fp32" else torch.float64), precision=prec))[0]
    assert rel_rms(y, S.H(x.astype(np.float64))) < 2 * TOLS[prec]
    b = host(plan.rhs(cuda(p.d), precision=prec))[0]
    assert rel_rms(b, S.rhs(p.d[0])) < 2 * TOLS[prec]


@pytest.mark.parametrize("fft_len", [1 << 11, 1 << 13, 1 << 15])
def test_operator_timing_leaves_the_kernels_loading_out(fft_len):
    """In a fresh process the first launch of a kernel loads it, which takes milliseconds
    where the kernels take tens of microseconds: the first timing agrees with the second."""
    import os
    import subprocess
    import sys
    code = f"""
from tests.gpu_helpers import make_plan
from tests.helpers import tiny_IQU
plan = make_plan(tiny_IQU(seed=190, n_per_det=20000, n_lags=40, n_ivl_lo=2000, n_ivl_hi=9000), fft_len={fft_len})
for prec in ("fp32", "fp64", "df64"):
    first, second = (plan.time_operator(prec, reps=2)[0] for _ in range(2))
    assert 0 < sum(first[:3]) < 5 * sum(second[:3]), (prec, first, second)
print("DONE")
"""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    out = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, cwd=root, timeout=300)
    assert "DONE" in out.stdout, out.stdout + out.stderr
