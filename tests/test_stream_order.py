"""Set-up copies and the streams that read them.

A plan's tables, tile lists and work buffers are written while it is set up and
read by kernels on the caller's stream or on the plan's own, which need not be
ordered after the legacy default stream.  A copy from pageable host memory on the
legacy stream may still be in flight when cudaMemcpy returns, so every host to
device copy has to be made on the stream that reads it (or be waited for).  The
race itself cannot be shown by running it; the first test reads the sources, the
second runs every set-up path from a non-blocking stream against the oracle.
"""

from __future__ import annotations

import glob
import os
import re

import numpy as np
import pytest

from tests.helpers import rel_rms, system_for, tiny_IQU

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _sources():
    files = glob.glob(os.path.join(ROOT, "paper_0906_1775_gb300", "csrc", "*.cu*"))
    assert len(files) >= 8
    for f in files:
        yield os.path.basename(f), re.sub(r"//[^\n]*", "", open(f).read())


def test_no_host_to_device_copy_is_left_to_the_legacy_stream():
    for name, src in _sources():
        for m in re.finditer(r"cudaMemcpy\((?:[^()]|\([^()]*\))*\)", src):
            assert "HostToDevice" not in m.group(0), (name, m.group(0))
        # a cudaMemset of device memory returns before it is done: the next statement waits for it
        for m in re.finditer(r"cudaMemset\([^;]*;([^;]*);", src):
            assert "cudaStreamSynchronize" in m.group(1), (name, m.group(0))


@pytest.mark.gpu
@pytest.mark.parametrize("fft_len", [0, 1 << 14, 1 << 17])
def test_plans_set_up_on_a_side_stream_match_the_oracle(fft_len):
    import torch
    from oracle.adjoint import solve_backward
    from tests.gpu_helpers import cuda, host, lib_lags, make_plan
    p = tiny_IQU(seed=61, n_per_det=4000, width=8, n_lags=40, n_ivl_lo=300, n_ivl_hi=2500)
    S = system_for(p)
    x = cuda(np.random.default_rng(1).standard_normal((S.n_obs, 3)), torch.float64)
    d, g = cuda(p.d[0]), cuda(np.random.default_rng(2).standard_normal((S.n_obs, 3)))
    torch.cuda.synchronize()
    kw = dict(precision="fp64", rel_tol=1e-12, max_iter=600)
    with torch.cuda.stream(torch.cuda.Stream()):
        plan = make_plan(p, lags=2 * lib_lags(p), fft_len=fft_len)
        plan.set_filters(lib_lags(p))
        ys = {prec: host(plan.apply_ATNA(x.to(torch.float32) if prec == "fp32" else x, precision=prec))[0]
              for prec in ("fp64", "df64", "fp32")}
        m, _ = plan.solve(d, **kw)
        ms, _ = plan.solve_batched(torch.stack([d, 2 * d, 4 * d]), **kw)   # exact in float32
        gd, gl, _ = plan.solve_backward(d, m, g, **kw)
        m, ms, gd, gl = host(m), host(ms), host(gd), host(gl)
    for prec, y in ys.items():
        ref = S.H(host(x).astype(np.float32).astype(np.float64) if prec == "fp32" else host(x))
        assert rel_rms(y, ref) < (2e-5 if prec == "fp32" else 1e-11), prec
    xo, _ = S.solve(p.d[0], rel_tol=1e-13, max_iter=600)
    assert rel_rms(m, xo) < 1e-10
    for k in range(3):
        assert rel_rms(ms[k], 2.0 ** k * xo) < 1e-10, k
    ogd, ogl, _ = solve_backward(S, p.d[0].astype(np.float64), m, host(g))
    assert rel_rms(gd, ogd) < 2e-5 and rel_rms(gl, ogl) < 2e-5
