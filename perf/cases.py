"""The measured work of the library: what a map-making program calls, and how often-used sizes spread.

Every case is one call (or, for the differentiable solve, one training step) through the public Python
entry points, on a plan that the program built once.  The families are

  ninv      N^-1 y of a timestream                         Plan.apply_ninv
  atna      one operator application A^T N^-1 A x          Plan.apply_ATNA
  rhs       the right-hand side A^T N^-1 d                 Plan.rhs
  solve     the map of one timestream                      Plan.solve
  batch     the maps of several timestreams, one scan      Plan.solve_batched
  train     solve, loss, gradients of d and of the noise   MadmapSolve + autograd

over the scans "flat" (cross-linked raster on a W x W grid, temperature or IQU), "ring" (spinning all-sky
scan on a HEALPix RING grid), "stripe" (the raster with white noise and one offset per baseline, i.e.
destriping) and "bore" (compressed boresight pointing expanded on the fly).
"""

import math

import numpy as np
import torch

import paper_0906_1775_gb300 as mm

DEV = "cuda"


# ----------------------------------------------------------------- the cases
def _case(name, family, scan, precision, n_det, n_per_det, n_side, n_lags, **more):
    c = dict(name=name, family=family, scan=scan, precision=precision, n_det=n_det, n_per_det=n_per_det,
             n_side=n_side, n_lags=n_lags, stokes=3, ivl_lo=0, ivl_hi=0, flagged=0.0, rel_tol=0.0, iters=1,
             n_rhs=1, autotune=False)
    c.update(more)
    return c


def listed():
    return [
        # the smallest call: the weighting of one short scan (a quick look, one subscan), latency only
        _case("ninv-short-f32", "ninv", "flat", "fp32", 1, 5000, 32, 64, stokes=1),
        # one operator application of a single-detector temperature map in double precision
        _case("atna-T-f64", "atna", "flat", "fp64", 1, 1 << 18, 64, 1 << 12, stokes=1),
        # the inner operator of the flat-sky IQU solve: four polarimeters, uneven stationary intervals
        _case("atna-flat-f32", "atna", "flat", "fp32", 4, 1 << 22, 512, 1 << 14, ivl_lo=1 << 16, ivl_hi=1 << 20),
        # the double-float right-hand side of an odd-sized scan with flagged samples
        _case("rhs-odd-df64", "rhs", "flat", "df64", 4, 777777, 301, 5000, ivl_lo=30011, ivl_hi=300007,
              flagged=0.01),
        # the inner operator of the all-sky solve: eight of its detectors, the largest call
        _case("atna-ring-f32", "atna", "ring", "fp32", 8, 1 << 24, 512, 1 << 15, ivl_lo=432000, ivl_hi=648000),
        # a whole double-precision temperature map: a latency-bound iteration
        _case("solve-T-f64", "solve", "flat", "fp64", 1, 1 << 18, 64, 1 << 12, stokes=1, rel_tol=1e-10, iters=16),
        # a whole flat-sky IQU map in mixed precision
        _case("solve-flat-mixed", "solve", "flat", "mixed", 4, 1 << 22, 512, 1 << 14, ivl_lo=1 << 16,
              ivl_hi=1 << 20, rel_tol=1e-8, iters=29),
        # a whole all-sky IQU map in mixed precision on an autotuned plan (four detectors, half the sky's rings)
        _case("solve-ring-mixed", "solve", "ring", "mixed", 4, 1 << 23, 512, 1 << 15, ivl_lo=432000,
              ivl_hi=648000, rel_tol=1e-8, iters=36, autotune=True),
        # noise Monte Carlo: several realisations over one scan, short uneven intervals
        _case("batch-T-mixed", "batch", "flat", "mixed", 1, 2500003, 64, 1 << 12, stokes=1, ivl_lo=1 << 12,
              ivl_hi=1 << 20, rel_tol=1e-8, iters=16, n_rhs=16),
        # one step of fitting the noise model: solve, backward, gradients of the data and of three
        # noise parameters per detector
        _case("train-flat-mixed", "train", "flat", "mixed", 8, 1 << 20, 256, 1 << 12, rel_tol=1e-8, iters=22),
        # destriping: white noise and one offset per baseline, no FFT
        _case("atna-stripe-f32", "atna", "stripe", "fp32", 4, 1 << 22, 512, 1, ivl_lo=6000, ivl_hi=6000),
        # the low-memory mode: pointing expanded from the boresight nodes on the fly
        _case("atna-bore-f32", "atna", "bore", "fp32", 4, 1 << 22, 512, 1 << 14, ivl_lo=1 << 16, ivl_hi=1 << 20),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the same families with sizes over the listed range (odd ones as they come)."""
    kind = rng.choice(["ninv", "atna-T", "atna-flat", "rhs", "atna-ring", "solve-T", "solve-flat", "solve-ring", "batch",
                       "train", "stripe", "bore"])
    if kind == "ninv":
        n = _logint(rng, 2000, 4000000)
        lags = _logint(rng, 16, min(n // 4, 20000))
        c = _case("", "ninv", "flat", rng.choice(["fp32", "fp64"]), 1, n, 64, lags, stokes=1)
    elif kind == "atna-T":
        n = _logint(rng, 1 << 16, 1 << 22)
        c = _case("", "atna", "flat", rng.choice(["fp32", "fp64", "df64"]), 1, n, rng.randint(30, 120),
                  _logint(rng, 100, 10000), stokes=1)
    elif kind in ("atna-flat", "rhs", "bore"):
        n = _logint(rng, 1 << 18, 1 << 22)
        lags = _logint(rng, 1000, 16384)
        w = int(math.sqrt(n / rng.uniform(8, 32)))
        fam, scan = ("rhs", "flat") if kind == "rhs" else ("atna", "bore" if kind == "bore" else "flat")
        c = _case("", fam, scan, "fp32" if kind != "rhs" else rng.choice(["fp32", "df64"]), 4, n, w, lags,
                  ivl_lo=4 * lags, ivl_hi=64 * lags, flagged=rng.choice([0.0, 0.01]) if scan == "flat" else 0.0)
    elif kind == "atna-ring":
        c = _case("", "atna", "ring", "fp32", 4, _logint(rng, 1 << 21, 1 << 24), rng.choice([128, 256, 512]),
                  _logint(rng, 8000, 32768), ivl_lo=300000, ivl_hi=648000)
    elif kind == "solve-T":
        n = _logint(rng, 1 << 16, 1 << 20)
        c = _case("", "solve", "flat", rng.choice(["fp64", "mixed"]), 1, n, rng.randint(30, 64),
                  _logint(rng, 500, 5000), stokes=1, rel_tol=1e-10, iters=16)
    elif kind == "solve-flat":
        n = _logint(rng, 1 << 18, 1 << 21)
        lags = _logint(rng, 1000, 16384)
        c = _case("", "solve", "flat", "mixed", 4, n, int(math.sqrt(n / rng.uniform(12, 32))), lags,
                  ivl_lo=4 * lags, ivl_hi=64 * lags, rel_tol=1e-8, iters=29)
    elif kind == "solve-ring":
        c = _case("", "solve", "ring", "mixed", 4, _logint(rng, 1 << 21, 1 << 22), rng.choice([128, 256]),
                  _logint(rng, 8000, 32768), ivl_lo=300000, ivl_hi=648000, rel_tol=1e-8, iters=36)
    elif kind == "batch":
        c = _case("", "batch", "flat", "mixed", 1, _logint(rng, 1 << 18, 1 << 21), rng.randint(30, 64), 1 << 12,
                  stokes=1, ivl_lo=1 << 12, ivl_hi=1 << 19, rel_tol=1e-8, iters=16, n_rhs=rng.randint(2, 16))
    elif kind == "train":
        n = _logint(rng, 1 << 17, 1 << 20)
        c = _case("", "train", "flat", "mixed", 4, n, int(math.sqrt(n / 16)), rng.choice([1 << 10, 1 << 11, 1 << 12]),
                  rel_tol=1e-8, iters=22)
    else:
        n = _logint(rng, 1 << 18, 1 << 22)
        base = rng.randint(500, 10000)
        c = _case("", "atna", "stripe", "fp32", 4, n, int(math.sqrt(n / rng.uniform(8, 32))), 1, ivl_lo=base,
                  ivl_hi=base)
    del c["name"]
    return c


# ----------------------------------------------------------------- scans
def _raster(c, g):
    """Pixels of one detector on the alternating raster (one sample per pixel step, jitter 0.3 pixel), and sweeps."""
    w, n = c["n_side"], c["n_per_det"]
    k = torch.arange(n, device=DEV)
    sweep, step = k // (w * w), k % (w * w)
    line, pos = step // w, step % w
    pos = torch.where(line % 2 == 0, pos, w - 1 - pos)
    horiz = sweep % 2 == 0
    jit = 0.3 * torch.randn((2, n), generator=g, device=DEV)
    r = torch.where(horiz, line, pos) + torch.floor(0.5 + jit[0]).to(torch.int64)
    q = torch.where(horiz, pos, line) + torch.floor(0.5 + jit[1]).to(torch.int64)
    return (r.clamp(0, w - 1) * w + q.clamp(0, w - 1)).to(torch.int32), sweep


def _healpix_ring(N, z, phi):
    """RING pixel of directions (z, phi) on the HEALPix grid of side N (Gorski et al. 2005)."""
    za = z.abs()
    tt = torch.remainder(phi / (math.pi / 2), 4.0)
    # equatorial belt
    a, b = N * (0.5 + tt), N * z * 0.75
    jp, jm = torch.floor(a - b).to(torch.int64), torch.floor(a + b).to(torch.int64)
    ir = N + 1 + jp - jm
    ks = 1 - (ir & 1)
    ip = torch.remainder(torch.div(jp + jm - N + ks + 1, 2, rounding_mode="floor"), 4 * N)
    eq = 2 * N * (N - 1) + (ir - 1) * 4 * N + ip
    # polar caps
    tp = tt - torch.floor(tt)
    t = N * torch.sqrt((3.0 * (1.0 - za)).clamp(min=0.0))
    jp, jm = torch.floor(tp * t).to(torch.int64), torch.floor((1.0 - tp) * t).to(torch.int64)
    ir = jp + jm + 1
    ip = torch.remainder(torch.floor(tt * ir).to(torch.int64), 4 * ir)
    cap = torch.where(z > 0, 2 * ir * (ir - 1) + ip, 12 * N * N - 2 * ir * (ir + 1) + ip)
    return torch.where(za <= 2.0 / 3.0, eq, cap).to(torch.int32)


def _ring(c, det, lam0):
    """Pixels and polariser angles of one detector: 1 rpm rings of half-angle 85 degrees at 180 Hz, the spin axis
    stepping 2.5 arcmin per ring; quadruples of detectors share a focal-plane offset and look at 0/45/90/135 degrees."""
    k = torch.arange(c["n_per_det"], dtype=torch.float64, device=DEV)
    ring = torch.floor(k / 10800)
    lam = lam0 + ring * math.radians(2.5 / 60)
    om = (k - ring * 10800) * (2 * math.pi / 10800)
    off = math.radians(0.25 * (det // 4))
    ca, sa = math.cos(math.radians(85) + off), math.sin(math.radians(85) + off)
    cl, sl, co, so = torch.cos(lam), torch.sin(lam), torch.cos(om), torch.sin(om)
    nx, ny, nz = ca * cl + sa * so * sl, ca * sl - sa * so * cl, sa * co
    vx, vy, vz = co * sl, -co * cl, -so
    north = -nz * (nx * vx + ny * vy) + (1 - nz * nz) * vz
    east = -ny * vx + nx * vy
    psi = torch.remainder(torch.atan2(east, north) + math.radians(45 * (det % 4)), math.pi)
    return _healpix_ring(c["n_side"], nz.clamp(-1, 1), torch.atan2(ny, nx)), psi.to(torch.float32)


def _boresight(c):
    """Nodes every 32 samples of a raster that overshoots the grid by one node interval at each end of a line; the
    focal plane turns once in 100,003 samples."""
    w, step, n = c["n_side"], 32, c["n_per_det"]
    length = ((w + 2 * step) // step + 1) * step        # samples per line
    u = np.arange((n - 1) // step + 2, dtype=np.int64) * step
    line, pos = u // length, (u % length).astype(np.float64) - step
    sweep = line // w
    pos = np.where(line % 2 == 0, pos, length - 2 * step - 1 - pos)
    cross = (line % w) + 0.5
    x, y = np.where(sweep % 2 == 0, pos, cross), np.where(sweep % 2 == 0, cross, pos)
    a = 2 * math.pi * u / 100003.0
    return torch.from_numpy(np.stack([x, y, np.cos(a), np.sin(a)], 1).astype(np.float32)).to(DEV), step


def _intervals(c, rng):
    """Offsets and filters: each detector cut into stationary intervals, one filter per detector (ring: one in all)."""
    lens, filt = [], []
    for det in range(c["n_det"]):
        left = c["n_per_det"]
        while left > 0:
            n = left if not c["ivl_lo"] else min(left, int(round(math.exp(rng.uniform(math.log(c["ivl_lo"]),
                                                                                      math.log(c["ivl_hi"]))))))
            if c["scan"] == "stripe":
                n = left                                # white noise: the offsets carry the correlations
            lens.append(n)
            filt.append(0 if c["scan"] == "ring" else det)
            left -= n
    return np.concatenate([[0], np.cumsum(lens)]).astype(np.int64), np.asarray(filt, dtype=np.int32)


def _noise(c, rng):
    """(sigma, f_knee, alpha) per filter and the sampling rate."""
    if c["scan"] == "ring":
        return np.array([[1.0, 0.03, 1.7]]), 180.0
    n = c["n_det"]
    return np.stack([rng.uniform(0.8, 1.2, n), rng.uniform(0.05, 0.2, n), rng.uniform(1.0, 2.0, n)], 1), 100.0


def _sky(n_rows, stokes, g, dtype):
    """Map values of unit intensity and a tenth of it in polarisation."""
    return (torch.randn((n_rows, stokes), generator=g, device=DEV, dtype=torch.float64)
            * torch.tensor([1.0, 0.1, 0.1][:stokes], device=DEV, dtype=torch.float64)).to(dtype)


def _inputs(case, seed):
    """Scan, noise and data from the seed alone (no library call)."""
    c = dict(_case("", "", "", "", 0, 0, 0, 0), **case)
    rng = np.random.default_rng(seed)
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    s = dict(case=c, fs=100.0)
    s["off"], s["filt"] = _intervals(c, rng)
    s["params"], s["fs"] = _noise(c, rng)
    n_t = c["n_det"] * c["n_per_det"]
    if c["scan"] == "bore":
        s["bore"], s["step"] = _boresight(c)
        ang = np.radians(45.0 * np.arange(c["n_det"]))
        s["det"] = np.stack([rng.uniform(-1, 1, c["n_det"]), rng.uniform(-1, 1, c["n_det"]), np.cos(ang),
                             np.sin(ang)], 1).astype(np.float32)
        s["n_pix"] = c["n_side"] ** 2
    else:
        pix, psi = [], []
        lam0 = 0.3                                      # the same rings, so the same observed pixels, for any seed
        for det in range(c["n_det"]):
            if c["scan"] == "ring":
                p, a = _ring(c, det, lam0)
                psi.append(a)
            else:
                p, sweep = _raster(c, g)
                psi.append(torch.remainder(math.radians(45.0 * det) + 2 * math.radians(22.5) * sweep.to(torch.float64),
                                           math.pi).to(torch.float32))
            pix.append(p)
        s["pix"] = torch.cat(pix)
        s["psi"] = torch.cat(psi) if c["stokes"] == 3 else None
        if c["flagged"] > 0:
            s["pix"][torch.rand(n_t, generator=g, device=DEV) < c["flagged"]] = -1
        s["n_pix"] = 12 * c["n_side"] ** 2 if c["scan"] == "ring" else c["n_side"] ** 2
        if c["scan"] == "stripe":
            t = torch.arange(c["n_per_det"], device=DEV) // c["ivl_lo"]
            per = int(t[-1]) + 1
            s["extra"] = (t.repeat(c["n_det"]) + per * torch.arange(c["n_det"], device=DEV)
                          .repeat_interleave(c["n_per_det"])).to(torch.int32)
            s["n_extra"] = per * c["n_det"]
    if c["family"] in ("ninv", "rhs", "solve", "batch", "train"):
        # signal of a random sky plus 1/f noise per detector
        nd, n = c["n_det"], c["n_per_det"]
        nu = torch.fft.rfftfreq(n, d=1.0 / s["fs"], device=DEV, dtype=torch.float64)
        nu[0] = nu[1]
        sky = _sky(s["n_pix"], c["stokes"], g, torch.float64)
        d = torch.empty((c["n_rhs"], nd * n), dtype=torch.float32, device=DEV)
        for det in range(nd):
            a, b = det * n, (det + 1) * n
            p = s["pix"][a:b].clamp(min=0).to(torch.int64)
            sig = sky[p, 0]
            if c["stokes"] == 3:
                two = 2 * s["psi"][a:b].to(torch.float64)
                sig = sig + sky[p, 1] * torch.cos(two) + sky[p, 2] * torch.sin(two)
            sg, fk, al = s["params"][0 if c["scan"] == "ring" else det]
            amp = sg * torch.sqrt(1 + (fk / nu) ** al)
            for r in range(c["n_rhs"]):
                w = torch.randn(n, generator=g, device=DEV, dtype=torch.float64)
                d[r, a:b] = (sig + torch.fft.irfft(torch.fft.rfft(w) * amp, n=n)).to(torch.float32)
        s["d"] = d
        if c["family"] == "ninv":
            s["y"] = d[0].to(torch.float64 if c["precision"] == "fp64" else torch.float32)
    s["g"] = g
    return s


def _map_input(s, n_rows):
    c = s["case"]
    return _sky(n_rows, c["stokes"], s["g"], torch.float32 if c["precision"] == "fp32" else torch.float64)


def _loss_target(s, n_rows):
    return _sky(n_rows, s["case"]["stokes"], s["g"], torch.float64)


def prepare(case, seed):
    s = _inputs(case, seed)
    c = s["case"]
    lags = np.stack([mm.noise_filter(c["n_lags"], s["fs"], *p) for p in s["params"]])
    if c["scan"] == "bore":
        s["plan"] = mm.Plan.from_boresight(s["bore"], s["step"], s["det"], c["n_per_det"], c["n_side"], c["n_side"], True,
                                           s["off"], s["filt"], lags)
    elif c["scan"] == "stripe":
        s["plan"] = mm.Plan(s["pix"], s["psi"], s["n_pix"], s["off"], s["filt"], lags, extra_index=s["extra"],
                            n_extra=s["n_extra"])
    else:
        s["plan"] = mm.Plan(s["pix"], s["psi"], s["n_pix"], s["off"], s["filt"], lags, autotune=c["autotune"])
    if c["family"] == "atna":
        s["x"] = _map_input(s, s["plan"].n_obs)
    if c["family"] == "train":
        s["target"] = _loss_target(s, s["plan"].n_obs)
        s["data"] = s["d"][0].clone().requires_grad_(True)
        s["noise"] = torch.from_numpy(s["params"]).requires_grad_(True)
    return s


def run(s):
    c, plan = s["case"], s["plan"]
    if c["family"] == "ninv":
        return plan.apply_ninv(s["y"], precision=c["precision"])
    if c["family"] == "atna":
        return plan.apply_ATNA(s["x"], precision=c["precision"])
    if c["family"] == "rhs":
        return plan.rhs(s["d"], precision=c["precision"])
    kw = dict(precision=c["precision"], rel_tol=c["rel_tol"], max_iter=500)
    if c["family"] == "solve":
        return plan.solve(s["d"][0], **kw)[0]
    if c["family"] == "batch":
        return plan.solve_batched(s["d"], **kw)[0]
    m = mm.MadmapSolve.apply(s["data"], s["noise"], plan, s["fs"], kw)
    loss = ((m - s["target"]) ** 2).sum()
    gd, gp = torch.autograd.grad(loss, [s["data"], s["noise"]])
    return {"map": m.detach(), "grad_d": gd, "grad_noise": gp}


# ----------------------------------------------------------------- what a pass cannot do without
def work(case):
    c = dict(_case("", "", "", "", 0, 0, 0, 0), **case)
    n = float(c["n_det"] * c["n_per_det"])
    es = {"fp32": 4, "mixed": 4, "df64": 8, "fp64": 8}[c["precision"]]
    pointing = (8.0 if c["stokes"] == 3 else 4.0) * n
    if c["scan"] == "stripe":
        pointing += 4.0 * n
    if c["scan"] == "bore":
        pointing = 16.0 * c["n_per_det"] / 32
    pixels = 12.0 * c["n_side"] ** 2 if c["scan"] == "ring" else float(c["n_side"]) ** 2
    maps = pixels * c["stokes"] * es
    # forward and inverse real transforms of four filter lengths (half of each is output), the filter, the pointing
    fft = 2 * 2 * 2.5 * math.log2(4 * c["n_lags"]) + 4 if c["n_lags"] > 1 else 1.0
    op = n * (fft + (10.0 if c["stokes"] == 3 else 2.0))
    if c["family"] == "ninv":
        return {"bytes": 2 * es * n, "flops": n * fft}
    if c["family"] == "atna":
        return {"bytes": pointing + 2 * maps, "flops": op}
    if c["family"] == "rhs":
        return {"bytes": pointing + 4 * n + maps, "flops": op}
    # one operator application per iteration (the scan is larger than the cache) and the data once
    its = c["iters"] * (2 if c["family"] == "train" else 1)
    r = c["n_rhs"]
    return {"bytes": its * (pointing + 2 * maps * r) + 4 * n * r + 8 * pixels * c["stokes"] * r + (4 * n if its > c["iters"] else 0),
            "flops": its * op * r}


def tolerance(case):
    """About four times what runs differ from 64 bits by."""
    fam, prec = case["family"], case["precision"]
    if fam in ("ninv", "atna", "rhs"):
        if prec == "fp64":
            return {"rel": 1e-14, "max": 1e-13}     # 4e-16: float64 sums and transforms in any order
        if prec == "df64":
            return {"rel": 5e-13, "max": 2e-11}     # 4e-14: 48-bit sums and products
        return {"rel": 3e-6, "max": 1e-4}           # 3e-7 to 6e-7: float32 sums and transforms in any order
    if prec == "fp64":
        return {"rel": 1e-9, "max": 1e-8}           # 1e-10: where the stopping rule ends
    if fam == "train":
        return {"rel": 3e-6, "max": 1e-4}           # 5e-7: float32 gradients of the data
    return {"rel": 1e-6, "max": 2e-5}               # 4e-8 to 2e-7: where the stopping rule ends, an iteration apart


# ----------------------------------------------------------------- the same in 64 bits with plain torch
def _lags64(c, params, fs):
    """The band-limited inverse noise filter: inverse DFT of 1 / PSD at 4 n_lags points, triangular taper."""
    L = 4 * c["n_lags"]
    j = torch.arange(L, device=DEV, dtype=torch.float64)
    nu = torch.minimum(j, L - j) * fs / L
    nu[0] = nu[1]
    q = 1 / (params[:, 0:1] ** 2 * (1 + (params[:, 1:2] / nu) ** params[:, 2:3]))
    t = torch.arange(c["n_lags"], device=DEV, dtype=torch.float64)
    return torch.fft.ifft(q, dim=1).real[:, : c["n_lags"]] * (1 - t / c["n_lags"])


class _Exact:
    """A, A^T and N^-1 of the inputs `s` in float64 torch."""

    def __init__(self, s):
        self.s, c = s, s["case"]
        self.c, self.ns = c, c["stokes"]
        w = None
        if c["scan"] == "bore":
            pix, c2, s2 = self._expand()
            w = (c2, s2)
        else:
            pix = s["pix"].to(torch.int64)
            if self.ns == 3:
                two = 2 * s["psi"].to(torch.float64)
                w = (torch.cos(two), torch.sin(two))
        obs = torch.zeros(s["n_pix"], dtype=torch.bool, device=DEV)
        obs[pix[pix >= 0]] = True
        g2o = torch.cumsum(obs.to(torch.int64), 0) - 1
        self.n_sky = int(obs.sum())
        self.ok = pix >= 0
        self.row = torch.where(self.ok, g2o[pix.clamp(min=0)], torch.zeros_like(pix))
        self.w = w
        self.n_rows = self.n_sky + s.get("n_extra", 0)
        self.lags = _lags64(c, torch.from_numpy(s["params"]).to(DEV), s["fs"])

    def _expand(self):
        s, c = self.s, self.c
        j = torch.arange(c["n_per_det"], device=DEV)
        u = j // s["step"]
        f = ((j % s["step"]).to(torch.float32) * (1.0 / s["step"]))[:, None]
        a, b = s["bore"][u], s["bore"][u + 1]
        v = a + f * (b - a)
        x, y, co, si = v.unbind(1)
        pix, c2, s2 = [], [], []
        W = c["n_side"]
        for dx, dy, cd, sd in torch.from_numpy(s["det"]).to(DEV):
            fx, fy = torch.floor(x + (co * dx - si * dy)), torch.floor(y + (si * dx + co * dy))
            C, S = (co * cd - si * sd).to(torch.float64), (si * cd + co * sd).to(torch.float64)
            n = C * C + S * S
            ok = (fx >= 0) & (fx < W) & (fy >= 0) & (fy < W) & (n > 0)
            pix.append(torch.where(ok, fy.to(torch.int64) * W + fx.to(torch.int64), -torch.ones_like(u)))
            c2.append((C * C - S * S) / n)
            s2.append(2 * C * S / n)
        return torch.cat(pix), torch.cat(c2), torch.cat(s2)

    def A(self, x):
        x = x.reshape(self.n_rows, self.ns).to(torch.float64)
        y = x[self.row, 0]
        if self.ns == 3:
            y = y + x[self.row, 1] * self.w[0] + x[self.row, 2] * self.w[1]
        if "extra" in self.s:
            y = y + x[self.n_sky + self.s["extra"].to(torch.int64), 0]
        return torch.where(self.ok, y, torch.zeros_like(y))

    def At(self, y):
        y = torch.where(self.ok, y, torch.zeros_like(y))
        out = torch.zeros((self.n_rows, self.ns), dtype=torch.float64, device=DEV)
        out[:, 0].index_add_(0, self.row, y)
        if self.ns == 3:
            out[:, 1].index_add_(0, self.row, y * self.w[0])
            out[:, 2].index_add_(0, self.row, y * self.w[1])
        if "extra" in self.s:
            out[:, 0].index_add_(0, self.n_sky + self.s["extra"].to(torch.int64), y)
        return out

    def Ninv(self, y, lags=None):
        lags = self.lags if lags is None else lags
        off, filt, parts = self.s["off"], self.s["filt"], []
        for i in range(len(filt)):
            a, b, f = int(off[i]), int(off[i + 1]), lags[int(filt[i])]
            if len(f) == 1:
                parts.append(y[a:b] * f[0])
                continue
            n = b - a
            L = 1 << (n + len(f) - 1).bit_length()
            m = min(len(f), n)
            k = torch.cat([f[:m], torch.zeros(L - 2 * m + 1, dtype=f.dtype, device=DEV), f[1:m].flip(0)])
            parts.append(torch.fft.irfft(torch.fft.rfft(y[a:b], n=L) * torch.fft.rfft(k), n=L)[:n])
        return torch.cat(parts)

    def solve(self, b):
        """H x = b by block-Jacobi PCG, far below the tested tolerances."""
        f0 = self.lags[:, 0][torch.from_numpy(np.repeat(self.s["filt"], np.diff(self.s["off"])).astype(np.int64)).to(DEV)]
        one = [torch.ones_like(f0)] + (list(self.w) if self.ns == 3 else [])
        B = torch.zeros((self.n_rows, self.ns, self.ns), dtype=torch.float64, device=DEV)
        f0 = torch.where(self.ok, f0, torch.zeros_like(f0))
        for i in range(self.ns):
            for j in range(i, self.ns):
                col = torch.zeros(self.n_rows, dtype=torch.float64, device=DEV).index_add_(0, self.row, f0 * one[i] * one[j])
                B[:, i, j] = B[:, j, i] = col
        P = 1 / B if self.ns == 1 else torch.linalg.inv(B)
        prec = lambda r: torch.einsum("kij,kj->ki", P, r)  # noqa: E731
        x, r = torch.zeros_like(b), b.clone()
        z = prec(r)
        p, rz, b2 = z.clone(), float((r * z).sum()), float((b * b).sum())
        for _ in range(400):
            q = self.At(self.Ninv(self.A(p)))
            alpha = rz / float((p * q).sum())
            x += alpha * p
            r -= alpha * q
            if float((r * r).sum()) <= 1e-26 * b2:
                break
            z = prec(r)
            new = float((r * z).sum())
            p = z + (new / rz) * p
            rz = new
        return x


def exact(case, seed):
    s = _inputs(case, seed)
    c = s["case"]
    E = _Exact(s)
    if c["family"] == "ninv":
        return E.Ninv(s["y"].to(torch.float64))[None]
    if c["family"] == "atna":
        return E.At(E.Ninv(E.A(_map_input(s, E.n_rows))))[None]
    if c["family"] == "rhs":
        return E.At(E.Ninv(s["d"][0].to(torch.float64)))[None]
    maps = [E.solve(E.At(E.Ninv(d.to(torch.float64)))) for d in s["d"]]
    if c["family"] == "solve":
        return maps[0]
    if c["family"] == "batch":
        return torch.stack(maps)
    m = maps[0]
    lam = E.solve(2 * (m - _loss_target(s, E.n_rows)))
    a, r = E.A(lam), s["d"][0].to(torch.float64) - E.A(m)
    prm = torch.from_numpy(s["params"]).to(DEV).requires_grad_(True)
    gp = torch.autograd.grad((a * E.Ninv(r, _lags64(c, prm, s["fs"]))).sum(), prm)[0]
    return {"map": m, "grad_d": E.Ninv(a), "grad_noise": gp}
