// Operator kernels with the transforms in registers (windows of M = 256 N1
// points, N1 = 64 .. 1024; included by operator_kernels.cuh).
//
// The same four-step window transform as k_f1, k_f2 and k_f3, cut so that an
// element crosses shared memory once per column transform and once per row
// transform instead of once per radix-8 pass:
//
//   k_c1  gather + 256-point column FFTs as 16 x 16: a thread holds 16 elements
//         of one column, transforms them, exchanges once, transforms again
//   k_c2  row FFTs, filter, inverse row FFTs as RA x RB (N1 = RA RB) by groups
//         of RB lanes of one warp, RA elements each; no CTA barrier
//   k_c3  inverse column FFTs as k_c1, then the scatter
//
// What bounds them: the L1 data pipe and the latency of pointing -> map loads.
// The radix-8 kernels spent a fifth of their L1 wavefronts on passes through
// shared memory and an eighth on strided twiddle tables built by every CTA;
// here each thread reads two or three 16-byte entries of tables laid out in
// its own access order, and a warp's pointing and scratch rows are 16 samples
// (128 bytes) long instead of 8.  Float32 operator, one launch of each kernel
// on half of 97 tiles of 2^17 (IQU, 512 x 512 raster): columns 67.7 -> 50.2 and
// 61.5 -> 59.1 us, rows 30.9 -> 23.6 us, one application 262 -> 213 us; on 103
// tiles of 2^18 (ring scan, N_side 512): 109 -> 77, 121 -> 112 and 65 -> 47 us,
// 531 -> 412 us (and to 201 and 387 us with the packed sums below).  Sixteen columns a CTA because 256 threads x 16 elements leave
// four CTAs per SM at 64 registers; three CTAs with twice or four times the
// loads in flight per thread measured slower (442 and 468 us on the ring scan),
// and so did loading the pointing one to four batches ahead of the map (373 -> 387
// to 458 us: at 64 registers the loads in flight cost more than they hide).
// The float64-size types run the same kernels on 8 columns, 128 threads and 128
// registers, with twiddles read whole (a product costs more).  Double-float is
// bound by issue, float64 by its pipe, which radix 16 spends 29 operations an
// element on per column transform instead of 32 to 35: 97 tiles of 2^17, columns
// 165 -> 147 and 196 -> 150 us per launch in double-float (one application 884
// -> 770 us), 476 -> 395 and 462 -> 382 us in float64 (2.96 -> 2.78 ms).  Rows of
// 512 and 1024 points of these types stay in shared memory: 32 elements a lane
// leave 8 warps per SM (double-float 129 -> 224 us per launch, float64 672 -> 730).
//
// Shorter windows would leave rows of less than 64 points to groups of fewer
// than 8 lanes (32-byte rows of scratch), longer ones need rows of more than
// 32 x 32: both stay with k_f1, k_f2 and k_f3.
//
// Scratch rows are in natural order of k2 and the spectrum in natural order
// [k2][k1] (bit-reversed in k1 for k_f2's rows).
#pragma once

// Multiplication by exp(-2 pi i k / 32), 0 <= k < 16 (INV: its conjugate); k is
// a compile-time constant after unrolling.
template <bool INV>
__device__ __forceinline__ float2 mul_w32(float2 v, int k) {
  constexpr float h = 0.70710678118654752440f;
  constexpr float cs[16] = {1.0f, 0.98078528040323044913f, 0.92387953251128675613f, 0.83146961230254523708f,
                            h, 0.55557023301960222474f, 0.38268343236508977173f, 0.19509032201612826785f,
                            0.0f, -0.19509032201612826785f, -0.38268343236508977173f, -0.55557023301960222474f,
                            -h, -0.83146961230254523708f, -0.92387953251128675613f, -0.98078528040323044913f};
  constexpr float sn[16] = {0.0f, 0.19509032201612826785f, 0.38268343236508977173f, 0.55557023301960222474f,
                            h, 0.83146961230254523708f, 0.92387953251128675613f, 0.98078528040323044913f,
                            1.0f, 0.98078528040323044913f, 0.92387953251128675613f, 0.83146961230254523708f,
                            h, 0.55557023301960222474f, 0.38268343236508977173f, 0.19509032201612826785f};
  if (k == 0) return v;
  if (k == 8) return INV ? make_float2(-v.y, v.x) : make_float2(v.y, -v.x);
  if (k == 4) return INV ? make_float2((v.x - v.y) * h, (v.x + v.y) * h) : make_float2((v.x + v.y) * h, (v.y - v.x) * h);
  if (k == 12) return INV ? make_float2(-(v.x + v.y) * h, (v.x - v.y) * h) : make_float2((v.y - v.x) * h, -(v.x + v.y) * h);
  const float c = cs[k], s = INV ? -sn[k] : sn[k];
  return make_float2(v.x * c + v.y * s, v.y * c - v.x * s);
}

// The float64-size types: eighths as in the shared-memory passes, else a
// product with the constant.
template <bool INV, typename C>
__device__ __forceinline__ C mul_w32(const C& v, int k) {
  typedef typename RealOf<C>::type R;
  constexpr double cs[16] = {1.0, 0.98078528040323044913, 0.92387953251128675613, 0.83146961230254523708,
                             0.70710678118654752440, 0.55557023301960222474, 0.38268343236508977173,
                             0.19509032201612826785, 0.0, -0.19509032201612826785, -0.38268343236508977173,
                             -0.55557023301960222474, -0.70710678118654752440, -0.83146961230254523708,
                             -0.92387953251128675613, -0.98078528040323044913};
  if (k == 0) return v;
  if (k == 4) return mul_w8<1, INV>(v);
  if (k == 8) return mul_w8<2, INV>(v);
  if (k == 12) return mul_w8<3, INV>(v);
  const C w = make_c<C, R>(R(cs[k]), R(k < 8 ? -cs[8 - k] : -cs[k - 8]));
  return INV ? cmulc(v, w) : cmul(v, w);
}

__device__ __forceinline__ float2 reg_add(float2 a, float2 b) { return add2(a, b); }
__device__ __forceinline__ float2 reg_sub(float2 a, float2 b) { return sub2(a, b); }
template <typename C>
__device__ __forceinline__ C reg_add(const C& a, const C& b) { return cadd(a, b); }
template <typename C>
__device__ __forceinline__ C reg_sub(const C& a, const C& b) { return csub(a, b); }

// 2^LG-point DFT (INV: inverse, unnormalised) of registers, natural order in,
// bit-reversed order out: radix-2 decimation in frequency, constant twiddles.
// Complex sums are one packed instruction each (add2, sub2): the row kernel
// issued on 69% of its cycles and half of its instructions were these (ring
// scan, 2^18: rows 46.7 -> 42.5, inverse columns 113 -> 103 us per launch, one
// application 416 -> 387 us).
template <int LG, bool INV, typename C>
__device__ __forceinline__ void reg_dft(C (&v)[1 << LG]) {
#pragma unroll
  for (int st = 0; st < LG; ++st) {
    const int span = 1 << (LG - 1 - st);
#pragma unroll
    for (int m = 0; m < (1 << LG); ++m) {
      if ((m & span) == 0) {
        const C x = v[m], y = v[m + span];
        v[m] = reg_add(x, y);
        v[m + span] = mul_w32<INV>(reg_sub(x, y), ((m & (span - 1)) << st) << (5 - LG));
      }
    }
  }
}
template <int LG>
__host__ __device__ constexpr int brev_lg(int m) {
  int r = 0;
  for (int b = 0; b < LG; ++b) r |= ((m >> b) & 1) << (LG - 1 - b);
  return r;
}

// Powers w^m, m < 2^LG, of a group's twiddle from w, w^2, w^4, w^8 (and w^16),
// each rounded once from its exact value: lo[m & 3] times mid[m >> 2], at most
// three products deep.
template <int LG>
struct Powers {
  static constexpr int NM = (1 << LG) / 4;
  float2 lo[4], mid[NM];
  __device__ __forceinline__ explicit Powers(const float4* __restrict__ b) {
    const float4 b0 = __ldg(b);
    lo[1] = make_float2(b0.x, b0.y);
    lo[2] = make_float2(b0.z, b0.w);
    lo[3] = cmul(lo[1], lo[2]);
    if constexpr (LG > 2) {
      const float4 b1 = __ldg(b + 1);
      mid[1] = make_float2(b1.x, b1.y);
      if constexpr (LG > 3) {
        mid[2] = make_float2(b1.z, b1.w);
        mid[3] = cmul(mid[1], mid[2]);
      }
      if constexpr (LG > 4) {
        const float4 b2 = __ldg(b + 2);
        mid[4] = make_float2(b2.x, b2.y);
#pragma unroll
        for (int k = 5; k < 8; ++k) mid[k] = cmul(mid[k - 4], mid[4]);
      }
    }
  }
  __device__ __forceinline__ float2 operator()(int m) const {  // m >= 1, compile-time after unrolling
    return (m & 3) == 0 ? mid[m >> 2] : (m >> 2) == 0 ? lo[m] : cmul(mid[m >> 2], lo[m & 3]);
  }
};

// Columns per CTA of k_c1 and k_c3 (16 threads x 16 elements a column): 16 in
// float32, at 64 registers and four CTAs per SM; 8 for the float64-size types,
// at 128 registers and four CTAs of 128 threads.
template <typename Real>
__host__ __device__ constexpr int reg_cols() {
  return sizeof(Real) == 4 ? 16 : 8;
}
constexpr int REG_CTAS = 4;
// Samples of each lane in flight per thread in the gather and the scatter (64
// registers in float32, 128 in the others).
template <typename Real>
__host__ __device__ constexpr int reg_batch() {
  return sizeof(Real) == 4 ? 2 : 4;
}

// Twiddles of the float64-size types, read whole (a product costs more than
// the read): entries of the plan's wide tables (wide_four), or of the float32 powers.
template <typename Real>
struct ColTwiddle {   // w^m = exp(-2 pi i j m / 256)
  typedef typename CxT<Real>::type C;
  const C* t;
  __device__ __forceinline__ ColTwiddle(const OpArgs& a, int j) : t(static_cast<const C*>(a.reg_wide) + j) {}
  __device__ __forceinline__ C operator()(int m) const { return t[16 * m]; }
};
template <>
struct ColTwiddle<float> : Powers<4> {
  __device__ __forceinline__ ColTwiddle(const OpArgs& a, int j) : Powers<4>(a.reg_col + 2 * j) {}
};
template <typename Real>
struct FourTwiddle {  // exp(-2 pi i n1 (p + 16 b) / M) by b
  typedef typename CxT<Real>::type C;
  const C* t;
  int logN1;
  __device__ __forceinline__ FourTwiddle(const OpArgs& a, int n1, int p) : logN1(a.reg_logN1) {
    t = static_cast<const C*>(a.reg_wide) + wide_four(logN1) + (p << logN1) + n1;
  }
  __device__ __forceinline__ C operator()(int b) const { return t[(long long)(16 * b) << logN1]; }
};
template <>
struct FourTwiddle<float> {
  const float2 w0;
  const Powers<4> w;
  __device__ __forceinline__ FourTwiddle(const OpArgs& a, int n1, int p)
      : w0(__ldg(a.reg_four0 + (p << a.reg_logN1) + n1)), w(a.reg_four + 2 * n1) {}
  __device__ __forceinline__ float2 operator()(int b) const { return b == 0 ? w0 : cmul(w0, w(b)); }
};

// ---------------------------------------------------------------- k_c1
// Thread (column c, group j): elements n2 = j + 16 u (u = 0 .. 15) of column n1.
// 256 = 16 x 16: X[k2 = p + 16 b] = sum_j W16^(j b) W256^(j p) sum_u x[j + 16 u] W16^(u p).
template <typename Real, int NS, int IN, int COLS>
__global__ void __launch_bounds__(16 * COLS, REG_CTAS * reg_cols<Real>() / COLS) k_c1(OpArgs a) {
  typedef typename CxT<Real>::type C;
  const Tile* T = a.tiles + a.tile0 + blockIdx.y;
  if (skip_tile(a, T)) return;
  __shared__ C buf[256 * COLS];
  const int c = threadIdx.x & (COLS - 1), j = threadIdx.x / COLS;
  const int n1 = blockIdx.x * COLS + c, logN1 = a.reg_logN1;
  LaneView<Real> L[2];
  L[0] = lane_view<Real, IN, OUT_MAP>(a, T->l[0]);
  L[1] = lane_view<Real, IN, OUT_MAP>(a, T->l[1]);
  constexpr int U = gathers(IN) ? reg_batch<Real>() : (sizeof(Real) == 4 ? 8 : 4);
  C v[16];
#pragma unroll
  for (int b = 0; b < 16 / U; ++b) {
    int nn[U];
    Real x[2][U];
#pragma unroll
    for (int k = 0; k < U; ++k) nn[k] = n1 + ((j + 16 * (U * b + k)) << logN1);
    gather_samples<Real, NS, IN, U>(a, L, nn, x);
#pragma unroll
    for (int k = 0; k < U; ++k) v[U * b + k] = make_c<C, Real>(x[0][k], x[1][k]);
  }
  reg_dft<4, false>(v);
  {
    const ColTwiddle<Real> w(a, j);
#pragma unroll
    for (int m = 0; m < 16; ++m) {
      const int p = brev_lg<4>(m);
      buf[(p * 16 + j) * COLS + c] = p == 0 ? v[m] : cmul(v[m], w(p));
    }
  }
  __syncthreads();
  // thread (c, p = j): all of group p's elements
#pragma unroll
  for (int m = 0; m < 16; ++m) v[m] = buf[(j * 16 + m) * COLS + c];
  reg_dft<4, false>(v);
  C* sc = static_cast<C*>(a.scratch) + (long long)blockIdx.y * a.M + n1;
  const FourTwiddle<Real> w(a, n1, j);
#pragma unroll
  for (int m = 0; m < 16; ++m) {
    const int b = brev_lg<4>(m);
    sc[(long long)(j + 16 * b) << logN1] = cmul(v[m], w(b));
  }
}

// ---------------------------------------------------------------- k_c2
// Rows of N1 = RA RB points: a group of RB lanes holds one row, lane l the
// elements l + RB u.  Forward: DFT over u, twiddle W^(l p), exchange, DFT over
// the lanes' index (lane l then holds k1 = p + RA b for p = l + RB q); the
// spectrum; the same steps back.  Exchange rows are padded to an odd stride
// (17 or 33), so both directions touch every bank once per half-warp.
template <int LA, int LB>
struct RowGeom {
  static constexpr int RA = 1 << LA, RB = 1 << LB;
  static constexpr int S = RB == 32 ? 33 : 17;
  static constexpr int ROW = RA * S + ((RB == 8 && (RA * S) % 16 == 0) ? 8 : 0);   // rows of 8 lanes: half the banks apart
  static constexpr int PER_WARP = 32 / RB, ROWS = 4 * PER_WARP;   // rows of a warp, and of four
};
template <typename Real, int LA, int LB>
struct RowTwiddle {   // exp(-2 pi i l m / N1) of lane l, m < RA; Inverse: of exchange row p, m < RB
  typedef typename CxT<Real>::type C;
  const C* t;
  __device__ __forceinline__ RowTwiddle(const OpArgs& a, int l)
      : t(static_cast<const C*>(a.reg_wide) + WIDE_ROW_F + l) {}
  __device__ __forceinline__ C operator()(int m) const { return t[m << LB]; }
  struct Inverse {
    const C* t;
    __device__ __forceinline__ Inverse(const OpArgs& a, int p)
        : t(static_cast<const C*>(a.reg_wide) + wide_row_i(LA + LB) + p) {}
    __device__ __forceinline__ C operator()(int m) const { return t[m << LA]; }
  };
};
template <int LA, int LB>
struct RowTwiddle<float, LA, LB> : Powers<LA> {
  __device__ __forceinline__ RowTwiddle(const OpArgs& a, int l) : Powers<LA>(a.reg_row + 4 * l) {}
  struct Inverse : Powers<LB> {
    __device__ __forceinline__ Inverse(const OpArgs& a, int p) : Powers<LB>(a.reg_row + 4 * p) {}
  };
};
template <typename Real, int LA, int LB, int WARPS>
__global__ void __launch_bounds__(32 * WARPS, (sizeof(Real) == 4 && LA < 5 ? 8 : 4) * 4 / WARPS) k_c2(OpArgs a) {
  typedef typename CxT<Real>::type C;
  typedef RowGeom<LA, LB> G;
  constexpr int RA = G::RA, RB = G::RB, Q = RA / RB, LN = LA + LB, ROWS = WARPS * G::PER_WARP;
  const Tile* T = a.tiles + a.tile0 + blockIdx.y;
  if (skip_tile(a, T)) return;
  __shared__ C buf[ROWS * G::ROW];
  const int l = threadIdx.x & (RB - 1), r = threadIdx.x / RB;
  C* const x = buf + r * G::ROW;
  const int row = blockIdx.x * ROWS + r;
  C* sc = static_cast<C*>(a.scratch) + (long long)blockIdx.y * a.M + ((long long)row << LN) + l;
  const Real* H = static_cast<const Real*>(a.H) + (long long)T->filter * a.M + ((long long)row << LN) + l;
  C v[RA];
#pragma unroll
  for (int u = 0; u < RA; ++u) v[u] = sc[RB * u];
  reg_dft<LA, false>(v);
  {
    const RowTwiddle<Real, LA, LB> w(a, l);
#pragma unroll
    for (int m = 0; m < RA; ++m) {
      const int p = brev_lg<LA>(m);
      x[p * G::S + l] = p == 0 ? v[m] : cmul(v[m], w(p));
    }
  }
  __syncwarp();
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    C z[RB], y[RB];
    Real h[RB];
#pragma unroll
    for (int b = 0; b < RB; ++b) h[b] = H[RB * q + RA * b];
#pragma unroll
    for (int m = 0; m < RB; ++m) z[m] = x[(l + RB * q) * G::S + m];
    reg_dft<LB, false>(z);
#pragma unroll
    for (int m = 0; m < RB; ++m) {
      const int b = brev_lg<LB>(m);
      y[b] = c_scale(z[m], h[b]);
    }
    reg_dft<LB, true>(y);
    const typename RowTwiddle<Real, LA, LB>::Inverse w(a, l + RB * q);
#pragma unroll
    for (int m = 0; m < RB; ++m) {
      const int p = brev_lg<LB>(m);
      x[(l + RB * q) * G::S + p] = p == 0 ? y[m] : cmulc(y[m], w(p));
    }
  }
  __syncwarp();
#pragma unroll
  for (int p = 0; p < RA; ++p) v[p] = x[p * G::S + l];
  reg_dft<LA, true>(v);
#pragma unroll
  for (int m = 0; m < RA; ++m) sc[RB * brev_lg<LA>(m)] = v[m];
}

// ---------------------------------------------------------------- k_c3
// The inverse of k_c1's transform, thread (c, p): k2 = p + 16 b, then thread
// (c, j): n2 = j + 16 u, and the outputs of those samples.
template <typename Real, int NS, int OUT, int COLS>
__global__ void __launch_bounds__(16 * COLS, REG_CTAS * reg_cols<Real>() / COLS) k_c3(OpArgs a) {
  typedef typename CxT<Real>::type C;
  typedef typename OutT<Real>::type Out;
  const Tile* T = a.tiles + a.tile0 + blockIdx.y;
  if (skip_tile(a, T)) return;
  __shared__ C buf[256 * COLS];
  // half-wave-plate sums of the CTA, per tile lane (extended pointing only)
  constexpr bool HWP = extended(NS) && OUT == OUT_MAP;
  __shared__ Out hacc[HWP ? 64 : 1];
  __shared__ int hgrp[2];
  if (HWP) {
    for (int i = threadIdx.x; i < 64; i += 16 * COLS) hacc[i] = 0;
    if (threadIdx.x < 2) hgrp[threadIdx.x] = -1;
  }
  const int c = threadIdx.x & (COLS - 1), j = threadIdx.x / COLS;
  const int n1 = blockIdx.x * COLS + c, logN1 = a.reg_logN1;
  const C* sc = static_cast<const C*>(a.scratch) + (long long)blockIdx.y * a.M + n1;
  C v[16], y[16];
#pragma unroll
  for (int b = 0; b < 16; ++b) v[b] = sc[(long long)(j + 16 * b) << logN1];
  {
    const FourTwiddle<Real> w(a, n1, j);
#pragma unroll
    for (int b = 0; b < 16; ++b) v[b] = cmulc(v[b], w(b));
  }
  reg_dft<4, true>(v);
  {
    const ColTwiddle<Real> w(a, j);
#pragma unroll
    for (int m = 0; m < 16; ++m) {
      const int q = brev_lg<4>(m);
      buf[(j * 16 + q) * COLS + c] = q == 0 ? v[m] : cmulc(v[m], w(q));
    }
  }
  __syncthreads();
#pragma unroll
  for (int p = 0; p < 16; ++p) v[p] = buf[(p * 16 + j) * COLS + c];
  reg_dft<4, true>(v);
#pragma unroll
  for (int m = 0; m < 16; ++m) y[brev_lg<4>(m)] = v[m];
  LaneView<Real> L[2];
  L[0] = lane_view<Real, IN_MAPX, OUT>(a, T->l[0]);
  L[1] = lane_view<Real, IN_MAPX, OUT>(a, T->l[1]);
  constexpr int U = OUT == OUT_MAP ? reg_batch<Real>() : (sizeof(Real) == 4 ? 8 : 4);
#pragma unroll
  for (int b = 0; b < 16 / U; ++b) {
    int nn[U];
    Real val[2][U];
#pragma unroll
    for (int k = 0; k < U; ++k) {
      nn[k] = n1 + ((j + 16 * (U * b + k)) << logN1);
      val[0][k] = c_re(y[U * b + k]);
      val[1][k] = c_im(y[U * b + k]);
    }
    scatter_samples<Real, NS, OUT, U, (sizeof(Real) == 4 ? REG_RUN : 0)>(a, L, nn, val, hacc, hgrp);
  }
  if constexpr (HWP) {
    if (a.hwp_base) {
      __syncthreads();
      for (int l = 0; l < 2; ++l)
        hwp_flush(static_cast<Out*>(L[l].out), map_ns(NS) == 3 ? 4 : 1, hacc + 32 * l, hgrp + l, 1);
    }
  }
}

// ---------------------------------------------------------------- k_xcorr
// Backward pass: row transforms of a window pair's a and r (scratch tiles 2 i
// and 2 i + 1, from k_c1) and their cross spectrum Re(conj(Z_a) Z_r), added in
// float64 to the filter's G [k2][k1].
template <int LA, int LB>
__device__ __forceinline__ void row_forward(const float2* sc, float2* x, const float4* row, int l,
                                            float2 (&z)[1 << LA]) {
  typedef RowGeom<LA, LB> G;
  constexpr int RA = G::RA, RB = G::RB, Q = RA / RB;
  float2 v[RA];
#pragma unroll
  for (int u = 0; u < RA; ++u) v[u] = sc[RB * u];
  reg_dft<LA, false>(v);
  const Powers<LA> w(row + 4 * l);
  __syncwarp();
#pragma unroll
  for (int m = 0; m < RA; ++m) {
    const int p = brev_lg<LA>(m);
    x[p * G::S + l] = p == 0 ? v[m] : cmul(v[m], w(p));
  }
  __syncwarp();
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    float2 t[RB];
#pragma unroll
    for (int m = 0; m < RB; ++m) t[m] = x[(l + RB * q) * G::S + m];
    reg_dft<LB, false>(t);
#pragma unroll
    for (int m = 0; m < RB; ++m) z[q * RB + brev_lg<LB>(m)] = t[m];
  }
}
template <int LA, int LB>
__global__ void __launch_bounds__(128, LA == 5 ? 2 : 4) k_xcorr(OpArgs a, double* G0) {
  typedef RowGeom<LA, LB> G;
  constexpr int RA = G::RA, RB = G::RB, Q = RA / RB, LN = LA + LB;
  __shared__ float2 buf[G::ROWS * G::ROW];
  const int l = threadIdx.x & (RB - 1), r = threadIdx.x / RB;
  const int row = blockIdx.x * G::ROWS + r;
  const int filt = a.tiles[a.tile0 + 2 * blockIdx.y].filter;
  const float2* sc = static_cast<const float2*>(a.scratch) + 2LL * blockIdx.y * a.M + ((long long)row << LN) + l;
  float2 za[RA], zr[RA];
  row_forward<LA, LB>(sc, buf + r * G::ROW, a.reg_row, l, za);
  row_forward<LA, LB>(sc + a.M, buf + r * G::ROW, a.reg_row, l, zr);
  double* g = G0 + (long long)filt * a.M + ((long long)row << LN) + l;
#pragma unroll
  for (int q = 0; q < Q; ++q)
#pragma unroll
    for (int b = 0; b < RB; ++b) {
      const float2 u = za[q * RB + b], v = zr[q * RB + b];
      atomicAdd(g + RB * q + RA * b, widen(u.x) * widen(v.x) + widen(u.y) * widen(v.y));
    }
}

// Row kernels: k_c2, and for rows of 512 and 1024 points of the float64-size
// types (32 elements a lane would not fit the registers) the shared-memory
// k_f2, whose spectrum stays bit-reversed within a row.
template <typename Real, int LA, int LB, int WARPS>
inline void launch_c2(const OpArgs& a, int nt, cudaStream_t s) {
  k_c2<Real, LA, LB, WARPS><<<dim3(256 / (WARPS * RowGeom<LA, LB>::PER_WARP), nt), 32 * WARPS, 0, s>>>(a);
}
// The shared-memory row kernel of the wide types and its shared memory (which is
// opted into ahead of a stream capture).
template <typename Real>
inline madmap_status wide_rows(int logN1, OpKernel& f2, int& B2, size_t& sm) {
  typedef typename CxT<Real>::type C;
  f2 = logN1 == 9 ? k_f2<Real, 9> : k_f2<Real, 10>;
  B2 = std::max(1, elems_per_cta<Real>() >> logN1);
  sm = ((size_t)B2 * lay_rs(sizeof(C), logN1, false) + ((size_t)1 << logN1)) * sizeof(C);
  MM_CUDA(set_smem(f2, sm));
  return MADMAP_OK;
}
template <typename Real, int WARPS>
inline madmap_status launch_rows(OpArgs a, int nt, cudaStream_t s) {
  typedef typename CxT<Real>::type C;
  switch (a.reg_logN1) {
    case 6: launch_c2<Real, 3, 3, WARPS>(a, nt, s); return MADMAP_OK;
    case 7: launch_c2<Real, 4, 3, WARPS>(a, nt, s); return MADMAP_OK;
    case 8: launch_c2<Real, 4, 4, WARPS>(a, nt, s); return MADMAP_OK;
  }
  if constexpr (sizeof(Real) == 4) {
    if (a.reg_logN1 == 9) launch_c2<Real, 5, 4, WARPS>(a, nt, s);
    else launch_c2<Real, 5, 5, WARPS>(a, nt, s);
  } else {
    a.logN1 = a.reg_logN1;
    a.N1 = 1 << a.logN1;
    a.tw = static_cast<const C*>(a.reg_wide) + wide_row(a.logN1);
    a.N2 = 1;                 // stride of the row twiddles
    OpKernel f2;
    size_t sm;
    const madmap_status st = wide_rows<Real>(a.logN1, f2, a.B2, sm);
    if (st != MADMAP_OK) return st;
    f2<<<dim3(REG_N2 / a.B2, nt), OP_THREADS, sm, s>>>(a);
  }
  return MADMAP_OK;
}
// Float64 on the smallest problems: with fewer than two column CTAs per SM the
// launch lasts as long as the SM with the most of them, whose float64 pipe every
// CTA waits for, so both column kernels run 2 columns and the rows one warp a CTA
// (one application, wide against narrow CTAs, at 16, 96, 176 and 344 wide CTAs a
// launch: temperature 62.7 and 56.7, 79.2 and 76.2, 134.8 and 109.1, 258 and 265 us;
// IQU 76.3 and 69.5, 93.6 and 87.5, 149 and 124, 286 and 301 us; from 350 on, 1 to
// 5% the other way, for coalescing).
template <typename Real, int NS>
constexpr bool narrow_ctas() {
  return std::is_same<Real, double>::value && (NS == 1 || NS == 3);
}
// The kernels of a plan with register transforms, and their grids for nt tiles
// (nt = 0 only prepares them).
template <typename Real, int NS, int IN, int OUT>
inline madmap_status launch_reg(const OpArgs& a, int nt, cudaStream_t s, cudaEvent_t* ev, int* ei) {
  constexpr int COLS = reg_cols<Real>();
  const int N1 = 1 << a.reg_logN1;
  bool narrow = false;
  if constexpr (narrow_ctas<Real, NS>()) narrow = (long long)(N1 / COLS) * nt < 2 * 152;
  if (ev) cudaEventRecord(ev[(*ei)++], s);
  if constexpr (narrow_ctas<Real, NS>()) {
    if (narrow) k_c1<Real, NS, IN, 2><<<dim3(N1 / 2, nt), 32, 0, s>>>(a);
  }
  if (!narrow) k_c1<Real, NS, IN, COLS><<<dim3(N1 / COLS, nt), 16 * COLS, 0, s>>>(a);
  if (ev) cudaEventRecord(ev[(*ei)++], s);
  madmap_status st = MADMAP_OK;
  if constexpr (narrow_ctas<Real, NS>()) {
    if (narrow) st = launch_rows<Real, 1>(a, nt, s);
  }
  if (!narrow) st = launch_rows<Real, 4>(a, nt, s);
  if (st != MADMAP_OK) return st;
  if (ev) cudaEventRecord(ev[(*ei)++], s);
  if constexpr (narrow_ctas<Real, NS>()) {
    if (narrow) k_c3<Real, NS, OUT, 2><<<dim3(N1 / 2, nt), 32, 0, s>>>(a);
  }
  if (!narrow) k_c3<Real, NS, OUT, COLS><<<dim3(N1 / COLS, nt), 16 * COLS, 0, s>>>(a);
  if (ev) cudaEventRecord(ev[(*ei)++], s);
  return MADMAP_OK;
}
