// Float32 operator kernels with the transforms in registers (windows of
// M = 256 N1 points, N1 = 64 .. 1024; included by operator_kernels.cuh).
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
// 531 -> 412 us (and to 201 and 365 us with the packed sums and short run sums
// below).  Sixteen columns a CTA because 256 threads x 16 elements leave
// four CTAs per SM at 64 registers; three CTAs with twice or four times the
// loads in flight per thread measured slower (442 and 468 us on the ring scan),
// and so did loading the pointing one to four batches ahead of the map (373 -> 387
// to 458 us: at 64 registers the loads in flight cost more than they hide).
// Shorter windows would leave rows of less than 64 points to groups of fewer
// than 8 lanes (32-byte rows of scratch), longer ones need rows of more than
// 32 x 32: both stay with k_f1, k_f2 and k_f3.
//
// Scratch rows are in natural order of k2 and the spectrum H32 in natural
// order [k2][k1], so no index is bit-reversed outside registers.
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

// 2^LG-point DFT (INV: inverse, unnormalised) of registers, natural order in,
// bit-reversed order out: radix-2 decimation in frequency, constant twiddles.
// Complex sums are one packed instruction each (add2, sub2): the row kernel
// issued on 69% of its cycles and half of its instructions were these (ring
// scan, 2^18: rows 46.7 -> 42.5, inverse columns 113 -> 103 us per launch, one
// application 416 -> 387 us).
template <int LG, bool INV>
__device__ __forceinline__ void reg_dft(float2 (&v)[1 << LG]) {
#pragma unroll
  for (int st = 0; st < LG; ++st) {
    const int span = 1 << (LG - 1 - st);
#pragma unroll
    for (int m = 0; m < (1 << LG); ++m) {
      if ((m & span) == 0) {
        const float2 x = v[m], y = v[m + span];
        v[m] = add2(x, y);
        v[m + span] = mul_w32<INV>(sub2(x, y), ((m & (span - 1)) << st) << (5 - LG));
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

// Lanes of a run sum in k_c3 (run_sum): a run of samples in one pixel adds once
// per aligned group of this many.  Four takes two shuffle steps of each of the
// three sums where a warp row of 16 samples takes four, for one atomic in two
// samples instead of one in three on the ring scan (0.65 repeats); the shuffles
// were a third of the kernel's L1 wavefronts (16, 8, 4 lanes: 103.5, 97.9, 97.6
// us per launch, 387, 377, 373 us per application).
constexpr int REG_RUN = 4;
constexpr int REG_COLS = 16;   // columns per CTA of k_c1 and k_c3 (256 threads x 16 elements)
#ifndef MM_MINB_C1
#define MM_MINB_C1 4
#endif
#ifndef MM_MINB_C3
#define MM_MINB_C3 4
#endif
#ifndef MM_U_C1
#define MM_U_C1 2
#endif
#ifndef MM_U_C3
#define MM_U_C3 2
#endif

// ---------------------------------------------------------------- k_c1
// Thread (column c, group j): elements n2 = j + 16 u (u = 0 .. 15) of column n1.
// 256 = 16 x 16: X[k2 = p + 16 b] = sum_j W16^(j b) W256^(j p) sum_u x[j + 16 u] W16^(u p).
template <int NS, int IN>
__global__ void __launch_bounds__(256, MM_MINB_C1) k_c1(OpArgs a) {
  const Tile* T = a.tiles + a.tile0 + blockIdx.y;
  if (skip_tile(a, T)) return;
  __shared__ float2 buf[256 * REG_COLS];
  const int c = threadIdx.x & (REG_COLS - 1), j = threadIdx.x / REG_COLS;
  const int n1 = blockIdx.x * REG_COLS + c, logN1 = a.reg_logN1, N1 = 1 << logN1;
  LaneView<float> L[2];
  L[0] = lane_view<float, IN, OUT_MAP>(a, T->l[0]);
  L[1] = lane_view<float, IN, OUT_MAP>(a, T->l[1]);
  constexpr int U = gathers(IN) ? MM_U_C1 : 8;
  float2 v[16];
#pragma unroll
  for (int b = 0; b < 16 / U; ++b) {
    int nn[U];
    float x[2][U];
#pragma unroll
    for (int k = 0; k < U; ++k) nn[k] = n1 + ((j + 16 * (U * b + k)) << logN1);
    gather_samples<float, NS, IN, U>(a, L, nn, x);
#pragma unroll
    for (int k = 0; k < U; ++k) v[U * b + k] = make_float2(x[0][k], x[1][k]);
  }
  reg_dft<4, false>(v);
  {
    const Powers<4> w(a.reg_col + 2 * j);
#pragma unroll
    for (int m = 0; m < 16; ++m) {
      const int p = brev_lg<4>(m);
      buf[(p * 16 + j) * REG_COLS + c] = p == 0 ? v[m] : cmul(v[m], w(p));
    }
  }
  __syncthreads();
  // thread (c, p = j): all of group p's elements
#pragma unroll
  for (int m = 0; m < 16; ++m) v[m] = buf[(j * 16 + m) * REG_COLS + c];
  reg_dft<4, false>(v);
  // four-step twiddle exp(-2 pi i n1 k2 / M), k2 = j + 16 b: w0 w^b
  float2* sc = static_cast<float2*>(a.scratch) + (long long)blockIdx.y * a.M + n1;
  const float2 w0 = __ldg(a.reg_four0 + j * N1 + n1);
  const Powers<4> w(a.reg_four + 2 * n1);
#pragma unroll
  for (int m = 0; m < 16; ++m) {
    const int b = brev_lg<4>(m);
    sc[(long long)(j + 16 * b) << logN1] = cmul(v[m], b == 0 ? w0 : cmul(w0, w(b)));
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
  static constexpr int WARPS = 4, PER_WARP = 32 / RB, ROWS = WARPS * PER_WARP;
};
template <int LA, int LB>
__global__ void __launch_bounds__(128, LA == 5 ? 4 : 8) k_c2(OpArgs a) {
  typedef RowGeom<LA, LB> G;
  constexpr int RA = G::RA, RB = G::RB, Q = RA / RB, LN = LA + LB;
  const Tile* T = a.tiles + a.tile0 + blockIdx.y;
  if (skip_tile(a, T)) return;
  __shared__ float2 buf[G::ROWS * G::ROW];
  const int l = threadIdx.x & (RB - 1), r = threadIdx.x / RB;
  float2* const x = buf + r * G::ROW;
  const int row = blockIdx.x * G::ROWS + r;
  float2* sc = static_cast<float2*>(a.scratch) + (long long)blockIdx.y * a.M + ((long long)row << LN) + l;
  const float* H = static_cast<const float*>(a.H) + (long long)T->filter * a.M + ((long long)row << LN) + l;
  float2 v[RA];
#pragma unroll
  for (int u = 0; u < RA; ++u) v[u] = sc[RB * u];
  reg_dft<LA, false>(v);
  {
    const Powers<LA> w(a.reg_row + 4 * l);
#pragma unroll
    for (int m = 0; m < RA; ++m) {
      const int p = brev_lg<LA>(m);
      x[p * G::S + l] = p == 0 ? v[m] : cmul(v[m], w(p));
    }
  }
  __syncwarp();
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    float2 z[RB], y[RB];
    float h[RB];
#pragma unroll
    for (int b = 0; b < RB; ++b) h[b] = __ldg(H + RB * q + RA * b);
#pragma unroll
    for (int m = 0; m < RB; ++m) z[m] = x[(l + RB * q) * G::S + m];
    reg_dft<LB, false>(z);
#pragma unroll
    for (int m = 0; m < RB; ++m) {
      const int b = brev_lg<LB>(m);
      y[b] = make_float2(z[m].x * h[b], z[m].y * h[b]);
    }
    reg_dft<LB, true>(y);
    const Powers<LB> w(a.reg_row + 4 * (l + RB * q));
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
template <int NS, int OUT>
__global__ void __launch_bounds__(256, MM_MINB_C3) k_c3(OpArgs a) {
  const Tile* T = a.tiles + a.tile0 + blockIdx.y;
  if (skip_tile(a, T)) return;
  __shared__ float2 buf[256 * REG_COLS];
  // half-wave-plate sums of the CTA, per tile lane (extended pointing only)
  constexpr bool HWP = extended(NS) && OUT == OUT_MAP;
  __shared__ float hacc[HWP ? 64 : 1];
  __shared__ int hgrp[2];
  if (HWP) {
    for (int i = threadIdx.x; i < 64; i += 256) hacc[i] = 0;
    if (threadIdx.x < 2) hgrp[threadIdx.x] = -1;
  }
  const int c = threadIdx.x & (REG_COLS - 1), j = threadIdx.x / REG_COLS;
  const int n1 = blockIdx.x * REG_COLS + c, logN1 = a.reg_logN1, N1 = 1 << logN1;
  const float2* sc = static_cast<const float2*>(a.scratch) + (long long)blockIdx.y * a.M + n1;
  float2 v[16], y[16];
#pragma unroll
  for (int b = 0; b < 16; ++b) v[b] = sc[(long long)(j + 16 * b) << logN1];
  {
    const float2 w0 = __ldg(a.reg_four0 + j * N1 + n1);
    const Powers<4> w(a.reg_four + 2 * n1);
#pragma unroll
    for (int b = 0; b < 16; ++b) v[b] = cmulc(v[b], b == 0 ? w0 : cmul(w0, w(b)));
  }
  reg_dft<4, true>(v);
  {
    const Powers<4> w(a.reg_col + 2 * j);
#pragma unroll
    for (int m = 0; m < 16; ++m) {
      const int q = brev_lg<4>(m);
      buf[(j * 16 + q) * REG_COLS + c] = q == 0 ? v[m] : cmulc(v[m], w(q));
    }
  }
  __syncthreads();
#pragma unroll
  for (int p = 0; p < 16; ++p) v[p] = buf[(p * 16 + j) * REG_COLS + c];
  reg_dft<4, true>(v);
#pragma unroll
  for (int m = 0; m < 16; ++m) y[brev_lg<4>(m)] = v[m];
  LaneView<float> L[2];
  L[0] = lane_view<float, IN_MAPX, OUT>(a, T->l[0]);
  L[1] = lane_view<float, IN_MAPX, OUT>(a, T->l[1]);
  constexpr int U = OUT == OUT_MAP ? MM_U_C3 : 8;
#pragma unroll
  for (int b = 0; b < 16 / U; ++b) {
    int nn[U];
    float val[2][U];
#pragma unroll
    for (int k = 0; k < U; ++k) {
      nn[k] = n1 + ((j + 16 * (U * b + k)) << logN1);
      val[0][k] = y[U * b + k].x;
      val[1][k] = y[U * b + k].y;
    }
    scatter_samples<float, NS, OUT, U, REG_RUN>(a, L, nn, val, hacc, hgrp);
  }
  if constexpr (HWP) {
    if (a.hwp_base) {
      __syncthreads();
      for (int l = 0; l < 2; ++l)
        hwp_flush(static_cast<float*>(L[l].out), map_ns(NS) == 3 ? 4 : 1, hacc + 32 * l, hgrp + l, 1);
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
      atomicAdd(g + RB * q + RA * b, (double)u.x * (double)v.x + (double)u.y * (double)v.y);
    }
}

// The kernels of a plan with register transforms, and their grids for nt tiles.
template <int NS, int IN, int OUT>
inline void launch_reg(const OpArgs& a, int nt, cudaStream_t s, cudaEvent_t* ev, int* ei) {
  const int N1 = 1 << a.reg_logN1;
  const dim3 g13(N1 / REG_COLS, nt);
  if (ev) cudaEventRecord(ev[(*ei)++], s);
  k_c1<NS, IN><<<g13, 256, 0, s>>>(a);
  if (ev) cudaEventRecord(ev[(*ei)++], s);
  switch (a.reg_logN1) {
    case 6: k_c2<3, 3><<<dim3(256 / RowGeom<3, 3>::ROWS, nt), 128, 0, s>>>(a); break;
    case 7: k_c2<4, 3><<<dim3(256 / RowGeom<4, 3>::ROWS, nt), 128, 0, s>>>(a); break;
    case 8: k_c2<4, 4><<<dim3(256 / RowGeom<4, 4>::ROWS, nt), 128, 0, s>>>(a); break;
    case 9: k_c2<5, 4><<<dim3(256 / RowGeom<5, 4>::ROWS, nt), 128, 0, s>>>(a); break;
    default: k_c2<5, 5><<<dim3(256 / RowGeom<5, 5>::ROWS, nt), 128, 0, s>>>(a); break;
  }
  if (ev) cudaEventRecord(ev[(*ei)++], s);
  k_c3<NS, OUT><<<g13, 256, 0, s>>>(a);
  if (ev) cudaEventRecord(ev[(*ei)++], s);
}
