// Float64 transforms of whole real sequences on the device: the filters'
// spectra when a plan is built or its filters change, and the way back from
// the backward pass's cross spectrum to lags.
//
// One complex FFT of length M = N1 N2 per filter in two kernels (columns, then
// rows), with the shared-memory passes of the operator kernels.  Both
// sequences are real and even up to what the caller drops, so only real parts
// leave the second kernel.  (Two filters in one complex transform would let the
// rounding of a large one into a much smaller one.)
//
// On the host the same transforms took 3.2 ms for 8 filters of M = 2^16 on 16
// cores, most of a set_filters call; they are latency-bound here (two launches
// of M / 2048 CTAs per filter, about 10^8 float64 operations).
#include <math.h>

#include <algorithm>
#include <cstring>
#include <string>
#include <vector>

#include "internal.cuh"

namespace mm {

namespace {

// SPEC: x(n) = the circulant embedding of filter f's lags, out: H64, Hdf and
// H32 / M in the operator kernels' order.  CORR: x(k) = the cross spectrum G
// [k mod 256][k / 256], out: the correlations at lags 0 .. n_lags - 1.
// LAGS: x(j) = 1 / PSD of filter f (symmetric in j), out: its tapered lags.
// VJP: x(t) = the tapered gradient of the lags, out: each CTA's share of the
// gradient of (sigma, f_knee, alpha).
enum { SPEC = 0, CORR = 1, LAGS = 2, VJP = 3 };
struct SpecArgs {
  int M, logN1, logN2, logB1, logB2, n_lags;
  const double* x;
  const double2* tw;   // [M] exp(-2 pi i j / M)
  double2* scratch;    // [filters of the launch][M]
  double* H64;
  float* H32;
  df64* Hdf;
  int reg_logN1;       // SPEC: H32 in the register kernels' order; CORR: G's row length
  unsigned long long* mins;  // SPEC: order-preserving bits of each filter's spectrum minimum
  double* grad;        // CORR, LAGS: [filters][n_lags]; VJP: [filters][CTAs of the row kernel][3]
  const double* prm;   // VJP: [filters][3]
  double fs;
};

// (f_knee / nu_j)^alpha and 1 / PSD at frequency j of a grid of L points (the
// zero frequency takes the first one's value), and the latter's gradient, as
// madmap_noise_filter states them.
__device__ __forceinline__ void inverse_psd(const double* prm, double fs, int j, int L, double& nu, double& r,
                                            double& q) {
  nu = (double)(j > 0 ? j : 1) * fs / (double)L;
  r = pow(prm[1] / nu, prm[2]);
  q = 1.0 / (prm[0] * prm[0] * (1.0 + r));
}
__global__ void k_inverse_psd(const double* prm, double fs, int L, int n_f, double* out) {
  const int n = L / 2 + 1;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < (long long)n * n_f;
       i += (long long)gridDim.x * blockDim.x) {
    double nu, r, q;
    inverse_psd(prm + 3 * (i / n), fs, (int)(i % n), L, nu, r, q);
    out[i] = q;
  }
}

__device__ __forceinline__ unsigned long long order_bits(double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}

template <int MODE>
__global__ void __launch_bounds__(OP_THREADS) k_spec_cols(SpecArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double2* buf = reinterpret_cast<double2*>(smem_raw);
  const int N1 = 1 << a.logN1, B1 = 1 << a.logB1, rs = lay_rs(16, a.logN2, true);
  constexpr int SW = 0;
  double2* tw = buf + B1 * rs;
  build_pass_twiddles(tw, a.logN2, a.tw, N1);
  const int f = blockIdx.y, n1_0 = blockIdx.x * B1, total = B1 << a.logN2;
  for (int e = threadIdx.x; e < total; e += OP_THREADS) {
    const int n = n1_0 + (e & (B1 - 1)) + ((e >> a.logB1) << a.logN1);
    double v;
    if (MODE == SPEC) {
      const int t = n < a.M - n ? n : a.M - n;
      v = t < a.n_lags ? a.x[(long long)f * a.n_lags + t] : 0.0;
    } else if (MODE == LAGS) {
      v = a.x[(long long)f * (a.M / 2 + 1) + (n < a.M - n ? n : a.M - n)];
    } else if (MODE == VJP) {
      v = n < a.n_lags ? (1.0 - (double)n / a.n_lags) * a.x[(long long)f * a.n_lags + n] : 0.0;
    } else {
      v = a.x[(long long)f * a.M + ((long long)(n & (REG_N2 - 1)) << a.reg_logN1) + (n >> 8)];
    }
    buf[(e & (B1 - 1)) * rs + swz<SW>(e >> a.logB1)] = make_double2(v, 0.0);
  }
  __syncthreads();
  fft_rows<double2, false, SW>(buf, B1, rs, a.logN2, tw);
  double2* sc = a.scratch + (long long)f * a.M;
  for (int e = threadIdx.x; e < total; e += OP_THREADS) {
    const int j = e & (B1 - 1), pos = e >> a.logB1;
    const double2 w = a.tw[((n1_0 + j) * brev_n(pos, a.logN2)) & (a.M - 1)];
    sc[((long long)pos << a.logN1) + n1_0 + j] = cmul(buf[j * rs + swz<SW>(pos)], w);
  }
}

template <int MODE>
__global__ void __launch_bounds__(OP_THREADS) k_spec_rows(SpecArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double2* buf = reinterpret_cast<double2*>(smem_raw);
  const int N1 = 1 << a.logN1, B2 = 1 << a.logB2, rs = lay_rs(16, a.logN1, false);
  constexpr int SW = 1;
  double2* tw = buf + B2 * rs;
  build_pass_twiddles(tw, a.logN1, a.tw, 1 << a.logN2);
  const int f = blockIdx.y, pos0 = blockIdx.x * B2, total = B2 << a.logN1;
  const double2* sc = a.scratch + (long long)f * a.M + ((long long)pos0 << a.logN1);
  for (int e = threadIdx.x; e < total; e += OP_THREADS)
    buf[(e >> a.logN1) * rs + swz<SW>(e & (N1 - 1))] = sc[e];
  __syncthreads();
  fft_rows<double2, false, SW>(buf, B2, rs, a.logN1, tw);
  const double inv = 1.0 / (double)a.M;   // a power of two
  unsigned long long mn = ~0ull;
  double sum[3] = {0.0, 0.0, 0.0};
  for (int e = threadIdx.x; e < total; e += OP_THREADS) {
    const int pos2 = pos0 + (e >> a.logN1), pos1 = e & (N1 - 1);
    const double v = buf[(e >> a.logN1) * rs + swz<SW>(pos1)].x * inv;
    const int k = brev_n(pos2, a.logN2) + (brev_n(pos1, a.logN1) << a.logN2);
    if (MODE == SPEC) {
      // a NaN orders above +inf as positive, so it is mapped below every value
      const unsigned long long b = v == v ? order_bits(v) : 0ull;
      mn = b < mn ? b : mn;
      long long o = (long long)f * a.M + ((long long)pos2 << a.logN1) + pos1, r = o;
      if (a.reg_logN1 > 0) {
        const int k1 = k >> 8;
        o = r = (long long)f * a.M + ((long long)(k & (REG_N2 - 1)) << a.reg_logN1);
        r += k1;
        o += a.reg_logN1 > 8 ? brev_n(k1, a.reg_logN1) : k1;
      }
      a.H64[o] = v;
      a.Hdf[o] = df64((float)v, (float)(v - (double)(float)v));
      a.H32[r] = (float)v;
    } else if (MODE == LAGS) {
      if (k < a.n_lags) a.grad[(long long)f * a.n_lags + k] = (1.0 - (double)k / a.n_lags) * v;
    } else if (MODE == VJP) {
      if (k <= a.M / 2) {
        const double* prm = a.prm + 3 * f;
        double nu, r, q;
        inverse_psd(prm, a.fs, k, a.M, nu, r, q);
        const double w = (k == 0 || k == a.M / 2) ? v : 2.0 * v;
        sum[0] += w * (-2.0 * q / prm[0]);
        if (prm[1] > 0.0) {
          const double c = -q * q * prm[0] * prm[0] * r * w;
          sum[1] += c * prm[2] / prm[1];
          sum[2] += c * log(prm[1] / nu);
        }
      }
    } else if (k < a.n_lags) {
      // c(tau) + c(-tau) = sum_k 2 G cos / M; tau = 0 counts once
      a.grad[(long long)f * a.n_lags + k] = k == 0 ? v : 2.0 * v;
    }
  }
  if (MODE == SPEC) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long b = __shfl_xor_sync(0xffffffffu, mn, o);
      mn = b < mn ? b : mn;
    }
    if ((threadIdx.x & 31) == 0) atomicMin(a.mins + f, mn);
  }
  if (MODE == VJP) {   // fixed order: the CTA's warps here, the CTAs on the host
    __shared__ double part[OP_THREADS / 32][3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      for (int o = 16; o > 0; o >>= 1) sum[i] += __shfl_xor_sync(0xffffffffu, sum[i], o);
      if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5][i] = sum[i];
    }
    __syncthreads();
    if (threadIdx.x < 3) {
      double t = 0.0;
      for (int w = 0; w < OP_THREADS / 32; ++w) t += part[w][threadIdx.x];
      a.grad[((long long)f * gridDim.x + blockIdx.x) * 3 + threadIdx.x] = t;
    }
  }
}

__global__ void k_fill_twiddles(double2* tw, int M) {
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < M; j += gridDim.x * blockDim.x) {
    double s, c;
    sincospi(2.0 * (double)j / (double)M, &s, &c);
    tw[j] = make_double2(c, -s);
  }
}

// The wide tables (wide_four) of length M = 256 N1 from the table of M-th roots.
template <typename C>
__global__ void k_wide_tables(const C* tw, C* out, int logN1) {
  const int N1 = 1 << logN1, M = N1 << 8, lb = wide_lb(logN1), la = logN1 - lb, n = wide_four(logN1) + M;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    int m;
    if (i < WIDE_ROW_F) {
      m = (i >> 4) * (i & 15) * N1;
    } else if (i < wide_row_i(logN1)) {
      const int e = i - WIDE_ROW_F;
      m = (e >> lb) * (e & ((1 << lb) - 1)) * REG_N2;
    } else if (i < wide_row(logN1)) {
      const int e = i - wide_row_i(logN1);
      m = (e >> la) * (e & ((1 << la) - 1)) * REG_N2;
    } else if (i < wide_four(logN1)) {
      m = (i - wide_row(logN1)) * REG_N2;
    } else {
      const int e = i - wide_four(logN1);
      m = (e >> logN1) * (e & (N1 - 1));
    }
    out[i] = tw[m & (M - 1)];
  }
}

// Both kernels over n_f filters, at most `batch` (filters of scratch) a launch.
template <int MODE>
madmap_status run_spec(SpecArgs a, int n_f, int batch, cudaStream_t s) {
  const int lg = a.logN1 + a.logN2, E = 11;   // 2048 elements per CTA
  a.logB1 = std::max(0, std::min(E - a.logN2, a.logN1));
  a.logB2 = std::max(0, std::min(E - a.logN1, a.logN2));
  const size_t s1 = (((size_t)lay_rs(16, a.logN2, true) << a.logB1) + ((size_t)1 << a.logN2)) * 16;
  const size_t s2 = (((size_t)lay_rs(16, a.logN1, false) << a.logB2) + ((size_t)1 << a.logN1)) * 16;
  MM_CUDA(cudaFuncSetAttribute(k_spec_cols<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 << 10));
  MM_CUDA(cudaFuncSetAttribute(k_spec_rows<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 << 10));
  MM_CHECK(s1 <= (96u << 10) && s2 <= (96u << 10) && lg <= 20, MADMAP_ERR_INTERNAL, "spectra: bad geometry");
  const SpecArgs b = a;
  batch = std::min(batch, 65535);
  for (int f = 0; f < n_f; f += batch) {
    const int n = std::min(batch, n_f - f);
    a.x = b.x + (long long)f * (MODE == CORR ? a.M : MODE == LAGS ? a.M / 2 + 1 : a.n_lags);
    if (MODE == VJP) {
      a.grad = b.grad + ((long long)f << (a.logN2 - a.logB2)) * 3;
      a.prm = b.prm + 3 * f;
    } else if (MODE == SPEC) {
      a.H64 = b.H64 + (long long)f * a.M;
      a.H32 = b.H32 + (long long)f * a.M;
      a.Hdf = b.Hdf + (long long)f * a.M;
      a.mins = b.mins + f;
    } else {
      a.grad = b.grad + (long long)f * a.n_lags;
    }
    k_spec_cols<MODE><<<dim3(1 << (a.logN1 - a.logB1), n), OP_THREADS, s1, s>>>(a);
    k_spec_rows<MODE><<<dim3(1 << (a.logN2 - a.logB2), n), OP_THREADS, s2, s>>>(a);
    count_launches(2);
  }
  MM_CUDA(cudaGetLastError());
  return MADMAP_OK;
}

}  // namespace

madmap_status fill_wide_tables(Plan* p, cudaStream_t s) {
  const int rl = p->reg.logN1, grid = (wide_four(rl) + p->M + 255) / 256;
  k_wide_tables<double2><<<grid, 256, 0, s>>>(p->tw64, p->wide64, rl);
  k_wide_tables<cdf64><<<grid, 256, 0, s>>>(p->twdf, p->wide_df, rl);
  MM_CUDA(cudaGetLastError());
  return MADMAP_OK;
}

// The spectra of all filters (p->lags) into p->H64, p->H32 and p->Hdf, using
// p->tw64 and p->scratch; waits for the stream and fails when a symbol is not
// positive.
madmap_status build_spectra(Plan* p, cudaStream_t s) {
  const int F = p->n_filters;
  const size_t nl = p->lags.size();
  // one temporary: lags, then the minima
  double* dl = nullptr;
  MM_CUDA(cudaMalloc(&dl, sizeof(double) * (nl + F)));
  unsigned long long* mins = reinterpret_cast<unsigned long long*>(dl + nl);
  std::vector<unsigned long long> h(F, ~0ull);
  cudaError_t e = cudaMemcpyAsync(dl, p->lags.data(), sizeof(double) * nl, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(mins, h.data(), sizeof(h[0]) * F, cudaMemcpyHostToDevice, s);
  madmap_status st = e == cudaSuccess ? MADMAP_OK : cuda_fail(e, "cudaMemcpy (lags)");
  if (st == MADMAP_OK) {
    SpecArgs a = {};
    a.M = p->M;
    a.logN1 = p->logN1;
    a.logN2 = p->logN2;
    a.n_lags = p->n_lags;
    a.x = dl;
    a.tw = p->tw64;
    a.scratch = static_cast<double2*>(p->scratch);
    a.H64 = p->H64;
    a.H32 = p->H32;
    a.Hdf = p->Hdf;
    a.reg_logN1 = p->reg.logN1;
    a.mins = mins;
    st = run_spec<SPEC>(a, F, p->scratch_slots * p->tiles_per_chunk, s);
  }
  if (st == MADMAP_OK) {
    e = cudaMemcpyAsync(h.data(), mins, sizeof(h[0]) * F, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) st = cuda_fail(e, "spectra");
  }
  cudaFree(dl);
  if (st != MADMAP_OK) return st;
  for (int f = 0; f < F; ++f) {
    const unsigned long long b = h[f];
    double mn = NAN;
    if (b != 0ull) {
      const unsigned long long u = (b >> 63) ? (b & 0x7fffffffffffffffull) : ~b;
      memcpy(&mn, &u, sizeof(mn));
      mn *= (double)p->M;
    }
    if (!(mn > 0.0)) {
      set_error("filter " + std::to_string(f) + " is not positive definite (circulant symbol minimum " +
                std::to_string(mn) + ")");
      return MADMAP_ERR_NOT_PD;
    }
  }
  return MADMAP_OK;
}

// ---------------------------------------------------------------- noise filters from their parameters
// madmap_noise_filter and its chain rule for all of a plan's filters at once, for
// lag counts whose grid of L = 4 n_lags frequencies the transforms take (on the host,
// filter by filter, where the device has no memory left for it).  8 filters
// of 4096 lags on host threads: 2.2 ms and 2.3 ms a training step.
namespace {

bool noise_on_device(const Plan* p) {
  return p->n_lags >= 64 && p->n_lags <= (1 << 18) && (p->n_lags & (p->n_lags - 1)) == 0;
}

madmap_status noise_setup(Plan* p, cudaStream_t s) {
  NoiseBuffers& b = p->noise;
  if (b.prm) return MADMAP_OK;
  const size_t L = 4 * (size_t)p->n_lags, F = (size_t)p->n_filters;
  b.batch = (int)std::max<size_t>(1, std::min<size_t>(F, ((size_t)64 << 20) / (16 * L)));
  // one allocation: all of it or, for the host's sums, none
  const size_t n_x = F * (L / 2 + 1), n_out = F * p->n_lags;
  double2* base = nullptr;
  const madmap_status st = dalloc_t(p, &base, (b.batch + 1) * L + (n_x + n_out + 3 * F + 1) / 2);
  if (st != MADMAP_OK) return st;
  b.scratch = base + L;
  b.x = reinterpret_cast<double*>(b.scratch + b.batch * L);
  b.out = b.x + n_x;
  k_fill_twiddles<<<(int)((L + 255) / 256), 256, 0, s>>>(base, (int)L);
  b.tw = base;
  b.prm = b.out + n_out;   // set last: the setup is complete
  return MADMAP_OK;
}

SpecArgs noise_args(const Plan* p, double fs) {
  SpecArgs a = {};
  a.M = 4 * p->n_lags;
  const int lg = ilog2((unsigned)a.M);
  a.logN2 = (lg + 1) / 2;
  a.logN1 = lg - a.logN2;
  a.n_lags = p->n_lags;
  a.tw = p->noise.tw;
  a.scratch = p->noise.scratch;
  a.prm = p->noise.prm;
  a.fs = fs;
  return a;
}

madmap_status check_noise(const Plan* p, double fs, const double* prm) {
  for (int f = 0; f < p->n_filters; ++f)
    MM_CHECK(fs > 0 && prm[3 * f] > 0 && prm[3 * f + 1] >= 0 && isfinite(prm[3 * f + 2]), MADMAP_ERR_INVALID_ARG,
             "noise_filter: need fs > 0, sigma > 0, fknee >= 0, finite alpha");
  return MADMAP_OK;
}

}  // namespace

// lags[filter][n_lags] (host) of the parameters prm[filter][3] (host).
madmap_status noise_lags(Plan* p, double fs, const double* prm, double* lags, cudaStream_t s) {
  madmap_status st = check_noise(p, fs, prm);
  if (st != MADMAP_OK) return st;
  const size_t F = (size_t)p->n_filters;
  if (!noise_on_device(p) || (st = noise_setup(p, s)) == MADMAP_ERR_OOM) {
    st = MADMAP_OK;
    for (size_t f = 0; f < F && st == MADMAP_OK; ++f)
      st = madmap_noise_filter(p->n_lags, fs, prm[3 * f], prm[3 * f + 1], prm[3 * f + 2], lags + f * p->n_lags, nullptr);
    return st;
  }
  if (st != MADMAP_OK) return st;
  MM_CUDA(cudaMemcpyAsync(p->noise.prm, prm, sizeof(double) * 3 * F, cudaMemcpyHostToDevice, s));
  SpecArgs a = noise_args(p, fs);
  const long long n = (long long)F * (a.M / 2 + 1);
  k_inverse_psd<<<(int)std::min<long long>((n + 127) / 128, 152LL * 16), 128, 0, s>>>(p->noise.prm, fs, a.M,
                                                                                      p->n_filters, p->noise.x);
  count_launches(1);
  a.x = p->noise.x;
  a.grad = p->noise.out;
  if ((st = run_spec<LAGS>(a, p->n_filters, p->noise.batch, s)) != MADMAP_OK) return st;
  MM_CUDA(cudaMemcpyAsync(lags, p->noise.out, sizeof(double) * F * p->n_lags, cudaMemcpyDeviceToHost, s));
  MM_CUDA(cudaStreamSynchronize(s));
  return MADMAP_OK;
}

// out[filter][3] (host) = the gradient of the parameters from grad_lags (device).
madmap_status noise_vjp(Plan* p, double fs, const double* prm, const double* grad_lags, double* out, cudaStream_t s) {
  madmap_status st = check_noise(p, fs, prm);
  if (st != MADMAP_OK) return st;
  const size_t F = (size_t)p->n_filters;
  if (!noise_on_device(p) || (st = noise_setup(p, s)) == MADMAP_ERR_OOM) {
    st = MADMAP_OK;
    std::vector<double> g(F * p->n_lags);
    MM_CUDA(cudaMemcpyAsync(g.data(), grad_lags, sizeof(double) * g.size(), cudaMemcpyDeviceToHost, s));
    MM_CUDA(cudaStreamSynchronize(s));
    for (size_t f = 0; f < F && st == MADMAP_OK; ++f)
      st = madmap_noise_filter_vjp(p->n_lags, fs, prm[3 * f], prm[3 * f + 1], prm[3 * f + 2], g.data() + f * p->n_lags,
                                   out + 3 * f);
    return st;
  }
  if (st != MADMAP_OK) return st;
  MM_CUDA(cudaMemcpyAsync(p->noise.prm, prm, sizeof(double) * 3 * F, cudaMemcpyHostToDevice, s));
  SpecArgs a = noise_args(p, fs);
  a.x = grad_lags;
  a.grad = p->noise.x;   // [F][CTAs][3] in [F][L / 2 + 1]
  const int ctas = 1 << (a.logN2 - std::max(0, std::min(11 - a.logN1, a.logN2)));
  MM_CHECK(3 * ctas <= a.M / 2 + 1, MADMAP_ERR_INTERNAL, "noise_vjp: partial sums do not fit");
  if ((st = run_spec<VJP>(a, p->n_filters, p->noise.batch, s)) != MADMAP_OK) return st;
  std::vector<double> part(F * ctas * 3);
  MM_CUDA(cudaMemcpyAsync(part.data(), p->noise.x, sizeof(double) * part.size(), cudaMemcpyDeviceToHost, s));
  MM_CUDA(cudaStreamSynchronize(s));
  for (size_t f = 0; f < F; ++f)
    for (int i = 0; i < 3; ++i) {
      double t = 0.0;
      for (int c = 0; c < ctas; ++c) t += part[(f * ctas + c) * 3 + i];
      out[3 * f + i] = t;
    }
  return MADMAP_OK;
}

// ---------------------------------------------------------------- lag correlation of the backward pass
// sum_{|t - t'| = tau} a_t r_t' per filter for tau < n_lags, by transforms: in
// each overlap-save window, a at the window's exact outputs and r over its
// whole input have the wanted circular correlations at +-tau, so the cross
// spectra Re(conj(Z_a) Z_r) of all windows of a filter are summed (float64) and
// one float64 transform per filter returns the lags.  Two windows share a
// complex transform: of conj(A + iA') (R + iR') the part that mixes them is odd
// in k after taking the real part and leaves the (even) cosine sum unchanged.
static constexpr int CORR_MAX_LAGS = 3 << 15;
static constexpr size_t CORR_SCRATCH = (size_t)128 << 20;

// The plan's own window length where it has register transforms, else the
// shortest one whose windows are at least half exact (a quarter at most lags).
static int corr_fft_len(const Plan* p) {
  if (reg_log_n1(p->M) > 0) return p->M;
  int M = 1 << 14;
  while (M < (1 << 18) && M < 4 * p->n_lags) M <<= 1;
  return M;
}

// Transforms or direct sums, by the time that each is expected to take (both
// measured at 2e3 to 2e7 samples in intervals of 100 to 2e6, 1 to 60000 lags and 1
// to 2000 filters): a pair of windows takes 17 ps a point, a filter's float64
// transform 100 ps a point, their launches 60 us; the direct sums 0.245 ns a sample
// per block of CORR_LB lags, 3.5 ns an item, 6 ps for each atomic it ends with, and
// at least 38 us for each thousand samples of the longest item.  So windows of 2^14
// points are not spent on short intervals (2e6 samples, 50 lags, direct against
// transforms: intervals of 100 0.57 and 2.77 ms, of 300 0.49 and 0.98 ms, of 1000
// 0.49 and 0.34 ms, of 10000 0.74 and 0.08 ms).
static bool fft_cheaper(const Plan* p) {
  if (p->n_lags > CORR_MAX_LAGS) return false;
  const long long M = corr_fft_len(p), h = p->n_lags - 1, U = M - 2 * h;
  std::vector<long long> windows(p->n_filters, 0);
  double samples = 0, items = 0, longest = 0;
  for (int i = 0; i < p->n_ivl; ++i) {
    const long long n = p->offsets[i + 1] - p->offsets[i];
    if (n <= 0) continue;
    windows[p->ivl_filter[i]] += n + h <= M ? 1 : (n + U - 1) / U;
    samples += (double)((n + 7) / 8 * 8);
    items += (double)((n + CORR_CHUNK - 1) / CORR_CHUNK);
    longest = std::max(longest, (double)std::min<long long>(n, CORR_CHUNK));
  }
  double pairs = 0;
  for (long long w : windows) pairs += (double)((w + 1) / 2);
  const double blocks = (double)((p->n_lags + CORR_LB - 1) / CORR_LB);
  const double t_fft = 60.0 + (17e-6 * pairs + 100e-6 * p->n_filters) * M;   // microseconds
  const double t_direct = std::max(blocks * (0.245e-3 * samples + 3.5e-3 * items) + 6e-6 * items * p->n_lags,
                                   38e-3 * longest);
  return t_fft < t_direct;
}

bool corr_by_fft(Plan* p) {
  if (p->corr.route == 0) p->corr.route = fft_cheaper(p) ? 1 : 2;
  return p->corr.route == 1;
}

madmap_status corr_setup(Plan* p, cudaStream_t s) {
  CorrPlan& c = p->corr;
  if (c.G) return MADMAP_OK;
  madmap_status st = MADMAP_OK;
  const int M = corr_fft_len(p);
  const bool own = reg_log_n1(p->M) == 0;   // tables of this pass's own
  c.M = M;
  const int rl = reg_log_n1(M), lg = rl + 8;
  c.logN2 = (lg + 1) / 2;
  c.logN1 = lg - c.logN2;
  // window pairs, each twice: a at the exact outputs (rhs 0), r over the input (rhs 1)
  std::vector<Tile> tiles, both;
  build_tiles(p->offsets, p->ivl_filter, p->n_filters, p->n_lags, M, tiles);
  for (const Tile& t : tiles) {
    Tile ta = t, tr = t;
    for (int l = 0; l < 2; ++l) {
      ta.l[l].lo = t.l[l].ws + t.l[l].out_lo;
      ta.l[l].hi = t.l[l].ws + t.l[l].out_hi;
      ta.l[l].rhs = 0;
      tr.l[l].rhs = 1;
    }
    both.push_back(ta);
    both.push_back(tr);
  }
  c.n_pairs = (int)tiles.size();
  c.per_chunk = (int)std::max<long long>(
      1, std::min<long long>(std::min<long long>(c.n_pairs, 32767), (long long)(CORR_SCRATCH / (2 * (size_t)M * sizeof(float2)))));
  // one buffer for the windows' transforms and then the float64 ones
  c.scratch_bytes = std::max((size_t)c.per_chunk * 2 * M * sizeof(float2), (size_t)M * sizeof(double2));
  // one allocation: all of it or, for the direct sums, none
  std::vector<float> h(own ? reg_table_floats(rl) : 0);
  size_t bytes = 0;
  auto part = [&bytes](size_t n) {
    const size_t o = bytes;
    bytes = (o + n + 255) & ~(size_t)255;
    return o;
  };
  const size_t o_scratch = part(c.scratch_bytes), o_G = part((size_t)p->n_filters * M * sizeof(double)),
               o_tiles = part(both.size() * sizeof(Tile)), o_tw = part(own ? (size_t)M * sizeof(double2) : 0),
               o_tab = part(h.size() * sizeof(float));
  char* base = nullptr;
  if ((st = dalloc_t(p, &base, bytes)) != MADMAP_OK) return st;
  c.scratch = base + o_scratch;
  c.tiles = reinterpret_cast<Tile*>(base + o_tiles);
  if ((st = upload(c.tiles, both.data(), sizeof(Tile) * both.size(), s)) != MADMAP_OK) return st;
  if (own) {
    reg_fill_tables(rl, h.data());
    if ((st = upload(base + o_tab, h.data(), sizeof(float) * h.size(), s)) != MADMAP_OK) return st;
    c.reg = reg_point_tables(rl, reinterpret_cast<const float*>(base + o_tab));
    double2* tw = reinterpret_cast<double2*>(base + o_tw);
    k_fill_twiddles<<<(M + 255) / 256, 256, 0, s>>>(tw, M);
    c.tw = tw;
  } else {
    c.reg = p->reg;
    c.tw = p->tw64;
  }
  c.G = reinterpret_cast<double*>(base + o_G);   // set last: the setup is complete
  return MADMAP_OK;
}

// grad[filter][tau] from p->bw_a, a and then r (corr_setup done).
madmap_status corr_run(Plan* p, double* grad, cudaStream_t s) {
  CorrPlan& c = p->corr;
  MM_CUDA(cudaMemsetAsync(c.G, 0, sizeof(double) * (size_t)p->n_filters * c.M, s));
  madmap_status st = corr_spectrum(p, s);
  if (st != MADMAP_OK) return st;
  SpecArgs a = {};
  a.M = c.M;
  a.logN1 = c.logN1;
  a.logN2 = c.logN2;
  a.n_lags = p->n_lags;
  a.x = c.G;
  a.tw = c.tw;
  a.scratch = static_cast<double2*>(c.scratch);
  a.reg_logN1 = c.reg.logN1;
  a.grad = grad;
  return run_spec<CORR>(a, p->n_filters, (int)std::min<size_t>(65535, c.scratch_bytes / ((size_t)c.M * sizeof(double2))), s);
}

}  // namespace mm

extern "C" madmap_status madmap_plan_noise_vjp(madmap_plan_t plan, double fs, const double* params,
                                               const double* grad_lags, double* grad_params, void* stream) {
  using namespace mm;
  MM_CHECK(plan && params && grad_lags && grad_params, MADMAP_ERR_INVALID_ARG, "plan_noise_vjp: NULL argument");
  return noise_vjp(reinterpret_cast<Plan*>(plan), fs, params, grad_lags, grad_params, static_cast<cudaStream_t>(stream));
}
