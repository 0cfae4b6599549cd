// The float operator kernels (see operator_kernels.cuh), compiled apart from
// the other precisions so the library's translation units build in parallel.
#include "operator_kernels.cuh"

namespace mm {

const OpImpl& op_impl_f32() {
  static const OpImpl impl = make_impl<float>();
  return impl;
}

// Cross spectra of the backward pass's windows (tiles of p->corr: a, then r of
// each pair), summed per filter into corr.G.
madmap_status corr_spectrum(Plan* p, cudaStream_t s) {
  const CorrPlan& c = p->corr;
  OpArgs a = {};
  a.M = c.M;
  a.tiles = c.tiles;
  a.in = p->bw_a;
  a.in_stride = p->n_t;
  a.scratch = c.scratch;
  a.reg_logN1 = c.reg.logN1;
  a.reg_col = c.reg.col;
  a.reg_row = c.reg.row;
  a.reg_four = c.reg.four;
  a.reg_four0 = c.reg.four0;
  for (int t0 = 0; t0 < c.n_pairs; t0 += c.per_chunk) {
    const int n = std::min(c.per_chunk, c.n_pairs - t0);
    a.tile0 = 2 * t0;
    k_c1<float, 1, IN_TODF, 16><<<dim3((1 << a.reg_logN1) / 16, 2 * n), 256, 0, s>>>(a);
    switch (a.reg_logN1) {
      case 6: k_xcorr<3, 3><<<dim3(256 / RowGeom<3, 3>::ROWS, n), 128, 0, s>>>(a, c.G); break;
      case 7: k_xcorr<4, 3><<<dim3(256 / RowGeom<4, 3>::ROWS, n), 128, 0, s>>>(a, c.G); break;
      case 8: k_xcorr<4, 4><<<dim3(256 / RowGeom<4, 4>::ROWS, n), 128, 0, s>>>(a, c.G); break;
      case 9: k_xcorr<5, 4><<<dim3(256 / RowGeom<5, 4>::ROWS, n), 128, 0, s>>>(a, c.G); break;
      default: k_xcorr<5, 5><<<dim3(256 / RowGeom<5, 5>::ROWS, n), 128, 0, s>>>(a, c.G); break;
    }
    count_launches(2);
  }
  MM_CUDA(cudaGetLastError());
  return MADMAP_OK;
}

}  // namespace mm
