// Mixed form (complex64 sweeps): the dispatch over sweep forms, the W > 64
// (row-chunked) variant and the W <= 16 one.  The W <= 32 and W <= 64 variants
// are compiled in k_xmatvec_c64_w32.cu and k_xmatvec_c64_w64.cu.
#include "xmatvec_mixed.cuh"

DY_SOLVE_VARIANT(float, 0)
DY_CHAIN_VARIANT(float, 16, k_xmatvec_m)

template <>
cudaError_t launch_xmatvec<float>(const Geo& g, const Bufs& b, int K, int j, int mixed, int ncols, cudaStream_t st) {
  if (g.W > DY_MAXW_SMEM) return run_xmatvec<float, 0>(g, b, K, j, mixed, ncols, st);
  if (g.W <= 16) return run_xmatvec_m<float, 16>(g, b, K, j, ncols, st);
  if (g.W <= 32) return run_xmatvec_m<float, 32>(g, b, K, j, ncols, st);
  return run_xmatvec_m<float, 64>(g, b, K, j, ncols, st);
}

template <>
cudaError_t launch_bsolve<float>(const Geo& g, const Bufs& b, int K, const cxd* q_dd, cxd* w_dd,
                                 cudaStream_t st) {
  if (g.W > DY_MAXW_SMEM) return run_bsolve<float, 0>(g, b, K, q_dd, w_dd, st);
  if (g.W <= 16) return run_bsolve_m<float, 16>(g, b, K, q_dd, w_dd, st);
  if (g.W <= 32) return run_bsolve_m<float, 32>(g, b, K, q_dd, w_dd, st);
  return run_bsolve_m<float, 64>(g, b, K, q_dd, w_dd, st);
}
