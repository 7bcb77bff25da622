// FP64 form (complex128 sweeps): the 8-warp sweep for 32 < W <= 64 and the
// row-chunked sweep for W > 64; the two-chain strips (W <= 32) are compiled in
// k_xmatvec_c128_chain.cu.
#include "solve_device.cuh"
#include "xmatvec_mixed.cuh"

DY_SOLVE_VARIANT(double, 0)
DY_SOLVE_VARIANT(double, 64)

template <>
cudaError_t launch_xmatvec<double>(const Geo& g, const Bufs& b, int K, int j, int mixed, int ncols, cudaStream_t st) {
  if (g.W > DY_MAXW_SMEM) return run_xmatvec<double, 0>(g, b, K, j, mixed, ncols, st);
  if (g.W > DY_TWO_MAXW64) return run_xmatvec<double, 64>(g, b, K, j, mixed, ncols, st);
  if (g.W <= 16) return run_xmatvec_m<double, 16>(g, b, K, j, ncols, st);
  return run_xmatvec_m<double, 32>(g, b, K, j, ncols, st);
}

template <>
cudaError_t launch_bsolve<double>(const Geo& g, const Bufs& b, int K, const cxd* q_dd, cxd* w_dd,
                                  cudaStream_t st) {
  if (g.W > DY_MAXW_SMEM) return run_bsolve<double, 0>(g, b, K, q_dd, w_dd, st);
  if (g.W > DY_TWO_MAXW64) return run_bsolve<double, 64>(g, b, K, q_dd, w_dd, st);
  if (g.W <= 16) return run_bsolve_m<double, 16>(g, b, K, q_dd, w_dd, st);
  return run_bsolve_m<double, 32>(g, b, K, q_dd, w_dd, st);
}
