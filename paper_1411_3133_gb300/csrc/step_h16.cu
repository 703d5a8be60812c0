// Fused time-step kernels, FP16 deviation storage with FP32 arithmetic:
// instantiations for the flat, cylindrical and ellipsoidal metrics.
#include "step_launch.cuh"

namespace lbgm {

cudaError_t launch_step_h16(int K, const __half* fin, __half* fout, const GeoDev<float>& geo,
                            const InstParams<float>* inst, const Dims& d, int* flag, int threads,
                            bool chained, cudaStream_t s) {
  return launch_pair_t<__half>(K, fin, fout, geo, inst, d, flag, threads, chained, s);
}

cudaError_t launch_step_list_h16(int K, const Dims& d, size_t smem, const void* recs, int count, const int* items,
                                 int tile, int threads, int grid, int parity, bool chained, cudaStream_t s) {
  return launch_pair_list_t<__half>(K, d, smem, recs, count, items, tile, threads, grid, parity, chained, s);
}

cudaError_t step_list_occupancy_h16(int K, const Dims& d, size_t smem, int threads, int* blocks_per_sm) {
  return pair_list_occupancy_t<__half>(K, d, smem, threads, blocks_per_sm);
}

}  // namespace lbgm
