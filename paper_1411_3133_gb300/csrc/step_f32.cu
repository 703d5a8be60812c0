// Fused time-step kernel, FP32 populations and arithmetic: instantiations for
// every metric.
#include "step_launch.cuh"

namespace lbgm {

cudaError_t launch_step_f32(int K, const float* fin, float* fout, const GeoDev<float>& geo,
                            const InstParams<float>* inst, const Dims& d, int* flag, int threads,
                            bool chained, cudaStream_t s) {
  return launch_step_t<float>(K, fin, fout, geo, inst, d, flag, threads, chained, s);
}

cudaError_t launch_step_list_f32(int K, const void* recs, int count, const int* items, int tile, int threads,
                                 int grid, int parity, bool chained, cudaStream_t s) {
  return launch_step_list_t<float>(K, recs, count, items, tile, threads, grid, parity, chained, s);
}

cudaError_t step_list_occupancy_f32(int K, int threads, int* blocks_per_sm) {
  return step_list_occupancy_t<float>(K, threads, blocks_per_sm);
}

}  // namespace lbgm
