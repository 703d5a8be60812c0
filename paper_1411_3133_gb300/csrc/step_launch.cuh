// Launcher of the fused step kernel for one storage/compute type pair; each
// step_*.cu translation unit instantiates one pair so that the large unrolled
// kernel bodies compile in parallel.
#pragma once

#include "kernels.cuh"
#include "launch.h"

namespace lbgm {

template <class S, class R>
cudaError_t launch_step_t(int K, const S* fin, S* fout, const GeoDev<R>& geo, const InstParams<R>* inst,
                          const Dims& d, int* flag, int threads, cudaStream_t s) {
  if (d.batch < 1 || d.batch > 65535) return cudaErrorInvalidValue;
  threads = threads < StepBounds<S, R>::maxt ? threads : StepBounds<S, R>::maxt;
  const dim3 blocks((uint32_t(d.ncell) + threads - 1) / threads, uint32_t(d.batch));
  switch (K) {
    case KFLAT: k_step<S, R, KFLAT><<<blocks, threads, 0, s>>>(fin, fout, geo, inst, d, flag); break;
    case KCYL: k_step<S, R, KCYL><<<blocks, threads, 0, s>>>(fin, fout, geo, inst, d, flag); break;
    case KELL: k_step<S, R, KELL><<<blocks, threads, 0, s>>>(fin, fout, geo, inst, d, flag); break;
    case KELT:  // the theta-resolved ellipsoid: FP64 / FP32 storage, this kernel only
      if constexpr (!Codec<S, R>::uses_ref) {
        k_step<S, R, KELT><<<blocks, threads, 0, s>>>(fin, fout, geo, inst, d, flag);
        break;
      }
      return cudaErrorInvalidValue;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

// Region-split step of 2-byte storage (flat and cylinder, periodic x3,
// bounce-back walls): the interior on stream s, then the 6 wall layers on
// stream se (the caller orders the two streams around the step). Launched
// second, the small wall-layer kernel takes SMs as interior blocks retire.
// Blocks must not straddle an i_r layer (split_supported).
template <class S>
cudaError_t launch_step_split_t(int K, const S* fin, S* fout, const GeoDev<float>& geo,
                                const InstParams<float>* inst, const Dims& d, int* flag, int threads,
                                cudaStream_t s, cudaStream_t se) {
  if (d.batch < 1 || d.batch > 65535 || !d.periodic3 || d.nr < 7) return cudaErrorInvalidValue;
  threads = threads < StepBounds<S, float>::maxt ? threads : StepBounds<S, float>::maxt;
  const uint32_t layer = uint32_t(d.nt) * uint32_t(d.n3);
  if (layer % uint32_t(threads)) return cudaErrorInvalidValue;
  const dim3 ge(6u * layer / threads, uint32_t(d.batch));
  const dim3 gb(uint32_t(d.nr - 6) * layer / threads, uint32_t(d.batch));
  switch (K) {
    case KFLAT:
      k_step_bulk_rowsm<S, KFLAT><<<gb, threads, 0, s>>>(fin, fout, geo, inst, d, flag);
      k_step_edge_rowsm<S, KFLAT><<<ge, threads, 0, se>>>(fin, fout, geo, inst, d, flag);
      break;
    case KCYL:
      k_step_bulk_rowsm<S, KCYL><<<gb, threads, 0, s>>>(fin, fout, geo, inst, d, flag);
      k_step_edge_rowsm<S, KCYL><<<ge, threads, 0, se>>>(fin, fout, geo, inst, d, flag);
      break;
    default:
      return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

// grid 0: one block per work item; otherwise `grid` persistent blocks. multi:
// the items are longer than one block.
template <class S, class R>
cudaError_t launch_step_list_t(int K, bool multi, const void* insts, const int4* work, int nwork, int threads,
                               int grid, int parity, cudaStream_t s) {
  if (nwork == 0) return cudaSuccess;
  const auto* I = static_cast<const ListInst<S, R>*>(insts);
  const int g = grid > 0 && grid < nwork ? grid : nwork;
#define LB_LIST(KK)                                                                      \
  if (multi) k_step_list<S, R, KK, true><<<g, threads, 0, s>>>(I, work, nwork, parity); \
  else k_step_list<S, R, KK, false><<<g, threads, 0, s>>>(I, work, nwork, parity)
  switch (K) {
    case KFLAT: LB_LIST(KFLAT); break;
    case KCYL: LB_LIST(KCYL); break;
    case KELL: LB_LIST(KELL); break;
    default: return cudaErrorInvalidValue;
  }
#undef LB_LIST
  return cudaGetLastError();
}

// Largest block of the work-list kernel (its launch bounds).
template <class S, class R>
int step_list_max_threads_t() {
  return StepBounds<S, R>::maxt;
}

// Resident blocks per SM of the work-list kernel at `threads` per block.
template <class S, class R>
cudaError_t step_list_occupancy_t(int K, int threads, int* blocks_per_sm) {
  switch (K) {
    case KFLAT:
      return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_step_list<S, R, KFLAT, false>, threads, 0);
    case KCYL:
      return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_step_list<S, R, KCYL, false>, threads, 0);
    case KELL:
      return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_step_list<S, R, KELL, false>, threads, 0);
    default:
      return cudaErrorInvalidValue;
  }
}

}  // namespace lbgm
