// Launchers of the fused step kernel for one storage type; each step_*.cu
// translation unit instantiates one so that the large unrolled kernel bodies
// compile in parallel.
#pragma once

#include <cstring>

#include "launch.h"
#include "pair.cuh"

namespace lbgm {

// Largest block of the step kernels (their launch bounds).
template <class S>
constexpr int step_max_threads() {
  return sizeof(S) == 2 ? LBGM_PAIR_MAXT : KBounds<S, KCYL>::maxt;
}

// Launch of a step kernel; `chained` if the launch before it on the stream is
// the step before (or host-synchronised work): the programmatic launch
// attribute lets the kernel start early (chain_wait). Not for streams that run
// beside others: blocks that wait would hold the other streams' slots.
template <class... P, class... A>
cudaError_t launch_chained(void (*kern)(P...), dim3 grid, int threads, size_t smem, cudaStream_t s, bool chained,
                           A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(unsigned(threads));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr = {};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = chained ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, P(args)...);
}

template <class R>
cudaError_t launch_step_t(int K, const R* fin, R* fout, const GeoDev<R>& geo, const InstParams<R>* inst,
                          const Dims& d, int* flag, int threads, bool chained, cudaStream_t s) {
  if (d.batch < 1 || d.batch > 65535) return cudaErrorInvalidValue;
  threads = threads < step_max_threads<R>() ? threads : step_max_threads<R>();
  const dim3 blocks((uint32_t(d.ncell) + threads - 1) / threads, uint32_t(d.batch));
  switch (K) {
    case KFLAT: return launch_chained(k_step<R, KFLAT>, blocks, threads, 0, s, chained, fin, fout, geo, inst, d, flag);
    case KCYL: return launch_chained(k_step<R, KCYL>, blocks, threads, 0, s, chained, fin, fout, geo, inst, d, flag);
    case KELL: return launch_chained(k_step<R, KELL>, blocks, threads, 0, s, chained, fin, fout, geo, inst, d, flag);
    case KELT: return launch_chained(k_step<R, KELT>, blocks, threads, 0, s, chained, fin, fout, geo, inst, d, flag);
    default: return cudaErrorInvalidValue;
  }
}

// Warps per block of the pair kernels and whether its warps share their
// staged rows: as many warps as asked for where they all lie in one
// (i_r, chunk) (ntheta a multiple of them) or need one row each, else pairs of
// warps (26.6 KB of staged rows a block unless they share them).
inline int pair_block(const Dims& d, int threads, bool* shared) {
  int w = (threads < LBGM_PAIR_MAXT ? threads : LBGM_PAIR_MAXT) / 32;
  *shared = false;
  if (d.st_row_r) return w;
  if (d.nt % w != 0) w = 2;
  *shared = d.nt % w == 0;
  return w;
}

// f(EVEN, ROW1) with the dispatch's compile-time choices for d.
template <int K, class F>
cudaError_t pair_dispatch(const Dims& d, F&& f) {
  const bool even = d.n3 % 2 == 0;
  if constexpr (K != KELL) {
    if (d.st_row_r)
      return even ? f(std::true_type{}, std::true_type{}) : f(std::false_type{}, std::true_type{});
  }
  return even ? f(std::true_type{}, std::false_type{}) : f(std::false_type{}, std::false_type{});
}

template <class S, int K>
cudaError_t launch_pair_k(const S* fin, S* fout, const GeoDev<float>& geo, const InstParams<float>* inst,
                          const Dims& d, int* flag, int threads, bool chained, cudaStream_t s) {
  return pair_dispatch<K>(d, [&](auto even, auto row1) {
    constexpr bool EVEN = decltype(even)::value, ROW1 = decltype(row1)::value;
    bool shared;
    const int w = pair_block(d, threads, &shared);
    const uint32_t warps = pair_warps(d);
    const dim3 grid((warps + w - 1) / w, uint32_t(d.batch));
    const size_t smem = pair_smem_bytes(d, w);
    return launch_chained(k_step_pair<S, K, EVEN, ROW1>, grid, w * 32, smem, s, chained, fin, fout, geo, inst, d, flag,
                          warps, shared ? 1 : 0);
  });
}

template <class S>
cudaError_t launch_pair_t(int K, const S* fin, S* fout, const GeoDev<float>& geo, const InstParams<float>* inst,
                          const Dims& d, int* flag, int threads, bool chained, cudaStream_t s) {
  if (d.batch < 1 || d.batch > 65535) return cudaErrorInvalidValue;
  switch (K) {
    case KFLAT: return launch_pair_k<S, KFLAT>(fin, fout, geo, inst, d, flag, threads, chained, s);
    case KCYL: return launch_pair_k<S, KCYL>(fin, fout, geo, inst, d, flag, threads, chained, s);
    case KELL: return launch_pair_k<S, KELL>(fin, fout, geo, inst, d, flag, threads, chained, s);
    default: return cudaErrorInvalidValue;
  }
}

// The arguments of one work-list launch over `count` records (at most
// ListArgs::N) of `items` tiles each.
template <class S, class R>
ListArgs<S, R> list_args(const void* recs, int count, const int* items, int tile, int parity) {
  ListArgs<S, R> a;
  std::memcpy(a.rec, recs, size_t(count) * sizeof(a.rec[0]));
  a.tile_start[0] = 0;
  for (int i = 0; i < count; ++i) a.tile_start[i + 1] = a.tile_start[i] + items[i];
  a.count = count;
  a.tile = tile;
  a.parity = parity;
  return a;
}

// grid 0: one block per work item; otherwise `grid` persistent blocks.
template <class R>
cudaError_t launch_step_list_t(int K, const void* recs, int count, const int* items, int tile, int threads, int grid,
                               int parity, bool chained, cudaStream_t s) {
  const ListArgs<R, R> a = list_args<R, R>(recs, count, items, tile, parity);
  const int n = a.tile_start[count], g = grid > 0 && grid < n ? grid : n;
  const bool loop = g < n || tile > threads;
#define LB_LIST(KK)                                                                         \
  return loop ? launch_chained(k_step_list<R, KK, true>, dim3(g), threads, 0, s, chained, a) \
              : launch_chained(k_step_list<R, KK, false>, dim3(g), threads, 0, s, chained, a)
  switch (K) {
    case KFLAT: LB_LIST(KFLAT);
    case KCYL: LB_LIST(KCYL);
    case KELL: LB_LIST(KELL);
    default: return cudaErrorInvalidValue;
  }
#undef LB_LIST
}

// The same for 2-byte storage; `d` is any instance of the group (one metric
// kind, row kind and parity of n3), smem the group's staged rows in bytes.
template <class S, int K>
cudaError_t launch_pair_list_k(const Dims& d, size_t smem, const ListArgs<S, float>& a, int threads, int grid,
                               bool chained, cudaStream_t s) {
  const int n = a.tile_start[a.count], g = grid > 0 && grid < n ? grid : n;
  return pair_dispatch<K>(d, [&](auto even, auto row1) {
    constexpr bool EVEN = decltype(even)::value, ROW1 = decltype(row1)::value;
    auto kern = k_step_pair_list<S, K, EVEN, ROW1>;
    if (smem > 40 * 1024) {
      cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
      if (e != cudaSuccess) return e;
    }
    return launch_chained(kern, dim3(g), threads, smem, s, chained, a);
  });
}

template <class S>
cudaError_t launch_pair_list_t(int K, const Dims& d, size_t smem, const void* recs, int count, const int* items,
                               int tile, int threads, int grid, int parity, bool chained, cudaStream_t s) {
  const ListArgs<S, float> a = list_args<S, float>(recs, count, items, tile, parity);
  switch (K) {
    case KFLAT: return launch_pair_list_k<S, KFLAT>(d, smem, a, threads, grid, chained, s);
    case KCYL: return launch_pair_list_k<S, KCYL>(d, smem, a, threads, grid, chained, s);
    case KELL: return launch_pair_list_k<S, KELL>(d, smem, a, threads, grid, chained, s);
    default: return cudaErrorInvalidValue;
  }
}

// Resident blocks per SM of the work-list kernel at `threads` per block.
template <class R>
cudaError_t step_list_occupancy_t(int K, int threads, int* out) {
  switch (K) {
    case KFLAT: return cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, k_step_list<R, KFLAT, false>, threads, 0);
    case KCYL: return cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, k_step_list<R, KCYL, false>, threads, 0);
    case KELL: return cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, k_step_list<R, KELL, false>, threads, 0);
    default: return cudaErrorInvalidValue;
  }
}

template <class S>
cudaError_t pair_list_occupancy_t(int K, const Dims& d, size_t smem, int threads, int* out) {
  auto occ = [&](auto kk) {
    constexpr int KK = decltype(kk)::value;
    return pair_dispatch<KK>(d, [&](auto even, auto row1) {
      return cudaOccupancyMaxActiveBlocksPerMultiprocessor(
          out, k_step_pair_list<S, KK, decltype(even)::value, decltype(row1)::value>, threads, smem);
    });
  };
  switch (K) {
    case KFLAT: return occ(std::integral_constant<int, KFLAT>{});
    case KCYL: return occ(std::integral_constant<int, KCYL>{});
    case KELL: return occ(std::integral_constant<int, KELL>{});
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace lbgm
