// Step kernels of 2-byte storage (FP16 / BF16 deviations, FP32 arithmetic):
// one thread updates the two nodes z, z + 1 (z even) of a row.
//
// With half the bytes of FP32 the one-node-per-thread step was bound by
// instruction issue (1340 instructions per update, DRAM 34 % busy). Two
// neighbours share their row addresses and predicates, a population of both
// is one 32-bit load or store where it is aligned, and the arithmetic runs in
// packed FP32x2 instructions (FFMA2, FADD2, FMUL2: two multiply-adds per
// issue slot at the same FP32 rate). The 41 gathered values stay packed in 41
// registers: they are unpacked once for the moments and again, one pair of
// velocities at a time, for the collision, which stores its results at once.
#pragma once

#include "kernels.cuh"

namespace lbgm {

// ---------------------------------------------------------------------------
// two nodes in one value
// ---------------------------------------------------------------------------
// Each lane of a PF2 is rounded like the scalar float instruction.
struct PF2 {
  float2 v;
  PF2() = default;
  __device__ __forceinline__ PF2(float2 a) : v(a) {}
  __device__ __forceinline__ PF2(float a, float b) : v(make_float2(a, b)) {}
  __device__ __forceinline__ explicit PF2(float a) : v(make_float2(a, a)) {}
  __device__ __forceinline__ explicit PF2(double c) : v(make_float2(float(c), float(c))) {}
};
// A product is a multiply-add of -0, from a constant the compiler cannot see
// through: CUDA 13.0's ptxas contracts mul.rn.f32x2 with the add.rn.f32x2 that
// uses it, -fmad=false and the rounding modifier or not, and a kernel's
// rounding would depend on where its compiler finds such pairs.
static __constant__ float2 c_neg_zero = {-0.0f, -0.0f};
__device__ __forceinline__ PF2 fmav(PF2 a, PF2 b, PF2 c) { return PF2(__ffma2_rn(a.v, b.v, c.v)); }
__device__ __forceinline__ PF2 operator+(PF2 a, PF2 b) { return PF2(__fadd2_rn(a.v, b.v)); }
__device__ __forceinline__ PF2 operator*(PF2 a, PF2 b) { return PF2(__ffma2_rn(a.v, b.v, c_neg_zero)); }
__device__ __forceinline__ PF2 operator-(PF2 a, PF2 b) { return fmav(b, PF2(-1.f, -1.f), a); }
__device__ __forceinline__ PF2 operator-(PF2 a) { return PF2(-a.v.x, -a.v.y); }
__device__ __forceinline__ PF2 rcpv(PF2 a) { return PF2(rcpv(a.v.x), rcpv(a.v.y)); }

// Packed storage of two values: unpack to FP32, pack rounding to nearest.
template <class S>
struct Pack2;
template <>
struct Pack2<__half> {
  __device__ static __forceinline__ PF2 unpack(uint32_t r) {
    return PF2(__half22float2(*reinterpret_cast<const __half2*>(&r)));
  }
  __device__ static __forceinline__ uint32_t pack(PF2 a) {
    const __half2 h = __float22half2_rn(a.v);
    return *reinterpret_cast<const uint32_t*>(&h);
  }
};
template <>
struct Pack2<__nv_bfloat16> {
  __device__ static __forceinline__ PF2 unpack(uint32_t r) {
    return PF2(__uint_as_float(r << 16), __uint_as_float(r & 0xffff0000u));
  }
  __device__ static __forceinline__ uint32_t pack(PF2 a) {
    const __nv_bfloat162 h = __float22bfloat162_rn(a.v);
    return *reinterpret_cast<const uint32_t*>(&h);
  }
};

// State reads: ordinary loads (gather_table).
__device__ __forceinline__ uint32_t ld16(const void* p) { return *static_cast<const unsigned short*>(p); }
__device__ __forceinline__ uint32_t ld32(const void* p) { return *static_cast<const uint32_t*>(p); }
__device__ __forceinline__ uint32_t join16(uint32_t lo, uint32_t hi) { return __byte_perm(lo, hi, 0x5410); }

// The gathered pair as the shell functions see it: reads unpack, results go
// straight to the output rows. EVEN (even n3): z and the row start are even,
// so a population of the pair is one aligned 32-bit word; else two 16-bit
// ones, the second absent at the end of an odd row.
template <class S, bool EVEN>
struct PairPop {
  uint32_t (&raw)[Q];
  S* out;
  uint32_t N, cell;
  bool first, second;
  template <int L>
  __device__ __forceinline__ PF2 get() const {
    return Pack2<S>::unpack(raw[L]);
  }
  template <int L>
  __device__ __forceinline__ void put(const PF2& v) const {
    const uint32_t w = Pack2<S>::pack(v);
    S* o = out + (uint32_t(L) * N + cell);
    if constexpr (EVEN) {
      if (first) *reinterpret_cast<uint32_t*>(o) = w;
    } else {
      unsigned short* u = reinterpret_cast<unsigned short*>(o);
      if (first) u[0] = static_cast<unsigned short>(w);
      if (second) u[1] = static_cast<unsigned short>(w >> 16);
    }
  }
};

// A pair's stream-table row in shared memory: both nodes' values of an entry
// next to each other (k_stream_table), so an entry is two 16-byte reads that
// are packed operands as they stand.
struct TabPair {
  const float4* st;
  int stride;
  __device__ __forceinline__ TabEntry<PF2> at(int k) const {
    const float4 a = st[(2 * k) * stride], b = st[(2 * k + 1) * stride];
    return {PF2(a.x, a.y), PF2(a.z, a.w), PF2(b.x, b.y), PF2(b.z, b.w)};
  }
};

__device__ __forceinline__ void copy_async16(float4* dst, const float4* __restrict__ src) {
  const uint32_t sa = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(sa), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_async_wait() {
  asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
}

// ---------------------------------------------------------------------------
// gather
// ---------------------------------------------------------------------------
// Streamed values of the pair far from every wall.
template <class S, bool EVEN>
__device__ __forceinline__ void gather_pair_far(const S* fin, const CellPos& p, bool second, const Dims& d,
                                                uint32_t (&raw)[Q]) {
  const uint32_t N = uint32_t(d.ncell);
  int rrow[7], tcol[7], zc[8];
#pragma unroll
  for (int c = -3; c <= 3; ++c) {
    rrow[c + 3] = (p.ir - c) * d.nt;
    tcol[c + 3] = wrap_small(p.it - c, d.nt);
  }
#pragma unroll
  for (int k = -3; k <= 4; ++k) {  // node z + k
    const int z = p.i3 + k;
    zc[k + 3] = d.periodic3 ? wrap_small(z, d.n3) : z;
  }
  raw[0] = EVEN ? ld32(fin + p.cell)
                : join16(ld16(fin + p.cell), ld16(fin + p.cell + (second ? 1 : 0)));
  static_for<0, 2 * NPAIR>([&](auto I_) {
    constexpr int I = decltype(I_)::value, P = I / 2, sg = I % 2 ? -1 : 1;
    using C = Pair<P>;
    constexpr int cx = sg * C::x, cy = sg * C::y, cz = sg * C::z, L = I + 1;
    const uint32_t row = uint32_t(L) * N + uint32_t((rrow[cx + 3] + tcol[cy + 3]) * d.n3);
    if constexpr (cz == 0 && EVEN) {
      raw[L] = ld32(fin + (row + uint32_t(p.i3)));
    } else {
      const int z0 = zc[3 - cz], z1 = EVEN || second ? zc[4 - cz] : z0;
      raw[L] = join16(ld16(fin + (row + uint32_t(z0))), ld16(fin + (row + uint32_t(z1))));
    }
  });
}

// Streamed values of the pair through the source table (gather_table), each
// node by its own key.
template <class S>
__device__ __forceinline__ void gather_pair_table(const S* fin, const CellPos& p, bool second, const Dims& d,
                                                  uint32_t (&raw)[Q]) {
  const int key = (axis_class(p.ir, d.nr) * d.src_nt + axis_class(p.it, d.nt)) * d.src_n3;
  const int one = second ? 1 : 0;
  const int4* __restrict__ r0 = d.src + (key + axis_class(p.i3, d.n3)) * SRC_ROW;
  const int4* __restrict__ r1 = d.src + (key + axis_class(p.i3 + one, d.n3)) * SRC_ROW;
  const int c0 = p.cell, c1 = p.cell + one;
  static_for<0, SRC_ROW>([&](auto J_) {
    constexpr int J = decltype(J_)::value;
    const int4 a = __ldg(r0 + J), b = __ldg(r1 + J);
    raw[4 * J] = join16(ld16(fin + uint32_t(c0 + a.x)), ld16(fin + uint32_t(c1 + b.x)));
    if constexpr (4 * J + 1 < Q) {
      raw[4 * J + 1] = join16(ld16(fin + uint32_t(c0 + a.y)), ld16(fin + uint32_t(c1 + b.y)));
      raw[4 * J + 2] = join16(ld16(fin + uint32_t(c0 + a.z)), ld16(fin + uint32_t(c1 + b.z)));
      raw[4 * J + 3] = join16(ld16(fin + uint32_t(c0 + a.w)), ld16(fin + uint32_t(c1 + b.w)));
    }
  });
}

template <int K, bool EVEN>
__device__ __forceinline__ NodeGeo<PF2, K> load_geo_pair(const GeoDev<float>& g, const Dims& d, const CellPos& p,
                                                         bool second) {
  NodeGeo<PF2, K> n;
  if constexpr (K == KELL) {
    const int row = p.ir * d.geo_rows3 + p.i3;
    auto two = [&](const float* a) {
      if constexpr (EVEN) return PF2(__ldg(reinterpret_cast<const float2*>(a + row)));
      else return PF2(__ldg(a + row), __ldg(a + row + (second ? 1 : 0)));
    };
    n.fth = two(g.fth);
    n.dtt = two(g.dtt);
    n.dpp = two(g.dpp);
    n.n_rtt = -two(g.g_rtt);
    n.n_trt = -two(g.g_trt);
    n.n_rpp = -two(g.g_rpp);
    n.n_prp = -two(g.g_prp);
    n.n_ttp = -two(g.g_ttp);
    n.n_ptt = -two(g.g_ptt);
  } else {
    const NodeGeo<float, K> a = load_geo<float, K>(g, p.ir);
    n.fth = PF2(a.fth);
    if constexpr (K == KCYL) {
      n.dtt = PF2(a.dtt);
      n.n_rtt = PF2(a.n_rtt);
      n.n_trt = PF2(a.n_trt);
    }
  }
  return n;
}

// ---------------------------------------------------------------------------
// the step
// ---------------------------------------------------------------------------
// One step of the pairs of warp `wrp` of one instance (state blocks fin and
// fout, reference table ref). `sm` is the block's staged rows; with `shared`
// (not ROW1) the block's warps lie in one (i_r, chunk) and stage its rows
// together.
template <typename S, int K, bool EVEN, bool ROW1>
__device__ __forceinline__ void step_pair(const S* fin, S* __restrict__ fout, const float* ref,
                                          const float4* __restrict__ st, const GeoDev<float>& geo,
                                          const InstParams<float>* __restrict__ inst, const Dims& d, uint32_t wrp,
                                          bool active, bool shared, float4* sm, int* __restrict__ flag) {
  const int lane = int(threadIdx.x & 31), wib = int(threadIdx.x >> 5);
  const int np = (d.n3 + 1) / 2;
  CellPos p;
  p.b = 0;
  bool live = active;
  TabPair tab;
  if (!active) wrp = 0;
  if constexpr (ROW1) {
    const uint32_t per = uint32_t(d.nt * np), wpl = (per + 31) / 32;
    p.ir = int(d.div_wl.div(wrp));
    uint32_t i = (wrp - uint32_t(p.ir) * wpl) * 32 + uint32_t(lane);
    if (i >= per) {
      live = false;
      i = per - 1;
    }
    p.it = int(d.div_np.div(i));
    p.i3 = 2 * int(i - uint32_t(p.it * np));
    float4* own = sm + wib * 2 * ST_K;
    if (lane < 2 * ST_K) copy_async16(own + lane, st + (lane * d.nr + p.ir));
    tab = {own, 1};
  } else {
    const uint32_t nch = uint32_t(np + 31) / 32, per = nch * uint32_t(d.nt);
    p.ir = int(d.div_wl.div(wrp));
    const uint32_t r = wrp - uint32_t(p.ir) * per;
    const int ch = int(d.div_nt.div(r));
    p.it = int(r) - ch * d.nt;
    int i = ch * 32 + lane;
    if (i >= np) {
      live = false;
      i = np - 1;
    }
    p.i3 = 2 * i;
    const float4* src = st + (p.ir * d.st_rows3 + (K == KELL ? i : pair_row(i, np)));
    const int stride = d.nr * d.st_rows3;
    float4* own = shared ? sm : sm + wib * 64 * ST_K;
    const int step = shared ? int(blockDim.x >> 5) : 1;
#pragma unroll 1
    for (int k = shared ? wib : 0; k < 2 * ST_K; k += step) copy_async16(own + k * 32 + lane, src + k * stride);
    tab = {own + lane, 32};
  }
  p.cell = (p.ir * d.nt + p.it) * d.n3 + p.i3;
  const bool pair = EVEN || p.i3 + 1 < d.n3;
  uint32_t raw[Q];
  bool near = near_wall(p, d);
  if constexpr (!ROW1) near = near || (!d.periodic3 && p.i3 + 1 > d.n3 - 4);
  chain_wait();
  if (__any_sync(0xffffffffu, near)) gather_pair_table<S>(fin, p, pair, d, raw);
  else gather_pair_far<S, EVEN>(fin, p, pair, d, raw);
  const InstParams<float> ip = *inst;
  const NodeGeo<PF2, K> g = load_geo_pair<K, EVEN>(geo, d, p, pair);
  copy_async_wait();
  if (!ROW1 && shared) __syncthreads();
  else __syncwarp();

  const PairPop<S, EVEN> pop{raw, fout, uint32_t(d.ncell), uint32_t(p.cell), live, live && pair};
  const TabEntry<PF2> ta = tab.at(0), tb = tab.at(1), tc = tab.at(2);
  const Moments<PF2> m0 = {ta.x, ta.y, ta.z, ta.w, tb.x, tb.y, tb.z, tb.w, tc.x, tc.y};
  const Moments<PF2> m = moments_shells<true, PF2>(pop, m0);
  if (live && !(finite_v(m.rho.v.x) && finite_v(pair ? m.rho.v.y : 0.0f))) {
    if (*flag == 0) atomicExch(flag, 1);
  }
  // keep the values packed across the moments (unpacked they would take 82 registers)
#pragma unroll
  for (int l = 0; l < Q; ++l) asm volatile("" : "+r"(raw[l]));
  const Coef<PF2> k = coefficients<PF2, K>(m, g, PF2(ip.kappa), PF2(ip.G));
  collide_shells<PF2, K>(pop, k, g, PF2(ip.omega), tab, tc.z);
  if (d.wall_eq && live) {
    // equilibrium-wall nodes leave the step as f^eq(rho', 0) of their own density
    const bool wr = p.ir == 0 || p.ir == d.nr - 1;
#pragma unroll 1
    for (int h = 0; h < (pair ? 2 : 1); ++h) {
      const int i3 = p.i3 + h;
      if (!wr && (d.periodic3 || (i3 != 0 && i3 != d.n3 - 1))) continue;
      CellPos ph = p;
      ph.i3 = i3;
      ph.cell = p.cell + h;
      float fe[Q];
      equilibrium<float, K>(h ? m.rho.v.y : m.rho.v.x, 0.0f, 0.0f, 0.0f,
                            load_geo<float, K>(geo, geo_row<K>(d, p.ir, i3)), fe);
      store_node<K>(fout, ref, ph, d, fe);
    }
  }
}

// Largest block and resident blocks per SM (168 registers, no spills).
// Measured on 24 64 x 4 x 256 channels in FP16, cylinder / four-wall ellipsoid,
// one launch a step: blocks of 128 threads, 3 / 4 / 5 of them 65 / 78, 68 / 97
// and 88 / 145 us a step (the last two spill); parking the gathered values in
// shared memory to fit 4 measured slower (109 / 126).
#ifndef LBGM_PAIR_MAXT
#define LBGM_PAIR_MAXT 128
#endif
#ifndef LBGM_PAIR_MINB
#define LBGM_PAIR_MINB 3
#endif

// Uniform batch: fin, fout are whole states, grid row y is instance y.
template <typename S, int K, bool EVEN, bool ROW1>
__global__ void __launch_bounds__(LBGM_PAIR_MAXT, LBGM_PAIR_MINB)
    k_step_pair(const S* fin, S* __restrict__ fout, GeoDev<float> geo,
                const InstParams<float>* __restrict__ inst, Dims d, int* __restrict__ flag, uint32_t warps,
                int shared) {
  extern __shared__ float4 sm[];
  chain_start();
  const uint32_t b = blockIdx.y, w = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const size_t base = size_t(b) * Q * uint32_t(d.ncell);
  step_pair<S, K, EVEN, ROW1>(fin + base, fout + base, ref_of(d, int(b)), stream_of(d, int(b)), geo, inst + b, d, w,
                              w < warps, shared != 0, sm, flag);
}

// Work list over instances of one metric kind and row parity (ListArgs; a tile
// is a number of warps).
template <typename S, int K, bool EVEN, bool ROW1>
__global__ void __launch_bounds__(LBGM_PAIR_MAXT, LBGM_PAIR_MINB)
    k_step_pair_list(const __grid_constant__ ListArgs<S, float> a) {
  extern __shared__ float4 sm[];
  chain_start();
  const int wpb = int(blockDim.x >> 5);
  for (int j = blockIdx.x; j < a.tile_start[a.count]; j += gridDim.x) {
    const int i = a.instance(j);
    const ListInst<S, float>& I = a.rec[i];
    const S* fin = a.parity ? I.f1 : I.f0;
    S* fout = const_cast<S*>(a.parity ? I.f0 : I.f1);
    const int warps = int(pair_warps(I.d)), first = (j - a.tile_start[i]) * a.tile;
    const bool shared = !ROW1 && I.d.nt % wpb == 0;
    for (int w0 = first; w0 < min(first + a.tile, warps); w0 += wpb) {
      if (j != int(blockIdx.x) || w0 != first) __syncthreads();  // the rows staged before have been read
      const int w = w0 + int(threadIdx.x >> 5);
      step_pair<S, K, EVEN, ROW1>(fin, fout, I.d.ref, I.d.st, I.geo, I.ip, I.d, uint32_t(w), w < warps, shared, sm,
                                  I.flag);
    }
  }
}

}  // namespace lbgm
