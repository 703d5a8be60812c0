// Device building blocks of the lattice Boltzmann update in generalized
// metrics (Sec. II of the paper): pull streaming with full bounce-back along
// the path, moments, equilibrium, non-equilibrium stress, forcing term, BGK.
//
// Arithmetic is organised per velocity pair (c, -c): every term is either even
// or odd in c, so each pair costs one evaluation of the even part E and of
// the odd part O, and f(+c) uses E + O while f(-c) uses E - O.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <cstdint>
#include <type_traits>

#include "collision.cuh"

namespace lbgm {

// ---------------------------------------------------------------------------
// launch geometry
// ---------------------------------------------------------------------------
// Division by a runtime-invariant unsigned integer (round-up multiply-shift).
struct FastDiv {
  uint32_t d, mul, shift;
  __host__ static FastDiv make(uint32_t d_) {
    FastDiv f{d_, 0u, 0u};
    if (d_ == 1) return f;
    uint32_t l = 0;
    while ((1ull << l) < d_) ++l;
    f.shift = l - 1;
    f.mul = uint32_t(((1ull << (32 + l)) + d_ - 1) / d_ - (1ull << 32));
    return f;
  }
  __device__ __forceinline__ uint32_t div(uint32_t n) const {
    if (d == 1) return n;
    uint32_t t = __umulhi(n, mul);
    return (t + ((n - t) >> 1)) >> shift;
  }
};

struct Dims {
  int nr, nt, n3;
  int ncell;       // nr * nt * n3 (one instance)
  int periodic3;   // 0: walls on x3
  int batch;
  int geo_rows3;   // geometry rows per i_r: n3 for the ellipsoid's (r, x3)
                   // rows, nt n3 for the theta-resolved one, 1 otherwise
  FastDiv div_ncell, div_n3, div_nt;
  // 2-byte storage: reference populations over the nr * geo_rows3 geometry
  // rows, per instance (ref_index; NULL for FP32 / FP64 storage)
  const float* ref;
  int wall_eq;     // 1: equilibrium (Dirichlet) walls on the end nodes
  // 2-byte storage: the stream table of each instance (stream_of; NULL for
  // FP32 / FP64 storage) over nr * st_rows3 stream rows, and the divisors of
  // the pair kernels' node numbering
  const float4* st;
  int st_rows3;    // rows per i_r: 1, the x3 pairs (n3 + 1) / 2, or their kinds (pair_rows)
  int st_row_r;    // 1: rows of i_r alone (flat and cylinder, periodic x3)
  FastDiv div_np, div_wl;  // x3 pairs per line, warps per i_r layer
  int geo_theta;   // 1: geometry rows (and observable weights) per node
  // source table (gather_table): SRC_ROW offsets per key of node classes
  const int4* src;
  int src_nt, src_n3;  // theta and x3 classes (the key's radices)
};

// Node class along an axis of n nodes: which of a node's sources lie beyond
// an end of the axis depends only on its distance to the ends, up to 3 nodes
// -- 0, 1, 2 (first nodes), 3 (inside), 4, 5, 6 (last nodes); every node is
// its own class on an axis shorter than 7.
__host__ __device__ __forceinline__ int axis_classes(int n) { return n < 7 ? n : 7; }
__host__ __device__ __forceinline__ int axis_class(int i, int n) {
  return n < 7 || i < 3 ? i : (i > n - 4 ? i - n + 7 : 3);
}
// A node of class c.
__host__ __device__ __forceinline__ int axis_class_node(int c, int n) { return n < 7 || c <= 3 ? c : n - 7 + c; }
// Stream rows of an i_r layer between x3 walls where the metric does not depend
// on x3 (flat, cylinder; np pairs of nodes along x3): the first two pairs, those
// whose nodes are all of class 3, the last two. With a row for every pair the
// table was larger than the state (416 B a pair; 259 MB for 24 cylinders of
// 130 x 1 x 400, 6.5 MB now), and lb_init of those, which writes it, took 356 us
// (now 178).
__host__ __device__ __forceinline__ int pair_rows(int np) { return np < 5 ? np : 5; }
__host__ __device__ __forceinline__ int pair_row(int i, int np) {
  return np < 5 || i < 2 ? i : (i >= np - 2 ? i - np + 5 : 2);
}
// A pair of row r.
__host__ __device__ __forceinline__ int pair_of_row(int r, int np) { return np < 5 || r < 3 ? r : np - 5 + r; }
constexpr int SRC_ROW = 11;  // int4 per key: 41 offsets, padded

// Index of reference population l of geometry row r in an instance's table:
// row-major [r][l] where rows are i_r only (cylinder, flat: a warp shares
// the row, and the offsets of a node's 41 entries are compile-time
// constants), population-major [l][r] for the ellipsoid's (i_r, i_3) rows
// (consecutive nodes read consecutive rows).
template <int K>
__device__ __forceinline__ uint32_t ref_index(const Dims& d, int l, int row) {
  if constexpr (K == KELL) return uint32_t(l) * uint32_t(d.nr) * uint32_t(d.geo_rows3) + uint32_t(row);
  else return uint32_t(row) * 41u + uint32_t(l);
}

// Geometry row of node (i_r, i_3): i_r * n3 + i_3 for the ellipsoid, i_r
// otherwise.
template <int K>
__device__ __forceinline__ int geo_row(const Dims& d, int ir, int i3) {
  if constexpr (K == KELL) return ir * d.geo_rows3 + i3;
  else return ir;
}

// Geometry row of node p for metric kind K: i_r (flat, cylinder), (i_r, i_3)
// (ellipsoid), the node itself (theta-resolved ellipsoid).
template <int K>
__device__ __forceinline__ int geo_row_node(const Dims& d, int ir, int it, int i3) {
  if constexpr (K == KELL) return ir * d.geo_rows3 + i3;
  else if constexpr (K == KELT) return ir * d.geo_rows3 + it * d.n3 + i3;
  else return ir;
}

// Reference table of instance b (see Dims::ref).
__device__ __forceinline__ const float* ref_of(const Dims& d, int b) {
  return d.ref ? d.ref + size_t(b) * 41 * size_t(d.nr) * size_t(d.geo_rows3) : nullptr;
}

// Stream table of instance b (2-byte storage). Which stored population (and
// whose geometry row's reference) a node receives in streaming does not
// depend on theta, and for the flat channel and the cylinder with a periodic
// x3 not on x3 either: a stream row is an i_r layer there, between x3 walls a
// kind of pair of the layer (pair_rows), in the ellipsoid the pair (i_3 = 2 p,
// 2 p + 1) of an (i_r, x3) line. A row holds 13 entries of 4
// values for both nodes of the pair, stored [2 k + half][row] as float4 (x of
// both nodes, y of both) and (z of both, w of both): consecutive pairs are
// consecutive float4. Entry k (f_l = w_l g_l + rho_l: g the stored deviation,
// rho_l the reference population of the stored value the node receives as
// population l, t_l = ((1 - omega) rho_l - r_l) / w_l with r_l the node's own
// reference):
//   k = 0: sum rho_l, sum c^x rho_l, sum c^y rho_l, sum c^z rho_l
//   k = 1: sum c^x c^x rho_l, c^y c^y, c^z c^z, c^x c^y
//   k = 2: sum c^x c^z rho_l, sum c^y c^z rho_l, t_0, 0
//   k = 3 + j, j = 0..9: E and O of slot 2 j, then of slot 2 j + 1. A slot
//           belongs to a pair (t_+ of population 2 P + 1, t_- of 2 P + 2) and
//           E, O hold te = (t_+ + t_-) / 2 and to = (t_+ - t_-) / 2 in
//           the coefficient space of the pair's shell: te, to themselves on
//           the axes; half sum and half difference of a face's two pairs; the
//           4-point Hadamard transform over 4 of a body shell's four
constexpr int ST_K = 13;
__device__ __forceinline__ const float4* stream_of(const Dims& d, int b) {
  return d.st + size_t(b) * 2 * ST_K * size_t(d.nr) * size_t(d.st_rows3);
}

// Geometry rows in the compute precision. A row is i_r * geo_rows3 + i_3 (or
// i_r). Only the components that are non-zero for the metric kind are read:
// every other Delta^ij, Gamma^i_jk and g^{i theta} is zero at theta = 0.
template <typename Real>
struct GeoDev {
  const Real* dtt;    // Delta^{theta theta}
  const Real* dpp;    // Delta^{33}
  const Real* g_rtt;  // h Gamma^r_{theta theta}
  const Real* g_rpp;  // h Gamma^r_{33}
  const Real* g_trt;  // h Gamma^theta_{r theta}
  const Real* g_prp;  // h Gamma^3_{r 3}
  const Real* g_ttp;  // h Gamma^theta_{theta 3}
  const Real* g_ptt;  // h Gamma^3_{theta theta}
  const Real* fth;    // g^{theta theta}
  // theta-resolved ellipsoid only: Delta^rr, Delta^{r theta}, Delta^{r 3},
  // Delta^{theta 3}, g^{r theta}, g^{3 theta} at ext + j * ext_stride
  const Real* ext;
  uint32_t ext_stride;
};

template <typename Real>
struct InstParams {
  Real omega;  // 1 / tau
  Real kappa;  // 1 - 1/(2 tau) (improved forcing) or 0 (old forcing)
  Real G;      // covariant streamwise force per step
  Real pad;
};

struct CellPos {
  int b, cell, ir, it, i3;
};

// Position of node `cell` of instance b.
__device__ __forceinline__ CellPos locate_cell(const Dims& d, int b, uint32_t cell) {
  CellPos p;
  p.b = b;
  p.cell = int(cell);
  uint32_t row = d.div_n3.div(cell);
  p.i3 = p.cell - int(row) * d.n3;
  p.ir = int(d.div_nt.div(row));
  p.it = int(row) - p.ir * d.nt;
  return p;
}

__device__ __forceinline__ CellPos locate(const Dims& d, uint32_t t) {
  CellPos p;
  p.b = int(d.div_ncell.div(t));
  p.cell = int(t) - p.b * d.ncell;
  uint32_t row = d.div_n3.div(uint32_t(p.cell));
  p.i3 = p.cell - int(row) * d.n3;
  p.ir = int(d.div_nt.div(row));
  p.it = int(row) - p.ir * d.nt;
  return p;
}

// ---------------------------------------------------------------------------
// population storage
// ---------------------------------------------------------------------------
// Codec<S, R> reads populations stored as S into the compute type R and back.
// For the reduced-precision formats the stored value is the scaled deviation
// (f_l - r_l) / w_l from a reference population r_l of the storing node's
// geometry row (a table entry, passed as a pointer), so every stored number
// is small whatever its weight: f_l = w_l s_l + r_l. With r_l = w_l this is
// the deviation from the rest state of unit density.
template <class S, class R>
struct Codec {
  static constexpr bool uses_ref = false;
  template <int L>
  __device__ static __forceinline__ R dec(S v, const float*) { return R(v); }
  template <int L>
  __device__ static __forceinline__ S enc(R f, const float*) { return S(f); }
};
template <>
struct Codec<__half, float> {
  static constexpr bool uses_ref = true;
  template <int L>
  __device__ static __forceinline__ float dec(__half v, const float* ref) {
    constexpr float w = float(WeightOf<L>::w);
    return fmaf(w, __half2float(v), __ldg(ref));
  }
  template <int L>
  __device__ static __forceinline__ __half enc(float f, const float* ref) {
    constexpr float iw = float(1.0 / WeightOf<L>::w);
    return __float2half_rn((f - __ldg(ref)) * iw);
  }
};
template <>
struct Codec<__nv_bfloat16, float> {
  static constexpr bool uses_ref = true;
  template <int L>
  __device__ static __forceinline__ float dec(__nv_bfloat16 v, const float* ref) {
    constexpr float w = float(WeightOf<L>::w);
    return fmaf(w, __bfloat162float(v), __ldg(ref));
  }
  template <int L>
  __device__ static __forceinline__ __nv_bfloat16 enc(float f, const float* ref) {
    constexpr float iw = float(1.0 / WeightOf<L>::w);
    return __float2bfloat16_rn((f - __ldg(ref)) * iw);
  }
};

// ---------------------------------------------------------------------------
// pull streaming
// ---------------------------------------------------------------------------
// periodic wrap of v in [-3, n + 3) onto [0, n)
__device__ __forceinline__ int wrap_small(int v, int n) {
  if (n >= 3) {
    v += (v < 0) ? n : 0;
    v -= (v >= n) ? n : 0;
    return v;
  }
  v %= n;
  return v < 0 ? v + n : v;
}

// Node offsets of the sources of one node far from every wall:
// source of population c is x - c (periodic in theta, and in x3 if periodic).
struct Neighbours {
  int rrow[7];  // (i_r - c) * nt for c = -3..3 (index c + 3)
  int tcol[7];  // wrap(i_t - c)
  int zcol[7];  // i_3 - c, wrapped if periodic
};

__device__ __forceinline__ void make_neighbours(const CellPos& p, const Dims& d, Neighbours& n) {
#pragma unroll
  for (int c = -3; c <= 3; ++c) {
    n.rrow[c + 3] = (p.ir - c) * d.nt;
    n.tcol[c + 3] = wrap_small(p.it - c, d.nt);
    int z = p.i3 - c;
    n.zcol[c + 3] = d.periodic3 ? wrap_small(z, d.n3) : z;
  }
}

template <int CX, int CY, int CZ>
__device__ __forceinline__ int src_far(const Neighbours& n, const Dims& d) {
  return (n.rrow[CX + 3] + n.tcol[CY + 3]) * d.n3 + n.zcol[CZ + 3];
}

// Source of population c arriving at a node near a wall. The population's
// path is a straight line x + q * sigma (sigma = c / s, q in lattice units
// along each non-zero axis); a wall reverses the whole velocity, so the path
// folds back and forth on the interval of the line inside the walls. In
// half-node units Q = 2 q the walls are odd integers lo < 0 < hi. Going back
// one time step means moving 2 s towards negative Q; each fold flips the
// population to its opposite.
__device__ __forceinline__ int src_wall(int cx, int cy, int cz, int s, const CellPos& p, const Dims& d, bool& flip,
                                        int& src_ir, int& src_i3) {
  const int sx = (cx > 0) - (cx < 0), sy = (cy > 0) - (cy < 0), sz = (cz > 0) - (cz < 0);
  int lo = -(1 << 30), hi = (1 << 30);
  if (sx != 0) {
    const int l_ = sx > 0 ? -1 - 2 * p.ir : 2 * p.ir + 1 - 2 * d.nr;
    const int h_ = sx > 0 ? 2 * d.nr - 1 - 2 * p.ir : 2 * p.ir + 1;
    lo = max(lo, l_);
    hi = min(hi, h_);
  }
  if (sz != 0 && !d.periodic3) {
    const int l_ = sz > 0 ? -1 - 2 * p.i3 : 2 * p.i3 + 1 - 2 * d.n3;
    const int h_ = sz > 0 ? 2 * d.n3 - 1 - 2 * p.i3 : 2 * p.i3 + 1;
    lo = max(lo, l_);
    hi = min(hi, h_);
  }
  const int D = 2 * s;
  int Qe;
  flip = false;
  if (-D >= lo) {
    Qe = -D;
  } else {
    int v = D + lo;  // distance left after the first fold (odd, < D)
    const int L = hi - lo;
    int k = 0;
    while (v > L) {  // at most D / 2 iterations
      v -= L;
      ++k;
    }
    flip = (k & 1) == 0;  // k + 1 folds
    Qe = (k & 1) ? hi - v : lo + v;
  }
  const int q = Qe / 2;
  const int yr = p.ir + q * sx;
  const int yt = wrap_small(p.it + q * sy, d.nt);
  int yz = p.i3 + q * sz;
  if (d.periodic3) yz = wrap_small(yz, d.n3);
  src_ir = yr;
  src_i3 = yz;
  return (yr * d.nt + yt) * d.n3 + yz;
}

__device__ __forceinline__ bool near_wall(const CellPos& p, const Dims& d) {
  return p.ir < 3 || p.ir > d.nr - 4 || (!d.periodic3 && (p.i3 < 3 || p.i3 > d.n3 - 4));
}

// Visit the sources of the 41 streamed populations of node p: fn(L, src,
// sl, row) with L a std::integral_constant (the population received), src
// the address in fin (one instance's block: population l of cell c at
// fin[l * ncell + c]) of the post-collision value it is streamed from, sl
// the population index stored there (L, or its opposite after a fold) and
// row the geometry row of the node that stored it (sl and row select the
// reference population of 2-byte storage). Near a wall every moving
// population comes from its (possibly folded) source; opposite velocities
// share their weight. Offsets are
// 32-bit: an instance block holds fewer than 2^32 bytes (checked when the
// context is created).
template <int K, class S, class Fn>
__device__ __forceinline__ void for_each_source_far(const S* fin, const CellPos& p, const Dims& d, Fn&& fn) {
  const uint32_t N = uint32_t(d.ncell);
  Neighbours nb;
  make_neighbours(p, d, nb);
  static_for<0, NPAIR>([&](auto P_) {
    constexpr int P = decltype(P_)::value;
    using C = Pair<P>;
    const uint32_t sp = uint32_t(src_far<C::x, C::y, C::z>(nb, d));
    const uint32_t sm = uint32_t(src_far<-C::x, -C::y, -C::z>(nb, d));
    fn(std::integral_constant<int, 2 * P + 1>{}, fin + ((2 * P + 1) * N + sp), 2 * P + 1,
       geo_row<K>(d, p.ir - C::x, nb.zcol[C::z + 3]));
    fn(std::integral_constant<int, 2 * P + 2>{}, fin + ((2 * P + 2) * N + sm), 2 * P + 2,
       geo_row<K>(d, p.ir + C::x, nb.zcol[-C::z + 3]));
  });
}

// Equilibrium walls: the source x - c with walled axes clamped onto the
// wall layer (periodic axes wrapped); no flip.
template <int K, class S, class Fn>
__device__ __forceinline__ void for_each_source_clamped(const S* __restrict__ fin, const CellPos& p,
                                                        const Dims& d, Fn&& fn) {
  const uint32_t N = uint32_t(d.ncell);
  auto src = [&](int cx, int cy, int cz, int& yr, int& yz) {
    yr = min(max(p.ir - cx, 0), d.nr - 1);
    const int yt = wrap_small(p.it - cy, d.nt);
    yz = p.i3 - cz;
    yz = d.periodic3 ? wrap_small(yz, d.n3) : min(max(yz, 0), d.n3 - 1);
    return uint32_t((yr * d.nt + yt) * d.n3 + yz);
  };
  static_for<0, NPAIR>([&](auto P_) {
    constexpr int P = decltype(P_)::value;
    using C = Pair<P>;
    int rp, zp, rm, zm;
    const uint32_t sp = src(C::x, C::y, C::z, rp, zp);
    const uint32_t sm = src(-C::x, -C::y, -C::z, rm, zm);
    fn(std::integral_constant<int, 2 * P + 1>{}, fin + ((2 * P + 1) * N + sp), 2 * P + 1, geo_row<K>(d, rp, zp));
    fn(std::integral_constant<int, 2 * P + 2>{}, fin + ((2 * P + 2) * N + sm), 2 * P + 2, geo_row<K>(d, rm, zm));
  });
}

template <int K, class S, class Fn>
__device__ __forceinline__ void for_each_source_wall(const S* __restrict__ fin, const CellPos& p, const Dims& d,
                                                     Fn&& fn) {
  if (d.wall_eq) {
    for_each_source_clamped<K>(fin, p, d, fn);
    return;
  }
  const uint32_t N = uint32_t(d.ncell);
  static_for<0, NPAIR>([&](auto P_) {
    constexpr int P = decltype(P_)::value;
    using C = Pair<P>;
    bool fp, fm;
    int rp, zp, rm, zm;
    const uint32_t sp = uint32_t(src_wall(C::x, C::y, C::z, C::s, p, d, fp, rp, zp));
    const uint32_t sm = uint32_t(src_wall(-C::x, -C::y, -C::z, C::s, p, d, fm, rm, zm));
    const int lp = fp ? 2 * P + 2 : 2 * P + 1, lm = fm ? 2 * P + 1 : 2 * P + 2;
    fn(std::integral_constant<int, 2 * P + 1>{}, fin + (lp * N + sp), lp, geo_row<K>(d, rp, zp));
    fn(std::integral_constant<int, 2 * P + 2>{}, fin + (lm * N + sm), lm, geo_row<K>(d, rm, zm));
  });
}

template <int K, class S, class Fn>
__device__ __forceinline__ void for_each_source(const S* __restrict__ fin, const CellPos& p, const Dims& d,
                                                Fn&& fn) {
  fn(std::integral_constant<int, 0>{}, fin + uint32_t(p.cell), 0, geo_row<K>(d, p.ir, p.i3));
  if (!near_wall(p, d))
    for_each_source_far<K>(fin, p, d, fn);
  else
    for_each_source_wall<K>(fin, p, d, fn);
}

// Sources for a node J = 0, 1, 2 layers from the r-wall on side SIDE (0: low,
// 1: high), at least 3 layers from the x3-walls (or x3 periodic), nr >= 7:
// only that wall can lie on a population's one-step path, so the wall rule of
// src_wall reduces to constants. A population whose backward path (along -c,
// length s = |c|_inf) meets the wall 2 J + 1 half-nodes away folds once: its
// source is x + (s - 1 - 2 J) sigma (sigma = c / s) and it arrives flipped;
// every other population comes from x - c as away from walls.
template <int SIDE, int J, int CX, int CY, int CZ, int S>
struct LayerFold {
  static constexpr int sx = (CX > 0) - (CX < 0), sy = (CY > 0) - (CY < 0), sz = (CZ > 0) - (CZ < 0);
  static constexpr bool hit = ((SIDE == 0 && sx > 0) || (SIDE == 1 && sx < 0)) && (2 * S > 1 + 2 * J);
  static constexpr int q = hit ? S - 1 - 2 * J : -S;
  static constexpr int dx = q * sx, dy = q * sy, dz = q * sz;  // source - node
};

template <int K, int SIDE, int J, class S, class Fn>
__device__ __forceinline__ void for_each_source_layer(const S* __restrict__ fin, const CellPos& p,
                                                      const Dims& d, Fn&& fn) {
  const uint32_t N = uint32_t(d.ncell);
  Neighbours nb;
  make_neighbours(p, d, nb);
  static_for<0, NPAIR>([&](auto P_) {
    constexpr int P = decltype(P_)::value;
    using C = Pair<P>;
    using Fp = LayerFold<SIDE, J, C::x, C::y, C::z, C::s>;
    using Fm = LayerFold<SIDE, J, -C::x, -C::y, -C::z, C::s>;
    const uint32_t sp = uint32_t((nb.rrow[3 - Fp::dx] + nb.tcol[3 - Fp::dy]) * d.n3 + nb.zcol[3 - Fp::dz]);
    const uint32_t sm = uint32_t((nb.rrow[3 - Fm::dx] + nb.tcol[3 - Fm::dy]) * d.n3 + nb.zcol[3 - Fm::dz]);
    constexpr int lp = Fp::hit ? 2 * P + 2 : 2 * P + 1, lm = Fm::hit ? 2 * P + 1 : 2 * P + 2;
    fn(std::integral_constant<int, 2 * P + 1>{}, fin + (lp * N + sp), lp,
       geo_row<K>(d, p.ir + Fp::dx, nb.zcol[3 - Fp::dz]));
    fn(std::integral_constant<int, 2 * P + 2>{}, fin + (lm * N + sm), lm,
       geo_row<K>(d, p.ir + Fm::dx, nb.zcol[3 - Fm::dz]));
  });
}

// Decoding visitor: f[L] from the stored value at src, with the reference
// row table ref (instance base; NULL for FP32 / FP64 storage).
template <int K, class S, class R>
struct DecodeInto {
  R (&f)[Q];
  const float* ref;
  const Dims& d;
  template <class LC>
  __device__ __forceinline__ void operator()(LC, const S* src, int sl, int row) const {
    constexpr int L = LC::value;
    if constexpr (Codec<S, R>::uses_ref)
      f[L] = Codec<S, R>::template dec<L>(__ldg(src), ref + ref_index<K>(d, sl, row));
    else
      f[L] = Codec<S, R>::template dec<L>(__ldg(src), nullptr);
  }
};

// Streamed populations of a node within 3 layers of an r-wall (x3 periodic or
// the node at least 3 layers from the x3-walls, nr >= 7) through the
// per-layer constant folds.
template <int K, class S, class Put>
__device__ __forceinline__ void gather_edge(const S* __restrict__ fin, const CellPos& p, const Dims& d,
                                            const Put& put) {
  put(std::integral_constant<int, 0>{}, fin + uint32_t(p.cell), 0, geo_row<K>(d, p.ir, p.i3));
  const int side = p.ir < 3 ? 0 : 1;
  const int j = side == 0 ? p.ir : d.nr - 1 - p.ir;
  switch (side * 3 + j) {
    case 0: for_each_source_layer<K, 0, 0>(fin, p, d, put); break;
    case 1: for_each_source_layer<K, 0, 1>(fin, p, d, put); break;
    case 2: for_each_source_layer<K, 0, 2>(fin, p, d, put); break;
    case 3: for_each_source_layer<K, 1, 0>(fin, p, d, put); break;
    case 4: for_each_source_layer<K, 1, 1>(fin, p, d, put); break;
    default: for_each_source_layer<K, 1, 2>(fin, p, d, put); break;
  }
}

// Load the 41 streamed populations of node p from the post-collision state
// (instance block fin, reference table ref), decoded (the observables and the
// half-force variant's step). Near an r-wall with bounce-back walls, at least
// 3 nodes away from any x3 wall, only the r-wall can lie on a population's
// path, and the compile-time folds of gather_edge replace the general wall
// rule (the same sources, fewer instructions).
template <int K, class S, class R>
__device__ __forceinline__ void gather(const S* __restrict__ fin, const float* ref, const CellPos& p,
                                       const Dims& d, R (&f)[Q]) {
  const DecodeInto<K, S, R> put{f, ref, d};
  const bool x3_clear = d.periodic3 || (p.i3 >= 3 && p.i3 <= d.n3 - 4);
  if (!d.wall_eq && d.nr >= 7 && x3_clear && (p.ir < 3 || p.ir > d.nr - 4)) {
    gather_edge<K>(fin, p, d, put);
    return;
  }
  for_each_source<K>(fin, p, d, put);
}

// The streamed populations of node p through the source table: entry L of the
// node's key is (stored population * ncell + source node) - node, so one
// 32-bit addition forms the address whatever the walls do to the path --
// folds along r, along x3, corner reflections, equilibrium walls' clamping and
// every periodic wrap. One code path for all of them keeps the step kernels
// small: with a compile-time variant per wall layer they were bound by
// instruction fetch (7 to 19 cycles per issue at the walls).
//
// The state is read by ordinary loads, through pointers that promise nothing:
// a chained step (launch_chained) starts while the step that writes its input
// still runs, so its input is not read-only for the kernel's lifetime as the
// non-coherent path needs (__ldg, const __restrict__ arguments), and only
// ordinary loads are ordered after chain_wait.
template <class S>
__device__ __forceinline__ void gather_table(const S* fin, const CellPos& p, const Dims& d, S (&f)[Q]) {
  const int key = (axis_class(p.ir, d.nr) * d.src_nt + axis_class(p.it, d.nt)) * d.src_n3 + axis_class(p.i3, d.n3);
  const int4* __restrict__ row = d.src + key * SRC_ROW;
  static_for<0, SRC_ROW>([&](auto J_) {
    constexpr int J = decltype(J_)::value;
    const int4 o = __ldg(row + J);
    f[4 * J] = fin[uint32_t(p.cell + o.x)];
    if constexpr (4 * J + 1 < Q) {
      f[4 * J + 1] = fin[uint32_t(p.cell + o.y)];
      f[4 * J + 2] = fin[uint32_t(p.cell + o.z)];
      f[4 * J + 3] = fin[uint32_t(p.cell + o.w)];
    }
  });
}

// The step's gather: nodes at least 3 nodes from every wall take their sources
// from the node's own neighbours, computed; a warp that holds any other node
// reads the source table for all its nodes, so it runs one of the two paths.
template <class S>
__device__ __forceinline__ void gather_step(const S* fin, const CellPos& p, const Dims& d, S (&f)[Q]) {
  if (__any_sync(__activemask(), near_wall(p, d))) {
    gather_table(fin, p, d, f);
  } else {
    f[0] = fin[uint32_t(p.cell)];
    for_each_source_far<KFLAT>(fin, p, d, [&](auto L_, const S* src, int, int) { f[decltype(L_)::value] = *src; });
  }
}

// Store the 41 post-collision populations of node p into the instance block
// `out` (32-bit offsets, as for_each_source).
template <int K, class S, class R>
__device__ __forceinline__ void store_node(S* __restrict__ out, const float* ref, const CellPos& p, const Dims& d,
                                           const R (&f)[Q]) {
  using Cd = Codec<S, R>;
  const uint32_t N = uint32_t(d.ncell), cell = uint32_t(p.cell);
  const int row = geo_row<K>(d, p.ir, p.i3);
  static_for<0, Q>([&](auto L_) {
    constexpr int L = decltype(L_)::value;
    if constexpr (Cd::uses_ref)
      out[uint32_t(L) * N + cell] = Cd::template enc<L>(f[L], ref + ref_index<K>(d, L, row));
    else
      out[uint32_t(L) * N + cell] = Cd::template enc<L>(f[L], nullptr);
  });
}

// ---------------------------------------------------------------------------
// geometry and stream-table rows
// ---------------------------------------------------------------------------
template <typename Real, int K>
__device__ __forceinline__ NodeGeo<Real, K> load_geo(const GeoDev<Real>& g, int row) {
  NodeGeo<Real, K> n;
  n.fth = __ldg(g.fth + row);
  if constexpr (K == KCYL || K == KELL || K == KELT) {
    n.dtt = __ldg(g.dtt + row);
    n.n_rtt = -__ldg(g.g_rtt + row);
    n.n_trt = -__ldg(g.g_trt + row);
  }
  if constexpr (K == KELL || K == KELT) {
    n.dpp = __ldg(g.dpp + row);
    n.n_rpp = -__ldg(g.g_rpp + row);
    n.n_prp = -__ldg(g.g_prp + row);
    n.n_ttp = -__ldg(g.g_ttp + row);
    n.n_ptt = -__ldg(g.g_ptt + row);
  }
  if constexpr (K == KELT) {
    const Real* e = g.ext + row;
    n.drr = __ldg(e);
    n.drt = __ldg(e + g.ext_stride);
    n.drp = __ldg(e + 2 * g.ext_stride);
    n.dtp = __ldg(e + 3 * g.ext_stride);
    n.fr = __ldg(e + 4 * g.ext_stride);
    n.fp = __ldg(e + 5 * g.ext_stride);
  }
  return n;
}

// ---------------------------------------------------------------------------
// work division of the pair kernels (2-byte storage, pair.cuh)
// ---------------------------------------------------------------------------
// Warps of one instance. A stream-table row belongs to i_r alone (st_row_r) or
// to a pair of the (i_r, x3) cross-section. In the first case a warp takes 32
// consecutive pairs of an i_r layer and holds one row; else 32 consecutive
// pairs of one (i_r, i_theta) line, warps of consecutive theta next to each
// other, so that a block whose warps share (i_r, chunk) -- ntheta a multiple
// of its warps -- holds their rows once.
__host__ __device__ __forceinline__ uint32_t pair_warps(const Dims& d) { return uint32_t(d.nr) * d.div_wl.d; }

// Bytes of staged table rows in a block of `warps` warps.
__host__ __device__ __forceinline__ size_t pair_smem_bytes(const Dims& d, int warps) {
  const int rows = d.st_row_r ? warps : (d.nt % warps == 0 ? 32 : 32 * warps);
  return size_t(2 * ST_K) * size_t(rows) * sizeof(float4);
}

}  // namespace lbgm
