// Kernels of the lattice Boltzmann path. One thread per lattice node; nodes
// are numbered with x3 fastest so that a warp shares (instance, i_r, i_theta)
// and the wall branch along r is warp-uniform.
#pragma once

#include "lbm_device.cuh"

namespace lbgm {

// Programmatic dependent launch between the steps of a chain (launch_chained):
// a step's blocks may start while the step before still runs -- they find
// their nodes, source-table rows and geometry -- and wait for its end and its
// memory before they touch the state (gather_table says how they may read it).
// Without the launch attribute both are no-ops.
// chain_start lets the next step's blocks in. FP32 arithmetic asks for them
// first of all. An FP64 step asks after its own wait, so that at most the step to
// come waits on the SMs: asked for at once, blocks of two or three steps sat
// there, some SMs got two blocks of one step and their FP64 units took twice as
// long. us a step, asked for at once / after the wait: one cylinder of 49 blocks
// 28.4 / 20.0; two contexts of 24 blocks side by side 29.1 / 21.7, four 35.5 /
// 24.7 (32.3 before steps were chained).
__device__ __forceinline__ void chain_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
template <class Real>
constexpr bool CHAIN_LATE = sizeof(Real) == 8;

// Fused time step (Eq. LB) of one node p of one instance whose state blocks
// start at fin and fout: pull streaming + walls (gather_step), moments,
// equilibrium, non-equilibrium stress, forcing, BGK, store. flag is set to 1
// when the node's density is not finite. Nodes on an equilibrium wall (the end
// nodes of the walled axes) leave the step as f^eq(rho', 0) of their own
// density and metric (Sec. III). FP32 and FP64 storage (2-byte storage:
// pair.cuh).
template <typename Real, int K>
__device__ __forceinline__ void step_node(const Real* fin, Real* __restrict__ fout,
                                          const GeoDev<Real>& geo, const InstParams<Real>& ip, const Dims& d,
                                          const CellPos& p, int* __restrict__ flag) {
  Real f[Q];
  const int row = geo_row_node<K>(d, p.ir, p.it, p.i3);
  NodeGeo<Real, K> g;
  // the theta-resolved ellipsoid's 15 values per node come from HBM: asked for
  // before the gather (2 x 65 x 64 x 128, FP32: 74.6 -> 69.8 us a step); rows
  // shared by nodes come from L1 and L2 and would only hold registers
  if constexpr (K == KELT) g = load_geo<Real, K>(geo, row);
  chain_wait();
  if constexpr (CHAIN_LATE<Real>) chain_start();
  gather_step(fin, p, d, f);
  const Moments<Real> m = step_moments(f);
  if (!finite_v(m.rho)) {  // NaN or Inf
    if (*flag == 0) atomicExch(flag, 1);
  }
  if constexpr (K != KELT) g = load_geo<Real, K>(geo, row);
  if (d.wall_eq && (p.ir == 0 || p.ir == d.nr - 1 || (!d.periodic3 && (p.i3 == 0 || p.i3 == d.n3 - 1)))) {
    equilibrium<Real, K>(m.rho, Real(0.0), Real(0.0), Real(0.0), g, f);
    store_node<K>(fout, nullptr, p, d, f);
    return;
  }
  const Coef<Real> k = coefficients<Real, K>(m, g, ip.kappa, ip.G);
  collide<Real, K>(f, k, g, ip.omega);
  store_node<K>(fout, nullptr, p, d, f);
}

// Launch bounds of the one-node-per-thread step. FP32: at most 128 threads per
// block and 5 resident blocks per SM (96 registers). Measured at 8 / 7 / 6 / 5 /
// 4 blocks with the instances held in L2 (lanes.h), us a step: 24 cylinders of
// 64 x 4 x 256 88 / 79 / 72 / 66 / -, 24 four-wall ellipsoids - / - / 80 / 68 /
// 69, the theta-resolved ellipsoid - / - / 83 / 75 / 78. FP64 keeps its
// registers (bound by the FP64 units). LBGM_STEP32_MAXT / LBGM_STEP32_MINB
// override the FP32 values for tuning builds.
#ifndef LBGM_STEP32_MAXT
#define LBGM_STEP32_MAXT 128
#endif
#ifndef LBGM_STEP32_MINB
#define LBGM_STEP32_MINB 5
#endif
template <class Real, int K>
struct KBounds {
  static constexpr int maxt = LBGM_STEP32_MAXT, minb = LBGM_STEP32_MINB;
};
template <int K>
struct KBounds<double, K> {
  static constexpr int maxt = 256, minb = 1;
};
// Uniform batch: fin/fout are whole states (batch blocks of Q * ncell);
// block (x, y) updates nodes [x blockDim, (x + 1) blockDim) of instance y, so
// the instance's block base is uniform across the thread block.
template <typename Real, int K>
__global__ void __launch_bounds__(KBounds<Real, K>::maxt, KBounds<Real, K>::minb)
    k_step(const Real* fin, Real* __restrict__ fout, GeoDev<Real> geo,
           const InstParams<Real>* __restrict__ inst, Dims d, int* __restrict__ flag) {
  if constexpr (!CHAIN_LATE<Real>) chain_start();
  const uint32_t cell = blockIdx.x * blockDim.x + threadIdx.x;
  if (cell >= uint32_t(d.ncell)) return;
  const int b = int(blockIdx.y);
  const CellPos p = locate_cell(d, b, cell);
  const size_t base = size_t(b) * Q * uint32_t(d.ncell);
  step_node<Real, K>(fin + base, fout + base, geo, inst[b], d, p, flag);
}

// One instance of a batch whose instances differ in geometry and size: its
// dimensions (batch 1), geometry tables, parameters, two state blocks and
// the flag that records a non-finite density.
template <typename S, typename Real>
struct ListInst {
  Dims d;
  GeoDev<Real> geo;
  const InstParams<Real>* ip;
  const S* f0;
  S* f1;
  int* flag;
};

// Arguments of a work-list launch: up to N instances and the first work item
// of each (tile_start[count] items in all). They travel in the kernel's
// parameters, so a block reads its instance's record through the constant
// cache with a block-uniform index, as the uniform-batch kernels read theirs:
// staged in shared memory the record took the step's registers (184 bytes
// spilled on the cylinder: 103.6 us a step against 82.4 for k_step on 24
// 64 x 4 x 256 cylinders in FP32).
template <typename S, typename Real>
struct ListArgs {
  static constexpr int N = 16;  // LIST_MAX
  ListInst<S, Real> rec[N];
  int tile_start[N + 1];
  int count, tile, parity;

  // Instance of work item j.
  __device__ __forceinline__ int instance(int j) const {
    int i = 0;
#pragma unroll
    for (int s = N / 2; s > 0; s >>= 1)
      if (i + s < count && tile_start[i + s] <= j) i += s;
    return i;
  }
};

// Work-list step over instances of one metric kind: item j is the j-th tile of
// `tile` consecutive nodes over all instances. One block per item of at most
// one block's worth of nodes, or with LOOP items of several blocks' worth and
// blocks that take items blockIdx.x, blockIdx.x + gridDim.x, ... (the loops
// cost registers: a separate instantiation). `parity` 0 reads f0 and writes
// f1, 1 the reverse.
template <typename Real, int K, bool LOOP>
__global__ void __launch_bounds__(KBounds<Real, K>::maxt, KBounds<Real, K>::minb)
    k_step_list(const __grid_constant__ ListArgs<Real, Real> a) {
  if constexpr (!CHAIN_LATE<Real>) chain_start();
  auto item = [&](int j) {
    const int i = a.instance(j);
    const ListInst<Real, Real>& I = a.rec[i];
    const Real* fin = a.parity ? I.f1 : I.f0;
    Real* fout = const_cast<Real*>(a.parity ? I.f0 : I.f1);
    const int first = (j - a.tile_start[i]) * a.tile, end = min(first + a.tile, I.d.ncell);
    int c = first + int(threadIdx.x);
    if (c >= end) return;
    do {
      step_node<Real, K>(fin, fout, I.geo, *I.ip, I.d, locate_cell(I.d, 0, uint32_t(c)), I.flag);
      c += int(blockDim.x);
    } while (LOOP && c < end);
  };
  if constexpr (LOOP) {
    for (int j = blockIdx.x; j < a.tile_start[a.count]; j += gridDim.x) item(j);
  } else {
    item(int(blockIdx.x));
  }
}

// Moments of the streamed populations of node p (the observables).
template <typename S, typename Real, int K>
__device__ __forceinline__ Moments<Real> streamed_moments(const S* __restrict__ fin, const float* ref,
                                                          const CellPos& p, const Dims& d) {
  Real f[Q];
  if constexpr (Codec<S, Real>::uses_ref) gather<K>(fin, ref, p, d, f);
  else gather_step(fin, p, d, f);
  return moments(f);
}

// rho' and u of the streamed populations (moments only). 2-byte storage asks
// for three blocks per SM: without it the ellipsoid's kernel takes 122 registers
// for 80, two blocks, and 8 four-wall 64 x 4 x 255 channels 100 us for 78.
template <typename S, typename Real, int K>
__global__ void __launch_bounds__(256, sizeof(S) == 2 ? 3 : 1)
    k_macros(const S* __restrict__ fin, double* __restrict__ rho, double* __restrict__ u, Dims d) {
  const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= uint32_t(d.batch) * uint32_t(d.ncell)) return;
  const CellPos p = locate(d, t);
  const Moments<Real> m = streamed_moments<S, Real, K>(fin + size_t(p.b) * Q * d.ncell, ref_of(d, p.b), p, d);
  const double r = double(m.rho);
  if (rho) rho[t] = r;
  if (u) {
    const size_t ub = size_t(p.b) * 3 * d.ncell + p.cell;
    u[ub] = double(m.jx / m.rho);
    u[ub + d.ncell] = double(m.jy / m.rho);
    u[ub + 2 * size_t(d.ncell)] = double(m.jz / m.rho);
  }
}

// Largest of the warp's 64-bit values.
__device__ __forceinline__ unsigned long long warp_max(unsigned long long v) {
  const uint32_t hi = __reduce_max_sync(0xffffffffu, uint32_t(v >> 32));
  const uint32_t lo = __reduce_max_sync(0xffffffffu, uint32_t(v >> 32) == hi ? uint32_t(v) : 0u);
  return (static_cast<unsigned long long>(hi) << 32) | lo;
}

// Convergence monitor: max |u - u_prev| and max |u| of instance blockIdx.y
// into out[2 b], out[2 b + 1] (zero before; non-negative doubles order like
// their bits), and u_prev = u. One pass over the state: the velocity goes
// nowhere else, and no reduction runs after it.
template <typename S, typename Real, int K>
__global__ void __launch_bounds__(256) k_velocity_change(const S* __restrict__ fin, double* __restrict__ u_prev,
                                                         Dims d, unsigned long long* __restrict__ out) {
  const uint32_t cell = blockIdx.x * blockDim.x + threadIdx.x;
  const int b = int(blockIdx.y);
  // the maxima as the bits of non-negative numbers: FP64 comparisons run on
  // the FP64 units (16 cycles a warp instruction), integer ones do not
  unsigned long long md = 0, mu = 0;
  if (cell < uint32_t(d.ncell)) {
    double* q = u_prev + size_t(b) * 3 * d.ncell + cell;
    const size_t N = size_t(d.ncell);
    const double old[3] = {q[0], q[N], q[2 * N]};
    const CellPos p = locate_cell(d, b, cell);
    const Moments<Real> m = streamed_moments<S, Real, K>(fin + size_t(b) * Q * d.ncell, ref_of(d, b), p, d);
    const Real v[3] = {m.jx / m.rho, m.jy / m.rho, m.jz / m.rho};
    Real um = Real(0);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const double x = double(v[i]);
      const unsigned long long e = static_cast<unsigned long long>(__double_as_longlong(fabs(x - old[i])));
      if (e > md && e <= 0x7ff0000000000000ull) md = e;  // a NaN does not count, as in fmax
      um = fmax(um, fabs(v[i]));
      q[i * N] = x;
    }
    mu = static_cast<unsigned long long>(__double_as_longlong(double(um)));
  }
  md = warp_max(md);
  mu = warp_max(mu);
  __shared__ unsigned long long s_m[8][2];
  if ((threadIdx.x & 31) == 0) {
    s_m[threadIdx.x >> 5][0] = md;
    s_m[threadIdx.x >> 5][1] = mu;
  }
  __syncthreads();
  if (threadIdx.x < 2) {
    unsigned long long m = 0;
    for (int w = 0; w < 8; ++w) m = max(m, s_m[w][threadIdx.x]);
    atomicMax(out + 2 * b + threadIdx.x, m);
  }
}

// SplitMix64: output number k (from 0) of the generator seeded with `seed`.
__device__ __forceinline__ uint64_t splitmix64_at(uint64_t seed, uint64_t k) {
  uint64_t z = seed + (k + 1ull) * 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

struct InitInst {
  unsigned long long seed;
  double amp;
};

// Initial state f = f^eq(rho', u): either from caller fields (rho_in, u_in
// non-NULL) or rho' = 1/sqrt(g), u = base(b, i_r) + noise.
template <typename S, typename Real, int K>
__global__ void __launch_bounds__(256) k_init(S* __restrict__ f, GeoDev<Real> geo,
                                              const double* __restrict__ sqrtg,
                                              const double* __restrict__ base_uth,
                                              const InitInst* __restrict__ ini,
                                              const double* __restrict__ rho_in,
                                              const double* __restrict__ u_in, Dims d) {
  const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= uint32_t(d.batch) * uint32_t(d.ncell)) return;
  const CellPos p = locate(d, t);
  double rho, u[3];
  if (rho_in) {
    rho = rho_in[t];
    const size_t ub = size_t(p.b) * 3 * d.ncell + p.cell;
    u[0] = u_in[ub];
    u[1] = u_in[ub + d.ncell];
    u[2] = u_in[ub + 2 * size_t(d.ncell)];
  } else {
    rho = 1.0 / sqrtg[d.geo_theta ? p.cell : p.ir * d.n3 + p.i3];
    u[0] = 0.0;
    u[1] = base_uth ? base_uth[size_t(p.b) * d.nr + p.ir] : 0.0;
    u[2] = 0.0;
    const InitInst in = ini[p.b];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const uint64_t s = splitmix64_at(in.seed, 3ull * uint64_t(p.cell) + uint64_t(i));
      const double U = double(s >> 11) * 0x1.0p-53;
      u[i] += in.amp * (2.0 * U - 1.0);
    }
  }
  const int row = geo_row_node<K>(d, p.ir, p.it, p.i3);
  const NodeGeo<Real, K> g = load_geo<Real, K>(geo, row);
  Real fe[Q];
  equilibrium<Real, K>(Real(rho), Real(u[0]), Real(u[1]), Real(u[2]), g, fe);
  store_node<K>(f + size_t(p.b) * Q * d.ncell, ref_of(d, p.b), p, d, fe);
}

// Reference populations of 2-byte storage (Codec): for instance b and
// geometry row r, mode 0: r_l = w_l (the rest state of unit density);
// mode 1: the equilibrium f^eq(rho', u) of the row's initial state: with
// caller fields (rho_in, u_in non-NULL) their mean over the row's nodes,
// else rho' = 1/sqrt(g) and u = (0, base(b, i_r), 0) (rest where base is
// NULL). Written at ref_index<K> of instance b's table.
template <int K>
__global__ void __launch_bounds__(256) k_ref_table(float* __restrict__ ref, GeoDev<float> geo,
                                                   const double* __restrict__ sqrtg,
                                                   const double* __restrict__ base_uth,
                                                   const double* __restrict__ rho_in,
                                                   const double* __restrict__ u_in, Dims d, int mode) {
  const uint32_t nrows = uint32_t(d.nr) * uint32_t(d.geo_rows3);
  const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= uint32_t(d.batch) * nrows) return;
  const uint32_t b = t / nrows, row = t - b * nrows;
  const int ir = int(row) / d.geo_rows3, i3 = int(row) - ir * d.geo_rows3;
  float fe[Q];
  if (mode == 0) {
    static_for<0, Q>([&](auto L_) {
      constexpr int L = decltype(L_)::value;
      fe[L] = float(WeightOf<L>::w);
    });
  } else if (rho_in) {
    // mean over the row's nodes: all (i_theta, i_3) of layer i_r, or all
    // i_theta of (i_r, i_3) for the ellipsoid's rows
    double rs = 0.0, us[3] = {0.0, 0.0, 0.0};
    const int n3s = d.geo_rows3 > 1 ? 1 : d.n3;
    int cnt = 0;
    for (int it = 0; it < d.nt; ++it)
      for (int k3 = 0; k3 < n3s; ++k3) {
        const size_t cell = (size_t(ir) * d.nt + it) * d.n3 + (d.geo_rows3 > 1 ? i3 : k3);
        rs += rho_in[size_t(b) * d.ncell + cell];
        const size_t ub = size_t(b) * 3 * d.ncell + cell;
        us[0] += u_in[ub];
        us[1] += u_in[ub + d.ncell];
        us[2] += u_in[ub + 2 * size_t(d.ncell)];
        ++cnt;
      }
    const NodeGeo<float, K> g = load_geo<float, K>(geo, int(row));
    equilibrium<float, K>(float(rs / cnt), float(us[0] / cnt), float(us[1] / cnt), float(us[2] / cnt), g, fe);
  } else {
    const double rho = 1.0 / sqrtg[ir * d.n3 + i3];
    const double uth = base_uth ? base_uth[size_t(b) * d.nr + ir] : 0.0;
    const NodeGeo<float, K> g = load_geo<float, K>(geo, int(row));
    equilibrium<float, K>(float(rho), 0.0f, float(uth), 0.0f, g, fe);
  }
  float* rb = ref + size_t(b) * Q * nrows;
#pragma unroll
  for (int l = 0; l < Q; ++l) rb[ref_index<K>(d, l, int(row))] = fe[l];
}

// Stream table entries of node p (stream_of): put(k, x, y, z, w). The sources
// of the node at theta = 0 give, for every population l, the stored population
// index and geometry row whose reference rho_l it receives -- the sources of the
// step's gather. rb is the instance's reference table, fin any state block of
// the context: its addresses are formed, never read.
template <int K, class S, class Put>
__device__ __forceinline__ void stream_entries(const float* __restrict__ rb, float omega, const S* fin,
                                               const CellPos& p, const Dims& d, Put&& put) {
  double rho_l[Q];
  for_each_source<K, S>(fin, p, d, [&](auto L_, const S*, int sl, int row) {
    constexpr int L = decltype(L_)::value;
    rho_l[L] = double(rb[ref_index<K>(d, sl, row)]);
  });
  const float om1 = 1.0f - omega;  // as the step computes it
  const int own = geo_row<K>(d, p.ir, p.i3);
  double tl[Q];
  double m[10] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
  static_for<0, Q>([&](auto L_) {
    constexpr int L = decltype(L_)::value;
    constexpr int cx = L == 0 ? 0 : ((L - 1) % 2 == 0 ? 1 : -1) * PAIRS[L == 0 ? 0 : (L - 1) / 2].x;
    constexpr int cy = L == 0 ? 0 : ((L - 1) % 2 == 0 ? 1 : -1) * PAIRS[L == 0 ? 0 : (L - 1) / 2].y;
    constexpr int cz = L == 0 ? 0 : ((L - 1) % 2 == 0 ? 1 : -1) * PAIRS[L == 0 ? 0 : (L - 1) / 2].z;
    const double r = rho_l[L];
    m[0] += r;
    auto add = [&](int i, auto C_) {
      if constexpr (decltype(C_)::value != 0) m[i] += decltype(C_)::value * r;
    };
    add(1, std::integral_constant<int, cx>{});
    add(2, std::integral_constant<int, cy>{});
    add(3, std::integral_constant<int, cz>{});
    add(4, std::integral_constant<int, cx * cx>{});
    add(5, std::integral_constant<int, cy * cy>{});
    add(6, std::integral_constant<int, cz * cz>{});
    add(7, std::integral_constant<int, cx * cy>{});
    add(8, std::integral_constant<int, cx * cz>{});
    add(9, std::integral_constant<int, cy * cz>{});
    tl[L] = (double(om1) * r - double(rb[ref_index<K>(d, L, own)])) / WeightOf<L>::w;
  });
  // even and odd parts of t per pair, then each shell's transform to the
  // coefficients its pairs are evaluated from (update_face, update_body)
  double te[NPAIR], to[NPAIR];
#pragma unroll
  for (int P = 0; P < NPAIR; ++P) {
    te[P] = 0.5 * (tl[2 * P + 1] + tl[2 * P + 2]);
    to[P] = 0.5 * (tl[2 * P + 1] - tl[2 * P + 2]);
  }
  auto face = [](double* v) {
    const double a = v[0], b2 = v[1];
    v[0] = 0.5 * (a + b2);
    v[1] = 0.5 * (a - b2);
  };
  auto body = [](double* v) {
    const double p2 = v[0] + v[1], q = v[2] + v[3], r = v[0] - v[1], s = v[2] - v[3];
    v[0] = 0.25 * (p2 + q);
    v[1] = 0.25 * (p2 - q);
    v[2] = 0.25 * (r + s);
    v[3] = 0.25 * (r - s);
  };
  for (double* v : {te, to}) {
    face(v + 3);
    face(v + 5);
    face(v + 7);
    body(v + 9);
    body(v + 16);
  }
  put(0, m[0], m[1], m[2], m[3]);
  put(1, m[4], m[5], m[6], m[7]);
  put(2, m[8], m[9], tl[0], 0.0);
#pragma unroll
  for (int j = 0; j < NPAIR / 2; ++j) put(3 + j, te[2 * j], to[2 * j], te[2 * j + 1], to[2 * j + 1]);
}

// Stream table of 2-byte storage: one thread per instance, stream row and node
// of the row's pair (the last pair of an odd line repeats its one node). FP64
// arithmetic bounds it: the zero products are left out, and a block is one warp,
// so that a cylinder's few rows are spread over the SMs (lb_init of one 64 x 4 x
// 256 cylinder in FP16 88 -> 81 us, of 24 four-wall 64 x 4 x 255 ellipsoids 1000
// -> 902).
constexpr int ST_THREADS = 32;
template <int K, class S>
__global__ void __launch_bounds__(ST_THREADS) k_stream_table(float4* __restrict__ st,
                                                             const float* __restrict__ ref,
                                                             const InstParams<float>* __restrict__ inst,
                                                             const S* fin, Dims d) {
  const uint32_t nrows = uint32_t(d.nr) * uint32_t(d.st_rows3);
  const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= uint32_t(d.batch) * nrows * 2u) return;
  const uint32_t half = t & 1u;
  const int b = int((t / 2) / nrows), srow = int(t / 2 - uint32_t(b) * nrows);
  CellPos p;
  p.b = b;
  p.it = 0;
  p.ir = srow / d.st_rows3;
  const int r3 = srow - p.ir * d.st_rows3;
  p.i3 = d.st_row_r ? 0 : 2 * (K == KELL ? r3 : pair_of_row(r3, (d.n3 + 1) / 2)) + int(half);
  if (p.i3 >= d.n3) p.i3 -= int(half);
  p.cell = (p.ir * d.nt + p.it) * d.n3 + p.i3;
  float* out = reinterpret_cast<float*>(st + size_t(b) * 2 * ST_K * nrows + uint32_t(srow)) + half;
  stream_entries<K, S>(ref + size_t(b) * Q * size_t(d.nr) * size_t(d.geo_rows3), inst[b].omega, fin, p, d,
                       [&](int k, double x, double y, double z, double w) {
                         float* o = out + size_t(2 * k) * nrows * 4;
                         o[0] = float(x);
                         o[2] = float(y);
                         o += size_t(nrows) * 4;
                         o[0] = float(z);
                         o[2] = float(w);
                       });
}

}  // namespace lbgm
