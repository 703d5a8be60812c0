// Initialisation, macroscopic fields, state conversion and the observables
// reduction (Sec. II initial state and moments; Sec. III-IV Dean number,
// mean velocity and mean vorticity).
#include <algorithm>

#include "kernels.cuh"
#include "launch.h"

namespace lbgm {

namespace {

uint32_t blocks_for(const Dims& d, int threads) {
  const uint32_t total = uint32_t(d.batch) * uint32_t(d.ncell);
  return (total + threads - 1) / threads;
}

template <typename S, typename Real>
cudaError_t macros_t(int K, const S* fin, double* rho, double* u, const Dims& d, cudaStream_t s) {
  const uint32_t nb = blocks_for(d, 256);
  switch (K) {
    case KFLAT: k_macros<S, Real, KFLAT><<<nb, 256, 0, s>>>(fin, rho, u, d); break;
    case KCYL: k_macros<S, Real, KCYL><<<nb, 256, 0, s>>>(fin, rho, u, d); break;
    case KELL: k_macros<S, Real, KELL><<<nb, 256, 0, s>>>(fin, rho, u, d); break;
    case KELT:
      if constexpr (!Codec<S, Real>::uses_ref) {  // FP64 / FP32 storage only
        k_macros<S, Real, KELT><<<nb, 256, 0, s>>>(fin, rho, u, d);
        break;
      }
      return cudaErrorInvalidValue;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

template <typename S, typename Real>
cudaError_t init_t(int K, S* f, const GeoDev<Real>& geo, const double* sqrtg, const double* base,
                   const InitInst* ini, const double* rho_in, const double* u_in, const Dims& d,
                   cudaStream_t s) {
  const uint32_t nb = blocks_for(d, 256);
  switch (K) {
    case KFLAT: k_init<S, Real, KFLAT><<<nb, 256, 0, s>>>(f, geo, sqrtg, base, ini, rho_in, u_in, d); break;
    case KCYL: k_init<S, Real, KCYL><<<nb, 256, 0, s>>>(f, geo, sqrtg, base, ini, rho_in, u_in, d); break;
    case KELL: k_init<S, Real, KELL><<<nb, 256, 0, s>>>(f, geo, sqrtg, base, ini, rho_in, u_in, d); break;
    case KELT:
      if constexpr (!Codec<S, Real>::uses_ref) {  // FP64 / FP32 storage only
        k_init<S, Real, KELT><<<nb, 256, 0, s>>>(f, geo, sqrtg, base, ini, rho_in, u_in, d);
        break;
      }
      return cudaErrorInvalidValue;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

// Velocities by population index, for code that loops over them.
struct VelTable {
  signed char c[Q][4];  // x, y, z, |c|_inf
};
constexpr VelTable make_velocities() {
  VelTable t{};
  for (int l = 1; l < Q; ++l) {
    int s = 0;
    for (int a = 0; a < 3; ++a) {
      const int v = vel(l, a);
      t.c[l][a] = static_cast<signed char>(v);
      s = v > s ? v : -v > s ? -v : s;
    }
    t.c[l][3] = static_cast<signed char>(s);
  }
  return t;
}
__constant__ VelTable c_vel = make_velocities();

// Source table (gather_table): one thread per key and entry, from the general
// source rule at a node of the key's classes.
__global__ void __launch_bounds__(256) k_source_table(int* __restrict__ tab, Dims d) {
  const int keys = axis_classes(d.nr) * d.src_nt * d.src_n3;
  const int t = int(blockIdx.x * blockDim.x + threadIdx.x), k = t / (4 * SRC_ROW), l = t - k * 4 * SRC_ROW;
  if (k >= keys) return;
  const int c3 = k % d.src_n3, ct = (k / d.src_n3) % d.src_nt, cr = k / (d.src_n3 * d.src_nt);
  CellPos p;
  p.b = 0;
  p.ir = axis_class_node(cr, d.nr);
  p.it = axis_class_node(ct, d.nt);
  p.i3 = axis_class_node(c3, d.n3);
  p.cell = (p.ir * d.nt + p.it) * d.n3 + p.i3;
  int off = 0;
  if (l > 0 && l < Q) {
    const int cx = c_vel.c[l][0], cy = c_vel.c[l][1], cz = c_vel.c[l][2];
    int yr, yz, src, from = l;
    if (d.wall_eq) {  // the source clamped onto the wall layers
      yr = min(max(p.ir - cx, 0), d.nr - 1);
      yz = p.i3 - cz;
      yz = d.periodic3 ? wrap_small(yz, d.n3) : min(max(yz, 0), d.n3 - 1);
      src = (yr * d.nt + wrap_small(p.it - cy, d.nt)) * d.n3 + yz;
    } else {
      bool flip;
      src = src_wall(cx, cy, cz, c_vel.c[l][3], p, d, flip, yr, yz);
      if (flip) from = ((l - 1) ^ 1) + 1;  // the opposite of l
    }
    off = from * d.ncell + src - p.cell;
  }
  tab[t] = off;
}

// weights by population index, for the element-wise conversions
__constant__ double c_weight[Q];

// stored value <-> f_l (2-byte formats: f = w s + r, Codec)
__device__ __forceinline__ double to_f(double v, double, double) { return v; }
__device__ __forceinline__ double to_f(float v, double, double) { return v; }
__device__ __forceinline__ double to_f(__half v, double w, double r) { return w * double(__half2float(v)) + r; }
__device__ __forceinline__ double to_f(__nv_bfloat16 v, double w, double r) {
  return w * double(__bfloat162float(v)) + r;
}
__device__ __forceinline__ void from_f(double& o, double f, double, double) { o = f; }
__device__ __forceinline__ void from_f(float& o, double f, double, double) { o = float(f); }
__device__ __forceinline__ void from_f(__half& o, double f, double w, double r) { o = __double2half((f - r) / w); }
__device__ __forceinline__ void from_f(__nv_bfloat16& o, double f, double w, double r) {
  o = __double2bfloat16((f - r) / w);
}

// state (documented population layout) <-> FP64 populations
template <typename S>
__global__ void k_convert(S* state, double* dbl, size_t n, Dims d, int to_double) {
  const size_t N = size_t(d.ncell), layer = size_t(d.nt) * size_t(d.n3);
  const size_t nrows = size_t(d.nr) * size_t(d.geo_rows3);
  for (size_t i = blockIdx.x * size_t(blockDim.x) + threadIdx.x; i < n;
       i += size_t(gridDim.x) * blockDim.x) {
    const size_t bl = i / N;  // b * Q + l
    const double w = c_weight[bl % Q];
    double r = 0.0;
    if (d.ref) {  // the reference table's layout of ref_index
      const size_t cell = i - bl * N, b = bl / Q, l = bl % Q;
      const size_t ir = cell / layer;
      const float* rb = d.ref + b * Q * nrows;
      r = d.geo_rows3 > 1 ? double(rb[l * nrows + ir * size_t(d.geo_rows3) + cell % size_t(d.n3)])
                          : double(rb[ir * Q + l]);
    }
    if (to_double)
      dbl[i] = to_f(state[i], w, r);
    else
      from_f(state[i], dbl[i], w, r);
  }
}

// Equilibrium walls: the wall nodes' velocity is the Dirichlet value 0 in
// every observable (their streamed moments are replaced in the collision).
__device__ __forceinline__ bool eq_wall_node(const Dims& d, int ir, int i3) {
  return d.wall_eq && (ir == 0 || ir == d.nr - 1 || (!d.periodic3 && (i3 == 0 || i3 == d.n3 - 1)));
}

// derivative along an axis from the values at offsets -2 .. +2 (u2m, um, u0,
// up, u2p); the bounce-back wall version uses u = 0 half a node outside the
// first and last node, the equilibrium-wall version second-order one-sided
// differences at the wall nodes (whose value is 0).
__device__ __forceinline__ double d_axis(double u2m, double um, double u0, double up, double u2p, int i, int n,
                                         bool walled, bool eqw) {
  if (!walled) return 0.5 * (up - um);
  if (n == 1) return 0.0;
  if (eqw) {
    if (i == 0) return 0.5 * (-3.0 * u0 + 4.0 * up - u2p);
    if (i == n - 1) return 0.5 * (3.0 * u0 - 4.0 * um + u2m);
    return 0.5 * (up - um);
  }
  if (i == 0) return u0 + up / 3.0;
  if (i == n - 1) return -(u0 + um / 3.0);
  return 0.5 * (up - um);
}

constexpr int DIAG_THREADS = 256;

__device__ __forceinline__ void block_reduce(double (&a)[DIAG_NQ], double* sh) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int q = 0; q < DIAG_NQ; ++q) {
    double v = a[q];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double w = __shfl_down_sync(0xffffffffu, v, o);
      v = (q == 7) ? fmax(v, w) : v + w;
    }
    if (lane == 0) sh[warp * DIAG_NQ + q] = v;
  }
  __syncthreads();
  if (threadIdx.x < DIAG_NQ) {
    const int q = threadIdx.x;
    double v = sh[q];
    for (int w = 1; w < DIAG_THREADS / 32; ++w)
      v = (q == 7) ? fmax(v, sh[w * DIAG_NQ + q]) : v + sh[w * DIAG_NQ + q];
    a[q] = v;  // valid in thread q only
  }
}

// isfinite without the FP64 units
__device__ __forceinline__ bool finite_bits(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }

// Per-block partial sums of one instance (blockIdx.y), in a fixed order.
//   0 rho'   1 rho' g   2 sqrt(g_thth) u^theta wA   3 wA   4 |omega| wOmega
//   5 (u^r)^2   6 (u^r - row mean)^2   7 max |u|^2   8 non-finite nodes
// A warp takes whole x3 rows: the row's mean of u^r first, then its nodes
// while the row is in L1. 89 us for 24 x 64 x 4 x 256 nodes, 42 of them the FP64
// units' (16 cycles a warp instruction), the rest latency at 16 warps per SM. So
// the weights come multiplied out (diag_weights), 5 is the sum of 6 and the
// rows' means, the square root of 7 is taken once at the end, comparisons are
// integer, and the two halves of the central differences are one factor of the
// weight: 14 FP64 operations a node.
__global__ void __launch_bounds__(DIAG_THREADS)
    k_diag_partial(const double* __restrict__ rho, const double* __restrict__ u, const double* __restrict__ geo64,
                   Dims d, double* __restrict__ partial, int nblk) {
  __shared__ double sh[(DIAG_THREADS / 32) * DIAG_NQ];
  const int b = blockIdx.y, lane = threadIdx.x & 31;
  const int N = d.ncell, n3 = d.n3;
  const double* ur = u + size_t(b) * 3 * N;
  const double* ut = ur + N;
  const double* uz = ur + 2 * size_t(N);
  const double* rb = rho + size_t(b) * N;
  const bool eqw = d.wall_eq != 0;
  double a[DIAG_NQ];
#pragma unroll
  for (int q = 0; q < DIAG_NQ; ++q) a[q] = 0.0;
  const double inv_n3 = 1.0 / n3;
  int bad = 0;
  bool direct = false;            // 5 from u^r itself, since a row with an infinity
  unsigned long long speed2 = 0;  // bits of the largest |u|^2
  for (int row = blockIdx.x * (DIAG_THREADS / 32) + (threadIdx.x >> 5); row < d.nr * d.nt;
       row += nblk * (DIAG_THREADS / 32)) {
    const int ir = row / d.nt, it = row - ir * d.nt;
    const double* r0 = ur + size_t(row) * n3;
    double s = 0.0;
    for (int i = lane; i < n3; i += 32) s += eq_wall_node(d, ir, i) ? 0.0 : r0[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    const double mean = s * inv_n3;
    if (!direct && !finite_bits(mean)) {  // no mean to split (u^r)^2 by, and 6 becomes a NaN
      a[5] += a[6];
      direct = true;
    }
    if (!direct) {
      if (lane == 0) a[5] = fma(double(n3) * mean, mean, a[5]);  // + sum fl^2 = sum (u^r)^2
    } else {
      for (int i = lane; i < n3; i += 32) {
        const double v = eq_wall_node(d, ir, i) ? 0.0 : r0[i];
        a[5] = fma(v, v, a[5]);
      }
    }
    for (int i3 = lane; i3 < n3; i3 += 32) {
      const int c = row * n3 + i3;
      const double* gr = geo64 + size_t(d.geo_theta ? c : ir * n3 + i3) * 4;
      const double r = rb[c];
      // velocity component at node (jr, j3) of this theta plane: 0 on an
      // equilibrium wall node and outside the node range
      auto U = [&](const double* a, int jr, int j3) -> double {
        if (jr < 0 || jr >= d.nr || j3 < 0 || j3 >= n3 || eq_wall_node(d, jr, j3)) return 0.0;
        return a[(size_t(jr) * d.nt + it) * n3 + j3];
      };
      const double u0 = U(ur, ir, i3), u1 = U(ut, ir, i3), u2 = U(uz, ir, i3);
      double om2;  // 2 (d_3 u^r - d_r u^3)
      if (ir > 0 && ir < d.nr - 1 && (d.periodic3 || (i3 > 0 && i3 < n3 - 1))) {
        const int jm = i3 == 0 ? n3 - 1 : i3 - 1, jp = i3 == n3 - 1 ? 0 : i3 + 1;
        om2 = (U(ur, ir, jp) - U(ur, ir, jm)) - (U(uz, ir + 1, i3) - U(uz, ir - 1, i3));
      } else {
        double d3ur;
        if (d.periodic3) {
          const int jm = i3 == 0 ? n3 - 1 : i3 - 1, jp = i3 == n3 - 1 ? 0 : i3 + 1;
          d3ur = d_axis(0.0, U(ur, ir, jm), u0, U(ur, ir, jp), 0.0, i3, n3, false, eqw);
        } else {
          d3ur = d_axis(U(ur, ir, i3 - 2), U(ur, ir, i3 - 1), u0, U(ur, ir, i3 + 1), U(ur, ir, i3 + 2), i3, n3,
                        true, eqw);
        }
        const double drz = d_axis(U(uz, ir - 2, i3), U(uz, ir - 1, i3), u2, U(uz, ir + 1, i3), U(uz, ir + 2, i3), ir,
                                  d.nr, true, eqw);
        om2 = 2.0 * (d3ur - drz);
      }
      const double fl = u0 - mean;
      a[0] += r;
      a[1] = fma(gr[0], r, a[1]);
      a[2] = fma(gr[1], u1, a[2]);
      a[3] += gr[2];
      a[4] = fma(fabs(om2), gr[3], a[4]);
      a[6] = fma(fl, fl, a[6]);
      const unsigned long long v2 =
          static_cast<unsigned long long>(__double_as_longlong(fma(u2, u2, fma(u1, u1, u0 * u0))));
      if (v2 > speed2 && v2 <= 0x7ff0000000000000ull) speed2 = v2;  // a NaN does not count, as in fmax
      bad += finite_bits(r) && finite_bits(u0) && finite_bits(u1) && finite_bits(u2) ? 0 : 1;
    }
  }
  if (!direct) a[5] += a[6];
  a[7] = __longlong_as_double(static_cast<long long>(speed2));
  a[8] = double(bad);
  block_reduce(a, sh);
  if (threadIdx.x < DIAG_NQ) partial[(size_t(b) * nblk + blockIdx.x) * DIAG_NQ + threadIdx.x] =
      a[threadIdx.x];
}

__global__ void __launch_bounds__(DIAG_THREADS)
    k_diag_final(const double* __restrict__ partial, int nblk, double* __restrict__ out) {
  __shared__ double sh[(DIAG_THREADS / 32) * DIAG_NQ];
  const int b = blockIdx.x;
  double a[DIAG_NQ];
#pragma unroll
  for (int q = 0; q < DIAG_NQ; ++q) a[q] = 0.0;
  for (int k = threadIdx.x; k < nblk; k += DIAG_THREADS) {
    const double* p = partial + (size_t(b) * nblk + k) * DIAG_NQ;
#pragma unroll
    for (int q = 0; q < DIAG_NQ; ++q) a[q] = (q == 7) ? fmax(a[q], p[q]) : a[q] + p[q];
  }
  block_reduce(a, sh);
  if (threadIdx.x < DIAG_NQ)
    out[size_t(b) * DIAG_NQ + threadIdx.x] = threadIdx.x == 7 ? sqrt(a[threadIdx.x]) : a[threadIdx.x];
}

}  // namespace

cudaError_t launch_macros(int prec, int K, const void* fin, double* rho, double* u, const Dims& d,
                          cudaStream_t s) {
  switch (prec) {
    case 0: return macros_t<double, double>(K, static_cast<const double*>(fin), rho, u, d, s);
    case 1: return macros_t<float, float>(K, static_cast<const float*>(fin), rho, u, d, s);
    case 2: return macros_t<__half, float>(K, static_cast<const __half*>(fin), rho, u, d, s);
    case 3: return macros_t<__nv_bfloat16, float>(K, static_cast<const __nv_bfloat16*>(fin), rho, u, d, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_init(int prec, int K, void* f, const void* geo, const double* sqrtg,
                        const double* base_uth, const InitInst* ini, const double* rho_in,
                        const double* u_in, const Dims& d, cudaStream_t s) {
  const GeoDev<float>& gf = *static_cast<const GeoDev<float>*>(geo);
  switch (prec) {
    case 0:
      return init_t<double, double>(K, static_cast<double*>(f), *static_cast<const GeoDev<double>*>(geo),
                                    sqrtg, base_uth, ini, rho_in, u_in, d, s);
    case 1: return init_t<float, float>(K, static_cast<float*>(f), gf, sqrtg, base_uth, ini, rho_in, u_in, d, s);
    case 2: return init_t<__half, float>(K, static_cast<__half*>(f), gf, sqrtg, base_uth, ini, rho_in, u_in, d, s);
    case 3:
      return init_t<__nv_bfloat16, float>(K, static_cast<__nv_bfloat16*>(f), gf, sqrtg, base_uth, ini, rho_in,
                                          u_in, d, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_convert(int prec, int to_double, void* state, double* dbl, size_t n, const Dims& d,
                           cudaStream_t s) {
  static bool weights_set = false;
  if (!weights_set) {
    double w[Q];
    for (int l = 0; l < Q; ++l) w[l] = weight(l);
    cudaError_t e = cudaMemcpyToSymbol(c_weight, w, sizeof(w));
    if (e != cudaSuccess) return e;
    weights_set = true;
  }
  const int threads = 256;
  const size_t want = (n + threads - 1) / threads;
  const int blocks = int(want < 152 * 16 ? (want ? want : 1) : 152 * 16);
  switch (prec) {
    case 0: k_convert<double><<<blocks, threads, 0, s>>>(static_cast<double*>(state), dbl, n, d, to_double); break;
    case 1: k_convert<float><<<blocks, threads, 0, s>>>(static_cast<float*>(state), dbl, n, d, to_double); break;
    case 2: k_convert<__half><<<blocks, threads, 0, s>>>(static_cast<__half*>(state), dbl, n, d, to_double); break;
    case 3:
      k_convert<__nv_bfloat16><<<blocks, threads, 0, s>>>(static_cast<__nv_bfloat16*>(state), dbl, n, d,
                                                          to_double);
      break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

namespace {
template <typename S, typename Real>
cudaError_t velocity_change_t(int K, const S* fin, double* u_prev, const Dims& d, double* out, cudaStream_t s) {
  auto* o = reinterpret_cast<unsigned long long*>(out);
  cudaError_t e = cudaMemsetAsync(out, 0, size_t(d.batch) * 2 * sizeof(double), s);
  if (e != cudaSuccess) return e;
  const dim3 g((uint32_t(d.ncell) + 255) / 256, uint32_t(d.batch));
  switch (K) {
    case KFLAT: k_velocity_change<S, Real, KFLAT><<<g, 256, 0, s>>>(fin, u_prev, d, o); break;
    case KCYL: k_velocity_change<S, Real, KCYL><<<g, 256, 0, s>>>(fin, u_prev, d, o); break;
    case KELL: k_velocity_change<S, Real, KELL><<<g, 256, 0, s>>>(fin, u_prev, d, o); break;
    case KELT:
      if constexpr (!Codec<S, Real>::uses_ref) {  // FP64 / FP32 storage only
        k_velocity_change<S, Real, KELT><<<g, 256, 0, s>>>(fin, u_prev, d, o);
        break;
      }
      return cudaErrorInvalidValue;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}
}  // namespace

cudaError_t launch_velocity_change(int prec, int K, const void* fin, double* u_prev, const Dims& d, double* out,
                                   cudaStream_t s) {
  switch (prec) {
    case 0: return velocity_change_t<double, double>(K, static_cast<const double*>(fin), u_prev, d, out, s);
    case 1: return velocity_change_t<float, float>(K, static_cast<const float*>(fin), u_prev, d, out, s);
    case 2: return velocity_change_t<__half, float>(K, static_cast<const __half*>(fin), u_prev, d, out, s);
    case 3:
      return velocity_change_t<__nv_bfloat16, float>(K, static_cast<const __nv_bfloat16*>(fin), u_prev, d, out, s);
    default: return cudaErrorInvalidValue;
  }
}

// Row means of FP64 populations into the reference table (ref_index
// layout): one thread per (instance, row, population).
__global__ void k_ref_from_state(const double* __restrict__ dbl, float* __restrict__ ref, Dims d) {
  const size_t nrows = size_t(d.nr) * size_t(d.geo_rows3);
  const size_t t = blockIdx.x * size_t(blockDim.x) + threadIdx.x;
  if (t >= size_t(d.batch) * nrows * Q) return;
  const size_t l = t % Q, br = t / Q, b = br / nrows, row = br - b * nrows;
  const int ir = int(row / size_t(d.geo_rows3)), i3 = int(row - size_t(ir) * d.geo_rows3);
  const bool ell = d.geo_rows3 > 1;
  const int n3s = ell ? 1 : d.n3;
  const double* f = dbl + (b * Q + l) * size_t(d.ncell);
  double s = 0.0;
  for (int it = 0; it < d.nt; ++it)
    for (int k3 = 0; k3 < n3s; ++k3) s += f[(size_t(ir) * d.nt + it) * d.n3 + (ell ? i3 : k3)];
  const double mean = s / double(d.nt * n3s);
  float* rb = ref + b * Q * nrows;
  rb[ell ? l * nrows + row : row * Q + l] = float(mean);
}

cudaError_t launch_ref_from_state(const double* dbl, float* ref, const Dims& d, cudaStream_t s) {
  const size_t n = size_t(d.batch) * size_t(d.nr) * size_t(d.geo_rows3) * Q;
  k_ref_from_state<<<unsigned((n + 255) / 256), 256, 0, s>>>(dbl, ref, d);
  return cudaGetLastError();
}

cudaError_t launch_ref_table(int K, float* ref, const GeoDev<float>& geo, const double* sqrtg,
                             const double* base_uth, const double* rho_in, const double* u_in, const Dims& d,
                             int mode, cudaStream_t s) {
  const uint32_t n = uint32_t(d.batch) * uint32_t(d.nr) * uint32_t(d.geo_rows3);
  const uint32_t nb = (n + 255) / 256;
  switch (K) {
    case KFLAT: k_ref_table<KFLAT><<<nb, 256, 0, s>>>(ref, geo, sqrtg, base_uth, rho_in, u_in, d, mode); break;
    case KCYL: k_ref_table<KCYL><<<nb, 256, 0, s>>>(ref, geo, sqrtg, base_uth, rho_in, u_in, d, mode); break;
    case KELL: k_ref_table<KELL><<<nb, 256, 0, s>>>(ref, geo, sqrtg, base_uth, rho_in, u_in, d, mode); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

template <class S>
cudaError_t launch_stream_table_t(int K, float4* st, const float* ref, const InstParams<float>* inst,
                                  const void* fin, const Dims& d, cudaStream_t s) {
  const uint32_t n = uint32_t(d.batch) * uint32_t(d.nr) * uint32_t(d.st_rows3) * 2u;
  const uint32_t nb = (n + ST_THREADS - 1) / ST_THREADS;
  const S* f = static_cast<const S*>(fin);
  if (K == KFLAT) k_stream_table<KFLAT, S><<<nb, ST_THREADS, 0, s>>>(st, ref, inst, f, d);
  else if (K == KCYL) k_stream_table<KCYL, S><<<nb, ST_THREADS, 0, s>>>(st, ref, inst, f, d);
  else if (K == KELL) k_stream_table<KELL, S><<<nb, ST_THREADS, 0, s>>>(st, ref, inst, f, d);
  else return cudaErrorInvalidValue;
  return cudaGetLastError();
}

cudaError_t launch_stream_table(int prec, int K, float4* st, const float* ref, const InstParams<float>* inst,
                                const void* fin, const Dims& d, cudaStream_t s) {
  if (!st || !ref || d.st != st) return cudaErrorInvalidValue;
  if (prec == 2) return launch_stream_table_t<__half>(K, st, ref, inst, fin, d, s);
  if (prec == 3) return launch_stream_table_t<__nv_bfloat16>(K, st, ref, inst, fin, d, s);
  return cudaErrorInvalidValue;
}

cudaError_t launch_source_table(int4* tab, const Dims& d, cudaStream_t s) {
  const int n = axis_classes(d.nr) * d.src_nt * d.src_n3 * 4 * SRC_ROW;
  k_source_table<<<(n + 255) / 256, 256, 0, s>>>(reinterpret_cast<int*>(tab), d);
  return cudaGetLastError();
}

cudaError_t launch_diag(const double* rho, const double* u, const double* geo64, const Dims& d, double* partial,
                        int nblk, double* out, cudaStream_t s) {
  // about two blocks per SM over all instances (the blocks' reductions cost as
  // much as three rows), no more than rows for their warps
  const int rows = (d.nr * d.nt + DIAG_THREADS / 32 - 1) / (DIAG_THREADS / 32);
  const int want = (304 + d.batch - 1) / d.batch;
  const int blocks = std::min(nblk, std::min(rows, want));
  k_diag_partial<<<dim3(blocks, d.batch), DIAG_THREADS, 0, s>>>(rho, u, geo64, d, partial, blocks);
  k_diag_final<<<d.batch, DIAG_THREADS, 0, s>>>(partial, blocks, out);
  return cudaGetLastError();
}

}  // namespace lbgm
