// Surrogate of developed channel flow: a multilayer perceptron mapping
// channel parameters (Dean number, curvature ratio, ...) and a node's
// position to the macroscopic fields (rho', u^r, u^theta, u^3) of a
// converged LB run, used to warm-start the LB (lb_init_fields). Hand-written
// kernels for the forward pass, the backward pass and the Adam update;
// weights are kept in FP32 (master copy, Adam moments) and used in BF16 by
// every product, which accumulates in FP32.
//
// Layers: features phi(x) = (p_1 .. p_P, sin(2 pi k z), cos(2 pi k z), k =
// 1..F) of an input row (p_1 .. p_P, z),
// then depth - 1 hidden layers of `width` units with SiLU, then a linear
// output layer of 4 units. Outputs are normalised per field: the network
// predicts (y - mean) / std.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <string>
#include <type_traits>
#include <vector>

#include "../../include/lbgm.h"

namespace {

constexpr int NOUT = 4;

// --------------------------------------------------------------------------
// kernels
// --------------------------------------------------------------------------
// Row i of x holds np plain inputs then z; its features are the plain
// inputs then sin(2 pi k z), cos(2 pi k z), k = 1..nf.
__global__ void k_features(const float* __restrict__ x, int n, int np, int nf, float* __restrict__ phi) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int nin = np + 2 * nf;
  const float* xi = x + size_t(i) * (np + 1);
  float* o = phi + size_t(i) * nin;
  for (int j = 0; j < np; ++j) o[j] = xi[j];
  const float z = xi[np];
  for (int k = 1; k <= nf; ++k) {
    float s, c;
    sincospif(2.0f * float(k) * z, &s, &c);
    o[np + 2 * k - 2] = s;
    o[np + 2 * k - 1] = c;
  }
}

__device__ __forceinline__ float sigmoidf(float z) { return 1.0f / (1.0f + expf(-z)); }

// Products C = A B on the tensor cores (mma.sync m16n8k16, BF16 operands, FP32
// accumulation) with FP32 operands taken apart into three BF16 terms: a = h +
// m + l, each term the rounding of what the ones before left, holds all 24 bits
// of a, so against a BF16 weight the three products are exact and against
// another FP32 operand the six largest of the nine leave out 2^-26 of the
// product. 64 x 64 output tiles, 8 warps of 16 x 32; 32-deep k slices go
// through registers (loaded while the slice before is multiplied, as 16-byte
// words where the operand allows it, VEC) and are taken apart on their way to
// shared memory. A 4096 x 256 x 256 layer: 28 us as multiply-adds on the FP32
// pipes with the same tiles (33 % busy, 14 warps an SM), 30 us before that.
constexpr int TM = 64, TN = 64, TK = 32;
// A slice in shared memory: 64 columns of 32 k (KC, rows padded to 40) or 32 k
// of 64 columns (padded to 72); both are free of ldmatrix bank conflicts.
constexpr int PLANE = 64 * 40;
constexpr int ROW_KC = 40, ROW_CK = 72;

__device__ __forceinline__ float4 load4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ uint2 load4(const __nv_bfloat16* p) { return *reinterpret_cast<const uint2*>(p); }
__device__ __forceinline__ float load1(const float* p) { return *p; }
__device__ __forceinline__ float load1(const __nv_bfloat16* p) { return __bfloat162float(*p); }

// 4 consecutive elements of an operand in registers.
template <class T>
struct Quad;
template <>
struct Quad<float> {
  float4 v;
  static constexpr int planes = 3;
};
template <>
struct Quad<__nv_bfloat16> {
  uint2 v;
  static constexpr int planes = 1;
};
__device__ __forceinline__ uint32_t bf16x2(float lo, float hi) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ float lo_f(uint32_t r) { return __uint_as_float(r << 16); }
__device__ __forceinline__ float hi_f(uint32_t r) { return __uint_as_float(r & 0xffff0000u); }
// what a term leaves of x; nothing of an infinity or NaN, which the term holds
__device__ __forceinline__ float rest(float x, float term) { return fabsf(term) <= 3.4e38f ? x - term : 0.0f; }

// One thread's two quads of a slice [k0, k0 + TK) x [c0, c0 + 64). Operand with
// k contiguous (KC): element (k, c) at p[c * ld + k], a quad is 4 k of one c;
// else at p[k * ld + c], 4 c of one k. Zero outside k < K, c < C.
template <bool KC>
__device__ __forceinline__ void quad_at(int i, int& k, int& c) {
  const int x = int(threadIdx.x) + i * 256;
  k = KC ? (x & 7) * 4 : x >> 4;
  c = KC ? x >> 3 : (x & 15) * 4;
}
template <bool KC, bool VEC, class T>
__device__ __forceinline__ Quad<T> slice_load(int i, const T* __restrict__ p, size_t ld, int k0, int c0, int K, int C) {
  int k, c;
  quad_at<KC>(i, k, c);
  k += k0;
  c += c0;
  Quad<T> r;
  r.v = {};
  if (k >= K || c >= C) return r;
  const T* q = KC ? p + size_t(c) * ld + k : p + size_t(k) * ld + c;
  if constexpr (VEC) {  // K (KC) or C is a multiple of 4: whole words
    r.v = load4(q);
  } else {
    const int left = KC ? K - k : C - c;
    float e[4] = {load1(q), 0.f, 0.f, 0.f};
    for (int j = 1; j < 4; ++j)
      if (j < left) e[j] = load1(q + j);
    if constexpr (std::is_same<T, float>::value) r.v = make_float4(e[0], e[1], e[2], e[3]);
    else r.v = make_uint2(bf16x2(e[0], e[1]), bf16x2(e[2], e[3]));
  }
  return r;
}
template <bool KC, class T>
__device__ __forceinline__ void slice_store(int i, __nv_bfloat16* s, const Quad<T>& r) {
  int k, c;
  quad_at<KC>(i, k, c);
  __nv_bfloat16* at = s + (KC ? c * ROW_KC + k : k * ROW_CK + c);
  if constexpr (std::is_same<T, float>::value) {
    float4 x = r.v;
#pragma unroll
    for (int t = 0; t < 3; ++t) {
      const uint32_t a = bf16x2(x.x, x.y), b = bf16x2(x.z, x.w);
      *reinterpret_cast<uint2*>(at + t * PLANE) = make_uint2(a, b);
      x = make_float4(rest(x.x, lo_f(a)), rest(x.y, hi_f(a)), rest(x.z, lo_f(b)), rest(x.w, hi_f(b)));
    }
  } else {
    *reinterpret_cast<uint2*>(at) = r.v;
  }
}

template <bool TRANS>
__device__ __forceinline__ void ldmatrix4(uint32_t (&r)[4], const __nv_bfloat16* p) {
  const uint32_t a = static_cast<uint32_t>(__cvta_generic_to_shared(p));
  if constexpr (TRANS)
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(a)
                 : "memory");
  else
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(a)
                 : "memory");
}
__device__ __forceinline__ void mma(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// The warp's 16 x 32 outputs: acc[j] holds columns 8 j .. 8 j + 7 of its 32, in
// the layout of mma's accumulator: rows lane / 4 and lane / 4 + 8, columns
// 2 (lane % 4) and the next. f(row, column, value) for each, in the tile.
template <class F>
__device__ __forceinline__ void for_outputs(const float (&acc)[4][4], F&& f) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int r = (w >> 1) * 16 + lane / 4, c = (w & 1) * 32 + 2 * (lane & 3);
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int e = 0; e < 4; ++e) f(r + (e >> 1) * 8, c + 8 * j + (e & 1), acc[j][e]);
}

// acc += the 64 x 64 tile at (m0, n0) of A B over k in [kb, ke); colsum (A not
// KC; NULL: none) += the sums over the thread's k of its 4 columns of A.
template <bool AKC, bool BKC, bool VEC, class TA, class TB>
__device__ __forceinline__ void tile_product(__nv_bfloat16* sm, const TA* __restrict__ A, size_t lda, int M,
                                             const TB* __restrict__ B, size_t ldb, int N, int kb, int ke, int m0,
                                             int n0, float (&acc)[4][4], float4* colsum) {
  constexpr int PA = Quad<TA>::planes, PB = Quad<TB>::planes;
  __nv_bfloat16* sa = sm;
  __nv_bfloat16* sb = sm + PA * PLANE;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int mw = (w >> 1) * 16, nw = (w & 1) * 32, q = lane >> 3, r = lane & 7;
  Quad<TA> ra[2];
  Quad<TB> rb[2];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    ra[i] = slice_load<AKC, VEC>(i, A, lda, kb, m0, ke, M);
    rb[i] = slice_load<BKC, VEC>(i, B, ldb, kb, n0, ke, N);
  }
  for (int k0 = kb; k0 < ke; k0 += TK) {
    if (k0 > kb) __syncthreads();  // every warp is done with the slice before
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      slice_store<AKC>(i, sa, ra[i]);
      slice_store<BKC>(i, sb, rb[i]);
      if constexpr (!AKC) {
        if (colsum) {
          colsum->x += ra[i].v.x;
          colsum->y += ra[i].v.y;
          colsum->z += ra[i].v.z;
          colsum->w += ra[i].v.w;
        }
      }
    }
    __syncthreads();
    if (k0 + TK < ke) {
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        ra[i] = slice_load<AKC, VEC>(i, A, lda, k0 + TK, m0, ke, M);
        rb[i] = slice_load<BKC, VEC>(i, B, ldb, k0 + TK, n0, ke, N);
      }
    }
#pragma unroll
    for (int kk = 0; kk < TK; kk += 16) {
      uint32_t a[PA][4], b[PB][2][4];
#pragma unroll
      for (int t = 0; t < PA; ++t) {
        const __nv_bfloat16* s = sa + t * PLANE;
        if constexpr (AKC) ldmatrix4<false>(a[t], s + (mw + (lane & 15)) * ROW_KC + kk + (lane >> 4) * 8);
        else ldmatrix4<true>(a[t], s + (kk + (q >> 1) * 8 + r) * ROW_CK + mw + (q & 1) * 8);
      }
#pragma unroll
      for (int t = 0; t < PB; ++t)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const __nv_bfloat16* s = sb + t * PLANE;
          const int n = nw + 16 * h;
          if constexpr (BKC) ldmatrix4<false>(b[t][h], s + (n + (q >> 1) * 8 + r) * ROW_KC + kk + (q & 1) * 8);
          else ldmatrix4<true>(b[t][h], s + (kk + (q & 1) * 8 + r) * ROW_CK + n + (q >> 1) * 8);
        }
      // the sum over 16 k from zero, smallest terms first, then added to the
      // accumulators by FP32 additions: mma cuts its sum off instead of
      // rounding it, and over a chain of them the cuts add up (error of the
      // gradients against FP64 4.9e-6 where the FP32 pipes give 7e-7)
      float part[4][4] = {};
#pragma unroll
      for (int ta = PA - 1; ta >= 0; --ta)
#pragma unroll
        for (int tb = PB - 1; tb >= 0; --tb) {
          if (ta + tb > 2) continue;
#pragma unroll
          for (int j = 0; j < 4; ++j) mma(part[j], a[ta], b[tb][j >> 1][(j & 1) * 2], b[tb][j >> 1][(j & 1) * 2 + 1]);
        }
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[j][e] += part[j][e];
    }
  }
}

// Hidden layer: Z = in W^T + b, H = SiLU(Z); in n x fi, W fo x fi.
template <bool VEC>
__global__ void __launch_bounds__(256) k_layer(int n, int fo, int fi, const float* __restrict__ in,
                                               const __nv_bfloat16* __restrict__ W, const float* __restrict__ bias,
                                               float* __restrict__ Z, float* __restrict__ H) {
  __shared__ __align__(16) __nv_bfloat16 sm[4 * PLANE];
  const int m0 = blockIdx.x * TM, n0 = blockIdx.y * TN;
  float acc[4][4] = {};
  tile_product<true, true, VEC>(sm, in, fi, n, W, fi, fo, 0, fi, m0, n0, acc, nullptr);
  for_outputs(acc, [&](int r, int c, float v) {
    if (m0 + r >= n || n0 + c >= fo) return;
    const size_t at = size_t(m0 + r) * fo + n0 + c;
    const float z = v + bias[n0 + c];
    Z[at] = z;
    H[at] = z * sigmoidf(z);
  });
}

// Backward through a hidden layer: Z = (dZ_next W) SiLU'(Z), in place; dZ_next
// n x fo, W fo x fi, Z n x fi.
template <bool VEC>
__global__ void __launch_bounds__(256) k_layer_back(int n, int fo, int fi, const float* __restrict__ dZn,
                                                    const __nv_bfloat16* __restrict__ W, float* __restrict__ Z) {
  __shared__ __align__(16) __nv_bfloat16 sm[4 * PLANE];
  const int m0 = blockIdx.x * TM, n0 = blockIdx.y * TN;
  float acc[4][4] = {};
  tile_product<true, false, VEC>(sm, dZn, fo, n, W, fi, fi, 0, fo, m0, n0, acc, nullptr);
  for_outputs(acc, [&](int r, int c, float v) {
    if (m0 + r >= n || n0 + c >= fi) return;
    const size_t at = size_t(m0 + r) * fi + n0 + c;
    const float z = Z[at], s = sigmoidf(z);
    Z[at] = v * (s * (1.0f + z * (1.0f - s)));
  });
}

// Output layer, one warp per row: Y = H W^T + b (4 outputs). Training (y not
// NULL): the gradient of the mean squared error of normalised outputs dY =
// 2 (Y - T) / (n NOUT), T = (y - mean) istd, its way back through the last
// hidden layer Z = (dY W) SiLU'(Z) (in place), and per-block partial sums of
// the squared error; else pred = Y std + mean.
__global__ void __launch_bounds__(256) k_output(int n, int fi, const float* __restrict__ H,
                                                const __nv_bfloat16* __restrict__ W, const float* __restrict__ bias,
                                                const float* __restrict__ scale, const float* __restrict__ y,
                                                float* __restrict__ dY, float* __restrict__ Z,
                                                float* __restrict__ partial, float* __restrict__ pred) {
  __shared__ float s_e[8];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int row = blockIdx.x * 8 + wib;
  float e2 = 0.0f;
  if (row < n) {
    float o[NOUT] = {};
    const float* h = H + size_t(row) * fi;
    for (int k = lane; k < fi; k += 32) {
      const float hv = h[k];
#pragma unroll
      for (int q = 0; q < NOUT; ++q) o[q] = fmaf(hv, load1(W + size_t(q) * fi + k), o[q]);
    }
#pragma unroll
    for (int q = 0; q < NOUT; ++q) {
#pragma unroll
      for (int s = 16; s > 0; s >>= 1) o[q] += __shfl_xor_sync(0xffffffffu, o[q], s);
      o[q] += bias[q];
    }
    const float* mean = scale;
    const float* istd = scale + NOUT;
    const float* sd = scale + 2 * NOUT;
    if (y) {
      float d[NOUT];
#pragma unroll
      for (int q = 0; q < NOUT; ++q) {
        const float t = (y[size_t(row) * NOUT + q] - mean[q]) * istd[q];
        const float e = o[q] - t;
        d[q] = 2.0f * e / float(n * NOUT);
        e2 += e * e;
        if (lane == q) dY[size_t(row) * NOUT + q] = d[q];
      }
      float* zr = Z + size_t(row) * fi;
      for (int k = lane; k < fi; k += 32) {
        float g = 0.0f;
#pragma unroll
        for (int q = 0; q < NOUT; ++q) g = fmaf(d[q], load1(W + size_t(q) * fi + k), g);
        const float z = zr[k], s = sigmoidf(z);
        zr[k] = g * (s * (1.0f + z * (1.0f - s)));
      }
    } else {
#pragma unroll
      for (int q = 0; q < NOUT; ++q)
        if (lane == q) pred[size_t(row) * NOUT + q] = o[q] * sd[q] + mean[q];
    }
  }
  if (!y) return;
  if (lane == 0) s_e[wib] = e2;
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = 0.0f;
    for (int w = 0; w < 8; ++w) t += s_e[w];
    partial[blockIdx.x] = t;
  }
}

// Weight gradients of every layer in one launch: dW[o][k] = sum_i dZ[i][o]
// in[i][k], db[o] = sum_i dZ[i][o]. Grid x: 64 x 64 tiles of all layers, grid
// y: chunks of rows, each with its own copy of the gradient (part + y *
// nparam), summed by k_adam in a fixed order -- one chunk alone would leave
// the 16 tiles of a 256 x 256 layer on 16 SMs.
constexpr int MAX_DEPTH = 16;
struct WeightJobs {
  int layers;
  struct {
    const float* dZ;
    const float* in;
    int fo, fi, tile0, vec;
    size_t w_off, b_off;
  } job[MAX_DEPTH];
};
__global__ void __launch_bounds__(256) k_weight_grads(WeightJobs jobs, int n, int chunk, float* __restrict__ part,
                                                      size_t nparam) {
  __shared__ __align__(16) __nv_bfloat16 sm[6 * PLANE];
  int l = 0;
  while (l + 1 < jobs.layers && int(blockIdx.x) >= jobs.job[l + 1].tile0) ++l;
  const auto& J = jobs.job[l];
  const int tiles_n = (J.fi + TN - 1) / TN, tile = int(blockIdx.x) - J.tile0;
  const int m0 = tile / tiles_n * TM, n0 = tile % tiles_n * TN;
  const int kb = int(blockIdx.y) * chunk, ke = min(n, kb + chunk);
  float acc[4][4] = {};
  float4 cs = make_float4(0.f, 0.f, 0.f, 0.f);
  float4* csp = n0 == 0 ? &cs : nullptr;
  if (J.vec) tile_product<false, false, true>(sm, J.dZ, J.fo, J.fo, J.in, J.fi, J.fi, kb, ke, m0, n0, acc, csp);
  else tile_product<false, false, false>(sm, J.dZ, J.fo, J.fo, J.in, J.fi, J.fi, kb, ke, m0, n0, acc, csp);
  float* g = part + size_t(blockIdx.y) * nparam;
  for_outputs(acc, [&](int r, int c, float v) {
    if (m0 + r < J.fo && n0 + c < J.fi) g[J.w_off + size_t(m0 + r) * J.fi + n0 + c] = v;
  });
  if (csp) {  // thread t holds the sums of columns 4 (t % 16) .. over its k: add the 16 threads'
    float* s = reinterpret_cast<float*>(sm);
    __syncthreads();
    *reinterpret_cast<float4*>(s + (threadIdx.x >> 4) * TM + (threadIdx.x & 15) * 4) = cs;
    __syncthreads();
    if (threadIdx.x < TM && m0 + int(threadIdx.x) < J.fo) {
      float t = 0.0f;
#pragma unroll
      for (int k = 0; k < 16; ++k) t += s[k * TM + threadIdx.x];
      g[J.b_off + m0 + threadIdx.x] = t;
    }
  }
}

// Sum of the chunks' gradients, then Adam on the FP32 master parameters and
// their BF16 copy. Block 0 also sums the loss.
__global__ void __launch_bounds__(256) k_adam(float* __restrict__ w, float* __restrict__ g,
                                              const float* __restrict__ part, int chunks, float* __restrict__ m,
                                              float* __restrict__ v, __nv_bfloat16* __restrict__ wb, size_t count,
                                              float lr, float b1, float b2, float c1, float c2, float eps,
                                              const float* __restrict__ loss_part, int nloss, float denom,
                                              float* __restrict__ loss) {
  const size_t i = blockIdx.x * size_t(blockDim.x) + threadIdx.x;
  if (i < count) {
    float gi = part[i];
    for (int c = 1; c < chunks; ++c) gi += part[size_t(c) * count + i];
    g[i] = gi;
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float wi = w[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    w[i] = wi;
    wb[i] = __float2bfloat16_rn(wi);
  }
  if (blockIdx.x == 0) {
    __shared__ float sh[256];
    float s = 0.0f;
    for (int k = threadIdx.x; k < nloss; k += 256) s += loss_part[k];
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int k = 128; k > 0; k >>= 1) {
      if (threadIdx.x < k) sh[threadIdx.x] += sh[threadIdx.x + k];
      __syncthreads();
    }
    if (threadIdx.x == 0) *loss = sh[0] / denom;
  }
}

__global__ void k_to_bf16(const float* __restrict__ w, __nv_bfloat16* __restrict__ wb, size_t count) {
  const size_t i = blockIdx.x * size_t(blockDim.x) + threadIdx.x;
  if (i < count) wb[i] = __float2bfloat16_rn(w[i]);
}

unsigned nblk(size_t n, int t = 256) { return unsigned((n + t - 1) / t); }

}  // namespace

struct lb_mlp {
  int np = 0, nf = 0, width = 0, depth = 0, max_batch = 0, nin = 0;
  cudaStream_t stream = nullptr;
  std::vector<int> fan_in, fan_out;       // per layer
  std::vector<size_t> w_off, b_off;       // offsets into the parameter arrays
  size_t nparam = 0;
  float *w = nullptr, *g = nullptr, *m = nullptr, *v = nullptr;
  __nv_bfloat16* wb = nullptr;
  float *phi = nullptr, *dY = nullptr, *partial = nullptr, *loss = nullptr;
  std::vector<float*> Z, H;                // per hidden layer [max_batch][width]; Z becomes dZ backwards
  float* part = nullptr;                   // [max_chunks][nparam] weight gradients of row chunks
  int max_chunks = 1;
  float* scale = nullptr;                  // mean[4], istd[4], std[4]
  long long steps = 0;
  std::string err;
  std::vector<void*> allocs;
};

namespace {

thread_local std::string g_mlp_err;

lb_status mfail(lb_mlp* n, lb_status s, const std::string& msg) {
  if (n) n->err = msg;
  else g_mlp_err = msg;
  return s;
}

#define LB_MCUDA(n, call)                                                                 \
  do {                                                                                    \
    cudaError_t e_ = (call);                                                              \
    if (e_ != cudaSuccess) return mfail(n, LB_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
  } while (0)

template <class T>
cudaError_t alloc(lb_mlp* n, T** p, size_t count) {
  void* q = nullptr;
  cudaError_t e = cudaMalloc(&q, count * sizeof(T) + 16);
  if (e == cudaSuccess) {
    n->allocs.push_back(q);
    *p = static_cast<T*>(q);
  }
  return e;
}

// Whole 16-byte (8-byte BF16) words: rows of ld elements from an aligned base.
bool words(const void* p, size_t elem, int ld) {
  return ld % 4 == 0 && reinterpret_cast<uintptr_t>(p) % (4 * elem) == 0;
}

// Hidden layers of n rows; the last one's outputs land in n->H[depth - 2].
cudaError_t forward(lb_mlp* net, const float* x, int n) {
  cudaStream_t s = net->stream;
  k_features<<<nblk(n, 64), 64, 0, s>>>(x, n, net->np, net->nf, net->phi);
  const float* in = net->phi;
  for (int l = 0; l < net->depth - 1; ++l) {
    const int fi = net->fan_in[l], fo = net->fan_out[l];
    const __nv_bfloat16* W = net->wb + net->w_off[l];
    const dim3 grid((n + TM - 1) / TM, (fo + TN - 1) / TN);
    const bool vec = words(in, 4, fi) && words(W, 2, fi);
    (vec ? k_layer<true> : k_layer<false>)<<<grid, 256, 0, s>>>(n, fo, fi, in, W, net->w + net->b_off[l], net->Z[l],
                                                                net->H[l]);
    in = net->H[l];
  }
  return cudaGetLastError();
}

// The output layer (k_output): training on y, or the fields pred.
cudaError_t output(lb_mlp* net, int n, const float* y, float* pred) {
  const int l = net->depth - 1;
  k_output<<<nblk(n, 8), 256, 0, net->stream>>>(n, net->fan_in[l], net->H[l - 1], net->wb + net->w_off[l],
                                                net->w + net->b_off[l], net->scale, y, net->dY, net->Z[l - 1],
                                                net->partial, pred);
  return cudaGetLastError();
}

}  // namespace

extern "C" {

lb_status lb_mlp_create(int n_plain, int n_fourier, int width, int depth, int max_batch, unsigned long long seed,
                        void* cuda_stream, lb_mlp** out) {
  if (!out) return mfail(nullptr, LB_ERR_ARG, "null argument");
  *out = nullptr;
  if (n_plain < 1 || n_plain > 16 || n_fourier < 0 || n_fourier > 16 || width < 4 || width > 4096 || depth < 2 ||
      depth > 16 || max_batch < 1 || max_batch > (1 << 22))
    return mfail(nullptr, LB_ERR_ARG, "need 1 <= n_plain <= 16, 0 <= n_fourier <= 16, 4 <= width <= 4096, "
                                      "2 <= depth <= 16, 1 <= max_batch <= 4M");
  lb_mlp* n = new lb_mlp();
  n->np = n_plain;
  n->nf = n_fourier;
  n->width = width;
  n->depth = depth;
  n->max_batch = max_batch;
  n->nin = n_plain + 2 * n_fourier;
  n->stream = static_cast<cudaStream_t>(cuda_stream);
  for (int l = 0; l < depth; ++l) {
    n->fan_in.push_back(l == 0 ? n->nin : width);
    n->fan_out.push_back(l == depth - 1 ? NOUT : width);
  }
  for (int l = 0; l < depth; ++l) {
    n->w_off.push_back(n->nparam);
    n->nparam += size_t(n->fan_in[l]) * n->fan_out[l];
    n->b_off.push_back(n->nparam);
    n->nparam += size_t(n->fan_out[l]);
  }
  auto bail = [&](cudaError_t e) {
    const std::string m = std::string("allocation: ") + cudaGetErrorString(e);
    lb_mlp_destroy(n);
    return mfail(nullptr, LB_ERR_CUDA, m);
  };
  cudaError_t e = cudaSuccess;
  for (float** p : {&n->w, &n->g, &n->m, &n->v})
    if (e == cudaSuccess) e = alloc(n, p, n->nparam);
  if (e == cudaSuccess) e = alloc(n, &n->wb, n->nparam);
  if (e == cudaSuccess) e = alloc(n, &n->phi, size_t(max_batch) * n->nin);
  if (e == cudaSuccess) e = alloc(n, &n->dY, size_t(max_batch) * NOUT);
  if (e == cudaSuccess) e = alloc(n, &n->partial, nblk(max_batch, 8));
  if (e == cudaSuccess) e = alloc(n, &n->loss, 1);
  if (e == cudaSuccess) e = alloc(n, &n->scale, 3 * NOUT);
  // row chunks of 256 for the weight gradients, as many as 64 MB of copies hold
  n->max_chunks = int(std::min<size_t>((size_t(max_batch) + 255) / 256, std::max<size_t>(1, (size_t(64) << 20) / (4 * n->nparam))));
  if (e == cudaSuccess) e = alloc(n, &n->part, n->max_chunks * n->nparam);
  n->Z.assign(depth - 1, nullptr);
  n->H.assign(depth - 1, nullptr);
  for (int l = 0; l < depth - 1 && e == cudaSuccess; ++l) {
    e = alloc(n, &n->Z[l], size_t(max_batch) * width);
    if (e == cudaSuccess) e = alloc(n, &n->H[l], size_t(max_batch) * width);
  }
  if (e != cudaSuccess) return bail(e);
  // He-uniform initial weights (SplitMix64 stream), zero biases and moments
  std::vector<float> h(n->nparam, 0.0f);
  uint64_t k = 0;
  for (int l = 0; l < depth; ++l) {
    const double a = std::sqrt(6.0 / n->fan_in[l]) * (l == depth - 1 ? 0.5 : 1.0);
    for (size_t i = 0; i < size_t(n->fan_in[l]) * n->fan_out[l]; ++i) {
      uint64_t z = seed + (++k) * 0x9E3779B97F4A7C15ull;
      z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
      z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
      z ^= z >> 31;
      const double u = double(z >> 11) * 0x1.0p-53;
      h[n->w_off[l] + i] = float(a * (2.0 * u - 1.0));
    }
  }
  const float sc[3 * NOUT] = {0, 0, 0, 0, 1, 1, 1, 1, 1, 1, 1, 1};
  e = cudaMemcpy(n->w, h.data(), n->nparam * sizeof(float), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemset(n->m, 0, n->nparam * sizeof(float));
  if (e == cudaSuccess) e = cudaMemset(n->v, 0, n->nparam * sizeof(float));
  if (e == cudaSuccess) e = cudaMemcpy(n->scale, sc, sizeof(sc), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    k_to_bf16<<<nblk(n->nparam), 256, 0, n->stream>>>(n->w, n->wb, n->nparam);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(n->stream);
  if (e != cudaSuccess) return bail(e);
  *out = n;
  return LB_OK;
}

size_t lb_mlp_param_count(const lb_mlp* n) { return n ? n->nparam : 0; }

lb_status lb_mlp_set_output_scale(lb_mlp* n, const float* mean, const float* sd) {
  if (!n || !mean || !sd) return mfail(n, LB_ERR_ARG, "null argument");
  float h[3 * NOUT];
  for (int q = 0; q < NOUT; ++q) {
    if (!(sd[q] > 0.0f) || !std::isfinite(mean[q])) return mfail(n, LB_ERR_ARG, "need finite mean, std > 0");
    h[q] = mean[q];
    h[NOUT + q] = 1.0f / sd[q];
    h[2 * NOUT + q] = sd[q];
  }
  LB_MCUDA(n, cudaMemcpyAsync(n->scale, h, sizeof(h), cudaMemcpyHostToDevice, n->stream));
  LB_MCUDA(n, cudaStreamSynchronize(n->stream));
  return LB_OK;
}

lb_status lb_mlp_get_params(lb_mlp* n, float* host, size_t count) {
  if (!n || !host || count != n->nparam) return mfail(n, LB_ERR_ARG, "need a host buffer of lb_mlp_param_count floats");
  LB_MCUDA(n, cudaMemcpyAsync(host, n->w, count * sizeof(float), cudaMemcpyDeviceToHost, n->stream));
  LB_MCUDA(n, cudaStreamSynchronize(n->stream));
  return LB_OK;
}

lb_status lb_mlp_set_params(lb_mlp* n, const float* host, size_t count) {
  if (!n || !host || count != n->nparam) return mfail(n, LB_ERR_ARG, "need a host buffer of lb_mlp_param_count floats");
  LB_MCUDA(n, cudaMemcpyAsync(n->w, host, count * sizeof(float), cudaMemcpyHostToDevice, n->stream));
  k_to_bf16<<<nblk(count), 256, 0, n->stream>>>(n->w, n->wb, count);
  LB_MCUDA(n, cudaGetLastError());
  LB_MCUDA(n, cudaMemsetAsync(n->m, 0, count * sizeof(float), n->stream));
  LB_MCUDA(n, cudaMemsetAsync(n->v, 0, count * sizeof(float), n->stream));
  LB_MCUDA(n, cudaStreamSynchronize(n->stream));
  n->steps = 0;
  return LB_OK;
}

lb_status lb_mlp_predict(lb_mlp* n, const float* x, int count, float* y) {
  if (!n || (!x && count) || (!y && count)) return mfail(n, LB_ERR_ARG, "null argument");
  if (count < 0 || count > n->max_batch) return mfail(n, LB_ERR_ARG, "need 0 <= count <= max_batch");
  if (count == 0) return LB_OK;
  LB_MCUDA(n, forward(n, x, count));
  LB_MCUDA(n, output(n, count, nullptr, y));
  return LB_OK;
}

lb_status lb_mlp_train_step(lb_mlp* n, const float* x, const float* y, int count, float lr, float* loss) {
  if (!n || !x || !y) return mfail(n, LB_ERR_ARG, "null argument");
  if (count < 1 || count > n->max_batch) return mfail(n, LB_ERR_ARG, "need 1 <= count <= max_batch");
  if (!(lr > 0.0f) || !std::isfinite(lr)) return mfail(n, LB_ERR_ARG, "need lr > 0");
  cudaStream_t s = n->stream;
  LB_MCUDA(n, forward(n, x, count));
  LB_MCUDA(n, output(n, count, y, nullptr));  // leaves dZ of the last hidden layer in its Z
  for (int l = n->depth - 2; l > 0; --l) {
    const int fi = n->fan_in[l], fo = n->fan_out[l];
    const __nv_bfloat16* W = n->wb + n->w_off[l];
    const dim3 grid((count + TM - 1) / TM, (fi + TN - 1) / TN);
    const bool vec = words(n->Z[l], 4, fo) && words(W, 2, fi);
    (vec ? k_layer_back<true> : k_layer_back<false>)<<<grid, 256, 0, s>>>(count, fo, fi, n->Z[l], W, n->Z[l - 1]);
  }
  LB_MCUDA(n, cudaGetLastError());
  WeightJobs jobs;
  jobs.layers = n->depth;
  int tiles = 0;
  for (int l = 0; l < n->depth; ++l) {
    auto& J = jobs.job[l];
    J.fi = n->fan_in[l];
    J.fo = n->fan_out[l];
    J.dZ = l == n->depth - 1 ? n->dY : n->Z[l];
    J.in = l == 0 ? n->phi : n->H[l - 1];
    J.vec = words(J.dZ, 4, J.fo) && words(J.in, 4, J.fi);
    J.tile0 = tiles;
    J.w_off = n->w_off[l];
    J.b_off = n->b_off[l];
    tiles += ((J.fo + TM - 1) / TM) * ((J.fi + TN - 1) / TN);
  }
  int chunks = std::min(n->max_chunks, (count + 255) / 256);
  const int chunk = ((count + chunks - 1) / chunks + TK - 1) / TK * TK;
  chunks = (count + chunk - 1) / chunk;
  k_weight_grads<<<dim3(tiles, chunks), 256, 0, s>>>(jobs, count, chunk, n->part, n->nparam);
  LB_MCUDA(n, cudaGetLastError());
  ++n->steps;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.0f - std::pow(b1, float(n->steps)), c2 = 1.0f - std::pow(b2, float(n->steps));
  k_adam<<<nblk(n->nparam), 256, 0, s>>>(n->w, n->g, n->part, chunks, n->m, n->v, n->wb, n->nparam, lr, b1, b2, c1,
                                         c2, 1e-8f, n->partial, int(nblk(count, 8)), float(count * NOUT), n->loss);
  LB_MCUDA(n, cudaGetLastError());
  if (loss) {
    LB_MCUDA(n, cudaMemcpyAsync(loss, n->loss, sizeof(float), cudaMemcpyDeviceToHost, s));
    LB_MCUDA(n, cudaStreamSynchronize(s));
  }
  return LB_OK;
}

lb_status lb_mlp_get_grads(lb_mlp* n, float* host, size_t count) {
  if (!n || !host || count != n->nparam) return mfail(n, LB_ERR_ARG, "need a host buffer of lb_mlp_param_count floats");
  LB_MCUDA(n, cudaMemcpyAsync(host, n->g, count * sizeof(float), cudaMemcpyDeviceToHost, n->stream));
  LB_MCUDA(n, cudaStreamSynchronize(n->stream));
  return LB_OK;
}

void lb_mlp_destroy(lb_mlp* n) {
  if (!n) return;
  if (n->stream) cudaStreamSynchronize(n->stream);
  else cudaDeviceSynchronize();
  for (void* p : n->allocs) cudaFree(p);
  delete n;
}

const char* lb_mlp_last_error(const lb_mlp* n) { return n ? n->err.c_str() : g_mlp_err.c_str(); }

}  // extern "C"
