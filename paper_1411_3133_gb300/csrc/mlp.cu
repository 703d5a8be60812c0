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

#include <cmath>
#include <cstdint>
#include <cstring>
#include <string>
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

// Products C = A B on the FP32 pipes. Every output is one chain of FP32
// multiply-adds in ascending k, whatever the tile: training amplifies rounding
// (a weight that rounds to the other BF16 neighbour changes the gradients by
// 1e-3 of their rms), so the kernels' sums keep one order. Tensor cores with
// the FP32 operands split into three BF16 terms ran the four steps below in
// 0.72 ms, but with sums of their own order.
// 64 x 64 output tiles, 128 threads with 8 x 4 outputs each: 26 us for 4096 x
// 256 x 256 (20 TFLOP/s), as 4 x 4 outputs of 256 threads take, which read 8
// values of shared memory for 16 multiply-adds; 8 x 8 leave three warps on an
// SM and take 34 us. 32-deep k slices, loaded as 16-byte words where the operand
// allows it (VEC) into registers while the slice before is multiplied, double
// buffered in shared memory. Column groups of 4 are swizzled by k / 4, so that
// stores along k and reads along the columns meet no bank conflicts.
constexpr int TL = 64, TK = 32, LTHREADS = 128, QUADS = TL * TK / 4 / LTHREADS;
struct Tiles {
  float A[2][TK][TL];
  float B[2][TK][TL];
};

__device__ __forceinline__ float4 load4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 load4(const __nv_bfloat16* p) {
  const uint2 r = *reinterpret_cast<const uint2*>(p);
  return make_float4(__uint_as_float(r.x << 16), __uint_as_float(r.x & 0xffff0000u), __uint_as_float(r.y << 16),
                     __uint_as_float(r.y & 0xffff0000u));
}
__device__ __forceinline__ float load1(const float* p) { return *p; }
__device__ __forceinline__ float load1(const __nv_bfloat16* p) { return __bfloat162float(*p); }

// One thread's i-th quad of a slice [k0, k0 + TK) x [c0, c0 + 64). Operand with
// k contiguous (KC): element (k, c) at p[c * ld + k], a quad is 4 k of one c;
// else at p[k * ld + c], 4 c of one k. Zero outside k < K, c < C.
template <bool KC>
__device__ __forceinline__ void quad_at(int i, int& k, int& c) {
  const int x = int(threadIdx.x) + i * LTHREADS;
  k = KC ? (x & 7) * 4 : x >> 4;
  c = KC ? x >> 3 : (x & 15) * 4;
}
template <bool KC, bool VEC, class E>
__device__ __forceinline__ float4 slice_load(int i, const E* __restrict__ p, size_t ld, int k0, int c0, int K, int C) {
  int k, c;
  quad_at<KC>(i, k, c);
  k += k0;
  c += c0;
  float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
  if (k >= K || c >= C) return r;
  const E* q = KC ? p + size_t(c) * ld + k : p + size_t(k) * ld + c;
  if constexpr (VEC) return load4(q);  // K (KC) or C is a multiple of 4: whole words
  const int left = KC ? K - k : C - c;
  r.x = load1(q);
  if (left > 1) r.y = load1(q + 1);
  if (left > 2) r.z = load1(q + 2);
  if (left > 3) r.w = load1(q + 3);
  return r;
}
__device__ __forceinline__ int swizzled(int k, int group) { return (group ^ (k >> 2)) * 4; }
template <bool KC>
__device__ __forceinline__ void slice_store(int i, float (&s)[TK][TL], const float4& r) {
  int k, c;
  quad_at<KC>(i, k, c);
  if constexpr (KC) {
    const int at = swizzled(k, c >> 2) + (c & 3);  // k / 4 is the same for all four
    s[k][at] = r.x;
    s[k + 1][at] = r.y;
    s[k + 2][at] = r.z;
    s[k + 3][at] = r.w;
  } else {
    *reinterpret_cast<float4*>(&s[k][swizzled(k, c >> 2)]) = r;
  }
}

// acc += the 64 x 64 tile at (m0, n0) of A B over k in [0, K): the thread's rows
// are 4 ty .. and 32 + 4 ty .., its columns 4 tx ..
template <bool AKC, bool BKC, bool VEC, class TA, class TB>
__device__ __forceinline__ void tile_product(Tiles& sh, const TA* __restrict__ A, size_t lda, int M,
                                             const TB* __restrict__ B, size_t ldb, int N, int K, int m0, int n0,
                                             float (&acc)[8][4]) {
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  float4 ra[QUADS], rb[QUADS];
#pragma unroll
  for (int i = 0; i < QUADS; ++i) {
    ra[i] = slice_load<AKC, VEC>(i, A, lda, 0, m0, K, M);
    rb[i] = slice_load<BKC, VEC>(i, B, ldb, 0, n0, K, N);
  }
  int buf = 0;
  for (int k0 = 0; k0 < K; k0 += TK, buf ^= 1) {
#pragma unroll
    for (int i = 0; i < QUADS; ++i) {
      slice_store<AKC>(i, sh.A[buf], ra[i]);
      slice_store<BKC>(i, sh.B[buf], rb[i]);
    }
    __syncthreads();  // also: every warp is done with the slice that used this buffer
    if (k0 + TK < K) {
#pragma unroll
      for (int i = 0; i < QUADS; ++i) {
        ra[i] = slice_load<AKC, VEC>(i, A, lda, k0 + TK, m0, K, M);
        rb[i] = slice_load<BKC, VEC>(i, B, ldb, k0 + TK, n0, K, N);
      }
    }
#pragma unroll
    for (int kk = 0; kk < TK; ++kk) {
      float av[8], bv[4];
      *reinterpret_cast<float4*>(av) = load4(&sh.A[buf][kk][swizzled(kk, ty)]);
      *reinterpret_cast<float4*>(av + 4) = load4(&sh.A[buf][kk][swizzled(kk, ty + 8)]);
      *reinterpret_cast<float4*>(bv) = load4(&sh.B[buf][kk][swizzled(kk, tx)]);
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
    }
  }
}

// f(row, column, value) for the thread's outputs, in the tile.
template <class F>
__device__ __forceinline__ void for_outputs(const float (&acc)[8][4], F&& f) {
  const int r = (threadIdx.x >> 4) * 4, c = (threadIdx.x & 15) * 4;
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) f(r + (i & 3) + 32 * (i >> 2), c + j, acc[i][j]);
}

// Hidden layer: Z = in W^T + b, H = SiLU(Z); in n x fi, W fo x fi.
template <bool VEC>
__global__ void __launch_bounds__(LTHREADS) k_layer(int n, int fo, int fi, const float* __restrict__ in,
                                                       const __nv_bfloat16* __restrict__ W,
                                                       const float* __restrict__ bias, float* __restrict__ Z,
                                                       float* __restrict__ H) {
  __shared__ Tiles sh;
  const int m0 = blockIdx.x * TL, n0 = blockIdx.y * TL;
  float acc[8][4] = {};
  tile_product<true, true, VEC>(sh, in, fi, n, W, fi, fo, fi, m0, n0, acc);
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
__global__ void __launch_bounds__(LTHREADS) k_layer_back(int n, int fo, int fi, const float* __restrict__ dZn,
                                                            const __nv_bfloat16* __restrict__ W,
                                                            float* __restrict__ Z) {
  __shared__ Tiles sh;
  const int m0 = blockIdx.x * TL, n0 = blockIdx.y * TL;
  float acc[8][4] = {};
  tile_product<true, false, VEC>(sh, dZn, fo, n, W, fi, fi, fo, m0, n0, acc);
  for_outputs(acc, [&](int r, int c, float v) {
    if (m0 + r >= n || n0 + c >= fi) return;
    const size_t at = size_t(m0 + r) * fi + n0 + c;
    const float z = Z[at], s = sigmoidf(z);
    Z[at] = v * (s * (1.0f + z * (1.0f - s)));
  });
}

// Output layer of OUT_ROWS rows: Y = H W^T + b (4 outputs, one thread each, H
// and W staged in shared memory 256 columns at a time: 15 us for 4096 rows, 24
// with H read where it is used). Training (y not NULL):
// the gradient of the mean squared error of normalised outputs dY = 2 (Y - T) /
// (n NOUT), T = (y - mean) istd, its way back through the last hidden layer Z =
// (dY W) SiLU'(Z) (in place), and the block's partial sum of the squared error;
// else pred = Y std + mean.
constexpr int OUT_ROWS = 16, OUT_COLS = 256;
__global__ void __launch_bounds__(256) k_output(int n, int fi, const float* __restrict__ H,
                                                const __nv_bfloat16* __restrict__ W, const float* __restrict__ bias,
                                                const float* __restrict__ scale, const float* __restrict__ y,
                                                float* __restrict__ dY, float* __restrict__ Z,
                                                float* __restrict__ partial, float* __restrict__ pred) {
  __shared__ float s_d[OUT_ROWS][NOUT], s_e[OUT_ROWS * NOUT];
  __shared__ float s_h[OUT_ROWS][OUT_COLS + 1], s_w[NOUT][OUT_COLS + 1];
  const int row0 = blockIdx.x * OUT_ROWS;
  const int r = threadIdx.x / NOUT, q = threadIdx.x % NOUT, row = row0 + r;
  float o = 0.0f;
  for (int k0 = 0; k0 < fi; k0 += OUT_COLS) {
    const int k = k0 + int(threadIdx.x), ke = min(OUT_COLS, fi - k0);
    if (k < fi) {
#pragma unroll
      for (int i = 0; i < OUT_ROWS; ++i) s_h[i][threadIdx.x] = row0 + i < n ? H[size_t(row0 + i) * fi + k] : 0.0f;
#pragma unroll
      for (int i = 0; i < NOUT; ++i) s_w[i][threadIdx.x] = load1(W + size_t(i) * fi + k);
    }
    __syncthreads();
    if (threadIdx.x < OUT_ROWS * NOUT) {
#pragma unroll 16
      for (int j = 0; j < ke; ++j) o = fmaf(s_h[r][j], s_w[q][j], o);
    }
    __syncthreads();
  }
  if (threadIdx.x < OUT_ROWS * NOUT) {
    float d = 0.0f, e2 = 0.0f;
    if (row < n) {
      o += bias[q];
      if (y) {
        const float t = (y[size_t(row) * NOUT + q] - scale[q]) * scale[NOUT + q];
        const float e = o - t;
        d = 2.0f * e / float(n * NOUT);
        e2 = e * e;
        dY[size_t(row) * NOUT + q] = d;
      } else {
        pred[size_t(row) * NOUT + q] = o * scale[2 * NOUT + q] + scale[q];
      }
    }
    s_d[r][q] = d;
    s_e[threadIdx.x] = e2;
  }
  if (!y) return;
  __syncthreads();
  const int rows = min(OUT_ROWS, n - row0);
  for (int k = threadIdx.x; k < fi; k += 256) {
    float w[NOUT];
#pragma unroll
    for (int q = 0; q < NOUT; ++q) w[q] = load1(W + size_t(q) * fi + k);
    for (int r = 0; r < rows; ++r) {
      float g = 0.0f;
#pragma unroll
      for (int q = 0; q < NOUT; ++q) g = fmaf(s_d[r][q], w[q], g);
      float* zr = Z + size_t(row0 + r) * fi + k;
      const float z = *zr, s = sigmoidf(z);
      *zr = g * (s * (1.0f + z * (1.0f - s)));
    }
  }
  if (threadIdx.x == 0) {
    float t = 0.0f;
    for (int i = 0; i < OUT_ROWS * NOUT; ++i) t += s_e[i];
    partial[blockIdx.x] = t;
  }
}

__device__ __forceinline__ void copy_async(void* dst, const float* src, int bytes, bool valid) {
  const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
  const int n = valid ? bytes : 0;  // the rest is filled with zeros
  if (bytes == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(n) : "memory");
  else asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(n) : "memory");
}

// Gradients of every layer in one launch: dW[o][k] = sum_i dZ[i][o] in[i][k] by
// 32 x 32 tiles of 128 threads with 4 x 2 outputs (a 256 x 256 layer alone is 64
// blocks; the sums over the rows stay one chain, so smaller tiles are what
// spreads them over the SMs). A further block per 32 rows of dW sums the bias'
// gradient db[o] = sum_i dZ[i][o]. Too few warps to hide a load behind another's
// arithmetic: the slices of 32 rows arrive by cp.async, three of them in
// flight. 105 us for the 5 x 256 network on 4096 rows; 157 us with the next
// slice in registers and db summed from global memory.
constexpr int MAX_DEPTH = 16;
constexpr int TG = 32, GTHREADS = 128, GROWS = 32, GSTAGES = 4;
struct WeightJobs {
  int layers;
  struct {
    const float* dZ;
    const float* in;
    int fo, fi, tile0;
    bool vec_z, vec_in;  // rows are whole 16-byte words
    size_t w_off, b_off;
  } job[MAX_DEPTH];
};
__global__ void __launch_bounds__(GTHREADS) k_weight_grads(const __grid_constant__ WeightJobs jobs, int n,
                                                           float* __restrict__ g) {
  __shared__ float4 st[GSTAGES][2][GROWS][TG / 4];
  int l = 0;
  while (l + 1 < jobs.layers && int(blockIdx.x) >= jobs.job[l + 1].tile0) ++l;
  const auto& J = jobs.job[l];
  const int fo = J.fo, fi = J.fi;
  const float* __restrict__ dZ = J.dZ;
  const float* __restrict__ in = J.in;
  const int tiles_n = (fi + TG - 1) / TG + 1, tile = int(blockIdx.x) - J.tile0;
  const int m0 = tile / tiles_n * TG, n0 = tile % tiles_n * TG;
  const bool bias = tile % tiles_n == tiles_n - 1;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  // rows [k0, k0 + 32) of columns [c0, c0 + 32) of an operand
  auto fetch_one = [&](float4 (&dst)[GROWS][TG / 4], const float* __restrict__ p, int cols, bool vec, int c0, int k0) {
    if (vec) {
      const int c = c0 + (threadIdx.x & 7) * 4;
#pragma unroll
      for (int i = 0; i < GROWS * TG / 4 / GTHREADS; ++i) {
        const int k = (threadIdx.x >> 3) + i * (GTHREADS / 8), row = k0 + k;
        const bool ok = row < n && c < cols;
        copy_async(&dst[k][threadIdx.x & 7], ok ? p + size_t(row) * cols + c : p, 16, ok);
      }
    } else {
      const int c = c0 + (threadIdx.x & 31);
#pragma unroll
      for (int i = 0; i < GROWS * TG / GTHREADS; ++i) {
        const int k = (threadIdx.x >> 5) + i * (GTHREADS / 32), row = k0 + k;
        const bool ok = row < n && c < cols;
        copy_async(reinterpret_cast<float*>(dst[k]) + (threadIdx.x & 31), ok ? p + size_t(row) * cols + c : p, 4, ok);
      }
    }
  };
  auto fetch = [&](int s, int k0) {
    fetch_one(st[s][0], dZ, fo, J.vec_z, m0, k0);
    if (!bias) fetch_one(st[s][1], in, fi, J.vec_in, n0, k0);
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  for (int s = 0; s < GSTAGES - 1; ++s) fetch(s, s * GROWS);
  float acc[4][2] = {};
  float col = 0.0f;
  int s = 0;
  for (int k0 = 0; k0 < n; k0 += GROWS, s = (s + 1) % GSTAGES) {
    asm volatile("cp.async.wait_group %0;" ::"n"(GSTAGES - 2) : "memory");
    __syncthreads();  // the slice is there, and the one before has been read
    fetch((s + GSTAGES - 1) % GSTAGES, k0 + (GSTAGES - 1) * GROWS);
    if (bias) {
      if (threadIdx.x < TG) {
        const float* z = reinterpret_cast<const float*>(st[s][0]) + threadIdx.x;
#pragma unroll
        for (int kk = 0; kk < GROWS; ++kk) col += z[kk * TG];
      }
      continue;
    }
#pragma unroll
    for (int kk = 0; kk < GROWS; ++kk) {
      const float4 a = st[s][0][kk][ty];
      const float2 b = reinterpret_cast<const float2*>(st[s][1][kk])[tx];
      const float av[4] = {a.x, a.y, a.z, a.w}, bv[2] = {b.x, b.y};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  if (bias) {
    if (threadIdx.x < TG && m0 + int(threadIdx.x) < fo) g[J.b_off + m0 + threadIdx.x] = col;
    return;
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j)
      if (m0 + ty * 4 + i < fo && n0 + tx * 2 + j < fi)
        g[J.w_off + size_t(m0 + ty * 4 + i) * fi + n0 + tx * 2 + j] = acc[i][j];
}

// Adam on the FP32 master parameters; refreshes their BF16 copy. Block 0 also
// sums the loss.
__global__ void __launch_bounds__(256) k_adam(float* __restrict__ w, const float* __restrict__ g,
                                              float* __restrict__ m, float* __restrict__ v,
                                              __nv_bfloat16* __restrict__ wb, size_t count, float lr, float b1,
                                              float b2, float c1, float c2, float eps,
                                              const float* __restrict__ loss_part, int nloss, float denom,
                                              float* __restrict__ loss) {
  const size_t i = blockIdx.x * size_t(blockDim.x) + threadIdx.x;
  if (i < count) {
    const float gi = g[i];
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
    const dim3 grid((n + TL - 1) / TL, (fo + TL - 1) / TL);
    const bool vec = words(in, 4, fi) && words(W, 2, fi);
    (vec ? k_layer<true> : k_layer<false>)<<<grid, LTHREADS, 0, s>>>(n, fo, fi, in, W, net->w + net->b_off[l], net->Z[l],
                                                                net->H[l]);
    in = net->H[l];
  }
  return cudaGetLastError();
}

// The output layer (k_output): training on y, or the fields pred.
cudaError_t output(lb_mlp* net, int n, const float* y, float* pred) {
  const int l = net->depth - 1;
  k_output<<<nblk(n, OUT_ROWS), 256, 0, net->stream>>>(n, net->fan_in[l], net->H[l - 1], net->wb + net->w_off[l],
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
  if (e == cudaSuccess) e = alloc(n, &n->partial, nblk(max_batch, OUT_ROWS));
  if (e == cudaSuccess) e = alloc(n, &n->loss, 1);
  if (e == cudaSuccess) e = alloc(n, &n->scale, 3 * NOUT);
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
    const dim3 grid((count + TL - 1) / TL, (fi + TL - 1) / TL);
    const bool vec = words(n->Z[l], 4, fo) && words(W, 2, fi);
    (vec ? k_layer_back<true> : k_layer_back<false>)<<<grid, LTHREADS, 0, s>>>(count, fo, fi, n->Z[l], W, n->Z[l - 1]);
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
    J.vec_z = words(J.dZ, 4, J.fo);
    J.vec_in = words(J.in, 4, J.fi);
    J.tile0 = tiles;
    J.w_off = n->w_off[l];
    J.b_off = n->b_off[l];
    tiles += ((J.fo + TG - 1) / TG) * ((J.fi + TG - 1) / TG + 1);
  }
  k_weight_grads<<<unsigned(tiles), GTHREADS, 0, s>>>(jobs, count, n->g);
  LB_MCUDA(n, cudaGetLastError());
  ++n->steps;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.0f - std::pow(b1, float(n->steps)), c2 = 1.0f - std::pow(b2, float(n->steps));
  k_adam<<<nblk(n->nparam), 256, 0, s>>>(n->w, n->g, n->m, n->v, n->wb, n->nparam, lr, b1, b2, c1, c2, 1e-8f,
                                         n->partial, int(nblk(count, OUT_ROWS)), float(count * NOUT), n->loss);
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
