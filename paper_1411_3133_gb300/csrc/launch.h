// Host-side launchers of the device kernels (one translation unit per
// precision for the step kernel so that the large unrolled bodies compile in
// parallel).
#pragma once

#include <cuda_runtime.h>

#include <string>

#include "lbm_device.cuh"

namespace lbgm {

struct InitInst;

constexpr int SMS = 152;  // of a GB300

// Whether an FP64 step of `blocks` blocks is worth chaining. An SM that holds two
// blocks of one step needs twice as long for it (its FP64 units bound the step),
// and the blocks of the next step, which sit on the SMs while they wait, bring
// that about where the caller's other contexts step beside it. Cylinders, us a
// step chained / unchained: one context alone 20.0 / 22.6 at 64 to 144 blocks;
// three of 64 side by side 36.6 / 31.6, two of 96 37.9 / 31.4, four of 96 46.6 /
// 46.7. Below a third of the SMs the waiting blocks find
// SMs of their own (two contexts of 49 21.8, four of 24 24.7). FP32 arithmetic is
// bound by latency there and gains in every size (144 blocks 3.5 / 4.6).
constexpr bool fp64_chains(long long blocks) { return 3 * blocks <= SMS || blocks >= SMS; }

// chained: see launch_chained.
cudaError_t launch_step_f64(int K, const double* fin, double* fout, const GeoDev<double>& geo,
                            const InstParams<double>* inst, const Dims& d, int* flag, int threads,
                            bool chained, cudaStream_t s);
cudaError_t launch_step_f32(int K, const float* fin, float* fout, const GeoDev<float>& geo,
                            const InstParams<float>* inst, const Dims& d, int* flag, int threads,
                            bool chained, cudaStream_t s);
cudaError_t launch_step_h16(int K, const __half* fin, __half* fout, const GeoDev<float>& geo,
                            const InstParams<float>* inst, const Dims& d, int* flag, int threads,
                            bool chained, cudaStream_t s);
cudaError_t launch_step_b16(int K, const __nv_bfloat16* fin, __nv_bfloat16* fout, const GeoDev<float>& geo,
                            const InstParams<float>* inst, const Dims& d, int* flag, int threads,
                            bool chained, cudaStream_t s);

// Plain step whose instances may use the half-force velocity variant
// (InstParams::pad = 1); see step_shift.cu.
cudaError_t launch_step_shift_f64(int K, const double* fin, double* fout, const GeoDev<double>& geo,
                                  const InstParams<double>* inst, const Dims& d, int* flag, int threads,
                                  bool chained, cudaStream_t s);
cudaError_t launch_step_shift_f32(int K, const float* fin, float* fout, const GeoDev<float>& geo,
                                  const InstParams<float>* inst, const Dims& d, int* flag, int threads,
                                  bool chained, cudaStream_t s);

// Work-list step over `count` (at most LIST_MAX) instances of different
// geometry: their host records (ListInst), the work items of each and the
// tile, the nodes (FP32, FP64) or warps (2-byte storage) of an item; grid 0
// launches one block per item. 2-byte storage: a group of one metric kind, row
// kind and parity of n3 -- d any of its instances, smem the bytes of staged
// rows a block needs.
constexpr int LIST_MAX = 16;
cudaError_t launch_step_list_f64(int K, const void* recs, int count, const int* items, int tile, int threads,
                                 int grid, int parity, bool chained, cudaStream_t s);
cudaError_t step_list_occupancy_f64(int K, int threads, int* blocks_per_sm);
cudaError_t launch_step_list_f32(int K, const void* recs, int count, const int* items, int tile, int threads,
                                 int grid, int parity, bool chained, cudaStream_t s);
cudaError_t step_list_occupancy_f32(int K, int threads, int* blocks_per_sm);
cudaError_t launch_step_list_h16(int K, const Dims& d, size_t smem, const void* recs, int count, const int* items,
                                 int tile, int threads, int grid, int parity, bool chained, cudaStream_t s);
cudaError_t step_list_occupancy_h16(int K, const Dims& d, size_t smem, int threads, int* blocks_per_sm);
cudaError_t launch_step_list_b16(int K, const Dims& d, size_t smem, const void* recs, int count, const int* items,
                                 int tile, int threads, int grid, int parity, bool chained, cudaStream_t s);
cudaError_t step_list_occupancy_b16(int K, const Dims& d, size_t smem, int threads, int* blocks_per_sm);

// TMA-pipelined FP32 step (n3 in {128, 256}); map is a CUtensorMap over the
// input state (make_state_tensor_map).
bool tma_step_supported(const Dims& d);
size_t tensor_map_bytes();
cudaError_t make_state_tensor_map(void* map_out, const float* base, const Dims& d);
cudaError_t launch_step_tma_f32(int K, const void* map, const float* fin, float* fout,
                                const GeoDev<float>& geo, const InstParams<float>* inst, const Dims& d,
                                int* flag, cudaStream_t s);

// prec: 0 = FP64, 1 = FP32, 2 = FP16 deviations, 3 = BF16 deviations (state
// pointers of the storage type; geo a GeoDev<double> for FP64, else GeoDev<float>)
cudaError_t launch_macros(int prec, int K, const void* fin, double* rho, double* u, const Dims& d,
                          cudaStream_t s);
cudaError_t launch_init(int prec, int K, void* f, const void* geo, const double* sqrtg,
                        const double* base_uth, const InitInst* ini, const double* rho_in,
                        const double* u_in, const Dims& d, cudaStream_t s);
cudaError_t launch_convert(int prec, int to_double, void* state, double* dbl, size_t n, const Dims& d,
                           cudaStream_t s);
// Per instance max |u - u_prev| and max |u| into out[2 b], out[2 b + 1], then
// u_prev = u (k_velocity_change).
cudaError_t launch_velocity_change(int prec, int K, const void* fin, double* u_prev, const Dims& d, double* out,
                                   cudaStream_t s);
// Reference table from the row means of FP64 populations (k_ref_from_state).
cudaError_t launch_ref_from_state(const double* dbl, float* ref, const Dims& d, cudaStream_t s);
// Reference populations of 2-byte storage (k_ref_table): mode 0 weights,
// 1 the initial rows' equilibria (from the row means of rho_in / u_in if
// given, else base_uth, which may be NULL: rest).
cudaError_t launch_ref_table(int K, float* ref, const GeoDev<float>& geo, const double* sqrtg,
                             const double* base_uth, const double* rho_in, const double* u_in, const Dims& d,
                             int mode, cudaStream_t s);

// Stream table of 2-byte storage (k_stream_table) from the reference table
// and the instances' omega; prec 2 (FP16) or 3 (BF16), fin any state block.
cudaError_t launch_stream_table(int prec, int K, float4* st, const float* ref, const InstParams<float>* inst,
                                const void* fin, const Dims& d, cudaStream_t s);

// Source table of a channel (k_source_table): keys * SRC_ROW int4 at tab.
cudaError_t launch_source_table(int4* tab, const Dims& d, cudaStream_t s);

// Observables: NQ sums per instance written to out[batch * DIAG_NQ]. geo64
// holds diag_weights of each row (node for the theta-resolved kind); partial
// batch * nblk * DIAG_NQ doubles.
constexpr int DIAG_NQ = 9;
inline __host__ __device__ void diag_weights(const double* w, double* out) {
  // from (sqrt g, sqrt g_thth, wA, wOmega): g, sqrt(g_thth) wA, wA, wOmega / 2
  out[0] = w[0] * w[0];
  out[1] = w[1] * w[2];
  out[2] = w[2];
  out[3] = 0.5 * w[3];
}
cudaError_t launch_diag(const double* rho, const double* u, const double* geo64, const Dims& d, double* partial,
                        int nblk, double* out, cudaStream_t s);

// Message for lb_last_error(NULL) from entry points without a context.
void set_last_error_noctx(const std::string& msg);

}  // namespace lbgm
