// Stand-in for the kernel launchers (see fake_runtime.cpp).
#include <cstring>
#include <utility>
#include <vector>

#include "../paper_1411_3133_gb300/csrc/kernels.cuh"
#include "../paper_1411_3133_gb300/csrc/launch.h"

using Instances = std::vector<std::pair<const void*, void*>>;
void fake_step(const char* kind, const Instances& inst, int elem, double nodes, bool chained, int threads, cudaStream_t s,
               int tile = 0);

namespace lbgm {
namespace {

template <class S>
cudaError_t uniform(const char* kind, const S* fin, S* fout, const Dims& d, bool chained, int threads,
                    cudaStream_t s) {
  Instances inst;
  const size_t per = size_t(Q) * size_t(d.ncell);
  for (int b = 0; b < d.batch; ++b) inst.push_back({fin + b * per, fout + b * per});
  fake_step(kind, inst, sizeof(S), double(d.ncell) * d.batch, chained, threads, s);
  return cudaSuccess;
}

template <class S, class R>
cudaError_t listed(const char* kind, const void* recs, int count, int tile, int parity, bool chained, int threads,
                   cudaStream_t s) {
  Instances inst;
  double nodes = 0;
  const ListInst<S, R>* r = static_cast<const ListInst<S, R>*>(recs);
  for (int i = 0; i < count; ++i) {
    inst.push_back({parity ? r[i].f1 : r[i].f0, const_cast<S*>(parity ? r[i].f0 : r[i].f1)});
    nodes += r[i].d.ncell;
  }
  fake_step(kind, inst, sizeof(S), nodes, chained, threads, s, tile);
  return cudaSuccess;
}

}  // namespace

#define FAKE_STEP(NAME, KIND, S, R)                                                                               \
  cudaError_t NAME(int, const S* fin, S* fout, const GeoDev<R>&, const InstParams<R>*, const Dims& d, int*, int t, \
                   bool ch, cudaStream_t s) {                                                                     \
    return uniform(KIND, fin, fout, d, ch, t, s);                                                                 \
  }
FAKE_STEP(launch_step_f64, "f64", double, double)
FAKE_STEP(launch_step_f32, "f32", float, float)
FAKE_STEP(launch_step_h16, "h16", __half, float)
FAKE_STEP(launch_step_b16, "b16", __nv_bfloat16, float)
FAKE_STEP(launch_step_shift_f64, "shift64", double, double)
FAKE_STEP(launch_step_shift_f32, "shift32", float, float)

cudaError_t launch_step_list_f64(int, const void* r, int n, const int*, int tile, int t, int, int par, bool ch, cudaStream_t s) {
  return listed<double, double>("list64", r, n, tile, par, ch, t, s);
}
cudaError_t launch_step_list_f32(int, const void* r, int n, const int*, int tile, int t, int, int par, bool ch, cudaStream_t s) {
  return listed<float, float>("list32", r, n, tile, par, ch, t, s);
}
cudaError_t launch_step_list_h16(int, const Dims&, size_t, const void* r, int n, const int*, int tile, int t, int, int par,
                                 bool ch, cudaStream_t s) {
  return listed<__half, float>("listh16", r, n, tile, par, ch, t, s);
}
cudaError_t launch_step_list_b16(int, const Dims&, size_t, const void* r, int n, const int*, int tile, int t, int, int par,
                                 bool ch, cudaStream_t s) {
  return listed<__nv_bfloat16, float>("listb16", r, n, tile, par, ch, t, s);
}
cudaError_t step_list_occupancy_f64(int, int, int* o) { *o = 2; return cudaSuccess; }
cudaError_t step_list_occupancy_f32(int, int, int* o) { *o = 5; return cudaSuccess; }
cudaError_t step_list_occupancy_h16(int, const Dims&, size_t, int, int* o) { *o = 3; return cudaSuccess; }
cudaError_t step_list_occupancy_b16(int, const Dims&, size_t, int, int* o) { *o = 3; return cudaSuccess; }

bool tma_step_supported(const Dims& d) { return d.n3 == 128 || d.n3 == 256; }
size_t tensor_map_bytes() { return 128; }
cudaError_t make_state_tensor_map(void*, const float*, const Dims&) { return cudaSuccess; }
cudaError_t launch_step_tma_f32(int, const void*, const float* fin, float* fout, const GeoDev<float>&,
                                const InstParams<float>*, const Dims& d, int*, cudaStream_t s) {
  return uniform("tma", fin, fout, d, false, 0, s);
}
cudaError_t launch_macros(int, int, const void*, double*, double*, const Dims&, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_init(int prec, int, void* f, const void*, const double*, const double*, const InitInst*,
                        const double*, const double*, const Dims& d, cudaStream_t) {
  const size_t e = prec == 0 ? 8 : prec == 1 ? 4 : 2;
  for (int b = 0; b < d.batch; ++b) std::memset(static_cast<char*>(f) + b * size_t(Q) * d.ncell * e, 0, e);
  return cudaSuccess;
}
cudaError_t launch_convert(int, int, void*, double*, size_t, const Dims&, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_velocity_change(int, int, const void*, double*, const Dims&, double*, cudaStream_t) {
  return cudaSuccess;
}
cudaError_t launch_ref_from_state(const double*, float*, const Dims&, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_ref_table(int, float*, const GeoDev<float>&, const double*, const double*, const double*,
                             const double*, const Dims&, int, cudaStream_t) {
  return cudaSuccess;
}
cudaError_t launch_stream_table(int, int, float4*, const float*, const InstParams<float>*, const void*, const Dims&,
                                cudaStream_t) {
  return cudaSuccess;
}
cudaError_t launch_source_table(int4*, const Dims&, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_diag(const double*, const double*, const double*, const Dims&, double*, int, double*, cudaStream_t) {
  return cudaSuccess;
}

}  // namespace lbgm
