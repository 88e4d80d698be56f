// smu.cu -- instantiations of smu.cuh: batches on float pairs, single calls in FP64.
#include "smu.cuh"

#include "internal.h"

namespace {
__global__ void __launch_bounds__(256) list_tables_kernel(const pw::smu::TabArgs<pwi::Wide>* t) {
  const pw::smu::TabArgs<pwi::Wide> a = t[blockIdx.x];
  pw::smu::tables(a, threadIdx.x, 256);
}
// One evaluation per thread, in blocks of 64 over the SMs.
__global__ void __launch_bounds__(64) one_tables_kernel(pw::smu::TabArgs<double2> t) {
  pw::smu::tables(t, blockIdx.x * 64 + threadIdx.x, gridDim.x * 64);
}
}  // namespace

namespace pwi {

cudaError_t launch_smu_list(int N, const pw::smu::Inst<Wide>* list, int n, int chunk, bool any_mu, cudaStream_t s) {
  switch (N) {
#define PW_CASE(NN) \
  case NN:          \
    return pw::smu::launch<NN, Wide>(list, {}, n, chunk, any_mu, s);
    PW_CASE(16) PW_CASE(32) PW_CASE(64) PW_CASE(96) PW_CASE(128)
#undef PW_CASE
    default:
      return cudaErrorInvalidValue;
  }
}

cudaError_t launch_smu_list_tables(const pw::smu::TabArgs<Wide>* list, int n, cudaStream_t s) {
  list_tables_kernel<<<n, 256, 0, s>>>(list);
  return cudaGetLastError();
}

cudaError_t launch_smu_one(const pw::smu::TabArgs<double2>& t, const pw::smu::Inst<double2>& q, cudaStream_t s) {
  one_tables_kernel<<<(5 * t.N + 63) / 64, 64, 0, s>>>(t);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  switch (q.N) {
#define PW_CASE(NN) \
  case NN:          \
    return pw::smu::launch<NN, double2>(nullptr, q, 1, 0, q.mu != nullptr, s);
    PW_CASE(4) PW_CASE(6) PW_CASE(8) PW_CASE(12) PW_CASE(16) PW_CASE(24) PW_CASE(32) PW_CASE(48) PW_CASE(64)
    PW_CASE(96) PW_CASE(128) PW_CASE(256)
#undef PW_CASE
    default:
      return cudaErrorInvalidValue;
  }
}

}  // namespace pwi
