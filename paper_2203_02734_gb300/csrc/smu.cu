// smu.cu -- instantiations of smu.cuh.
#include "smu.cuh"

#include "internal.h"

namespace pwi {

cudaError_t launch_smu(int N, const pw::smu::Inst* list, const pw::smu::Inst& one, int n, int chunk, bool any_mu,
                       cudaStream_t s) {
  switch (N) {
#define PW_CASE(NN) \
  case NN:          \
    return pw::smu::launch<NN>(list, one, n, chunk, any_mu, s);
    PW_CASE(16) PW_CASE(32) PW_CASE(64) PW_CASE(96) PW_CASE(128)
#undef PW_CASE
    default:
      return cudaErrorInvalidValue;
  }
}

}  // namespace pwi
