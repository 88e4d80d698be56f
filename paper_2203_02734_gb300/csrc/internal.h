// internal.h -- what the translation units of the library share.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>

#include "../../include/pywolf_gb.h"

namespace pw {
namespace smu {
struct Inst;
}
}  // namespace pw

namespace pwi {

// Sets the thread's message returned by pw_last_error().
void set_last_error(const char* msg);

// Tensor maps of a work buffer in the V layout and of W in planes (pywolf_gb.cu).
pw_status encode_vmap(CUtensorMap* map, void* work, int N);
pw_status encode_wmap(CUtensorMap* map, void* W, int N);

// Propagation of a GSM source plane by plane (plane.cuh) from its FP64-derived tables.
struct PlaneArgs {
  const float2* F;
  const float* G;
  const float2* tw;
  const float2* Eout;
  float2* work;  // 2 N^3 table values
  float2* W;
  float* S;
  float A, scale;
  float2* row;  // W(P1, .) or nullptr
  int iP, jP;
};
// ev: nullptr or three events around the two passes; err: flag of a bounded wait (N = 256 only).
cudaError_t dispatch_planes(int N, const CUtensorMap& wmap, const PlaneArgs& q, int* err, cudaStream_t s,
                            cudaEvent_t* ev);

// S and mu without the CSDA (smu.cuh) of the instances of grid size N and launch round `chunk` in
// list[0 .. n) (device), or of the one instance `one` where list is null (n = 1).
cudaError_t launch_smu(int N, const pw::smu::Inst* list, const pw::smu::Inst& one, int n, int chunk, bool any_mu,
                       cudaStream_t s);

}  // namespace pwi
