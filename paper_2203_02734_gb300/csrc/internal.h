// internal.h -- what the translation units of the library share.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>

#include "../../include/pywolf_gb.h"

namespace pw {
struct ff2;
namespace smu {
template <class C> struct Inst;
template <class C> struct TabArgs;
}
}  // namespace pw

namespace pwi {

using Wide = pw::ff2;  // arithmetic of the batch's S and mu (smu.cuh)

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
  double A, scale;
  pw::ff2* tw2;  // N = 256: room for N twiddles
  float2* row;   // W(P1, .) or nullptr
  int iP, jP;
};
// ev: nullptr or three events around the two passes; err: flag of a bounded wait that gave up.
cudaError_t dispatch_planes(int N, const CUtensorMap& wmap, const PlaneArgs& q, int* err, cudaStream_t s,
                            cudaEvent_t* ev);

// S and mu without the CSDA (smu.cuh): the tables of n instances, then those of grid size N and launch round
// `chunk` among them (device lists, float pairs); or one instance (FP64).
cudaError_t launch_smu_list_tables(const pw::smu::TabArgs<Wide>* list, int n, cudaStream_t s);
cudaError_t launch_smu_list(int N, const pw::smu::Inst<Wide>* list, int n, int chunk, bool any_mu, cudaStream_t s);
cudaError_t launch_smu_one(const pw::smu::TabArgs<double2>& t, const pw::smu::Inst<double2>& q, cudaStream_t s);

}  // namespace pwi
