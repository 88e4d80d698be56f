// pywolf_gb.cu -- C ABI of include/pywolf_gb.h: handle state, argument checks, FP64 table
// set-up and the launch sequence of one propagation (by source: planes, passes over an array, closed
// form, dense contractions).
#include <cuda.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/pywolf_gb.h"
#include "internal.h"
#include "propagate.cuh"
#include "d256.cuh"
#include "dense.cuh"
#include "dense_tc.cuh"
#include "t256.cuh"
#include "delta.cuh"
#include "grad.cuh"
#include "plane.cuh"
#include "small.cuh"
#include "smu.cuh"
#include "r128.cuh"
#include "r64.cuh"
#include "r96.cuh"

namespace {

thread_local std::string g_err;

pw_status fail(pw_status s, const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof buf, fmt, ap);
  va_end(ap);
  g_err = buf;
  return s;
}

pw_status cuda_fail(cudaError_t e, const char* what) {
  cudaGetLastError();  // clear a sticky launch error so the next call starts clean
  return fail(PW_ECUDA, "%s: %s", what, cudaGetErrorString(e));
}

bool finite_pos(double v) { return std::isfinite(v) && v > 0.0; }

// Device pointers are dereferenced as 16-byte bulk / tensor copies (the CSDA buffers), 8-byte
// complex values (masks, uploaded arrays, mu) or floats (S, diagonals).
bool aligned(const void* p, size_t a) { return reinterpret_cast<uintptr_t>(p) % a == 0; }

enum SourceKind { SRC_NONE = 0, SRC_GSM = 1, SRC_ARRAY = 2, SRC_PROPAGATED = 3, SRC_DIAGONAL = 4 };

}  // namespace

namespace pwi {
void set_last_error(const char* msg) { g_err = msg; }
}  // namespace pwi

struct pw_csd {
  int N;
  double d;       // sampling of the current plane
  double lambda;
  pw_c32* W;
  pw_c32* work;
  cudaStream_t stream;
  // source of the current plane
  SourceKind kind;
  double sigma_S, sigma_mu, A;
  const pw_c32* W0;
  const float* diag;  // diagonal source values (SRC_DIAGONAL)
  int grad_rows[2];   // blocks of the adjoint's gradient kernel without and with a mu term (0: not queried yet)
  int hermitian;
  // masks of the current plane
  double aperture;  // <= 0: none
  double lens_f;    // 0: none
  const pw_c32* mask;
  // small device tables (one allocation)
  void* tables;
  float2* F;
  float2* M0;
  float* G;
  float2* tw;
  float2* Eout;
  float2* Ein;    // per-axis input factors
  float* S;       // S of the last propagated plane (the last pass's epilogue)
  int* err;       // device flag: a bounded wait in a kernel gave up
  unsigned* maxes;  // dense path: bits of the largest input component of each contraction (8 slots)
  // adjoint scratch (O(N^2)): the adjoint source (diagonal, P1 row), partial sums, the
  // GSM factor and far-field factors of the source grid, and a spare gradient triple
  float* adj_d;
  float2* adj_c;
  double* gpart;
  float* gtab;
  float2* qtab;
  double* g3tmp;
  CUtensorMap vmap;  // TMA map of the work buffer in the V layout
  CUtensorMap ymap;  // N = 256: the second pass's tiles of the work buffer
  CUtensorMap y3map;  // N = 256: the third pass's tiles of the work buffer
  CUtensorMap y1map;  // N = 256: the first pass's stores (four rows per warp) into the work buffer
  CUtensorMap wmap;   // planes of W, at N = 256 its column tiles (plane.cuh)
  int dft_mode;      // PW_DFT_AUTO, PW_DFT_FP32 or PW_DFT_TC_BF16X3
  int Nz;            // zero padding: transform size (0 = none); the dense path runs when set
  void* qbuf;        // split DFT matrices of the tensor-core dense path (allocated on first use)
  int stall;         // failure-detection test: chunk whose copy CTA 0 leaves out, next dense TC run only
  // optional per-pass timing: 4 events per recorded propagation (before the first pass, after it,
  // after the last, and between the second and third passes of the N = 256 engine)
  std::vector<cudaEvent_t> events;
  std::vector<char> three;  // per recorded propagation: the middle event was recorded
  int timed;
};

namespace {

bool supported(int N) {
  switch (N) {
    case 2: case 4: case 6: case 8: case 12: case 16: case 24: case 32: case 48: case 64:
    case 96: case 128: case 256:
      return true;
    default:
      return false;
  }
}

size_t table_bytes(int N) {
  const size_t NN = (size_t)N * N;
  const size_t base = NN * sizeof(float2) * 2 + NN * sizeof(float) * 2 + (size_t)N * sizeof(float2) * 3 + 1024 + 256;
  const size_t adj = NN * (sizeof(float) + sizeof(float2) + 3 * sizeof(double) + sizeof(float)) +
                     (size_t)N * sizeof(float2) + 3 * sizeof(double) + 6 * 256;
  return base + adj;
}

int num_sms() {
  static int n = 0;
  if (n == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (n <= 0) n = 1;
  }
  return n;
}

// Persistent grid: as many CTAs as fit on the device at once, at most one per slice.
template <class K>
cudaError_t persistent_grid(K kernel, int threads, size_t smem, int slices, int* grid) {
  int per_sm = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) per_sm = 1;
  const long g = (long)per_sm * num_sms();
  *grid = (int)(g < slices ? g : slices);
  return cudaSuccess;
}

template <int N>
cudaError_t launch_a(const CUtensorMap& vmap, const pw::PassAArgs& a, cudaStream_t s) {
  constexpr size_t smem = pw::pass_a_smem<N>();
  static int grid = 0;
  if (grid == 0) {
    cudaError_t e = cudaFuncSetAttribute(pw::pass_a_kernel<N, pw::SRC_ARRAY>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    e = persistent_grid(pw::pass_a_kernel<N, pw::SRC_ARRAY>, pw::Plan<N>::NT, smem, N * N, &grid);
    if (e != cudaSuccess) return e;
  }
  pw::pass_a_kernel<N, pw::SRC_ARRAY><<<grid, pw::Plan<N>::NT, smem, s>>>(vmap, a);
  return cudaGetLastError();
}

// N = 128: register-resident pass A (r128.cuh).
struct R128Extra {
  const float2* Ein;
  const float2* mask;
  int ap_ithr;
  int* err;
};

template <bool MASK>
cudaError_t launch_a_r128(const CUtensorMap& vmap, const pw::PassAArgs& a, const R128Extra& x, cudaStream_t s) {
  constexpr size_t smem = pw::r128::pass_a_smem();
  static int grid = 0;
  if (grid == 0) {
    cudaError_t e = cudaFuncSetAttribute(pw::r128::pass_a_r128<MASK>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    e = persistent_grid(pw::r128::pass_a_r128<MASK>, pw::r128::NT, smem, 128 * 128, &grid);
    if (e != cudaSuccess) return e;
  }
  pw::r128::pass_a_r128<MASK><<<grid, pw::r128::NT, smem, s>>>(vmap, a, x.Ein, x.mask, x.ap_ithr);
  return cudaGetLastError();
}

// N = 128, Hermitian store: register-resident pass B with prefetched gather (r128.cuh).
cudaError_t launch_b_r128(const pw::PassBArgs& b, cudaStream_t s) {
  constexpr size_t smem = pw::r128::pass_b_smem();
  static int grid = 0;
  if (grid == 0) {
    cudaError_t e = cudaFuncSetAttribute(pw::r128::pass_b_r128,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    e = persistent_grid(pw::r128::pass_b_r128, pw::r128::NT, smem, 128 * 128, &grid);
    if (e != cudaSuccess) return e;
  }
  pw::r128::pass_b_r128<<<grid, pw::r128::NT, smem, s>>>(b);
  return cudaGetLastError();
}

// N = 96: register-resident passes (r96.cuh), two CTAs per SM.
template <bool MASK>
cudaError_t launch_a_r96(const CUtensorMap& vmap, const pw::PassAArgs& a, const R128Extra& x, cudaStream_t s) {
  constexpr size_t smem = pw::r96::pass_a_smem();
  static int grid = 0;
  if (grid == 0) {
    cudaError_t e = cudaFuncSetAttribute(pw::r96::pass_a_r96<MASK>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    e = persistent_grid(pw::r96::pass_a_r96<MASK>, pw::r96::NT, smem, 96 * 96, &grid);
    if (e != cudaSuccess) return e;
  }
  pw::r96::pass_a_r96<MASK><<<grid, pw::r96::NT, smem, s>>>(vmap, a, x.Ein, x.mask, x.ap_ithr);
  return cudaGetLastError();
}

cudaError_t launch_b_r96(const pw::PassBArgs& b, cudaStream_t s) {
  constexpr size_t smem = pw::r96::pass_b_smem();
  static int grid = 0;
  if (grid == 0) {
    cudaError_t e = cudaFuncSetAttribute(pw::r96::pass_b_r96,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    e = persistent_grid(pw::r96::pass_b_r96, pw::r96::NT, smem, 96 * 96, &grid);
    if (e != cudaSuccess) return e;
  }
  pw::r96::pass_b_r96<<<grid, pw::r96::NT, smem, s>>>(b);
  return cudaGetLastError();
}

// N = 64: register-resident passes (r64.cuh), three CTAs per SM.
template <class K>
cudaError_t grid_r64(K kernel, int* grid) {
  if (*grid) return cudaSuccess;
  const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pw::r64::smem_bytes());
  return e != cudaSuccess ? e : persistent_grid(kernel, pw::r64::NT, pw::r64::smem_bytes(), 64 * 64, grid);
}

cudaError_t launch_a_r64(const CUtensorMap& vmap, const pw::PassAArgs& a, cudaStream_t s) {
  static int grid = 0;
  const cudaError_t e = grid_r64(pw::r64::pass_a_r64, &grid);
  if (e != cudaSuccess) return e;
  pw::r64::pass_a_r64<<<grid, pw::r64::NT, pw::r64::smem_bytes(), s>>>(vmap, a);
  return cudaGetLastError();
}

cudaError_t launch_b_r64(const pw::PassBArgs& b, cudaStream_t s) {
  static int grid = 0;
  const cudaError_t e = grid_r64(pw::r64::pass_b_r64, &grid);
  if (e != cudaSuccess) return e;
  pw::r64::pass_b_r64<<<grid, pw::r64::NT, pw::r64::smem_bytes(), s>>>(b);
  return cudaGetLastError();
}

// Number of CTAs of the largest grid of `cs`-CTA clusters of `kernel` that can be co-resident.
template <class K>
cudaError_t cluster_capacity(K kernel, int cs, int threads, size_t smem, int* grid) {
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cs;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cfg.gridDim = dim3(cs * num_sms());
  int nclusters = 0;
  e = cudaOccupancyMaxActiveClusters(&nclusters, kernel, &cfg);
  if (e != cudaSuccess) return e;
  if (nclusters < 1) return cudaErrorInvalidConfiguration;
  *grid = nclusters * cs;
  return cudaSuccess;
}

// Persistent launch of a kernel compiled for clusters of `cs` CTAs: as many clusters as can be
// co-resident (queried once per kernel, unless *grid is already set).
template <class K, class... Args>
cudaError_t launch_clusters(K kernel, int cs, int threads, size_t smem, int* grid, cudaStream_t s, Args... args) {
  if (*grid == 0) {
    cudaError_t e = cluster_capacity(kernel, cs, threads, smem, grid);
    if (e != cudaSuccess) return e;
  }
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cs;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cfg.gridDim = dim3(*grid);
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// N = 256, GSM source, first stage on the tensor cores: the comparison mode.
template <bool MASK>
cudaError_t launch_a_d256(const CUtensorMap& vmap, const pw::PassAArgs& a, const R128Extra& x, cudaStream_t s) {
  static int grid = 0;
  constexpr int CS = pw::d256::CLUSTER_A;
  if (grid == 0) {
    // The occupancy calculator fits one CTA per SM for a kernel that uses tensor memory (15
    // clusters of 8 instead of 36, measured). This one allocates 128 of an SM's 512 columns and
    // has the registers, threads and shared memory of its FP32 twin, which caps residency at two
    // CTAs per SM, so it takes the twin's grid (two per SM co-resident, measured: 53.8 -> 32.3 ms).
    cudaError_t e = cudaFuncSetAttribute(pw::d256::pass_a_d256<CS, MASK, true>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pw::d256::pass_a_smem<CS>());
    if (e != cudaSuccess) return e;
    e = cluster_capacity(pw::d256::pass_a_d256<CS, MASK, false>, CS, pw::d256::Geo<CS>::NT,
                         pw::d256::pass_a_smem<CS>(), &grid);
    if (e != cudaSuccess) return e;
  }
  return launch_clusters(pw::d256::pass_a_d256<CS, MASK, true>, CS, pw::d256::Geo<CS>::NT,
                         pw::d256::pass_a_smem<CS>(), &grid, s, vmap, a, x.Ein, x.mask, x.ap_ithr, x.err);
}

cudaError_t launch_b_d256(const pw::PassBArgs& b, cudaStream_t s) {
  static int grid = 0;
  constexpr int CS = pw::d256::CLUSTER_B;
  return launch_clusters(pw::d256::pass_b_d256<CS>, CS, pw::d256::Geo<CS>::NT, pw::d256::pass_b_smem<CS>(), &grid,
                         s, b);
}

template <int N, int WST>
cudaError_t launch_b(const pw::PassBArgs& b, cudaStream_t s) {
  constexpr size_t smem = pw::pass_b_smem<N>();
  static int grid = 0;
  if (grid == 0) {
    cudaError_t e = cudaFuncSetAttribute(pw::pass_b_kernel<N, WST>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    e = persistent_grid(pw::pass_b_kernel<N, WST>, pw::Plan<N>::NT, smem, N * N, &grid);
    if (e != cudaSuccess) return e;
  }
  pw::pass_b_kernel<N, WST><<<grid, pw::Plan<N>::NT, smem, s>>>(b);
  return cudaGetLastError();
}

// The two general passes of an uploaded or propagated array (N <= 128), or at N = 256 of a GSM source in the
// tensor-core comparison mode.  ev: nullptr or three events recorded before pass A, between the
// passes and after pass B.
template <int N>
cudaError_t launch_passes(bool herm, const CUtensorMap& vmap, const pw::PassAArgs& a, const pw::PassBArgs& b,
                          const R128Extra& x, cudaStream_t s, cudaEvent_t* ev) {
  cudaError_t e;
  if (ev && (e = cudaEventRecord(ev[0], s)) != cudaSuccess) return e;
  if constexpr (N == 256) e = x.mask ? launch_a_d256<true>(vmap, a, x, s) : launch_a_d256<false>(vmap, a, x, s);
  else if constexpr (N == 128) e = x.mask ? launch_a_r128<true>(vmap, a, x, s) : launch_a_r128<false>(vmap, a, x, s);
  else if constexpr (N == 96) e = x.mask ? launch_a_r96<true>(vmap, a, x, s) : launch_a_r96<false>(vmap, a, x, s);
  else if constexpr (N == 64) e = launch_a_r64(vmap, a, s);
  else e = launch_a<N>(vmap, a, s);
  if (e != cudaSuccess) return e;
  if (ev && (e = cudaEventRecord(ev[1], s)) != cudaSuccess) return e;
  if constexpr (N == 256) e = launch_b_d256(b, s);
  else if (!herm) e = launch_b<N, pw::W_GENERAL>(b, s);
  else if constexpr (N == 128) e = launch_b_r128(b, s);
  else if constexpr (N == 96) e = launch_b_r96(b, s);
  else if constexpr (N == 64) e = launch_b_r64(b, s);
  else e = launch_b<N, pw::W_HERM>(b, s);
  if (e != cudaSuccess) return e;
  if (ev && (e = cudaEventRecord(ev[2], s)) != cudaSuccess) return e;
  return cudaSuccess;
}

cudaError_t dispatch(int N, bool herm, const CUtensorMap& vmap, const pw::PassAArgs& a, const pw::PassBArgs& b,
                     const R128Extra& x, cudaStream_t s, cudaEvent_t* ev) {
  switch (N) {
#define PW_CASE(NN) \
  case NN:          \
    return launch_passes<NN>(herm, vmap, a, b, x, s, ev);
    PW_CASE(2) PW_CASE(4) PW_CASE(6) PW_CASE(8) PW_CASE(12) PW_CASE(16) PW_CASE(24)
    PW_CASE(32) PW_CASE(48) PW_CASE(64) PW_CASE(96) PW_CASE(128) PW_CASE(256)
#undef PW_CASE
    default:
      return cudaErrorInvalidValue;
  }
}

using pwi::PlaneArgs;

// N <= 16: tables and planes in one kernel (small.cuh), timed as the planes.
template <int N>
cudaError_t launch_small(const PlaneArgs& q, cudaStream_t s, cudaEvent_t* ev) {
  cudaError_t e;
  if (ev && ((e = cudaEventRecord(ev[0], s)) != cudaSuccess || (e = cudaEventRecord(ev[1], s)) != cudaSuccess)) return e;
  const pw::small::Scale sA(q.scale, q.A);
  const pw::small::Args a{q.F, q.G, q.tw, q.Eout, q.W, q.S, sA.scale, sA.pow2, q.row, q.iP, q.jP};
  if ((e = pw::small::launch<N>(a, s)) != cudaSuccess) return e;
  return ev ? cudaEventRecord(ev[2], s) : cudaSuccess;
}

template <int N>
cudaError_t launch_planes(const CUtensorMap& wmap, const PlaneArgs& q, int* err, cudaStream_t s, cudaEvent_t* ev) {
  namespace P = pw::plane;
  constexpr size_t N3 = (size_t)N * N * N;
  static int grid = 0;  // of the plane kernel
  cudaError_t e;
  constexpr auto kernel = [] {
    if constexpr (N == 64) return pw::r64::plane64_kernel;
    else if constexpr (N == 96) return P::plane96_kernel;
    else if constexpr (N == 128) return P::plane128_kernel;
    else return P::plane_kernel<N>;
  }();
  constexpr int nt = N == 64 ? pw::r64::NT : N == 96 ? pw::r96::NT : N == 128 ? pw::r128::NT : pw::Plan<N>::NT;
  constexpr size_t smem = N == 64 ? pw::r64::smem_bytes() : N == 96 ? P::plane96_smem() : N == 128 ? P::plane128_smem() : P::plane_smem<N>();
  if (grid == 0) {
    if ((e = cudaFuncSetAttribute(P::table_kernel<N>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)P::tab_smem<N>())) != cudaSuccess ||
        (e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess ||
        (e = persistent_grid(kernel, nt, smem, N * N, &grid)) != cudaSuccess)
      return e;
  }
  if (ev && (e = cudaEventRecord(ev[0], s)) != cudaSuccess) return e;
  const P::TabArgs ta{q.F, q.G, q.tw, q.Eout, q.work, q.work + N3, (float)q.A};
  P::table_kernel<N><<<dim3(N * (N / P::tab_lines<N>()), 2), P::tab_nt<N>(), P::tab_smem<N>(), s>>>(ta);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if (ev && (e = cudaEventRecord(ev[1], s)) != cudaSuccess) return e;
  const P::Args a{ta.H, ta.T, q.tw, q.Eout, q.W, q.S, (float)q.scale, q.row, q.iP, q.jP};
  if constexpr (N == 128) {
    kernel<<<grid, nt, smem, s>>>(a, err);
    P::diag_row_kernel<<<N * N / 256, 256, 0, s>>>(a, N);
  } else if constexpr (N == 64) {
    kernel<<<grid, nt, smem, s>>>(a);
  } else {
    kernel<<<grid, nt, smem, s>>>(wmap, a);
  }
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if (ev && (e = cudaEventRecord(ev[2], s)) != cudaSuccess) return e;
  return cudaSuccess;
}

cudaError_t launch_planes256(const CUtensorMap& wmap, const PlaneArgs& q, int* err, cudaStream_t s, cudaEvent_t* ev) {
  namespace P = pw::plane;
  constexpr int N = 256;
  constexpr size_t N3 = (size_t)N * N * N;
  static int grid = 0;  // of the column kernel
  cudaError_t e;
  if (grid == 0) {
    if ((e = cudaFuncSetAttribute(P::table256_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)P::table256_smem())) != cudaSuccess ||
        (e = cudaFuncSetAttribute(P::rows256_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)P::rows256_smem())) != cudaSuccess ||
        (e = cudaFuncSetAttribute(P::cols256_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)P::cols256_smem())) != cudaSuccess ||
        (e = persistent_grid(P::cols256_kernel, P::NT256, P::cols256_smem(), 1 << 30, &grid)) != cudaSuccess)
      return e;
  }
  if (ev && (e = cudaEventRecord(ev[0], s)) != cudaSuccess) return e;
  const P::TabArgs ta{q.F, q.G, q.tw, q.Eout, q.work, q.work + N3, (float)q.A};
  P::table256_tw_kernel<<<1, N, 0, s>>>(q.tw2);
  P::table256_kernel<<<dim3(N * (N / P::TAB_L256), 2), P::TAB_NT256, P::table256_smem(), s>>>(ta, q.tw2);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const P::Args a{ta.H, ta.T, q.tw, q.Eout, q.W, q.S, (float)q.scale, nullptr, 0, 0};
  P::rows256_kernel<<<N * (N / 16) * (N / P::ROWS_C), P::NT256, P::rows256_smem(), s>>>(a);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if (ev && (e = cudaEventRecord(ev[1], s)) != cudaSuccess) return e;
  P::cols256_kernel<<<grid, P::NT256, P::cols256_smem(), s>>>(wmap, a, err);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if (ev && (e = cudaEventRecord(ev[2], s)) != cudaSuccess) return e;
  return cudaSuccess;
}

}  // namespace

namespace pwi {
cudaError_t dispatch_planes(int N, const CUtensorMap& wmap, const PlaneArgs& q, int* err, cudaStream_t s,
                            cudaEvent_t* ev) {
  switch (N) {
#define PW_CASE(NN) \
  case NN:          \
    return launch_planes<NN>(wmap, q, err, s, ev);
    PW_CASE(24) PW_CASE(32) PW_CASE(48) PW_CASE(64) PW_CASE(96) PW_CASE(128)
#undef PW_CASE
#define PW_CASE(NN) \
  case NN:          \
    return launch_small<NN>(q, s, ev);
    PW_CASE(2) PW_CASE(4) PW_CASE(6) PW_CASE(8) PW_CASE(12) PW_CASE(16)
#undef PW_CASE
    case 256:
      return launch_planes256(wmap, q, err, s, ev);
    default:
      return cudaErrorInvalidValue;
  }
}

}  // namespace pwi

namespace {

// cuTensorMapEncodeTiled through the runtime's driver entry point (no link against libcuda).
PFN_cuTensorMapEncodeTiled_v12000 encode_tiled() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }
  return fn;
}

// N = 256 (three-pass engine): Y[a][b][k_l'][d' / 8][r][d' mod 8] in the work buffer as floats
// {64, 32, 64, N, N} (the innermost 64 floats are one 256-byte run of 4 r x 8 d'), with the second
// pass's box {64, 1, 1, N, 1} (one run for every b) and the third pass's box {16, 4, 1, 1, N} (the
// 64-byte pieces of one k_h in four consecutive runs, for every a); the first pass stores through
// the same array as floats {16, 4, 32, 64, N^2} with box {16, 1, 32, 4, 1} (four k_l' rows of
// one r: 128 pieces of 64 bytes).
pw_status make_t256_maps(pw_csd* h) {
  auto enc = encode_tiled();
  if (!enc) return fail(PW_ECUDA, "cuTensorMapEncodeTiled is not available from the driver");
  constexpr cuuint64_t N = 256, run = 64 * sizeof(float);
  cuuint32_t estr[5] = {1, 1, 1, 1, 1};
  const cuuint64_t dims[5] = {64, 32, 64, N, N};
  const cuuint64_t strides[4] = {run, run * 32, run * 32 * 64, run * 32 * 64 * N};
  const cuuint32_t box2[5] = {64, 1, 1, (cuuint32_t)N, 1}, box3[5] = {16, 4, 1, 1, (cuuint32_t)N};
  CUresult r = enc(&h->ymap, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 5, h->work, dims, strides, box2, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return fail(PW_ECUDA, "cuTensorMapEncodeTiled (second-pass tiles) failed (CUresult %d)", (int)r);
  r = enc(&h->y3map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 5, h->work, dims, strides, box3, estr,
          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE,
          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return fail(PW_ECUDA, "cuTensorMapEncodeTiled (third-pass tiles) failed (CUresult %d)", (int)r);
  {
    const cuuint64_t d1[5] = {16, 4, 32, 64, N * N};
    const cuuint64_t s1[4] = {64, 256, 256 * 32, 256 * 32 * 64};
    const cuuint32_t b1[5] = {16, 1, 32, 4, 1};
    r = enc(&h->y1map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 5, h->work, d1, s1, b1, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(PW_ECUDA, "cuTensorMapEncodeTiled (first-pass rows) failed (CUresult %d)", (int)r);
  }
  return PW_OK;
}

pw_status make_vmap(pw_csd* h) {
  pw_status st = pwi::encode_vmap(&h->vmap, h->work, h->N);
  if (st == PW_OK) st = pwi::encode_wmap(&h->wmap, h->W, h->N);
  if (st == PW_OK && h->N == 256) st = make_t256_maps(h);
  return st;
}

// Fill F, G, tw, Eout for a propagation over z (z <= 0: source-plane view only), and M0 where it is used.
pw_status build_tables(pw_csd* h, double z, bool farfield, bool want_m0 = false) {
  const int N = h->N;
  const double d = h->d, lam = h->lambda;
  pw::TableArgs t{};
  t.N = N;
  const double invf = h->lens_f != 0.0 ? 1.0 / h->lens_f : 0.0;
  const double base = d * d / (2.0 * lam);
  t.K0 = -base * invf;
  if (z > 0.0) {
    t.Kin = farfield ? -base * invf : base * (1.0 / z - invf);
    const double dx = lam * z / (N * d);
    t.Kout = dx * dx / (2.0 * lam * z);
  }
  if (h->kind == SRC_GSM) {
    t.gs = d * d / (4.0 * h->sigma_S * h->sigma_S);
    t.gm = d * d / (2.0 * h->sigma_mu * h->sigma_mu);
    t.G = h->G;
  }
  if (h->aperture > 0.0) {
    const double rp = h->aperture / d;
    t.ap_thr = rp * rp;
  } else {
    t.ap_thr = -1.0;
  }
  t.mask = reinterpret_cast<const float2*>(h->mask);
  t.F = h->F;
  t.M0 = want_m0 ? h->M0 : nullptr;
  t.tw = h->tw;
  t.Eout = h->Eout;
  t.Ein = h->Ein;
  pw::tables_kernel<<<pw::tables_grid(t), pw::TABLE_NT, 0, h->stream>>>(t);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e, "table kernel launch");
  return PW_OK;
}

// The output plane becomes the current plane: its CSDA is in W, its masks are unset.
void to_output_plane(pw_csd* h, double dx, bool herm) {
  h->d = dx;
  h->kind = SRC_PROPAGATED;
  h->hermitian = herm ? 1 : 0;
  h->W0 = nullptr;
  h->diag = nullptr;
  h->aperture = 0.0;
  h->lens_f = 0.0;
  h->mask = nullptr;
}

// The next recorded propagation's events, or nullptr.
cudaEvent_t* next_events(pw_csd* h) {
  if (h->events.empty() || (size_t)(4 * (h->timed + 1)) > h->events.size()) return nullptr;
  h->three[h->timed] = 0;
  return &h->events[4 * h->timed++];
}

bool has_masks(const pw_csd* h) { return h->aperture > 0.0 || h->lens_f != 0.0 || h->mask != nullptr; }

// Launches one tensor-core contraction of the dense path.
cudaError_t launch_axis_tc(const pw::dense_tc::Args& ax, int mode, const unsigned char* q, int* err, cudaStream_t s) {
  namespace T = pw::dense_tc;
  static size_t smem_set = 0;  // the limit is raised once per size
  const size_t smem = T::smem_bytes(ax.N);
  auto set = [&](auto k) { return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem); };
  auto all = [&](auto f) -> cudaError_t {
    cudaError_t e;
    if ((e = f(T::axis_tc_kernel<2, T::IN_COLS>)) != cudaSuccess || (e = f(T::axis_tc_kernel<2, T::IN_ROWS>)) != cudaSuccess ||
        (e = f(T::axis_tc_kernel<2, T::IN_MASK>)) != cudaSuccess || (e = f(T::axis_tc_kernel<2, T::IN_PRODUCT>)) != cudaSuccess ||
        (e = f(T::axis_tc_kernel<3, T::IN_COLS>)) != cudaSuccess || (e = f(T::axis_tc_kernel<3, T::IN_ROWS>)) != cudaSuccess ||
        (e = f(T::axis_tc_kernel<3, T::IN_MASK>)) != cudaSuccess)
      return e;
    return f(T::axis_tc_kernel<3, T::IN_PRODUCT>);
  };
  if (smem > smem_set) {
    const cudaError_t e = all(set);
    if (e != cudaSuccess) return e;
    smem_set = smem;
  }
  const dim3 grid((unsigned)((ax.ncols + 127) / 128 * T::parts(ax.N)));
  auto go = [&](auto k) { k<<<grid, T::NT, smem, s>>>(ax, q, err); };
  const bool two = T::b_buffers(ax.N) == 2;
  switch (mode) {
    case T::IN_COLS: two ? go(T::axis_tc_kernel<2, T::IN_COLS>) : go(T::axis_tc_kernel<3, T::IN_COLS>); break;
    case T::IN_ROWS: two ? go(T::axis_tc_kernel<2, T::IN_ROWS>) : go(T::axis_tc_kernel<3, T::IN_ROWS>); break;
    case T::IN_MASK: two ? go(T::axis_tc_kernel<2, T::IN_MASK>) : go(T::axis_tc_kernel<3, T::IN_MASK>); break;
    default: two ? go(T::axis_tc_kernel<2, T::IN_PRODUCT>) : go(T::axis_tc_kernel<3, T::IN_PRODUCT>); break;
  }
  return cudaGetLastError();
}

// Zero padding (Nz > N) or a grid size without an FFT plan: dense axis contractions (dense.cuh).
//   Tensor cores (dense_tc.cuh), GSM source: the tables H and T (in W), then d (-> work) and a (-> W, with
//     the scale and S).  Other sources: d (masks applied on the way in), c, b, a, alternating between
//     work and W.
//   CUDA cores: W0 is built in W, then d (W -> work), c (work -> W), b (W -> work) and a (work -> W).
// Events as for the FFT passes: the first half of the contractions counts as the first pass.
pw_status propagate_dense(pw_csd* h, double z, bool farfield, bool herm) {
  const int N = h->N, Nz = h->Nz > 0 ? h->Nz : N;
  pw_status st = build_tables(h, z, farfield, true);  // G and M0 (the FFT factors are not used here)
  if (st != PW_OK) return st;
  const double d = h->d, lz = h->lambda * z, dx = lz / (Nz * d);
  cudaStream_t s = h->stream;
  cudaEvent_t* ev = next_events(h);
  cudaError_t e = cudaSuccess;
  if (ev && (e = cudaEventRecord(ev[0], s)) != cudaSuccess) return cuda_fail(e, "event record");
  pw::dense::TabArgs t{};
  t.N = N;
  t.Nz = Nz;
  t.Kin = farfield ? 0.0 : d * d / (2.0 * lz);
  t.Kout = dx * dx / (2.0 * lz);
  t.E = h->F;  // the FFT input factor's storage (N x N complex) holds E on this path
  t.max = h->maxes;
  const int NN = N * N;
  pw::dense::tables_kernel<<<(NN + 255) / 256, 256, 0, s>>>(t);
  pw::dense::SrcArgs sa{};
  sa.N = N;
  sa.mode = h->kind == SRC_GSM ? pw::SRC_GSM : (h->kind == SRC_DIAGONAL ? pw::SRC_DIAG : pw::SRC_ARRAY);
  sa.G = h->G;
  sa.M0 = h->M0;
  sa.W0 = reinterpret_cast<const float2*>(h->kind == SRC_PROPAGATED ? h->W : h->W0);
  sa.diag = h->diag;
  sa.A = (float)h->A;
  sa.W = reinterpret_cast<float2*>(h->W);
  const bool tc = h->dft_mode != PW_DFT_FP32 && N <= pw::dense_tc::MAX_N;
  float2* Wf = reinterpret_cast<float2*>(h->W);
  float2* Xf = reinterpret_cast<float2*>(h->work);
  const long long L[4] = {1, N, (long long)N * N, (long long)N * N * N};
  const float scale = (float)((d * d / lz) * (d * d / lz));
  if (tc) {
    namespace T = pw::dense_tc;
    // the split matrices of E (point 2) and conj(E) (point 1)
    const size_t qb = T::q_bytes(N);
    if (!h->qbuf && (e = cudaMalloc(&h->qbuf, 2 * qb)) != cudaSuccess) return cuda_fail(e, "cudaMalloc of the split DFT matrices");
    unsigned char* q = reinterpret_cast<unsigned char*>(h->qbuf);
    for (int cj = 0; cj < 2; ++cj) {
      T::QArgs qa{N, h->F, cj, q + cj * qb};
      T::qsplit_kernel<<<num_sms() * 4, 256, 0, s>>>(qa);
    }
    unsigned* mx = h->maxes;  // zeroed by tables_kernel
    T::Args ax{};
    ax.N = N;
    ax.scale = 1.0f;
    ax.vec = 1;
    const int stall = h->stall;  // first contraction of the N^4 array only, then cleared
    h->stall = 0;
    if (sa.mode == pw::SRC_GSM) {
      const size_t N3 = (size_t)N * N * N;
      unsigned* cm = reinterpret_cast<unsigned*>(h->adj_c);  // 2 N^2 column maxima in the adjoint's scratch
      T::TableArgs ta{N, h->G, h->M0, (float)h->A, Xf, Xf + N3, cm};
      T::table_source_kernel<<<dim3((N + T::TS_D - 1) / T::TS_D, N, 2), T::TS_D * T::TS_B, 0, s>>>(ta);
      float2 *H = Wf, *Tt = Wf + N3;
      ax.L = N;
      ax.ncols = (long long)NN;
      ax.in = ta.H0;
      ax.out = H;
      ax.max_col = cm;
      if ((e = launch_axis_tc(ax, T::IN_COLS, q + qb, h->err, s)) != cudaSuccess) return cuda_fail(e, "table contraction");
      ax.in = ta.T0;
      ax.out = Tt;
      ax.max_col = cm + NN;
      if ((e = launch_axis_tc(ax, T::IN_COLS, q, h->err, s)) != cudaSuccess) return cuda_fail(e, "table contraction");
      T::table_max_kernel<<<(NN + 255) / 256, 256, 0, s>>>(N, H, Tt, mx + 2);
      ax.L = 1;
      ax.ncols = (long long)N3;
      ax.in = nullptr;
      ax.max_col = nullptr;
      ax.H = H;
      ax.T = Tt;
      ax.out = Xf;
      ax.max_in = mx + 2;
      ax.max_out = mx + 3;
      ax.stall = stall;
      if ((e = launch_axis_tc(ax, T::IN_PRODUCT, q, h->err, s)) != cudaSuccess) return cuda_fail(e, "dense contraction");
      if (ev && (e = cudaEventRecord(ev[1], s)) != cudaSuccess) return cuda_fail(e, "event record");
      ax.stall = 0;
      ax.L = L[3];
      ax.in = Xf;
      ax.out = Wf;
      ax.scale = scale;
      ax.S = h->S;
      ax.max_in = mx + 3;
      ax.max_out = nullptr;
      if ((e = launch_axis_tc(ax, T::IN_COLS, q + qb, h->err, s)) != cudaSuccess) return cuda_fail(e, "dense contraction");
    } else {
      const float2* src = sa.W0;
      int mode = T::IN_MASK;
      if (sa.mode == pw::SRC_DIAG) {  // N^2 non-zeros: built in W
        sa.max = mx;
        pw::dense::source_kernel<<<num_sms() * 8, 256, 0, s>>>(sa);
        src = Wf;
        mode = T::IN_ROWS;
      } else {
        T::masked_max_kernel<<<std::min(NN, num_sms() * 8), 256, 0, s>>>(N, src, h->M0, mx);
      }
      ax.ncols = (long long)N * NN;
      ax.M0 = h->M0;
      for (int pass = 0; pass < 4; ++pass) {
        ax.L = L[pass];
        ax.in = pass == 0 ? src : pass % 2 == 0 ? Wf : Xf;
        ax.vec = aligned(ax.in, 16) ? 1 : 0;
        ax.out = pass % 2 == 0 ? Xf : Wf;
        ax.scale = pass == 3 ? scale : 1.0f;
        ax.S = pass == 3 ? h->S : nullptr;
        ax.max_in = mx + pass;
        ax.max_out = pass < 3 ? mx + pass + 1 : nullptr;
        ax.stall = pass == 0 ? stall : 0;
        if ((e = launch_axis_tc(ax, pass == 0 ? mode : T::IN_COLS, q + (pass < 2 ? 0 : qb), h->err, s)) != cudaSuccess)
          return cuda_fail(e, "dense contraction");
        if (pass == 1 && ev && (e = cudaEventRecord(ev[1], s)) != cudaSuccess) return cuda_fail(e, "event record");
      }
    }
  } else {
    pw::dense::source_kernel<<<num_sms() * 8, 256, 0, s>>>(sa);
    pw::dense::AxisArgs ax{};
    ax.N = N;
    ax.ncols = (long long)N * NN;
    ax.E = h->F;
    ax.S = h->S;
    const dim3 grid((unsigned)(((ax.ncols + pw::dense::BN - 1) / pw::dense::BN) * ((N + pw::dense::BM - 1) / pw::dense::BM)));
    for (int pass = 0; pass < 4; ++pass) {
      ax.L = L[pass];
      ax.in = pass % 2 == 0 ? Wf : Xf;
      ax.out = pass % 2 == 0 ? Xf : Wf;
      ax.scale = pass == 3 ? scale : 1.0f;
      if (pass < 2)
        pw::dense::axis_kernel<false, false><<<grid, pw::dense::NT, 0, s>>>(ax);
      else if (pass == 2)
        pw::dense::axis_kernel<true, false><<<grid, pw::dense::NT, 0, s>>>(ax);
      else
        pw::dense::axis_kernel<true, true><<<grid, pw::dense::NT, 0, s>>>(ax);
      if (pass == 1 && ev && (e = cudaEventRecord(ev[1], s)) != cudaSuccess) return cuda_fail(e, "event record");
    }
  }
  if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(e, "dense propagation launch");
  if (ev && (e = cudaEventRecord(ev[2], s)) != cudaSuccess) return cuda_fail(e, "event record");
  to_output_plane(h, dx, herm);
  return PW_OK;
}

// N = 256, three streaming passes (t256.cuh): the array with the point-2 DFT over (m, d) into the
// work buffer, the radix-4 over r and the DFT over b in place there, the DFT over a with the output
// factors and S from the work buffer into W.  Uploaded and propagated arrays (Hermitian or not; W0 may be W
// itself, since the first pass writes only the work buffer).  Events: the first pass, then the
// second and third apart.
pw_status propagate_t256(pw_csd* h, double z, bool herm) {
  namespace T = pw::t256;
  pw::PassAArgs a{};
  a.F = h->F;
  a.tw = h->tw;
  a.W0 = reinterpret_cast<const float2*>(h->kind == SRC_PROPAGATED ? h->W : h->W0);
  pw::PassBArgs b{};
  b.tw = h->tw;
  b.Eout = h->Eout;
  b.W = reinterpret_cast<float2*>(h->W);
  b.S = h->S;
  const double lz = h->lambda * z;
  b.scale = (float)((h->d * h->d / lz) * (h->d * h->d / lz));
  static int g2 = 0, g3 = 0;
  cudaError_t e = cudaSuccess;
  if (g2 == 0) {
    if ((e = cudaFuncSetAttribute(T::pass1_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)T::pass1_smem())) != cudaSuccess ||
        (e = cudaFuncSetAttribute(T::pass2_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)T::pass2_smem())) != cudaSuccess ||
        (e = cudaFuncSetAttribute(T::pass3_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)T::pass3_smem())) != cudaSuccess ||
        (e = persistent_grid(T::pass2_kernel, T::NT2, T::pass2_smem(), 1 << 30, &g2)) != cudaSuccess ||
        (e = persistent_grid(T::pass3_kernel, T::NT2, T::pass3_smem(), 1 << 30, &g3)) != cudaSuccess)
      return cuda_fail(e, "set-up of the N = 256 passes");
  }
  cudaEvent_t* ev = nullptr;
  if (!h->events.empty() && (size_t)(4 * (h->timed + 1)) <= h->events.size()) {
    h->three[h->timed] = 1;
    ev = &h->events[4 * h->timed++];
  }
  if (ev && (e = cudaEventRecord(ev[0], h->stream)) != cudaSuccess) return cuda_fail(e, "event record");
  T::pass1_kernel<<<num_sms(), T::NT1, T::pass1_smem(), h->stream>>>(h->y1map, a);  // one CTA per SM
  e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e, "first-pass launch (N = 256)");
  if (ev && (e = cudaEventRecord(ev[1], h->stream)) != cudaSuccess) return cuda_fail(e, "event record");
  T::pass2_kernel<<<g2, T::NT2, T::pass2_smem(), h->stream>>>(h->ymap, h->tw, reinterpret_cast<float2*>(h->work), h->err);
  if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(e, "second-pass launch (N = 256)");
  if (ev && (e = cudaEventRecord(ev[3], h->stream)) != cudaSuccess) return cuda_fail(e, "event record");
  T::pass3_kernel<<<g3, T::NT2, T::pass3_smem(), h->stream>>>(h->y3map, b, h->err);
  if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(e, "third-pass launch (N = 256)");
  if (ev && (e = cudaEventRecord(ev[2], h->stream)) != cudaSuccess) return cuda_fail(e, "event record");
  to_output_plane(h, lz / (h->N * h->d), herm);
  return PW_OK;
}

// GSM sources, plane by plane (plane.cuh).  The work buffer holds the two tables.  Events: the tables
// (at N = 256 with the row pass) as the first pass, the planes (the column pass) as the second.
pw_status propagate_planes(pw_csd* h, double z) {
  cudaEvent_t* ev = next_events(h);
  const double lz = h->lambda * z;
  PlaneArgs q{};
  q.F = h->F;
  q.G = h->G;
  q.tw = h->tw;
  q.Eout = h->Eout;
  q.work = reinterpret_cast<float2*>(h->work);
  q.W = reinterpret_cast<float2*>(h->W);
  q.S = h->S;
  q.A = h->A;
  q.scale = (h->d * h->d / lz) * (h->d * h->d / lz);
  q.tw2 = reinterpret_cast<pw::ff2*>(h->gpart);  // N = 256: in the adjoint's scratch
  cudaError_t e = pwi::dispatch_planes(h->N, h->wmap, q, h->err, h->stream, ev);
  if (e != cudaSuccess) return cuda_fail(e, "propagation kernel launch (GSM source)");
  to_output_plane(h, lz / (h->N * h->d), true);
  return PW_OK;
}

// Aperture as n_i^2 + n_j^2 <= threshold: the integer floor of the table kernel's FP64 threshold (r^2 is an
// integer, the same decision), -1 for none.
int aperture_threshold(const pw_csd* h) {
  if (!(h->aperture > 0.0)) return -1;
  const double rp = h->aperture / h->d, thr = rp * rp;
  return thr >= 2147483647.0 ? 2147483647 : (int)std::floor(thr);
}

// Tables of a sparse source (delta.cuh) into the work buffer: D, and with a row al and be.
cudaError_t delta_tables(pw_csd* h, pw::delta::TabArgs& t) {
  const int N = h->N, G = pw::delta::table_groups(N);
  const size_t NN = (size_t)N * N;
  t.N = N;
  t.F = h->F;
  t.tw = h->tw;
  t.Eout = h->Eout;
  t.D = reinterpret_cast<float2*>(h->work);
  t.al = t.D + NN;
  t.be = t.al + NN;
  pw::delta::tables_kernel<<<dim3(N, t.cross ? 2 : 1), N * G, (size_t)(G + 1) * N * sizeof(float2), h->stream>>>(t, G);
  return cudaGetLastError();
}

cudaError_t delta_write(pw_csd* h, const pw::delta::TabArgs& t, bool cross, bool conj, double kappa, float* S) {
  const int N = h->N, H = N / 2;
  const pw::delta::WriteArgs w{N, t.Eout, t.q, t.D, t.al, t.be, (float)kappa, reinterpret_cast<float2*>(h->W), S};
  const int grid = std::min(N * N, num_sms() * 8), nt = 256 / H * H;
  if (cross && conj) pw::delta::write_kernel<true, true><<<grid, nt, 0, h->stream>>>(w);
  else if (conj) pw::delta::write_kernel<false, true><<<grid, nt, 0, h->stream>>>(w);
  else pw::delta::write_kernel<false, false><<<grid, nt, 0, h->stream>>>(w);
  return cudaGetLastError();
}

// A delta-correlated source: W depends on x1 - x2 but for the output factors (delta.cuh).  Events: the table
// as the first pass, the write as the second.
pw_status propagate_diagonal(pw_csd* h, double z) {
  const double lz = h->lambda * z, s = (h->d * h->d / lz) * (h->d * h->d / lz);
  cudaEvent_t* ev = next_events(h);
  cudaError_t e;
  pw::delta::TabArgs t{};
  t.d = h->diag;
  t.A = (float)h->A;
  if (ev && (e = cudaEventRecord(ev[0], h->stream)) != cudaSuccess) return cuda_fail(e, "event record");
  if ((e = delta_tables(h, t)) != cudaSuccess) return cuda_fail(e, "table launch (delta-correlated source)");
  if (ev && (e = cudaEventRecord(ev[1], h->stream)) != cudaSuccess) return cuda_fail(e, "event record");
  if ((e = delta_write(h, t, false, false, s, h->S)) != cudaSuccess) return cuda_fail(e, "write launch (delta-correlated source)");
  if (ev && (e = cudaEventRecord(ev[2], h->stream)) != cudaSuccess) return cuda_fail(e, "event record");
  to_output_plane(h, lz / (h->N * h->d), true);
  return PW_OK;
}

pw_status propagate(pw_csd* h, double z, bool farfield) {
  if (!h) return fail(PW_EINVAL, "null handle");
  if (!finite_pos(z)) return fail(PW_EINVAL, "propagation distance must be finite and > 0 (got %g)", z);
  if (h->kind == SRC_NONE) return fail(PW_ESTATE, "no source set for the current plane");
  const bool herm = h->kind == SRC_GSM || h->kind == SRC_DIAGONAL || h->hermitian != 0;
  if (h->Nz > 0 || !supported(h->N)) return propagate_dense(h, z, farfield, herm);
  if (h->dft_mode == PW_DFT_TC_BF16X3 && h->kind != SRC_GSM)
    return fail(PW_EUNSUPPORTED, "the tensor-core first stage is built for Gaussian Schell-model sources only");
  pw_status st = build_tables(h, z, farfield);
  if (st != PW_OK) return st;
  // GSM sources: plane by plane, one 2D transform over (a, d) per (b', c') from tables of N^3 values
  // (N = 128: 0.87 against 1.67 ms on the two general passes; N = 96: 0.31 against 0.68; N = 256: 16.3
  // against 31.3 ms; N = 32: 2 us less).  The exception is the tensor-core comparison mode at N = 256.
  const bool tc256 = h->N == 256 && h->dft_mode == PW_DFT_TC_BF16X3;
  if (h->kind == SRC_GSM && !tc256) return propagate_planes(h, z);
  if (h->kind == SRC_DIAGONAL) return propagate_diagonal(h, z);
  // N = 256: the three streaming passes (t256.cuh); the cluster engine (d256.cuh) runs
  // only the comparison mode with the tensor-core first stage
  if (h->N == 256 && !tc256) return propagate_t256(h, z, herm);
  pw::PassAArgs a{};
  a.F = h->F;
  a.G = h->G;
  a.tw = h->tw;
  a.W0 = tc256 ? nullptr : reinterpret_cast<const float2*>(h->kind == SRC_PROPAGATED ? h->W : h->W0);
  a.A = (float)h->A;
  pw::PassBArgs b{};
  b.V = reinterpret_cast<const float2*>(h->work);
  b.tw = h->tw;
  b.Eout = h->Eout;
  b.W = reinterpret_cast<float2*>(h->W);
  b.S = h->S;
  const double lz = h->lambda * z;
  b.scale = (float)((h->d * h->d / lz) * (h->d * h->d / lz));
  R128Extra x{};
  x.Ein = h->Ein;
  x.mask = reinterpret_cast<const float2*>(h->mask);
  x.ap_ithr = aperture_threshold(h);
  x.err = h->err;
  cudaError_t e = dispatch(h->N, herm, h->vmap, a, b, x, h->stream, next_events(h));
  if (e != cudaSuccess) return cuda_fail(e, "propagation kernel launch");
  to_output_plane(h, lz / (h->N * h->d), herm);
  return PW_OK;
}

// S and mu(P1, .) after a propagation of the recorded GSM source, without it (smu.cuh).
pw_status gsm_s_mu(pw_csd* h, double z, bool farfield, int iP, int jP, float* S, pw_c32* mu) {
  if (h->kind != SRC_GSM) return fail(PW_ESTATE, "no Gaussian Schell-model source recorded for the current plane");
  if (h->Nz > 0 || !supported(h->N) || h->N < 4)
    return fail(PW_EUNSUPPORTED, "S and mu alone need an unpadded grid with an FFT plan, N >= 4");
  const int N = h->N;
  const double d = h->d, lam = h->lambda, lz = lam * z, dx = lz / (N * d), base = d * d / (2.0 * lam);
  const double invf = h->lens_f != 0.0 ? 1.0 / h->lens_f : 0.0;
  double2* w = reinterpret_cast<double2*>(h->work);  // 6 N^2 values of scratch, then 5.5 N of tables
  pw::smu::TabArgs<double2> t{};
  t.N = N;
  t.Kin = farfield ? -base * invf : base * (1.0 / z - invf);
  t.Kout = dx * dx / (2.0 * lz);
  t.gs = d * d / (4.0 * h->sigma_S * h->sigma_S);
  t.gm = d * d / (2.0 * h->sigma_mu * h->sigma_mu);
  t.amp = 1.0;
  t.tw = w + (size_t)6 * N * N;
  t.P1 = t.tw + 2 * N;
  t.Eout = t.P1 + N;
  t.k = reinterpret_cast<double*>(t.Eout + N);
  pw::smu::Inst<double2> q{};
  q.N = N;
  q.iP = iP;
  q.jP = jP;
  q.factor = (d * d / lz) * (d * d / lz) * h->A / (4.0 * N * N);
  q.tw = t.tw;
  q.P1 = t.P1;
  q.Eout = t.Eout;
  q.k = t.k;
  q.K = t.k + N;
  q.mask = reinterpret_cast<const float2*>(h->mask);
  q.ap_ithr = aperture_threshold(h);
  q.scratch = w;
  q.S = S;
  q.mu = reinterpret_cast<float2*>(mu);
  const cudaError_t e = pwi::launch_smu_one(t, q, h->stream);
  if (e != cudaSuccess) return cuda_fail(e, "S/mu launch (GSM source)");
  return PW_OK;
}

pw_status s_mu(pw_csd* h, int iP, int jP, float* S, pw_c32* mu) {
  if (h->kind == SRC_NONE) return fail(PW_ESTATE, "no source set for the current plane");
  // A propagated plane without masks needs no tables: S comes from the last pass's epilogue.
  if (h->kind != SRC_PROPAGATED || has_masks(h)) {
    pw_status st = build_tables(h, 0.0, false, true);
    if (st != PW_OK) return st;
  }
  pw::SMuArgs a{};
  a.N = h->N;
  a.mode = h->kind == SRC_GSM ? 0 : (h->kind == SRC_ARRAY ? 1 : (h->kind == SRC_DIAGONAL ? 3 : 2));
  a.diag = h->diag;
  a.G = h->G;
  a.A = (float)h->A;
  a.M0 = has_masks(h) ? h->M0 : nullptr;
  a.Wsrc = reinterpret_cast<const float2*>(h->kind == SRC_ARRAY ? h->W0 : h->W);
  a.Sprop = h->S;
  a.iP = iP;
  a.jP = jP;
  a.S_out = S;
  a.mu_out = reinterpret_cast<float2*>(mu);
  const int NN = h->N * h->N;
  pw::s_mu_kernel<<<(NN + 255) / 256, 256, 0, h->stream>>>(a);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e, "S/mu kernel launch");
  return PW_OK;
}

}  // namespace

namespace pwi {
// 5D map of a work buffer in the V layout, as 32-bit floats: dims (innermost first)
// (2g floats of one d' run, b, a, d'/g, c'); box = one whole slice {2g, 1, 1, N/g, N}
// (N = 256: each CTA of a cluster stores a tile of N / CLUSTER_A columns, d256.cuh).
pw_status encode_vmap(CUtensorMap* map, void* work, int N) {
  const int g = pw::vgroup_of(N);
  auto enc = encode_tiled();
  if (!enc) return fail(PW_ECUDA, "cuTensorMapEncodeTiled is not available from the driver");
  const cuuint64_t run = (cuuint64_t)2 * g * sizeof(float);
  cuuint64_t dims[5] = {(cuuint64_t)2 * g, (cuuint64_t)N, (cuuint64_t)N, (cuuint64_t)(N / g), (cuuint64_t)N};
  cuuint64_t strides[4] = {run, run * N, run * N * N, run * N * N * (N / g)};
  // N = 256 (cluster engine): each CTA stores N / CLUSTER_A columns of the slice; N = 128: each
  // warp stores its eight rows; otherwise the whole slice in one box
  const int cols = N == 256 ? N / pw::d256::CLUSTER_A : N;
  const int rows = N == 128 ? 8 : N;
  cuuint32_t box[5] = {(cuuint32_t)(2 * g), 1, 1, (cuuint32_t)(cols / g), (cuuint32_t)rows};
  cuuint32_t estr[5] = {1, 1, 1, 1, 1};
  CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 5, work, dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return fail(PW_ECUDA, "cuTensorMapEncodeTiled failed (CUresult %d)", (int)r);
  return PW_OK;
}

// 5D map of W for the plane kernels: a plane (b', c') is the N rows W(a', b', c', .), left whole (N <= 96); at
// N = 256 the column pass's tiles, 64 floats of every a.  (N = 64 and 128 need none.)
pw_status encode_wmap(CUtensorMap* map, void* W, int N) {
  if (N <= pw::small::MAX_N || N == 64 || N == 128) return PW_OK;
  auto enc = encode_tiled();
  if (!enc) return fail(PW_ECUDA, "cuTensorMapEncodeTiled is not available from the driver");
  const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
  if (N == 256) {
    const cuuint64_t dims[5] = {64, 256 * 256 * 8, 256, 1, 1};
    const cuuint64_t strides[4] = {256, (cuuint64_t)256 * 256 * 256 * 8, (cuuint64_t)1 << 35, (cuuint64_t)1 << 35};
    const cuuint32_t box[5] = {64, 1, 256, 1, 1};
    CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 5, W, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                     CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(PW_ECUDA, "cuTensorMapEncodeTiled (column tiles of W) failed (CUresult %d)", (int)r);
    return PW_OK;
  }
  const cuuint64_t n = N, row = 2 * n * sizeof(float);
  const cuuint64_t dims[5] = {2 * n, n, n, n, 1};
  const cuuint64_t strides[4] = {row, row * n, row * n * n, row * n * n * n};
  const cuuint32_t box[5] = {(cuuint32_t)(2 * N), 1, 1, (cuuint32_t)N, 1};
  CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 5, W, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                   CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return fail(PW_ECUDA, "cuTensorMapEncodeTiled (planes of W) failed (CUresult %d)", (int)r);
  return PW_OK;
}

}  // namespace pwi

extern "C" {

const char* pw_last_error(void) { return g_err.c_str(); }

const char* pw_status_string(pw_status s) {
  switch (s) {
    case PW_OK: return "PW_OK";
    case PW_EINVAL: return "PW_EINVAL";
    case PW_ESIZE: return "PW_ESIZE";
    case PW_ECUDA: return "PW_ECUDA";
    case PW_ETIMEOUT: return "PW_ETIMEOUT";
    case PW_ESTATE: return "PW_ESTATE";
    case PW_EUNSUPPORTED: return "PW_EUNSUPPORTED";
  }
  return "PW_UNKNOWN";
}

int pw_supported_n(int N) { return supported(N) ? 1 : 0; }

size_t pw_csda_bytes(int N) {
  if (N <= 0) return 0;
  const size_t n = (size_t)N;
  return n * n * n * n * sizeof(pw_c32);
}

pw_status pw_csd_create(pw_csd** out, int N, double dxi_m, double lambda_m, pw_c32* dev_W,
                        size_t W_bytes, pw_c32* dev_work, size_t work_bytes, void* stream) {
  g_err.clear();
  if (!out) return fail(PW_EINVAL, "out is null");
  *out = nullptr;
  if (N < 2 || (N & 1)) return fail(PW_EINVAL, "N must be even and >= 2 (got %d)", N);
  if (!finite_pos(dxi_m)) return fail(PW_EINVAL, "sampling must be finite and > 0 (got %g)", dxi_m);
  if (!finite_pos(lambda_m)) return fail(PW_EINVAL, "wavelength must be finite and > 0 (got %g)", lambda_m);
  if (N > PW_MAX_N) return fail(PW_EUNSUPPORTED, "no propagation plan for N = %d (at most %d)", N, PW_MAX_N);
  if (!dev_W || !dev_work) return fail(PW_EINVAL, "dev_W and dev_work must be non-null");
  const size_t need = pw_csda_bytes(N);
  if (W_bytes < need || work_bytes < need)
    return fail(PW_ESIZE, "buffers need %zu bytes each (got W %zu, work %zu)", need, W_bytes, work_bytes);
  {
    const char* a0 = reinterpret_cast<const char*>(dev_W);
    const char* b0 = reinterpret_cast<const char*>(dev_work);
    if (a0 < b0 + need && b0 < a0 + need) return fail(PW_EINVAL, "dev_W and dev_work overlap");
  }
  if (!aligned(dev_W, 16) || !aligned(dev_work, 16)) return fail(PW_EINVAL, "dev_W and dev_work must be 16-byte aligned");
  pw_csd* h = new pw_csd{};
  h->N = N;
  h->d = dxi_m;
  h->lambda = lambda_m;
  h->W = dev_W;
  h->work = dev_work;
  h->stream = reinterpret_cast<cudaStream_t>(stream);
  h->kind = SRC_NONE;
  h->A = 1.0;
  cudaError_t e = cudaMalloc(&h->tables, table_bytes(N));
  if (e != cudaSuccess) {
    delete h;
    return cuda_fail(e, "cudaMalloc of the handle tables");
  }
  const size_t NN = (size_t)N * N;
  char* p = reinterpret_cast<char*>(h->tables);
  h->F = reinterpret_cast<float2*>(p);
  p += NN * sizeof(float2);
  h->M0 = reinterpret_cast<float2*>(p);
  p += NN * sizeof(float2);
  h->G = reinterpret_cast<float*>(p);
  p += NN * sizeof(float);
  h->S = reinterpret_cast<float*>(p);
  p += NN * sizeof(float);
  h->tw = reinterpret_cast<float2*>(p);
  p += N * sizeof(float2);
  h->Eout = reinterpret_cast<float2*>(p);
  p += N * sizeof(float2);
  h->Ein = reinterpret_cast<float2*>(p);
  p += N * sizeof(float2);
  h->err = reinterpret_cast<int*>(p);
  h->maxes = reinterpret_cast<unsigned*>(p + 64);
  p += 256;
  auto carve = [&](size_t bytes) {
    char* q = p;
    p += (bytes + 255) / 256 * 256;
    return q;
  };
  h->adj_d = reinterpret_cast<float*>(carve(NN * sizeof(float)));
  h->adj_c = reinterpret_cast<float2*>(carve(NN * sizeof(float2)));
  h->gpart = reinterpret_cast<double*>(carve(NN * 3 * sizeof(double)));
  h->gtab = reinterpret_cast<float*>(carve(NN * sizeof(float)));
  h->qtab = reinterpret_cast<float2*>(carve((size_t)N * sizeof(float2)));
  h->g3tmp = reinterpret_cast<double*>(carve(3 * sizeof(double)));
  e = cudaMemsetAsync(h->err, 0, sizeof(int), h->stream);
  if (e != cudaSuccess) {
    cudaFree(h->tables);
    delete h;
    return cuda_fail(e, "clearing the error flag");
  }
  pw_status st = supported(N) ? make_vmap(h) : PW_OK;  // the dense path needs no tensor map
  if (st != PW_OK) {
    cudaFree(h->tables);
    delete h;
    return st;
  }
  *out = h;
  return PW_OK;
}

static void free_events(pw_csd* h) {
  for (cudaEvent_t e : h->events) cudaEventDestroy(e);
  h->events.clear();
  h->three.clear();
  h->timed = 0;
}

pw_status pw_csd_destroy(pw_csd* h) {
  g_err.clear();
  if (!h) return PW_OK;
  cudaError_t e1 = cudaStreamSynchronize(h->stream);
  free_events(h);
  cudaError_t e2 = cudaFree(h->tables);
  if (h->qbuf) cudaFree(h->qbuf);
  delete h;
  if (e1 != cudaSuccess) return cuda_fail(e1, "stream synchronize in destroy");
  if (e2 != cudaSuccess) return cuda_fail(e2, "cudaFree of the handle tables");
  return PW_OK;
}

pw_status pw_csd_set_stream(pw_csd* h, void* stream) {
  g_err.clear();
  if (!h) return fail(PW_EINVAL, "null handle");
  h->stream = reinterpret_cast<cudaStream_t>(stream);
  return PW_OK;
}

pw_status pw_csd_reset(pw_csd* h, double dxi_m) {
  g_err.clear();
  if (!h) return fail(PW_EINVAL, "null handle");
  if (!finite_pos(dxi_m)) return fail(PW_EINVAL, "sampling must be finite and > 0 (got %g)", dxi_m);
  h->d = dxi_m;
  h->kind = SRC_NONE;
  h->W0 = nullptr;
  h->A = 1.0;
  h->aperture = 0.0;
  h->lens_f = 0.0;
  h->mask = nullptr;
  return PW_OK;
}

pw_status pw_csd_check(pw_csd* h) {
  g_err.clear();
  if (!h) return fail(PW_EINVAL, "null handle");
  int flag = 0;
  cudaError_t e = cudaMemcpyAsync(&flag, h->err, sizeof(int), cudaMemcpyDeviceToHost, h->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
  if (e != cudaSuccess) return cuda_fail(e, "reading the error flag");
  if (flag) {
    e = cudaMemsetAsync(h->err, 0, sizeof(int), h->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    if (e != cudaSuccess) return cuda_fail(e, "clearing the error flag");
    return fail(PW_ETIMEOUT, "a bounded device-side wait gave up; the last result is invalid");
  }
  return PW_OK;
}

pw_status pw_csd_enable_timing(pw_csd* h, int max_props) {
  g_err.clear();
  if (!h) return fail(PW_EINVAL, "null handle");
  if (max_props < 0) return fail(PW_EINVAL, "max_props must be >= 0");
  free_events(h);
  h->events.resize((size_t)4 * max_props);
  h->three.assign((size_t)max_props, 0);
  for (size_t i = 0; i < h->events.size(); ++i) {
    cudaError_t e = cudaEventCreate(&h->events[i]);
    if (e != cudaSuccess) {
      h->events.resize(i);
      free_events(h);
      return cuda_fail(e, "cudaEventCreate");
    }
  }
  return PW_OK;
}

pw_status pw_csd_pass_times3(pw_csd* h, double* ms_first, double* ms_second, double* ms_third, int* count) {
  g_err.clear();
  if (!h || !ms_first || !ms_second || !ms_third || !count) return fail(PW_EINVAL, "null argument");
  double sa = 0.0, sb = 0.0, sc = 0.0;
  for (int k = 0; k < h->timed; ++k) {
    cudaEvent_t* ev = &h->events[4 * k];
    float t1 = 0.f, t2 = 0.f, t3 = 0.f;
    cudaError_t e = cudaEventSynchronize(ev[2]);
    if (e == cudaSuccess) e = cudaEventElapsedTime(&t1, ev[0], ev[1]);
    if (e == cudaSuccess) {
      if (h->three[k]) {
        e = cudaEventElapsedTime(&t2, ev[1], ev[3]);
        if (e == cudaSuccess) e = cudaEventElapsedTime(&t3, ev[3], ev[2]);
      } else {
        e = cudaEventElapsedTime(&t2, ev[1], ev[2]);
      }
    }
    if (e != cudaSuccess) return cuda_fail(e, "pass timing events");
    sa += t1;
    sb += t2;
    sc += t3;
  }
  *ms_first = sa;
  *ms_second = sb;
  *ms_third = sc;
  *count = h->timed;
  h->timed = 0;
  return PW_OK;
}

pw_status pw_csd_pass_times(pw_csd* h, double* ms_first, double* ms_second, int* count) {
  double m3 = 0.0;
  pw_status st = pw_csd_pass_times3(h, ms_first, ms_second, &m3, count);
  if (st == PW_OK) *ms_second += m3;
  return st;
}

pw_status pw_csd_set_padding(pw_csd* h, int Nz) {
  g_err.clear();
  if (!h) return fail(PW_EINVAL, "null handle");
  if (Nz != 0 && (Nz < h->N || (Nz - h->N) % 2 != 0 || Nz > (1 << 20)))
    return fail(PW_EINVAL, "padded size must be 0 or N <= Nz <= 2^20 with Nz - N even (N = %d, Nz = %d)", h->N, Nz);
  h->Nz = Nz == h->N ? 0 : Nz;
  return PW_OK;
}

pw_status pw_csd_get_padding(const pw_csd* h, int* Nz) {
  g_err.clear();
  if (!h || !Nz) return fail(PW_EINVAL, "null argument");
  *Nz = h->Nz > 0 ? h->Nz : h->N;
  return PW_OK;
}

pw_status pw_csd_inject_stall(pw_csd* h, int chunk) {
  g_err.clear();
  if (!h) return fail(PW_EINVAL, "null handle");
  h->stall = chunk;
  return PW_OK;
}

pw_status pw_csd_set_dft_mode(pw_csd* h, int mode) {
  g_err.clear();
  if (!h) return fail(PW_EINVAL, "null handle");
  if (mode != PW_DFT_AUTO && mode != PW_DFT_FP32 && mode != PW_DFT_TC_BF16X3)
    return fail(PW_EINVAL, "unknown DFT mode %d", mode);
  if (mode == PW_DFT_TC_BF16X3 && h->N > pw::dense_tc::MAX_N)
    return fail(PW_EUNSUPPORTED, "the tensor-core paths exist for N <= %d (N = %d)", pw::dense_tc::MAX_N, h->N);
  h->dft_mode = mode;
  return PW_OK;
}

pw_status pw_csd_get_dft_mode(const pw_csd* h, int* mode) {
  g_err.clear();
  if (!h || !mode) return fail(PW_EINVAL, "null argument");
  *mode = h->dft_mode;
  return PW_OK;
}

pw_status pw_source_gsm(pw_csd* h, double sigma_S_m, double sigma_mu_m, double amplitude) {
  g_err.clear();
  if (!h) return fail(PW_EINVAL, "null handle");
  if (!finite_pos(sigma_S_m) || !finite_pos(sigma_mu_m))
    return fail(PW_EINVAL, "sigma_S and sigma_mu must be finite and > 0 (got %g, %g)", sigma_S_m, sigma_mu_m);
  if (!std::isfinite(amplitude)) return fail(PW_EINVAL, "amplitude must be finite");
  h->kind = SRC_GSM;
  h->sigma_S = sigma_S_m;
  h->sigma_mu = sigma_mu_m;
  h->A = amplitude;
  h->W0 = nullptr;
  return PW_OK;
}

pw_status pw_source_aperture(pw_csd* h, double radius_m) {
  g_err.clear();
  if (!h) return fail(PW_EINVAL, "null handle");
  if (!std::isfinite(radius_m)) return fail(PW_EINVAL, "aperture radius must be finite");
  h->aperture = radius_m > 0.0 ? radius_m : 0.0;
  return PW_OK;
}

pw_status pw_source_lens(pw_csd* h, double focal_m) {
  g_err.clear();
  if (!h) return fail(PW_EINVAL, "null handle");
  if (!std::isfinite(focal_m)) return fail(PW_EINVAL, "focal length must be finite");
  h->lens_f = focal_m;
  return PW_OK;
}

pw_status pw_source_mask(pw_csd* h, const pw_c32* dev_mask) {
  g_err.clear();
  if (!h) return fail(PW_EINVAL, "null handle");
  if (dev_mask && !aligned(dev_mask, 8)) return fail(PW_EINVAL, "dev_mask must be 8-byte aligned");
  h->mask = dev_mask;
  return PW_OK;
}

pw_status pw_source_array(pw_csd* h, const pw_c32* dev_W0, int hermitian) {
  g_err.clear();
  if (!h) return fail(PW_EINVAL, "null handle");
  if (!dev_W0) return fail(PW_EINVAL, "dev_W0 is null");
  if (!aligned(dev_W0, 8)) return fail(PW_EINVAL, "dev_W0 must be 8-byte aligned");
  {
    const size_t need = pw_csda_bytes(h->N);
    const char* a0 = reinterpret_cast<const char*>(dev_W0);
    const char* b0 = reinterpret_cast<const char*>(h->work);
    if (a0 < b0 + need && b0 < a0 + need) return fail(PW_EINVAL, "dev_W0 overlaps the work buffer");
  }
  h->kind = SRC_ARRAY;
  h->W0 = dev_W0;
  h->hermitian = hermitian ? 1 : 0;
  h->A = 1.0;
  return PW_OK;
}

pw_status pw_source_diagonal(pw_csd* h, const float* dev_d, double weight) {
  g_err.clear();
  if (!h) return fail(PW_EINVAL, "null handle");
  if (!dev_d) return fail(PW_EINVAL, "dev_d is null");
  if (!aligned(dev_d, 4)) return fail(PW_EINVAL, "dev_d must be 4-byte aligned");
  if (!std::isfinite(weight)) return fail(PW_EINVAL, "weight must be finite");
  h->kind = SRC_DIAGONAL;
  h->diag = dev_d;
  h->W0 = nullptr;
  h->A = weight;
  return PW_OK;
}

pw_status pw_gsm_gradient(pw_csd* h, double sigma_S_m, double sigma_mu_m, double amplitude, const float* dev_amask,
                          double lambda_m, double z_m, int farfield, double* dev_grad3, float* dev_grad_mask) {
  g_err.clear();
  if (!h || !dev_grad3) return fail(PW_EINVAL, "null argument");
  if (!finite_pos(sigma_S_m) || !finite_pos(sigma_mu_m) || !finite_pos(lambda_m) || !finite_pos(z_m))
    return fail(PW_EINVAL, "lengths must be finite and > 0");
  if (!std::isfinite(amplitude)) return fail(PW_EINVAL, "amplitude must be finite");
  if (h->kind != SRC_PROPAGATED) return fail(PW_ESTATE, "no propagated CSDA (run the adjoint propagation first)");
  if (h->Nz > 0 || !supported(h->N))
    return fail(PW_EUNSUPPORTED, "the GSM gradient needs an unpadded grid with an FFT plan");
  const int N = h->N;
  const double d = h->d;                    // the source plane of the forward propagation
  const double dx = lambda_m * z_m / (N * d);  // its output plane
  pw::GradArgs g{};
  g.N = N;
  g.d = d;
  g.sigma_S = sigma_S_m;
  g.sigma_mu = sigma_mu_m;
  g.A = amplitude;
  g.amask = dev_amask;
  g.R = reinterpret_cast<const float2*>(h->W);
  g.c = std::pow(d / dx, 4);
  g.farfield = farfield ? 1 : 0;
  g.Kq = d * d / (2.0 * lambda_m * z_m);
  g.g3 = dev_grad3;
  g.gmask = dev_grad_mask;
  // the work buffer is scratch between propagations: partial sums, then the FP64-built tables
  g.part = reinterpret_cast<double*>(h->work);
  g.rows = N * N;
  g.gtab = reinterpret_cast<float*>(g.part + (size_t)N * N * 3);
  g.qtab = reinterpret_cast<float2*>(g.gtab + (size_t)N * N + (N & 1));
  pw::gsm_gradient_tables<<<(N * N + 255) / 256, 256, 0, h->stream>>>(g);
  cudaError_t e0 = cudaGetLastError();
  if (e0 != cudaSuccess) return cuda_fail(e0, "gradient table launch");
  const size_t sh = 2 * N * sizeof(float) + 2 * N * sizeof(float2) + 32 * sizeof(double) + 64;
  if (g.farfield) pw::gsm_gradient_kernel<true><<<N * N, 256, sh, h->stream>>>(g);
  else pw::gsm_gradient_kernel<false><<<N * N, 256, sh, h->stream>>>(g);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e, "gradient kernel launch");
  pw::gsm_gradient_reduce<<<1, 256, 0, h->stream>>>(g);
  e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e, "gradient reduction launch");
  return PW_OK;
}

}  // extern "C"

namespace {

// The adjoint of one propagation (Fresnel or far field over z) for a loss on S and mu of its
// output plane; the handle's current plane is that output plane.  See pw_propagate_fresnel_adjoint.
pw_status adjoint(pw_csd* h, double z, bool farfield, const pw_adjoint* a) {
  if (!h || !a) return fail(PW_EINVAL, "null argument");
  if (!finite_pos(z)) return fail(PW_EINVAL, "propagation distance must be finite and > 0 (got %g)", z);
  if (h->Nz > 0 || !supported(h->N))
    return fail(PW_EUNSUPPORTED, "the adjoint propagation needs an unpadded grid with an FFT plan");
  const int N = h->N;
  const bool has_mu = a->dev_dmu != nullptr;
  if (!a->dev_dS && !has_mu) return fail(PW_EINVAL, "no upstream gradient (dev_dS and dev_dmu are both null)");
  if (has_mu) {
    if (!a->dev_S || !a->dev_mu) return fail(PW_EINVAL, "dev_dmu needs the output plane's dev_S and dev_mu");
    if (a->iP < 0 || a->jP < 0 || a->iP >= N || a->jP >= N)
      return fail(PW_EINVAL, "P1 = (%d, %d) outside the %d x %d grid", a->iP, a->jP, N, N);
  }
  const bool params = a->dev_grad3 != nullptr || a->dev_grad_amask != nullptr;
  if (!params && !a->grad_W0) return fail(PW_EINVAL, "no gradient requested");
  if (params && (!finite_pos(a->sigma_S_m) || !finite_pos(a->sigma_mu_m) || !std::isfinite(a->amplitude)))
    return fail(PW_EINVAL, "the GSM parameters must be finite (sigma_S, sigma_mu > 0)");
  if ((a->dev_dS && !aligned(a->dev_dS, 4)) || (a->dev_S && !aligned(a->dev_S, 4)) ||
      (a->dev_amask && !aligned(a->dev_amask, 4)) || (a->dev_grad_amask && !aligned(a->dev_grad_amask, 4)) ||
      (a->dev_dmu && !aligned(a->dev_dmu, 8)) || (a->dev_mu && !aligned(a->dev_mu, 8)) ||
      (a->dev_grad3 && !aligned(a->dev_grad3, 8)))
    return fail(PW_EINVAL, "misaligned device pointer");
  const double dx = h->d, lam = h->lambda, d = lam * z / (N * dx);
  const double c = std::pow(d / dx, 4);
  cudaStream_t st = h->stream;

  // the handle ends at the source plane, with no source recorded
  auto done = [&](pw_status r) {
    h->d = d;
    h->kind = SRC_NONE;
    h->W0 = nullptr;
    h->diag = nullptr;
    h->aperture = 0.0;
    h->lens_f = 0.0;
    h->mask = nullptr;
    return r;
  };
  if (h->dft_mode == PW_DFT_TC_BF16X3)
    return done(fail(PW_EUNSUPPORTED, "the tensor-core first stage is built for Gaussian Schell-model sources only"));

  // the (conjugated) adjoint source on the output plane
  const int NN = N * N, nprep = (NN + 1023) / 1024;
  pw::AdjPrepArgs pa{};
  pa.N = N;
  pa.iP = a->iP;
  pa.jP = a->jP;
  pa.gS = a->dev_dS;
  pa.gmu = reinterpret_cast<const float2*>(a->dev_dmu);
  pa.S = a->dev_S;
  pa.mu = reinterpret_cast<const float2*>(a->dev_mu);
  pa.d = h->adj_d;
  pa.cross = h->adj_c;
  pa.part = h->gpart;
  pw::adjoint_prep_kernel<<<nprep, 1024, 0, st>>>(pa);
  // the GSM factor (parameter gradients) and the far-field factors of the source grid
  pw::GradArgs g{};
  g.N = N;
  g.d = d;
  g.sigma_S = params ? a->sigma_S_m : 0.0;
  g.sigma_mu = params ? a->sigma_mu_m : 0.0;
  g.A = a->amplitude;
  g.c = c;
  g.Kq = d * d / (2.0 * lam * z);
  g.part = h->gpart;
  g.gtab = h->gtab;
  g.qtab = h->qtab;
  g.g3 = a->dev_grad3 ? a->dev_grad3 : h->g3tmp;
  if (params || farfield) pw::gsm_gradient_tables<<<(NN + 255) / 256, 256, 0, st>>>(g);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return done(cuda_fail(e, "adjoint set-up launch"));

  // the adjoint propagation is a Fresnel propagation over z from the output sampling dx of the
  // conjugated source, back onto the source grid d, in closed form (delta.cuh)
  h->d = dx;
  h->kind = SRC_DIAGONAL;  // no GSM table
  pw_status r = build_tables(h, z, false);
  if (r != PW_OK) return done(r);
  const double lz = lam * z, s = (dx * dx / lz) * (dx * dx / lz);
  cudaEvent_t* ev = next_events(h);
  if (ev && (e = cudaEventRecord(ev[0], st)) != cudaSuccess) return done(cuda_fail(e, "event record"));
  pw::delta::TabArgs t{};
  t.d = h->adj_d;
  t.A = 1.0f;
  t.q = farfield ? h->qtab : nullptr;
  t.cross = has_mu ? h->adj_c : nullptr;
  t.iP = a->iP;
  t.jP = a->jP;
  t.part = has_mu ? h->gpart : nullptr;
  t.npart = nprep;
  t.S = a->dev_S;
  if ((e = delta_tables(h, t)) != cudaSuccess) return done(cuda_fail(e, "adjoint table launch"));
  if (ev && (e = cudaEventRecord(ev[1], st)) != cudaSuccess) return done(cuda_fail(e, "event record"));
  if (params) {
    // the Hermitian part of the source suffices: dW0/dtheta is Hermitian
    const int rows = std::max(1, 256 / N), nt = (rows * N + 31) / 32 * 32;
    const pw::delta::GradArgs ga{N, h->Eout, t.q, t.D, t.al, t.be, h->gtab, a->dev_amask, (float)s, (float)(d * d),
                                 h->gpart, a->dev_grad_amask, (float)(4.0 * c * a->amplitude)};
    const int nc = N % 4 == 0 ? 4 : 2;  // columns a block takes together
    const size_t sh = N * sizeof(float2);
    auto grad = [&](auto k) -> cudaError_t {  // one wave of resident blocks
      int& rows_of_k = h->grad_rows[has_mu];
      const cudaError_t r = rows_of_k ? cudaSuccess : persistent_grid(k, nt, sh, NN / nc, &rows_of_k);
      g.rows = rows_of_k;
      if (r == cudaSuccess) k<<<g.rows, nt, sh, st>>>(ga);
      return r;
    };
    if (nc == 4) e = has_mu ? grad(pw::delta::grad_kernel<true, 4>) : grad(pw::delta::grad_kernel<false, 4>);
    else e = has_mu ? grad(pw::delta::grad_kernel<true, 2>) : grad(pw::delta::grad_kernel<false, 2>);
    if (e != cudaSuccess) return done(cuda_fail(e, "gradient launch"));
    pw::gsm_gradient_reduce<<<1, 256, 0, st>>>(g);
    if ((e = cudaGetLastError()) != cudaSuccess) return done(cuda_fail(e, "gradient launch"));
  }
  // a general complex W0: the whole adjoint (the P1 row without its mirrored column), as
  // dL/dRe W0 + i dL/dIm W0 = 2 c conj(R)
  if (a->grad_W0 && (e = delta_write(h, t, has_mu, true, 2.0 * c * s, nullptr)) != cudaSuccess)
    return done(cuda_fail(e, "gradient write launch"));
  if (ev && (e = cudaEventRecord(ev[2], st)) != cudaSuccess) return done(cuda_fail(e, "event record"));
  return done(PW_OK);
}

}  // namespace

extern "C" {

pw_status pw_propagate_fresnel_adjoint(pw_csd* h, double z_m, const pw_adjoint* a) {
  g_err.clear();
  return adjoint(h, z_m, false, a);
}

pw_status pw_propagate_farfield_adjoint(pw_csd* h, double z_m, const pw_adjoint* a) {
  g_err.clear();
  return adjoint(h, z_m, true, a);
}

pw_status pw_gsm_s_mu(pw_csd* h, double z_m, int farfield, int iP, int jP, float* dev_S, pw_c32* dev_mu) {
  g_err.clear();
  if (!h || !dev_S) return fail(PW_EINVAL, "null argument");
  if (!finite_pos(z_m)) return fail(PW_EINVAL, "propagation distance must be finite and > 0 (got %g)", z_m);
  if (!aligned(dev_S, 4)) return fail(PW_EINVAL, "dev_S must be 4-byte aligned");
  if (dev_mu && !aligned(dev_mu, 8)) return fail(PW_EINVAL, "dev_mu must be 8-byte aligned");
  if (iP < 0 || jP < 0 || iP >= h->N || jP >= h->N)
    return fail(PW_EINVAL, "P1 = (%d, %d) outside the %d x %d grid", iP, jP, h->N, h->N);
  return gsm_s_mu(h, z_m, farfield != 0, iP, jP, dev_S, dev_mu);
}

pw_status pw_propagate_fresnel(pw_csd* h, double z_m) {
  g_err.clear();
  return propagate(h, z_m, false);
}

pw_status pw_propagate_farfield(pw_csd* h, double z_m) {
  g_err.clear();
  return propagate(h, z_m, true);
}

pw_status pw_get_sampling(const pw_csd* h, double* d_m) {
  g_err.clear();
  if (!h || !d_m) return fail(PW_EINVAL, "null argument");
  *d_m = h->d;
  return PW_OK;
}

pw_status pw_spectral_density(pw_csd* h, float* dev_S) {
  g_err.clear();
  if (!h || !dev_S) return fail(PW_EINVAL, "null argument");
  if (!aligned(dev_S, 4)) return fail(PW_EINVAL, "dev_S must be 4-byte aligned");
  return s_mu(h, 0, 0, dev_S, nullptr);
}

pw_status pw_degree_of_coherence(pw_csd* h, int iP, int jP, pw_c32* dev_mu) {
  g_err.clear();
  if (!h || !dev_mu) return fail(PW_EINVAL, "null argument");
  if (!aligned(dev_mu, 8)) return fail(PW_EINVAL, "dev_mu must be 8-byte aligned");
  if (iP < 0 || jP < 0 || iP >= h->N || jP >= h->N)
    return fail(PW_EINVAL, "P1 = (%d, %d) outside the %d x %d grid", iP, jP, h->N, h->N);
  return s_mu(h, iP, jP, nullptr, dev_mu);
}

}  // extern "C"
