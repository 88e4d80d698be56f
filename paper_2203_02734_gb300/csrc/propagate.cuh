// propagate.cuh -- the two fused passes of one propagation, the FP64 table kernel and the
// S / mu kernel.
//
// With index centring (x(i) = (i - N/2) d, and the same for the flipped second axis), the
// discretised Eq. W_fresnel factorises exactly as
//   W_B(a',b',c',d') = s conj(E(a') E(b')) E(c') E(d')
//                        sum_{a,b} e^{+2 pi i (a a' + b b')/N}  sum_{c,d} e^{-2 pi i (c c' + d d')/N}
//                        conj(F(a,b)) F(c,d) W0core(a,b,c,d)
// where F(i,j) = (-1)^(i+j) exp(2 pi i (tau_i + tau_j)) Y(i,j) m(i,j) folds the input
// propagator q(xi) (Algorithm 3), a thin lens q*(f, xi), the aperture Y and a mask m, and
// E(i) = (-1)^i exp(2 pi i tau'_i) is the output propagator on the new grid; the
// checkerboards carry the centring and s = d^4/(lambda z)^2.  (a,b) is point 1, (c,d) point 2.
//
// Pass A (one CTA per point-1 pair (a,b), contiguous slice): generate conj(F(a,b)) F(c,d)
//   A G(a,c) G(b,d) (GSM) or read the uploaded W0 slice, run the direct 2D DFT over (c,d)
//   in shared memory, store the slice of V once.
// Pass B (one CTA per point-2 output pair (c',d'), strided slice): gather V(., ., c', d'),
//   run the inverse-sign 2D DFT over (a,b), apply s and the output propagators, write S on
//   the diagonal and store.  Because a CSD is Hermitian (Sec. 3.3), the column
//   W_B(., ., c', d') is stored conjugated as the contiguous row W_B(c', d', ., .); the
//   general (non-Hermitian) variant stores the column in place.
//
// Layout of V (the corner turn between the passes): V[c'][d'/g][a][b][d' mod g], g = vgroup_of(N).
// Pass A writes each (c', d'/g) run of g outputs as one piece (a 32-byte sector for g = 4); the g
// columns of one group sit in one contiguous N^2 g-element block, and consecutive (a, b) of one
// column are g elements apart.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "cluster.cuh"
#include "fft.cuh"

namespace pw {

__device__ __forceinline__ double frac_turns(double t) { return t - rint(t); }

// exp(2 pi i t) from turns t, reduced to [-1/2, 1/2] in FP64 before sincospi.
__device__ __forceinline__ float2 cis_turns(double t) {
  double s, c;
  sincospi(2.0 * frac_turns(t), &s, &c);
  return make_float2((float)c, (float)s);
}

struct TableArgs {
  int N;
  double Kin;     // turns per n^2 of the point-2 input factor (propagator and lens)
  double K0;      // turns per n^2 of the lens alone (source-plane view, no propagator)
  double Kout;    // turns per n^2 of the output propagator
  double gs, gm;  // GSM: d^2/(4 sigma_S^2) and d^2/(2 sigma_mu^2)
  double ap_thr;  // aperture: n_i^2 + n_j^2 <= ap_thr (pixels^2), < 0 = none
  const float2* mask;  // user mask (N x N) or nullptr
  float2* F;      // N x N input factor
  float2* M0;     // N x N source-plane mask Y * lens * m (or nullptr)
  float* G;       // N x N GSM axis factor (or nullptr)
  float2* tw;     // N twiddles exp(-2 pi i m / N)
  float2* Eout;   // N output factors
  float2* Ein;    // N per-axis input factors (-1)^i exp(2 pi i Kin n_i^2), or nullptr
};

// One FP64 sincospi or exp per thread (blockIdx.y: 0 F, 1 the per-axis tables, 2 G, 3 M0), in small blocks
// spread over the SMs: an SM issues about two FP64 FMAs a cycle, so a block of 256 threads that evaluated
// five of them each took 10 to 14 us at any N up to 128.
constexpr int TABLE_NT = 64;
inline dim3 tables_grid(const TableArgs& t) {
  return dim3((t.N * t.N + TABLE_NT - 1) / TABLE_NT, t.M0 ? 4 : t.G ? 3 : 2);
}
static __global__ void __launch_bounds__(TABLE_NT) tables_kernel(TableArgs t) {
  const int N = t.N, M = N / 2, NN = N * N, role = blockIdx.y;
  const int idx = blockIdx.x * TABLE_NT + threadIdx.x;
  if (role == 1) {
    for (int q = idx; q < 3 * N; q += gridDim.x * TABLE_NT) {
      const int kind = q / N, i = q - kind * N;
      const double n = (double)(i - M), odd = 0.5 * (i & 1);
      if (kind == 0) t.tw[i] = cis_turns(-(double)i / (double)N);
      else if (kind == 1) t.Eout[i] = cis_turns(frac_turns(n * n * t.Kout) + odd);
      else if (t.Ein) t.Ein[i] = cis_turns(frac_turns(n * n * t.Kin) + odd);
    }
    return;
  }
  if (idx >= NN) return;
  const int i = idx / N, j = idx - i * N;
  const double ni = (double)(i - M), nj = (double)(j - M);
  const double n2i = ni * ni, n2j = nj * nj;
  if (role == 2) {
    if (!t.G) return;
    const double dij = (double)(i - j);
    t.G[idx] = (float)exp(-(n2i + n2j) * t.gs - dij * dij * t.gm);
    return;
  }
  const bool inside = t.ap_thr < 0.0 || (n2i + n2j) <= t.ap_thr;
  float2 m = t.mask ? t.mask[idx] : make_float2(1.f, 0.f);
  if (!inside) m = make_float2(0.f, 0.f);
  if (role == 0) t.F[idx] = cmul(cis_turns(frac_turns(n2i * t.Kin) + frac_turns(n2j * t.Kin) + 0.5 * ((i + j) & 1)), m);
  else t.M0[idx] = cmul(cis_turns(frac_turns(n2i * t.K0) + frac_turns(n2j * t.K0)), m);
}

// Sources: the GSM model, an uploaded CSDA, and (dense path) a diagonal source.
enum SrcMode { SRC_GSM = 0, SRC_ARRAY = 1, SRC_DIAG = 2 };

struct PassAArgs {
  const float2* F;
  const float* G;
  const float2* tw;
  const float2* W0;   // uploaded source (SRC_ARRAY) or nullptr
  float A;            // GSM amplitude
};

template <int N> __host__ __device__ constexpr int pitch() { return N + 1; }
// Width g of the d' runs of the V layout: 4 (one 32-byte sector per run; 2 when 4 does not
// divide N).  Narrower 16-byte runs halve pass B's gather traffic but make pass A's TMA store
// issue twice as many half-sector writes, which costs more than it saves (measured at N = 128).
// g = 4 makes each run one 32-byte sector.  N = 256 uses g = 8: its pass A leaves each 128 KB
// output tile by TMA between two uses of the same shared buffer, and the store of 64-byte runs
// drains in half the time (pass B's 8-byte gathers cost about the same either way).
__host__ __device__ constexpr int vgroup_of(int n) { return n == 256 ? 8 : n % 4 == 0 ? 4 : 2; }
template <int N> __host__ __device__ constexpr int vgroup() { return vgroup_of(N); }
// Row of c' along V's c' index.  At N = 128 the eight rows c' = w + 16 i that one pass-A warp
// finishes are adjacent (8 w + i), so that the warp leaves them by one TMA store; other N keep c'.
template <int N> __host__ __device__ constexpr int vrow(int c) { return N == 128 ? 8 * (c & 15) + (c >> 4) : c; }
// offset of V(a, b, c', d') in the V layout
template <int N>
__device__ __forceinline__ size_t v_offset(int ab, int c, int d) {
  constexpr int g = vgroup<N>();
  return (((size_t)(vrow<N>(c) * (N / g) + d / g) * (N * N) + ab) * g) + (d % g);
}

template <int N> __host__ __device__ constexpr size_t pass_a_smem() {
  return (size_t)N * pitch<N>() * sizeof(float2) + N * sizeof(float2) + 2 * N * sizeof(float);
}
template <int N> __host__ __device__ constexpr size_t pass_b_smem() {
  return (size_t)N * pitch<N>() * sizeof(float2) + 2 * N * sizeof(float2);
}

// ---- bulk asynchronous copies (TMA) issued by one thread, tracked as bulk groups ----
__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
// Orders this thread's completed async-proxy writes to global memory (bulk / tensor stores)
// before its later generic-proxy operations (a release that publishes them).
__device__ __forceinline__ void fence_proxy_async_global() {
  asm volatile("fence.proxy.async.global;" ::: "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// wait until every committed bulk copy of this thread has finished reading shared memory
__device__ __forceinline__ void bulk_wait_read_all() {
  asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}
// wait until every committed bulk copy of this thread is complete
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
// tiled 5D tensor store from shared memory (box and layout fixed by the tensor map)
__device__ __forceinline__ void tma_store_5d(const void* tmap, const void* smem, int c0, int c1, int c2,
                                             int c3, int c4) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile(
      "cp.async.bulk.tensor.5d.global.shared::cta.tile.bulk_group [%0, {%2, %3, %4, %5, %6}], [%1];" ::"l"(tmap),
      "r"(s), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4)
      : "memory");
}
// contiguous bulk store of `bytes` (multiple of 16, both addresses 16-byte aligned)
__device__ __forceinline__ void bulk_store(void* gdst, const void* smem, unsigned bytes) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(gdst), "r"(s), "r"(bytes)
               : "memory");
}

// Barrier that first lets thread 0 wait for its earlier bulk stores to finish reading shared
// memory: used before a slice's first write into the buffer the previous slice is leaving by TMA.
struct SmemFreeMid {
  __device__ __forceinline__ void operator()() const {
    if (threadIdx.x == 0) bulk_wait_read_all();
    __syncthreads();
  }
};

// In-place shared-memory stages I..IEND-1 along AXIS (0: along the second index, element
// (line, pos) at line*P + pos; 1: along the first index, element (pos, line) at pos*P + line).
template <int N, int SIGN, int AXIS, int I, int IEND, int NT = Plan<N>::NT>
__device__ __forceinline__ void smem_stages(float2* buf, const float2* tw) {
  if constexpr (I < IEND) {
    constexpr int P = pitch<N>();
    constexpr int R = StageInfo<N, I>::R, NS = StageInfo<N, I>::NS;
    auto ld = [buf](int line, int pos) { return AXIS == 0 ? buf[line * P + pos] : buf[pos * P + line]; };
    auto st = [buf](int line, int pos, float2 v) {
      if (AXIS == 0) buf[line * P + pos] = v; else buf[pos * P + line] = v;
    };
    fft_stage<N, R, NS, SIGN, false, NT>(tw, ld, SyncMid{}, st);
    __syncthreads();
    smem_stages<N, SIGN, AXIS, I + 1, IEND, NT>(buf, tw);
  }
}

// Pass A, persistent: CTA blockIdx.x handles point-1 pairs ab = blockIdx.x + k gridDim.x.
// Per slice: generate + DFT along c (lanes along d), DFT along d, write the natural-order slice
// into shared memory and leave it by one TMA tensor store into the V layout (the 5D box
// {2g floats, 1, 1, N/g, N} over (d' mod g, b, a, d'/g, c')).
template <int N, int SRC>
__global__ void __launch_bounds__(Plan<N>::NT, 1) pass_a_kernel(const __grid_constant__ CUtensorMap vmap, PassAArgs p) {
  constexpr bool ARRAY = SRC == SRC_ARRAY;
  constexpr int NT = Plan<N>::NT, P = pitch<N>(), S = Plan<N>::stages;
  extern __shared__ __align__(1024) float2 smem[];
  float2* buf = smem;
  float2* tw = buf + N * P;
  float* gA = reinterpret_cast<float*>(tw + N);
  float* gB = gA + N;
  for (int i = threadIdx.x; i < N; i += NT) tw[i] = p.tw[i];
  const float2* F = p.F;
  for (int ab = blockIdx.x; ab < N * N; ab += gridDim.x) {
    const int a = ab / N, b = ab - a * N;
    if (SRC == SRC_GSM) {
      for (int i = threadIdx.x; i < N; i += NT) {
        gA[i] = p.G[a * N + i];
        gB[i] = p.G[b * N + i];
      }
    }
    __syncthreads();
    float2 s_ab = cconj(__ldg(F + ab));
    if (SRC == SRC_GSM) s_ab = cscale(s_ab, p.A);
    const float2* W0 = ARRAY ? p.W0 + (size_t)ab * N * N : nullptr;
    auto gen = [&](int d, int c) -> float2 {
      const float2 f = __ldg(F + c * N + d);
      if (ARRAY) return cmul(cmul(s_ab, __ldg(W0 + c * N + d)), f);
      return cscale(cmul(s_ab, f), gA[c] * gB[d]);
    };
    auto st1 = [buf](int d, int c, float2 v) { buf[c * P + d] = v; };
    fft_stage<N, StageInfo<N, 0>::R, 1, -1, false, NT>(tw, gen, SmemFreeMid{}, st1);
    __syncthreads();
    smem_stages<N, -1, 1, 1, S>(buf, tw);
    smem_stages<N, -1, 0, 0, S - 1>(buf, tw);
    auto ld0 = [buf](int c, int d) { return buf[c * P + d]; };
    auto nat = [buf](int c, int d, float2 v) { buf[c * N + d] = v; };
    fft_stage<N, StageInfo<N, S - 1>::R, StageInfo<N, S - 1>::NS, -1, true, NT>(tw, ld0, SyncMid{}, nat);
    fence_proxy_async_smem();
    __syncthreads();
    if (threadIdx.x == 0) {
      tma_store_5d(&vmap, buf, 0, b, a, 0, 0);
      bulk_commit();
    }
  }
  if (threadIdx.x == 0) bulk_wait_all();
}

struct PassBArgs {
  const float2* V;
  const float2* tw;
  const float2* Eout;
  float2* W;
  float* S;
  float scale;
};

// What pass B stores of the propagated CSDA: the conjugated column as the contiguous row (Hermitian
// CSDA) or every element at its own place.
enum WStore { W_HERM = 1, W_GENERAL = 2 };

// Pass B, persistent: CTA blockIdx.x handles point-2 output pairs cd = blockIdx.x + k gridDim.x.
// Per slice: gather V(., ., c', d') + DFT along a (lanes along b), DFT along b with the
// epilogue (scale, output propagators, S on the diagonal).  WST = W_HERM:
// the conjugated column is the contiguous row W(c', d', ., .), written to shared memory and left
// by one bulk store; W_GENERAL: strided stores.
template <int N, int WST>
__global__ void __launch_bounds__(Plan<N>::NT, 1) pass_b_kernel(PassBArgs p) {
  constexpr int NT = Plan<N>::NT, P = pitch<N>(), S = Plan<N>::stages;
  constexpr size_t NN = (size_t)N * N;
  extern __shared__ __align__(1024) float2 smem[];
  float2* buf = smem;
  float2* tw = buf + N * P;
  float2* eo = tw + N;
  for (int i = threadIdx.x; i < N; i += NT) {
    tw[i] = p.tw[i];
    eo[i] = p.Eout[i];
  }
  // The g columns of one (c', d'/g) share one block of V; the CTA of column j brings part j of the
  // block of its column after next into L2, so that the gathers (8 bytes from every 32-byte run)
  // hit L2 instead of waiting on DRAM (V is larger than L2 from N = 32 on).
  constexpr int g = vgroup<N>();
  auto prefetch = [&](int cdn) {
    if (N >= 32 && threadIdx.x == 0 && cdn < N * N) {
      const int cn = cdn / N, dn = cdn % N;
      bulk_prefetch_l2(p.V + ((size_t)(vrow<N>(cn) * (N / g) + dn / g) * g + dn % g) * NN, (unsigned)(NN * sizeof(float2)));
    }
  };
  prefetch(blockIdx.x);
  prefetch(blockIdx.x + gridDim.x);
  __syncthreads();
  for (int cd = blockIdx.x; cd < N * N; cd += gridDim.x) {
    prefetch(cd + 2 * gridDim.x);
    const int c = cd / N, d = cd - c * N;
    const float2* Vg = p.V + v_offset<N>(0, c, d);
    auto gather = [Vg](int b, int a) { return __ldg(Vg + (size_t)(a * N + b) * vgroup<N>()); };
    auto st1 = [buf](int b, int a, float2 v) { buf[a * P + b] = v; };
    fft_stage<N, StageInfo<N, 0>::R, 1, +1, false, NT>(tw, gather, SmemFreeMid{}, st1);
    __syncthreads();
    smem_stages<N, +1, 1, 1, S>(buf, tw);
    smem_stages<N, +1, 0, 0, S - 1>(buf, tw);
    const float2 ecd = cscale(cmul(eo[c], eo[d]), p.scale);
    float* Sd = p.S;
    auto ld0 = [buf](int a, int b) { return buf[a * P + b]; };
    if constexpr (WST == W_HERM) {
      auto epi = [=](int a, int b, float2 y) {
        const float2 w = cmul(cmul(cconj(cmul(eo[a], eo[b])), ecd), y);
        if (a == c && b == d) Sd[cd] = w.x;
        buf[a * N + b] = cconj(w);
      };
      fft_stage<N, StageInfo<N, S - 1>::R, StageInfo<N, S - 1>::NS, +1, true, NT>(tw, ld0, SyncMid{}, epi);
      fence_proxy_async_smem();
      __syncthreads();
      if (threadIdx.x == 0) {
        bulk_store(p.W + (size_t)cd * NN, buf, (unsigned)(NN * sizeof(float2)));
        bulk_commit();
      }
    } else {
      float2* W = p.W;
      auto epi = [=](int a, int b, float2 y) {
        const float2 w = cmul(cmul(cconj(cmul(eo[a], eo[b])), ecd), y);
        if (a == c && b == d) Sd[cd] = w.x;
        W[(size_t)(a * N + b) * NN + cd] = w;
      };
      fft_stage<N, StageInfo<N, S - 1>::R, StageInfo<N, S - 1>::NS, +1, true, NT>(tw, ld0, NoMid{}, epi);
    }
  }
  if (threadIdx.x == 0) bulk_wait_all();
}

// S and mu of the current plane (Eq. defS / Algorithm 4, Eq. defMu / Algorithm coherence),
// including masks recorded for this plane (W+ = conj(M0(x1)) W M0(x2)).
struct SMuArgs {
  int N;
  int mode;            // 0: GSM model, 1: CSDA in Wsrc (S from its diagonal), 2: CSDA + S in Sprop,
                       // 3: diagonal source A d(x)
  const float* G;
  float A;
  const float2* M0;    // nullptr = no mask
  const float2* Wsrc;
  const float* Sprop;
  const float* diag;
  int iP, jP;
  float* S_out;        // nullptr = skip
  float2* mu_out;      // nullptr = skip
};

__device__ __forceinline__ float smu_S(const SMuArgs& a, int x) {
  const int N = a.N, i = x / N, j = x - i * N;
  float s;
  if (a.mode == 0) s = a.A * a.G[i * N + i] * a.G[j * N + j];
  else if (a.mode == 3) s = a.A * a.diag[x];
  else if (a.mode == 2) s = a.Sprop[x];
  else s = a.Wsrc[(size_t)x * N * N + x].x;
  if (a.M0) {
    const float2 m = a.M0[x];
    s *= m.x * m.x + m.y * m.y;
  }
  return s;
}

static __global__ void s_mu_kernel(SMuArgs a) {
  const int N = a.N, NN = N * N;
  const int xp = a.iP * N + a.jP;
  const float sp = smu_S(a, xp);
  for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < NN; x += gridDim.x * blockDim.x) {
    const float sx = smu_S(a, x);
    if (a.S_out) a.S_out[x] = sx;
    if (a.mu_out) {
      const int i = x / N, j = x - i * N;
      float2 w;
      if (a.mode == 0) {
        w = make_float2(a.A * a.G[a.iP * N + i] * a.G[a.jP * N + j], 0.f);
      } else if (a.mode == 3) {
        w = make_float2(x == xp ? a.A * a.diag[x] : 0.f, 0.f);
      } else {
        w = a.Wsrc[(size_t)xp * NN + x];
      }
      if (a.M0) w = cmul(cmul(cconj(a.M0[xp]), a.M0[x]), w);
      const float den = sp * sx;
      a.mu_out[x] = den > 0.f ? cscale(w, rsqrtf(den)) : make_float2(0.f, 0.f);
    }
  }
}

}  // namespace pw
