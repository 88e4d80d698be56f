// r64.cuh -- register-resident 2D DFT of a 64 x 64 slice: the plane kernel of a GSM source and the two
// general passes at N = 64.
//
// 64 = 4 x 4 x 4 per axis: three 2D Stockham stages of radix (4, 4), 256 threads, 16 points per thread;
// thread t has butterfly (jp, jq) = (t / 16, t mod 16) in every stage:
//   stage 1: inputs (jp + 16 rp, jq + 16 rq), outputs (4 jp + rp, 4 jq + rq);
//   stage 2: the same inputs, twiddles w16^(rp (jp mod 4)) w16^(rq (jq mod 4)), outputs (16 (jp / 4) +
//            jp mod 4 + 4 rp, 16 (jq / 4) + jq mod 4 + 4 rq);
//   stage 3: the same inputs, twiddles w64^(rp jp) w64^(rq jq), outputs in natural order at the input
//            positions
// (w_L = exp(+-2 pi i / L)).  Points move between stages through two 32 KB buffers, so that two block
// barriers a slice are enough; the column index is XOR-swizzled (q ^ ((q >> 4) & 3), then
// q ^ (((q >> 4) & 3) << 2)) so that 16 lanes touch 16 distinct 8-byte bank pairs on both sides.  Three CTAs share
// an SM (65 KB of shared memory each) and hide each other's loads and barriers.  The generic engine
// (radices 8, 8 per axis in shared memory) moved each point through shared memory seven times: plane 68 us,
// first pass 62 us, second pass 84 us at 16.8 million points.
#pragma once
#include "plane.cuh"
#include "r128.cuh"

namespace pw {
namespace r64 {

constexpr int N = 64, NT = 256, CTAS = 3;
constexpr size_t smem_bytes() { return (size_t)(2 * N * N + 2 * N) * sizeof(float2); }

__device__ __forceinline__ int sw1(int q) { return q ^ ((q >> 4) & 3); }
__device__ __forceinline__ int sw2(int q) { return q ^ (((q >> 4) & 3) << 2); }

// Stages 1 to 3 on the thread's points v (sign SP along p, SQ along q).  Contract: A is free on entry (the
// block has passed a barrier since its last use); on return B may still be read by other threads, A not.
template <int SP, int SQ>
__device__ __forceinline__ void transform(float2 (&v)[4][4], float2* A, float2* B, const float2* tw) {
  const int jp = threadIdx.x >> 4, jq = threadIdx.x & 15;
  r128::dft2d<4, 4, SP, SQ>(v);
#pragma unroll
  for (int rp = 0; rp < 4; ++rp)
#pragma unroll
    for (int rq = 0; rq < 4; ++rq) A[(4 * jp + rp) * N + sw1(4 * jq + rq)] = v[rp][rq];
  __syncthreads();
#pragma unroll
  for (int rp = 0; rp < 4; ++rp)
#pragma unroll
    for (int rq = 0; rq < 4; ++rq) v[rp][rq] = A[(jp + 16 * rp) * N + sw1(jq + 16 * rq)];
  r128::twiddle2d<4, 4, SP, SQ>(v, tw, 4 * (jp & 3), 4 * (jq & 3));
  r128::dft2d<4, 4, SP, SQ>(v);
#pragma unroll
  for (int rp = 0; rp < 4; ++rp)
#pragma unroll
    for (int rq = 0; rq < 4; ++rq)
      B[(16 * (jp >> 2) + (jp & 3) + 4 * rp) * N + sw2(16 * (jq >> 2) + (jq & 3) + 4 * rq)] = v[rp][rq];
  __syncthreads();
#pragma unroll
  for (int rp = 0; rp < 4; ++rp)
#pragma unroll
    for (int rq = 0; rq < 4; ++rq) v[rp][rq] = B[(jp + 16 * rp) * N + sw2(jq + 16 * rq)];
  r128::twiddle2d<4, 4, SP, SQ>(v, tw, jp, jq);
  r128::dft2d<4, 4, SP, SQ>(v);
}

// A plane (b', c') of a GSM source (plane.cuh) per block iteration, stored from registers (128-byte runs).
__global__ void __launch_bounds__(NT, CTAS) plane64_kernel(plane::Args p) {
  extern __shared__ __align__(1024) float2 smem[];
  float2 *A = smem, *B = A + N * N, *tw = B + N * N, *eo = tw + N;
  const int t = threadIdx.x, jp = t >> 4, jq = t & 15;
  if (t < N) {
    tw[t] = p.tw[t];
    eo[t] = p.Eout[t];
  }
  __syncthreads();
  for (int bc = blockIdx.x; bc < N * N; bc += gridDim.x) {
    const int bq = bc / N, cq = bc - bq * N;
    const float2* __restrict__ H = p.H + (size_t)bq * N * N + jp * N + jq;
    const float2* __restrict__ T = p.T + (size_t)cq * N * N + jp * N + jq;
    float2 v[4][4];
#pragma unroll
    for (int rp = 0; rp < 4; ++rp)
#pragma unroll
      for (int rq = 0; rq < 4; ++rq) v[rp][rq] = cmul(__ldg(H + 16 * (rp * N + rq)), __ldg(T + 16 * (rp * N + rq)));
    transform<+1, -1>(v, A, B, tw);
    float2* Wt = p.W + ((size_t)jp * N * N + bc) * N + jq;
#pragma unroll
    for (int rp = 0; rp < 4; ++rp) {
      const int aq = jp + 16 * rp;
      const float2 ea = cscale(cconj(eo[aq]), p.scale);
#pragma unroll
      for (int rq = 0; rq < 4; ++rq) {
        const int dq = jq + 16 * rq;
        const float2 w = cmul(cmul(ea, eo[dq]), v[rp][rq]);
        Wt[(size_t)16 * rp * N * N * N + 16 * rq] = w;
        if (aq == cq && dq == bq) p.S[cq * N + bq] = w.x;
        if (p.row && bq == p.jP && aq == p.iP) p.row[cq * N + dq] = w;
      }
    }
  }
}

// Pass A (propagate.cuh) of an uploaded or propagated array: slice (a, b), sign - over (c, d), left in
// natural order by one TMA store into the V layout.
__global__ void __launch_bounds__(NT, CTAS) pass_a_r64(const __grid_constant__ CUtensorMap vmap, PassAArgs p) {
  extern __shared__ __align__(1024) float2 smem[];
  float2 *A = smem, *B = A + N * N, *tw = B + N * N;
  const int t = threadIdx.x, jp = t >> 4, jq = t & 15;
  if (t < N) tw[t] = p.tw[t];
  const float2* __restrict__ F = p.F + jp * N + jq;
  for (int ab = blockIdx.x; ab < N * N; ab += gridDim.x) {
    const int a = ab / N, b = ab - a * N;
    const float2 s_ab = cconj(__ldg(p.F + ab));
    const float2* __restrict__ W0 = p.W0 + (size_t)ab * N * N + jp * N + jq;
    float2 v[4][4];
#pragma unroll
    for (int rp = 0; rp < 4; ++rp)
#pragma unroll
      for (int rq = 0; rq < 4; ++rq)
        v[rp][rq] = cmul(cmul(s_ab, __ldg(W0 + 16 * (rp * N + rq))), __ldg(F + 16 * (rp * N + rq)));
    if (t == 0) bulk_wait_read_all();  // the previous slice's store has left A
    __syncthreads();
    transform<-1, -1>(v, A, B, tw);
#pragma unroll
    for (int rp = 0; rp < 4; ++rp)
#pragma unroll
      for (int rq = 0; rq < 4; ++rq) A[(jp + 16 * rp) * N + jq + 16 * rq] = v[rp][rq];
    fence_proxy_async_smem();
    __syncthreads();
    if (t == 0) {
      tma_store_5d(&vmap, A, 0, b, a, 0, 0);
      bulk_commit();
    }
  }
  if (t == 0) bulk_wait_all();
}

// Pass B of a Hermitian array: column (c', d') gathered from V (its group's block brought into L2 two columns
// ahead), sign + over (a, b), the conjugated column stored as the row W(c', d', ., .) from registers.
__global__ void __launch_bounds__(NT, CTAS) pass_b_r64(PassBArgs p) {
  extern __shared__ __align__(1024) float2 smem[];
  float2 *A = smem, *B = A + N * N, *tw = B + N * N, *eo = tw + N;
  constexpr int g = vgroup<N>();
  const int t = threadIdx.x, jp = t >> 4, jq = t & 15;
  if (t < N) {
    tw[t] = p.tw[t];
    eo[t] = p.Eout[t];
  }
  auto prefetch = [&](int cd) {
    if (t == 0 && cd < N * N)
      bulk_prefetch_l2(p.V + (size_t)cd * N * N, (unsigned)(N * N * sizeof(float2)));
  };
  prefetch(blockIdx.x);
  prefetch(blockIdx.x + gridDim.x);
  __syncthreads();
  for (int cd = blockIdx.x; cd < N * N; cd += gridDim.x) {
    const int c = cd / N, d = cd - c * N;
    prefetch(cd + 2 * gridDim.x);
    const float2* __restrict__ Vg = p.V + v_offset<N>(jp * N + jq, c, d);
    float2 v[4][4];
#pragma unroll
    for (int rp = 0; rp < 4; ++rp)
#pragma unroll
      for (int rq = 0; rq < 4; ++rq) v[rp][rq] = __ldg(Vg + (size_t)16 * (rp * N + rq) * g);
    transform<+1, +1>(v, A, B, tw);
    const float2 ecd = cscale(cmul(eo[c], eo[d]), p.scale);
    float2* Wrow = p.W + (size_t)cd * N * N + jp * N + jq;
#pragma unroll
    for (int rp = 0; rp < 4; ++rp) {
      const int a = jp + 16 * rp;
      const float2 ea = cmul(cconj(eo[a]), ecd);
#pragma unroll
      for (int rq = 0; rq < 4; ++rq) {
        const int b = jq + 16 * rq;
        const float2 w = cmul(cmul(ea, cconj(eo[b])), v[rp][rq]);
        if (a == c && b == d) p.S[cd] = w.x;
        Wrow[16 * (rp * N + rq)] = cconj(w);
      }
    }
  }
}

}  // namespace r64
}  // namespace pw
