// plane.cuh -- the propagation of a Gaussian Schell-model source, one plane of the output at a time.
//
// The source W1(a, b, c, d) = A conj F(a, b) F(c, d) G(a, c) G(b, d) couples its indices in a ring
// (a-b and c-d through the masks F, a-c and b-d through the coherence G).  With a and d fixed, b and
// c are independent of each other, so for any masks their transforms are tables of N^3 values:
//   H(b'; a, d) = conj E(b') sum_b e^{+2 pi i b b'/N} A conj F(a, b) G(b, d)
//   T(c'; a, d) = E(c') sum_c e^{-2 pi i c c'/N} F(c, d) G(a, c)
// and the propagated CSDA is, for each (b', c'), one 2D transform over (a, d) of their product:
//   W(a', b', c', d') = s conj E(a') E(d') sum_{a,d} e^{+2 pi i a a'/N - 2 pi i d d'/N} H(b'; a, d) T(c'; a, d).
// Two of the four transforms over N^4 values shrink to N^3, there is no half-transformed N^4 array
// and no corner turn: at N <= 128 a plane (a, d) lives in one SM's registers and its result rows
// W(a', b', c', .) are final, so the whole propagation writes its 8 bytes a point once and reads the
// tables from L2.  (The general path moves 24 bytes a point, 40 at N = 256.)
//   table_kernel (table256_kernel): N^2 columns of length N of each table, into the work buffer.
//   plane kernels (24 <= N <= 128; r64.cuh at N = 64, small.cuh with its own tables up to N = 16): one
//   (b', c') per CTA iteration.
//   N = 256: the rows (a, d) and the columns of a plane in two passes, 24 bytes a point.
#pragma once
#include <cuda.h>
#include <cstdint>

#include "ff.cuh"
#include "propagate.cuh"
#include "r128.cuh"
#include "r96.cuh"
#include "t256.cuh"
#include "tc16.cuh"

namespace pw {
namespace plane {

struct TabArgs {
  const float2* F;     // N x N input factors (propagator, lens, aperture, mask, checkerboard)
  const float* G;      // N x N GSM axis factor
  const float2* tw;    // N twiddles exp(-2 pi i m / N)
  const float2* Eout;  // N output factors
  float2* H;           // N^3
  float2* T;           // N^3
  float A;
};

// In-place stages I .. IEND - 1 of the plan on the shared buffer x (a barrier after each).
template <int N, int SIGN, int LINES, int NT, int I, int IEND>
__device__ __forceinline__ void line_stages(float2* x, const float2* tw) {
  if constexpr (I < IEND) {
    auto ld = [x](int line, int pos) { return x[pos * LINES + line]; };
    auto st = [x](int line, int pos, float2 v) { x[pos * LINES + line] = v; };
    line_stage<N, StageInfo<N, I>::R, StageInfo<N, I>::NS, SIGN, LINES, NT>(tw, ld, SyncMid{}, st);
    __syncthreads();
    line_stages<N, SIGN, LINES, NT, I + 1, IEND>(x, tw);
  }
}

// Columns per block and threads of table_kernel (LINES divides N).
template <int N> __host__ __device__ constexpr int tab_lines() { return N <= 32 ? N : N % 32 == 0 ? 32 : 16; }
template <int N> __host__ __device__ constexpr int tab_nt() { return N >= 128 ? 256 : N >= 48 ? 128 : 64; }
template <int N> constexpr size_t tab_smem() { return (size_t)(N * tab_lines<N>() + N) * sizeof(float2); }

// The tables: block (a, LINES columns d) of H (blockIdx.y = 0) or T (1).
template <int N, int SIGN, class Gen, class Out>
__device__ __forceinline__ void table_lines(float2* x, const float2* tw, Gen gen, Out out) {
  constexpr int S = Plan<N>::stages, LINES = tab_lines<N>(), NT = tab_nt<N>();
  if constexpr (S == 1) {
    line_stage<N, StageInfo<N, 0>::R, 1, SIGN, LINES, NT>(tw, gen, NoMid{}, out);
  } else {
    auto st = [x](int line, int pos, float2 v) { x[pos * LINES + line] = v; };
    line_stage<N, StageInfo<N, 0>::R, 1, SIGN, LINES, NT>(tw, gen, NoMid{}, st);
    __syncthreads();
    line_stages<N, SIGN, LINES, NT, 1, S - 1>(x, tw);
    auto ld = [x](int line, int pos) { return x[pos * LINES + line]; };
    line_stage<N, StageInfo<N, S - 1>::R, StageInfo<N, S - 1>::NS, SIGN, LINES, NT>(tw, ld, NoMid{}, out);
  }
}

template <int N>
__global__ void __launch_bounds__(tab_nt<N>()) table_kernel(TabArgs p) {
  constexpr int LINES = tab_lines<N>();
  extern __shared__ __align__(1024) float2 smem[];
  float2* x = smem;
  float2* tw = x + N * LINES;
  for (int i = threadIdx.x; i < N; i += tab_nt<N>()) tw[i] = p.tw[i];
  __syncthreads();
  const int a = blockIdx.x / (N / LINES), d0 = (blockIdx.x % (N / LINES)) * LINES;
  const float2* F = p.F;
  const float* G = p.G;
  const float2* E = p.Eout;
  const float A = p.A;
  if (blockIdx.y == 0) {
    auto gen = [=](int line, int b) { return cscale(cscale(cconj(__ldg(F + a * N + b)), A), __ldg(G + b * N + d0 + line)); };
    float2* H = p.H + (size_t)a * N + d0;
    auto out = [=](int line, int b, float2 v) { H[(size_t)b * N * N + line] = cmul(cconj(__ldg(E + b)), v); };
    table_lines<N, +1>(x, tw, gen, out);
  } else {
    auto gen = [=](int line, int c) { return cscale(__ldg(F + c * N + d0 + line), __ldg(G + a * N + c)); };
    float2* T = p.T + (size_t)a * N + d0;
    auto out = [=](int line, int c, float2 v) { T[(size_t)c * N * N + line] = cmul(__ldg(E + c), v); };
    table_lines<N, -1>(x, tw, gen, out);
  }
}

// N = 256: the same on pairs of floats (ff.cuh), rounded once at the end.  A line of a table goes into 256 planes, and
// most of a row W(P1, .) lies where the planes cancel: the rounding of the FP32 transforms took mu's error from 2.8e-7
// (three passes) to 4.1e-7, here 2.6e-7 (S 1.1e-7, 1.3e-7, 0.9e-7).  16.65 ms a propagation against 16.28 ms with
// FP32 tables, bound by FP32 issue; 4 to 16 columns a block and 128 to 512 threads within 0.07 ms of each other.
constexpr int TAB_L256 = 16, TAB_NT256 = 256, TAB_P256 = TAB_L256 + 1;
constexpr size_t table256_smem() { return (size_t)(256 * TAB_P256 + 256) * sizeof(ff2); }

__global__ void __launch_bounds__(256) table256_tw_kernel(ff2* tw) {
  double sn, cs;
  sincospi(-2.0 * (double)threadIdx.x / 256.0, &sn, &cs);
  tw[threadIdx.x] = make_c(ff(cs), ff(sn));
}

template <int SIGN, int NS = 1>
__device__ __forceinline__ void table256_stages(ff2* x, const ff2* tw) {
  if constexpr (NS < 256) {
    auto ld = [x](int line, int pos) { return x[pos * TAB_P256 + line]; };
    auto st = [x](int line, int pos, ff2 v) { x[pos * TAB_P256 + line] = v; };
    line_stage<256, 4, NS, SIGN, TAB_L256, TAB_NT256>(tw, ld, SyncMid{}, st);
    __syncthreads();
    table256_stages<SIGN, 4 * NS>(x, tw);
  }
}

__global__ void __launch_bounds__(TAB_NT256) table256_kernel(TabArgs p, const ff2* __restrict__ tw2) {
  constexpr int N = 256;
  extern __shared__ __align__(1024) float2 smem[];
  ff2* x = reinterpret_cast<ff2*>(smem);
  ff2* tw = x + N * TAB_P256;
  tw[threadIdx.x] = tw2[threadIdx.x];
  const int a = blockIdx.x / (N / TAB_L256), d0 = (blockIdx.x % (N / TAB_L256)) * TAB_L256;
  const bool h = blockIdx.y == 0;
  const ff A = ff(p.A);
  for (int e = threadIdx.x; e < N * TAB_L256; e += TAB_NT256) {
    const int line = e % TAB_L256, b = e / TAB_L256;  // b, or c of T
    const float2 f = __ldg(p.F + (h ? a * N + b : b * N + d0 + line));
    const ff g = h ? A * ff(__ldg(p.G + b * N + d0 + line)) : ff(__ldg(p.G + a * N + b));
    x[b * TAB_P256 + line] = make_c(ff(f.x) * g, ff(h ? -f.y : f.y) * g);
  }
  __syncthreads();
  if (h) table256_stages<+1>(x, tw);
  else table256_stages<-1>(x, tw);
  float2* out = (h ? p.H : p.T) + (size_t)a * N + d0;
  for (int e = threadIdx.x; e < N * TAB_L256; e += TAB_NT256) {
    const int line = e % TAB_L256, k = e / TAB_L256;
    const float2 E = __ldg(p.Eout + k);
    const ff2 v = cmul(x[k * TAB_P256 + line], make_c(ff(E.x), ff(h ? -E.y : E.y)));
    out[(size_t)k * N * N + line] = make_float2((float)v.x, (float)v.y);
  }
}

struct Args {
  const float2* H;
  const float2* T;
  const float2* tw;
  const float2* Eout;
  float2* W;
  float* S;
  float scale;
  float2* row;  // optional: row[x] = W(P1, x), P1 = (iP, jP)
  int iP, jP;
};

// S and the P1 row from the finished plane (b', c') in shared memory (row a' at buf + at(a') N): thread i of
// n takes part.
template <int N, class At>
__device__ __forceinline__ void plane_s_row(const Args& p, const float2* buf, At at, int bq, int cq, int i, int n) {
  if (i == 0) p.S[cq * N + bq] = buf[at(cq) * N + bq].x;
  if (p.row && bq == p.jP)
    for (int d = i; d < N; d += n) p.row[cq * N + d] = buf[at(p.iP) * N + d];
}

// ---------------------------------------------------------------------------------------------
// N = 24 to 48 (small.cuh up to 16): the generic shared-memory 2D transform of propagate.cuh, one plane per
// block iteration; the natural-order plane leaves by one TMA tensor store (box {2 N floats, 1, 1, N} of W).
template <int N> constexpr size_t plane_smem() {
  return (size_t)N * pitch<N>() * sizeof(float2) + 2 * N * sizeof(float2);
}
template <int N>
__global__ void __launch_bounds__(Plan<N>::NT, 1) plane_kernel(const __grid_constant__ CUtensorMap wmap, Args p) {
  constexpr int NT = Plan<N>::NT, P = pitch<N>(), S = Plan<N>::stages;
  extern __shared__ __align__(1024) float2 smem[];
  float2* buf = smem;
  float2* tw = buf + N * P;
  float2* eo = tw + N;
  for (int i = threadIdx.x; i < N; i += NT) {
    tw[i] = p.tw[i];
    eo[i] = p.Eout[i];
  }
  __syncthreads();
  for (int bc = blockIdx.x; bc < N * N; bc += gridDim.x) {
    const int bq = bc / N, cq = bc - bq * N;
    const float2* __restrict__ H = p.H + (size_t)bq * N * N;
    const float2* __restrict__ T = p.T + (size_t)cq * N * N;
    auto gen = [=](int d, int a) { return cmul(__ldg(H + a * N + d), __ldg(T + a * N + d)); };
    auto st1 = [buf](int d, int a, float2 v) { buf[a * P + d] = v; };
    fft_stage<N, StageInfo<N, 0>::R, 1, +1, false, NT>(tw, gen, SmemFreeMid{}, st1);
    __syncthreads();
    smem_stages<N, +1, 1, 1, S>(buf, tw);
    smem_stages<N, -1, 0, 0, S - 1>(buf, tw);
    auto ld0 = [buf](int a, int d) { return buf[a * P + d]; };
    auto epi = [&](int aq, int dq, float2 y) {
      buf[aq * N + dq] = cmul(cmul(cconj(eo[aq]), cscale(eo[dq], p.scale)), y);
    };
    fft_stage<N, StageInfo<N, S - 1>::R, StageInfo<N, S - 1>::NS, -1, true, NT>(tw, ld0, SyncMid{}, epi);
    fence_proxy_async_smem();
    __syncthreads();
    if (threadIdx.x == 0) {
      tma_store_5d(&wmap, buf, 0, cq, bq, 0, 0);
      bulk_commit();
    }
    plane_s_row<N>(p, buf, [](int a) { return a; }, bq, cq, threadIdx.x, NT);
  }
  if (threadIdx.x == 0) bulk_wait_all();
}

// ---------------------------------------------------------------------------------------------
// N = 96: the register stages of r96.cuh (two CTAs per SM), the plane left by one TMA store.
__global__ void __launch_bounds__(r96::NT, 2) plane96_kernel(const __grid_constant__ CUtensorMap wmap, Args p) {
  using r96::N;
  using r96::NT;
  extern __shared__ __align__(1024) float2 smem[];
  float2* X = smem;
  float2* tw = X + N * r96::P;
  float2* eo = tw + N;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  for (int i = t; i < N; i += NT) {
    tw[i] = p.tw[i];
    eo[i] = p.Eout[i];
  }
  __syncthreads();
  for (int bc = blockIdx.x; bc < N * N; bc += gridDim.x) {
    const int bq = bc / N, cq = bc - bq * N;
    const float2* __restrict__ H = p.H + (size_t)bq * N * N;
    const float2* __restrict__ T = p.T + (size_t)cq * N * N;
    float2 v[2][8][3];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int kp = 0; kp < 8; ++kp)
#pragma unroll
        for (int kq = 0; kq < 3; ++kq) {
          const int ad = (warp + 6 * i + 12 * kp) * N + lane + 32 * kq;
          v[i][kp][kq] = cmul(__ldg(H + ad), __ldg(T + ad));
        }
    if (t == 0) bulk_wait_read_all();  // the previous plane's TMA store has left X
    __syncthreads();
    float2 w3[3][4][4];
    r96::stages<+1, -1>(v, w3, X, tw);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const int u = t + NT * i, jq = u % 24, jp = u / 24;
#pragma unroll
      for (int kp = 0; kp < 4; ++kp) {
        const int aq = jp + 24 * kp;
        const float2 ea = cscale(cconj(eo[aq]), p.scale);
#pragma unroll
        for (int kq = 0; kq < 4; ++kq) {
          const int dq = jq + 24 * kq;
          X[aq * N + dq] = cmul(cmul(ea, eo[dq]), w3[i][kp][kq]);
        }
      }
    }
    fence_proxy_async_smem();
    __syncthreads();
    if (t == 0) {
      tma_store_5d(&wmap, X, 0, cq, bq, 0, 0);
      bulk_commit();
    }
    plane_s_row<N>(p, X, [](int a) { return a; }, bq, cq, t, NT);
  }
  if (t == 0) bulk_wait_all();
}
constexpr size_t plane96_smem() { return (size_t)96 * r96::P * sizeof(float2) + 2 * 96 * sizeof(float2); }

// ---------------------------------------------------------------------------------------------
// N = 128: the register stages of r128.cuh, one CTA per SM, each CTA a contiguous range of planes (c' fastest).
// Reading both factors when a plane starts brings 256 KB into an SM while nothing computes (4096 cycles
// of its L2 bandwidth, 0.97 ms in all), so they come ahead of time, each warp's own rows by its own bulk
// copies on its own mbarrier:
//   - the 8 rows of T of the next plane land in the warp's eight buffer rows as soon as it has read its
//     stage-3 inputs from them (the second exchange permutes rows by vrow, so these are its own);
//   - six of its 8 rows of H stay in shared memory while b' is the same (96 KB; two are read through L2).
// Stage 1 reads and exchange 1 writes only the warp's own rows, so three block barriers a plane are
// enough.  Results go straight from registers to W, 16 bytes a lane; S and the P1 row are read back from
// W by diag_row_kernel (tests for them in the store loop were 5 % of the plane's instructions).  0.844 ms:
// bound by issue, 62 % active at 77 instructions a point; the write of W alone would take 0.32 ms.
constexpr int HROWS128 = 6;
constexpr size_t plane128_smem() {
  return (size_t)(128 * 128 + 16 * HROWS128 * 128 + 2 * 128) * sizeof(float2) + 16 * sizeof(uint64_t);
}
__global__ void __launch_bounds__(r128::NT, 1) plane128_kernel(Args p, int* err) {
  using r128::N;
  using r128::NT;
  constexpr int HR = HROWS128;
  extern __shared__ __align__(1024) float2 smem[];
  float2* buf = smem;
  float2* hs = buf + N * N;  // 16 warps x HR rows of H
  float2* tw = hs + 16 * HR * N;
  float2* eo = tw + N;
  uint64_t* mbars = reinterpret_cast<uint64_t*>(eo + N);
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  for (int i = t; i < N; i += NT) {
    tw[i] = p.tw[i];
    eo[i] = p.Eout[i];
  }
  float2* rows = buf + 8 * warp * N;   // the warp's buffer rows: T rows a = warp + 16 rp
  float2* hrows = hs + HR * warp * N;  // H rows a = warp + 16 rp, rp < HR
  uint64_t* mbar = mbars + warp;
  const int p0 = (int)((long long)blockIdx.x * N * N / gridDim.x), p1 = (int)((long long)(blockIdx.x + 1) * N * N / gridDim.x);
  // lane 0: copies for plane bc (with H where b' is new to the warp)
  auto fetch = [&](int bc, bool with_h) {
    const int bq = bc / N, cq = bc - bq * N;
    fence_proxy_async_smem();
    t256::mbar_expect(mbar, (uint32_t)((8 + (with_h ? HR : 0)) * N * sizeof(float2)));
    for (int rp = 0; rp < 8; ++rp)
      bulk_g2s(rows + rp * N, p.T + ((size_t)cq * N + warp + 16 * rp) * N, N * sizeof(float2), mbar);
    if (with_h)
      for (int rp = 0; rp < HR; ++rp)
        bulk_g2s(hrows + rp * N, p.H + ((size_t)bq * N + warp + 16 * rp) * N, N * sizeof(float2), mbar);
  };
  if (lane == 0) {
    tc16::mbar_init(mbar);
    if (p0 < p1) fetch(p0, true);
  }
  __syncthreads();  // tw, eo
  uint32_t parity = 0;
  int ok = 1;  // (lane 0) a wait that gave up sets *err; the warp then waits and copies no more, its results are
               // invalid, and parity stays that of the phase in flight for the last wait below
  for (int bc = p0; bc < p1; ++bc, parity ^= (uint32_t)ok) {
    const int bq = bc / N, cq = bc - bq * N;
    const float2* __restrict__ H = p.H + (size_t)bq * N * N;
    float2 hx[8 - HR][4];
#pragma unroll
    for (int rp = HR; rp < 8; ++rp)
#pragma unroll
      for (int rq = 0; rq < 4; ++rq) hx[rp - HR][rq] = __ldg(H + (warp + 16 * rp) * N + lane + 32 * rq);
    if (lane == 0 && ok) {
      ok = tc16::mbar_wait(mbar, parity) ? 1 : 0;
      if (!ok) atomicExch(err, 1);
    }
    __syncwarp();
    float2 v[8][4];
#pragma unroll
    for (int rp = 0; rp < 8; ++rp)
#pragma unroll
      for (int rq = 0; rq < 4; ++rq)
        v[rp][rq] = cmul(rp < HR ? hrows[rp * N + lane + 32 * rq] : hx[rp < HR ? 0 : rp - HR][rq], rows[rp * N + lane + 32 * rq]);
    r128::dft2d<8, 4, +1, -1>(v);
    __syncwarp();  // the warp has read its rows of T; exchange 1 writes them
    float2 w3[2][4][4];
    r128::stages_23<+1, true, -1, true>(v, w3, buf, tw, [&]() {
      __syncwarp();
      if (lane == 0 && ok && bc + 1 < p1) fetch(bc + 1, cq == N - 1);
    });
    const int half = lane >> 4, dq0 = 2 * (lane & 15);
    float2* Wt = p.W + ((size_t)(warp + 16 * half) * N * N + bc) * N + dq0;
    float4 ed[4];
#pragma unroll
    for (int rq = 0; rq < 4; ++rq) ed[rq] = *reinterpret_cast<const float4*>(eo + dq0 + 32 * rq);
#pragma unroll
    for (int rp = 0; rp < 4; ++rp) {
      const float2 ea = cscale(cconj(eo[warp + 16 * half + 32 * rp]), p.scale);
#pragma unroll
      for (int rq = 0; rq < 4; ++rq) {
        const float2 w0 = cmul(cmul(ea, make_float2(ed[rq].x, ed[rq].y)), w3[0][rp][rq]);
        const float2 w1 = cmul(cmul(ea, make_float2(ed[rq].z, ed[rq].w)), w3[1][rp][rq]);
        *reinterpret_cast<float4*>(Wt + (size_t)32 * rp * N * N * N + 32 * rq) = make_float4(w0.x, w0.y, w1.x, w1.y);
      }
    }
  }
  if (!ok && lane == 0) tc16::mbar_wait(mbar, parity);  // a copy left in flight by a failed wait
  __syncthreads();
}

__global__ void __launch_bounds__(256) diag_row_kernel(Args p, int N) {
  const int NN = N * N, x = blockIdx.x * 256 + threadIdx.x;
  if (x >= NN) return;
  p.S[x] = p.W[(size_t)x * NN + x].x;
  if (p.row) p.row[x] = p.W[(size_t)(p.iP * N + p.jP) * NN + x];
}

// ---------------------------------------------------------------------------------------------
// N = 256: a plane (512 KB) does not fit an SM, so its rows and its columns are two passes: rows over d
// into W (8 bytes a point written), columns over a in place in W (16 bytes), both in W's natural
// layout.
constexpr int N256 = 256, NT256 = 256;

// Rows: Y(a, b', c', d') = sum_d e^{-2 pi i d d'/N} H(b'; a, d) T(c'; a, d).  A block owns one a, 16
// values of b' (two per warp, one per half-warp) and half of the c'; each lane keeps its 16 points of
// the row of H in registers and meets one row of T after another, which all warps of the block read
// at about the same time (L1), so the tables cost one L2 read per block instead of 16 bytes a point.
// The row transform is 16 x 16: radix 16, twiddle, a transpose through the half-warp's own shared
// memory (pitch 17, no block barrier), radix 16.
constexpr int XP = 17, ROWS_C = 128;
constexpr size_t rows256_smem() { return (size_t)(8 * 2 * 16 * XP + 256) * sizeof(float2); }

__global__ void __launch_bounds__(NT256, 2) rows256_kernel(Args p) {
  constexpr int N = N256;
  extern __shared__ __align__(1024) float2 smem[];
  float2* tr = smem;                  // 8 warps x 2 rows x 16 x XP
  float2* tw = tr + 8 * 2 * 16 * XP;  // w256^(k2 l) at 16 k2 + l
  const int t = threadIdx.x, lane = t & 31, w = t >> 5, l = lane & 15, half = lane >> 4;
  tw[t] = p.tw[(t >> 4) * (t & 15)];
  const int g = blockIdx.x & 15, c0 = ((blockIdx.x >> 4) & 1) * ROWS_C, a = blockIdx.x >> 5;
  const int bq = 16 * g + 2 * w + half;
  const float2* __restrict__ H = p.H + ((size_t)bq * N + a) * N + l;
  const float2* __restrict__ T = p.T + ((size_t)c0 * N + a) * N + l;
  float2* Y = p.W + (((size_t)a * N + bq) * N + c0) * N + l;
  float2* x16 = tr + (w * 2 + half) * 16 * XP;
  float2 h[16], tn[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    h[i] = __ldg(H + 16 * i);
    tn[i] = __ldg(T + 16 * i);
  }
  __syncthreads();  // tw
#pragma unroll 1
  for (int c = 0; c < ROWS_C; ++c, Y += N) {
    float2 x[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) x[i] = cmul(h[i], tn[i]);
    T += (size_t)N * N;
    if (c + 1 < ROWS_C) {
#pragma unroll
      for (int i = 0; i < 16; ++i) tn[i] = __ldg(T + 16 * i);
    }
    Dft<16, -1>::run(x);
#pragma unroll
    for (int k2 = 1; k2 < 16; ++k2) x[k2] = cmul(x[k2], tw[16 * k2 + l]);
    __syncwarp();
#pragma unroll
    for (int k2 = 0; k2 < 16; ++k2) x16[k2 * XP + l] = x[k2];
    __syncwarp();
#pragma unroll
    for (int n1 = 0; n1 < 16; ++n1) x[n1] = x16[l * XP + n1];
    Dft<16, -1>::run(x);  // x[k1] = output d' = l + 16 k1
#pragma unroll
    for (int k1 = 0; k1 < 16; ++k1) Y[16 * k1] = x[k1];
  }
}

// Columns: W(a', b', c', d') = s conj E(a') E(d') sum_a e^{+2 pi i a a'/N} Y(a, b', c', d').  Tile of 32
// consecutive columns, all a: 64 KB by one TMA load (tensor map: W as floats {64, N^3 / 32, 256}), DFT-256
// as two radix-16 stages (line = lane), S, stored back to the same places.  Two CTAs per SM: one
// CTA's load overlaps the other's DFT.
constexpr size_t cols256_smem() { return (size_t)(256 * 32 + 2 * 256) * sizeof(float2) + 64; }

__global__ void __launch_bounds__(NT256, 2) cols256_kernel(const __grid_constant__ CUtensorMap wmap, Args p, int* err) {
  constexpr int N = N256;
  using t256::twid;
  extern __shared__ __align__(1024) float2 smem[];
  float2* X = smem;  // [256][32]
  float2* tw = X + N * 32;
  float2* eo = tw + N;
  uint64_t* mbar = reinterpret_cast<uint64_t*>(eo + N);
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  for (int i = t; i < N; i += NT256) {
    tw[i] = p.tw[i];
    eo[i] = p.Eout[i];
  }
  constexpr int NTILES = N * N * 8;
  auto issue = [&](int tile) {
    fence_proxy_async_smem();
    t256::mbar_expect(mbar, (uint32_t)(N * 32 * sizeof(float2)));
    t256::tma_load_5d(X, &wmap, mbar, 0, tile, 0, 0, 0);
  };
  bool pending = false;  // thread 0: a load was issued and not yet seen complete
  if (t == 0) {
    tc16::mbar_init(mbar);
    if ((int)blockIdx.x < NTILES) {
      issue(blockIdx.x);
      pending = true;
    }
  }
  __syncthreads();
  uint32_t parity = 0;
  for (int tile = blockIdx.x; tile < NTILES; tile += gridDim.x, parity ^= 1u) {
    const int dq = 32 * (tile & 7) + lane, cq = (tile >> 3) & 255, bq = tile >> 11;
    if (!t256::tile_arrived(mbar, parity, err)) break;
    pending = false;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int n1 = 2 * w + e;
      float2 x[16];
#pragma unroll
      for (int n2 = 0; n2 < 16; ++n2) x[n2] = X[(n1 + 16 * n2) * 32 + lane];
      Dft<16, +1>::run(x);
#pragma unroll
      for (int k2 = 1; k2 < 16; ++k2) x[k2] = cmul(x[k2], twid<+1>(tw, n1 * k2));
#pragma unroll
      for (int k2 = 0; k2 < 16; ++k2) X[(n1 + 16 * k2) * 32 + lane] = x[k2];
    }
    __syncthreads();
    float2 y[2][16];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int k2 = 2 * w + e;
#pragma unroll
      for (int n1 = 0; n1 < 16; ++n1) y[e][n1] = X[(n1 + 16 * k2) * 32 + lane];
      Dft<16, +1>::run(y[e]);
    }
    __syncthreads();  // every thread has read X: the next tile may land there
    if (t == 0 && tile + (int)gridDim.x < NTILES) {
      issue(tile + gridDim.x);
      pending = true;
    }
    const float2 ed = cscale(eo[dq], p.scale);
    float2* Wt = p.W + (size_t)tile * 32 + lane;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int k2 = 2 * w + e;
#pragma unroll
      for (int k1 = 0; k1 < 16; ++k1) {
        const int aq = k2 + 16 * k1;
        const float2 v = cmul(cmul(cconj(eo[aq]), ed), y[e][k1]);
        Wt[(size_t)aq * N * N * N] = v;
        if (aq == cq && bq == dq) p.S[cq * N + bq] = v.x;
      }
    }
  }
  if (t == 0 && pending) tc16::mbar_wait(mbar, parity);  // a load left in flight by a failed wait
  __syncthreads();
}

}  // namespace plane
}  // namespace pw
