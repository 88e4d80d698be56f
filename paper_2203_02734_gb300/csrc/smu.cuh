// smu.cuh -- S and mu(P1, .) of a propagated Gaussian Schell-model source without its CSDA.
//
// The GSM axis factor is a product, G(a, c) = h(a) h(c) k(a - c) with h(n) = exp(-n^2 d^2/(4 sigma_S^2)) and
// k(u) = exp(-u^2 d^2/(2 sigma_mu^2)), so with the source field P(a, b) = F(a, b) h(a) h(b)
//   S(a', b') = s A sum_{u,v} e^{-2 pi i (u a' + v b')/N} k(u) k(v) C(u, v),
//   C(u, v) = sum_{a,b} conj P(a, b) P(a + u, b + v)
// (the output propagators cancel), and the numerator of mu is
//   W(P1; c', d') = s A conj(E(iP) E(jP)) E(c') E(d') sum_{c,d} e^{-2 pi i (c c' + d d')/N} P(c, d) R(c, d),
//   R = (k x k) * [conj P(a, b) e^{+2 pi i (a iP + b jP)/N}].
// Both the correlation C and the convolution R come from the zero-padded transform P^ of P (L = 2 N per
// axis): C is the inverse transform of |P^|^2, and R that of
//   K(m) K(n) conj P^(2 iP - m, 2 jP - n), K = the transform of k,
// so an instance costs a few FFTs of (2N)^2 points in place of an N^4 array.  (The 4D route took 0.99 ms
// for one instance at N = 128, 87 ms for a batch of 192.)  A few lags carry most of S, so every output takes the
// rounding of the largest: in FP32 the relative error of S was 1e-3 where S is 1e-4 of its maximum (the 4D route,
// whose errors average over N^2 terms, 1e-5), and some dim S came out negative.  So a batch runs on pairs of
// floats (ff.cuh), which leaves the rounding of the outputs alone: 2.6e-8 of S in L2, 6e-8 at every point,
// against 1.8e-7 and 6e-6 in FP32 on well-lit outputs.  192 instances of N = 64 to 128 take 0.62 ms; 0.26 ms in
// FP32, 2.62 ms in FP64.  The single call, for a host loop that waits for it, runs in FP64 (8 MFLOP at N = 96).
//   k1: columns b, transform over a              -> X1[m][b]   (L x N)
//   k2: rows m, transform over b; |P^|^2 back to v, times k(v), to b' -> Z1[m][b'];
//       the R product back to d                  -> Z2[m][d]   (L x N each)
//   k3: columns, Z1 back to u, times k(u), to a' -> S;  Z2 back to c, times P(c, d), to c' -> X3[c'][d]
//   k4: rows c', transform over d                -> mu
// One launch of each covers every instance of one N (blockIdx.y).  A block holds LINES lines in shared
// memory as x[pos * (LINES + 1) + line], so lanes may walk along lines or across them without bank
// conflicts and every global access is contiguous along one of the two.
#pragma once
#include <cuda_runtime.h>

#include <type_traits>

#include "ff.cuh"
#include "propagate.cuh"

namespace pw {
namespace smu {

template <class C>
struct Inst {
  using R = real_t<C>;
  int N, iP, jP;
  int chunk;            // launch round: instances of one round have scratch of their own
  R factor;             // s A / L^2 (float pairs: its sign, the rest is in P1)
  const C* tw;          // L twiddles exp(-2 pi i m / L)
  const C* P1;          // N: Ein(i) h(i)
  const C* Eout;        // N
  const R* k;           // N: k(u)
  R* K;                 // L: transform of k over |u| < N (written by k1)
  const float2* mask;   // N x N or nullptr
  int ap_ithr;          // aperture, as in batch.cuh
  C* scratch;           // 3 L N values
  float* S;             // N x N
  float2* mu;           // N x N or nullptr
};

template <class C> __device__ __forceinline__ C ldc(const C* p) { return __ldg(p); }
__device__ __forceinline__ ff2 ldc(const ff2* p) {
  const float4 v = __ldg(reinterpret_cast<const float4*>(p));
  return make_c(ff(v.x, v.y), ff(v.z, v.w));
}
__device__ __forceinline__ ff ldc(const ff* p) {
  const float2 v = __ldg(reinterpret_cast<const float2*>(p));
  return ff(v.x, v.y);
}

// Lines per block.  Batches (float pairs) fill the chip with instances, and four 16-byte lines make 64-byte runs of
// the column accesses (polychromatic batch of 192, pairs renormalised after every operation: 1216 / 799 / 687 /
// 736 us with 1 / 2 / 4 / 8 lines; 621 us without that).  FP64 calls are one instance: a line per block puts an SM's
// FP64 pipe behind each (N = 96: 16 lines a block left 6 to 12 blocks, 247 us a call; one line 74 us, with the
// radices below 55 us; two lines 58 us).
template <int N, class C> __host__ __device__ constexpr int lines() { return std::is_same<C, ff2>::value ? 4 : 1; }
template <int N, class C> __host__ __device__ constexpr int threads() {
  return N >= 64 ? 256 : 128;
}
template <int N, class C> constexpr size_t smem_bytes() {
  return (size_t)(2 * 2 * N * (lines<N, C>() + 1) + 3 * N) * sizeof(C);
}

// In-place transform of the block's lines (length LEN, natural order), after a barrier and ending with one.
// NS: points already combined.  Radices are fours and then threes and twos: fft.cuh's plans are made for FP32
// registers, and at 2 FP64 operations a clock and SM a radix-16 butterfly keeps its warp for 5 us while most
// warps of the block have none.
template <int LEN, int SIGN, int LINES, int NT, int NS = 1, class C>
__device__ __forceinline__ void fft_lines(C* x, const C* tw) {
  if constexpr (NS < LEN) {
    constexpr int LP = LINES + 1, REM = LEN / NS;
    constexpr int RD = REM % 4 == 0 ? 4 : REM % 3 == 0 ? 3 : 2;
    auto ld = [x](int line, int pos) { return x[pos * LP + line]; };
    auto st = [x](int line, int pos, C v) { x[pos * LP + line] = v; };
    line_stage<LEN, RD, NS, SIGN, LINES, NT>(tw, ld, SyncMid{}, st);
    __syncthreads();
    fft_lines<LEN, SIGN, LINES, NT, NS * RD>(x, tw);
  }
}

// The tables of a block: tw (L) and twN (N = every other entry).
template <int N, class C>
__device__ __forceinline__ void load_tw(const Inst<C>& in, C* tw, C* twN) {
  for (int i = threadIdx.x; i < 2 * N; i += threads<N, C>()) {
    const C v = in.tw[i];
    tw[i] = v;
    if (!(i & 1)) twN[i >> 1] = v;
  }
}

// P(a, b): source field at a point.
template <int N, class C>
__device__ __forceinline__ C field(const Inst<C>& in, int a, int b) {
  using R = real_t<C>;
  const int na = a - N / 2, nb = b - N / 2;
  if (in.ap_ithr >= 0 && na * na + nb * nb > in.ap_ithr) return make_c((R)0.f, (R)0.f);
  C v = cmul(ldc(in.P1 + a), ldc(in.P1 + b));
  if (in.mask) {
    const float2 m = __ldg(in.mask + a * N + b);
    v = cmul(v, make_c((R)m.x, (R)m.y));
  }
  return v;
}

// x[v] <- k(v) x[v] + k(N - v) x[v + N] for v < N: the weighted lags v and v - N, folded mod N.
template <int N, int LINES, int NT, class C>
__device__ __forceinline__ void fold(C* x, const real_t<C>* k) {
  constexpr int LP = LINES + 1;
  for (int e = threadIdx.x; e < N * LINES; e += NT) {
    const int line = e % LINES, v = e / LINES;
    C y = cscale(x[v * LP + line], ldc(k + v));
    if (v > 0) y = cadd(y, cscale(x[(v + N) * LP + line], ldc(k + N - v)));
    x[v * LP + line] = y;
  }
  __syncthreads();
}

template <class C>
__device__ __forceinline__ Inst<C> pick(const Inst<C>* list, const Inst<C>& one) {
  return list ? list[blockIdx.y] : one;
}

template <int N, class C>
__global__ void __launch_bounds__(threads<N, C>()) k1(const Inst<C>* list, Inst<C> one, int chunk) {
  using R = real_t<C>;
  constexpr int L = 2 * N, LINES = lines<N, C>(), LP = LINES + 1, NT = threads<N, C>();
  const Inst<C> in = pick(list, one);
  if (in.N != N || in.chunk != chunk) return;
  extern __shared__ __align__(16) unsigned char smem[];
  C *x = reinterpret_cast<C*>(smem), *tw = x + 2 * L * LP, *twN = tw + L;
  load_tw<N>(in, tw, twN);
  const int b0 = blockIdx.x * LINES;
  if (b0 == N) {  // the last block: K
    for (int e = threadIdx.x; e < L * LINES; e += NT) {
      const int line = e % LINES, u = e / LINES;
      x[u * LP + line] = make_c(line || u == N ? (R)0.f : ldc(in.k + (u < N ? u : L - u)), (R)0.f);
    }
    __syncthreads();
    fft_lines<L, -1, LINES, NT>(x, tw);
    for (int m = threadIdx.x; m < L; m += NT) in.K[m] = x[m * LP].x;
    return;
  }
  for (int e = threadIdx.x; e < L * LINES; e += NT) {
    const int line = e % LINES, a = e / LINES;
    x[a * LP + line] = a < N ? field<N, C>(in, a, b0 + line) : make_c((R)0.f, (R)0.f);
  }
  __syncthreads();
  fft_lines<L, -1, LINES, NT>(x, tw);
  for (int e = threadIdx.x; e < L * LINES; e += NT) {
    const int line = e % LINES, m = e / LINES;
    in.scratch[m * N + b0 + line] = x[m * LP + line];
  }
}

template <int N, class C>
__global__ void __launch_bounds__(threads<N, C>()) k2(const Inst<C>* list, Inst<C> one, int chunk) {
  using R = real_t<C>;
  constexpr int L = 2 * N, LINES = lines<N, C>(), LP = LINES + 1, NT = threads<N, C>();
  const Inst<C> in = pick(list, one);
  if (in.N != N || in.chunk != chunk) return;
  extern __shared__ __align__(16) unsigned char smem[];
  C *x = reinterpret_cast<C*>(smem), *y = x + L * LP, *tw = y + L * LP, *twN = tw + L;
  load_tw<N>(in, tw, twN);
  const int m0 = blockIdx.x * LINES;
  const C* X1 = in.scratch;
  C* Z1 = in.scratch + (size_t)L * N;
  C* Z2 = Z1 + (size_t)L * N;
  for (int e = threadIdx.x; e < L * LINES; e += NT) {
    const int b = e % L, line = e / L;
    x[b * LP + line] = b < N ? X1[(m0 + line) * N + b] : make_c((R)0.f, (R)0.f);
  }
  __syncthreads();
  fft_lines<L, -1, LINES, NT>(x, tw);  // P^(m, n)
  if (in.mu) {
    for (int e = threadIdx.x; e < L * LINES; e += NT) {  // row m' = 2 iP - m of the R product
      const int line = e % LINES, n = e / LINES;
      int mm = 2 * in.iP - (m0 + line), nn = 2 * in.jP - n;
      mm += mm < 0 ? L : 0;
      nn += nn < 0 ? L : 0;
      y[n * LP + line] = cscale(cconj(x[nn * LP + line]), ldc(in.K + mm) * ldc(in.K + n));
    }
    __syncthreads();
  }
  for (int e = threadIdx.x; e < L * LINES; e += NT) {
    const int line = e % LINES, n = e / LINES;
    const C v = x[n * LP + line];
    x[n * LP + line] = make_c(fma_(v.x, v.x, v.y * v.y), (R)0.f);
  }
  __syncthreads();
  fft_lines<L, +1, LINES, NT>(x, tw);
  fold<N, LINES, NT>(x, in.k);
  fft_lines<N, -1, LINES, NT>(x, twN);
  for (int e = threadIdx.x; e < N * LINES; e += NT) {
    const int b = e % N, line = e / N;
    Z1[(m0 + line) * N + b] = x[b * LP + line];
  }
  if (in.mu) {
    fft_lines<L, +1, LINES, NT>(y, tw);
    for (int e = threadIdx.x; e < N * LINES; e += NT) {
      const int d = e % N, line = e / N;
      int mm = 2 * in.iP - (m0 + line);
      mm += mm < 0 ? L : 0;
      Z2[mm * N + d] = y[d * LP + line];
    }
  }
}

template <int N, class C>
__global__ void __launch_bounds__(threads<N, C>()) k3(const Inst<C>* list, Inst<C> one, int chunk) {
  using R = real_t<C>;
  constexpr int L = 2 * N, LINES = lines<N, C>(), LP = LINES + 1, NT = threads<N, C>();
  const Inst<C> in = pick(list, one);
  if (in.N != N || in.chunk != chunk) return;
  extern __shared__ __align__(16) unsigned char smem[];
  C *x = reinterpret_cast<C*>(smem), *tw = x + 2 * L * LP, *twN = tw + L;
  load_tw<N>(in, tw, twN);
  const int b0 = blockIdx.x * LINES;
  C* X3 = in.scratch;
  const C* Z1 = in.scratch + (size_t)L * N;
  const C* Z2 = Z1 + (size_t)L * N;
  for (int e = threadIdx.x; e < L * LINES; e += NT) {
    const int line = e % LINES, m = e / LINES;
    x[m * LP + line] = Z1[m * N + b0 + line];
  }
  __syncthreads();
  fft_lines<L, +1, LINES, NT>(x, tw);
  fold<N, LINES, NT>(x, in.k);
  fft_lines<N, -1, LINES, NT>(x, twN);
  for (int e = threadIdx.x; e < N * LINES; e += NT) {
    const int line = e % LINES, a = e / LINES;
    in.S[a * N + b0 + line] = (float)(x[a * LP + line].x * in.factor);
  }
  if (!in.mu) return;
  __syncthreads();
  for (int e = threadIdx.x; e < L * LINES; e += NT) {
    const int line = e % LINES, m = e / LINES;
    x[m * LP + line] = Z2[m * N + b0 + line];
  }
  __syncthreads();
  fft_lines<L, +1, LINES, NT>(x, tw);
  for (int e = threadIdx.x; e < N * LINES; e += NT) {
    const int line = e % LINES, c = e / LINES;
    x[c * LP + line] = cmul(field<N, C>(in, c, b0 + line), x[c * LP + line]);
  }
  __syncthreads();
  fft_lines<N, -1, LINES, NT>(x, twN);
  for (int e = threadIdx.x; e < N * LINES; e += NT) {
    const int line = e % LINES, c = e / LINES;
    X3[c * N + b0 + line] = x[c * LP + line];
  }
}

template <int N, class C>
__global__ void __launch_bounds__(threads<N, C>()) k4(const Inst<C>* list, Inst<C> one, int chunk) {
  using R = real_t<C>;
  constexpr int LINES = lines<N, C>(), LP = LINES + 1, NT = threads<N, C>(), L = 2 * N;
  const Inst<C> in = pick(list, one);
  if (in.N != N || in.chunk != chunk || !in.mu) return;
  extern __shared__ __align__(16) unsigned char smem[];
  C *x = reinterpret_cast<C*>(smem), *tw = x + 2 * L * LP, *twN = tw + L;
  load_tw<N>(in, tw, twN);
  const int c0 = blockIdx.x * LINES;
  for (int e = threadIdx.x; e < N * LINES; e += NT) {
    const int d = e % N, line = e / N;
    x[d * LP + line] = in.scratch[(c0 + line) * N + d];
  }
  __syncthreads();
  fft_lines<N, -1, LINES, NT>(x, twN);
  const float sp = in.S[in.iP * N + in.jP];
  const C ep = cscale(cconj(cmul(ldc(in.Eout + in.iP), ldc(in.Eout + in.jP))), in.factor);
  for (int e = threadIdx.x; e < N * LINES; e += NT) {
    const int d = e % N, line = e / N, c = c0 + line;
    const float den = sp * in.S[c * N + d];
    const C row = cmul(cmul(ep, cmul(ldc(in.Eout + c), ldc(in.Eout + d))), x[d * LP + line]);
    const float inv = rsqrtf(den);
    in.mu[c * N + d] = den > 0.f ? make_float2((float)row.x * inv, (float)row.y * inv) : make_float2(0.f, 0.f);
  }
}

// FP64-derived tables of one instance: twiddles, per-axis factors, coherence.
template <class C>
struct TabArgs {
  int N;
  double Kin, Kout;  // turns per n^2 of the input factor (propagator, lens) and of the output propagator
  double gs, gm;     // d^2/(4 sigma_S^2), d^2/(2 sigma_mu^2)
  double amp;        // factor of P1: with (s |A| / L^2)^(1/4) the sums between are of the size of S, whatever A and
                     // the masks are by themselves (float pairs have FP32's range; FP64: 1)
  C *tw, *P1, *Eout;
  real_t<C>* k;
};

// One FP64 evaluation per task: tasks 0..L-1 tw, then P1, Eout and k of each index.
template <class C>
__device__ __forceinline__ void tables(const TabArgs<C>& t, int q0, int step) {
  using R = real_t<C>;
  const int N = t.N, L = 2 * N, M = N / 2;
  for (int q = q0; q < L + 3 * N; q += step) {
    const int kind = q < L ? -1 : (q - L) / N, i = q < L ? q : (q - L) - kind * N;
    const double n2 = (double)(i - M) * (double)(i - M);
    if (kind == 2) {
      t.k[i] = (R)exp(-(double)i * (double)i * t.gm);
      continue;
    }
    const double turns = kind < 0 ? -(double)i / (double)L : frac_turns(n2 * (kind == 0 ? t.Kin : t.Kout)) + 0.5 * (i & 1);
    double sn, cs;
    sincospi(2.0 * frac_turns(turns), &sn, &cs);
    if (kind < 0) {
      t.tw[i] = make_c((R)cs, (R)sn);
    } else if (kind == 1) {
      t.Eout[i] = make_c((R)cs, (R)sn);
    } else {
      const double hh = t.amp * exp(-n2 * t.gs);
      t.P1[i] = make_c((R)(cs * hh), (R)(sn * hh));
    }
  }
}

template <int N, class C>
cudaError_t launch(const Inst<C>* list, const Inst<C>& one, int n, int chunk, bool any_mu, cudaStream_t s) {
  constexpr int LINES = lines<N, C>(), NT = threads<N, C>();
  constexpr size_t sm = smem_bytes<N, C>();
  static bool ready = false;
  cudaError_t e = cudaSuccess;
  if (!ready) {
    if ((e = cudaFuncSetAttribute(k1<N, C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm)) != cudaSuccess ||
        (e = cudaFuncSetAttribute(k2<N, C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm)) != cudaSuccess ||
        (e = cudaFuncSetAttribute(k3<N, C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm)) != cudaSuccess ||
        (e = cudaFuncSetAttribute(k4<N, C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm)) != cudaSuccess)
      return e;
    ready = true;
  }
  k1<N, C><<<dim3(N / LINES + 1, n), NT, sm, s>>>(list, one, chunk);
  k2<N, C><<<dim3(2 * N / LINES, n), NT, sm, s>>>(list, one, chunk);
  k3<N, C><<<dim3(N / LINES, n), NT, sm, s>>>(list, one, chunk);
  if (any_mu) k4<N, C><<<dim3(N / LINES, n), NT, sm, s>>>(list, one, chunk);
  return cudaGetLastError();
}

}  // namespace smu
}  // namespace pw
