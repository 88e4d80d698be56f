// small.cuh -- the planes of plane.cuh for N <= 16, tables included, in one kernel.
//
// One block per output plane (b', c'), one thread per point.  H(b'; a, d) and T(c'; a, d) are sums of N terms
// of which a plane needs one b' and one c': at N = 16 the block forms them by direct sums in as many
// instructions as its two transforms, and a separate table launch (5 us of latency for 0.2 us of work) is
// saved.  The transforms are direct sums too: 256 planes of 256 points keep every SM busy for about a
// microsecond.  Above N = 16 the O(N) sums per point cost more than the launch (at N = 32 some 10 us of
// shared-memory reads against 5 us for table_kernel).
// The allocation-free call at N = 16: 15.4 us in three launches (tables, two passes of 5 us each), 11.5 in two.
#pragma once
#include <cuda_runtime.h>

#include <cmath>

#include "fft.cuh"

namespace pw {
namespace small {

constexpr int MAX_N = 16;

struct Args {
  const float2* F;     // N x N input factors
  const float* G;      // N x N GSM axis factor
  const float2* tw;    // N twiddles exp(-2 pi i m / N)
  const float2* Eout;  // N output factors
  float2* W;
  float* S;
  float scale, pow2;  // s A = scale pow2
  float2* row;  // optional: row[x] = W(P1, x), P1 = (iP, jP)
  int iP, jP;
};

// The scale s A in two factors: a power of two that goes to the source without rounding, so that a large A meets weak
// masks there and not after their product, and the rest, rounded once.
struct Scale {
  float scale, pow2;
  Scale(double s, double A) {
    int k = 0;
    const double m = std::frexp(A, &k);  // A = 2 m 2^(k - 1): the power of any finite float is one
    scale = (float)(s * 2.0 * m);
    pow2 = std::ldexp(1.0f, k - 1);
  }
};

template <int N>
__global__ void __launch_bounds__(N * N) kernel(Args p) {
  constexpr int NN = N * N;
  __shared__ float2 fb[NN], fc[NN], x[NN], y[NN], tw[N];
  __shared__ float g[NN];
  const int t = threadIdx.x, i = t / N, j = t % N, bp = blockIdx.y, cp = blockIdx.x;
  if (t < N) tw[t] = p.tw[t];
  g[t] = p.G[t];
  const float2 f = p.F[t];
  const float2 e = cmul(cconj(p.Eout[bp]), p.Eout[cp]);  // of H T
  const float2 eo = cmul(cconj(p.Eout[i]), p.Eout[j]);   // of (a', d')
  fb[t] = cmul(cscale(cconj(f), p.pow2), cconj(p.tw[j * bp % N]));  // (a, b) = (i, j)
  fc[t] = cmul(f, p.tw[i * cp % N]);                                // (c, d) = (i, j)
  __syncthreads();
  // Sums in four shares: as one chain each, they took the error of W from 1.55e-7 (general passes) to 1.82e-7 at
  // N = 16; in shares, and with A in the scale, 1.53e-7.  (Their time is made up for by a barrier less, with the first
  // twiddles from memory, and by indices i a mod N in place of running ones: two launches 7.05 -> 6.96 us in a graph.)
  auto total = [](const float2 (&v)[4]) { return cadd(cadd(v[0], v[1]), cadd(v[2], v[3])); };
  auto add = [](float2& s, float2 v, float2 w) {  // s += v w
    s = make_float2(fmaf(v.x, w.x, fmaf(-v.y, w.y, s.x)), fmaf(v.x, w.y, fmaf(v.y, w.x, s.y)));
  };
  // (a, d) = (i, j)
  float2 h[4] = {}, u[4] = {};
#pragma unroll
  for (int n = 0; n < N; ++n) {
    const float2 a = fb[i * N + n], b = fc[n * N + j];
    const float gb = g[n * N + j], gc = g[i * N + n];
    float2 &hn = h[n & 3], &un = u[n & 3];
    hn = make_float2(fmaf(a.x, gb, hn.x), fmaf(a.y, gb, hn.y));
    un = make_float2(fmaf(b.x, gc, un.x), fmaf(b.y, gc, un.y));
  }
  x[t] = cmul(cmul(total(h), total(u)), e);
  __syncthreads();
  float2 r[4] = {};
#pragma unroll
  for (int d = 0; d < N; ++d) add(r[d & 3], x[i * N + d], tw[j * d % N]);
  y[t] = total(r);  // (a, d')
  __syncthreads();
  float2 q[4] = {};
#pragma unroll
  for (int a = 0; a < N; ++a) add(q[a & 3], y[a * N + j], cconj(tw[i * a % N]));
  const float2 s = total(q);
  const float2 w = cscale(cmul(s, eo), p.scale);  // W(a' = i, b', c', d' = j)
  p.W[(size_t)((i * N + bp) * N + cp) * N + j] = w;
  if (i == cp && j == bp) p.S[t] = w.x;
  if (p.row && i == p.iP && bp == p.jP) p.row[cp * N + j] = w;
}

template <int N>
cudaError_t launch(const Args& a, cudaStream_t s) {
  kernel<N><<<dim3(N, N), N * N, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace small
}  // namespace pw
