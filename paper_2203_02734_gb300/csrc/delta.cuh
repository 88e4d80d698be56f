// delta.cuh -- propagation of sources with N^2 non-zeros: the delta-correlated (incoherent) source and the
// adjoint source of a loss on S and mu (the diagonal plus the row of P1).
//
// A point of the source becomes a plane wave, so the propagated array of the diagonal
// d(x1) delta(x1 - x2) depends on x1' - x2' only, apart from the output factors, and the row of P1 gives a
// product of two vectors.  With k = (a', b') and e(k) = E(a') E(b'):
//   W(k1, k2) = s conj e(k1) e(k2) [ D(k1 - k2) + cross(k1, k2) ],
//   D(u) = sum_x d(x) |F(x)|^2 e^{+2 pi i x.u/N}                       (N^2 values, indices mod N)
//   cross = rho(k1) r^(k2) for the row alone, its Hermitian part (the row halved and mirrored as the column)
//           1/2 [rho(k1) r^(k2) + conj(r^(k1) rho(k2))],
//   rho(k) = conj F(P1) e^{+2 pi i P1.k/N},  r^(k) = sum_x F(x) r(x) e^{-2 pi i x.k/N}.
// So the array is written once from tables (8 bytes a point), or not at all where only sums over it are
// wanted.  (Writing V as plane waves and transforming it took 24 bytes a point and a 2D DFT of every
// column: 1.45 ms at N = 128 for an annulus, and 0.64 ms at N = 96 for the parameter gradients.)
#pragma once
#include <cuda_runtime.h>

#include "grad.cuh"

namespace pw {
namespace delta {

struct TabArgs {
  int N;
  const float2* F;
  const float2* tw;
  const float* d;       // N x N diagonal
  float A;              // its weight
  const float2* Eout;   // N output factors
  const float2* q;      // N far-field factors of the adjoint, or nullptr: e takes conj q
  const float2* cross;  // N x N row r, or nullptr
  int iP, jP;
  // correction of d(P1) by the mu term: -1/2 sum(part) / (2 S(P1)) where S(P1) > 0 (adjoint_prep)
  const double* part;   // npart partial sums of r, or nullptr
  int npart;
  const float* S;
  float2* D;            // N x N
  float2* al;           // N x N: conj e(k) rho(k)
  float2* be;           // N x N: e(k) r^(k)
};

// e of one axis.
__device__ __forceinline__ float2 axis_e(const float2* E, const float2* q, int i) {
  const float2 e = __ldg(E + i);
  return q ? cmul(e, cconj(__ldg(q + i))) : e;
}

// Row u of D (blockIdx.y = 0) or row a' of al and be (1): sums over the first axis for every b (G groups of N
// threads share them), then over b.  2 N^3 products in one launch of N blocks.
__global__ void tables_kernel(TabArgs p, int G) {
  extern __shared__ float2 sh[];
  const int N = p.N, t = threadIdx.x, b = t % N, g = t / N;
  float2 *tw = sh, *acc = sh + N;  // acc: G x N
  for (int i = t; i < N; i += blockDim.x) tw[i] = p.tw[i];
  const bool row = blockIdx.y == 1;
  const int u = blockIdx.x, xp = p.iP * N + p.jP;
  float fix = 0.f;
  if (!row && p.part) {
    double rs = 0.0;
    for (int i = 0; i < p.npart; ++i) rs += p.part[i];
    const float sp = p.S[xp];
    if (sp > 0.f) fix = 0.5f * (float)(rs / (2.0 * (double)sp));
  }
  __syncthreads();
  // sum over a of e^{+-2 pi i a u / N} x(a, b)
  float2 s = make_float2(0.f, 0.f);
  const int step = (int)((long long)G * u % N);
  int ia = (int)((long long)g * u % N);
#pragma unroll 4
  for (int a = g; a < N; a += G) {
    const float2 f = __ldg(p.F + a * N + b);
    float2 w = tw[ia];
    if (!row) {
      w.y = -w.y;
      float dv = __ldg(p.d + a * N + b);
      if (a * N + b == xp) dv -= fix;
      const float ad = p.A * dv;  // |F|^2 alone would underflow behind weak masks
      s = cadd(s, cscale(w, fmaf(ad * f.x, f.x, ad * f.y * f.y)));
    } else {
      s = cadd(s, cmul(w, cmul(f, __ldg(p.cross + a * N + b))));
    }
    ia += step;
    ia -= ia >= N ? N : 0;
  }
  acc[g * N + b] = s;
  __syncthreads();
  if (g == 0) {
    for (int k = 1; k < G; ++k) s = cadd(s, acc[k * N + b]);
    acc[b] = s;
  }
  __syncthreads();
  float2 z = make_float2(0.f, 0.f);
  const int v = b, stv = (int)((long long)G * v % N);
  int ib = (int)((long long)g * v % N);
#pragma unroll 4
  for (int c = g; c < N; c += G) {
    float2 w = tw[ib];
    if (!row) w.y = -w.y;
    z = cadd(z, cmul(w, acc[c]));
    ib += stv;
    ib -= ib >= N ? N : 0;
  }
  __syncthreads();
  acc[g * N + v] = z;
  __syncthreads();
  if (g != 0) return;
  for (int k = 1; k < G; ++k) z = cadd(z, acc[k * N + v]);
  if (!row) {
    p.D[u * N + v] = z;
  } else {
    const float2 e = cmul(axis_e(p.Eout, p.q, u), axis_e(p.Eout, p.q, v));
    const int m = (int)(((long long)p.iP * u + (long long)p.jP * v) % N);
    p.al[u * N + v] = cmul(cconj(e), cmul(cconj(__ldg(p.F + xp)), cconj(tw[m])));
    p.be[u * N + v] = cmul(e, z);
  }
}
// Threads of tables_kernel: G groups of N (N even, at most 256).
inline int table_groups(int N) { return N >= 512 ? 1 : 512 / N; }

struct WriteArgs {
  int N;
  const float2* Eout;
  const float2* q;
  const float2* D;
  const float2 *al, *be;  // CROSS
  float kappa;
  float2* W;              // N^4, 16-byte aligned
  float* S;               // N x N: Re W(x, x), or nullptr
};

// W(k1, k2) = kappa [conj e(k1) e(k2) D(k1 - k2) + al(k1) be(k2)], or its conjugate.  A block writes the N^2
// consecutive values of k1 = (a', b'), blocks in order; a thread keeps two neighbouring d' (16-byte
// stores) and walks over c'.  The table D (N^2 values) is read from L1 / L2.  Bound by the write:
// 2.15 GB in 0.33 ms at N = 128.
template <bool CROSS, bool CONJ>
__global__ void __launch_bounds__(256) write_kernel(WriteArgs p) {
  const int N = p.N, H = N / 2, rows = blockDim.x / H;
  const int pd = threadIdx.x % H, r0 = threadIdx.x / H, d0 = 2 * pd;
  const float2 ed0 = axis_e(p.Eout, p.q, d0), ed1 = axis_e(p.Eout, p.q, d0 + 1);
  for (int k1 = blockIdx.x; k1 < N * N; k1 += gridDim.x) {
    const int a = k1 / N, b = k1 - a * N;
    const float2 e1 = cscale(cconj(cmul(axis_e(p.Eout, p.q, a), axis_e(p.Eout, p.q, b))), p.kappa);
    float2 al = make_float2(0.f, 0.f);
    if (CROSS) al = cscale(__ldg(p.al + k1), p.kappa);
    int i0 = b - d0, i1 = i0 - 1;
    i0 += i0 < 0 ? N : 0;
    i1 += i1 < 0 ? N : 0;
    float2* W = p.W + (size_t)k1 * N * N + d0;
#pragma unroll 4
    for (int c = r0; c < N; c += rows) {
      int u = a - c;
      u += u < 0 ? N : 0;
      const float2 f = cmul(e1, axis_e(p.Eout, p.q, c));
      float2 w0 = cmul(cmul(f, ed0), __ldg(p.D + u * N + i0));
      float2 w1 = cmul(cmul(f, ed1), __ldg(p.D + u * N + i1));
      if (CROSS) {
        const float4 be = __ldg(reinterpret_cast<const float4*>(p.be + c * N + d0));
        w0 = cadd(w0, cmul(al, make_float2(be.x, be.y)));
        w1 = cadd(w1, cmul(al, make_float2(be.z, be.w)));
      }
      if (p.S && c == a && (b & ~1) == d0) p.S[k1] = (b & 1) ? w1.x : w0.x;
      if (CONJ) {
        w0.y = -w0.y;
        w1.y = -w1.y;
      }
      *reinterpret_cast<float4*>(W + c * N) = make_float4(w0.x, w0.y, w1.x, w1.y);
    }
  }
}

// Parameter gradients of the amplitude-masked GSM source W0 = A a(x1) a(x2) G(x1, x2) from the adjoint array
// R = kappa conj e(k1) e(k2) [D + Hermitian cross], which is never stored: with
//   t(x1, x2) = Re R(x1, x2) G(x1, x2) a(x1),
// a block takes NC neighbouring columns x2 = (c, d .. d + NC - 1) after one another and adds, over x1,
//   sum t (r^2(x1) + r^2(x2)), sum t |x1 - x2|^2, sum t   (r^2 and |x1 - x2|^2 in pixels^2),
// the last one also as the mask gradient of x2.  Re R = kappa [Re(conj e1 (e2 D)) + Re(al1 be2 + al2 be1) / 2].
// A thread owns one b and walks over a; what depends on x1 alone is loaded once for the NC columns (one
// column at a time took 254 us at N = 96, six loads a term).  N^4 terms of about 20 instructions, 85
// million at N = 96.  FP32 terms and per-thread sums (N^2 / threads terms each), pairs of floats over threads
// and columns (FP64 additions there were 40 % of the kernel), FP64 over blocks, in a fixed order.
struct Pair {  // an unevaluated sum h + l, about 48 bits
  float h = 0.f, l = 0.f;
  __device__ __forceinline__ void add(float x) {
    const float s = h + x, z = s - h;
    l += (h - (s - z)) + (x - z);
    h = s;
  }
  __device__ __forceinline__ void add(Pair o) {
    add(o.h);
    l += o.l;
  }
  __device__ __forceinline__ Pair from(int lanes) const {  // the pair of the lane `lanes` further down
    Pair o;
    o.h = __shfl_down_sync(0xffffffffu, h, lanes);
    o.l = __shfl_down_sync(0xffffffffu, l, lanes);
    return o;
  }
};
struct GradArgs {
  int N;
  const float2* Eout;
  const float2* q;
  const float2* D;
  const float2 *al, *be;  // CROSS
  const float* gtab;      // N x N GSM axis factor
  const float* amask;     // N x N or nullptr
  float kappa, d2;        // d2: d^2 of the source grid
  double* part;           // gridDim.x x 3
  float* gmask;           // N x N or nullptr
  float gscale;           // 4 c A
};

template <bool CROSS, int NC>
__global__ void __launch_bounds__(256) grad_kernel(GradArgs p) {
  __shared__ double red[3][8];
  __shared__ float col[NC][256];
  extern __shared__ float2 ea[];  // N: e of one axis
  const int N = p.N, M = N / 2, rows = blockDim.x / N;
  const int b = threadIdx.x % N, a0 = threadIdx.x / N;
  const bool on = a0 < rows;  // threads beyond the last whole group of N only reduce
  for (int i = threadIdx.x; i < N; i += blockDim.x) ea[i] = axis_e(p.Eout, p.q, i);
  __syncthreads();
  const float2 eb = ea[b];
  const float rb = (float)((b - M) * (b - M));
  Pair tot[3];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int k2 = NC * blockIdx.x; k2 < N * N; k2 += NC * gridDim.x) {
    const int c = k2 / N, d = k2 - c * N;  // NC divides N: one row c
    float sS[NC], sM[NC], sA[NC];
#pragma unroll
    for (int j = 0; j < NC; ++j) sS[j] = sM[j] = sA[j] = 0.f;
    if (on) {
      float2 f2[NC], al2[CROSS ? NC : 1], be2[CROSS ? NC : 1];
      float gb[NC], fb[NC];
      int v[NC];
#pragma unroll
      for (int j = 0; j < NC; ++j) {
        f2[j] = cmul(cconj(eb), cscale(cmul(ea[c], ea[d + j]), p.kappa));  // conj e(b) kappa e(c) e(d)
        if (CROSS) {
          al2[j] = cscale(__ldg(p.al + k2 + j), 0.5f * p.kappa);
          be2[j] = cscale(__ldg(p.be + k2 + j), 0.5f * p.kappa);
        }
        gb[j] = __ldg(p.gtab + b * N + d + j);
        v[j] = b - d - j;
        fb[j] = (float)(v[j] * v[j]);
        v[j] += v[j] < 0 ? N : 0;
      }
#pragma unroll 2
      for (int a = a0; a < N; a += rows) {
        int u = a - c;
        const float fa = (float)(u * u), r1 = (float)((a - M) * (a - M)) + rb;
        u += u < 0 ? N : 0;
        const float2 e1 = ea[a];
        const float2* Du = p.D + u * N;
        float m = __ldg(p.gtab + a * N + c);
        if (p.amask) m *= __ldg(p.amask + a * N + b);
        float2 al1 = make_float2(0.f, 0.f), be1 = al1;
        if (CROSS) {
          al1 = __ldg(p.al + a * N + b);
          be1 = __ldg(p.be + a * N + b);
        }
#pragma unroll
        for (int j = 0; j < NC; ++j) {
          const float2 z = cmul(f2[j], __ldg(Du + v[j]));
          float R = fmaf(e1.x, z.x, e1.y * z.y);
          if (CROSS) {
            R = fmaf(al1.x, be2[j].x, R);
            R = fmaf(-al1.y, be2[j].y, R);
            R = fmaf(al2[j].x, be1.x, R);
            R = fmaf(-al2[j].y, be1.y, R);
          }
          const float tt = R * (m * gb[j]);
          sS[j] = fmaf(tt, r1, sS[j]);
          sM[j] = fmaf(tt, fa + fb[j], sM[j]);
          sA[j] += tt;
        }
      }
    }
#pragma unroll
    for (int j = 0; j < NC; ++j) {
      const float rc = (float)((c - M) * (c - M) + (d + j - M) * (d + j - M));
      const float a2 = p.amask ? __ldg(p.amask + k2 + j) : 1.f;
      tot[0].add(fmaf(rc, sA[j], sS[j]) * a2);
      tot[1].add(sM[j] * a2);
      tot[2].add(sA[j] * a2);
    }
    if (p.gmask) {
      __syncthreads();  // col of the previous columns is read
#pragma unroll
      for (int j = 0; j < NC; ++j) col[j][threadIdx.x] = sA[j];
      __syncthreads();
      for (int j = warp; j < NC; j += nw) {
        Pair x;
        for (int i = lane; i < (int)blockDim.x; i += 32) x.add(col[j][i]);
        for (int o = 16; o > 0; o >>= 1) x.add(x.from(o));
        if (lane == 0) p.gmask[k2 + j] = (float)(p.gscale * ((double)x.h + (double)x.l));
      }
    }
  }
  for (int k = 0; k < 3; ++k) {
    double x = (double)tot[k].h + (double)tot[k].l;
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    if (lane == 0) red[k][warp] = x;
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    double x = 0.0;
    for (int w = 0; w < nw; ++w) x += red[threadIdx.x][w];
    p.part[(size_t)blockIdx.x * 3 + threadIdx.x] = threadIdx.x < 2 ? x * p.d2 : x;
  }
}

}  // namespace delta
}  // namespace pw
