// grad.cuh -- parameter gradients of a loss through the propagation, from the adjoint.
//
// For W_B = P(W0) and a real loss L, the conjugate-Wirtinger gradient W0bar = dL/dW0* equals
// P^H(dL/dW_B*), and P^H of a Fresnel propagation over z from sampling d is the conjugate of a
// Fresnel propagation over the same z of the conjugated array, started from the output sampling
// dx = lambda z/(N d) and scaled by (d/dx)^4 (the factorisation P = s D_out F D_in with
// F^H = conj F).  The caller runs that forward propagation; its result R on the source grid gives
// conj(W0bar) = c R (c = (d/dx)^4, times q(xi1) q*(xi2) for a far-field forward P).  This kernel
// then forms, for the amplitude-masked GSM source W0 = A a(xi1) a(xi2) G(xi1, xi2) (Sec. 5.4),
//   dL/dtheta = 2 Re sum conj(W0bar) dW0/dtheta   (theta = sigma_S, sigma_mu, A, a(eta)),
// reading R once; W0 and dW0/dtheta are generated in registers.
#pragma once
#include "propagate.cuh"

namespace pw {

struct GradArgs {
  int N;
  double d;           // source sampling
  double sigma_S, sigma_mu, A;
  const float* amask; // N x N amplitude mask or nullptr (a = 1)
  const float2* R;    // N^4 result of the adjoint propagation
  double c;           // (d/dx)^4
  int farfield;
  double Kq;          // far field: q(xi) = exp(2 pi i Kq n^2) per axis, Kq = d^2/(2 lambda z)
  double* part;       // rows x 3 partial sums (scratch)
  int rows;           // number of partial sums: N^2 from gsm_gradient_kernel
  float* gtab;        // N x N GSM axis factor G(i, k) (scratch, filled by gsm_gradient_tables)
  float2* qtab;       // N far-field factors q(x_i) (scratch)
  double* g3;         // [dL/dsigma_S, dL/dsigma_mu, dL/dA]
  float* gmask;       // N x N dL/da or nullptr
};

// The GSM axis factor G(i, k) = exp(-(x_i^2 + x_k^2)/(4 sigma_S^2) - (x_i - x_k)^2/(2 sigma_mu^2))
// (the same table serves both axes: y_j = -x_j) and the far-field factors, in FP64, once.
__global__ void gsm_gradient_tables(GradArgs g) {
  const int N = g.N, M = N / 2;
  const double d = g.d;
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < N * N; idx += gridDim.x * blockDim.x) {
    const int i = idx / N, k = idx - i * N;
    const double xi = (i - M) * d, xk = (k - M) * d;
    if (g.sigma_S > 0.0)
      g.gtab[idx] = (float)exp(-(xi * xi + xk * xk) / (4 * g.sigma_S * g.sigma_S) -
                               (xi - xk) * (xi - xk) / (2 * g.sigma_mu * g.sigma_mu));
    if (idx < N) {
      const double n2 = (double)(idx - M) * (idx - M);
      g.qtab[idx] = cis_turns(frac_turns(n2 * g.Kq));
    }
  }
}

// One CTA per row eta = (ea, eb) of R; R is Hermitian, so the column sums of the mask gradient
// equal the row sums and dL/da(eta) = 4 Re sum_xi2 conj(W0bar)(eta, xi2) A a(xi2) G(eta, xi2).
// The row is read as pairs of adjacent elements (16-byte loads, N even), two pairs in flight per
// thread, with the pair's (c, e) advanced incrementally; the row's three parameter sums go to
// g.part (reduced by gsm_gradient_reduce).  FF: far-field forward propagation.
template <bool FF>
__global__ void __launch_bounds__(256) gsm_gradient_kernel(GradArgs g) {
  extern __shared__ double gsm_sh[];
  const int N = g.N, M = N / 2;
  const int eta = blockIdx.x;
  const int ea = eta / N, eb = eta - ea * N;
  float* gx = reinterpret_cast<float*>(gsm_sh);  // G along the first axis for row ea
  float* gy = gx + N;                            // G along the second axis for row eb
  float2* qx = reinterpret_cast<float2*>(gy + N);  // far field: q(x_c) conj factors
  double* red = reinterpret_cast<double*>(qx + 2 * N);
  const double d = g.d;
  for (int i = threadIdx.x; i < N; i += blockDim.x) {
    gx[i] = g.gtab[ea * N + i];  // G along the first axis for row ea
    gy[i] = g.gtab[eb * N + i];  // G along the second axis for row eb (y_j = -x_j)
    if (FF) qx[i] = g.qtab[i];
  }
  __syncthreads();
  // conj(W0bar)(eta, xi2) = c R q(eta) q*(xi2) in the far field (q of both axes)
  float2 qe = make_float2(1.f, 0.f);
  if (FF) qe = cmul(qx[ea], qx[eb]);
  const float* amask = g.amask;
  const float ae = amask ? amask[eta] : 1.f;
  const float d2 = (float)(d * d);
  const float r2e = (float)((ea - M) * (ea - M) + (M - eb) * (M - eb));  // in units of d^2
  // per-thread partial sums in FP32 (each thread adds N^2 / blockDim terms), reduced in FP64
  float sS = 0.f, sM = 0.f, sA = 0.f;
  const float4* Rrow = reinterpret_cast<const float4*>(g.R + (size_t)eta * N * N);
  const int NP = N * N / 2, step = blockDim.x;
  auto term = [&](float2 r, int c, int e, float ax) {
    if (FF) r = cmul(r, cmul(qe, cconj(cmul(qx[c], qx[e]))));
    const float tG = r.x * ax * gx[c] * gy[e];  // dW0/dtheta is real: only Re(conj(W0bar)) enters
    const float r2x = (float)((c - M) * (c - M) + (M - e) * (M - e));
    const float dx2 = (float)((ea - c) * (ea - c) + (eb - e) * (eb - e));
    sS = fmaf(tG, r2e + r2x, sS);
    sM = fmaf(tG, dx2, sM);
    sA += tG;
  };
  // element x = 2 p of the pair: (c, e) = (x / N, x mod N), e even (N even)
  const int dc = (2 * step) / N, de = (2 * step) - dc * N;
  int c = (2 * threadIdx.x) / N, e = 2 * threadIdx.x - c * N;
#pragma unroll 2
  for (int p = threadIdx.x; p < NP; p += step) {
    const float4 rr = __ldg(Rrow + p);
    const int x = 2 * p;
    float2 am = make_float2(1.f, 1.f);
    if (amask) am = make_float2(__ldg(amask + x), __ldg(amask + x + 1));  // 4-byte alignment only
    term(make_float2(rr.x, rr.y), c, e, am.x);
    term(make_float2(rr.z, rr.w), c, e + 1, am.y);
    e += de;
    c += dc;
    if (e >= N) {
      e -= N;
      ++c;
    }
  }
  // the mask-gradient sum is A * sA; the others scale with w0 = A a(eta) a(xi2) G
  const float sa = sA;
  sS *= ae * d2;
  sM *= ae * d2;
  sA *= ae;
  // block reduction of the four sums
  double v[4] = {(double)sS, (double)sM, (double)sA, (double)sa};
  for (int k = 0; k < 4; ++k) {
    double x = v[k];
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    if ((threadIdx.x & 31) == 0) red[k * 8 + (threadIdx.x >> 5)] = x;
  }
  __syncthreads();
  if (threadIdx.x < 4) {
    double x = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) x += red[threadIdx.x * 8 + w];
    // sS, sM carry a(eta) a(xi2) G t (r^2 terms), sA carries a(eta) a(xi2) G t, sa carries a(xi2) G t
    if (threadIdx.x < 3) g.part[(size_t)eta * 3 + threadIdx.x] = x;
    if (threadIdx.x == 3 && g.gmask) g.gmask[eta] = (float)(4.0 * g.c * g.A * x);
  }
}

// g3 from the partial sums: one CTA, FP64, a fixed summation order (deterministic).
__global__ void __launch_bounds__(256) gsm_gradient_reduce(GradArgs g) {
  __shared__ double red[3][8];
  const int rows = g.rows;
  double v[3] = {0.0, 0.0, 0.0};
  for (int r = threadIdx.x; r < rows; r += blockDim.x)
    for (int k = 0; k < 3; ++k) v[k] += g.part[(size_t)r * 3 + k];
  for (int k = 0; k < 3; ++k) {
    double x = v[k];
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    if ((threadIdx.x & 31) == 0) red[k][threadIdx.x >> 5] = x;
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    double x = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) x += red[threadIdx.x][w];
    const double s3 = g.sigma_S * g.sigma_S * g.sigma_S, m3 = g.sigma_mu * g.sigma_mu * g.sigma_mu;
    const double scale = threadIdx.x == 0 ? g.A / s3 : (threadIdx.x == 1 ? 2.0 * g.A / m3 : 2.0);
    g.g3[threadIdx.x] = g.c * scale * x;
  }
}

// ---- the adjoint source of a loss on S and mu (reading R22), on the output plane -----------------
// Given the real gradients gS = dL/dS and gmu = dL/dRe mu + i dL/dIm mu of mu(P1, .), and S, mu of
// the output plane: with D(x) = sqrt(S(P1) S(x)), r(x) = Re(conj(gmu(x)) mu(x)) (0 where D = 0),
//   dL/dS(y) = gS(y) - r(y) / (2 S(y)) - [y = P1] sum_x r(x) / (2 S(P1)),
//   dL/dW_B* = (1/2) dL/dS(y) on the diagonal (y, y) and (1/2) gmu(x) / D(x) on the row (P1, x).
// The kernel writes the source of the adjoint propagation, the conjugate of that array: d(y) =
// (1/2) dL/dS(y) and cross(x) = conj((1/2) gmu(x) / D(x)), all but the sum over x at P1: each block leaves its
// share of the sum in part (FP64, a fixed order) and delta.cuh's tables take it in.
struct AdjPrepArgs {
  int N, iP, jP;
  const float* gS;     // N x N or nullptr
  const float2* gmu;   // N x N or nullptr
  const float* S;      // N x N (with gmu)
  const float2* mu;    // N x N (with gmu)
  float* d;            // out: N x N
  float2* cross;       // out: N x N
  double* part;        // out: one sum per block (with gmu)
};

__global__ void __launch_bounds__(1024) adjoint_prep_kernel(AdjPrepArgs a) {
  __shared__ double red[32];
  const int NN = a.N * a.N, xp = a.iP * a.N + a.jP;
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  double rs = 0.0;
  if (x < NN) {
    float dS = a.gS ? a.gS[x] : 0.f;
    float2 c = make_float2(0.f, 0.f);
    if (a.gmu) {
      const float sx = a.S[x], sp = a.S[xp];
      if (sp * sx > 0.f) {
        const float2 g = a.gmu[x], m = a.mu[x];
        const float r = g.x * m.x + g.y * m.y;
        rs = (double)r;
        if (sx > 0.f) dS -= r / (2.f * sx);
        const float inv = rsqrtf(sp * sx);
        c = make_float2(0.5f * g.x * inv, -0.5f * g.y * inv);
      }
    }
    a.d[x] = 0.5f * dS;
    a.cross[x] = c;
  }
  if (!a.gmu) return;
  for (int o = 16; o > 0; o >>= 1) rs += __shfl_down_sync(0xffffffffu, rs, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = rs;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
    a.part[blockIdx.x] = t;
  }
}

}  // namespace pw
