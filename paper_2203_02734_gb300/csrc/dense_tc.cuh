// dense_tc.cuh -- the dense axis contraction of dense.cuh on the tensor cores (tcgen05.mma,
// kind::f16, FP16 operands split in two, FP32 accumulators in tensor memory), N <= 256.
//
// C[k][j] = scale sum_n A(k, n) B[n][j] as a real GEMM D = X Q^T per tile of 128 columns j:
//   X (128 x 2Np): row = column j, (Re B[n][j], Im B[n][j]) at 2n, 2n + 1 (zero for n >= N);
//   Q (2Np x 2Np): Q(2k, 2n) = Re A, Q(2k, 2n+1) = -Im A, Q(2k+1, 2n) = Im A, Q(2k+1, 2n+1) = Re A;
//   D (128 x 2Np FP32, tensor memory lanes x columns): (Re C[k][j], Im C[k][j]) at 2k, 2k + 1;
// Np = N rounded up to 16.  Each operand is x = x1 + x2 with x1 = fp16(x), x2 = fp16(x - x1): 22 to 24
// bits of x, and D accumulates x1 q1 + x1 q2 + x2 q1 (the dropped x2 q2 is below 2^-23).  FP16 has no
// exponent to spare, so both operands are scaled by powers of two: Q by 2^10 (|A| = 1), X so that the
// largest component of the whole input array comes to [2^13, 2^14).  Values down to 2^-16 of the largest
// keep their 22 bits, smaller ones an absolute error of 2^-39 of it (a relative 2^-18 at 2^-20).  An output of
// a full set of contractions mixes every input with unit-modulus weights, so its FP32 rounding noise (2^-24 of
// the largest terms) covers that floor.  Every contraction leaves the largest component of its output for the
// next one (max_out / max_in); the first takes it from the source.  The tables of a GSM source are not such a
// full set: a and d of H(a, b', d) T(a, c', d) only meet the other point's mask in the product, which may
// leave nothing but lines where both tables are small.  So there every column (a, d) has a scale of its own.
// (With one scale for a table, an opaque disc of 32 pixels before a beam of sigma_S = 5 pixels, N = 90, cost 5e-3
// of W; now 1e-7.)
// Measured against FP64 (relative L2 of W): 1.7e-6 at N = 200 padded to 512, 2.9e-6 at N = 90, where BF16
// operands in three parts with six products gave 2.1e-6 and 5.4e-6: the error is that of the accumulation,
// which has half as many steps now.
//
// Up to Np = 128 a CTA computes all 2 Np output reals of its tile; above, two CTAs compute half of them
// each (both split the same inputs, the second from L2): an accumulator of at most 256 tensor-memory
// columns and 113 KB of shared memory let two CTAs share an SM, so that one's set-up and first
// loads (4100 cycles at N = 200) and epilogue (7000 by columns, 11000 by rows) overlap the other's chunks
// (2050 cycles each, 624 of them MMA).  One CTA of 512 converter threads with all 2 Np outputs splits every
// input once, but nothing covers its ends: 22.7 ms a propagation at N = 200 against 19.2.  K runs in chunks of 16 complex inputs (32 reals,
// two MMA K-steps), 6 MMAs (M 128, N = NOUT, K 16) each.  Q is split once per propagation by
// qsplit_kernel into a global buffer laid out half by half and chunk by chunk in the canonical K-major
// layout (no swizzle): per chunk, split s and K-step ks, core matrices [kb < 2][row group < NOUT / 8] of 8
// rows x 16 bytes, so one chunk is 128 NOUT contiguous bytes and arrives by bulk copies into one of BBUF
// chunk buffers.  The A tile (16 KB) of a chunk is built by the 256 converter threads in one of two
// tiles, from inputs that were loaded two chunks earlier (without that the converters waited for HBM
// in every chunk, which was the larger part of the 41 us a tile took at N = 200).
//
// Roles: eight warps split the operand chunks into A tiles and read the result back; one warp
// copies B and issues the MMAs (see axis_tc_kernel for the mbarrier hand-offs).
#pragma once
#include <cuda_fp16.h>
#include <cstdint>

#include "dense.cuh"
#include "tc16.cuh"

namespace pw {
namespace dense_tc {

constexpr int NT = 288;  // 8 converter warps + 1 issuer warp
constexpr int MAX_N = 256;

__host__ __device__ constexpr int npad(int N) { return (N + 15) / 16 * 16; }
// Output reals of one CTA, and CTAs per tile.
__host__ __device__ constexpr int parts(int N) { return npad(N) > 128 ? 2 : 1; }
__host__ __device__ constexpr int nout(int N) { return 2 * npad(N) / parts(N); }
__host__ __device__ constexpr size_t chunk_bytes(int N) { return (size_t)128 * nout(N); }
__host__ __device__ constexpr int nchunks(int N) { return npad(N) / 16; }
constexpr int ABUF = 2;
constexpr uint32_t A_BYTES = 2 * 2 * 4096;  // 2 splits x 2 K-steps x (128 rows x 16 fp16)
// B chunk buffers: three, so that a copy has two chunks' MMAs to land; two where only that lets two
// CTAs share an SM.
__host__ __device__ constexpr int b_buffers(int N) { return nout(N) > 208 ? 2 : 3; }
constexpr size_t EPI_BYTES = (size_t)8 * 32 * 33 * 8;  // per-warp transposes of the L = 1 epilogue
__host__ __device__ constexpr size_t operand_bytes(int N) {
  const size_t b = ABUF * A_BYTES + b_buffers(N) * chunk_bytes(N);
  return b > EPI_BYTES ? b : EPI_BYTES;
}
__host__ __device__ constexpr size_t smem_bytes(int N) { return operand_bytes(N) + 128; }
static_assert(2 * (smem_bytes(208) + 1024) <= 233472 && 2 * (smem_bytes(256) + 1024) <= 233472, "two CTAs per SM");
constexpr float QSCALE = 1024.f;  // scale of Q

// Exponent e of the input scale 2^e from the bits of the largest magnitude m: m 2^e in [2^13, 2^14); 0 where
// m is 0 or not finite (its column comes out as NaN, as it should), at most 126.
__device__ __forceinline__ int scale_exp(unsigned bits) {
  if (bits == 0u || bits >= 0x7f800000u) return 0;
  const int ex = (int)(bits >> 23) - 127;  // -127 for a denormal
  const int e = 13 - ex;
  return e > 126 ? 126 : e;
}
__device__ __forceinline__ float exp2_int(int e) {  // |e| <= 126
  return __uint_as_float((unsigned)(e + 127) << 23);
}
// Leaves the warp's largest magnitude in *out (bits of a non-negative float order as integers; a NaN
// does not count).
__device__ __forceinline__ void warp_max(unsigned* out, float m) {
  const unsigned b = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
  if ((threadIdx.x & 31) == 0 && b > *reinterpret_cast<volatile unsigned*>(out)) atomicMax(out, b);
}
// Tensor-memory columns to allocate: a power of two >= 32 holding D's NOUT columns.
__host__ __device__ constexpr uint32_t tmem_cols(int N) {
  return nout(N) <= 32 ? 32 : nout(N) <= 64 ? 64 : nout(N) <= 128 ? 128 : 256;
}

// Instruction descriptor: D FP32, A and B FP16, K-major, M = 128, N = n (a multiple of 16 <= 256).
__host__ __device__ constexpr uint32_t idesc(int n) {
  return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((128u >> 4) << 24);
}

// Split Q: element (row r < 2Np, K index kk < 32) of chunk c and split s goes to part r / NOUT, chunk c,
// block (s, ks = kk / 16), core matrix (kb = (kk mod 16) / 8, row group (r mod NOUT) / 8).
struct QArgs {
  int N;
  const float2* E;  // N x N, row k, column n
  int conj;         // A = conj(E)
  unsigned char* Q; // parts x nchunks x chunk_bytes
};
__host__ __device__ constexpr size_t q_bytes(int N) { return (size_t)parts(N) * nchunks(N) * chunk_bytes(N); }

__global__ void qsplit_kernel(QArgs a) {
  const int N = a.N, Np = npad(N), R = 2 * Np, NO = nout(N);
  const int total = nchunks(N) * R * 32;
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += gridDim.x * blockDim.x) {
    const int c = idx / (R * 32), rem = idx - c * R * 32, r = rem / 32, kk = rem - r * 32;
    const int k = r >> 1, cp = r & 1, n = c * 16 + (kk >> 1), cc = kk & 1;
    float v = 0.f;
    if (k < N && n < N) {
      float2 e = a.E[k * N + n];
      if (a.conj) e.y = -e.y;
      v = cp == 0 ? (cc == 0 ? e.x : -e.y) : (cc == 0 ? e.y : e.x);
    }
    v *= QSCALE;
    const __half s1 = __float2half_rn(v);
    const __half s2 = __float2half_rn(v - __half2float(s1));
    const int part = r / NO, rr = r - part * NO, ks = kk >> 4, kb = (kk >> 3) & 1, e8 = kk & 7;
    const size_t block = (size_t)32 * NO;  // bytes of one (split, K-step) block
    const size_t off = (size_t)(part * nchunks(N) + c) * chunk_bytes(N) + (size_t)ks * block +
                       (size_t)((kb * (NO / 8) + (rr >> 3)) * 128 + (rr & 7) * 16 + e8 * 2);
    *reinterpret_cast<__half*>(a.Q + off) = s1;
    *reinterpret_cast<__half*>(a.Q + off + 2 * block) = s2;
  }
}

// ---- the tables of a GSM source ----------------------------------------------------------------
// As in plane.cuh, b and c of the GSM source contract into tables of N^3 values,
//   H[a][b'][d] = sum_b conj E(b', b) A conj M0(a, b) G(b, d),  T[a][c'][d] = sum_c E(c', c) M0(c, d) G(a, c),
// themselves contractions of N^2 columns on axis_tc_kernel, and only d and a are left for the N^4 array
// H[a][b'][d] T[a][c'][d]: two contractions of N^3 columns instead of four.
struct TableArgs {
  int N;
  const float* G;
  const float2* M0;
  float A;
  float2 *H0, *T0;     // N^3 each: [a][b][d], [a][c][d]
  unsigned* max;       // 2 x N x N: largest component of each column (a, d) of H0, then of T0
};
constexpr int TS_D = 32, TS_B = 8;  // a block: 32 columns d of one a, of H0 (blockIdx.z = 0) or T0, in 8 shares of b or c
__global__ void __launch_bounds__(TS_D * TS_B) table_source_kernel(TableArgs p) {
  __shared__ float share[TS_B][TS_D];
  const int N = p.N, tx = threadIdx.x % TS_D, ty = threadIdx.x / TS_D, d = blockIdx.x * TS_D + tx, a = blockIdx.y;
  const bool h = blockIdx.z == 0;
  const size_t col = (size_t)a * N * N + d;
  float m = 0.f;
  if (d < N)
    for (int b = ty; b < N; b += TS_B) {
      const int ab = a * N + b, bd = b * N + d;
      const float2 v = h ? cscale(cconj(__ldg(p.M0 + ab)), p.A * __ldg(p.G + bd)) : cscale(__ldg(p.M0 + bd), __ldg(p.G + ab));
      (h ? p.H0 : p.T0)[col + (size_t)b * N] = v;
      m = fmaxf(m, fmaxf(fabsf(v.x), fabsf(v.y)));
    }
  share[ty][tx] = m;
  __syncthreads();
  if (ty != 0 || d >= N) return;
  for (int k = 1; k < TS_B; ++k) m = fmaxf(m, share[k][tx]);
  p.max[((h ? 0 : N) + a) * N + d] = __float_as_uint(m);
}
// Largest |H T| over the N^4 array: for each (a, d) the largest |H| over b' times the largest |T| over c'.
__global__ void __launch_bounds__(256) table_max_kernel(int N, const float2* __restrict__ H, const float2* __restrict__ T,
                                                        unsigned* max) {
  float m = 0.f;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < N * N) {
    const int a = i / N, d = i - a * N;
    const size_t base = (size_t)a * N * N + d;
    float h = 0.f, t = 0.f;
#pragma unroll 4
    for (int b = 0; b < N; ++b) {
      const float2 x = __ldg(H + base + (size_t)b * N), y = __ldg(T + base + (size_t)b * N);
      h = fmaxf(h, hypotf(x.x, x.y));
      t = fmaxf(t, hypotf(y.x, y.y));
    }
    m = h * t;
  }
  warp_max(max, m);
}

// Largest component of conj(M0(a, b)) W0(a, b, c, d) M0(c, d) over an uploaded or propagated array.
__global__ void __launch_bounds__(256) masked_max_kernel(int N, const float2* __restrict__ W0, const float2* __restrict__ M0,
                                                         unsigned* max) {
  const int NN = N * N;
  float m = 0.f;
  for (int ab = blockIdx.x; ab < NN; ab += gridDim.x) {
    const float2 m1 = cconj(__ldg(M0 + ab));
    const float2* w = W0 + (size_t)ab * NN;
#pragma unroll 4
    for (int cd = threadIdx.x; cd < NN; cd += 256) {
      const float2 v = cmul(cmul(m1, __ldg(w + cd)), __ldg(M0 + cd));
      m = fmaxf(m, fmaxf(fabsf(v.x), fabsf(v.y)));
    }
  }
  warp_max(max, m);
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* mbar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(mbar)), "r"(bytes) : "memory");
}

__device__ __forceinline__ void mma_np(uint32_t d, uint64_t a, uint64_t b, uint32_t id, uint32_t acc) {
  asm volatile("{.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
               "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;}" ::"r"(d),
               "l"(a), "l"(b), "r"(id), "r"(acc));
}

__device__ __forceinline__ void tmem_ld16(float* r, uint32_t taddr) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]), "=f"(r[7]), "=f"(r[8]),
        "=f"(r[9]), "=f"(r[10]), "=f"(r[11]), "=f"(r[12]), "=f"(r[13]), "=f"(r[14]), "=f"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_ld32(float (&r)[32], uint32_t taddr) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]), "=f"(r[7]), "=f"(r[8]),
        "=f"(r[9]), "=f"(r[10]), "=f"(r[11]), "=f"(r[12]), "=f"(r[13]), "=f"(r[14]), "=f"(r[15]), "=f"(r[16]),
        "=f"(r[17]), "=f"(r[18]), "=f"(r[19]), "=f"(r[20]), "=f"(r[21]), "=f"(r[22]), "=f"(r[23]), "=f"(r[24]),
        "=f"(r[25]), "=f"(r[26]), "=f"(r[27]), "=f"(r[28]), "=f"(r[29]), "=f"(r[30]), "=f"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// The inputs of a contraction: columns that are contiguous across j (L > 1), or along n (L = 1): an
// array, a masked array, or the product of the GSM tables.
enum Mode { IN_COLS = 0, IN_ROWS = 1, IN_MASK = 2, IN_PRODUCT = 3 };

struct Args {
  int N;
  long long L;      // elements after the contracted axis
  long long ncols;  // columns
  const float2* in; // all but IN_PRODUCT
  float2* out;
  float scale;
  float* S;         // last pass: S(a', b') = Re C at k = a', j = (b', a', b'); else nullptr
  int vec;          // L = 1: `in` is 16-byte aligned
  const float2* M0; // IN_MASK
  const float2 *H, *T;       // IN_PRODUCT (j = (a, b', c'))
  const unsigned* max_in;    // bits of the largest input component
  const unsigned* max_col;   // IN_COLS: the same of each column j, in place of max_in; or nullptr
  unsigned* max_out;         // the same of the output, or nullptr
  int stall;  // failure-detection test (0 = off): CTA 0 never copies operand chunk `stall` (> 0), or never
              // announces A tile -stall (< 0)
};

// One tile of 128 columns j and one part of its outputs per CTA (grid = parts x ceil(ncols / 128)), NT = 288
// threads: warps 0-7 split the operand and read the result back, warp 8 (one lane) copies B and issues
// the MMAs.  No block-wide barrier inside the chunk loop: the roles
// hand off through mbarriers -- afull[b] (8 warp arrivals: A tile b is written), bfull[b] (bytes
// of B buffer b have landed), mdone[b] (tcgen05.commit: the MMAs of the last chunk with parity b
// have completed, so its A tile and B buffer are free).  A tile c mod 2 and B buffer c mod BBUF hold
// chunk c; no barrier can run two phases ahead of a wait on it (each next fill depends
// on the completion being waited for).  Every wait is bounded; a wait that gives up sets the
// shared abort flag and *err, after which no role waits again, and the tile's outputs are not
// written.  Inputs: with L > 1 thread t owns column t mod 128 and the 8 n of K-step t / 128 (a warp reads
// 256 contiguous bytes); with L = 1 eight lanes share a column's 16 n (128 contiguous bytes) and a
// thread has four columns (one column per lane costs 32 L1 wavefronts a load there, eight times as many).
// Epilogue: with L > 1 a warp's 32 lanes are consecutive in memory (256-byte stores); with
// L = 1 a lane's k are, so each warp turns 32 columns x 32 outputs through shared memory (the
// operand buffers are free by then) and stores rows of 256 bytes.
// At most 112 registers, so that two CTAs share an SM.
template <int BBUF, int MODE>
__global__ void __launch_bounds__(NT, 2) axis_tc_kernel(Args p, const unsigned char* __restrict__ Q, int* err) {
  extern __shared__ __align__(1024) unsigned char sm[];
  constexpr bool ROWS = MODE != IN_COLS;
  const int N = p.N, NO = nout(N), nch = nchunks(N);
  const int part = parts(N) == 2 ? blockIdx.x & 1 : 0;
  const unsigned tile = parts(N) == 2 ? blockIdx.x >> 1 : blockIdx.x;
  const uint32_t cb = (uint32_t)chunk_bytes(N);
  unsigned char* As0 = sm;
  unsigned char* Bs0 = sm + ABUF * A_BYTES;
  uint64_t* bfull = reinterpret_cast<uint64_t*>(sm + operand_bytes(N));  // [3]
  uint64_t* mdone = bfull + 3;                                           // [2]
  uint64_t* afull = bfull + 5;                                           // [2]
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bfull + 7);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tslot + 1);
  volatile int* committed = abort_flag + 1;  // the last chunk whose MMAs the issuer committed
  // Issuer lane only: chunks whose B copies were started (bit c) and whose bfull wait completed
  // (bit c); on an abort, copies still in flight are drained before the CTA exits.
  uint32_t b_issued = 0, b_landed = 0;
  const int t = threadIdx.x, w = t >> 5, lane = t & 31;
  const long long L = p.L;
  // 32-bit column arithmetic: j < N^3 <= 2^24 and L <= N^3
  const unsigned ncols = (unsigned)p.ncols, Lu = (unsigned)L;
  int sexp = 0;  // exponent of the input scale; per column, thread t's being that of its epilogue too

  // the converter's inputs: eight values of a chunk, loaded two chunks ahead (three sets in turn).
  // ROWS: n = 16 c + 2 (t mod 8) + {0, 1} of the columns tile * 128 + t / 8 + 32 i, i < 4.
  const int m = t & 127, ks = (t >> 7) & 1, l8 = t & 7;
  const float2* src = nullptr;  // row of the first column (T itself for IN_PRODUCT)
  unsigned st[4], sf[4];        // offsets of the four columns' rows from src, and from their factors' array
  float2 gcol[MODE == IN_MASK ? 4 : 1];
  bool live[ROWS ? 4 : 1];
  if constexpr (ROWS) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const unsigned j = tile * 128 + (t >> 3) + 32 * i;
      live[i] = t < 256 && j < ncols;
      const unsigned jj = live[i] ? j : 0u;
      const int c = (int)(jj % N), b = (int)(jj / N % N), a = (int)(jj / (N * N));
      if constexpr (MODE == IN_PRODUCT) {
        st[i] = (a * N + c) * N + 2 * l8;
        sf[i] = (a * N + b) * N + 2 * l8;
      } else {
        st[i] = 32 * i * N;
        sf[i] = c * N + 2 * l8;
        if constexpr (MODE == IN_MASK) gcol[i] = cconj(__ldg(p.M0 + a * N + b));
      }
    }
    src = MODE == IN_PRODUCT ? p.T : p.in + (size_t)(tile * 128 + (t >> 3)) * N + 2 * l8;
    sexp = scale_exp(*p.max_in);
  } else {
    const unsigned j = tile * 128 + m;
    live[0] = t < 256 && j < ncols;
    const unsigned jj = live[0] ? j : 0u;
    src = p.in + (size_t)(jj / Lu) * L * N + jj % Lu;
    sexp = scale_exp(p.max_col ? p.max_col[jj] : *p.max_in);
  }
  auto load = [&](int c, float2 (&x)[8]) {
    if constexpr (ROWS) {
      const int n0 = 16 * c + 2 * l8;  // N is even: both values or none
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const bool ok = live[i] && n0 < N;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (MODE == IN_PRODUCT || p.vec) {
          if (ok) v = *reinterpret_cast<const float4*>(src + st[i] + 16 * c);
        } else if (ok) {
          const float2 u0 = src[st[i] + 16 * c], u1 = src[st[i] + 16 * c + 1];
          v = make_float4(u0.x, u0.y, u1.x, u1.y);
        }
        x[2 * i] = make_float2(v.x, v.y);
        x[2 * i + 1] = make_float2(v.z, v.w);
      }
    } else {
      const int n0 = 16 * c + 8 * ks;
#pragma unroll
      for (int i = 0; i < 8; ++i) x[i] = live[0] && n0 + i < N ? src[(long long)(n0 + i) * L] : make_float2(0.f, 0.f);
    }
  };
  float2 x0[8], x1[8], x2[8];
  if (w < 8) {  // before the set-up below, to hide it
    load(0, x0);
    load(1, x1);  // past the last chunk: zeros, nothing is read
  }

  if (w == 8) tc16::tmem_alloc(tslot, tmem_cols(N));
  if (t == 0) {
    for (int b = 0; b < BBUF; ++b) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&bfull[b])));
    for (int b = 0; b < 2; ++b) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&mdone[b])));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 8;" ::"r"(smem_u32(&afull[b])));
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    *abort_flag = 0;
    *committed = -1;
  }
  tc16::fence_before_sync();
  __syncthreads();
  tc16::fence_after_sync();
  const uint32_t tmem = *tslot;
  auto fail_now = [&]() {
    *abort_flag = 1;
    atomicExch(err, 1);
  };
  // bounded wait that also gives up at once when another role has aborted
  auto wait = [&](uint64_t* bar, uint32_t parity) -> bool {
    if (*abort_flag) return false;
    if (tc16::mbar_wait(bar, parity)) return true;
    fail_now();
    return false;
  };

  if (w == 8) {
    // ---- the issuer: B copies and MMAs, one lane
    if (lane == 0) {
      const uint32_t id = idesc(NO);
      Q += (size_t)part * nch * cb;
      auto load_chunk = [&](int c) {
        if (p.stall > 0 && c == p.stall && blockIdx.x == 0) return;  // injected: this phase never completes
        b_issued |= 1u << c;
        unsigned char* dst = Bs0 + (c % BBUF) * cb;
        const unsigned char* src = Q + (size_t)c * cb;
        mbar_expect_tx(&bfull[c % BBUF], cb);
        const uint32_t piece = cb / 4;  // 32 NOUT bytes, a multiple of 16
        for (int q = 0; q < 4; ++q) bulk_g2s(dst + q * piece, src + (size_t)q * piece, piece, &bfull[c % BBUF]);
      };
      for (int c = 0; c < BBUF && c < nch; ++c) load_chunk(c);
      constexpr int ti[3] = {0, 0, 1}, tj[3] = {0, 1, 0};
      const uint32_t blk = (uint32_t)(32 * NO);
      for (int c = 0; c < nch; ++c) {
        if (!wait(&afull[c & 1], (uint32_t)((c >> 1) & 1))) break;
        if (!wait(&bfull[c % BBUF], (uint32_t)((c / BBUF) & 1))) break;
        b_landed |= 1u << c;
        tc16::fence_after_sync();
        const uint64_t a0 = tc16::sdesc(smem_u32(As0 + (c & 1) * A_BYTES), 2048, 128);
        const uint64_t b0 = tc16::sdesc(smem_u32(Bs0 + (c % BBUF) * cb), (uint32_t)(16 * NO), 128);
#pragma unroll
        for (int q = 0; q < 3; ++q)
#pragma unroll
          for (int s2 = 0; s2 < 2; ++s2) {
            const uint64_t ad = a0 + (uint64_t)((ti[q] * 8192 + s2 * 4096) >> 4);
            const uint64_t bd = b0 + (uint64_t)(((tj[q] * 2 + s2) * blk) >> 4);
            mma_np(tmem, ad, bd, id, (c | q | s2) ? 1u : 0u);
          }
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                         smem_u32(&mdone[c & 1]))
                     : "memory");
        *committed = c;
        // the buffer of chunk c - 1 takes chunk c - 1 + BBUF once those MMAs are done
        if (c >= 1 && c - 1 + BBUF < nch) {
          if (!wait(&mdone[(c - 1) & 1], (uint32_t)(((c - 1) >> 1) & 1))) break;
          load_chunk(c - 1 + BBUF);
        }
      }
    }
  } else {
    // ---- the converters: split the operand chunk by chunk, then read the result back
    const float sx = exp2_int(sexp);
    auto split = [&](float2 v, uint32_t& h, uint32_t& l) {
      v = cscale(v, sx);
      const __half2 h1 = __floats2half2_rn(v.x, v.y);
      const float2 r1 = __half22float2(h1);
      const __half2 h2 = __floats2half2_rn(v.x - r1.x, v.y - r1.y);
      h = *reinterpret_cast<const uint32_t*>(&h1);
      l = *reinterpret_cast<const uint32_t*>(&h2);
    };
    auto convert = [&](int c, const float2 (&x)[8]) -> bool {
      // the factors of a row: shared by the columns of one (a, b') (H) or c (M0), from L1
      float4 f[4];
      if constexpr (MODE == IN_MASK || MODE == IN_PRODUCT) {
        const float2* fac = MODE == IN_MASK ? p.M0 : p.H;
#pragma unroll
        for (int i = 0; i < 4; ++i)
          f[i] = live[i] && 16 * c + 2 * l8 < N ? __ldg(reinterpret_cast<const float4*>(fac + sf[i] + 16 * c))
                                               : make_float4(0.f, 0.f, 0.f, 0.f);
      }
      // the split values first (hi, lo words of the thread's 16 reals), so that only the stores wait for
      // the tile
      uint32_t hi[8], lo[8];
      if constexpr (ROWS) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          float2 v0 = x[2 * i], v1 = x[2 * i + 1];
          if constexpr (MODE == IN_MASK) {
            v0 = cmul(gcol[i], v0);
            v1 = cmul(gcol[i], v1);
          }
          if constexpr (MODE != IN_ROWS) {
            v0 = cmul(v0, make_float2(f[i].x, f[i].y));
            v1 = cmul(v1, make_float2(f[i].z, f[i].w));
          }
          split(v0, hi[2 * i], lo[2 * i]);
          split(v1, hi[2 * i + 1], lo[2 * i + 1]);
        }
      } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) split(x[i], hi[i], lo[i]);
      }
      if (c >= ABUF) {  // A tile c mod 2 last held chunk c - 2
        const int pc = c - ABUF;
        bool ok = true;
        if (lane == 0) ok = wait(&mdone[pc & 1], (uint32_t)((pc >> 1) & 1));
        ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
        if (!ok) return false;
      }
      unsigned char* As = As0 + (c & 1) * A_BYTES;
      if constexpr (ROWS) {
        // reals 4 l8 .. 4 l8 + 3 of the chunk: K-step l8 / 4, core matrix (l8 / 2) mod 2, half l8 mod 2 of its row
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int col = (t >> 3) + 32 * i;
          unsigned char* dst = As + (l8 >> 2) * 4096 + (((l8 >> 1) & 1) * 16 + (col >> 3)) * 128 + (col & 7) * 16 + (l8 & 1) * 8;
          *reinterpret_cast<uint2*>(dst) = make_uint2(hi[2 * i], hi[2 * i + 1]);
          *reinterpret_cast<uint2*>(dst + 8192) = make_uint2(lo[2 * i], lo[2 * i + 1]);
        }
      } else {
        unsigned char* dst = As + ks * 4096 + (m >> 3) * 128 + (m & 7) * 16;
#pragma unroll
        for (int kb = 0; kb < 2; ++kb) {
          *reinterpret_cast<uint4*>(dst + kb * 2048) = make_uint4(hi[4 * kb], hi[4 * kb + 1], hi[4 * kb + 2], hi[4 * kb + 3]);
          *reinterpret_cast<uint4*>(dst + 8192 + kb * 2048) = make_uint4(lo[4 * kb], lo[4 * kb + 1], lo[4 * kb + 2], lo[4 * kb + 3]);
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      // injected (p.stall < 0): CTA 0 never announces A tile -p.stall, so the issuer's wait gives up
      // while the B copy of that chunk may still be in flight
      const bool skip = p.stall < 0 && c == -p.stall && blockIdx.x == 0;
      if (lane == 0 && !skip)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&afull[c & 1])) : "memory");
      return true;
    };
    // inputs are loaded two chunks ahead (three sets of registers, in turn)
    for (int c = 0; c < nch; c += 3) {
      load(c + 2, x2);
      if (!convert(c, x0)) break;
      if (c + 1 >= nch) break;
      load(c + 3, x0);
      if (!convert(c + 1, x1)) break;
      if (c + 2 >= nch) break;
      load(c + 4, x1);
      if (!convert(c + 2, x2)) break;
    }
    // the last chunk's MMAs complete after all earlier ones
    bool ok = true;
    if (lane == 0) ok = wait(&mdone[(nch - 1) & 1], (uint32_t)(((nch - 1) >> 1) & 1));
    ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
    tc16::fence_after_sync();
    if (ok && !*abort_flag) {
      // warp w reads lanes 32 (w mod 4) .. + 31 (columns j) of every second group of outputs (w / 4)
      const int h = w >> 2, kp = part * NO / 2;  // first output of the part
      const uint32_t tw = tmem + ((uint32_t)(32 * (w & 3)) << 16);
      const float s1 = p.scale / QSCALE, s2 = exp2_int(-sexp);
      const unsigned row0 = tile * 128 + 32 * (w & 3), j = row0 + lane;
      const bool in_range = j < ncols;
      float mx = 0.f;
      if constexpr (ROWS) {
        float2* turn = reinterpret_cast<float2*>(sm) + w * 32 * 33;
        for (int k0 = 32 * h; k0 < NO / 2; k0 += 64) {
          const int cnt = min(32, NO / 2 - k0);  // a multiple of 8
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            if (16 * q < cnt) {
              float r[32];
              const int n16 = min(16, cnt - 16 * q);
              if (n16 == 16) tmem_ld32(r, tw + (uint32_t)(2 * k0 + 32 * q));
              else tmem_ld16(r, tw + (uint32_t)(2 * k0 + 32 * q));
#pragma unroll
              for (int i = 0; i < 16; ++i) {
                if (i < n16) {
                  const float2 v = make_float2(r[2 * i] * s1 * s2, r[2 * i + 1] * s1 * s2);
                  if (in_range && kp + k0 + 16 * q + i < N) mx = fmaxf(mx, fmaxf(fabsf(v.x), fabsf(v.y)));
                  turn[lane * 33 + 16 * q + i] = v;
                }
              }
            }
          }
          __syncwarp();
          const int k = kp + k0 + lane;
          if (lane < cnt && k < N) {
            const int rows = row0 < ncols ? min(32u, ncols - row0) : 0;
            float2* o = p.out + (size_t)row0 * N + k;
            int r = 0;
            for (; r + 8 <= rows; r += 8, o += 8 * N) {  // eight loads, then eight stores: one by one 14800 cycles a CTA
              float2 v[8];
#pragma unroll
              for (int i = 0; i < 8; ++i) v[i] = turn[(r + i) * 33 + lane];
#pragma unroll
              for (int i = 0; i < 8; ++i) o[i * N] = v[i];
            }
            for (; r < rows; ++r, o += N) *o = turn[r * 33 + lane];
          }
          __syncwarp();
        }
      } else {
        const unsigned jj = in_range ? j : 0u;
        float2* out = p.out + (size_t)(jj / Lu) * L * N + jj % Lu;
        // S: the column (b', a', d') with d' = b' holds S(a', b') at k = a'
        const int sb = (int)(jj / (N * N)), sk = p.S && in_range && (int)(jj % N) == sb ? (int)(jj / N % N) : -1;
        for (int q = h; q < (NO + 31) / 32; q += 2) {  // 32 columns (16 complex outputs) per load, or a last 16
          float r[32];
          const int n16 = 32 * q + 32 <= NO ? 16 : 8;
          if (n16 == 16) tmem_ld32(r, tw + (uint32_t)(32 * q));
          else tmem_ld16(r, tw + (uint32_t)(32 * q));
          const int k0 = kp + 16 * q;
          float2* o = out + (long long)k0 * L;
#pragma unroll
          for (int i = 0; i < 16; ++i, o += L) {
            if (in_range && i < n16 && k0 + i < N) {
              const float2 v = make_float2(r[2 * i] * s1 * s2, r[2 * i + 1] * s1 * s2);
              mx = fmaxf(mx, fmaxf(fabsf(v.x), fabsf(v.y)));
              *o = v;
              if (k0 + i == sk) p.S[sk * N + sb] = v.x;
            }
          }
        }
      }
      if (p.max_out) warp_max(p.max_out, mx);
    }
  }
  tc16::fence_before_sync();
  __syncthreads();
  if (w == 8 && lane == 0 && *abort_flag) {
    // no MMA may still write tensor memory when it is freed: the last commit covers all (bounded)
    if (*committed >= 0) {
      const int lc = *committed;
      tc16::mbar_wait(&mdone[lc & 1], (uint32_t)((lc >> 1) & 1));
    }
    // no bulk copy may still write shared memory when the CTA exits: wait (bounded) for every B
    // copy that was started and not yet seen complete; at most one is outstanding per buffer
    for (int c = 0; c < nch; ++c)
      if ((b_issued >> c) & 1u && !((b_landed >> c) & 1u)) tc16::mbar_wait(&bfull[c % BBUF], (uint32_t)((c / BBUF) & 1));
  }
  __syncthreads();
  tc16::fence_after_sync();
  if (w == 8) tc16::tmem_dealloc(tmem, tmem_cols(N));
}

}  // namespace dense_tc
}  // namespace pw
