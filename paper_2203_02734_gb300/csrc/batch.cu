// batch.cu -- C ABI of the batched run (pw_batch_*): instance descriptors, workspace layout,
// item list, launch sequence and the chunk-size autotuner.  Instances that keep no W run on smu.cuh
// (S and mu without the CSDA); the others on the plane kernels one after the other, or in the
// persistent launch.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdint>
#include <cstdio>
#include <vector>

#include "../../include/pywolf_gb.h"
#include "batch.cuh"
#include "internal.h"
#include "smu.cuh"

namespace {

pw_status fail(pw_status s, const char* fmt, ...) {
  char msg[320];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(msg, sizeof msg, fmt, ap);
  va_end(ap);
  pwi::set_last_error(msg);
  return s;
}

pw_status cuda_fail(cudaError_t e, const char* what) {
  cudaGetLastError();
  return fail(PW_ECUDA, "%s: %s", what, cudaGetErrorString(e));
}

bool finite_pos(double v) { return std::isfinite(v) && v > 0.0; }

bool batch_n(int N) { return N == 16 || N == 32 || N == 64 || N == 96 || N == 128; }

bool aligned(const void* p, size_t a) { return reinterpret_cast<uintptr_t>(p) % a == 0; }

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// Workspace layout (offsets from the base, each part 256-byte aligned).
struct Layout {
  size_t inst, targs, mu, items, counters, tmaps, wts, tables, pool, total;
  int max_items;
  size_t slot_bytes;
};

constexpr int kMinChunk = 4;

Layout layout(const pw_instance* in, int n, int pool) {
  Layout L{};
  size_t off = 0;
  L.inst = off;
  off = align256(off + sizeof(pw::batch::Inst) * n);
  L.targs = off;
  off = align256(off + sizeof(pw::TableArgs) * n);
  L.mu = off;
  off = align256(off + sizeof(float2*) * n);
  long items = 0;
  int maxN = 0;
  for (int i = 0; i < n; ++i) {
    const long s = (long)in[i].N * in[i].N;
    items += 2 * ((s + kMinChunk - 1) / kMinChunk);
    if (in[i].N > maxN) maxN = in[i].N;
  }
  L.max_items = (int)items;
  L.items = off;
  off = align256(off + sizeof(pw::batch::Item) * items);
  L.counters = off;
  off = align256(off + sizeof(int) * (2 * (size_t)n + 2));
  L.tmaps = off;  // one tensor map per pool slot (N = 128 instances store V by TMA)
  off = align256(off + sizeof(CUtensorMap) * pool);
  L.wts = off;    // per-instance weights of pw_batch_spectral_sum
  off = align256(off + sizeof(double) * n);
  L.tables = off;
  for (int i = 0; i < n; ++i) {
    const size_t N = in[i].N, NN = N * N;
    off = align256(off + NN * sizeof(float2));  // F
    off = align256(off + NN * sizeof(float));   // G
    off = align256(off + N * sizeof(float2));   // twiddles
    off = align256(off + N * sizeof(float2));   // output propagators
    off = align256(off + N * sizeof(float2));   // per-axis input factors
    off = align256(off + NN * sizeof(float2));  // W(P1, .)
  }
  L.pool = off;
  L.slot_bytes = align256((size_t)maxN * maxN * maxN * maxN * sizeof(float2));
  off += L.slot_bytes * pool;
  L.total = off;
  return L;
}

}  // namespace

struct pw_batch {
  int n, pool, chunk;
  int mode;  // PW_BATCH_PERSISTENT or PW_BATCH_SEQUENCED
  std::vector<CUtensorMap> wmaps;  // per instance with W: its planes (plane.cuh)
  std::vector<pw::TableArgs> targs;   // FP64 tables, uploaded with N = 0 for the instances on smu.cuh
  std::vector<pw::smu::Inst<pwi::Wide>> smu;     // the instances on smu.cuh, by pw_instance index where direct
  std::vector<pw::smu::TabArgs<pwi::Wide>> smu_t;
  std::vector<float2*> mus;           // dev_mu of every instance
  struct Round {                      // one launch round of the instances on smu.cuh
    int chunk;
    bool mu;
    std::vector<int> Ns;
  };
  std::vector<Round> rounds;
  int ndirect;                        // instances on smu.cuh
  const pw::smu::Inst<pwi::Wide>* dev_smu;
  const pw::smu::TabArgs<pwi::Wide>* dev_smu_t;
  char* base;
  Layout L;
  cudaStream_t stream;
  std::vector<pw::batch::Inst> inst;
  std::vector<int> stalled;  // instances whose pass-A items are left out (failure-detection test)
  std::vector<double> A, scale;  // amplitude and scale of every instance
  std::vector<double> dx_out;  // output sampling of every instance (lambda z / (N dxi))
  int nitems;
  long long wait_cycles;
};

namespace {

// Instances that keep no W need no half-transformed array and run on smu.cuh, in either mode (192
// instances of N = 64 to 128: 87 ms on the half-transformed arrays).  With a stall injected the whole list
// stays in the persistent launch, whose waits are under test.
bool stalled(const pw_batch* b) { return std::find(b->stalled.begin(), b->stalled.end(), 1) != b->stalled.end(); }
bool direct(const pw_batch* b, int i) {
  return b->inst[i].W == nullptr && !(b->mode == PW_BATCH_PERSISTENT && stalled(b));
}

// The instances in the launch.
std::vector<int> members(const pw_batch* b) {
  std::vector<int> m;
  for (int i = 0; i < b->n; ++i)
    if (!direct(b, i)) m.push_back(i);
  return m;
}

pw_status build_items(pw_batch* b) {
  std::vector<int> Ns;
  for (const auto& d : b->inst) Ns.push_back(d.N);
  const std::vector<pw::batch::Item> items = pw::batch::items(members(b), Ns, b->stalled, b->chunk, b->pool);
  if ((int)items.size() > b->L.max_items) return fail(PW_EINVAL, "item list exceeds the workspace");
  b->nitems = (int)items.size();
  cudaError_t e = cudaMemcpyAsync(b->base + b->L.items, items.data(), items.size() * sizeof(pw::batch::Item),
                                  cudaMemcpyHostToDevice, b->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
  if (e != cudaSuccess) return cuda_fail(e, "uploading the item list");
  return PW_OK;
}

// Uploads what depends on which instances run on smu.cuh: the FP64 table arguments, the slots and mu outputs
// of the others, the smu.cuh descriptors, and the item list.  The descriptors sit at the end of the
// item area, in the room of the items that these instances do not have (2560 bytes each at least);
// their scratch is the V pool, in as many rounds as it takes.
pw_status upload(pw_batch* b) {
  const int n = b->n;
  const size_t pool_bytes = b->L.slot_bytes * b->pool;
  std::vector<pw::TableArgs> targs(b->targs);
  std::vector<float2*> mus(b->mus);
  std::vector<pw::smu::Inst<pwi::Wide>> list;
  std::vector<pw::smu::TabArgs<pwi::Wide>> tabs;
  b->rounds.clear();
  size_t used = 0;
  int chunk = 0;
  for (int i = 0; i < n; ++i) {
    if (!direct(b, i)) continue;
    targs[i].N = 0;
    mus[i] = nullptr;
    pw::smu::Inst<pwi::Wide> q = b->smu[i];
    const size_t need = align256((size_t)6 * q.N * q.N * sizeof(pwi::Wide));
    if (used + need > pool_bytes) {
      ++chunk;
      used = 0;
    }
    if (b->rounds.empty() || b->rounds.back().chunk != chunk) b->rounds.push_back({chunk, false, {}});
    auto& r = b->rounds.back();
    r.mu = r.mu || q.mu;
    if (std::find(r.Ns.begin(), r.Ns.end(), q.N) == r.Ns.end()) r.Ns.push_back(q.N);
    q.chunk = chunk;
    q.scratch = reinterpret_cast<pwi::Wide*>(b->base + b->L.pool + used);
    used += need;
    list.push_back(q);
    tabs.push_back(b->smu_t[i]);
  }
  b->ndirect = (int)list.size();
  const size_t lb = align256(list.size() * sizeof(pw::smu::Inst<pwi::Wide>)), tb = align256(tabs.size() * sizeof(pw::smu::TabArgs<pwi::Wide>));
  char* tail = b->base + (b->L.items + sizeof(pw::batch::Item) * (size_t)b->L.max_items) / 256 * 256 - lb - tb;
  b->dev_smu = reinterpret_cast<pw::smu::Inst<pwi::Wide>*>(tail);
  b->dev_smu_t = reinterpret_cast<pw::smu::TabArgs<pwi::Wide>*>(tail + lb);
  const std::vector<pw::batch::Place> at = pw::batch::places(members(b), n, b->pool);
  for (int i = 0; i < n; ++i) {
    pw::batch::Inst& d = b->inst[i];
    d.prev = at[i].prev;
    d.V = reinterpret_cast<float2*>(b->base + b->L.pool + b->L.slot_bytes * at[i].slot);
    d.vmap = d.N == 128 ? b->base + b->L.tmaps + sizeof(CUtensorMap) * at[i].slot : nullptr;
  }
  cudaError_t e = cudaMemcpyAsync(b->base + b->L.inst, b->inst.data(), sizeof(pw::batch::Inst) * n, cudaMemcpyHostToDevice,
                                  b->stream);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(b->base + b->L.targs, targs.data(), sizeof(pw::TableArgs) * n, cudaMemcpyHostToDevice, b->stream);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(b->base + b->L.mu, mus.data(), sizeof(float2*) * n, cudaMemcpyHostToDevice, b->stream);
  if (e == cudaSuccess && b->ndirect)
    e = cudaMemcpyAsync(tail, list.data(), list.size() * sizeof(pw::smu::Inst<pwi::Wide>), cudaMemcpyHostToDevice, b->stream);
  if (e == cudaSuccess && b->ndirect)
    e = cudaMemcpyAsync(tail + lb, tabs.data(), tabs.size() * sizeof(pw::smu::TabArgs<pwi::Wide>), cudaMemcpyHostToDevice, b->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
  if (e != cudaSuccess) return cuda_fail(e, "uploading the batch descriptors");
  return build_items(b);
}

int num_sms() {
  int dev = 0, n = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
  return n > 0 ? n : 1;
}

}  // namespace

extern "C" {

size_t pw_batch_workspace_bytes(const pw_instance* inst, int n, int pool) {
  if (!inst || n <= 0 || pool <= 0) return 0;
  return layout(inst, n, pool).total;
}

pw_status pw_batch_create(pw_batch** out, const pw_instance* in, int n, int pool, void* dev_ws, size_t ws_bytes,
                          void* stream) {
  pwi::set_last_error("");
  if (!out) return fail(PW_EINVAL, "out is null");
  *out = nullptr;
  if (!in || n <= 0) return fail(PW_EINVAL, "need at least one instance");
  if (pool <= 0) return fail(PW_EINVAL, "pool depth must be >= 1");
  if (!dev_ws) return fail(PW_EINVAL, "workspace is null");
  if (!aligned(dev_ws, 16)) return fail(PW_EINVAL, "the workspace must be 16-byte aligned");
  for (int i = 0; i < n; ++i) {
    const pw_instance& q = in[i];
    if (!batch_n(q.N)) return fail(PW_EUNSUPPORTED, "instance %d: N = %d (batched runs take N in {16, 32, 64, 96, 128})", i, q.N);
    if (!finite_pos(q.dxi_m) || !finite_pos(q.lambda_m) || !finite_pos(q.z_m) || !finite_pos(q.sigma_S_m) ||
        !finite_pos(q.sigma_mu_m))
      return fail(PW_EINVAL, "instance %d: lengths must be finite and > 0", i);
    if (!std::isfinite(q.amplitude) || !std::isfinite(q.aperture_m) || !std::isfinite(q.lens_f_m))
      return fail(PW_EINVAL, "instance %d: amplitude, aperture and focal length must be finite", i);
    if (q.iP < 0 || q.jP < 0 || q.iP >= q.N || q.jP >= q.N) return fail(PW_EINVAL, "instance %d: P1 outside the grid", i);
    if (!q.dev_S) return fail(PW_EINVAL, "instance %d: dev_S is required", i);
    if (!aligned(q.dev_W, 16) || !aligned(q.dev_S, 4) || !aligned(q.dev_mu, 8) || !aligned(q.dev_mask, 8))
      return fail(PW_EINVAL, "instance %d: misaligned device pointer (dev_W 16 bytes, dev_mu and dev_mask 8, dev_S 4)", i);
  }
  const Layout L = layout(in, n, pool);
  if (ws_bytes < L.total) return fail(PW_ESIZE, "workspace needs %zu bytes (got %zu)", L.total, ws_bytes);
  pw_batch* b = new pw_batch{};
  b->n = n;
  b->pool = pool;
  b->chunk = 8;
  b->base = reinterpret_cast<char*>(dev_ws);
  b->L = L;
  b->stream = reinterpret_cast<cudaStream_t>(stream);
  b->stalled.assign(n, 0);
  b->wait_cycles = 2000000000LL;  // ~1 s at 2 GHz
  // sequenced launches fill the GPU with one instance at a time from N = 64 on; smaller instances
  // are too small for that and share the persistent launch
  bool all_large = true;
  for (int i = 0; i < n; ++i) all_large = all_large && in[i].N >= 64;
  b->mode = all_large ? PW_BATCH_SEQUENCED : PW_BATCH_PERSISTENT;
  b->wmaps.resize(n);
  for (int i = 0; i < n; ++i) {
    pw_status st = in[i].dev_W ? pwi::encode_wmap(&b->wmaps[i], in[i].dev_W, in[i].N) : PW_OK;
    if (st != PW_OK) {
      delete b;
      return st;
    }
  }
  std::vector<pw::TableArgs>& targs = b->targs;
  std::vector<float2*>& mus = b->mus;
  targs.resize(n);
  mus.resize(n);
  b->smu.resize(n);
  b->smu_t.resize(n);
  b->inst.resize(n);
  size_t off = L.tables;
  for (int i = 0; i < n; ++i) {
    const pw_instance& q = in[i];
    const int N = q.N;
    const size_t NN = (size_t)N * N;
    pw::batch::Inst& d = b->inst[i];
    d.N = N;
    d.iP = q.iP;
    d.jP = q.jP;
    d.slices = (int)NN;
    d.A = (float)q.amplitude;
    const double lz = q.lambda_m * q.z_m;
    const double s2 = (q.dxi_m * q.dxi_m / lz) * (q.dxi_m * q.dxi_m / lz);
    d.scale = (float)s2;
    b->scale.push_back(s2);
    b->A.push_back(q.amplitude);
    float2* F = reinterpret_cast<float2*>(b->base + off);
    off = align256(off + NN * sizeof(float2));
    float* G = reinterpret_cast<float*>(b->base + off);
    off = align256(off + NN * sizeof(float));
    float2* tw = reinterpret_cast<float2*>(b->base + off);
    off = align256(off + N * sizeof(float2));
    float2* Eo = reinterpret_cast<float2*>(b->base + off);
    off = align256(off + N * sizeof(float2));
    float2* Ei = reinterpret_cast<float2*>(b->base + off);
    off = align256(off + N * sizeof(float2));
    d.row = reinterpret_cast<float2*>(b->base + off);
    off = align256(off + NN * sizeof(float2));
    d.F = F;
    d.G = G;
    d.tw = tw;
    d.Eout = Eo;
    d.Ein = Ei;
    d.mask = reinterpret_cast<const float2*>(q.dev_mask);
    d.W = reinterpret_cast<float2*>(q.dev_W);
    d.S = q.dev_S;
    mus[i] = reinterpret_cast<float2*>(q.dev_mu);
    // FP64 tables: same quantities as the single-instance path (propagator phases in turns)
    pw::TableArgs& t = targs[i];
    t = pw::TableArgs{};
    t.N = N;
    const double invf = q.lens_f_m != 0.0 ? 1.0 / q.lens_f_m : 0.0;
    const double base = q.dxi_m * q.dxi_m / (2.0 * q.lambda_m);
    t.Kin = q.farfield ? -base * invf : base * (1.0 / q.z_m - invf);
    const double dx = lz / (N * q.dxi_m);
    t.Kout = dx * dx / (2.0 * lz);
    b->dx_out.push_back(dx);
    t.gs = q.dxi_m * q.dxi_m / (4.0 * q.sigma_S_m * q.sigma_S_m);
    t.gm = q.dxi_m * q.dxi_m / (2.0 * q.sigma_mu_m * q.sigma_mu_m);
    if (q.aperture_m > 0.0) {
      const double rp = q.aperture_m / q.dxi_m;
      t.ap_thr = rp * rp;  // r^2 is an integer: the integer floor gives the same decision
      d.ap_ithr = t.ap_thr >= 2147483647.0 ? 2147483647 : (int)std::floor(t.ap_thr);
    } else {
      t.ap_thr = -1.0;
      d.ap_ithr = -1;
    }
    t.mask = reinterpret_cast<const float2*>(q.dev_mask);
    t.F = F;
    t.G = G;
    t.tw = tw;
    t.Eout = Eo;
    t.Ein = Ei;
    // smu.cuh: its tables take the place of F (88 N of the 8 N^2 bytes)
    pw::smu::TabArgs<pwi::Wide>& ta = b->smu_t[i];
    ta.N = N;
    ta.Kin = t.Kin;
    ta.Kout = t.Kout;
    ta.gs = t.gs;
    ta.gm = t.gm;
    ta.amp = std::sqrt(std::sqrt(s2 * std::fabs(q.amplitude) / (4.0 * (double)NN)));
    ta.tw = reinterpret_cast<pwi::Wide*>(F);
    ta.P1 = ta.tw + 2 * N;
    ta.Eout = ta.P1 + N;
    ta.k = reinterpret_cast<pw::real_t<pwi::Wide>*>(ta.Eout + N);
    pw::smu::Inst<pwi::Wide>& si = b->smu[i];
    si.N = N;
    si.iP = q.iP;
    si.jP = q.jP;
    si.factor = q.amplitude < 0.0 ? -1.0 : 1.0;
    si.tw = ta.tw;
    si.P1 = ta.P1;
    si.Eout = ta.Eout;
    si.k = ta.k;
    si.K = ta.k + N;
    si.mask = d.mask;
    si.ap_ithr = d.ap_ithr;
    si.S = q.dev_S;
    si.mu = mus[i];
  }
  bool any128 = false;
  for (int i = 0; i < n; ++i) any128 = any128 || in[i].N == 128;
  std::vector<CUtensorMap> maps(pool);
  if (any128) {
    for (int k = 0; k < pool; ++k) {
      pw_status st = pwi::encode_vmap(&maps[k], b->base + L.pool + L.slot_bytes * k, 128);
      if (st != PW_OK) {
        delete b;
        return st;
      }
    }
  }
  cudaError_t e = cudaSuccess;
  if (any128)
    e = cudaMemcpyAsync(b->base + L.tmaps, maps.data(), sizeof(CUtensorMap) * pool, cudaMemcpyHostToDevice,
                        b->stream);
  if (e == cudaSuccess)  // counters and the error flag start at zero (the workspace may hold old data)
    e = cudaMemsetAsync(b->base + L.counters, 0, sizeof(int) * (2 * (size_t)n + 2), b->stream);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(pw::batch::batch_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)pw::batch::smem_bytes());
  if (e != cudaSuccess) {
    delete b;
    return cuda_fail(e, "batch set-up");
  }
  pw_status st = upload(b);
  if (st != PW_OK) {
    delete b;
    return st;
  }
  *out = b;
  return PW_OK;
}

pw_status pw_batch_run(pw_batch* b) {
  pwi::set_last_error("");
  if (!b) return fail(PW_EINVAL, "null batch");
  cudaError_t e;
  if (b->ndirect) {
    if ((e = pwi::launch_smu_list_tables(b->dev_smu_t, b->ndirect, b->stream)) != cudaSuccess)
      return cuda_fail(e, "batch S/mu tables launch");
    for (const auto& r : b->rounds)
      for (int N : r.Ns)
        if ((e = pwi::launch_smu_list(N, b->dev_smu, b->ndirect, r.chunk, r.mu, b->stream)) != cudaSuccess)
          return cuda_fail(e, "batch S/mu launch");
    if (b->ndirect == b->n) return PW_OK;
  }
  int* cnt = reinterpret_cast<int*>(b->base + b->L.counters);
  if (b->mode == PW_BATCH_PERSISTENT) {
    e = cudaMemsetAsync(cnt, 0, sizeof(int) * (2 * (size_t)b->n + 1), b->stream);
    if (e != cudaSuccess) return cuda_fail(e, "resetting the batch counters");
  }
  int maxNN = 0;
  for (const auto& d : b->inst) maxNN = d.slices > maxNN ? d.slices : maxNN;
  dim3 tg((maxNN + 255) / 256, b->n);
  pw::batch::batch_tables_kernel<<<tg, 256, 0, b->stream>>>(reinterpret_cast<const pw::TableArgs*>(b->base + b->L.targs));
  if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(e, "batch tables launch");
  // mu of the instances that are not on smu.cuh (the others' entries are null)
  auto mu = [&]() -> pw_status {
    dim3 mg((maxNN + 255) / 256, b->n);
    pw::batch::batch_mu_kernel<<<mg, 256, 0, b->stream>>>(reinterpret_cast<const pw::batch::Inst*>(b->base + b->L.inst),
                                                          reinterpret_cast<float2* const*>(b->base + b->L.mu));
    const cudaError_t r = cudaGetLastError();
    return r == cudaSuccess ? PW_OK : cuda_fail(r, "batch mu launch");
  };
  if (b->mode == PW_BATCH_SEQUENCED) {
    // one instance after the other on the plane kernels (stream order reuses the slots)
    for (int i = 0; i < b->n; ++i) {
      const pw::batch::Inst& d = b->inst[i];
      if (direct(b, i)) continue;
      pwi::PlaneArgs q{};
      q.F = d.F;
      q.G = d.G;
      q.tw = d.tw;
      q.Eout = d.Eout;
      q.work = d.V;
      q.W = d.W;
      q.S = d.S;
      q.A = b->A[i];
      q.scale = b->scale[i];
      q.row = d.row;
      q.iP = d.iP;
      q.jP = d.jP;
      e = pwi::dispatch_planes(d.N, b->wmaps[i], q, cnt + 2 * b->n + 1, b->stream, nullptr);
      if (e != cudaSuccess) return cuda_fail(e, "batch instance launch");
    }
    return mu();
  }
  pw::batch::Args g{};
  g.inst = reinterpret_cast<const pw::batch::Inst*>(b->base + b->L.inst);
  g.items = reinterpret_cast<const pw::batch::Item*>(b->base + b->L.items);
  g.nitems = b->nitems;
  g.next = cnt + 2 * b->n;
  g.doneA = cnt;
  g.doneB = cnt + b->n;
  g.err = cnt + 2 * b->n + 1;
  g.wait_cycles = b->wait_cycles;
  pw::batch::batch_kernel<<<num_sms(), pw::batch::NT, pw::batch::smem_bytes(), b->stream>>>(g);
  if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(e, "batch kernel launch");
  return mu();
}

pw_status pw_batch_check(pw_batch* b) {
  pwi::set_last_error("");
  if (!b) return fail(PW_EINVAL, "null batch");
  int flag = 0;
  int* err = reinterpret_cast<int*>(b->base + b->L.counters) + 2 * b->n + 1;
  cudaError_t e = cudaMemcpyAsync(&flag, err, sizeof(int), cudaMemcpyDeviceToHost, b->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
  if (e != cudaSuccess) return cuda_fail(e, "reading the batch error flag");
  if (flag) {
    e = cudaMemsetAsync(err, 0, sizeof(int), b->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) return cuda_fail(e, "clearing the batch error flag");
    return fail(PW_ETIMEOUT, "a bounded wait of the batched launch gave up; some outputs are invalid");
  }
  return PW_OK;
}

pw_status pw_batch_set_chunk(pw_batch* b, int chunk) {
  pwi::set_last_error("");
  if (!b) return fail(PW_EINVAL, "null batch");
  if (chunk < kMinChunk) return fail(PW_EINVAL, "chunk must be >= %d", kMinChunk);
  b->chunk = chunk;
  return build_items(b);
}

pw_status pw_batch_spectral_sum(pw_batch* b, const double* weights, float* dev_I) {
  pwi::set_last_error("");
  if (!b || !weights || !dev_I) return fail(PW_EINVAL, "null argument");
  const int N = b->inst[0].N;
  for (int i = 0; i < b->n; ++i) {
    if (b->inst[i].N != N) return fail(PW_EINVAL, "instance %d: N = %d differs from instance 0 (N = %d)", i, b->inst[i].N, N);
    if (std::fabs(b->dx_out[i] / b->dx_out[0] - 1.0) > 1e-9)
      return fail(PW_EINVAL, "instance %d: output sampling %.9g m differs from instance 0 (%.9g m): no common grid",
                  i, b->dx_out[i], b->dx_out[0]);
    if (!std::isfinite(weights[i])) return fail(PW_EINVAL, "weight %d is not finite", i);
  }
  double* w = reinterpret_cast<double*>(b->base + b->L.wts);
  cudaError_t e = cudaMemcpyAsync(w, weights, sizeof(double) * b->n, cudaMemcpyHostToDevice, b->stream);
  if (e != cudaSuccess) return cuda_fail(e, "uploading the weights");
  const int NN = N * N;
  pw::batch::batch_sum_kernel<<<(NN + 255) / 256, 256, 0, b->stream>>>(
      reinterpret_cast<const pw::batch::Inst*>(b->base + b->L.inst), w, b->n, dev_I, NN);
  if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(e, "spectral sum launch");
  return PW_OK;
}

// The mode decides where a stalled batch runs its instances without W.
static pw_status change_mode(pw_batch* b, int mode) {
  const bool again = mode != b->mode && stalled(b);
  b->mode = mode;
  return again ? upload(b) : PW_OK;
}

pw_status pw_batch_set_mode(pw_batch* b, int mode) {
  pwi::set_last_error("");
  if (!b) return fail(PW_EINVAL, "null batch");
  if (mode != PW_BATCH_PERSISTENT && mode != PW_BATCH_SEQUENCED) return fail(PW_EINVAL, "unknown batch mode %d", mode);
  return change_mode(b, mode);
}

pw_status pw_batch_get_mode(const pw_batch* b, int* mode) {
  pwi::set_last_error("");
  if (!b || !mode) return fail(PW_EINVAL, "null argument");
  *mode = b->mode;
  return PW_OK;
}

pw_status pw_batch_get_chunk(const pw_batch* b, int* chunk) {
  pwi::set_last_error("");
  if (!b || !chunk) return fail(PW_EINVAL, "null argument");
  *chunk = b->chunk;
  return PW_OK;
}

pw_status pw_batch_autotune(pw_batch* b, int* chunk_out) {
  pwi::set_last_error("");
  if (!b) return fail(PW_EINVAL, "null batch");
  // candidates: the sequenced launches, and the persistent launch at each chunk size
  const int cand[][2] = {{PW_BATCH_SEQUENCED, 0},   {PW_BATCH_PERSISTENT, 4},  {PW_BATCH_PERSISTENT, 8},
                         {PW_BATCH_PERSISTENT, 16}, {PW_BATCH_PERSISTENT, 32}, {PW_BATCH_PERSISTENT, 64}};
  cudaEvent_t e0, e1;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess)
    return cuda_fail(cudaGetLastError(), "autotune events");
  float best = 1e30f;
  int best_m = b->mode, best_c = b->chunk;
  pw_status st = PW_OK;
  for (const auto& mc : cand) {
    if ((st = change_mode(b, mc[0])) != PW_OK) break;
    if (mc[0] == PW_BATCH_PERSISTENT && (st = pw_batch_set_chunk(b, mc[1])) != PW_OK) break;
    if ((st = pw_batch_run(b)) != PW_OK) break;  // warm-up
    cudaEventRecord(e0, b->stream);
    if ((st = pw_batch_run(b)) != PW_OK) break;
    cudaEventRecord(e1, b->stream);
    cudaEventSynchronize(e1);
    float ms = 0.f;
    cudaEventElapsedTime(&ms, e0, e1);
    if (ms < best) {
      best = ms;
      best_m = mc[0];
      best_c = mc[0] == PW_BATCH_PERSISTENT ? mc[1] : best_c;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (st != PW_OK) return st;
  if ((st = pw_batch_check(b)) != PW_OK) return st;
  if ((st = change_mode(b, best_m)) != PW_OK) return st;
  if (chunk_out) *chunk_out = best_c;
  return pw_batch_set_chunk(b, best_c);
}

pw_status pw_batch_inject_stall(pw_batch* b, int instance, double wait_s) {
  pwi::set_last_error("");
  if (!b) return fail(PW_EINVAL, "null batch");
  if (instance < 0 || instance >= b->n) return fail(PW_EINVAL, "instance out of range");
  if (!(wait_s > 0.0) || !std::isfinite(wait_s)) return fail(PW_EINVAL, "wait must be finite and > 0");
  b->stalled[instance] = 1;
  b->wait_cycles = (long long)(wait_s * 2.0e9);
  return upload(b);
}

pw_status pw_batch_destroy(pw_batch* b) {
  pwi::set_last_error("");
  if (!b) return PW_OK;
  cudaError_t e = cudaStreamSynchronize(b->stream);
  delete b;
  if (e != cudaSuccess) return cuda_fail(e, "stream synchronize in batch destroy");
  return PW_OK;
}

}  // extern "C"
