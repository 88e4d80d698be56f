"""Slots and work order of the persistent batch launch (csrc/batch_plan.h): on the CPU that no instance can
overwrite a slot that an earlier one still reads, whatever instances outside the launch stand between them;
on the GPU that batches which mix instances with and without W give the outputs of the single calls."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2203_02734_gb300", "csrc")
D, LAM = 20e-6, 633e-9

# Replays every list of 1 to 9 instances (any subset in the launch), pools of 1 to 5 slots and three chunk sizes.
CHECK = r"""
#include <cstdio>
#include <map>
#include "batch_plan.h"
using namespace pw::batch;
int main() {
  const int sizes[3] = {16, 32, 128};
  for (int n = 1; n <= 9; ++n)
    for (int mask = 0; mask < 1 << n; ++mask)
      for (int pool = 1; pool <= 5; ++pool)
        for (int chunk : {4, 24, 64}) {
          std::vector<int> m, N, none(n, 0);
          for (int i = 0; i < n; ++i) {
            if (mask >> i & 1) m.push_back(i);
            N.push_back(sizes[(i + mask) % 3]);
          }
          const auto at = places(m, n, pool);
          const auto list = items(m, N, none, chunk, pool);
          std::map<int, int> holder;  // the latest member in each slot
          for (int i : m) {
            if (at[i].slot < 0 || at[i].slot >= pool) return printf("slot\n"), 1;
            const int last = holder.count(at[i].slot) ? holder[at[i].slot] : -1;
            if (at[i].prev != last) return printf("n %d mask %x pool %d: %d waits for %d, not %d\n", n, mask, pool, i, at[i].prev, last), 1;
            holder[at[i].slot] = i;
          }
          std::vector<int> done[2] = {std::vector<int>(n, 0), std::vector<int>(n, 0)};
          for (const auto& it : list) {
            const int i = it.inst;  // what it waits for is listed before it
            if (it.pass == 1 && done[0][i] != N[i] * N[i]) return printf("B before A\n"), 1;
            if (it.pass == 0 && at[i].prev >= 0 && done[1][at[i].prev] != N[at[i].prev] * N[at[i].prev]) return printf("A before B of its slot\n"), 1;
            if (it.first + (it.count - 1) * it.stride >= N[i] * N[i]) return printf("range\n"), 1;
            done[it.pass][i] += it.count;
          }
          for (int i : m)
            if (done[0][i] != N[i] * N[i] || done[1][i] != N[i] * N[i]) return printf("slices\n"), 1;
        }
  return 0;
}
"""


def test_slots_and_order(tmp_path):
    src = tmp_path / "plan.cpp"
    src.write_text(CHECK)
    exe = str(tmp_path / "plan")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, "-o", exe, str(src)], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


# W: keeps W, -: S and mu only.  In each pattern a slot passes from one instance with W to another whose
# predecessor by index (i - pool) has none.  Two FP32 engines, each within 1e-6 in L2 (see test_planes.py).
@pytest.mark.gpu
@pytest.mark.parametrize("N", [16, 32, 64, 96, 128])
@pytest.mark.parametrize("pattern,pool", [("W-W", 1), ("W-------W", 4), ("WW-WW", 2), ("W--W-W", 1)])
def test_mixed_batch_matches_single_calls(N, pattern, pool):
    import torch
    import paper_2203_02734_gb300 as pw
    n, P1 = len(pattern), (N // 2 - 1, N // 2)
    S = torch.empty(n, N, N, device="cuda")
    mu = torch.empty(n, N, N, dtype=torch.complex64, device="cuda")
    W = {i: torch.empty(N, N, N, N, dtype=torch.complex64, device="cuda") for i in range(n) if pattern[i] == "W"}
    insts = []
    for i in range(n):
        q = pw.pw_instance()
        q.N, q.dxi_m, q.lambda_m, q.z_m, q.farfield = N, D, LAM * (1 + 0.03 * i), 0.3 + 0.1 * i, i % 2
        q.sigma_S_m, q.sigma_mu_m, q.amplitude = 5 * D, 1.5 * D, 0.8 + 0.1 * i
        (q.iP, q.jP), q.dev_S, q.dev_mu = P1, S[i].data_ptr(), mu[i].data_ptr()
        if i in W:
            q.dev_W = W[i].data_ptr()
        insts.append(q)
    ref = {}
    for i in W:
        c = pw.CSD(N, D, insts[i].lambda_m)
        c.source_gsm(5 * D, 1.5 * D, insts[i].amplitude)
        (c.propagate_farfield if i % 2 else c.propagate_fresnel)(insts[i].z_m)
        ref[i] = c.W, c.spectral_density(), c.degree_of_coherence(*P1)
        c.close()
    nb = pw.pw_batch_workspace_bytes(insts, pool)
    ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
    b = pw.pw_batch_create(insts, pool, ws.data_ptr(), nb, torch.cuda.current_stream().cuda_stream)
    pw.pw_batch_set_mode(b, pw.PW_BATCH_PERSISTENT)
    norm = lambda t: float(torch.linalg.vector_norm(torch.view_as_real(t) if t.is_complex() else t))  # noqa: E731
    for chunk in (4, 8, 32):
        pw.pw_batch_set_chunk(b, chunk)
        for _ in range(3):
            for w in W.values():
                w.fill_(float("nan"))
            pw.pw_batch_run(b)
            pw.pw_batch_check(b)
            for i, (Wr, Sr, mur) in ref.items():
                assert norm(W[i] - Wr) < 2e-6 * norm(Wr)
                assert norm(S[i] - Sr) < 2e-6 * norm(Sr)
                bright = Sr >= 1e-2 * Sr.max()
                assert float((mu[i] - mur)[bright].abs().max()) < 2e-5
    pw.pw_batch_destroy(b)
