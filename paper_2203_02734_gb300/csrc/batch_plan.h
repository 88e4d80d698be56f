// batch_plan.h -- which slot of the V pool each instance of the persistent launch uses, whom it waits for, and
// the order of the work items (host only).
#pragma once
#include <vector>

namespace pw {
namespace batch {

struct Item {
  int inst;
  int pass;  // 0 = A, 1 = B
  int first, count, stride;
};

// Slot of the pool, and the instance that used it before (-1: none).
struct Place {
  int slot = 0, prev = -1;
};

// `members`: the instances in the launch, ascending.  They take the slots in turn, so that an instance and the
// one whose slot it reuses are always `pool` members apart, whatever instances outside the launch stand
// between them; pass A waits for pass B of `prev`, and by induction for every earlier holder.
inline std::vector<Place> places(const std::vector<int>& members, int n, int pool) {
  std::vector<Place> p(n);
  for (int r = 0; r < (int)members.size(); ++r) {
    p[members[r]].slot = r % pool;
    p[members[r]].prev = r >= pool ? members[r - pool] : -1;
  }
  return p;
}

// Lookahead of L members: A(0) .. A(L-1), then B(r), A(r + L) for r = 0, 1, ...  B(r) waits for A(r), listed L
// phases earlier; A(r + L) reuses the slot of member r + L - pool and waits for its pass B, listed pool - L
// phases earlier.  L = pool - 2 (at least 1) leaves two phases between every wait and the items it waits on,
// and every awaited item precedes its waiter.
// One pass = J = ceil(slices / chunk) items.  N = 128 (register-resident engine, whose pass B gathers 8 bytes
// from every 32-byte run of V): strided items, item j takes slices j, j + J, j + 2 J, ..., so that neighbouring
// CTAs gather the columns of one run together.  Other sizes: contiguous ranges of chunk slices (measured
// slightly faster there).  left_out: instances whose pass A is left out (failure-detection test).
inline std::vector<Item> items(const std::vector<int>& members, const std::vector<int>& N, const std::vector<int>& left_out,
                               int chunk, int pool) {
  std::vector<Item> list;
  auto add = [&](int r, int pass) {
    const int i = members[r], S = N[i] * N[i], J = (S + chunk - 1) / chunk;
    if (pass == 0 && left_out[i]) return;
    for (int j = 0; j < J; ++j) {
      if (N[i] == 128) list.push_back({i, pass, j, (S - j + J - 1) / J, J});
      else list.push_back({i, pass, j * chunk, j + 1 < J ? chunk : S - j * chunk, 1});
    }
  };
  const int n = (int)members.size(), L = pool >= 3 ? pool - 2 : 1;
  for (int r = 0; r < L && r < n; ++r) add(r, 0);
  for (int r = 0; r < n; ++r) {
    add(r, 1);
    if (r + L < n) add(r + L, 0);
  }
  return list;
}

}  // namespace batch
}  // namespace pw
