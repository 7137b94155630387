// The walks' stack rule (csrc/gfs_internal.cuh) on hierarchies of any depth: a
// walk whose children are kept by a seeded chance, for a bounded number of
// rounds; returns the largest stack it needed.
#include "gfs_internal.cuh"

extern "C" int walk_take_host(int levels, int cap, int width, int keep, int rounds, unsigned seed, int* reserve) {
  using namespace gfs;
  *reserve = kFan;
  if (levels > kMaxLevels) return -1;
  static int stk[1 << 16];
  int sp = 0, most = 0;
  for (int j = 0; j < kFan; ++j) stk[sp++] = levels - 1;
  most = sp;
  for (int r = 0; r < rounds && sp > 0; ++r) {
    const int take = walk_take(sp, cap, width);
    if (take < 1 || take > sp || take > width) return -2;
    int add[4096], n = 0;
    for (int t = 0; t < take; ++t) {
      const int lev = stk[sp - 1 - t];
      if (lev == 0) continue;
      for (int c = 0; c < kFan; ++c) {
        seed = seed * 1664525u + 1013904223u;
        if (int(seed >> 24) < keep) add[n++] = lev - 1;
      }
    }
    sp -= take;
    for (int k = 0; k < n; ++k) stk[sp++] = add[k];
    most = sp > most ? sp : most;
  }
  return most;
}
