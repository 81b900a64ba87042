// Test helper (host code only): for every subspace m up to 160, on clusters of 8 and of 16, the
// shared-memory reads of the one-cluster Rayleigh-Ritz sweep by the kernel's own index functions.  One
// line each:
//   m  threads  active  items  highest float index read in a copy  floats of a copy
//   bytes the layout ends at  bytes asked for (b = 1)  entries hit exactly once (1 or 0)
#include <cstdio>
#include <vector>

#include "ritz_layout.cuh"

using namespace fe;

int main() {
  for (int k = 0; k < 2 * kRitzOneMax; ++k) {
    const int m = k / 2 + 1;
    const RitzShape sh = ritz_shape(m, k % 2 != 0);
    const int mp = m + (m & 1), np = mp / 2, nitems = ritz_items(np), nact = ritz_active(np, sh.threads);
    int top = 4 * nitems + np - 1;   // the pivots
    for (int tid = 0; tid < nact; ++tid)
      for (int u = 0; u < sh.items; ++u)
        for (int v = 0; v < 4; ++v) top = std::max(top, v * nitems + ritz_read(tid + u * nact, nitems));
    std::vector<int> hit(ritz_copy(np), 0);
    bool once = true;
    for (int a = 0; a < mp; ++a)
      for (int b = a + 1; b < mp; ++b) {
        const int e = ritz_entry(a, b, mp);
        if (e < 0 || e >= (int)hit.size() || hit[e]++) once = false;
      }
    const long end = 8L * np + 16L * mp + 2 * 4L * ritz_copy(np);
    printf("%d %d %d %d %d %d %ld %zu %d\n", m, sh.threads, nact, sh.items, top, ritz_copy(np), end,
           ritz_cluster_smem(m, 1, sh.ncta), once && (size_t)mp * (mp - 1) / 2 == hit.size() ? 1 : 0);
  }
  for (int max_sweeps : {1, 2, 5, 6, 7, 60}) {   // "sweeps max_sweeps: first, then all later ones" if every cap is used
    int left = max_sweeps, later = 0;
    for (int it = 1; it < 40; ++it) {
      const int cap = ritz_sweep_cap(it, left);
      later += cap;
      left -= cap;
    }
    printf("sweeps %d %d %d\n", max_sweeps, ritz_sweep_cap(0, max_sweeps), later);
  }
  return 0;
}
