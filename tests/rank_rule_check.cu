// Host-side check of which instance of rank_cluster_kernel a call takes (rank.cu), built by
// tests/test_rank_rule.py with nvcc and run on the CPU: two CTAs per SM only where the clusters
// do not all run together at one, and only where two CTAs' shared memory fits an SM.
#include <cstdio>

#include "../paper_2608_28911_gb300/csrc/rank.cu"

using namespace semkv;

int main() {
  int bad = 0;
  const size_t per_sm = 228 * 1024, reserved = 1024, fixed = 49424;
  ClusterLimits l;
  l.resident = 15;
  l.two_dynamic = two_cta_dynamic(per_sm, reserved, fixed);
  for (int B = 1; B <= 64; ++B)
    for (uint32_t T = 8192; cluster_chunk(T) <= kSmemKeys; T += 1003) {
      const size_t dyn = cluster_chunk(T) * sizeof(uint32_t);
      const bool fits = 2 * (reserved + fixed + dyn) <= per_sm;
      if (two_clusters_per_sm(B, dyn, l) != (B > 15 && fits)) bad++;
    }
  // a fixed part that leaves no room for two CTAs at all
  if (two_cta_dynamic(100 * 1024, 1024, 50 * 1024) != 0) bad++;
  printf("%s\n", bad ? "FAILED" : "rule ok");
  return bad != 0;
}
