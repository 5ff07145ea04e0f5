// Host-side check of the decode work plan (make_decode_plan in decode.cu) over caches with
// an empty pool, and over many short ones with staged tails, built by
// tests/test_decode_plan_one_sided.py with nvcc and run on the CPU (no kernel is launched).
//
// Required of every plan: weights that are not negative and add up (W = w_hi tiles_hi +
// w_lo tiles_lo, the length of a pair's range that the kernels and the combine work from);
// every tile in exactly one CTA's range; every partial slot, the staged tail's included,
// inside the pair's stride; the stride within the caller's limit (a plan that needs more is
// a refused call, and none of these may be refused); the pools' CTAs, and the staged tails'
// where the plan makes room for them or the fast kernel runs them, within one wave.
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "../paper_2608_28911_gb300/csrc/decode.cu"

using namespace semkv;

static int check(int L_hi, int L_lo, int B, int H, int G, long hi, long lo, int stage_n, int sms,
                 int max_stride) {
  const DecodePlan P = make_decode_plan(SEMKV_BASE_AFFINE, L_hi, L_lo, B, H, G * H, hi, lo, stage_n,
                                        sms, max_stride);
  const long pairs = (long)B * H, total = pairs * P.W;
  const int st = stage_n > 0 ? 1 : 0;
  int bad = 0;
  if (P.stride > max_stride) bad++;
  if (P.w_hi < 0 || P.w_lo < 0) bad++;
  if (P.W != (int64_t)P.w_hi * P.tiles_hi + (int64_t)P.w_lo * P.tiles_lo) bad++;
  if (P.ctas > 2L * sms) bad++;
  if (st && !P.tails_apart && 2L * sms >= 4 * pairs && P.ctas + pairs > 2L * sms) bad++;
  // the fast kernel's tails never come after a full wave
  if (st && P.fast && !P.tails_apart && P.ctas + pairs > 2L * sms) bad++;
  for (long bh = 0; bh < pairs && !bad; ++bh) {
    int n_hi, n_lo;
    pair_slots(P, bh, n_hi, n_lo);
    if (n_hi < 0 || n_lo < 0 || pair_partials(P, bh) > P.stride) bad++;
    for (int src = 0; src < 2; ++src) {
      const int tiles = src ? P.tiles_lo : P.tiles_hi;
      const long w = src ? P.w_lo : P.w_hi;
      const long S = bh * P.W + (src ? (long)P.w_hi * P.tiles_hi : 0), E = S + w * tiles;
      std::vector<int> owners(tiles, 0);
      for (long c = 0; c < P.ctas; ++c) {
        const long start = c * P.per, end = start + P.per < total ? start + P.per : total;
        if (E <= S || E <= start || S >= end) continue;
        const long x0 = (start > S ? start : S) - S, x1 = (end < E ? end : E) - S;
        const long t0 = (x0 + w - 1) / w, t1l = (x1 + w - 1) / w, t1 = t1l < tiles ? t1l : tiles;
        for (long t = t0; t < t1; ++t) owners[t]++;
        const long slot = (c - S / P.per) + (src ? n_hi : 0);
        if (slot < 0 || slot >= (src ? n_hi + n_lo : n_hi)) bad++;
      }
      for (int t = 0; t < tiles; ++t)
        if (owners[t] != 1) bad++;
    }
  }
  if (bad)
    printf("L%d/%d B%d H%d G%d hi %ld lo %ld stage %d sms %d max_stride %d: ctas %d stride %d per %lld "
           "w %d/%d W %lld: BAD\n",
           L_hi, L_lo, B, H, G, hi, lo, stage_n, sms, max_stride, P.ctas, P.stride, (long long)P.per,
           P.w_hi, P.w_lo, (long long)P.W);
  return bad ? 1 : 0;
}

int main() {
  int bad = 0, n = 0;
  const long sizes[] = {1, 1000, 4096, 16384, 16640, 16656, 20000, 32768, 65536, 131072, 500000};
  for (int H = 1; H <= 8; ++H)
    for (long t : sizes)
      for (int side = 0; side < 2; ++side)
        for (int stage_n : {0, 77})
          for (int fast = 0; fast < 2; ++fast, ++n)
            bad += check(fast ? 6 : 8, fast ? 5 : 3, 1, H, 4, side ? 0 : t, side ? t : 0, stage_n, 152, 65);
  // staged tails beside the short pools of many pairs
  for (int B = 8; B <= 64; B += 2)
    for (long t : {250L, 500L, 1000L, 2048L, 3500L})
      for (int H : {4, 8}) {
        bad += check(6, 5, B, H, 4, t / 4, t - t / 4, 77, 152, 65);
        bad += check(4, 4, B, H, 4, t / 4, t - t / 4, 77, 152, 65);
        n += 2;
      }
  srand(4321);
  for (int i = 0; i < 3000; ++i, ++n) {
    const int B = 1 + rand() % 6, H = 1 + rand() % 4, G = rand() % 2 ? 4 : 8, stage_n = rand() % 2;
    const long big = 1 + (long)(rand() % 500000) / (1 + rand() % 50);
    const int side = rand() % 3, L = 2 + rand() % 7;
    const long hi = side == 1 ? 0 : big, lo = side == 0 ? 0 : big / 2 + 1;
    // (the least the entry points accept: three slots and the staged tail's)
    const int max_stride = rand() % 2 ? 65 : 3 + stage_n + rand() % 62;
    bad += check(L, L > 2 ? L - 1 : 2, B, H, G, hi, lo, stage_n, 20 + rand() % 180, max_stride < 65 ? max_stride : 65);
  }
  printf("%d plans, %d bad\n%s\n", n, bad, bad ? "FAILED" : "all plans ok");
  return bad != 0;
}
