// Host check of the exchange's limb arithmetic (cg_exact.cuh): sums of many addends
// through the three words against 128-bit sums.  Prints "ok" or the first mismatch.
#include <algorithm>
#include <cstdio>
#include <random>

#include "../paper_2608_09647_gb300/csrc/cg_exact.cuh"

using namespace cg_exact;

static int check(int G, int warps, int e0, std::mt19937_64& r, bool extreme) {
  const int B = std::max(1, e0 - kRoom);
  unsigned long long d[3] = {0, 0, 0};
  i128 total = 0;
  int left_out = 0;
  for (int g = 0; g < G; ++g) {
    unsigned long long w[3] = {0, 0, 0};
    bool exc = false;
    for (int k = 0; k < warps; ++k) {
      int E = std::max(1, e0 - (int)(r() % 90) + (int)(r() % 12));
      i128 S = ((i128)(long long)r() << 5) >> (r() % 62);
      if (r() & 1) S = -S;
      if (extreme) {
        E = B;
        S = (((i128)1 << 104) - 1) * ((g & 1) ? 1 : -1);
      }
      if (to_scale(&S, E, false, B)) {
        total += S;
        for (int l = 0; l < 3; ++l) w[l] += limb(S, l);
      } else {
        exc = true;
      }
    }
    left_out += exc;
    for (int l = 0; l < 3; ++l) d[l] += w[l] + (1ull << kCountAt);
    if (exc) d[2] += 1ull << kExcAt;
  }
  int ex = 0;
  const i128 j = join_limbs(d[0], d[1], d[2], &ex);
  for (int l = 0; l < 3; ++l)
    if ((int)(d[l] >> kCountAt) != G) return 1;
  return (j != total) * 2 + (ex != left_out) * 4;
}

int main() {
  std::mt19937_64 r(20);
  for (int it = 0; it < 6000; ++it) {
    const bool wide = it & 1;  // 8 warps of up to 511 CTAs, 16 of up to 255
    const int G = it < 4 ? (wide ? 255 : kMaxAddends) : 1 + (int)(r() % (wide ? 255 : kMaxAddends));
    const int bad = check(G, wide ? 16 : 8, 1 + (int)(r() % 2040), r, it < 4);
    if (bad) {
      std::printf("case %d: G %d mismatch %d\n", it, G, bad);
      return 1;
    }
  }
  i128 S = 1;
  if (to_scale(&S, 5, true, 5) || enough_bits(0.0, 100) || !enough_bits(0.0, 1)) {
    std::printf("flags\n");
    return 1;
  }
  std::printf("ok\n");
  return 0;
}
