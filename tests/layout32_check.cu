// The 32-bit forms of the layout arithmetic that the kernels use, on the host:
// equal to the 64-bit ones (layout64.h) at every node of small trees, at every
// level's ends and at places spread over the tallest trees there can be (30 levels).
#include <cstdio>

#include "layout64.h"

using namespace bdl;

static int bad = 0;
#define CHECK(c)                                   \
  do {                                             \
    if (!(c) && bad++ < 10) printf("line %d\n", __LINE__); \
  } while (0)

int main() {
  for (int h = 1; h <= 30; ++h) {
    for (int t = 0; t <= h; ++t) {
      const int64_t n = (int64_t)1 << t, step = n <= 4096 ? 1 : n / 4093;
      for (int64_t i = 0; i < n; i += step) {
        CHECK(veb_slot(h + 1, t, i) == veb_slot32(h + 1, t, (int)i));
        if (t < h && (t == 0 || ((h - t) & 1) == 0)) CHECK(packed_slot(h, t, i) == packed_slot32(h, t, (int)i));
      }
      CHECK(veb_slot(h + 1, t, n - 1) == veb_slot32(h + 1, t, (int)(n - 1)));
    }
    const int64_t n = packed_nrec(h), step = n <= 50000 ? 1 : n / 49999;
    for (int64_t g = 0; g < n; g += step) {
      int t, t2, i2;
      int64_t i;
      packed_record_of(h, g, t, i);
      packed_record_of32(h, (int)g, t2, i2);
      CHECK(t == t2 && i == i2);
    }
  }
  // the depths that go to one block: none above them holds more nodes than
  // that, also where trees of several heights make a shallow depth the largest
  const int64_t even[] = {1, 2, 4, 8, 16, 32, 64, 128, 256, 512, 1024, 2048, 4096};
  const int64_t mixed[] = {501, 1002, 2004, 4008, 8016, 16032, 32064, 64128, 128256, 512};
  const int64_t many[] = {2000, 4000, 512};
  CHECK(one_block_depths(even, 13) == 11 && one_block_depths(even, 5) == 5);
  CHECK(one_block_depths(mixed, 10) == 2 && one_block_depths(many, 3) == 0 && one_block_depths(many, 0) == 0);
  // the tallest trees there can be (2^31 - 1 points, leaves of two), the levels
  // of records that a walk goes down in one, and the warp-per-query kernel's
  // node stack: what a wide round may leave on it and the rest one by one
  CHECK(tree_height(INT32_MAX, 2) == kMaxHeight);
  int levels = 0;
  for (int t = 0; t < kMaxHeight; t += packed_step(kMaxHeight, t)) ++levels;
  CHECK(kWWide - 8 + 32 + 3 * levels <= kWStack);
  CHECK(kMaxLevel + 1 + 32 <= kWWide);   // (the walk starts with every tree's root)
  // a grid barrier waits several times as long as the longest phase of a build
  // can take: one block's select over the most points there can be, 6 ns each
  CHECK(kBarrierNs >= 4 * 6 * (unsigned long long)INT32_MAX);
  puts(bad ? "BAD" : "ok");
  return bad != 0;
}
