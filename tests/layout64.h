// The packed k-NN records' layout in plain 64-bit arithmetic, as the 32-bit forms
// of the kernels are checked against it.
#pragma once
#include "../paper_2112_06188_gb300/csrc/bdl_internal.cuh"

namespace bdl {

// Position of node (level u, index i) in the vEB order of a complete 4-ary
// tree of H levels, split into top and bottom levels as veb_slot does.
inline int64_t veb4_slot(int H, int u, int64_t i) {
  int64_t off = 0;
  while (H > 1) {
    const int Hb = veb_bottom(H);
    const int Ht = H - Hb;
    if (u < Ht) {
      H = Ht;
    } else {
      const int uu = u - Ht;
      const int64_t j = i >> (2 * uu);
      off += quad_count(Ht) + j * quad_count(Hb);
      i &= ((int64_t)1 << (2 * uu)) - 1;
      u = uu;
      H = Hb;
    }
  }
  return off;
}

// Slot of the record of the node at depth t, index i (see packed_slot32).
inline int64_t packed_slot(int h, int t, int64_t i) {
  if (!(h & 1)) return veb4_slot(h / 2, t / 2, i);
  if (t == 0) return 0;
  const int64_t sub = i >> (t - 1), il = i & (((int64_t)1 << (t - 1)) - 1);
  return 1 + sub * quad_count((h - 1) / 2) + veb4_slot((h - 1) / 2, (t - 1) / 2, il);
}

// The g-th record in level order: depth t and index i of its node.
inline void packed_record_of(int h, int64_t g, int &t, int64_t &i) {
  const int odd = h & 1;
  if (odd && g == 0) {
    t = 0;
    i = 0;
    return;
  }
  int64_t y = odd ? g - 1 : g;
  int u = 0;
  while (y >= ((int64_t)(1 + odd) << (2 * u))) {   // 2 * 4^u (odd h) or 4^u nodes on level u
    y -= (int64_t)(1 + odd) << (2 * u);
    ++u;
  }
  t = 2 * u + odd;
  i = y;
}

}  // namespace bdl
