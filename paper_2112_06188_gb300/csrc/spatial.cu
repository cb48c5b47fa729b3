// spatial.cu -- construction of the static kd-trees of one Insert_L with the
// spatial-median splitting rule of Sec. V-C: a node splits its points at the
// midpoint v = floor((min + max) / 2) of their coordinates in its dimension,
// points with coordinate <= v to the left (reading G12).  The trees keep the
// shape of the object-median trees (h split levels, nodes in vEB slots), so
// queries and erases run on them unchanged; only the build differs.
//
// GPU design: the sizes of a node's children now depend on the data, so the
// build carries each segment's bounds in arrays instead of closed form.  All
// new trees of one dimension advance level by level together; the trees are
// ordered by height, so the trees still splitting at level t are a prefix of
// that order and so are their records in the staging buffer.  A record's
// segment at level t is s = j * 2^t + i (tree j, node i of depth t), and its
// child's is 2s or 2s + 1.  k_sp_levels runs all levels in one cooperative
// launch.  Per level, with a grid barrier after each:
//   scatter -- left records fill the child's range from its start, right
//              ones from its end (aggregated atomic cursors); records of a
//              tree whose children are leaves go straight to the tree; the
//              others also give their child segment's min and max of the next
//              level's split coordinate, so only the first level needs a pass
//              for its bounds (block-, then warp-aggregated atomics);
//   split   -- the node's key and children, the children's bounds, and the
//              leaf offsets of trees that end here.
// Order inside a child is not kept (the sets are what the rule fixes).  Then
// leaf boxes, boxes bottom-up and the packed k-NN records.
#include "bdl_internal.cuh"

#include <algorithm>
#include <numeric>

namespace bdl {

namespace {

constexpr int kT = 256;   // threads per block of the record passes

struct SpTree {           // one tree of a spatial build, as the kernels see it
  Node *node;
  int32_t *box, *live, *leaf_off, *pts;
  int64_t toff, size;     // first staging position, points
  int64_t from_cleared;   // records that come from cleared trees (first in the tree)
  int32_t h, pad_;
  unsigned long long *err;
  unsigned long long *skew;   // mapped host word for the sum of squared leaf sizes, or nullptr
};

struct SpGather {         // one source of a tree's points
  const int32_t *src;     // a cleared tree's records (live ones move), or nullptr: a pool chunk
  int64_t count;
  const int32_t *pbuf;    // pool chunk: the forest's pool (sorted buffer ids, then ids)
  int64_t pnbuf;
  const int32_t *parr;
  int64_t pfirst, pool_lo;
  const int32_t *idtab;
  int64_t dst0;           // pool chunk: first position inside its tree
  int32_t tree, pad_;
};

int64_t cdiv(int64_t a, int64_t b) { return (a + b - 1) / b; }
size_t al256(size_t x) { return (x + 255) / 256 * 256; }

__device__ __forceinline__ int find_entry(const int64_t *pre, int n, int64_t x) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (pre[mid] <= x) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

__device__ __forceinline__ void copy_rec(int32_t *dst, const int32_t *src, int rs) {
  for (int c = 0; c < rs; c += 4)
    *reinterpret_cast<int4 *>(dst + c) = *reinterpret_cast<const int4 *>(src + c);
}

// Gather: the live records of the cleared trees (any order) and the pool
// chunks (in order behind them) into staging -- or, for a tree that is a
// single leaf, straight into the tree.  Level-0 segment of a record = its tree.
__global__ void k_sp_gather(const SpGather *G, const int64_t *pre, int ng, const SpTree *T, int dim,
                            int32_t *stg, int32_t *seg, unsigned long long *cursor) {
  const int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int lane = threadIdx.x & 31;
  const bool act = x < pre[ng];
  const int j = act ? find_entry(pre, ng, x) : 0;
  const SpGather &g = G[j];
  const int64_t i = x - pre[j];
  const int rs = rec_ints(dim);
  int32_t r[rec_ints(kMaxDim)];
  bool keep = false;
  int tree = g.tree;
  if (act) {
    if (g.src) {
      const int32_t *src = g.src + i * rs;
      for (int c = 0; c < rs; ++c) r[c] = src[c];
      keep = r[dim] >= 0;               // tombstoned records stay behind
    } else {
      const int64_t k = g.pool_lo + i;
      const int32_t id = k < g.pnbuf ? g.pbuf[k] : (g.parr ? g.parr[k - g.pnbuf] : (int32_t)(g.pfirst + (k - g.pnbuf)));
      for (int c = 0; c < rs; ++c) r[c] = 0;
      for (int c = 0; c < dim; ++c) r[c] = g.idtab[(int64_t)id * dim + c];
      r[dim] = id;
      keep = true;
    }
  }
  // positions: cleared records take the next free slot of their tree (warp-
  // aggregated per tree), pool records a fixed slot after them
  int64_t pos = 0;
  const bool from_cleared = act && keep && g.src;
  const unsigned cm = __ballot_sync(0xffffffffu, from_cleared);
  if (from_cleared) {
    const unsigned peers = __match_any_sync(cm, tree);
    const int leader = __ffs(peers) - 1;
    unsigned long long base = 0;
    if (lane == leader) base = atomicAdd(&cursor[tree], (unsigned long long)__popc(peers));
    base = __shfl_sync(peers, base, leader);
    pos = (int64_t)base + __popc(peers & ((1u << lane) - 1));
  } else if (act && keep) {
    pos = g.dst0 + i;
  }
  if (!(act && keep)) return;
  const SpTree &tr = T[tree];
  if (pos < 0 || pos >= (g.src ? tr.from_cleared : tr.size)) {
    atomicOr(tr.err, kErrGather);
    return;
  }
  if (tr.h == 0) {
    for (int c = 0; c < rs; c += 4)
      *reinterpret_cast<int4 *>(tr.pts + pos * rs + c) = make_int4(r[c], r[c + 1], r[c + 2], r[c + 3]);
  } else {
    const int64_t p = tr.toff + pos;
    for (int c = 0; c < rs; c += 4)
      *reinterpret_cast<int4 *>(stg + p * rs + c) = make_int4(r[c], r[c + 1], r[c + 2], r[c + 3]);
    seg[p] = tree;
  }
}

// All levels of the new trees in one cooperative launch.
//
// A step's batch is a few microseconds of work per level, so three launches
// per level (clearing, scatter, split) and an upload per table were what it
// cost: 100K points into 1M 2-D ones, insert call 380 us, this way 306; 5,000
// into 100K 250 -> 170; builds of 100K and 1M 2-D points 328 -> 238 and 634 ->
// 567 us.  Large builds are bound by the records' gathers and scatters and
// want the warps: 10M 3-D points 3,705 us in launches, here 3,860 at four
// blocks per SM (58 registers), 3,580 at five, 3,222 at six and 3,345 at eight.
constexpr int kSpBlocks = 6;

struct SpLevels {
  const SpTree *T;
  const int64_t *seg_n;    // [hmax] segments of each level
  const int64_t *rec_n;    // [hmax] records still splitting at each level
  int ntree, dim, hmax;
  int32_t *stg[2], *seg[2];
  int32_t *mn[2], *mx[2];  // split-coordinate bounds of this level's and the next level's segments
  int64_t *lo[2];
  int32_t *n[2];
  uint32_t *curL, *curR;
  unsigned *bar;
  unsigned long long *err;
};

// First level's bounds from the records [p0, p0 + kT).
__device__ __forceinline__ void sp_minmax(const int32_t *stg, const int32_t *seg, int64_t p0, int64_t A, int rs,
                                          int c, int32_t *mn, int32_t *mx) {
  __shared__ int32_t s_mn[kT / 32], s_mx[kT / 32];
  const int64_t p = p0 + threadIdx.x;
  const bool act = p < A;
  const int s = act ? seg[p] : -1;
  const int32_t x = act ? stg[p * rs + c] : 0;
  const int s0 = seg[p0];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int32_t xl = act ? x : INT32_MAX, xh = act ? x : INT32_MIN;
  if (__syncthreads_and(!act || s == s0)) {
    // the whole block in one segment: one atomic pair
    const int32_t wl = __reduce_min_sync(0xffffffffu, xl), wh = __reduce_max_sync(0xffffffffu, xh);
    if (lane == 0) {
      s_mn[warp] = wl;
      s_mx[warp] = wh;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      int32_t a = s_mn[0], b = s_mx[0];
      for (int w = 1; w < kT / 32; ++w) {
        a = min(a, s_mn[w]);
        b = max(b, s_mx[w]);
      }
      atomicMin(&mn[s0], a);
      atomicMax(&mx[s0], b);
    }
    return;
  }
  const int ws = __shfl_sync(0xffffffffu, s, 0);
  if (__all_sync(0xffffffffu, !act || s == ws)) {
    const int32_t wl = __reduce_min_sync(0xffffffffu, xl), wh = __reduce_max_sync(0xffffffffu, xh);
    if (lane == 0 && ws >= 0) {
      atomicMin(&mn[ws], wl);
      atomicMax(&mx[ws], wh);
    }
    return;
  }
  if (act) {
    atomicMin(&mn[s], x);
    atomicMax(&mx[s], x);
  }
}

// The records [p0, p0 + kT) of level t.  Left records fill [lo, lo + nl) from
// the start, right ones [lo + nl, lo + m) from the end, so neither side needs
// the other's count first.
__device__ __forceinline__ void sp_scatter(const SpLevels &P, int t, int64_t p0, int64_t A) {
  const int dim = P.dim, c = t % dim;
  const int32_t *stg = P.stg[t & 1], *seg = P.seg[t & 1], *mn = P.mn[t & 1], *mx = P.mx[t & 1];
  int32_t *mn_next = P.mn[(t & 1) ^ 1], *mx_next = P.mx[(t & 1) ^ 1];
  const int64_t *lo = P.lo[t & 1];
  const int32_t *n = P.n[t & 1];
  uint32_t *curL = P.curL, *curR = P.curR;
  const SpTree *T = P.T;
  __shared__ uint32_t s_cnt[2][kT / 32];
  __shared__ uint32_t s_base[2];
  __shared__ int32_t s_bnd[4][kT / 32];   // per warp: left min, left max, right min, right max
  const int rs = rec_ints(dim);
  const int64_t p = p0 + threadIdx.x;
  const bool act = p < A;
  const int s = act ? seg[p] : -1;
  const int s0 = seg[p0];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int32_t x = act ? stg[p * rs + c] : 0;
  const bool left = act && x <= ((act ? mn[s] + mx[s] : 0) >> 1);
  const bool right = act && !left;
  const unsigned lt_mask = (1u << lane) - 1;
  // the next level's split coordinate, for the records whose children split on
  const int cn = (t + 1) % dim;
  const bool more = act && t + 2 <= T[s >> t].h;
  const int32_t xn = more ? stg[p * rs + cn] : 0;
  uint32_t rank = 0;
  if (__syncthreads_and(!act || s == s0)) {
    const unsigned bl = __ballot_sync(0xffffffffu, left), br = __ballot_sync(0xffffffffu, right);
    const int32_t lmn = __reduce_min_sync(0xffffffffu, more && left ? xn : INT32_MAX);
    const int32_t lmx = __reduce_max_sync(0xffffffffu, more && left ? xn : INT32_MIN);
    const int32_t rmn = __reduce_min_sync(0xffffffffu, more && right ? xn : INT32_MAX);
    const int32_t rmx = __reduce_max_sync(0xffffffffu, more && right ? xn : INT32_MIN);
    if (lane == 0) {
      s_cnt[0][warp] = __popc(bl);
      s_cnt[1][warp] = __popc(br);
      s_bnd[0][warp] = lmn;
      s_bnd[1][warp] = lmx;
      s_bnd[2][warp] = rmn;
      s_bnd[3][warp] = rmx;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      uint32_t tl = 0, tr = 0;
      int32_t a0 = INT32_MAX, a1 = INT32_MIN, a2 = INT32_MAX, a3 = INT32_MIN;
      for (int w = 0; w < kT / 32; ++w) {
        const uint32_t a = s_cnt[0][w], b = s_cnt[1][w];
        s_cnt[0][w] = tl;
        s_cnt[1][w] = tr;
        tl += a;
        tr += b;
        a0 = min(a0, s_bnd[0][w]);
        a1 = max(a1, s_bnd[1][w]);
        a2 = min(a2, s_bnd[2][w]);
        a3 = max(a3, s_bnd[3][w]);
      }
      s_base[0] = tl ? atomicAdd(&curL[s0], tl) : 0;
      s_base[1] = tr ? atomicAdd(&curR[s0], tr) : 0;
      if (a0 <= a1) {
        atomicMin(&mn_next[2 * s0], a0);
        atomicMax(&mx_next[2 * s0], a1);
      }
      if (a2 <= a3) {
        atomicMin(&mn_next[2 * s0 + 1], a2);
        atomicMax(&mx_next[2 * s0 + 1], a3);
      }
    }
    __syncthreads();
    rank = left ? s_base[0] + s_cnt[0][warp] + __popc(bl & lt_mask)
                : s_base[1] + s_cnt[1][warp] + __popc(br & lt_mask);
  } else {
    // groups of lanes with the same (segment, side)
    const int key = act ? 2 * s + (left ? 0 : 1) : -1 - lane;
    const unsigned peers = __match_any_sync(0xffffffffu, key);
    const int leader = __ffs(peers) - 1;
    uint32_t base = 0;
    if (act && lane == leader) base = atomicAdd(left ? &curL[s] : &curR[s], (uint32_t)__popc(peers));
    base = __shfl_sync(0xffffffffu, base, leader);
    rank = base + __popc(peers & lt_mask);
    // the group's bounds of the next coordinate (every lane of a group is in
    // the same tree, so `more` is the same for all of them)
    const int32_t gmn = __reduce_min_sync(peers, more ? xn : INT32_MAX);
    const int32_t gmx = __reduce_max_sync(peers, more ? xn : INT32_MIN);
    if (more && lane == leader) {
      atomicMin(&mn_next[2 * s + (left ? 0 : 1)], gmn);
      atomicMax(&mx_next[2 * s + (left ? 0 : 1)], gmx);
    }
  }
  if (!act) return;
  const int j = s >> t;
  const SpTree &tr = T[j];
  const int64_t m = n[s];
  if ((int64_t)rank >= m) {
    atomicOr(tr.err, kErrPartition);
    return;
  }
  const int64_t pos = left ? lo[s] + rank : lo[s] + m - 1 - rank;
  if (t + 1 == tr.h) {                    // the children are leaves: into the tree
    copy_rec(tr.pts + (pos - tr.toff) * rs, stg + p * rs, rs);
  } else {
    copy_rec(P.stg[(t & 1) ^ 1] + pos * rs, stg + p * rs, rs);
    P.seg[(t & 1) ^ 1][pos] = 2 * s + (left ? 0 : 1);
  }
}

// Segment s of level t: the node's key and children, the children's bounds for
// the next level, or the leaves' offsets and records when the children are
// leaves.
__device__ __forceinline__ void sp_split(const SpLevels &P, int t, int64_t s) {
  const int j = (int)(s >> t);
  const int64_t i = s & (((int64_t)1 << t) - 1);
  const SpTree &tr = P.T[j];
  const int64_t lo = P.lo[t & 1][s], m = P.n[t & 1][s];
  const int64_t nl = P.curL[s];
  if (nl + (int64_t)P.curR[s] != m) atomicOr(tr.err, kErrPartition);
  const int64_t v = m > 0 ? ((int64_t)P.mn[t & 1][s] + (int64_t)P.mx[t & 1][s]) >> 1 : 0;
  const int l = tr.h + 1;
  const int cl = veb_slot32(l, t + 1, 2 * (int)i), cr = veb_slot32(l, t + 1, 2 * (int)i + 1);
  tr.node[veb_slot32(l, t, (int)i)] = Node{(uint64_t)((v << 31) | 0x7FFFFFFF), cl, cr};
  if (t + 1 == tr.h) {
    tr.leaf_off[2 * i] = (int32_t)(lo - tr.toff);
    tr.leaf_off[2 * i + 1] = (int32_t)(lo + nl - tr.toff);
    tr.node[cl] = Node{0, (int32_t)(-1 - 2 * i), 0};
    tr.node[cr] = Node{0, (int32_t)(-2 - 2 * i), 0};
  } else {
    int64_t *lo_next = P.lo[(t & 1) ^ 1];
    int32_t *n_next = P.n[(t & 1) ^ 1];
    lo_next[2 * s] = lo;
    n_next[2 * s] = (int32_t)nl;
    lo_next[2 * s + 1] = lo + nl;
    n_next[2 * s + 1] = (int32_t)(m - nl);
  }
}

__global__ void __launch_bounds__(kT, kSpBlocks) k_sp_levels(const __grid_constant__ SpLevels P) {
  const int64_t t0 = (int64_t)blockIdx.x * kT + threadIdx.x, step = (int64_t)gridDim.x * kT;
  const int64_t r0 = (int64_t)blockIdx.x * kT;   // the block's first record, a multiple of kT (whole blocks go on)
  auto clear_cursors = [&](int64_t s) {
    P.curL[s] = 0;
    P.curR[s] = 0;
  };
  auto clear_bounds = [&](int t, int64_t s) {
    P.mn[t & 1][s] = INT32_MAX;
    P.mx[t & 1][s] = INT32_MIN;
  };
  // bounds of every splitting tree; the leaf-offset sentinels; the single leaf
  // of a tree with h = 0
  for (int64_t j = t0; j < P.ntree; j += step) {
    const SpTree &tr = P.T[j];
    tr.leaf_off[(int64_t)1 << tr.h] = (int32_t)tr.size;
    if (tr.h == 0) {
      tr.leaf_off[0] = 0;
      tr.node[0] = Node{0, -1, 0};
    } else {
      P.lo[0][j] = tr.toff;
      P.n[0][j] = (int32_t)tr.size;
      clear_cursors(j);
    }
  }
  if (P.hmax == 0) return;
  for (int t = 0; t < min(P.hmax, 2); ++t)
    for (int64_t s = t0; s < P.seg_n[t]; s += step) clear_bounds(t, s);
  unsigned epoch = 0;
  grid_barrier(P.bar, epoch, P.err);
  for (int64_t p = r0; p < P.rec_n[0]; p += step)
    sp_minmax(P.stg[0], P.seg[0], p, P.rec_n[0], rec_ints(P.dim), 0, P.mn[0], P.mx[0]);
  for (int t = 0; t < P.hmax; ++t) {
    grid_barrier(P.bar, epoch, P.err);
    const int64_t A = P.rec_n[t], N = P.seg_n[t];
    for (int64_t p = r0; p < A; p += step) sp_scatter(P, t, p, A);
    grid_barrier(P.bar, epoch, P.err);
    // a thread clears for the next levels what it alone reads here (s), and
    // the places behind N, which nobody reads here: a level has at most twice
    // the segments of the one before it
    const int64_t N1 = t + 1 < P.hmax ? P.seg_n[t + 1] : 0, N2 = t + 2 < P.hmax ? P.seg_n[t + 2] : 0;
    for (int64_t s = t0; s < N; s += step) {
      sp_split(P, t, s);
      for (int64_t i = s; i < N1; i += N) clear_cursors(i);
      for (int64_t i = s; i < N2; i += N) clear_bounds(t, i);
    }
  }
}

// Boxes and live counts: every leaf from its points, then the nodes of depth
// t = hmax - 1 .. 0 from their children, in one cooperative launch (a grid
// barrier between depths; one launch per depth took about 3 us each, 17 of
// them for a tree of 2^16 leaves).  An empty leaf gets the empty box
// [INT32_MAX, INT32_MIN].
//
// A warp takes 32 leaves: a lane its own leaf where that holds at most
// kLaneLeaf points, the whole warp the others in turn.  The rule bounds the
// depth and not the leaves, so clustered points leave leaves of thousands,
// and a lane per leaf took as long as the largest one.  1M 2-D points of 100
// clusters, a batch of 100K inserted and the buffer's tree: 1,121 us in 24
// launches, this way 174 in two.  Points in one place, or nearly, leave a leaf
// of any size: those of more than kHugeLeaf points are listed and dealt to
// all warps in pieces, so that the other blocks never wait at a barrier for
// one warp to go through a leaf of millions.
constexpr int kLaneLeaf = 32;
constexpr int kHugeLeaf = 8192;

struct HugeLeaf {
  int32_t tree, leaf;
};

struct SpBoxParams {
  const SpTree *T;
  const int64_t *leaf_pre;  // [ntree + 1] prefix of the trees' leaves
  const int64_t *depth;     // [hmax] nodes of each depth over the trees that have it
  unsigned long long *sq;   // [ntree] sum of the squared leaf sizes (zeroed)
  HugeLeaf *huge;           // the leaves of more than kHugeLeaf points ...
  unsigned *nhuge;          // ... and their number (zeroed)
  int ntree, dim, hmax;
  int one;                  // depths 0 .. one - 1 are one block's (one_block_depths)
  unsigned *bar;
  unsigned long long *err;
};

// Smallest and largest of x[r * rs] over [a, b), by a whole warp.
__device__ __forceinline__ void warp_extent(const int32_t *x, int rs, int64_t a, int64_t b, int32_t &lo, int32_t &hi) {
  lo = INT32_MAX;
  hi = INT32_MIN;
#pragma unroll 4
  for (int64_t r = a + (threadIdx.x & 31); r < b; r += 32) {
    const int32_t y = x[r * rs];
    lo = min(lo, y);
    hi = max(hi, y);
  }
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
}

__device__ __forceinline__ void sp_leaf_boxes(const SpBoxParams &P, int64_t x0) {
  const int lane = threadIdx.x & 31, dim = P.dim, rs = rec_ints(dim);
  const int64_t x = x0 + lane;
  const bool act = x < P.leaf_pre[P.ntree];
  const int j = act ? find_entry(P.leaf_pre, P.ntree, x) : 0;
  const SpTree &tr = P.T[j];
  const int64_t leaf = act ? x - P.leaf_pre[j] : 0;
  int64_t a = 0, b = 0, v = 0;
  bool ok = act;
  if (act) {
    a = tr.leaf_off[leaf];
    b = tr.leaf_off[leaf + 1];
    v = veb_slot32(tr.h + 1, tr.h, (int)leaf);
    if (a < 0 || b > tr.size || a > b) {
      atomicOr(tr.err, kErrLeaf);
      ok = false;
    }
  }
  const bool own = ok && b - a <= kLaneLeaf;
  for (int c = 0; c < dim; ++c) {
    if (!own) continue;
    int32_t lo = INT32_MAX, hi = INT32_MIN;
    for (int64_t r = a; r < b; ++r) {
      const int32_t y = tr.pts[r * rs + c];
      lo = min(lo, y);
      hi = max(hi, y);
    }
    tr.box[v * 2 * dim + c] = lo;
    tr.box[v * 2 * dim + dim + c] = hi;
  }
  if (ok) tr.live[v] = (int32_t)(b - a);
  unsigned long long sq = ok ? (unsigned long long)((b - a) * (b - a)) : 0;
  const int j0 = __shfl_sync(0xffffffffu, j, 0);   // (every lane takes part in every warp operation)
  if (__all_sync(0xffffffffu, !act || j == j0)) {
    for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
    if (lane == 0) atomicAdd(&P.sq[j], sq);
  } else if (ok) {
    atomicAdd(&P.sq[j], sq);
  }
  const bool huge = ok && b - a > kHugeLeaf;
  if (huge) {
    for (int c = 0; c < dim; ++c) {
      tr.box[v * 2 * dim + c] = INT32_MAX;
      tr.box[v * 2 * dim + dim + c] = INT32_MIN;
    }
    P.huge[atomicAdd(P.nhuge, 1u)] = HugeLeaf{j, (int32_t)leaf};
  }
  unsigned big = __ballot_sync(0xffffffffu, ok && !own && !huge);
  while (big) {
    const int src = __ffs(big) - 1;
    big &= big - 1;
    const SpTree &w = P.T[__shfl_sync(0xffffffffu, j, src)];
    const int64_t wa = __shfl_sync(0xffffffffu, a, src), wb = __shfl_sync(0xffffffffu, b, src),
                  wv = __shfl_sync(0xffffffffu, v, src);
    for (int c = 0; c < dim; ++c) {
      int32_t lo, hi;
      warp_extent(w.pts + c, rs, wa, wb, lo, hi);
      if (lane == 0) {
        w.box[wv * 2 * dim + c] = lo;
        w.box[wv * 2 * dim + dim + c] = hi;
      }
    }
  }
}

// The listed leaves' boxes, empty so far, from their points: kHugeLeaf at a
// time, the pieces of all leaves one after another to the grid's warps.
__device__ __forceinline__ void sp_huge_leaf_boxes(const SpBoxParams &P, unsigned nhuge) {
  const int lane = threadIdx.x & 31, dim = P.dim, rs = rec_ints(dim);
  const int64_t nwarp = (int64_t)gridDim.x * (kT / 32), warp = (int64_t)blockIdx.x * (kT / 32) + (threadIdx.x >> 5);
  int64_t first = 0;   // the warp that takes the next leaf's first piece
  for (unsigned e = 0; e < nhuge; ++e) {
    const HugeLeaf H = P.huge[e];
    const SpTree &tr = P.T[H.tree];
    const int64_t a = tr.leaf_off[H.leaf], b = tr.leaf_off[H.leaf + 1], n = (b - a + kHugeLeaf - 1) / kHugeLeaf;
    const int64_t v = veb_slot32(tr.h + 1, tr.h, H.leaf);
    for (int64_t i = warp >= first ? warp - first : warp - first + nwarp; i < n; i += nwarp) {
      const int64_t p = a + i * kHugeLeaf;
      for (int c = 0; c < dim; ++c) {
        int32_t lo, hi;
        warp_extent(tr.pts + c, rs, p, min(p + kHugeLeaf, b), lo, hi);
        if (lane == 0) {
          atomicMin(&tr.box[v * 2 * dim + c], lo);
          atomicMax(&tr.box[v * 2 * dim + dim + c], hi);
        }
      }
    }
    first = (first + n) % nwarp;
  }
}

__global__ void __launch_bounds__(kT) k_sp_boxes(const SpBoxParams P) {
  const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
  for (int64_t x = t0 & ~(int64_t)31; x < P.leaf_pre[P.ntree]; x += step) sp_leaf_boxes(P, x);
  const int dim = P.dim;
  auto node = [&](int t, int64_t s) {
    const SpTree &tr = P.T[s >> t];
    const int i = (int)(s & (((int64_t)1 << t) - 1));
    const int l = tr.h + 1;
    const int64_t v = veb_slot32(l, t, i), a = veb_slot32(l, t + 1, 2 * i), b = veb_slot32(l, t + 1, 2 * i + 1);
    for (int c = 0; c < dim; ++c) {
      tr.box[v * 2 * dim + c] = min(tr.box[a * 2 * dim + c], tr.box[b * 2 * dim + c]);
      tr.box[v * 2 * dim + dim + c] = max(tr.box[a * 2 * dim + dim + c], tr.box[b * 2 * dim + dim + c]);
    }
    tr.live[v] = tr.live[a] + tr.live[b];
    if (t == 0 && tr.skew) *tr.skew = P.sq[s];   // to the host, whenever it arrives (a hint)
  };
  unsigned epoch = 0;
  grid_barrier(P.bar, epoch, P.err);
  const unsigned nhuge = *P.nhuge;   // (final: every leaf has been looked at)
  if (nhuge > 0) {
    sp_huge_leaf_boxes(P, nhuge);
    grid_barrier(P.bar, epoch, P.err);
  }
  int t = P.hmax - 1;
  for (; t >= P.one; --t) {
    for (int64_t s = t0; s < P.depth[t]; s += step) node(t, s);
    grid_barrier(P.bar, epoch, P.err);
  }
  if (blockIdx.x > 0) return;
  for (; t >= 0; --t) {
    for (int64_t s = threadIdx.x; s < P.depth[t]; s += blockDim.x) node(t, s);
    __syncthreads();
  }
}

}  // namespace

int build_trees_spatial(bdl_forest *af, int dim, std::vector<BuildTree> &bt, const std::vector<ClearedSrc> &cl,
                        cudaStream_t s) {
  if (bt.empty()) return BDL_OK;
  const int ntree = (int)bt.size();
  // trees by height, tallest first: the trees still splitting at a level are a prefix
  std::vector<int> order(ntree);
  std::iota(order.begin(), order.end(), 0);
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return bt[a].h > bt[b].h; });
  std::vector<int> rank_of(ntree);
  for (int r = 0; r < ntree; ++r) rank_of[order[r]] = r;
  std::vector<SpTree> tr(ntree);
  int64_t S = 0;
  int hmax = 0;
  for (int r = 0; r < ntree; ++r) {
    const BuildTree &b = bt[order[r]];
    SpTree &x = tr[r];
    memset(&x, 0, sizeof(x));
    x.node = b.tree->node;
    x.box = b.tree->box;
    x.live = b.tree->live_nodes;
    x.leaf_off = b.tree->leaf_off;
    x.pts = b.tree->pts;
    x.size = b.s;
    x.from_cleared = b.from_cleared;
    x.h = b.h;
    x.err = b.err;
    x.skew = b.skew;
    x.toff = S;
    if (b.h > 0) S += b.s;
    hmax = std::max(hmax, b.h);
  }
  std::vector<int> nact(hmax + 1, 0);     // trees still splitting at level t
  for (int t = 0; t <= hmax; ++t)
    for (int r = 0; r < ntree; ++r)
      if (tr[r].h > t) nact[t]++;
  int64_t Nmax = 1, leaves = 0;
  for (int t = 0; t < hmax; ++t) Nmax = std::max(Nmax, (int64_t)nact[t] << t);
  std::vector<int64_t> leaf_pre(1, 0);
  for (int r = 0; r < ntree; ++r) leaf_pre.push_back(leaf_pre.back() + ((int64_t)1 << tr[r].h));
  leaves = leaf_pre.back();
  // gather sources: cleared trees' records, then each tree's pool chunk
  std::vector<SpGather> ga;
  std::vector<int64_t> gpre(1, 0);
  for (const ClearedSrc &c : cl) {
    SpGather g;
    memset(&g, 0, sizeof(g));
    g.src = c.pts;
    g.count = c.size;
    g.tree = rank_of[c.dst];
    ga.push_back(g);
    gpre.push_back(gpre.back() + c.size);
  }
  for (int k = 0; k < ntree; ++k) {
    const BuildTree &b = bt[k];
    SpGather g;
    memset(&g, 0, sizeof(g));
    g.count = b.s - b.from_cleared;
    g.pbuf = b.pool.buf;
    g.pnbuf = b.pool.nbuf;
    g.parr = b.pool.arr;
    g.pfirst = b.pool.first;
    g.pool_lo = b.pool_lo;
    g.idtab = b.idtab;
    g.dst0 = b.from_cleared;
    g.tree = rank_of[k];
    ga.push_back(g);
    gpre.push_back(gpre.back() + g.count);
  }
  // ---- one device block: staging, per-level arrays, tables ----
  const int rs = rec_ints(dim);
  const size_t b_stg = al256((size_t)std::max<int64_t>(S, 1) * rs * 4);
  const size_t b_seg = al256((size_t)std::max<int64_t>(S, 1) * 4);
  const size_t b_i32 = al256((size_t)Nmax * 4), b_i64 = al256((size_t)Nmax * 8);
  const size_t b_tr = al256(ntree * sizeof(SpTree)), b_ga = al256(ga.size() * sizeof(SpGather));
  const size_t b_gpre = al256(gpre.size() * 8), b_lpre = al256(leaf_pre.size() * 8);
  // zeroed: gather cursors, sums of squared leaf sizes, the two barriers, the number of huge leaves
  const size_t b_cur = 2 * al256((size_t)ntree * 8) + 256;
  std::vector<int64_t> depth(std::max(hmax, 1), 0);
  std::vector<int64_t> recs(depth.size(), 0);   // records still splitting at each level
  for (int t = 0; t < hmax; ++t) {
    depth[t] = (int64_t)nact[t] << t;
    recs[t] = tr[nact[t] - 1].toff + tr[nact[t] - 1].size;
  }
  const size_t b_depth = al256(depth.size() * 8);
  std::vector<TreeSeg> pk;
  std::vector<int64_t> pk_pre;
  {
    std::vector<Tree *> trees;
    for (auto &b : bt) trees.push_back(b.tree);
    pack_nodes_entries(trees, dim, pk, pk_pre);
  }
  const size_t b_pk = al256(pk.size() * sizeof(TreeSeg)), b_pkpre = al256(pk_pre.size() * 8);
  const size_t total = 2 * b_stg + 2 * b_seg + 6 * b_i32 + 2 * (b_i64 + b_i32) + b_tr + b_ga + b_gpre + b_lpre +
                       b_cur + b_pk + b_pkpre + 2 * b_depth;
  void *block = nullptr;
  int st = dev_alloc(af, &block, total, s);
  if (st) return st;
  unsigned char *p = (unsigned char *)block;
  auto take = [&](size_t bytes) {
    void *q = p;
    p += bytes;
    return q;
  };
  int32_t *stg[2], *seg[2];
  stg[0] = (int32_t *)take(b_stg);
  stg[1] = (int32_t *)take(b_stg);
  seg[0] = (int32_t *)take(b_seg);
  seg[1] = (int32_t *)take(b_seg);
  int32_t *mn[2], *mx[2];   // split-coordinate bounds of this level's and the next level's segments
  mn[0] = (int32_t *)take(b_i32);
  mx[0] = (int32_t *)take(b_i32);
  mn[1] = (int32_t *)take(b_i32);
  mx[1] = (int32_t *)take(b_i32);
  uint32_t *curL = (uint32_t *)take(b_i32), *curR = (uint32_t *)take(b_i32);
  int64_t *lo[2];
  int32_t *nn[2];
  lo[0] = (int64_t *)take(b_i64);
  nn[0] = (int32_t *)take(b_i32);
  lo[1] = (int64_t *)take(b_i64);
  nn[1] = (int32_t *)take(b_i32);
  // the tables, in one upload
  std::vector<unsigned char> img;
  unsigned char *const tables = p;
  auto table = [&](const void *src, size_t bytes, size_t room) {
    img.resize((size_t)(p - tables) + bytes);
    if (bytes) memcpy(img.data() + (p - tables), src, bytes);
    return take(room);
  };
  SpTree *d_tr = (SpTree *)table(tr.data(), ntree * sizeof(SpTree), b_tr);
  SpGather *d_ga = (SpGather *)table(ga.data(), ga.size() * sizeof(SpGather), b_ga);
  int64_t *d_gpre = (int64_t *)table(gpre.data(), gpre.size() * 8, b_gpre);
  int64_t *d_lpre = (int64_t *)table(leaf_pre.data(), leaf_pre.size() * 8, b_lpre);
  int64_t *d_depth = (int64_t *)table(depth.data(), depth.size() * 8, b_depth);
  int64_t *d_recs = (int64_t *)table(recs.data(), recs.size() * 8, b_depth);
  TreeSeg *d_pk = (TreeSeg *)table(pk.data(), pk.size() * sizeof(TreeSeg), b_pk);
  int64_t *d_pkpre = (int64_t *)table(pk_pre.data(), pk_pre.size() * 8, b_pkpre);
  unsigned long long *cursor = (unsigned long long *)take(b_cur);
  unsigned long long *sq = (unsigned long long *)((char *)cursor + al256((size_t)ntree * 8));
  unsigned *bar = (unsigned *)((char *)cursor + 2 * al256((size_t)ntree * 8));   // [0] and [32]; [16]: huge leaves
  st = h2d_and_zero(tables, img.data(), img.size(), cursor, b_cur, s);
  if (st) {
    dev_free(af, block, total, s);
    return st;
  }
  // ---- gather, levels ----
  if (gpre.back() > 0) {
    KScope ks_(kK_sp_gather, s);
    k_sp_gather<<<(unsigned)cdiv(gpre.back(), kT), kT, 0, s>>>(d_ga, d_gpre, (int)ga.size(), d_tr, dim, stg[0],
                                                               seg[0], cursor);
  }
  {
    SpLevels P;
    P.T = d_tr;
    P.seg_n = d_depth;
    P.rec_n = d_recs;
    P.ntree = ntree;
    P.dim = dim;
    P.hmax = hmax;
    for (int i = 0; i < 2; ++i) {
      P.stg[i] = stg[i];
      P.seg[i] = seg[i];
      P.mn[i] = mn[i];
      P.mx[i] = mx[i];
      P.lo[i] = lo[i];
      P.n[i] = nn[i];
    }
    P.curL = curL;
    P.curR = curR;
    P.bar = bar + 32;
    P.err = bt[0].err;
    st = launch_coop((const void *)k_sp_levels, kT, std::max<int64_t>(S, ntree), &P, kK_sp_levels, 0, s);
  }
  // ---- boxes, live counts, packed records ----
  {
    SpBoxParams P;
    P.T = d_tr;
    P.leaf_pre = d_lpre;
    P.depth = d_depth;
    P.sq = sq;
    P.huge = (HugeLeaf *)stg[0];   // (staging is free again; S / kHugeLeaf entries at most)
    P.nhuge = bar + 16;
    P.ntree = ntree;
    P.dim = dim;
    P.hmax = hmax;
    P.one = one_block_depths(depth.data(), hmax);
    P.bar = bar;
    P.err = bt[0].err;
    if (!st) st = launch_coop((const void *)k_sp_boxes, kT, leaves, &P, kK_sp_box, 0, s);
  }
  launch_pack_nodes(d_pk, d_pkpre, (int)pk.size(), pk_pre.back(), s);
  const int err = st ? st : cuda_check(cudaGetLastError(), "spatial build kernels");
  dev_free(af, block, total, s);
  return err;
}

}  // namespace bdl
