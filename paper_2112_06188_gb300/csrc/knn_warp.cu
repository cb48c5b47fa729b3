// knn_warp.cu -- kNN_L (Alg. 5) with one warp per query.
//
// The thread-per-query kernel (knn.cu) walks one query's tree nodes and leaf
// points one after another in one lane: a small batch leaves most of the GPU
// idle and waits for the longest such chain.  Here the 32 lanes of a warp work
// on one query together:
//  * a node round takes up to eight records off the query's stack at once and
//    gives each of their 32 entries to a lane (box distance, prune test);
//  * a leaf round gives 32 leaf points, of up to four leaves, a lane each;
//  * the k <= 32 best candidates live in registers, lane i holding the i-th
//    best; a few candidates enter one by one by a ballot (the rank) and a
//    shift, more than ten are sorted across the warp and merged;
//  * all trees of the forest are walked together: the stack starts with every
//    tree's root, the largest tree's on top, and an entry names its tree;
//  * a warp that answers several queries one after another starts each but the
//    first with a bound: the k neighbours just found are k live points, so the
//    next query's k-th distance is at most its distance to the farthest of
//    them.  A walk whose bound were the true k-th distance from the start
//    would take 25 to 36% less; this way it takes 3 to 19% less (below);
//  * while there is no bound, a node round takes two records only: what it
//    takes beside the nearest is mostly what the first leaves rule out.
// The answer does not depend on the order of the walk: every subtree whose
// box is not strictly farther than the k-th distance is visited, and the k
// best by (d2, id) of all points seen are unique.
//
// What bounds it: small batches by the chain of about 2 x 20 rounds per query
// (a dependent L2 read each); large ones by instruction issue (about 3,900
// warp instructions per query on 2M 3-D points, 9,500 on 2M 7-D ones, 67 to
// 75% of the issue slots) and by the shared/L1 data pipe (53 to 59%).
// Measured against the thread-per-query kernel as it was when this one came,
// whole calls: 1M 5-D points, k = 10, 316 queries 1,212 -> 51 us (the kernel 43 to
// 67 by the inputs: its longest chain); 50K 16-D points, k = 8, 1,000 queries 1,526
// -> 48; 500K 4-D points, k = 32, 100K queries 3,644 -> 779; 10M 7-D points of 100
// clusters, k = 5, 1M queries 31.4 -> 17.9 ms.
// Without the starting bound and the narrow first rounds, and with them, in one
// run: those four 50.5 -> 47, 55 -> 52, 840 -> 768 us and 20.3 -> 17.8 ms; 10M 3-D
// points, k = 10, 30K queries 235 -> 202 us; 1M 2-D points of 100 clusters, spatial
// median, k = 5, 100K queries 1,057 -> 865 us.
#include "bdl_internal.cuh"

#include <algorithm>
#include <cmath>

namespace bdl {

namespace {

constexpr int kWarpsPerBlock = 4;
constexpr int kWLeaves = 80;    // leaf stack entries per warp
constexpr int kWTrees = kMaxLevel + 1;
constexpr float kWBoundUp = 1.00000393390655517578125f;   // see TopK in knn.cu

// What a walk needs of a tree.
struct WTree {
  const int32_t *pk, *pts, *leaf_off;
  int64_t size;
  int32_t nrec, nleaf;
};

struct __align__(16) WarpMem {
  int32_t q[kMaxDim];        // the query
  uint64_t node[kWStack];    // (box distance bits, low 6 bits: tree) << 32 | record
  uint64_t leaf[kWLeaves];   // (box distance bits, low 6 bits: tree) << 32 | leaf
  uint64_t sel[8];           // the records of this round
};

// The k best candidates, lane i holding the i-th of the best 32.
struct WarpTop {
  uint64_t d;
  int32_t id;
  float kdf;       // pruning bound: k-th distance rounded up, scaled up (see box_dist_f in knn.cu)
  uint64_t kd;     // k-th pair
  int32_t kid;
  float cap;       // a bound known beforehand, in the form of kdf
};

__device__ __forceinline__ void top_bound(WarpTop &b, int k) {
  b.kd = __shfl_sync(0xffffffffu, b.d, k - 1);
  b.kid = __shfl_sync(0xffffffffu, b.id, k - 1);
  b.kdf = b.kd == ~0ull ? b.cap : fminf(b.cap, __fmul_ru(__ull2float_ru(b.kd), kWBoundUp));
}

__device__ __forceinline__ bool pair_less(uint64_t d, int32_t i, uint64_t e, int32_t j) {
  return d < e || (d == e && i < j);
}

// The candidates (d, id) of the lanes with `have` join the list.
__device__ __forceinline__ void top_add(WarpTop &b, int k, bool have, uint64_t d, int32_t id) {
  const int lane = threadIdx.x & 31;
  unsigned mask = __ballot_sync(0xffffffffu, have);
  if (!mask) return;
  if (__popc(mask) > 10) {
    // many at once: sort them across the warp, then merge the two sorted
    // lists (the smaller of element i and element 31 - i, a bitonic sequence)
    const bool empty = __shfl_sync(0xffffffffu, b.d, 0) == ~0ull;
    if (!have) {
      d = ~0ull;
      id = INT32_MAX;
    }
#pragma unroll
    for (int size = 2; size <= 64; size <<= 1) {
      if (size == 64) {
        if (empty) break;
        const uint64_t rd = __shfl_xor_sync(0xffffffffu, d, 31);
        const int32_t ri = __shfl_xor_sync(0xffffffffu, id, 31);
        const bool mine = pair_less(b.d, b.id, rd, ri);
        d = mine ? b.d : rd;
        id = mine ? b.id : ri;
      }
#pragma unroll
      for (int stride = size == 64 ? 16 : size >> 1; stride > 0; stride >>= 1) {
        const uint64_t od = __shfl_xor_sync(0xffffffffu, d, stride);
        const int32_t oi = __shfl_xor_sync(0xffffffffu, id, stride);
        const bool up = size >= 32 || (lane & size) == 0;
        const bool keep_min = ((lane & stride) == 0) == up;
        if (pair_less(od, oi, d, id) == keep_min) {
          d = od;
          id = oi;
        }
      }
    }
    b.d = d;
    b.id = id;
  } else {
    do {
      const int src = __ffs(mask) - 1;
      mask &= mask - 1;
      const uint64_t cd = __shfl_sync(0xffffffffu, d, src);
      const int32_t ci = __shfl_sync(0xffffffffu, id, src);
      const bool less = pair_less(b.d, b.id, cd, ci);
      const int pos = __popc(__ballot_sync(0xffffffffu, less));
      const uint64_t ud = __shfl_up_sync(0xffffffffu, b.d, 1);
      const int32_t ui = __shfl_up_sync(0xffffffffu, b.id, 1);
      if (!less) {
        b.d = lane == pos ? cd : ud;
        b.id = lane == pos ? ci : ui;
      }
    } while (mask);
  }
  top_bound(b, k);
}

// Query row qi of job J against the nt trees of the table (smallest first), then
// the buffer.  Called by a whole warp.  `near_id`: lane i < k comes with the id of
// a live point of the forest (all k different), or some lane with -1, and
// leaves with the query's i-th neighbour, or -1.
template <int D>
__device__ __forceinline__ void warp_query(const KnnJob &J, WarpMem &W, const WTree *tree, int nt,
                                           int64_t qi, int k, int32_t &near_id) {
  constexpr int DM = D ? D : kMaxDim;
  const int dim = D ? D : J.dim;
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1;
  const float kInf = __int_as_float(0x7f800000);
  __syncwarp();
  if (lane < dim) W.q[lane] = J.q[qi * dim + lane];
  __syncwarp();
  // the query as floats 2^23 + x, exact for |x| < 2^23; farther off the grid its
  // two roundings are below 4.6 * 2^-24 of any gap to the grid, which with the
  // sum's own (d + 1) * 2^-24 stays inside kWBoundUp's 2^-18
  float q[DM];
#pragma unroll
  for (int c = 0; c < DM; ++c)
    if (c < dim) q[c] = (float)W.q[c] + kBiasF;
  float cap = kInf;
  if (__all_sync(0xffffffffu, lane >= k || near_id >= 0)) {
    uint64_t s = 0;
    if (lane < k) {
      const int32_t *p = J.idtab + (int64_t)near_id * dim;
#pragma unroll
      for (int c = 0; c < DM; ++c)
        if (c < dim) {
          const int32_t g = W.q[c] - p[c];
          s += (uint64_t)((int64_t)g * g);
        }
    }
    const float f = __fmul_ru(__ull2float_ru(s), kWBoundUp);   // (not negative: ordered as its bits)
    cap = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(f)));
  }
  WarpTop best;
  best.d = ~0ull;
  best.id = INT32_MAX;
  best.kd = ~0ull;
  best.kid = INT32_MAX;
  best.kdf = best.cap = cap;
  int sp = 0, ls = 0;
  // the roots, largest tree last (on top), at distance zero: a root is seldom
  // pruned, and its box would be a read that everything waits for
  for (int b = 0; b < nt; b += 32) {
    const int ti = b + lane;
    const bool ok = ti < nt, leaf = ok && tree[ti].nrec == 0;
    const uint64_t e = (uint64_t)(unsigned)ti << 32;
    const unsigned nm = __ballot_sync(0xffffffffu, ok && !leaf), lm = __ballot_sync(0xffffffffu, ok && leaf);
    if (ok && !leaf) W.node[sp + __popc(nm & lt)] = e;
    if (ok && leaf) W.leaf[ls + __popc(lm & lt)] = e;
    sp += __popc(nm);
    ls += __popc(lm);
  }
  __syncwarp();
  const int rs = rec_ints(dim), rec = packed_node_ints(dim);
  while (sp > 0 || ls > 0) {
    // ---- leaf rounds: the points of up to four leaves, 32 at a time ----
    while (ls >= 2 || (sp == 0 && ls > 0)) {
      const int nl = min(ls, 4);
      uint32_t key = 0;    // box distance bits, low 6 bits: tree
      int pa = 0, n = 0;
      if (lane < nl) {
        const uint64_t e = W.leaf[ls - 1 - lane];
        key = (uint32_t)(e >> 32);
        if (!(__uint_as_float(key & ~63u) > best.kdf)) {
          const WTree &T = tree[key & 63u];
          const uint32_t lf = (uint32_t)e;
          int pz = 0;
          unsigned long long bad = kErrChild;
          if (lf < (uint32_t)T.nleaf) {
            pa = T.leaf_off[lf];
            pz = T.leaf_off[lf + 1];
            bad = pa < 0 || pz > T.size || pa > pz ? kErrLeaf : 0;
          }
          if (bad) atomicOr(J.err, bad);
          else n = pz - pa;
        }
      }
      ls -= nl;
      // each leaf's first place among the round's points
      int inc = n;
      int y = __shfl_up_sync(0xffffffffu, inc, 1);
      if (lane >= 1) inc += y;
      y = __shfl_up_sync(0xffffffffu, inc, 2);
      if (lane >= 2) inc += y;
      const int total = __shfl_sync(0xffffffffu, inc, 3);
      const int start = inc - n;
      const int s1 = __shfl_sync(0xffffffffu, start, 1);
      const int s2 = __shfl_sync(0xffffffffu, start, 2);
      const int s3 = __shfl_sync(0xffffffffu, start, 3);
      const int off = pa - start;
      for (int b = 0; b < total; b += 32) {
        const int x = b + lane;
        const int own = (x >= s1) + (x >= s2) + (x >= s3);
        const int po = __shfl_sync(0xffffffffu, off, own) + x;
        const uint32_t pk = __shfl_sync(0xffffffffu, key, own);
        bool have = false;
        uint64_t s = 0;
        int32_t id = 0;
        if (x < total && !(__uint_as_float(pk & ~63u) > best.kdf)) {
          const int32_t *src = tree[pk & 63u].pts + (int64_t)po * rs;
          int32_t p[D ? rec_ints(D) : rec_ints(kMaxDim)];
#pragma unroll
          for (int c4 = 0; c4 < (D ? rec_ints(D) : rec_ints(kMaxDim)); c4 += 4)
            if (c4 < rs) {
              const int4 v = *reinterpret_cast<const int4 *>(src + c4);
              p[c4] = v.x;
              p[c4 + 1] = v.y;
              p[c4 + 2] = v.z;
              p[c4 + 3] = v.w;
            }
          id = D ? p[D ? D : 0] : src[dim];
          float sf = 0.f;
#pragma unroll
          for (int c = 0; c < DM; ++c)
            if (c < dim) {
              const float g = q[c] - __int_as_float(p[c] | kBias);
              sf = fmaf(g, g, sf);
            }
          if (!(sf > best.kdf) && id >= 0) {
#pragma unroll
            for (int c4 = 0; c4 < DM; c4 += 4) {
              const int4 x4 = *reinterpret_cast<const int4 *>(W.q + c4);
              const int32_t xq[4] = {x4.x, x4.y, x4.z, x4.w};
#pragma unroll
              for (int e = 0; e < 4; ++e)
                if (c4 + e < DM && c4 + e < dim) {
                  const int32_t g = xq[e] - p[c4 + e];
                  s += (uint64_t)((int64_t)g * g);
                }
            }
            have = pair_less(s, id, best.kd, best.kid);
          }
        }
        top_add(best, k, have, s, id);
      }
    }
    if (sp == 0) continue;
    // ---- node round: the entries of up to eight records (two while there is no bound) ----
    const int win = min(sp, 32);
    const uint64_t e0 = lane < win ? W.node[sp - 1 - lane] : 0;
    const bool ok0 = lane < win && !(__uint_as_float((uint32_t)(e0 >> 32) & ~63u) > best.kdf);
    const unsigned om = __ballot_sync(0xffffffffu, ok0);
    const int ord = __popc(om & lt);
    const bool tk0 = ok0 && ord < (sp > kWWide ? 1 : best.kdf == kInf ? 2 : 8);
    if (tk0) W.sel[ord] = e0;
    const unsigned tk = __ballot_sync(0xffffffffu, tk0);
    // what leaves the stack: the records taken and the pruned ones above them
    sp -= tk == om ? win : 32 - __clz(tk);
    if (tk == 0) continue;
    __syncwarp();
    const int r = lane >> 2, a = lane & 3;
    uint32_t b = 0x7f800000u | a;   // box distance bits, low 2 bits: the entry's number
    int32_t code = 0;
    uint32_t tr = 0;
    if (r < __popc(tk)) {
      const uint64_t e = W.sel[r];
      tr = (uint32_t)(e >> 32) & 63u;
      const WTree &T = tree[tr];
      if ((uint32_t)e >= (uint32_t)T.nrec || sp > kWStack - 4) {
        atomicOr(J.err, (uint32_t)e >= (uint32_t)T.nrec ? kErrChild : kErrStack);
      } else {
        const int32_t *rp = T.pk + (int64_t)(uint32_t)e * rec;
        float s = 0.f;
        int32_t lv;
        auto gap = [&](int c, float lo, float hi) {
          const float g = fmaxf(fmaxf(lo - q[c], q[c] - hi), 0.f);
          s = fmaf(g, g, s);
        };
        if (D && !packed_by_entry(D)) {
          code = rp[packed_code_at(D, a)];
          lv = rp[packed_live_at(D, a)];
#pragma unroll
          for (int c = 0; c < DM; ++c)
            gap(c, __int_as_float(rp[packed_lo_at(D, a, c)] | kBias), __int_as_float(rp[packed_hi_at(D, a, c)] | kBias));
        } else if (dim & 1) {
          const int4 w0 = *reinterpret_cast<const int4 *>(rp + packed_quad_at(a, 0));
          code = w0.x;
          lv = w0.y;
          gap(0, __int_as_float(w0.z), __int_as_float(w0.w));
#pragma unroll
          for (int c = 1; c + 1 < DM; c += 2)
            if (c < dim) {
              const float4 w = *reinterpret_cast<const float4 *>(rp + packed_quad_at(a, 2 + 2 * c));
              gap(c, w.x, w.y);
              gap(c + 1, w.z, w.w);
            }
        } else {
          const int2 cl = *reinterpret_cast<const int2 *>(rp + packed_code_at(dim, a));
          code = cl.x;
          lv = cl.y;
#pragma unroll
          for (int c = 0; c + 1 < DM; c += 2)
            if (c < dim) {
              const float4 w = *reinterpret_cast<const float4 *>(rp + packed_quad_at(a, 2 * c));
              gap(c, w.x, w.y);
              gap(c + 1, w.z, w.w);
            }
        }
        if (lv > 0 && !(s > best.kdf)) b = (__float_as_uint(s) & ~3u) | a;
      }
    }
    // the entries that stay go onto their stack, the nearest of a record
    // last, the record nearest the old stack's top last of all
    const uint32_t b1 = __shfl_xor_sync(0xffffffffu, b, 1), b2 = __shfl_xor_sync(0xffffffffu, b, 2),
                   b3 = __shfl_xor_sync(0xffffffffu, b, 3);
    const int near = (b1 < b) + (b2 < b) + (b3 < b);   // entries that do not stay compare greater
    const bool in = b < 0x7f800000u;
    const unsigned nm = __ballot_sync(0xffffffffu, in && code >= 0);
    const unsigned lm = __ballot_sync(0xffffffffu, in && code < 0);
    const unsigned from = 0xffffffffu << (lane & ~3);   // this record's lanes and those taken after it
    const uint64_t e = ((uint64_t)((b & ~63u) | tr) << 32) | (uint32_t)(code < 0 ? ~code : code);
    if (in) {
      uint64_t *dst = code < 0 ? &W.leaf[ls + __popc(lm & from)] : &W.node[sp + __popc(nm & from)];
      dst[-1 - near] = e;
    }
    sp += __popc(nm);
    ls += __popc(lm);
    __syncwarp();
  }
  // the buffer's points, where they have no tree
  for (int64_t b = 0; b < J.nbuf; b += 32) {
    const int64_t j = b + lane;
    bool have = false;
    uint64_t s = 0;
    int32_t id = 0;
    if (j < J.nbuf) {
      id = J.buf[j];
      const int32_t *p = J.idtab + (int64_t)id * dim;
      for (int c = 0; c < dim; ++c) {
        const int32_t g = W.q[c] - p[c];
        s += (uint64_t)((int64_t)g * g);
      }
      have = pair_less(s, id, best.kd, best.kid);
    }
    top_add(best, k, have, s, id);
  }
  near_id = best.d != ~0ull ? best.id : -1;
  if (lane < k) {
    const bool ok = best.d != ~0ull;
    J.oi[qi * k + lane] = ok ? best.id : -1;
    J.od[qi * k + lane] = ok ? (int64_t)best.d : INT64_MAX;
  }
}

// The walk's tree table (smallest tree first) from the nt views.
__device__ __forceinline__ void fill_trees(WTree *tree, const TreeView *views, int nt, int at, int step) {
  for (int ti = at; ti < nt; ti += step) {
    const TreeView &V = views[nt - 1 - ti];
    WTree w;
    w.pk = V.pk;
    w.pts = V.pts;
    w.leaf_off = V.leaf_off;
    w.size = V.size;
    w.nrec = (int32_t)packed_nrec(V.h);
    w.nleaf = (int32_t)((int64_t)1 << V.h);
    tree[ti] = w;
  }
}

// One forest: every warp answers `per` consecutive queries of the processing
// order.
template <int D>
__global__ void __launch_bounds__(kWarpsPerBlock * 32)
    k_knn_warp_one(const __grid_constant__ KnnOne P, int k, int per) {
  __shared__ WarpMem W[kWarpsPerBlock];
  __shared__ WTree tree[kWTrees];
  fill_trees(tree, P.trees, P.job.ntrees, threadIdx.x, blockDim.x);
  __syncthreads();
  const int64_t t0 = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * per;
  const int64_t t1 = min(t0 + per, P.job.m);
  int32_t near_id = -1;
  for (int64_t t = t0; t < t1; ++t)
    warp_query<D>(P.job, W[threadIdx.x >> 5], tree, P.job.ntrees, P.job.perm ? P.job.perm[t] : t, k, near_id);
}

// Many forests: warp w answers the (w - job_warp[j])-th `per` queries of its
// job j.
template <int D>
__global__ void __launch_bounds__(kWarpsPerBlock * 32)
    k_knn_warp(const KnnJob *jobs, const int64_t *job_warp, int njobs, int k, int per) {
  __shared__ WarpMem W[kWarpsPerBlock];
  __shared__ WTree tree[kWarpsPerBlock][kWTrees];
  __shared__ KnnJob s_job[kWarpsPerBlock];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (w >= job_warp[njobs]) return;
  int lo = 0, hi = njobs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (job_warp[mid] <= w) lo = mid;
    else hi = mid - 1;
  }
  KnnJob &J = s_job[warp];
  if (lane == 0) J = jobs[lo];
  __syncwarp();
  const int64_t t0 = (w - job_warp[lo]) * per, t1 = min(t0 + per, J.m);
  fill_trees(tree[warp], J.trees, J.ntrees, lane, 32);
  __syncwarp();
  int32_t near_id = -1;
  for (int64_t t = t0; t < t1; ++t)
    warp_query<D>(J, W[warp], tree[warp], J.ntrees, J.perm ? J.perm[t] : t, k, near_id);
}

template <int D>
void warp_one(const KnnOne &P, int k, int per, cudaStream_t s) {
  const int64_t blk = (int64_t)kWarpsPerBlock * per;
  KScope ks_(kK_knn_warp, s);
  k_knn_warp_one<D><<<(unsigned)((P.job.m + blk - 1) / blk), kWarpsPerBlock * 32, 0, s>>>(P, k, per);
}

template <int D>
void warp_table(const KnnJob *jobs, const int64_t *job_warp, int njobs, int64_t warps, int k, int per,
                cudaStream_t s) {
  KScope ks_(kK_knn_warp, s);
  k_knn_warp<D><<<(unsigned)((warps + kWarpsPerBlock - 1) / kWarpsPerBlock), kWarpsPerBlock * 32, 0, s>>>(
      jobs, job_warp, njobs, k, per);
}

}  // namespace

// Up to eight neighbouring queries per warp, which find their paths in L1 and
// start with a bound, while that leaves about six times the warps the GPU can
// hold.  10M 7-D points, 1M queries: 23.5 -> 17.8 ms; with 16 per warp 17.9,
// with 32 19.2.  1M 7-D points, 50K queries: one per warp 0.99 ms, three 1.08.
int knn_warp_per(int64_t m) { return (int)std::min<int64_t>(8, std::max<int64_t>(1, m / 30000)); }

// Between the size of one forest, which sets the length of a walk, and the size
// of all, which sets how far apart a warp's queries and its reads lie: their
// geometric mean.  us by all / by one / by the mean: 64 forests of 10K 3-D
// points, 1,200 queries each, k = 8: 234 / 182 / 181; 5-D, 5,000 queries, k = 5:
// 1202 / 1336 / 1337; 32 forests of 12K 7-D points, 10,000 queries, k = 1: uniform
// 1017 / 1505 / 1015, clustered 828 / 529 / 829; 128 of 5K 8-D points, clustered,
// 2,000 queries, k = 1: 526 / 253 / 526.
int64_t knn_forest_size(double mn, int64_t m, double n) {
  return (int64_t)std::sqrt(mn / (double)std::max<int64_t>(m, 1) * n);
}

// Where the two kernels cost the same: thousands of queries, for k = 1, 5, 16
// and 32 on forests of 2,000, 10,000, 30,000, 100,000 and a million points, by
// dimension (the last row: 9 and more; 9999: beyond 2.5 million, from the 1.28
// million that were measured).  The warp-per-query kernel's time grows with the
// queries (3 to 20 ns each) from a few dozen microseconds; the
// thread-per-query kernel's stays near that of its slowest warps until about
// 130,000 queries fill the GPU, and then grows more slowly where its walks are
// short (low dimensions, small forests) and for small k (its top-k lists take
// 12 k bytes of shared memory per thread: past k = 16 they cost it resident
// warps).  Each entry is the geometric mean of the crossings of uniform points
// and of points in 100 clusters (a million: with those of 4 or 10 million; 9 and
// more: of 10, 13 and 16 dimensions; uniform points from 30,000 on in 8 and more
// dimensions, where the thread-per-query kernel is several times slower, count as
// 5 million).  2,500 to 1.28 million queries at points of the forest, thread /
// warp in us on either side of a crossing:
//   dim 1, k = 5:  n = 10,000, 10K queries 43 / 35, 20K 42 / 52
//   dim 2, k = 5:  n = 100,000, 20K 92 / 69, 40K 106 / 147
//   dim 3, k = 5:  n = 1M, 40K 278 / 205, 80K 282 / 340; n = 10M, 40K 282 / 216, 80K 307 / 390
//          k = 16: n = 1M, 80K 550 / 441, 160K 695 / 805
//   dim 4, k = 1:  n = 30,000, 40K 144 / 140, 80K 156 / 199
//   dim 5, k = 1:  n = 2,000 clustered, 10K 36 / 31, 20K 38 / 47
//          k = 16: n = 30,000, 80K 917 / 583, 160K 1049 / 1058
//   dim 6, k = 5:  n = 10,000, 80K 504 / 374, 160K 587 / 682
//   dim 7, k = 1:  n = 10,000, 160K 396 / 350, 320K 488 / 601; clustered, 20K 72 / 59, 40K 90 / 124
//          k = 5:  n = 4M clustered, 1.28M 33527 / 19327
//   dim 8, k = 1:  n = 2,000 clustered, 20K 51 / 50, 40K 70 / 106
//          k = 5:  n = 10,000, 160K 1525 / 1406, 320K 1914 / 2558
//   dim 10, k = 1: n = 2,000 clustered, 20K 96 / 68, 40K 114 / 138
//   dim 16, k = 1: n = 2,000 clustered, 20K 112 / 68, 40K 121 / 138
// Over all 3,121 of those launches the choice costs 1.9% more than the better
// kernel each time; at worst, between the crossings of uniform and of clustered
// points, 2.0 times where the warp-per-query kernel is taken and 2.8 times where
// the other is (1-D points of which most lie in the same places).
//
// Leaves of hundreds of points and more (spatial-median trees of clustered
// points) are scanned by one lane in the thread-per-query kernel, 32 points at
// a time here.  The second table, for 10,000, 100,000, 1 and 10 million points,
// stands where it is the higher one; it hardly depends on the dimension (1 to 5
// measured).  100 clusters, thread / warp in us:
//   dim 2, k = 1:  n = 100,000, 40K queries 224 / 166, 160K 287 / 403
//          k = 5:  n = 1M, 160K 2580 / 1255, 640K 3057 / 3947; n = 10M, 640K 14439 / 11371, 1.28M 17280 / 19153
//   dim 3, k = 5:  n = 100,000, 80K 436 / 303, 160K 464 / 542
//          k = 1:  n = 10M, 640K 18455 / 13107, 1.28M 23134 / 21732
// Over 796 such launches from 10,000 points on: 1.3% more than the better kernel.
namespace {

constexpr int kAtK[4] = {1, 5, 16, 32};

// Thousands of queries at (k, n) from a table over kAtK and N sizes: linear in
// k and log n between its entries, for the logarithm.
template <int N>
float crossing(const float (&most)[4][N], const float (&at_n)[N], int k, int64_t n) {
  const int ik = k < 5 ? 0 : k < 16 ? 1 : 2;
  const float wk = (float)(k - kAtK[ik]) / (float)(kAtK[ik + 1] - kAtK[ik]);
  int in = 0;
  while (in < N - 2 && (float)n >= at_n[in + 1]) ++in;
  const float x = std::log((float)std::max<int64_t>(n, 1) / at_n[in]) / std::log(at_n[in + 1] / at_n[in]);
  const float wn = std::min(std::max(x, 0.f), 1.f);
  auto at = [&](int i) { return (1 - wn) * std::log(most[i][in]) + wn * std::log(most[i][in + 1]); };
  return std::exp((1 - wk) * at(ik) + wk * at(ik + 1));
}

}  // namespace

bool knn_by_warp(int dim, int k, int64_t m, int64_t n, bool skewed) {
  static constexpr float kAtN[5] = {2000, 10000, 30000, 100000, 1e6};
  static constexpr float kMost[9][4][5] = {
      {{3, 9, 16, 19, 68}, {16, 15, 22, 26, 77}, {33, 33, 41, 49, 120}, {91, 61, 140, 170, 290}},
      {{12, 14, 21, 16, 27}, {24, 28, 31, 31, 42}, {41, 57, 81, 83, 100}, {120, 180, 450, 2100, 9999}},
      {{15, 24, 29, 25, 39}, {30, 39, 53, 50, 76}, {53, 79, 110, 140, 140}, {140, 440, 1600, 9999, 9999}},
      {{16, 21, 34, 32, 47}, {33, 44, 56, 59, 120}, {82, 98, 130, 190, 770}, {250, 1000, 1700, 9999, 9999}},
      {{21, 30, 49, 49, 130}, {37, 51, 82, 120, 590}, {94, 100, 150, 260, 9999}, {300, 1100, 1700, 9999, 9999}},
      {{23, 60, 92, 87, 690}, {44, 72, 120, 220, 9999}, {98, 130, 220, 1300, 9999}, {260, 1000, 1700, 9999, 9999}},
      {{35, 73, 160, 200, 9999}, {52, 95, 180, 9999, 9999}, {190, 230, 560, 9999, 9999}, {880, 1700, 9999, 9999, 9999}},
      {{37, 100, 460, 860, 9999}, {48, 110, 770, 9999, 9999}, {100, 150, 1100, 9999, 9999}, {260, 1200, 9999, 9999, 9999}},
      {{160, 460, 890, 9999, 9999}, {100, 220, 1100, 9999, 9999}, {550, 300, 1500, 9999, 9999}, {650, 9999, 9999, 9999, 9999}}};
  static constexpr float kAtSkewedN[4] = {1e4, 1e5, 1e6, 1e7};
  static constexpr float kMostSkewed[4][4] = {
      {26, 65, 300, 2000}, {40, 130, 500, 3000}, {110, 270, 900, 9999}, {450, 9999, 9999, 9999}};
  float most = crossing(kMost[std::min(dim, 9) - 1], kAtN, k, n);
  if (skewed) most = std::max(most, crossing(kMostSkewed, kAtSkewedN, k, n));
  return (float)m <= 1000 * most;
}

int launch_knn_warp_one(const KnnOne &P, int dim, int k, int per, cudaStream_t s) {
  switch (dim) {
    case 1: warp_one<1>(P, k, per, s); break;
    case 2: warp_one<2>(P, k, per, s); break;
    case 3: warp_one<3>(P, k, per, s); break;
    case 4: warp_one<4>(P, k, per, s); break;
    case 5: warp_one<5>(P, k, per, s); break;
    case 6: warp_one<6>(P, k, per, s); break;
    case 7: warp_one<7>(P, k, per, s); break;
    case 8: warp_one<8>(P, k, per, s); break;
    default: warp_one<0>(P, k, per, s); break;
  }
  return cuda_check(cudaGetLastError(), "knn kernel");
}

int launch_knn_warp_table(const void *table, int njobs, int64_t warps, int dim, int k, int per, cudaStream_t s) {
  if (warps == 0) return BDL_OK;
  const KnnJob *jobs = (const KnnJob *)table;
  const int64_t *job_warp = (const int64_t *)((const char *)table + njobs * sizeof(KnnJob));
  switch (dim) {
    case 1: warp_table<1>(jobs, job_warp, njobs, warps, k, per, s); break;
    case 2: warp_table<2>(jobs, job_warp, njobs, warps, k, per, s); break;
    case 3: warp_table<3>(jobs, job_warp, njobs, warps, k, per, s); break;
    case 4: warp_table<4>(jobs, job_warp, njobs, warps, k, per, s); break;
    case 5: warp_table<5>(jobs, job_warp, njobs, warps, k, per, s); break;
    case 6: warp_table<6>(jobs, job_warp, njobs, warps, k, per, s); break;
    case 7: warp_table<7>(jobs, job_warp, njobs, warps, k, per, s); break;
    case 8: warp_table<8>(jobs, job_warp, njobs, warps, k, per, s); break;
    default: warp_table<0>(jobs, job_warp, njobs, warps, k, per, s); break;
  }
  return cuda_check(cudaGetLastError(), "knn kernel");
}

}  // namespace bdl
