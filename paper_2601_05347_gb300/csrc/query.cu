// query.cu -- batched k-NN, range count and range list (Sec 2.2) on either
// tree layout (SPaC summary tree or P-Orth), one warp per query (k-NN of k <= 32
// over many queries: two per warp, and of k <= 16 one per thread, knn_lane.cu),
// queries taken in curve order so that neighbouring warps walk the same nodes
// out of L2.
//
// k-NN: depth-first traversal that enters children in increasing order of
// their box distance (Appendix "Implementation Details": subtrees are visited
// in increasing minimum distance to the query) and prunes a subtree whose box
// is farther than the current k-th best.  A node's children are evaluated one
// per lane; each level of the current path keeps its children's distance keys
// and a bitmask of those still to visit in shared memory, and a warp minimum
// picks the next one.  The search starts from seed leaves at the query's own
// curve position (SPaC, and P-Orth queries that are sorted).  The k best (d2, id) pairs live in
// a KList (klist.cuh).  Squared distances are exact int64 (|dx| < 2^31 for
// coordinates in [0, 2^31)).
//
// Range count: children inside the box add their subtree count; children that
// straddle the box are descended; straddling leaves are scanned.
// Range list: the same traversal counts first; after an exclusive scan of the
// counts a second traversal writes each query's ids at its offset (a
// subtree inside the box is enumerated without further box tests).
#include <cmath>
#include <type_traits>

#include "bitonic.cuh"
#include "index.cuh"
#include "keys.cuh"
#include "klist.cuh"
#include "knn.cuh"

namespace psi {

// Curve order of a query batch and its sorted keys; owns the sort buffers.
struct QueryOrder {
  Buf<uint64_t> k0, k1;
  Buf<uint32_t> v0, v1;
  const uint32_t *order = nullptr;
  const uint64_t *keys = nullptr;
  int key_shift = 0;
  uint32_t *spare = nullptr;    // 2 nq free words (the key buffer the sort left unused)
  uint32_t *spare_v = nullptr;  // nq free words (the position buffer it left unused)
};

namespace {

constexpr int QW = 4;         // warps per block
constexpr int STACK = 256;    // stack entries per warp (>= depth * fanout)
constexpr uint32_t INSIDE = 0x80000000u;

template <int D>
__device__ __forceinline__ uint32_t box_key(const TreeView &t, uint32_t node, const int32_t *qc) {
  int32_t lo[D], hi[D];
#pragma unroll
  for (int d = 0; d < D; ++d) {
    lo[d] = t.lo[d][node];
    hi[d] = t.hi[d][node];
  }
  return box_key_of<D>(lo, hi, qc);
}

// 0: disjoint, 1: straddles, 2: node box inside the query box.
template <int D>
__device__ __forceinline__ int box_relation(const TreeView &t, uint32_t node, const int32_t *blo, const int32_t *bhi) {
  bool inside = true, disjoint = false;
#pragma unroll
  for (int d = 0; d < D; ++d) {
    const int32_t lo = t.lo[d][node], hi = t.hi[d][node];
    disjoint |= hi < blo[d] || lo > bhi[d];
    inside &= blo[d] <= lo && hi <= bhi[d];
  }
  return disjoint ? 0 : (inside ? 2 : 1);
}

// Scan one leaf: every point whose (d2, id) beats the current k-th enters the
// list (klist_offer: in bulk when many enter at once, the seed leaves of a
// query; one at a time otherwise).
// Slots [s0, s0 + cnt).
// EMPTY: the list is known to be empty (the first leaf a query scans).
template <int D, int KPL, bool EMPTY = false>
__device__ __forceinline__ void knn_scan_slots(const TreeView &t, uint32_t s0, int cnt, const int32_t *qc,
                                               KList<KPL> &kl, KWait *wt, int &nw, int k) {
  const int lane = threadIdx.x & 31;
  for (int b = 0; b < cnt; b += 32) {
    const int s = b + lane;
    int64_t d2 = INT64_MAX;
    uint32_t id = 0xFFFFFFFFu;
    const bool valid = s < cnt;
    if (valid) {
      const uint32_t slot = s0 + (uint32_t)s;
      id = t.pid[slot];
      d2 = 0;
#pragma unroll
      for (int d = 0; d < D; ++d) {
        // both in [0, 2^31): the difference is exact in 32 bits, its square
        // one widening multiply
        const int32_t dd = t.px[d][slot] - qc[d];
        d2 += (int64_t)dd * dd;
      }
    }
    if (EMPTY && b == 0)  // the list holds nothing yet: every point enters
      klist_fill(kl, valid, d2, id, k);
    else if constexpr (KPL > 1)
      klist_wait(kl, *wt, nw, valid && kl.admits(d2, id), d2, id, k);
    else
      klist_offer(kl, valid && kl.admits(d2, id), d2, id, k);
  }
}

template <int D, int KPL, bool EMPTY = false>
__device__ __forceinline__ void knn_scan_leaf(const TreeView &t, uint32_t node, const int32_t *qc, KList<KPL> &kl,
                                              KWait *wt, int &nw, int k) {
  knn_scan_slots<D, KPL, EMPTY>(t, t.ref[node], t.cnt[node], qc, kl, wt, nw, k);
}

struct KnnStats {
  // [0] internal nodes expanded, [1] leaves scanned, [2] points scanned, [3] queries,
  // [4] child descriptors read (children evaluated by the expansions)
  unsigned long long *c;
};

// Queries per warp of the grouped k-NN kernel (k <= 32, queries in curve order).
constexpr int kGroup = 2;
// Flag of a stack entry that is a leaf to scan (in its count word).
constexpr uint32_t kLeafEntry = 0x80000000u;

// Last position p in [0, n) whose first key (>> shift) is <= key, or 0 when
// the key precedes every position (binary search by one thread).
template <typename FirstKey>
__device__ __forceinline__ int64_t seed_search(FirstKey first_key, int64_t n, uint64_t key, int shift) {
  int64_t lo = 0, hi = n;  // first position whose first key is greater
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if ((first_key(mid) >> shift) <= key)
      lo = mid + 1;
    else
      hi = mid;
  }
  return lo > 0 ? lo - 1 : 0;
}

// The same search by a whole warp (32 probes per step: four steps for 1e6
// positions), for one query: its steps are dependent loads.
__device__ __forceinline__ int64_t seed_search_warp(const uint64_t *first_key, int64_t n, uint64_t key) {
  const int lane = threadIdx.x & 31;
  int64_t lo = 0, hi = n;  // first position whose first key is greater
  while (hi - lo > 32) {
    const int64_t len = hi - lo;
    const int c = __popc(__ballot_sync(0xFFFFFFFFu, first_key[lo + len * (lane + 1) / 33] <= key));
    const int64_t l0 = lo;
    if (c > 0) lo = l0 + len * c / 33 + 1;
    if (c < 32) hi = l0 + len * (c + 1) / 33;
  }
  lo += __popc(__ballot_sync(0xFFFFFFFFu, lo + lane < hi && first_key[lo + lane] <= key));
  return lo > 0 ? lo - 1 : 0;
}

// Seed position of every query (queries in curve order), one thread each:
// SPaC, the node of the last leaf of the query's index whose first key is at
// most the query's key; P-Orth, the position in the key-ordered leaf list of
// the last leaf whose cell starts at or before the query's key.  Many
// independent searches in flight hide the dependent loads that one warp-wide
// search per query would wait on.
__global__ void k_knn_seed(const KnnSeed sd, const uint32_t *ref, const uint32_t *order, int64_t nq, uint32_t *pos) {
  for (int64_t qi = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; qi < nq; qi += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t key = sd.qkey[qi] & sd.qkey_mask;
    int64_t p = 0;
    if (sd.qseg) {
      const int64_t q = order ? (int64_t)order[qi] : qi;
      const int sg = sd.qseg[q];
      const int64_t lb = sd.node_off[sg];
      const int64_t L = (sd.off[sg + 1] - sd.off[sg] + sd.phi - 1) / sd.phi;
      if (L > 0) p = lb + seed_search([&](int64_t x) { return sd.pkey[ref[lb + x]]; }, L, key, sd.key_shift);
    } else if (sd.L > 0) {
      p = seed_search([&](int64_t x) { return sd.sep_key[x]; }, sd.L, key, sd.key_shift);
    }
    pos[qi] = (uint32_t)p;
  }
}

// One warp per query: depth-first search over a per-warp stack in shared
// memory.  Expanding a node evaluates its children one per lane and pushes
// those not farther than the current k-th distance, the nearest one on top, so
// the search enters the nearest child first (Appendix "Implementation
// Details": children in increasing box distance) and takes its siblings later,
// each re-checked against the k-th distance of that moment when it is popped.
// Seed (SPaC): the leaf that holds the query's own curve position is scanned
// first.  SPaC leaves are consecutive runs of the curve and their boxes
// overlap, so the nearest box is often not the leaf around the query; the
// curve neighbours make the k-th distance nearly final before the search
// starts (so the order of the later pops matters little), and the search then
// skips the seed leaves.  Seed (P-Orth): the leaf whose cell holds the query's
// key (or the last leaf before it in key order), alone.
template <int D, int KPL, bool STATS, bool BATCH, bool LIST = false, bool SELF = false, bool WIDE = false>
__global__ __launch_bounds__(QW * 32) void k_knn(KnnArgs a, KnnStats stats) {
  // internal nodes still to visit: (node, key, first child, children)
  __shared__ uint4 s_stk[QW][KSTACK];
  __shared__ KWait s_wait[KPL > 1 ? QW : 1];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  KWait *wt = &s_wait[KPL > 1 ? w : 0];
  const int64_t warps = (int64_t)gridDim.x * QW;
  const KnnTake<LIST> take(a);
  const int64_t nq = take.nq();
  const TreeView &t = a.t;
  __shared__ alignas(16) uint8_t s_tab[SELF ? kCurveTabBytes : 16];
  if (SELF && a.seed.curve == CURVE_HILBERT) {
    curve_table_init<D, CURVE_HILBERT>(s_tab);
    __syncthreads();
  }
  unsigned long long n_int = 0, n_leaf = 0, n_pts = 0, n_kids = 0;
  for (int64_t qi = (int64_t)blockIdx.x * QW + w; qi < nq; qi += warps) {
    const int64_t q = take.query(qi);
    int32_t qc[D];
#pragma unroll
    for (int d = 0; d < D; ++d) qc[d] = a.q[q * D + d];
    KList<KPL> kl;
    kl.init();
    int nw = 0;  // candidates waiting
    const int32_t root = a.qroot ? a.qroot[q] : t.root;
    // seed leaves [s_lo, s_hi]: the leaf at the query's curve position, widened
    // along the curve until it holds at least k points
    int64_t s_lo = 0, s_hi = -1;
    const KnnSeed &sd = a.seed;
    int64_t lb = 0, L = sd.L;  // the query's leaves are nodes [lb, lb + L)
    if (sd.qkey && sd.qseg) {
      const int sg = sd.qseg[q];
      lb = sd.node_off[sg];
      L = (sd.off[sg + 1] - sd.off[sg] + sd.phi - 1) / sd.phi;
    }
    if (SELF) {
      bool bad;  // (a query may lie outside the grid; its seed is then any leaf)
      const uint64_t key = sd.curve == CURVE_HILBERT ? point_key<D, CURVE_HILBERT>(s_tab, qc, sd.self_bits, bad)
                                                     : point_key<D, CURVE_MORTON>(s_tab, qc, sd.self_bits, bad);
      s_lo = s_hi = seed_search_warp(sd.sep_key, sd.L, key);
      knn_scan_leaf<D, KPL, true>(t, (uint32_t)s_lo, qc, kl, wt, nw, a.k);
    } else if (sd.qkey && root >= 0) {
      const int64_t pos = take.pos(qi);  // k_knn_seed
      if (L > 0) {
        // P-Orth: pos is a position in the key-ordered leaf list
        const int64_t j = sd.leaf_node ? (int64_t)sd.leaf_node[pos] : pos;
        const int64_t le = lb + L;
        knn_scan_leaf<D, KPL, true>(t, (uint32_t)j, qc, kl, wt, nw, a.k);
        int64_t got = t.cnt[j];
        if (STATS) {
          ++n_leaf;
          n_pts += got;
        }
        s_lo = j;
        s_hi = j;
        // widened along the curve only where leaves are consecutive nodes
        // (SPaC; P-Orth's key-order neighbours give a loose bound in 3D and
        // did not cut the leaves its search scans)
        while (!sd.leaf_node && got < a.k && (s_lo > lb || s_hi + 1 < le)) {
          int64_t nx;
          if (s_hi + 1 < le && (s_lo == lb || s_hi - j <= j - s_lo))
            nx = ++s_hi;
          else
            nx = --s_lo;
          knn_scan_leaf<D, KPL>(t, (uint32_t)nx, qc, kl, wt, nw, a.k);
          got += t.cnt[nx];
          if (STATS) {
            ++n_leaf;
            n_pts += t.cnt[nx];
          }
        }
      }
    }
    // seed leaves as a node range [slo, shi] (empty: slo > shi)
    const uint32_t slo = s_hi < s_lo ? 1u : (uint32_t)s_lo;
    const uint32_t shi = s_hi < s_lo ? 0u : (uint32_t)s_hi;
    if (KPL > 1 && nw) klist_flush(kl, *wt, nw, a.k);
    uint32_t kdk = order_key(kl.kd);
    int sp = 0;
    // Children [c0, c0 + nk) of an expanded node: the internal ones that may
    // hold a neighbour are pushed (the nearest on top); the leaves that may
    // are scanned at once, nearest first, each re-checked against the k-th
    // distance left by the ones before it.  Where a node has both (P-Orth),
    // only the leaves nearer than every internal survivor are scanned at once
    // and the others are pushed beside the internal ones (count | kLeafEntry),
    // so the search still takes the nearest child first.  A popped leaf entry
    // comes back here as `pl` (its lane 0 stands for the leaf).  Each lane
    // loads its child's reference and count with its box, so a popped entry
    // needs no further load before its own children are read.
    // WIDE (P-Orth): each group of CW lanes has a node (or leaf entry) of its own.
    constexpr int CW = WIDE ? 8 : 32;  // at least 2^D
    const int cl = lane % CW;
    auto expand = [&](uint32_t c0, int nk, bool pl, uint32_t pkey) {
      const uint32_t c = c0 + (uint32_t)cl;
      uint32_t key = 0xFFFFFFFFu;  // above any k-th distance key
      bool leafc = false;
      uint32_t cref = 0;
      int ccnt = 0;
      if (pl) {
        if (cl == 0) {
          key = pkey;
          leafc = true;
          cref = c0;
          ccnt = nk;
        }
      } else if (cl < nk) {  // every node of every layout holds a point
        cref = t.ref[c];
        if (a.leaf_limit >= 0) {
          leafc = (int64_t)c < a.leaf_limit;
          ccnt = leafc ? t.cnt[c] : t.kids[c];
        } else {
          const int ck = t.kids[c], cn = t.cnt[c];
          leafc = ck == 0;
          ccnt = leafc ? cn : ck;
        }
        key = box_key<D>(t, c, qc);
        if (leafc && c >= slo && c <= shi) key = 0xFFFFFFFFu;  // scanned as a seed
      }
      const bool in = key <= kdk;
      if (STATS && !pl) {
        ++n_int;
        n_kids += nk;
      }
      uint32_t mi = __ballot_sync(0xFFFFFFFFu, in && !leafc);
      uint32_t ml = __ballot_sync(0xFFFFFFFFu, in && leafc);
      if (mi && ml) {  // warp-uniform: leaves not nearer than the nearest internal survivor wait
        const uint32_t imin = __reduce_min_sync(0xFFFFFFFFu, ((mi >> lane) & 1u) ? key : 0xFFFFFFFFu);
        const uint32_t defer = __ballot_sync(0xFFFFFFFFu, in && leafc && key >= imin);
        ml &= ~defer;
        mi |= defer;
      }
      if (mi) {
        const int n = __popc(mi);
        if (sp + n > KSTACK) {  // cannot happen within the depth bound above
          if (lane == 0) atomicOr(a.status, ST_STACK);
        } else {
          // the nearest survivor (lowest lane on ties) takes the top slot, the
          // one that held the top slot takes its place
          const bool ii = (mi >> lane) & 1u;
          const uint32_t mn = __reduce_min_sync(0xFFFFFFFFu, ii ? key : 0xFFFFFFFFu);
          const int win = __ffs(__ballot_sync(0xFFFFFFFFu, ii && key == mn)) - 1;
          int pos = __popc(mi & lanemask_lt());
          if (lane == win)
            pos = n - 1;
          else if (pos == n - 1)
            pos = __popc(mi & ((1u << win) - 1u));
          __syncwarp();
          if (ii) s_stk[w][sp + pos] = make_uint4(c, key, cref, (uint32_t)ccnt | (leafc ? kLeafEntry : 0u));
          sp += n;
          __syncwarp();
        }
      }
      // BATCH (P-Orth): leaves in batches, taken nearest first (each still
      // within the k-th distance of that moment) while their points fit one
      // round of 32 lanes, then scanned together, so that small leaves (a few
      // points each in 3D) share one k-list merge; a leaf of more than 32
      // points is a batch of its own, scanned in rounds.  Otherwise (SPaC,
      // whose leaves fill a round) a leaf at a time, each re-checked.
      if constexpr (!BATCH) {
        while (ml) {
          const uint32_t mn = __reduce_min_sync(0xFFFFFFFFu, (ml >> lane) & 1u ? key : 0xFFFFFFFFu);
          if (mn > kdk) break;  // every remaining leaf is farther than the k-th distance
          const int src = __ffs(__ballot_sync(0xFFFFFFFFu, ((ml >> lane) & 1u) && key == mn)) - 1;
          ml &= ~(1u << src);
          const uint32_t lref = __shfl_sync(0xFFFFFFFFu, cref, src);
          const int lcnt = __shfl_sync(0xFFFFFFFFu, ccnt, src);
          knn_scan_slots<D, KPL>(t, lref, lcnt, qc, kl, wt, nw, a.k);
          kdk = order_key(kl.kd);
          if (STATS) {
            ++n_leaf;
            n_pts += lcnt;
          }
        }
      }
      while (BATCH && ml) {
        uint32_t bl = 0;  // the batch's children (lanes)
        int tot = 0;
        while (ml) {
          const uint32_t mn = __reduce_min_sync(0xFFFFFFFFu, (ml >> lane) & 1u ? key : 0xFFFFFFFFu);
          if (mn > kdk) {  // every remaining leaf is farther than the k-th distance
            ml = 0;
            break;
          }
          const int src = __ffs(__ballot_sync(0xFFFFFFFFu, ((ml >> lane) & 1u) && key == mn)) - 1;
          const int c = __shfl_sync(0xFFFFFFFFu, ccnt, src);
          if (bl && tot + c > 32) break;
          bl |= 1u << src;
          ml &= ~(1u << src);
          tot += c;
          if (STATS) {
            ++n_leaf;
            n_pts += c;
          }
          if (tot >= 32) break;
        }
        if (!bl) break;
        // batch position of each member leaf's first point (in lane order)
        const int mine = (bl >> lane) & 1u ? ccnt : 0;
        int incl = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
          if (lane >= o) incl += y;
        }
        const int excl = incl - mine;
        for (int r = 0; r < tot; r += 32) {
          const int p = r + lane;
          uint32_t slot = 0;
          bool valid = false;
          for (uint32_t mb = bl; mb; mb &= mb - 1) {
            const int b = __ffs(mb) - 1;
            const int eb = __shfl_sync(0xFFFFFFFFu, excl, b);
            const int cb = __shfl_sync(0xFFFFFFFFu, ccnt, b);
            const uint32_t rb = __shfl_sync(0xFFFFFFFFu, cref, b);
            if (p >= eb && p < eb + cb) {
              valid = true;
              slot = rb + (uint32_t)(p - eb);
            }
          }
          int64_t d2 = INT64_MAX;
          uint32_t id = 0xFFFFFFFFu;
          if (valid) {
            id = t.pid[slot];
            d2 = 0;
#pragma unroll
            for (int d = 0; d < D; ++d) {
              const int32_t dd = t.px[d][slot] - qc[d];  // exact: both in [0, 2^31)
              d2 += (int64_t)dd * dd;
            }
          }
          if constexpr (KPL > 1)
            klist_wait(kl, *wt, nw, valid && kl.admits(d2, id), d2, id, a.k);
          else
            klist_offer(kl, valid && kl.admits(d2, id), d2, id, a.k);
        }
        kdk = order_key(kl.kd);
      }
    };
    if (root >= 0) {
      if (t.kids[root] == 0) {
        if (!((uint32_t)root >= slo && (uint32_t)root <= shi))
          knn_scan_leaf<D, KPL>(t, (uint32_t)root, qc, kl, wt, nw, a.k);
      } else {
        // the root as the first entry: one call site keeps `expand` inlined
        uint32_t c0 = t.ref[root], pkey = 0;
        int nk = t.kids[root];
        bool pl = false;
        if (WIDE && lane >= CW) nk = 0;
        for (;;) {
          expand(c0, nk, pl, pkey);
          uint4 e = make_uint4(0, 0, 0, 0);
          bool more = false;
          // WIDE: the top entries, one per group of lanes, once the list is full
          // and while the stack has room for the most that single pops may add
          // (2^D - 1 per level)
          while (WIDE && sp > 0 && !more) {
            const int g = lane / CW, pops = sp <= 64 && kdk < kNoBound ? min(sp, 32 / CW) : 1;
            e = g < pops ? s_stk[w][sp - 1 - g] : make_uint4(0, 0xFFFFFFFFu, 0, 0);
            sp -= pops;
            if (e.y > kdk) e = make_uint4(0, 0, 0, 0);  // no children
            more = __any_sync(0xFFFFFFFFu, e.w != 0);
          }
          while (!WIDE && sp > 0) {
            e = s_stk[w][--sp];
            if (e.y <= kdk) {  // else farther than the k-th distance found since the push
              more = true;
              break;
            }
          }
          if (!more) break;
          c0 = e.z;
          nk = (int)(e.w & ~kLeafEntry);
          pl = (e.w & kLeafEntry) != 0;
          pkey = e.y;
        }
      }
    }
    if (KPL > 1 && nw) klist_flush(kl, *wt, nw, a.k);
#pragma unroll
    for (int r = 0; r < KPL; ++r) {
      const int e = r * 32 + lane;
      if (e < a.k) {
        a.out_id[q * a.k + e] = kl.i[r];
        a.out_d2[q * a.k + e] = kl.d[r];
      }
    }
    if (STATS && lane == 0) atomicAdd(&stats.c[3], 1ull);
  }
  if (STATS && lane == 0) {
    atomicAdd(&stats.c[0], n_int);
    atomicAdd(&stats.c[1], n_leaf);
    atomicAdd(&stats.c[2], n_pts);
    atomicAdd(&stats.c[4], n_kids);
  }
}

// Scan one leaf for the queries of a group whose bit is set in qmask (warp-
// uniform): every lane loads one point once and offers it to each of those
// queries' lists.  FILL: the lists are known to be empty (the group's first
// leaf).
template <int D, int G, bool FILL>
__device__ __forceinline__ void knn_scan_group(const TreeView &t, uint32_t s0, int cnt, const int32_t (&qc)[G][D],
                                               KList<1> (&kl)[G], int k, uint32_t qmask) {
  const int lane = threadIdx.x & 31;
  for (int b = 0; b < cnt; b += 32) {
    const int s = b + lane;
    const bool valid = s < cnt;
    int32_t p[D];
    uint32_t id = 0xFFFFFFFFu;
    if (valid) {
      const uint32_t slot = s0 + (uint32_t)s;
      id = t.pid[slot];
#pragma unroll
      for (int d = 0; d < D; ++d) p[d] = t.px[d][slot];
    }
#pragma unroll
    for (int g = 0; g < G; ++g) {
      if (!((qmask >> g) & 1u)) continue;
      int64_t d2 = INT64_MAX;
      if (valid) {
        d2 = 0;
#pragma unroll
        for (int d = 0; d < D; ++d) {
          const int32_t dd = p[d] - qc[g][d];  // exact: both in [0, 2^31)
          d2 += (int64_t)dd * dd;
        }
      }
      if (FILL && b == 0)
        klist_fill(kl[g], valid, d2, id, k);
      else
        klist_offer(kl[g], valid && kl[g].admits(d2, id), d2, id, k);
    }
  }
}

// k-NN for k <= 32 with G consecutive queries (in curve order) per warp.
// Neighbouring queries visit nearly the same nodes and leaves, so the group
// shares one depth-first traversal: each child box is loaded once and tested
// against every query of the group (a child is needed if some query's k-th
// distance admits it), and each leaf's points are loaded once and offered to
// the lists of the queries that need the leaf.  Per query the result is the
// same as k_knn's: exact (distance, id) order, each query pruned by its own
// k-th distance.  Seeds: the distinct seed leaves of the group's queries are
// scanned first, for all of them.
template <int D, int G, bool STATS, bool RECHECK, bool LIST = false>
__global__ __launch_bounds__(QW * 32) void k_knn_group(KnnArgs a, KnnStats stats) {
  static_assert(G <= 2 || !RECHECK, "a stack entry holds the box keys of two queries");
  // internal nodes still to visit: (first child, children) and, with RECHECK,
  // the box keys of queries 0 and G - 1
  using Entry = typename std::conditional<RECHECK, uint4, uint2>::type;
  __shared__ Entry s_stk[QW][KSTACK];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const TreeView &t = a.t;
  const KnnSeed &sd = a.seed;
  const KnnTake<LIST> take(a);
  const int64_t nq = take.nq();
  const int64_t ngroups = (nq + G - 1) / G;
  unsigned long long n_int = 0, n_leaf = 0, n_pts = 0, n_kids = 0;
  for (int64_t gi = (int64_t)blockIdx.x * QW + w; gi < ngroups; gi += (int64_t)gridDim.x * QW) {
    const int64_t qi0 = gi * G;
    const int ng = (int)min((int64_t)G, nq - qi0);
    int32_t qc[G][D];
    uint32_t seed[G];
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const int64_t qi = qi0 + min(g, ng - 1);  // a short last group repeats its last query
      const int64_t q = take.query(qi);
#pragma unroll
      for (int d = 0; d < D; ++d) qc[g][d] = a.q[q * D + d];
      seed[g] = !sd.qkey ? 0xFFFFFFFFu : sd.leaf_node ? (uint32_t)sd.leaf_node[take.pos(qi)] : take.pos(qi);
    }
    KList<1> kl[G];
#pragma unroll
    for (int g = 0; g < G; ++g) kl[g].init();
    const uint32_t all = (1u << G) - 1u;
    const int32_t root = t.root;
    if (sd.qkey && root >= 0) {
      // the distinct seed leaves (positions are non-decreasing in curve order)
#pragma unroll
      for (int g = 0; g < G; ++g) {
        if (g > 0 && seed[g] == seed[g - 1]) continue;
        const uint32_t j = seed[g];
        if (g == 0)
          knn_scan_group<D, G, true>(t, t.ref[j], t.cnt[j], qc, kl, a.k, all);
        else
          knn_scan_group<D, G, false>(t, t.ref[j], t.cnt[j], qc, kl, a.k, all);
        if (STATS) {
          ++n_leaf;
          n_pts += t.cnt[j];
        }
      }
    }
    uint32_t kdk[G];
#pragma unroll
    for (int g = 0; g < G; ++g) kdk[g] = order_key(kl[g].kd);
    int sp = 0;
    // Children [c0, c0 + nk): the internal ones some query may need are pushed
    // (the one nearest to some query on top); the leaves some query may need
    // are scanned at once, nearest first, for the queries that still need them.
    // With RECHECK (P-Orth), leaves that are not nearer than every internal
    // survivor are pushed too (count | kLeafEntry) and come back as `pl`, as
    // in k_knn.
    auto expand = [&](uint32_t c0, int nk, bool pl, uint32_t pk0, uint32_t pk1) {
      const uint32_t c = c0 + (uint32_t)lane;
      uint32_t key[G];
#pragma unroll
      for (int g = 0; g < G; ++g) key[g] = 0xFFFFFFFFu;
      uint32_t need = 0, mkey = 0xFFFFFFFFu;  // queries that may need the child; its smallest key
      bool leafc = false;
      uint32_t cref = 0;
      int ccnt = 0;
      if (RECHECK && pl) {
        if (lane == 0) {
          key[0] = pk0;
          if (G > 1) key[G - 1] = pk1;
          leafc = true;
          cref = c0;
          ccnt = nk;
#pragma unroll
          for (int g = 0; g < G; ++g)
            if (key[g] <= kdk[g]) {
              need |= 1u << g;
              mkey = min(mkey, key[g]);
            }
        }
      } else if (lane < nk) {
        cref = t.ref[c];
        if (a.leaf_limit >= 0) {
          leafc = (int64_t)c < a.leaf_limit;
          ccnt = leafc ? t.cnt[c] : t.kids[c];
        } else {
          const int ck = t.kids[c], cn = t.cnt[c];
          leafc = ck == 0;
          ccnt = leafc ? cn : ck;
        }
        int32_t lo[D], hi[D];
#pragma unroll
        for (int d = 0; d < D; ++d) {
          lo[d] = t.lo[d][c];
          hi[d] = t.hi[d][c];
        }
#pragma unroll
        for (int g = 0; g < G; ++g) {
          key[g] = box_key_of<D>(lo, hi, qc[g]);
          if (key[g] <= kdk[g]) {
            need |= 1u << g;
            mkey = min(mkey, key[g]);
          }
        }
        if (leafc) {
#pragma unroll
          for (int g = 0; g < G; ++g)
            if (c == seed[g]) need = 0;  // scanned as a seed
        }
      }
      if (STATS && !(RECHECK && pl)) {
        ++n_int;
        n_kids += nk;
      }
      uint32_t mi = __ballot_sync(0xFFFFFFFFu, need && !leafc);
      uint32_t ml = __ballot_sync(0xFFFFFFFFu, need && leafc);
      if (RECHECK && mi && ml) {  // warp-uniform
        const uint32_t imin = __reduce_min_sync(0xFFFFFFFFu, ((mi >> lane) & 1u) ? mkey : 0xFFFFFFFFu);
        const uint32_t defer = __ballot_sync(0xFFFFFFFFu, need && leafc && mkey >= imin);
        ml &= ~defer;
        mi |= defer;
      }
      if (mi) {
        const int n = __popc(mi);
        if (sp + n > KSTACK) {  // cannot happen within the depth bound
          if (lane == 0) atomicOr(a.status, ST_STACK);
        } else {
          const bool ii = (mi >> lane) & 1u;
          const uint32_t mn = __reduce_min_sync(0xFFFFFFFFu, ii ? mkey : 0xFFFFFFFFu);
          const int win = __ffs(__ballot_sync(0xFFFFFFFFu, ii && mkey == mn)) - 1;
          int pos = __popc(mi & lanemask_lt());
          if (lane == win)
            pos = n - 1;
          else if (pos == n - 1)
            pos = __popc(mi & ((1u << win) - 1u));
          __syncwarp();
          if (ii) {
            if constexpr (RECHECK)
              s_stk[w][sp + pos] = make_uint4(cref, (uint32_t)ccnt | (leafc ? kLeafEntry : 0u), key[0],
                                              G > 1 ? key[G - 1] : 0xFFFFFFFFu);
            else
              s_stk[w][sp + pos] = make_uint2(cref, (uint32_t)ccnt);
          }
          sp += n;
          __syncwarp();
        }
      }
      while (ml) {
        // queries that still need each remaining leaf under the current bounds
        uint32_t now = 0, nkey = 0xFFFFFFFFu;
        if ((ml >> lane) & 1u) {
#pragma unroll
          for (int g = 0; g < G; ++g)
            if (((need >> g) & 1u) && key[g] <= kdk[g]) {
              now |= 1u << g;
              nkey = min(nkey, key[g]);
            }
        }
        const uint32_t mn = __reduce_min_sync(0xFFFFFFFFu, nkey);
        if (mn == 0xFFFFFFFFu) break;  // no query needs any remaining leaf
        const int src = __ffs(__ballot_sync(0xFFFFFFFFu, now && nkey == mn)) - 1;
        ml &= ~(1u << src);
        const uint32_t qm = __shfl_sync(0xFFFFFFFFu, now, src);
        const uint32_t lref = __shfl_sync(0xFFFFFFFFu, cref, src);
        const int lcnt = __shfl_sync(0xFFFFFFFFu, ccnt, src);
        knn_scan_group<D, G, false>(t, lref, lcnt, qc, kl, a.k, qm);
#pragma unroll
        for (int g = 0; g < G; ++g) kdk[g] = order_key(kl[g].kd);
        if (STATS) {
          ++n_leaf;
          n_pts += lcnt;
        }
      }
    };
    if (root >= 0) {
      if (t.kids[root] == 0) {
        bool sd_root = false;
#pragma unroll
        for (int g = 0; g < G; ++g) sd_root |= seed[g] == (uint32_t)root;
        if (!sd_root) knn_scan_group<D, G, false>(t, t.ref[root], t.cnt[root], qc, kl, a.k, all);
      } else {
        uint32_t c0 = t.ref[root], pk0 = 0, pk1 = 0;
        int nk = t.kids[root];
        bool pl = false;
        for (;;) {  // one call site keeps `expand` inlined
          expand(c0, nk, pl, pk0, pk1);
          // RECHECK: the next entry that some query still needs under its
          // k-th distance of this moment (the others are dropped unexpanded)
          bool more = false;
          while (sp > 0) {
            const Entry e = s_stk[w][--sp];
            bool need = true;
            if constexpr (RECHECK) {
              need = e.z <= kdk[0] || (G > 1 && e.w <= kdk[G - 1]);
              pl = (e.y & kLeafEntry) != 0;
              pk0 = e.z;
              pk1 = e.w;
            }
            if (need) {
              c0 = e.x;
              nk = (int)(e.y & ~kLeafEntry);
              more = true;
              break;
            }
          }
          if (!more) break;
        }
      }
    }
#pragma unroll
    for (int g = 0; g < G; ++g) {
      if (g < ng && lane < a.k) {
        const int64_t q = take.query(qi0 + g);
        a.out_id[q * a.k + lane] = kl[g].i[0];
        a.out_d2[q * a.k + lane] = kl[g].d[0];
      }
    }
    if (STATS && lane == 0) atomicAdd(&stats.c[3], (unsigned long long)ng);
  }
  if (STATS && lane == 0) {
    atomicAdd(&stats.c[0], n_int);
    atomicAdd(&stats.c[1], n_leaf);
    atomicAdd(&stats.c[2], n_pts);
    atomicAdd(&stats.c[4], n_kids);
  }
}

struct RangeArgs {
  TreeView t;
  const int32_t *boxes;
  int64_t nq;
  int64_t *counts;          // count pass
  const int64_t *offsets;   // emit pass
  uint32_t *out_ids;
  int *status;
};

template <int D>
__device__ __forceinline__ bool point_in(const TreeView &t, uint32_t slot, const int32_t *blo, const int32_t *bhi) {
  bool in = true;
#pragma unroll
  for (int d = 0; d < D; ++d) {
    const int32_t c = t.px[d][slot];
    in &= c >= blo[d] && c <= bhi[d];
  }
  return in;
}

// EMIT = false: count; EMIT = true: write ids.
// One warp per box.  The internal nodes the box reaches wait on a stack as
// (first child, children | INSIDE), taken from their parent's expansion, so a
// pop reads no node record.  Expanding a node loads every child's record and
// box in one round of loads; internal children are pushed, and leaf children
// are scanned at once (slot range and count already in registers): a leaf
// costs one dependent load of its points instead of a trip through the stack.
// The count pass adds the count of a node inside the box without descending.
template <int D, bool EMIT>
__global__ __launch_bounds__(QW * 32) void k_range(RangeArgs a) {
  __shared__ uint2 s_node[QW][STACK];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t nw = (int64_t)gridDim.x * QW;
  const TreeView &t = a.t;
  for (int64_t q = (int64_t)blockIdx.x * QW + w; q < a.nq; q += nw) {
    int32_t blo[D], bhi[D];
#pragma unroll
    for (int d = 0; d < D; ++d) {
      blo[d] = a.boxes[q * 2 * D + d];
      bhi[d] = a.boxes[q * 2 * D + D + d];
    }
    int64_t acc = 0;                               // count pass: per-lane partial
    int64_t cursor = EMIT ? a.offsets[q] : 0;      // emit pass: warp-uniform
    // the root enters as the one child of a virtual node
    int sp = 0;
    if (t.root >= 0) {
      if (lane == 0) s_node[w][0] = make_uint2((uint32_t)t.root, 1u);
      sp = 1;
    }
    __syncwarp();
    while (sp > 0) {
      --sp;
      const uint2 e = s_node[w][sp];
      __syncwarp();
      const uint32_t c0 = e.x;
      const int nk = (int)(e.y & ~INSIDE);
      const bool inside = (e.y & INSIDE) != 0;
      // children per node: at most 32 (SPaC fanout <= 32, P-Orth 2^D <= 8)
      if (nk > 32 && lane == 0) atomicOr(a.status, ST_STACK);
      bool ok = false, lf = false;
      int rel = 0, ccnt = 0, ck = 0;
      uint32_t cref = 0;
      if (lane < nk) {
        const uint32_t c = c0 + (uint32_t)lane;
        ck = t.kids[c];
        cref = t.ref[c];
        ccnt = t.cnt[c];
        rel = inside ? 2 : box_relation<D>(t, c, blo, bhi);
        lf = ck == 0;
        if (rel == 2 && !EMIT)
          acc += ccnt;
        else
          ok = rel != 0;
      }
      // internal children: pushed
      const bool push = ok && !lf;
      const uint32_t m = __ballot_sync(0xFFFFFFFFu, push);
      if (sp + __popc(m) > STACK) {
        if (lane == 0) atomicOr(a.status, ST_STACK);
        break;
      }
      if (push) s_node[w][sp + __popc(m & lanemask_lt())] = make_uint2(cref, (uint32_t)ck | (rel == 2 ? INSIDE : 0u));
      sp += __popc(m);
      __syncwarp();
      // leaf children: scanned now
      uint32_t ml = __ballot_sync(0xFFFFFFFFu, ok && lf);
      if constexpr (!EMIT) {
        while (ml) {
          const int src = __ffs(ml) - 1;
          ml &= ml - 1;
          const uint32_t s0 = __shfl_sync(0xFFFFFFFFu, cref, src);
          const int cnt = __shfl_sync(0xFFFFFFFFu, ccnt, src);
          const bool lin = __shfl_sync(0xFFFFFFFFu, rel, src) == 2;  // leaf box inside the query box
          for (int b = 0; b < cnt; b += 32) {
            const int s = b + lane;
            acc += s < cnt && (lin || point_in<D>(t, s0 + (uint32_t)s, blo, bhi));
          }
        }
      } else {
        // two leaves per round, each lane's points and ids loaded together, so
        // that the loads of both leaves are in flight at once
        while (ml) {
          const int sa = __ffs(ml) - 1;
          ml &= ml - 1;
          const bool two = ml != 0;
          const int sb = two ? __ffs(ml) - 1 : sa;
          if (two) ml &= ml - 1;
          const uint32_t s0a = __shfl_sync(0xFFFFFFFFu, cref, sa), s0b = __shfl_sync(0xFFFFFFFFu, cref, sb);
          const int cna = __shfl_sync(0xFFFFFFFFu, ccnt, sa);
          const int cnb = two ? __shfl_sync(0xFFFFFFFFu, ccnt, sb) : 0;
          const bool lina = __shfl_sync(0xFFFFFFFFu, rel, sa) == 2, linb = __shfl_sync(0xFFFFFFFFu, rel, sb) == 2;
          // the first 32 slots of both leaves
          const bool va = lane < cna, vb = lane < cnb;
          int32_t pa[D], pb[D];
#pragma unroll
          for (int d = 0; d < D; ++d) {
            pa[d] = va && !lina ? t.px[d][s0a + lane] : 0;
            pb[d] = vb && !linb ? t.px[d][s0b + lane] : 0;
          }
          const uint32_t ia = va ? t.pid[s0a + lane] : 0u, ib = vb ? t.pid[s0b + lane] : 0u;
          bool ha = va, hb = vb;
#pragma unroll
          for (int d = 0; d < D; ++d) {
            ha &= lina || (pa[d] >= blo[d] && pa[d] <= bhi[d]);
            hb &= linb || (pb[d] >= blo[d] && pb[d] <= bhi[d]);
          }
          const uint32_t ma = __ballot_sync(0xFFFFFFFFu, ha);
          if (ha) a.out_ids[cursor + __popc(ma & lanemask_lt())] = ia;
          cursor += __popc(ma);
          const uint32_t mb = __ballot_sync(0xFFFFFFFFu, hb);
          if (hb) a.out_ids[cursor + __popc(mb & lanemask_lt())] = ib;
          cursor += __popc(mb);
          // leaves of more than 32 points: their remaining slots
#pragma unroll 1
          for (int u = 0; u < 2; ++u) {
            const uint32_t s0 = u ? s0b : s0a;
            const int cnt = u ? cnb : cna;
            const bool lin = u ? linb : lina;
            for (int b = 32; b < cnt; b += 32) {
              const int s = b + lane;
              const bool hit = s < cnt && (lin || point_in<D>(t, s0 + (uint32_t)s, blo, bhi));
              const uint32_t hm = __ballot_sync(0xFFFFFFFFu, hit);
              if (hit) a.out_ids[cursor + __popc(hm & lanemask_lt())] = t.pid[s0 + s];
              cursor += __popc(hm);
            }
          }
        }
      }
    }
    if (!EMIT) {
      for (int o = 16; o; o >>= 1) acc += __shfl_down_sync(0xFFFFFFFFu, acc, o);
      if (lane == 0) a.counts[q] = acc;
    }
  }
}

// ---- ascending sort of each query's ids ------------------------------------
// Bitonic sort of T * E values held E per thread (value e of thread t at
// position t * E + e) by a group of T threads: strides below E between a
// thread's own registers, strides below 32 E by warp shuffles, the others
// through shared memory ([E][T]; T > 32 only).  HALF: the group is one of the
// halves of a block of 2 T threads, with a barrier of its own.
template <int T, bool HALF>
__device__ __forceinline__ void seg_sync() {
  if (T == 32)
    __syncwarp();
  else if (HALF && threadIdx.x < T)  // (numbers known to the compiler: three barriers in all)
    asm volatile("bar.sync 1, %0;" ::"n"(T) : "memory");
  else if (HALF)
    asm volatile("bar.sync 2, %0;" ::"n"(T) : "memory");
  else
    __syncthreads();
}

template <int T, int E, bool HALF = false>
__device__ __forceinline__ void seg_bitonic(uint32_t (&v)[E], uint32_t *sm) {
  const int t = T == 32 || HALF ? (int)(threadIdx.x & (T - 1)) : (int)threadIdx.x;
  // strides from .. 1 between the thread's own values: stage k < E, whose runs
  // alternate inside the thread, or (k >= E) an ascending merge
  auto own = [&](int from, int k) {
#pragma unroll
    for (int j = E / 2; j > 0; j >>= 1)
      if (j <= from) {
#pragma unroll
        for (int e = 0; e < E; ++e)
          if (!(e & j)) {
            const bool asc = k >= E || (e & k) == 0;
            const uint32_t a = min(v[e], v[e | j]), b = max(v[e], v[e | j]);
            v[e] = asc ? a : b;
            v[e | j] = asc ? b : a;
          }
      }
  };
  // From stage E on a run is a thread's or several threads': the threads of a
  // descending one hold complements, so that every exchange ascends.
  uint32_t flip = 0;
  auto turn = [&](int k) {
    const uint32_t f = (t * E & k) == 0 ? 0u : 0xFFFFFFFFu;
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] ^= flip ^ f;
    flip = f;
  };
#pragma unroll
  for (int k = 2; k < E; k <<= 1) own(k / 2, k);
  if (E > 1) {
    turn(E);
    own(E / 2, E);
  }
#pragma unroll 1
  for (int k = 2 * E; k <= T * E; k <<= 1) {
    turn(k);
    int j = k / 2;
    if (T > 32) {
#pragma unroll 1
      for (; j >= 32 * E; j >>= 1) {
        seg_sync<T, HALF>();
#pragma unroll
        for (int e = 0; e < E; ++e) sm[e * T + t] = v[e];
        seg_sync<T, HALF>();
        const int x = t ^ (j / E);
        const bool low = (t & (j / E)) == 0;
#pragma unroll
        for (int e = 0; e < E; ++e) {
          const uint32_t o = sm[e * T + x];
          v[e] = low ? min(v[e], o) : max(v[e], o);
        }
      }
    }
#pragma unroll 1
    for (; j >= E; j >>= 1) {
      const bool low = (t & (j / E)) == 0;
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const uint32_t o = __shfl_xor_sync(0xFFFFFFFFu, v[e], j / E);
        v[e] = low ? min(v[e], o) : max(v[e], o);
      }
    }
    own(E / 2, k);
  }
}

// Sorts ids[0, len), len <= T * E.  The order of the values on the way in is
// free, so they are read coalesced; they leave through shared memory, where
// the group holds T * (E + 1) words.
template <int T, int E, bool HALF = false>
__device__ __forceinline__ void seg_sort(uint32_t *ids, int len, uint32_t *sm) {
  const int t = T == 32 || HALF ? (int)(threadIdx.x & (T - 1)) : (int)threadIdx.x;
  uint32_t v[E];
#pragma unroll
  for (int e = 0; e < E; ++e) v[e] = e * T + t < len ? ids[e * T + t] : 0xFFFFFFFFu;
  seg_bitonic<T, E, HALF>(v, sm);
  seg_sync<T, HALF>();
  constexpr int S = E > 1 ? E + 1 : 1;  // a word of padding per thread: no bank conflicts
#pragma unroll
  for (int e = 0; e < E; ++e) sm[t * S + e] = v[e];
  seg_sync<T, HALF>();
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int p = e * T + t;
    if (p < len) ids[p] = sm[p / E * S + p % E];
  }
  seg_sync<T, HALF>();
}

// The segments by length, each class sorted by a kernel of its own: a warp per
// segment up to 1024 ids, then 64, 128 and 512 threads (the first two in one
// launch: a launch costs a small report 4 us), then k_sort_seg_any.  Many values per thread keep most of the network in registers:
// at 1024 ids, 15 of its 55 stages are shuffles (whose rate bounds it) with 32
// values per thread; 28 are between threads with 8.  The classes are listed
// first and every warp or block takes the next segment of its list: taken in
// strides over all segments, some find more of their class than others.  5e4
// boxes of 1259 ids on average (6.3e7 ids): 590 us, against 6.1 ms for one
// 1024-thread block per segment with a network in shared memory and a barrier
// per stage; bound by instruction issue (about 110 per id and 32 lanes).
constexpr int kSegClasses = 5;
constexpr int kSeg0 = 1024, kSeg1 = 2048, kSeg2 = 4096, kSeg3 = 16384;  // largest of classes 0 to 3

struct SegLists {
  uint32_t *list;  // [kSegClasses][nq]
  uint32_t *ctr;   // [kSegClasses] lengths of the lists, [kSegClasses] next to take
  int64_t nq;
};

__global__ __launch_bounds__(256) void k_seg_classes(const int64_t *offsets, SegLists l) {
  const int lane = threadIdx.x & 31;
  const int64_t rounds = (l.nq + 31) / 32 * 32;
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < rounds; q += (int64_t)gridDim.x * blockDim.x) {
    const int64_t len = q < l.nq ? offsets[q + 1] - offsets[q] : 0;
    const int c = len < 2 ? -1 : (len > kSeg0) + (len > kSeg1) + (len > kSeg2) + (len > kSeg3);
#pragma unroll
    for (int x = 0; x < kSegClasses; ++x) {
      const uint32_t m = __ballot_sync(0xFFFFFFFFu, c == x);
      if (!m) continue;
      uint32_t base = 0;
      if (lane == 0) base = atomicAdd(&l.ctr[x], (uint32_t)__popc(m));
      base = __shfl_sync(0xFFFFFFFFu, base, 0);
      if (c == x) l.list[x * l.nq + base + __popc(m & lanemask_lt())] = (uint32_t)q;
    }
  }
}

// Class 0: a warp per segment, E chosen so that at least half of the positions
// hold ids.
__global__ __launch_bounds__(128, 8) void k_sort_seg_warp(const int64_t *offsets, SegLists l, uint32_t *ids) {
  __shared__ uint32_t sm[4][32 * 33];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t n = l.ctr[0];
  for (;;) {
    uint32_t x = 0;
    if (lane == 0) x = atomicAdd(&l.ctr[kSegClasses], 1u);
    x = __shfl_sync(0xFFFFFFFFu, x, 0);
    if (x >= n) break;
    const int64_t q = l.list[x], b = offsets[q];
    const int len = (int)(offsets[q + 1] - b);
    if (len <= 32)
      seg_sort<32, 1>(ids + b, len, sm[w]);
    else if (len <= 64)
      seg_sort<32, 2>(ids + b, len, sm[w]);
    else if (len <= 128)
      seg_sort<32, 4>(ids + b, len, sm[w]);
    else if (len <= 256)
      seg_sort<32, 8>(ids + b, len, sm[w]);
    else if (len <= 512)
      seg_sort<32, 16>(ids + b, len, sm[w]);
    else
      seg_sort<32, 32>(ids + b, len, sm[w]);
  }
}

// The next segment of class c for a group of threads (lead: one of them), or
// its number past the class's end.
template <int T, bool HALF>
__device__ __forceinline__ uint32_t seg_next(const SegLists &l, int c, uint32_t &slot, bool lead) {
  if (lead) slot = atomicAdd(&l.ctr[kSegClasses + c], 1u);
  seg_sync<T, HALF>();
  const uint32_t x = slot;
  seg_sync<T, HALF>();
  return x;
}

// Class 1 by the halves of a block, 64 threads each, then class 2 by whole
// blocks: one launch for both.
__global__ __launch_bounds__(128, 8) void k_sort_seg_mid(const int64_t *offsets, SegLists l, uint32_t *ids) {
  __shared__ uint32_t sm[128 * 33];
  __shared__ uint32_t next[2];
  const int h = threadIdx.x >> 6;
  for (const uint32_t n = l.ctr[1];;) {
    const uint32_t x = seg_next<64, true>(l, 1, next[h], (threadIdx.x & 63) == 0);
    if (x >= n) break;
    const int64_t q = l.list[l.nq + x], b = offsets[q];
    seg_sort<64, 32, true>(ids + b, (int)(offsets[q + 1] - b), sm + h * (64 * 33));
  }
  __syncthreads();
  for (const uint32_t n = l.ctr[2];;) {
    const uint32_t x = seg_next<128, false>(l, 2, next[0], threadIdx.x == 0);
    if (x >= n) break;
    const int64_t q = l.list[2 * l.nq + x], b = offsets[q];
    seg_sort<128, 32>(ids + b, (int)(offsets[q + 1] - b), sm);
  }
}

// Class 3: a block of 512 threads per segment.
__global__ __launch_bounds__(512, 2) void k_sort_seg_block(const int64_t *offsets, SegLists l, uint32_t *ids) {
  extern __shared__ uint32_t sm_seg[];  // 512 * 33
  __shared__ uint32_t next;
  for (const uint32_t n = l.ctr[3];;) {
    const uint32_t x = seg_next<512, false>(l, 3, next, threadIdx.x == 0);
    if (x >= n) break;
    const int64_t q = l.list[3 * l.nq + x], b = offsets[q];
    const int len = (int)(offsets[q + 1] - b);
    if (len <= 16 * 512)
      seg_sort<512, 16>(ids + b, len, sm_seg);
    else
      seg_sort<512, 32>(ids + b, len, sm_seg);
  }
}

// A block of 1024 threads per segment of any length: all segments of a call of
// few boxes, or (LIST) those of the last class.  Up to 16384 ids in registers,
// longer ones in place in global memory, where the network is bound by the
// threads at work: 8 lists of 2e5 ids 11.8 ms with 1024 threads, 20.4 with 512.
constexpr int kSegT = 1024, kSegTMax = 16 * kSegT;

template <bool LIST>
__global__ __launch_bounds__(kSegT, 1) void k_sort_seg_any(const int64_t *offsets, SegLists l, uint32_t *ids) {
  extern __shared__ uint32_t sm_seg[];  // kSegT * 17
  const int64_t n = LIST ? (int64_t)l.ctr[kSegClasses - 1] : l.nq;
  for (int64_t x = blockIdx.x; x < n; x += gridDim.x) {
    const int64_t q = LIST ? (int64_t)l.list[(kSegClasses - 1) * l.nq + x] : x;
    const int64_t b = offsets[q], len = offsets[q + 1] - b;
    uint32_t *v = ids + b;
    if (len < 2) continue;
    if (len > kSegTMax) {
      bitonic_ascending(
          len, [&](int64_t i, int64_t j) { return v[i] < v[j]; },
          [&](int64_t i, int64_t j) {
            const uint32_t tmp = v[i];
            v[i] = v[j];
            v[j] = tmp;
          });
    } else if (!LIST) {
      if (len <= 256) {  // one warp: no barriers
        if (threadIdx.x < 32) {
          if (len <= 32)
            seg_sort<32, 1>(v, (int)len, sm_seg);
          else if (len <= 64)
            seg_sort<32, 2>(v, (int)len, sm_seg);
          else
            seg_sort<32, 8>(v, (int)len, sm_seg);
        }
        __syncthreads();
      } else if (len <= 1 * kSegT) {
        seg_sort<kSegT, 1>(v, (int)len, sm_seg);
      } else if (len <= 4 * kSegT) {
        seg_sort<kSegT, 4>(v, (int)len, sm_seg);
      } else {
        seg_sort<kSegT, 16>(v, (int)len, sm_seg);
      }
    }
  }
}

template <bool LIST>
psi_status launch_sort_seg_any(const int64_t *offsets, const SegLists &l, uint32_t *ids, cudaStream_t s) {
  const size_t smem = LIST ? 0 : sizeof(uint32_t) * kSegT * 17;
  if (smem > 48 * 1024)
    PSI_CK(cudaFuncSetAttribute(k_sort_seg_any<LIST>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  PSI_LAUNCH_NAMED("k_sort_seg_any", k_sort_seg_any<LIST>,
                   (int)std::min<int64_t>(l.nq, (int64_t)num_sms() * (LIST ? 2 : 1)), kSegT, smem, s, offsets, l, ids);
  return PSI_OK;
}

// With at most a segment per SM one launch sorts them all, without lists: 10
// lists of 30 ids 5.7 us (by classes 34 with their launches, under the event
// timer), 150 of 3000 14.8 (50.0), 150 of 20000 586 (644).  More lists queue up
// behind its one block per SM: 300 of 20000 1156 us (919).
psi_status sort_segments(const int64_t *offsets, int64_t nq, uint32_t *ids, cudaStream_t s) {
  if (nq <= num_sms()) return launch_sort_seg_any<false>(offsets, SegLists{nullptr, nullptr, nq}, ids, s);
  Buf<uint32_t> list, ctr;
  psi_status st;
  if ((st = list.alloc(kSegClasses * nq, s)) || (st = ctr.alloc(2 * kSegClasses, s))) return st;
  PSI_CK(cudaMemsetAsync(ctr.p, 0, sizeof(uint32_t) * 2 * kSegClasses, s));
  const SegLists l{list.p, ctr.p, nq};
  PSI_LAUNCH(k_seg_classes, (int)std::min<int64_t>(ceil_div(nq, 256), (int64_t)num_sms() * 8), 256, 0, s, offsets, l);
  PSI_LAUNCH(k_sort_seg_warp, (int)std::min<int64_t>(ceil_div(nq, 4), (int64_t)num_sms() * 8), 128, 0, s, offsets, l,
             ids);
  PSI_LAUNCH(k_sort_seg_mid, (int)std::min<int64_t>(nq, (int64_t)num_sms() * 8), 128, 0, s, offsets, l, ids);
  const size_t smem = sizeof(uint32_t) * 512 * 33;
  PSI_CK(cudaFuncSetAttribute(k_sort_seg_block, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  PSI_LAUNCH(k_sort_seg_block, (int)std::min<int64_t>(nq, (int64_t)num_sms() * 2), 512, smem, s, offsets, l, ids);
  return launch_sort_seg_any<true>(offsets, l, ids, s);
}

// Grid of a grid-stride query kernel: the blocks that are resident at once
// (a larger grid would run as a second, partly idle wave).
template <typename Kern>
int resident_query_grid(Kern kern, int64_t nq) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, QW * 32, 0) != cudaSuccess || per_sm < 1) {
    cudaGetLastError();
    per_sm = 1;
  }
  return (int)std::max<int64_t>(1, std::min<int64_t>(ceil_div(nq, QW), (int64_t)num_sms() * per_sm));
}

}  // namespace

// Sorts the query points along the index's curve so that neighbouring warps
// traverse neighbouring parts of the tree; returns the permutation in *order
// and the sorted keys (curve key >> *key_shift) in *qkeys.
psi_status query_order(const psi_index *ix, const int32_t *q, int64_t nq, QueryOrder &qo, cudaStream_t s) {
  qo.order = nullptr;
  qo.keys = nullptr;
  if (nq < 4096) return PSI_OK;
  psi_status st;
  if ((st = qo.k0.alloc(nq, s)) || (st = qo.k1.alloc(nq, s)) || (st = qo.v0.alloc(nq, s)) ||
      (st = qo.v1.alloc(nq, s)))
    return st;
  // locality only needs the top bits of the curve key: 48 bits, 6 digit passes
  EncodeSpec e = encode_spec(ix, q);
  const int order_bits = std::min(48, ix->key_bits);
  e.key_shift = ix->key_bits - order_bits;
  SortResult r;
  if ((st = sort_pairs(e, nullptr, nullptr, nq, order_bits, nullptr, qo.k0.p, qo.v0.p, qo.k1.p, qo.v1.p,
                       ix->d_status, s, &r)))
    return st;
  qo.order = r.vals;
  qo.keys = r.keys;
  qo.key_shift = e.key_shift;
  qo.spare = reinterpret_cast<uint32_t *>(r.keys == qo.k0.p ? qo.k1.p : qo.k0.p);
  qo.spare_v = r.vals == qo.v0.p ? qo.v1.p : qo.v0.p;
  return PSI_OK;
}

// Fewest queries for which the one-query-per-thread kernel is the faster one,
// over n points on a chip of sms multiprocessors.  It needs the chip full of
// queries (a wave is 8 blocks of 128 per SM), more of them the longer the lists
// and, above some 3e6 points, the farther apart the queries of a warp are, whose
// shared walk is the longer.  The lines are read from 8e3 timings, 3e5 to 1e8
// points, uniform and Varden, 2e4 to 2e6 queries.  Other kernel / this one, in
// us, 10-NN at data points: 2D SPaC-H 3e5 queries on 3e6 points 562 / 395, on 1e8
// 706 / 732, 1e6 on 1e8 2072 / 1340; 3D SPaC-H 3e5 on 3e5 710 / 464, on 1e8 1141 /
// 1486, 1e6 on 1e8 3348 / 3025; 3D P-Orth 6e5 on 3e6 2014 / 1196, on 3e7 2364 /
// 2218.  A batch's other kernel takes one query per warp and is ahead for longer
// in 3D: 64 indexes of 1e6 uniform points, 10-NN of 4.7e5 queries 1484 / 1604, of
// 1.2e6 3906 / 2913 (Varden 1616 / 2474, 4187 / 5319).
static int64_t lane_min_queries(int sms, int D, int k, bool porth, bool batch, int64_t n) {
  if (k > kLaneMaxK) return INT64_MAX;
  // [P-Orth][D - 2]: waves at 3e6 points by k, and the exponent of the points
  static constexpr struct {
    double k1, k5, k10, k13, k16, c;
  } kFit[2][2] = {{{0.33, 0.36, 0.55, 0.8, 0.8, 0.35}, {0.38, 0.5, 0.85, 1.5, 1.5, 0.38}},
                  {{0.3, 0.35, 0.45, 0.9, 1.2, 0.3}, {0.33, 0.6, 1.1, 1.6, 3.0, 0.33}}};
  const auto &f = kFit[porth][D - 2];
  double waves = k == 1 ? f.k1 : k <= 5 ? f.k5 : k <= 10 ? f.k10 : k <= 13 ? f.k13 : f.k16;
  waves *= std::pow(std::max(1.0, (double)n / 3e6), f.c);
  if (batch && D == 3) waves *= 1.2;
  // (P-Orth queries away from the data are only listed here: at one wave the
  // whole call is 0.80 to 0.89 times as fast, at two 0.85 to 1)
  return (int64_t)((double)sms * 1024 * std::max(waves, porth && k > 1 ? 1.9 : 1.0));
}

// On P-Orth, one query per warp with small leaves scanned together, for few
// queries (the chip is not full, a query's latency counts), long lists and large
// trees; else two queries per warp with one leaf at a time.  The line is fitted
// to the same timings.  Two per warp / one, in us, at data points: 3D uniform 3e6
// points 10-NN 2e4 queries 165 / 130, 6e5 2014 / 2403; 3D Varden 3e5 points 10-NN
// 6e5 2082 / 3034; 3D uniform 1e8 points 32-NN 2e4 1023 / 256, 6e5 8781 / 5345.
static int64_t porth_single_max(int D, int k, int64_t n) {
  const double m = (double)n / 1e6;
  const double line =
      D == 2 ? 7450 * std::pow((double)k, 0.7) * std::pow(m, 0.3) : 5960 * k * std::pow(std::max(m, 0.6), 0.6);
  return (int64_t)std::max(line, 12000.0);
}
static bool porth_single(int D, int k, int64_t nq, int64_t n) { return nq < porth_single_max(D, k, n); }

psi_status run_knn_roots(const TreeView &tv, int64_t n, const int32_t *q, int64_t nq, int k, const uint32_t *order,
                         const int32_t *qroot, int D, uint32_t *out_id, int64_t *out_d2, int *status,
                         unsigned long long *d_stats, cudaStream_t s, const KnnSeed &seed, int64_t leaf_limit,
                         bool porth, const KnnHard &hard) {
  if (nq == 0) return PSI_OK;
  KnnArgs a{tv, q, nq, k, order, qroot, seed, leaf_limit, out_id, out_d2, status};
  KnnStats stats{d_stats};
  if (seed.qkey) {
    if (!seed.pos) {
      set_error("k-NN seed without its scratch");
      return PSI_ERR_INVALID;
    }
    const int gs = (int)std::max<int64_t>(1, std::min<int64_t>(ceil_div(nq, 256), (int64_t)num_sms() * 16));
    PSI_LAUNCH(k_knn_seed, gs, 256, 0, s, seed, tv.ref, order, nq, seed.pos);
  }
  if (hard.q && !d_stats && nq >= lane_min_queries(num_sms(), D, k, porth, qroot != nullptr, n)) {
    PSI_CK(cudaMemsetAsync(hard.n, 0, sizeof(uint32_t), s));
    LaneArgs l{a, hard.q, hard.pos, hard.n};
    psi_status st = run_knn_lane(l, D, porth, s);
    if (st) return st;
    // the queries it left out, a warp for each or (SPaC, and long lists on P-Orth)
    // for two: their number is known on the device only, so on P-Orth both kernels
    // are launched and one of them finds nothing to do.  Neighbours on a short list
    // are rarely neighbours in space, so up to a quarter of the queries its line
    // lies three times as high (6.2e5 10-NN on 3e5 3D Varden points, 1.27 times as
    // fast with a warp each).
    a.all_order = order;
    a.all_pos = seed.pos;
    a.order = hard.q;
    a.seed.pos = hard.pos;
    a.d_nq = hard.n;
#define KNN_LIST(DD, PP)                                                                                            \
  do {                                                                                                              \
    const int64_t one = porth_single_max(D, k, n);                                                                  \
    const int64_t split = PP ? std::max(one, std::min(3 * one, nq / 4)) : qroot ? INT64_MAX : 0;                     \
    if (split > 0) {                                                                                                 \
      a.list_lo = 0;                                                                                                 \
      a.list_hi = split;                                                                                             \
      PSI_LAUNCH_NAMED("k_knn", (k_knn<DD, 1, false, PP, true>),                                                     \
                       resident_query_grid(k_knn<DD, 1, false, PP, true>, nq), QW * 32, 0, s, a, stats);             \
    }                                                                                                                \
    if (split < INT64_MAX) {                                                                                         \
      a.list_lo = split;                                                                                             \
      a.list_hi = INT64_MAX;                                                                                         \
      PSI_LAUNCH_NAMED("k_knn", (k_knn_group<DD, kGroup, false, PP, true>),                                          \
                       resident_query_grid(k_knn_group<DD, kGroup, false, PP, true>, ceil_div(nq, kGroup)), QW * 32, \
                       0, s, a, stats);                                                                              \
    }                                                                                                                \
  } while (0)
    if (D == 2) {
      if (porth) KNN_LIST(2, true);
      else KNN_LIST(2, false);
    } else {
      if (porth) KNN_LIST(3, true);
      else KNN_LIST(3, false);
    }
#undef KNN_LIST
    PSI_CK(cudaGetLastError());
    return PSI_OK;
  }
  const int kpl = k <= 32 ? 1 : (k <= 64 ? 2 : 4);
  // k <= 32 over one tree with queries in curve order: kGroup queries per warp
  if (kpl == 1 && !qroot && order && kGroup > 1 && !(porth && porth_single(D, k, nq, n))) {
#define KNN_GROUP(DD, RC)                                                                                   \
  do {                                                                                                      \
    if (d_stats)                                                                                            \
      PSI_LAUNCH_NAMED("k_knn_stats", (k_knn_group<DD, kGroup, true, RC>),                                  \
                       resident_query_grid(k_knn_group<DD, kGroup, true, RC>, ceil_div(nq, kGroup)), QW * 32, \
                       0, s, a, stats);                                                                     \
    else                                                                                                    \
      PSI_LAUNCH_NAMED("k_knn", (k_knn_group<DD, kGroup, false, RC>),                                       \
                       resident_query_grid(k_knn_group<DD, kGroup, false, RC>, ceil_div(nq, kGroup)), QW * 32, \
                       0, s, a, stats);                                                                     \
  } while (0)
    // Popped nodes are re-checked against the k-th distances where the
    // search pushes many that later bounds rule out: P-Orth, whose nodes mix
    // leaf and internal children at every depth.  SPaC's seeds make the
    // bounds nearly final before the first push, and there the larger stack
    // entries cost more than the re-check saves.
    const bool recheck = porth;
    if (D == 2) {
      if (recheck) KNN_GROUP(2, true);
      else KNN_GROUP(2, false);
    } else {
      if (recheck) KNN_GROUP(3, true);
      else KNN_GROUP(3, false);
    }
#undef KNN_GROUP
    PSI_CK(cudaGetLastError());
    return PSI_OK;
  }
  // few queries on a SPaC tree: each warp finds its query's seed leaf itself
  // (its steps are dependent loads, a few microseconds; without the seed the
  // search entered 2.6 to 7 times as many leaves: 1e3 10-NN on 1e7 Varden
  // points, 2D SPaC-H 65 -> 36 us, 3D SPaC-Z 287 -> 35 us).  For k > 32 the
  // search is long beside what the seed saves: 0.85 to 1.18 times as fast.  On
  // P-Orth, whose nearest-box-first descent is near its floor, a seed of 32
  // points around the query in key order cost more than it saved (41 -> 51 us).
  if (seed.self_bits > 0 && kpl == 1 && !d_stats) {
    if (D == 2)
      PSI_LAUNCH_NAMED("k_knn", (k_knn<2, 1, false, false, false, true>),
                       resident_query_grid(k_knn<2, 1, false, false, false, true>, nq), QW * 32, 0, s, a, stats);
    else
      PSI_LAUNCH_NAMED("k_knn", (k_knn<3, 1, false, false, false, true>),
                       resident_query_grid(k_knn<3, 1, false, false, false, true>, nq), QW * 32, 0, s, a, stats);
    PSI_CK(cudaGetLastError());
    return PSI_OK;
  }
  // Few queries on P-Orth leave the chip waiting on the chain of dependent node
  // loads of each search: once a query's list is full, up to four nodes are
  // expanded at once, at the price of some that single steps would have pruned.
  // Before that there is no bound and the nearest node is the one wanted: four at
  // once from the start took 18.5 us for 4e3 1-NN at data points of 1e6 3D uniform
  // points, single steps 14.4.  Over 2D and 3D, 3e4 to 2e7 points, 1 to 4e3 queries
  // at, near and away from the data: 1.00 to 1.38 times as fast as single steps.
  if (porth && kpl == 1 && !order && !d_stats) {
    if (D == 2)
      PSI_LAUNCH_NAMED("k_knn", (k_knn<2, 1, false, true, false, false, true>),
                       resident_query_grid(k_knn<2, 1, false, true, false, false, true>, nq), QW * 32, 0, s, a, stats);
    else
      PSI_LAUNCH_NAMED("k_knn", (k_knn<3, 1, false, true, false, false, true>),
                       resident_query_grid(k_knn<3, 1, false, true, false, false, true>, nq), QW * 32, 0, s, a, stats);
    PSI_CK(cudaGetLastError());
    return PSI_OK;
  }
#define KNN_CASE1(DD, KK, BB)                                                                          \
  do {                                                                                                 \
    if (d_stats)                                                                                       \
      PSI_LAUNCH_NAMED("k_knn_stats", (k_knn<DD, KK, true, BB>),                                       \
                       resident_query_grid(k_knn<DD, KK, true, BB>, nq), QW * 32, 0, s, a, stats);     \
    else                                                                                               \
      PSI_LAUNCH_NAMED("k_knn", (k_knn<DD, KK, false, BB>), resident_query_grid(k_knn<DD, KK, false, BB>, nq), \
                       QW * 32, 0, s, a, stats);                                                       \
  } while (0)
  // small leaves in batches where leaves are not one round each (P-Orth)
#define KNN_CASE(DD, KK)                  \
  do {                                    \
    if (porth)                            \
      KNN_CASE1(DD, KK, true);            \
    else                                  \
      KNN_CASE1(DD, KK, false);           \
  } while (0)
  if (D == 2) {
    if (kpl == 1) KNN_CASE(2, 1);
    else if (kpl == 2) KNN_CASE(2, 2);
    else KNN_CASE(2, 4);
  } else {
    if (kpl == 1) KNN_CASE(3, 1);
    else if (kpl == 2) KNN_CASE(3, 2);
    else KNN_CASE(3, 4);
  }
#undef KNN_CASE
#undef KNN_CASE1
  PSI_CK(cudaGetLastError());
  return PSI_OK;
}



psi_status run_knn(const psi_index *ix, const int32_t *q, int64_t nq, int k, uint32_t *out_id, int64_t *out_d2,
                   unsigned long long *d_stats, cudaStream_t s) {
  if (nq == 0) return PSI_OK;
  QueryOrder qo;
  psi_status st = query_order(ix, q, nq, qo, s);
  if (st) return st;
  KnnSeed seed;
  KnnHard hard;
  Buf<uint32_t> nhard;
  if (qo.keys) {
    if ((st = nhard.alloc(1, s))) return st;
    hard.q = qo.spare + nq;
    hard.pos = qo.spare_v;
    hard.n = nhard.p;
    seed.qkey = qo.keys;
    seed.L = ix->L;
    seed.key_shift = qo.key_shift;
    seed.pos = qo.spare;
    seed.sep_key = ix->sep_key;
    if (ix->cfg.kind == PSI_PORTH) {
      // the leaf whose cell holds (or last precedes) the query's key
      seed.sep_key = ix->pl.key;
      seed.leaf_node = ix->leaf_node;
    }
  }
  if (!qo.keys && ix->L > 0 && ix->cfg.kind != PSI_PORTH) {  // few queries, not sorted
    seed.self_bits = ix->cfg.coord_bits;
    seed.curve = ix->curve;
    seed.sep_key = ix->sep_key;
    seed.L = ix->L;
  }
  return run_knn_roots(ix->view(), ix->n, q, nq, k, qo.order, nullptr, ix->D, out_id, out_d2, ix->d_status, d_stats, s,
                       seed, ix->cfg.kind == PSI_PORTH ? -1 : ix->L, ix->cfg.kind == PSI_PORTH, hard);
}

psi_status run_range_count(const psi_index *ix, const int32_t *boxes, int64_t nq, int64_t *counts, cudaStream_t s) {
  if (nq == 0) return PSI_OK;
  RangeArgs a{ix->view(), boxes, nq, counts, nullptr, nullptr, ix->d_status};
  if (ix->D == 2)
    PSI_LAUNCH_NAMED("k_range_count", (k_range<2, false>), resident_query_grid(k_range<2, false>, nq), QW * 32, 0, s,
                     a);
  else
    PSI_LAUNCH_NAMED("k_range_count", (k_range<3, false>), resident_query_grid(k_range<3, false>, nq), QW * 32, 0, s,
                     a);
  PSI_CK(cudaGetLastError());
  return PSI_OK;
}

psi_status run_range_emit(const psi_index *ix, const int32_t *boxes, int64_t nq, const int64_t *offsets,
                          uint32_t *ids, bool sorted, cudaStream_t s) {
  if (nq == 0) return PSI_OK;
  RangeArgs a{ix->view(), boxes, nq, nullptr, offsets, ids, ix->d_status};
  if (ix->D == 2)
    PSI_LAUNCH_NAMED("k_range_emit", (k_range<2, true>), resident_query_grid(k_range<2, true>, nq), QW * 32, 0, s, a);
  else
    PSI_LAUNCH_NAMED("k_range_emit", (k_range<3, true>), resident_query_grid(k_range<3, true>, nq), QW * 32, 0, s, a);
  if (sorted) {
    psi_status st = sort_segments(offsets, nq, ids, s);
    if (st) return st;
  }
  PSI_CK(cudaGetLastError());
  return PSI_OK;
}

}  // namespace psi

// Test hook of the rules above: the kernel that psi_knn chooses for queries in
// curve order on one index ('L' one query per thread, 'S' one per warp, 'G' two).
extern "C" int32_t psi_test_knn_form(int32_t dim, int32_t k, int32_t porth, int64_t nq, int64_t n, int32_t sms) {
  using namespace psi;
  if ((dim != 2 && dim != 3) || k < 1 || k > 128 || sms < 1 || n < 0) return 0;
  if (nq >= lane_min_queries(sms, dim, k, porth != 0, false, n)) return 'L';
  if (k > 32 || (porth && porth_single(dim, k, nq, n))) return 'S';
  return 'G';
}
