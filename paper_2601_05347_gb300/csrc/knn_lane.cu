// knn_lane.cu -- batched k-NN (Sec 2.2) with one query per thread, for small k
// and many queries.
//
// A warp takes 32 queries adjacent in curve order.  The tree search is shared:
// the warp walks one depth-first stack, its lanes test a node's children (one
// each) against the box around its queries, and each child that passes is
// tested by every query for itself.  Each (leaf, query) pair found goes into
// the warp's pool; when the pool is full, and at the end, the pairs are
// scanned 32 at a time, a lane per pair whichever query it belongs to.  So the
// box tests of the tree cost a warp once for 32 queries, a point costs one
// lane's instructions instead of a whole warp's, and the lanes stay busy
// however unevenly the leaves fall to the queries; queries far apart (few
// queries over many points) only make the shared walk longer.
//
// A query first bounds its k-th distance from its seed leaves, the ones at its
// place on the curve: the k smallest of the 32-bit images (rounded up) of their
// points' squared distances, two min/max per entry to take one in.  It then
// only notes the slots of the points within that bound; the seeds are good
// enough that few more than k are noted, and the bound is taken again from the
// notes only when they run out of room or the queue has filled.  At the end
// the notes are put in exact (distance, id) order by a sorting network.
//
// What bounds it: instruction issue and the latency of the scattered loads
// (ncu, 1e6 10-NN on 1e7 2D Varden points: 456 warp instructions per query
// against 1190 for two queries per warp, issue slots 55 % busy, 26 of 64 warps
// resident, L1 hits 65 %, DRAM 7 %).  Blocks of 128 threads at 64 to 80
// registers: at 72 to 96 registers there were no spills, but fewer warps, and
// 3D SPaC-H 10-NN took 7 to 8 % longer.  The pool is shared by the warp because queries that
// scan their own queues of leaves leave lanes idle when the lengths differ.
// 1e7 10-NN on 1e8 2D Varden points, whole call: 18.9 -> 8.2 ms.
//
// Exactness is k_knn's: exact int64 distances, ties by id, a child or leaf
// skipped only when a lower bound of its distance exceeds the k-th distance.
#include "klist.cuh"
#include "knn.cuh"

namespace psi {
namespace {

constexpr int LT = 128;      // threads per block
constexpr int LW = LT / 32;
constexpr int kPool = 128;   // (leaf, query) pairs a warp may have waiting
constexpr int kSeedPoints = 24;  // points a P-Orth query's seeds should hold
constexpr int kSeedMax = 12;     // seed leaves at most (the widened ones)
constexpr float kLoose = 8.0f;   // k-th squared distance over the seed leaves' squared diagonal
template <int D>
constexpr int kLong = D == 2 ? 32 : 64;  // leaves queued by one query
constexpr int kLaneStack = 96;   // nodes waiting; a warp that needs more leaves its queries to the other kernel
// A waiting pair: the leaf's first slot, and in one word the leaf's box key
// (its low bits cleared), the query's lane and the leaf's count.
constexpr uint32_t kCntMask = 255u, kPairMask = (1u << 13) - 1u;
__device__ __forceinline__ uint32_t pair_word(uint32_t key, int lane, int cnt) {
  return (key & ~kPairMask) | (uint32_t)lane << 8 | (uint32_t)cnt;
}
// Points a query may have noted (few, for the sake of the L1 cache beside);
// when fewer than kSpare places are left after 32 pairs, its bound is taken
// again and the notes beyond it dropped.
constexpr int kSpare = 10;
template <int K>
constexpr int kNotesOf = K + 22;
// Slots of the final sorting network; further notes are inserted one by one.
template <int K>
constexpr int kNetOf = K == 1 ? 4 : K <= 5 ? 8 : 16;

template <int D>
__device__ __forceinline__ uint32_t lane_box_key(const TreeView &t, uint32_t node, const int32_t *qc) {
  int32_t lo[D], hi[D];
#pragma unroll
  for (int d = 0; d < D; ++d) {
    lo[d] = t.lo[d][node];
    hi[d] = t.hi[d][node];
  }
  return box_key_of<D>(lo, hi, qc);
}

// f(slot, d2, inside) for the points of each lane's slots [s0, s0 + cnt)
// (cnt 0: none), their squared distances from q; four per step in one 16-byte
// load per coordinate from the aligned slots around them (the pool is a
// multiple of four slots long).  Slots around the range: inside = false.
template <int D, class Point>
__device__ __forceinline__ void walk_slots(const TreeView &t, const int32_t (&q)[D], uint32_t s0, int cnt, Point f) {
  const uint32_t end = s0 + (uint32_t)cnt;
  for (uint32_t b = s0 & ~3u; b < end; b += 4) {
    int4 v[D];
#pragma unroll
    for (int d = 0; d < D; ++d) v[d] = *reinterpret_cast<const int4 *>(t.px[d] + b);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      int64_t d2 = 0;
#pragma unroll
      for (int d = 0; d < D; ++d) {
        const int32_t c = u == 0 ? v[d].x : u == 1 ? v[d].y : u == 2 ? v[d].z : v[d].w;
        const int32_t dd = c - q[d];  // exact: both in [0, 2^31)
        d2 += (int64_t)dd * dd;
      }
      const uint32_t slot = b + u;
      f(slot, d2, slot >= s0 && slot < end);
    }
  }
}

// The search state of one query.  F: the K smallest images of the squared
// distances taken in so far, ascending (a shorter list starts with K - k
// zeros); image(d2) = ceil(d2 / 2^sh), 2^32 - 1 where that does not fit.  A
// point farther than kb = F[K - 1] << sh cannot be among the k nearest.
// note: the slots of the points found within the bound of their time; the
// first nd are in F.
template <int D, int K>
struct LaneSearch {
  const TreeView &t;
  int32_t qc[D];
  uint32_t F[K];
  int64_t kb;
  int sh;
  uint32_t *note;  // LT apart
  int nn, nd;
  static constexpr int kNotes = kNotesOf<K>, kRoom = kNotes - kSpare;
  bool full;  // more points within the bound than notes

  // Images at a scale where the squared extent `ext` takes 30 bits.
  __device__ __forceinline__ void init(int k, float ext) {
    nn = nd = 0;
    full = false;
    kb = INT64_MAX;
    sh = min(max((int)(__float_as_uint(ext) >> 23) - 127 - 30, 0), 31);
#pragma unroll
    for (int j = 0; j < K; ++j) F[j] = j < K - k ? 0u : 0xFFFFFFFFu;
  }

  __device__ __forceinline__ uint32_t image(int64_t d2) const {
    const uint32_t hi = (uint32_t)((uint64_t)d2 >> 32), lo = (uint32_t)d2;
    const uint32_t v = __funnelshift_r(lo, hi, sh);
    return (hi >> sh) || v == 0xFFFFFFFFu ? 0xFFFFFFFFu : v + (sh ? 1u : 0u);
  }

  __device__ __forceinline__ void take(uint32_t f) {
#pragma unroll
    for (int x = K - 1; x > 0; --x) F[x] = max(F[x - 1], min(F[x], f));
    F[0] = min(F[0], f);
  }

  __device__ __forceinline__ void set_bound() {
    kb = F[K - 1] == 0xFFFFFFFFu ? INT64_MAX : (int64_t)((uint64_t)F[K - 1] << sh);
  }

  __device__ __forceinline__ int64_t dist(uint32_t slot) const {
    int64_t d2 = 0;
#pragma unroll
    for (int d = 0; d < D; ++d) {
      const int32_t dd = t.px[d][slot] - qc[d];  // exact: both in [0, 2^31)
      d2 += (int64_t)dd * dd;
    }
    return d2;
  }

  // Every lane's new notes into its F.
  __device__ __forceinline__ void digest() {
    const int most = __reduce_max_sync(0xFFFFFFFFu, nn - nd);
    for (int j = 0; j < most; j += 2) {  // two per round: their loads are in flight together
      uint32_t f[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        f[u] = 0xFFFFFFFFu;
        if (nd + j + u < nn) f[u] = image(dist(note[(nd + j + u) * LT]));
      }
      take(f[0]);
      take(f[1]);
    }
    nd = nn;
    set_bound();
  }

  // Drops the notes beyond the bound.
  __device__ __forceinline__ void compact() {
    const int most = __reduce_max_sync(0xFFFFFFFFu, nn);
    int o = 0;
    for (int j = 0; j < most; ++j)
      if (j < nn) {
        const uint32_t slot = note[j * LT];
        if (dist(slot) <= kb) note[LT * o++] = slot;
      }
    nn = nd = o;
    if (o > kRoom) {  // piles of equal distances: left to the warp-per-query kernel
      full = true;
      nn = nd = 0;
      kb = -1;
    }
  }

  // The points of this lane's slots [s0, s0 + cnt) into F.
  __device__ __forceinline__ void bound_by(uint32_t s0, int cnt) {
    walk_slots<D>(t, qc, s0, cnt, [&](uint32_t, int64_t d2, bool in) { take(in ? image(d2) : 0xFFFFFFFFu); });
  }
};

// Squared diagonal of a node's box, rounded down.
template <int D>
__device__ __forceinline__ float box_diag2(const TreeView &t, uint32_t node) {
  float s = 0.0f;
#pragma unroll
  for (int d = 0; d < D; ++d) {
    const float g = __int2float_rd(t.hi[d][node] - t.lo[d][node]);
    s += g * g;
  }
  return s;
}

template <int D, int K, bool PORTH>
__global__ __launch_bounds__(LT, K <= 10 ? (D == 2 ? 8 : 7) : 6) void k_knn_lane(LaneArgs la) {
  __shared__ uint2 s_stk[LW][kLaneStack];  // nodes to expand: (first child, children)
  __shared__ uint2 s_pool[LW][kPool];      // pairs waiting
  __shared__ uint32_t s_note[kNotesOf<K>][LT];
  __shared__ int s_nn[LT];  // notes of each query, counted here while pairs are scanned
  const KnnArgs &a = la.a;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const TreeView &t = a.t;
  const KnnSeed &sd = a.seed;
  const int64_t qi = (int64_t)blockIdx.x * LT + tid;
  const bool valid = qi < a.nq;
  const int64_t qs = valid ? qi : a.nq - 1;
  const uint32_t q = a.order[qs];
  LaneSearch<D, K> S{t};
  S.note = &s_note[0][tid];
#pragma unroll
  for (int d = 0; d < D; ++d) S.qc[d] = a.q[(int64_t)q * D + d];
  const int32_t root = valid ? (a.qroot ? a.qroot[q] : t.root) : -1;

  // Seed leaves [lo, hi]: SPaC, node numbers; P-Orth, positions in the
  // key-ordered leaf list.
  int lb = 0, le = 0, lo = 0, hi = -1, j = 0;  // node numbers fit 31 bits
  if (root >= 0) {
    le = (int)sd.L;
    if (sd.qseg) {
      const int sg = sd.qseg[q];
      lb = (int)sd.node_off[sg];
      le = lb + (int)((sd.off[sg + 1] - sd.off[sg] + sd.phi - 1) / sd.phi);
    }
    if (le > lb) lo = hi = j = (int)sd.pos[qi];
  }
  // The leaf at the query's place on the curve, widened on both sides until
  // the seeds hold enough points (at most kSeedMax leaves), bounds the k-th
  // distance.  diag: squared diagonal of a seed leaf's box, the widest one's
  // (P-Orth), the narrowest one's of the leaf and its neighbours (SPaC).
  float diag = 0.0f;
  uint32_t wlo = 1u, whi = 0u;  // P-Orth: the seeds' slots [wlo, whi)
  bool hard = false;
  // lower bounds of the squared distances to the seeds and (SPaC) to the leaves beside them
  uint32_t skey = 0x7F800000u, nkey[2] = {0x7F800000u, 0x7F800000u};
  if (hi >= lo) {
    const uint32_t nd = PORTH ? (uint32_t)sd.leaf_node[j] : (uint32_t)j;
    diag = box_diag2<D>(t, nd);
    skey = lane_box_key<D>(t, nd, S.qc);
  }
  S.init(a.k, diag);
  {
    const int want = PORTH ? (K == 1 ? 4 : max(a.k, kSeedPoints)) : a.k;
    if (hi >= lo) {
      const uint32_t nd = PORTH ? (uint32_t)sd.leaf_node[j] : (uint32_t)j;
      int got = t.cnt[nd];
      if (PORTH) {
        wlo = t.ref[nd];
        whi = wlo + (uint32_t)got;
      }
      bool up = hi + 1 < le, down = lo > lb;  // sides that can still be taken
      while (got < want && hi - lo + 1 < kSeedMax && (up || down)) {
        const bool right = up && (!down || hi - j <= j - lo);
        const int nx = right ? hi + 1 : lo - 1;
        const uint32_t e = PORTH ? (uint32_t)sd.leaf_node[nx] : (uint32_t)nx;
        const int c = t.cnt[e];
        if (PORTH) {  // only leaves whose slots adjoin the others'
          const uint32_t r = t.ref[e];
          if (right ? r != whi : r + (uint32_t)c != wlo) {
            (right ? up : down) = false;
            continue;
          }
          if (right)
            whi += (uint32_t)c;
          else
            wlo = r;
          diag = fmaxf(diag, box_diag2<D>(t, e));
        }
        skey = min(skey, lane_box_key<D>(t, e, S.qc));
        (right ? hi : lo) = nx;
        got += c;
        up = hi + 1 < le && (up || !right);
        down = lo > lb && (down || right);
      }
      if (PORTH) {
        // a pile of duplicate points, which one lane alone would walk, or seeds
        // whose boxes already show that they are far from the query
        hard = whi - wlo > kCntMask || __uint_as_float(skey) > kLoose * diag;
        if (!hard) S.bound_by(wlo, (int)(whi - wlo));
      } else {
        for (int side = 0; side < 2; ++side) {
          const int nb = side ? hi + 1 : lo - 1;
          if (nb < lb || nb >= le) continue;
          diag = fminf(diag, box_diag2<D>(t, (uint32_t)nb));
          nkey[side] = lane_box_key<D>(t, (uint32_t)nb, S.qc);
        }
        const float far = kLoose * diag;
        hard = __uint_as_float(min(skey, min(nkey[0], nkey[1]))) > far;
        if (!hard)
          for (int x = lo; x <= hi; ++x) S.bound_by(t.ref[x], t.cnt[x]);
      }
    }
    __syncwarp();
    S.set_bound();
  }
  uint32_t kdk = order_key(S.kb);
  const int seen_end = hi;
  int np = 0;     // pairs waiting (warp-uniform)
  int total = 0;  // leaves this query has put in the pool in its search

  // The leaves just before and after the seeds, where they may hold a
  // neighbour (SPaC): a seed leaf that spans a jump of the curve (or a gap
  // between clusters) gives the queries beside it a bound as wide as the jump,
  // and the leaf on their side of it the true one.
  int seen = lo;  // next of the seed leaves, which are in F but not noted
  if (!PORTH) {
    // a query away from the data: neither the seeds nor the leaves beside them
    // are near it on their own scale
    const float far = kLoose * diag;
    hard |= hi >= lo && __uint_as_float(kdk) > far && __uint_as_float(min(nkey[0], nkey[1])) > far;
    for (int side = 0; side < 2; ++side) {
      const bool need = !hard && hi >= lo && nkey[side] < 0x7F800000u && nkey[side] <= kdk;
      const uint32_t nm = __ballot_sync(0xFFFFFFFFu, need);
      if (need) {
        const int nb = side ? hi + 1 : lo - 1;
        s_pool[w][np + __popc(nm & lanemask_lt())] = make_uint2(t.ref[nb], pair_word(nkey[side], lane, t.cnt[nb]));
        (side ? hi : lo) = nb;
      }
      np += __popc(nm);
    }
  }
  if (hard) seen = seen_end + 1;
  // SPaC: the seeds as node numbers [slo, shi]
  const uint32_t slo = hi >= lo ? (uint32_t)lo : 1u, shi = hi >= lo ? (uint32_t)hi : 0u;

  // The search, in rounds: pairs are put in the pool until it is full or there
  // are no more, then scanned.  Stage 0 takes the seeds' neighbours (above),
  // stage 1 the seeds themselves, to note their points under the bound of all
  // of them; stage 2 walks the tree, once per distinct root among the warp's
  // queries (one index: once).
  int stage = PORTH ? 1 : 0;
  uint32_t pending = 0, m = 0, lm = 0, gk = 0, c0 = 0;
  int sp = 0, nk = 0;
  bool act = false, leafc = false;
  int32_t lo_[D], hi_[D], glo[D], ghi[D];
  uint32_t cref = 0;
  int ccnt = 0;
  for (;;) {
    bool more = true;
    if (stage == 1) {
      const bool need = seen <= seen_end;
      uint32_t s0 = 0;
      int c = 0;
      if (need) {
        s0 = PORTH ? wlo : t.ref[seen];
        c = PORTH ? (int)(whi - wlo) : t.cnt[seen];
        seen = PORTH ? seen_end + 1 : seen + 1;
      }
      const uint32_t nm = __ballot_sync(0xFFFFFFFFu, need);
      if (need) s_pool[w][__popc(nm & lanemask_lt())] = make_uint2(s0, pair_word(0, lane, c));
      np = __popc(nm);
    } else if (stage == 2) {
      for (;;) {
        if (!m) {
          if (sp == 0) {  // the next root, as the only child of a virtual node
            if (!pending) {
              more = false;
              break;
            }
            const int32_t rt = __shfl_sync(0xFFFFFFFFu, root, __ffs(pending) - 1);
            act = root == rt && !hard;
            pending &= ~__ballot_sync(0xFFFFFFFFu, root == rt);
#pragma unroll
            for (int d = 0; d < D; ++d) {  // box around the active queries
              glo[d] = __reduce_min_sync(0xFFFFFFFFu, act ? S.qc[d] : INT32_MAX);
              ghi[d] = __reduce_max_sync(0xFFFFFFFFu, act ? S.qc[d] : INT32_MIN);
            }
            gk = __reduce_max_sync(0xFFFFFFFFu, act ? kdk : 0u);
            c0 = (uint32_t)rt;
            nk = lane == 0 ? 1 : 0;
          } else {  // SPaC: one node of up to 32 children; P-Orth: as many nodes as fit
            constexpr int W = PORTH ? 1 << D : 32;
            const int g = lane / W;
            __syncwarp();
            const uint2 e = g < sp ? s_stk[w][sp - 1 - g] : make_uint2(0u, 0u);
            __syncwarp();
            sp = max(sp - 32 / W, 0);
            c0 = e.x;
            nk = (int)e.y - lane % W;  // > 0: this lane's child exists
            if (PORTH) c0 -= (uint32_t)(g * W);
          }
          // expand: a lane per child, against the box around the queries
          const uint32_t c = c0 + (uint32_t)lane;
          bool near = false;
          leafc = false;
          if (nk > 0) {
            cref = t.ref[c];
            if (a.leaf_limit >= 0) {
              leafc = (int64_t)c < a.leaf_limit;
              ccnt = leafc ? t.cnt[c] : t.kids[c];
            } else {
              const int ck = t.kids[c], cn = t.cnt[c];
              leafc = ck == 0;
              ccnt = leafc ? cn : ck;
            }
            float f = 0.0f;
#pragma unroll
            for (int d = 0; d < D; ++d) {
              lo_[d] = t.lo[d][c];
              hi_[d] = t.hi[d][c];
              const int32_t g = max(0, max(lo_[d] - ghi[d], glo[d] - hi_[d]));  // all in [0, 2^31)
              const float gf = __int2float_rd(g);
              f = __fadd_rd(f, __fmul_rd(gf, gf));
            }
            near = __float_as_uint(f) <= gk;
          }
          m = __ballot_sync(0xFFFFFFFFu, near);
          lm = __ballot_sync(0xFFFFFFFFu, leafc);
          continue;
        }
        // test: one child that passed, by every query
        const int src = __ffs(m) - 1;
        m &= m - 1;
        int32_t blo[D], bhi[D];
#pragma unroll
        for (int d = 0; d < D; ++d) {
          blo[d] = __shfl_sync(0xFFFFFFFFu, lo_[d], src);
          bhi[d] = __shfl_sync(0xFFFFFFFFu, hi_[d], src);
        }
        const uint32_t key = box_key_of<D>(blo, bhi, S.qc);
        const uint32_t bref = __shfl_sync(0xFFFFFFFFu, cref, src);
        const bool leaf = (lm >> src) & 1u;  // warp-uniform
        bool need = act && key <= kdk;
        if (leaf) {
          if (PORTH)
            need &= !(bref >= wlo && bref < whi);
          else
            need &= !(c0 + (uint32_t)src >= slo && c0 + (uint32_t)src <= shi);
        }
        if (!__any_sync(0xFFFFFFFFu, need)) continue;
        const int bcnt = __shfl_sync(0xFFFFFFFFu, ccnt, src);
        if (leaf && !(PORTH && bcnt > (int)kCntMask)) {
          const uint32_t nm = __ballot_sync(0xFFFFFFFFu, need);
          if (need) {
            s_pool[w][np + __popc(nm & lanemask_lt())] = make_uint2(bref, pair_word(key, lane, bcnt));
            ++total;
          }
          np += __popc(nm);
          if (np > kPool - 32) break;
        } else if (!leaf && sp < kLaneStack) {
          if (lane == 0) s_stk[w][sp] = make_uint2(bref, (uint32_t)bcnt);
          ++sp;
        } else {  // a pile of duplicate points, or too many nodes waiting
          hard |= need;
          act &= !need;
        }
      }
    }
    // the pool, a lane per pair
    s_nn[tid] = S.nn;
    __syncwarp();
    for (int x0 = 0; x0 < np; x0 += 32) {
      const uint2 e = x0 + lane < np ? s_pool[w][x0 + lane] : make_uint2(0u, (uint32_t)lane << 8);
      const int o = (int)(e.y >> 8) & 31;  // the pair's query
      int32_t oq[D];
#pragma unroll
      for (int d = 0; d < D; ++d) oq[d] = __shfl_sync(0xFFFFFFFFu, S.qc[d], o);
      const int64_t okb = __shfl_sync(0xFFFFFFFFu, S.kb, o);
      const uint32_t ok = __shfl_sync(0xFFFFFFFFu, kdk, o);
      const int c = (e.y & ~kPairMask) <= ok ? (int)(e.y & kCntMask) : 0;
      int *on = &s_nn[w * 32 + o];
      uint32_t *onote = &s_note[0][w * 32 + o];
      walk_slots<D>(t, oq, e.x, c, [&](uint32_t slot, int64_t d2, bool in) {
        if (in && d2 <= okb) {
          const int p = atomicAdd(on, 1);
          if (p < kNotesOf<K>) onote[LT * p] = slot;
        }
      });
      __syncwarp();
      S.nn = s_nn[tid];
      if (S.nn > kNotesOf<K>) {  // some were not noted
        S.full = true;
        S.nn = S.nd = 0;
        S.kb = -1;
      }
      if (__any_sync(0xFFFFFFFFu, S.nn > LaneSearch<D, K>::kRoom)) {
        if (stage != 1) S.digest();
        else S.nd = S.nn;
        S.compact();
      }
      s_nn[tid] = S.nn;
      __syncwarp();
    }
    np = 0;
    if (stage == 1) {
      S.nd = S.nn;
      if (!__any_sync(0xFFFFFFFFu, seen <= seen_end)) {
        // A k-th distance far above the seeds' own extent (a query away from
        // the data, too few points in the seeds): left to the other kernel.
        hard |= S.full || !(__uint_as_float(kdk) <= kLoose * diag);
        hard &= root >= 0;
        pending = __ballot_sync(0xFFFFFFFFu, root >= 0 && !hard);
        stage = 2;
      }
      continue;
    }
    if (!more) break;
    S.digest();
    kdk = order_key(S.kb);
    if (stage == 0) {
      stage = 1;
      continue;
    }
    if (S.full || total > kLong<D>) {  // a long search: left to the other kernel
      hard |= act;
      act = false;
    }
    gk = __reduce_max_sync(0xFFFFFFFFu, act ? kdk : 0u);
  }

  // the notes in exact order
  constexpr int N = kNetOf<K>;
  int64_t od[N];
  uint32_t oi[N];
#pragma unroll
  for (int x = 0; x < N; ++x) {
    od[x] = INT64_MAX;
    oi[x] = 0xFFFFFFFFu;
    if (x < S.nn) {
      const uint32_t slot = S.note[x * LT];
      od[x] = S.dist(slot);
      oi[x] = t.pid[slot];
    }
  }
  pair_network(od, oi);
  const int most = __reduce_max_sync(0xFFFFFFFFu, S.nn);
  for (int x = N; x < most; ++x) {
    int64_t d2 = INT64_MAX;
    uint32_t id = 0xFFFFFFFFu;
    if (x < S.nn) {
      const uint32_t slot = S.note[x * LT];
      d2 = S.dist(slot);
      id = t.pid[slot];
    }
    if (__any_sync(0xFFFFFFFFu, pair_less(d2, id, od[K - 1], oi[K - 1]))) pair_insert<K>(od, oi, d2, id);
  }
  hard |= S.full;
  const uint32_t hm = __ballot_sync(0xFFFFFFFFu, hard);
  uint32_t hbase = 0;
  if (hm && lane == 0) hbase = atomicAdd(la.hn, (uint32_t)__popc(hm));
  hbase = __shfl_sync(0xFFFFFFFFu, hbase, 0);
  if (hard) {
    const uint32_t x = hbase + __popc(hm & lanemask_lt());
    la.hq[x] = q;
    la.hpos[x] = sd.pos[qi];
  } else if (valid) {
#pragma unroll
    for (int x = 0; x < K; ++x)
      if (x < a.k) {
        a.out_id[(int64_t)q * a.k + x] = oi[x];
        a.out_d2[(int64_t)q * a.k + x] = od[x];
      }
  }
}

}  // namespace

psi_status run_knn_lane(const LaneArgs &a, int D, bool porth, cudaStream_t s) {
  const int k = a.a.k;
  const unsigned grid = (unsigned)ceil_div(a.a.nq, LT);
#define LANE(DD, KK)                                                                     \
  do {                                                                                   \
    if (porth)                                                                           \
      PSI_LAUNCH_NAMED("k_knn", (k_knn_lane<DD, KK, true>), grid, LT, 0, s, a);          \
    else                                                                                 \
      PSI_LAUNCH_NAMED("k_knn", (k_knn_lane<DD, KK, false>), grid, LT, 0, s, a);         \
  } while (0)
#define LANE_K(DD)               \
  do {                           \
    if (k == 1) LANE(DD, 1);   \
    else if (k <= 5) LANE(DD, 5);   \
    else if (k <= 10) LANE(DD, 10); \
    else LANE(DD, kLaneMaxK);    \
  } while (0)
  if (D == 2) LANE_K(2);
  else LANE_K(3);
#undef LANE_K
#undef LANE
  PSI_CK(cudaGetLastError());
  return PSI_OK;
}

}  // namespace psi
