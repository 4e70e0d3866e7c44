// knn.cuh -- what the k-NN kernels share: their arguments and the pruning keys.
#pragma once
#include "index.cuh"

namespace psi {

// Pruning key of a child box: the float bits of a lower bound of its squared
// distance to the query, computed on the FP32 pipe (the ALU pipe is the
// k-NN kernel's bottleneck): each gap is an exact int32 difference converted,
// squared and summed with rounding toward -inf, so the bound never exceeds the
// exact distance; a float at or below the exact k-th distance is at or below
// that distance rounded to nearest, so comparing float bits never prunes a box
// that holds a neighbour.
template <int D>
__device__ __forceinline__ uint32_t box_key_of(const int32_t *lo, const int32_t *hi, const int32_t *qc) {
  float s = 0.0f;
#pragma unroll
  for (int d = 0; d < D; ++d) {
    const int32_t q = qc[d];
    const int32_t g = q < lo[d] ? lo[d] - q : (q > hi[d] ? q - hi[d] : 0);
    const float gf = __int2float_rd(g);
    s = __fadd_rd(s, __fmul_rd(gf, gf));
  }
  return __float_as_uint(s);
}

// 32-bit image of a non-negative distance for pruning: the float bits of the
// distance rounded up, built from its two 32-bit halves (a conversion from a
// 64-bit integer would run on the FP64 unit, which is very slow on this GPU).
// A child key is its box distance rounded down, so a child whose key exceeds
// the image of the k-th distance is farther than that distance: pruning by
// keys never skips a node that could hold a neighbour; it may keep a few that
// cannot, which costs time, not exactness.
__device__ __forceinline__ uint32_t order_key(int64_t md) {
  const uint32_t hi = (uint32_t)((uint64_t)md >> 32), lo = (uint32_t)md;
  return __float_as_uint(__fmaf_ru(__uint2float_ru(hi), 4294967296.0f, __uint2float_ru(lo)));
}

// order_key of the k-th distance of a list that is not full yet.
constexpr uint32_t kNoBound = 0x5F000000u;

struct KnnArgs {
  TreeView t;
  const int32_t *q;
  int64_t nq;
  int k;
  const uint32_t *order;
  const int32_t *qroot;  // per-query root (many indexes in one node array), or null
  KnnSeed seed;        // SPaC: leaves scanned before the search
  int64_t leaf_limit;  // >= 0: the leaves are exactly the nodes [0, leaf_limit) (one SPaC index)
  uint32_t *out_id;
  int64_t *out_d2;
  int *status;
  // listed queries: their number (at most nq), and the order and seed positions
  // of all nq queries
  const uint32_t *d_nq = nullptr;
  const uint32_t *all_order = nullptr, *all_pos = nullptr;
  int64_t list_lo = 0, list_hi = INT64_MAX;  // a list of any other length is left to another kernel
};

// The queries a kernel over a list takes: the list; or, where it holds three
// quarters of them, all (the others' results are written again, the same).  The
// list is in the order in which warps came to append to it, while neighbours of
// the curve order read the same nodes: 2e6 8-NN of uniform queries on 3e6 Varden
// points (2D P-Orth), listed 12.2 ms, in curve order 9.1.
// (Without a list everything is read from the arguments, which cost no registers.)
template <bool LIST>
struct KnnTake {
  const KnnArgs &a;
  const uint32_t *order = nullptr, *seeds = nullptr;
  int64_t number = 0;
  __device__ __forceinline__ explicit KnnTake(const KnnArgs &args) : a(args) {
    if (!LIST) return;
    const int64_t n = (int64_t)*a.d_nq;
    const bool all = 4 * n >= 3 * a.nq;
    order = all ? a.all_order : a.order;
    seeds = all ? a.all_pos : a.seed.pos;
    number = n < a.list_lo || n >= a.list_hi ? 0 : all ? a.nq : n;
  }
  __device__ __forceinline__ int64_t nq() const { return LIST ? number : a.nq; }
  __device__ __forceinline__ int64_t query(int64_t i) const {
    return LIST ? (int64_t)order[i] : a.order ? (int64_t)a.order[i] : i;
  }
  __device__ __forceinline__ uint32_t pos(int64_t i) const { return LIST ? seeds[i] : a.seed.pos[i]; }
};

// Per-warp depth-first stack of the k-NN search: an expanded node pushes at
// most F - 1 more entries than it pops, so depth x 31 + 32 entries suffice
// (SPaC: 7 levels at 1e9 points; P-Orth: at most 2^D children per level).
constexpr int KSTACK = 256;

// k-NN with one query per thread (knn_lane.cu), k <= kLaneMaxK, queries in
// curve order with seeds.  Queries whose seed bounds them badly (or whose
// search turns out long) are left out and listed: hq[i] = query, hpos[i] = its
// seed position, *hn of them (zero on entry), for the warp-per-query kernels.
constexpr int kLaneMaxK = 16;
struct LaneArgs {
  KnnArgs a;
  uint32_t *hq, *hpos, *hn;
};
psi_status run_knn_lane(const LaneArgs &a, int D, bool porth, cudaStream_t s);

}  // namespace psi
