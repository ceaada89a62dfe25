// Batched GreedySearch (Algorithm 2) and k-recall@k (§4).
//
// Queries are taken from an atomic counter.  Two kernels hold the search list
// differently:
//   search_reg_kernel   L <= 256: the list lives in one warp's registers, sorted,
//                       entry i in slot i % S of lane i / S.  Every entry sees
//                       for itself whether it stays, moves up by one or makes
//                       room for the new point, so adding a point takes two
//                       shuffles and a few selects per slot.
//   search_list_kernel  longer lists: in shared memory, sorted by (distance, id);
//                       new points are sorted and merged 32 at a time.  It also takes
//                       the float queries that met so many near-equal distances that
//                       the first kernel gave them up (kFineBudget).
//
// Algorithm 2 keeps a set: adding a point that is already in the list has
// no effect.  A point that was in the list and was cut may be added again by
// a later neighbour list, and then it is cut again at once: from the first cut
// on the list holds L members and its L-th (distance, id) only decreases, so
// the point still lies behind it.  (An expanded point that is cut is the same
// case: it comes back behind the L-th and is never the closest unexpanded
// member.)  So the only membership test the search needs is "is v in the
// list now?".  A small direct-mapped cache of recently met ids in shared memory
// skips most repeated distance computations; a miss only costs one more
// distance, never a different result.
//
// Neighbours are added one at a time or in batches, the list cut to L after
// each; the L closest of a union are the L closest of the L closest of its
// parts, so this equals adding the whole list and cutting once.
//
// Distances (row_keys): 4, 8 or 32 lanes share a row (by its length), lane s of
// G taking its 16-byte chunks s, s + G, ..., so that whole 32-byte sectors are
// read and every load of a step is in flight at once.  Every kernel sums a
// distance the same way, so a query's results do not depend on the kernel.
//
// Ordering: uint8 distances are exact integers.  float32 distances carry a
// rigorous single-precision error bound (lane_rel_bound); when two intervals
// overlap, both distances are recomputed in float-float arithmetic (bound about
// d 2^-46 relative), and only if those intervals still overlap in binary64
// (index order, no fused multiply-add), so every comparison agrees with the
// binary64 reading.
#include <cfloat>
#include <climits>
#include <map>
#include <mutex>
#include <tuple>
#include <type_traits>

#include "internal.h"

namespace rpk {

namespace {

constexpr int kWarps = 4;  // warps (queries in flight) per CTA
constexpr int kTeam = 5;        // warps per query of the team form: the list's warp and four that read rows
constexpr unsigned kVisited = 0x80000000u;
constexpr unsigned kIdMask = 0x7fffffffu;
// A float query's close decisions in search_reg_kernel are made one at a time by the
// whole warp, which is dear where distances tie all the time (rows of zeros and ones,
// rows many times over).  A query that has spent more than kFineBudget on them leaves
// kSearchRedo as its first id and is searched again by search_list_kernel, which keeps
// such distances and settles 32 at a time.  The benchmark's shapes make 0.2 (400,000 x
// 96, L = 100) to 20 a query (30,000 x 960, L = 200; no query above 47).  20,000 x 96
// zeros and ones, L = 100, 5,000 queries: every decision made here 2,963 ms, with the
// budget 55, by the list kernel alone 55.
// One that binary64 has to settle takes two sums in index order, by a lane each, and
// costs kFineF64.  30,000 x 960 rows give one to a query in 2,200; were that query
// given up, its call of 1,000 would take 9 to 18 ms where it takes 4.7.
constexpr int kFineBudget = 128;
constexpr int kFineF64 = 32;

struct SearchArgs {
  const uint8_t* X;
  int64_t row_bytes;
  int d;
  int64_t n;
  const int64_t* row_ptr;
  const int32_t* col;
  int64_t start;
  const SearchGraph* graphs;  // per-query graphs (with q_graph), or nullptr
  const int32_t* q_graph;     // index into graphs per query, or nullptr
  const int32_t* q_L;         // list size per query (k <= q_L <= L), or nullptr
  const uint8_t* Q;
  int64_t nq;
  int L;                      // largest list size; sizes the shared memory
  int k;
  int32_t* out_ids;
  float* out_dists;
  int cache_bits;             // log2 of the id-cache entries per warp
  unsigned int* work;
  DevStatus* status;
  // graph construction (Vamana): query i is base point q_point[i]; the graph
  // is held as adj_deg[v] ids at col + v * adj_stride; the expanded points of
  // query i go to visited[i * visited_cap ..] (the first visited_cap of them),
  // their number to visited_cnt[i]
  const int32_t* q_point;
  const int32_t* adj_deg;
  int64_t adj_stride;
  int32_t* visited;
  int32_t* visited_cnt;
  int visited_cap;
  int fine_budget;            // search_reg_kernel: most that a query may spend on close decisions
};

struct WarpSmem {
  unsigned* key;   // the list: distance bits, sorted by (distance, id)
  unsigned* idv;   // its ids (| kVisited once expanded)
  double* d64;     // float data: binary64 distances of the list (NaN until computed)
  unsigned* ckey;  // a batch's new members, then
  unsigned* cid;
  int* clo;        // their insertion points (sorted: the merge's shift table)
  double* cd64;
  uint8_t* q;
  unsigned* cache;  // direct-mapped ids met by this query (0xffffffff = empty)
};

__host__ __device__ inline size_t list_cap(int L) { return (size_t(L) + 3) & ~size_t(3); }

__host__ __device__ inline size_t warp_bytes(int L, int64_t row_bytes, bool f32, int cache_bits) {
  const size_t cap = list_cap(L);
  size_t b = cap * 8 + 32 * 12;  // list keys + ids; batch keys, ids, insertion points
  if (f32) b += cap * 8 + 32 * 8;
  b += size_t(row_bytes);
  b += size_t(4) << cache_bits;
  return (b + 127) & ~size_t(127);
}

__device__ inline WarpSmem carve(unsigned char* base, int L, int64_t row_bytes, bool f32, int cache_bits) {
  WarpSmem w;
  const size_t cap = list_cap(L);
  unsigned char* p = base;
  w.cache = reinterpret_cast<unsigned*>(p);
  p += size_t(4) << cache_bits;
  if (f32) {
    w.d64 = reinterpret_cast<double*>(p);
    p += cap * 8;
    w.cd64 = reinterpret_cast<double*>(p);
    p += 32 * 8;
  } else {
    w.d64 = w.cd64 = nullptr;
  }
  w.q = p;  // 16-byte aligned: cap is a multiple of 4 and row_bytes of 16
  p += row_bytes;
  w.key = reinterpret_cast<unsigned*>(p);
  p += cap * 4;
  w.idv = reinterpret_cast<unsigned*>(p);
  p += cap * 4;
  w.ckey = reinterpret_cast<unsigned*>(p);
  p += 32 * 4;
  w.cid = reinterpret_cast<unsigned*>(p);
  p += 32 * 4;
  w.clo = reinterpret_cast<int*>(p);
  return w;
}

// Lanes that share a row of nch 16-byte chunks: 4 for rows of up to 384 bytes (a
// step of eight rows then has at most six loads per lane), 8 up to 1 KB, else
// the whole warp.
__host__ __device__ constexpr int row_lanes(int nch) { return nch <= 24 ? 4 : nch <= 64 ? 8 : 32; }

// Relative bound of a float distance as row_keys sums it: each term carries two
// roundings of its difference, ceil(nch / G) fused adds into one of its lane's
// four sums, two to join those and log2 G to join the lanes; six ulps more
// cover the comparisons built on it.
__device__ __forceinline__ float lane_rel_bound(int nch) {
  const int G = row_lanes(nch);
  return float((nch + G - 1) / G + 2 + (G == 4 ? 2 : G == 8 ? 3 : 5) + 8) * 5.9604645e-08f;
}

// What one lane has summed of a row's distance.  uint8: |x|^2 - 2 <q, x>,
// exact in 32-bit modular arithmetic (d2 = |q|^2 + |x|^2 - 2 <q, x> < 2^32).
// float: four sums of squared differences, one per component of a chunk.
template <int DT>
struct LaneSum;
template <>
struct LaneSum<kU8> {
  unsigned dot = 0, xx = 0;
  __device__ __forceinline__ void add(uint4 q, uint4 x) {
    dot = __dp4a(q.x, x.x, dot);
    dot = __dp4a(q.y, x.y, dot);
    dot = __dp4a(q.z, x.z, dot);
    dot = __dp4a(q.w, x.w, dot);
    xx = __dp4a(x.x, x.x, xx);
    xx = __dp4a(x.y, x.y, xx);
    xx = __dp4a(x.z, x.z, xx);
    xx = __dp4a(x.w, x.w, xx);
  }
  template <int G>
  __device__ __forceinline__ unsigned finish(unsigned qn) {  // over the G lanes of a row
    unsigned v = xx - 2u * dot;
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return qn + v;
  }
};
template <>
struct LaneSum<kF32> {
  float x = 0.f, y = 0.f, z = 0.f, w = 0.f;
  __device__ __forceinline__ void add(uint4 q, uint4 b) {
    float t;
    t = __uint_as_float(q.x) - __uint_as_float(b.x); x = fmaf(t, t, x);
    t = __uint_as_float(q.y) - __uint_as_float(b.y); y = fmaf(t, t, y);
    t = __uint_as_float(q.z) - __uint_as_float(b.z); z = fmaf(t, t, z);
    t = __uint_as_float(q.w) - __uint_as_float(b.w); w = fmaf(t, t, w);
  }
  template <int G>
  __device__ __forceinline__ unsigned finish(unsigned) {
    float v = (x + y) + (z + w);
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return __float_as_uint(v);
  }
};

// Rows r, r + step, ... (U of them, those below nf) for each group of G lanes,
// in blocks of KC chunks per lane; a block's loads are all issued before the
// first is used.  Rows past nf repeat row nf - 1 and are not stored.  WHOLE:
// nch = G KC, so that no load needs a test.
template <int DT, int G, int KC, int U, bool WHOLE>
__device__ __forceinline__ void row_keys_step(const uint8_t* __restrict__ X, int64_t row_bytes, int nch,
                                              const uint8_t* q, const unsigned* cid, unsigned* ckey, int nf, int r,
                                              int step, unsigned qn) {
  const int sub = threadIdx.x & (G - 1);
  const uint4* px[U];
#pragma unroll
  for (int u = 0; u < U; ++u)
    px[u] = reinterpret_cast<const uint4*>(X + int64_t(cid[min(r + u * step, nf - 1)]) * row_bytes) + sub;
  const uint4* pq = reinterpret_cast<const uint4*>(q) + sub;
  LaneSum<DT> a[U];
  for (int c0 = 0; c0 < nch; c0 += G * KC) {
    uint4 x[U][KC];
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int c = 0; c < KC; ++c)
        x[u][c] = WHOLE || sub + c0 + G * c < nch ? __ldg(px[u] + c0 + G * c) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int c = 0; c < KC; ++c) {
      if (WHOLE || sub + c0 + G * c < nch) {
        const uint4 qv = pq[c0 + G * c];
#pragma unroll
        for (int u = 0; u < U; ++u) a[u].add(qv, x[u][c]);
      }
    }
    if (WHOLE) break;
  }
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const unsigned k = a[u].template finish<G>(qn);
    if (r + u * step < nf) ckey[r + u * step] = k;  // the same value from each of the G lanes
  }
}

// d2(q, cid[r]) as order-preserving bits into ckey[r] for the rows r < nf that
// fall to this warp, number `wi` of `nw` that share them.  All lanes of the
// warp take part; cid, q and ckey are in shared memory.  W: the kernel's warps
// per query (one: registers are short, so fewer loads at a time; 960-float rows,
// 1,000 queries on teams of three: 4 loads per lane in flight 5.48 ms, 8 4.58 ms).
template <int DT, int W>
__device__ __forceinline__ void row_keys(const uint8_t* __restrict__ X, int64_t row_bytes, const uint8_t* q,
                                         const unsigned* cid, unsigned* ckey, int nf, int wi, int nw, unsigned qn) {
  const int lane = threadIdx.x & 31;
  const int nch = int(row_bytes / 16);
#define RP_ROWS(G, KC, U, WHOLE)                                  \
  for (int b = (32 / G) * wi; b < nf; b += (32 / G) * U * nw)     \
    row_keys_step<DT, G, KC, U, WHOLE>(X, row_bytes, nch, q, cid, ckey, nf, b + lane / G, (32 / G) * nw, qn)
  if (nch <= 24) {  // row_lanes(nch) = 4: eight rows a step
    if (nch == 8) RP_ROWS(4, 2, 2, true);
    else if (nch == 24) RP_ROWS(4, 6, 1, true);
    else if (nch == 16) RP_ROWS(4, 4, 1, true);
    else RP_ROWS(4, 3, 1, false);
  } else if (nch <= 64) {
    RP_ROWS(8, 4, 1, false);
  } else {
    RP_ROWS(32, (W == 1 ? 4 : 8), (W == kTeam ? 2 : 1), false);
  }
#undef RP_ROWS
}

// Total order on (distance, id) entries.  For float data `d64a`/`d64b` point to
// the slots caching the binary64 distances (NaN until computed).
template <int DT>
__device__ __forceinline__ bool entry_less(unsigned ka, unsigned ia, double* d64a, unsigned kb, unsigned ib,
                                           double* d64b, const SearchArgs& a, const uint8_t* q, float E,
                                           float Eabs) {
  if constexpr (DT == kU8) {
    return ka < kb || (ka == kb && ia < ib);
  } else {
    if (ia == ib) return false;  // the same point: never less than itself (no binary64 needed)
    const float fa = __uint_as_float(ka), fb = __uint_as_float(kb);
    if (sure_less(fa, fb, E, Eabs)) return true;
    if (sure_less(fb, fa, E, Eabs)) return false;
    const float* qf = reinterpret_cast<const float*>(q);
    const int64_t stride = a.row_bytes / 4;
    const float* X = reinterpret_cast<const float*>(a.X);
    double xa = *d64a, xb = *d64b;
    // float-float first (cached, sign-marked), binary64 only if still undecided
    if (isnan(xa)) *d64a = xa = -ff_d2(qf, X + int64_t(ia) * stride, a.row_bytes);
    if (isnan(xb)) *d64b = xb = -ff_d2(qf, X + int64_t(ib) * stride, a.row_bytes);
    const int o = slot_order(xa, xb, ff_bound(a.d));
    if (o >= 0) return o == 1;
    if (signbit(xa)) {
      xa = canon_d2_f32(qf, X + int64_t(ia) * stride, a.d);
      *d64a = xa;
      atomicAdd(&a.status->fp64_search, 1ull);
    }
    if (signbit(xb)) {
      xb = canon_d2_f32(qf, X + int64_t(ib) * stride, a.d);
      *d64b = xb;
      atomicAdd(&a.status->fp64_search, 1ull);
    }
    return xa < xb || (xa == xb && ia < ib);
  }
}

// The list in shared memory, for L > kRegL.  A batch of 32 neighbours: those
// the id cache does not hold get their distances, those that enter the list
// are sorted by a bitonic network and merged in place.
// REDO: any L, only the queries that hold kSearchRedo (spread over the grid's warps).
// With a lane per row before and its rows shared by lanes now, 300 queries on 20,000
// rows, L = 300 and 1,024: 96 floats 3.78 and 17.2 ms, now 3.21 and 13.5; 960 floats 20.8
// and 126, 15.5 and 75.5; 128 uint8 1.46 and 6.28, 1.49 and 6.27.
template <int DT, bool REDO>
__global__ void __launch_bounds__(kWarps * 32, 8) search_list_kernel(SearchArgs a) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool f32 = DT == kF32;
  WarpSmem S = carve(smem_raw + size_t(w) * warp_bytes(a.L, a.row_bytes, f32, a.cache_bits), a.L, a.row_bytes, f32,
                     a.cache_bits);
  const int cshift = 32 - a.cache_bits;
  const int centries = 1 << a.cache_bits;
  const float E = lane_rel_bound(int(a.row_bytes / 16)), Eabs = abs_bound(a.d);
  const double qnan = __longlong_as_double(0x7ff8000000000000ll);
  // REDO: lane l looks at query rb + l * rstep
  const int64_t rstep = int64_t(gridDim.x) * kWarps;
  int64_t rb = int64_t(w) * gridDim.x + blockIdx.x - 32 * rstep;
  unsigned redo = 0;

  for (;;) {
    unsigned qi = 0;
    if constexpr (REDO) {
      while (!redo) {
        rb += 32 * rstep;
        if (rb >= a.nq) return;
        const int64_t q = rb + lane * rstep;
        redo = __ballot_sync(0xffffffffu, q < a.nq && a.out_ids[q * a.k] == kSearchRedo);
      }
      qi = unsigned(rb + (__ffs(int(redo)) - 1) * rstep);
      redo &= redo - 1;
    } else {
      if (lane == 0) qi = atomicAdd(a.work, 1u);
      qi = __shfl_sync(0xffffffffu, qi, 0);
      if (qi >= a.nq) break;
    }
    const int64_t* __restrict__ row_ptr = a.row_ptr;
    const int32_t* __restrict__ col = a.col;
    int64_t start = a.start;
    if (a.q_graph) {
      const SearchGraph g = a.graphs[a.q_graph[qi]];
      row_ptr = g.row_ptr;
      col = g.col;
      start = g.start;
    }
    const int L = a.q_L ? a.q_L[qi] : a.L;
    // stage the query row
    const uint4* src = reinterpret_cast<const uint4*>(
        a.q_point ? a.X + int64_t(a.q_point[qi]) * a.row_bytes : a.Q + int64_t(qi) * a.row_bytes);
    for (int c = lane; c < a.row_bytes / 16; c += 32) reinterpret_cast<uint4*>(S.q)[c] = src[c];
    for (int c = lane; c < centries; c += 32) S.cache[c] = 0xffffffffu;
    __syncwarp();
    unsigned qn = 0;  // uint8: |q|^2
    if constexpr (DT == kU8) {
      for (int w4 = lane; w4 < a.row_bytes / 4; w4 += 32) {
        const unsigned qw = reinterpret_cast<const unsigned*>(S.q)[w4];
        qn = __dp4a(qw, qw, qn);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) qn += __shfl_xor_sync(0xffffffffu, qn, o);
    }

    unsigned* const keyc = S.key;
    unsigned* const idc = S.idv;
    double* const dc = S.d64;
    int size = 1;
    int f = 0;  // the members before index f are all expanded
    if (lane == 0) {
      const unsigned s = unsigned(start);
      S.cid[0] = s;
      idc[0] = s;
      if (f32) dc[0] = qnan;
      S.cache[(s * 0x9E3779B1u) >> cshift] = s;
    }
    __syncwarp();
    row_keys<DT, 1>(a.X, a.row_bytes, S.q, S.cid, keyc, 1, 0, 1, qn);
    __syncwarp();

    int64_t iters = 0;
    for (;;) {
      // the closest member not yet expanded
      int pos = -1;
      for (int c0 = f & ~31; c0 < size; c0 += 32) {
        const int i = c0 + lane;
        const bool open = i < size && !(idc[i] & kVisited);
        const unsigned b = __ballot_sync(0xffffffffu, open);
        if (b) {
          pos = c0 + __ffs(b) - 1;
          break;
        }
      }
      if (pos < 0) break;
      if (++iters > a.n + 1) {  // cannot happen: each point is expanded at most once
        if (lane == 0) raise_status(a.status, kDevOverflow, qi);
        break;
      }
      const unsigned ps = idc[pos] & kIdMask;
      __syncwarp();
      if (lane == 0) idc[pos] |= kVisited;
      __syncwarp();
      f = pos + 1;
      if (a.visited && lane == 0 && iters <= a.visited_cap) a.visited[int64_t(qi) * a.visited_cap + iters - 1] = int32_t(ps);
      int64_t e0, e1;
      if (a.adj_deg) {
        e0 = int64_t(ps) * a.adj_stride;
        e1 = e0 + a.adj_deg[ps];
      } else {
        e0 = row_ptr[ps];
        e1 = row_ptr[ps + 1];
      }
      for (int64_t eb = e0; eb < e1; eb += 32) {
        // ---- new neighbours of this batch
        const int64_t e = eb + lane;
        bool fresh = false;
        unsigned v = 0;
        if (e < e1) {
          v = unsigned(col[e]);
          // a row holds distinct ids, so lanes that share a cache entry hold
          // different ids: whichever write lands, no lane skips a new id
          const unsigned h = (v * 0x9E3779B1u) >> cshift;
          fresh = S.cache[h] != v;
          if (fresh) S.cache[h] = v;
        }
        const unsigned frm = __ballot_sync(0xffffffffu, fresh);
        if (!frm) continue;
        const int fr = __popc(frm & ((1u << lane) - 1u));
        if (fresh) S.cid[fr] = v;
        __syncwarp();
        row_keys<DT, 1>(a.X, a.row_bytes, S.q, S.cid, S.ckey, __popc(frm), 0, 1, qn);
        __syncwarp();
        const unsigned kv = fresh ? S.ckey[fr] : 0xffffffffu;
        __syncwarp();
        // A full list keeps only entries before its L-th: a point behind it
        // would be cut right after the merge, so it skips the merge.
        bool enters = fresh;
        double cand_d64 = qnan;
        if (enters && size == L) {
          enters = entry_less<DT>(kv, v, f32 ? &cand_d64 : nullptr, keyc[L - 1],
                                  idc[L - 1] & kIdMask, f32 ? &dc[L - 1] : nullptr, a, S.q,
                                  E, Eabs);
        }
        // Already in the list?  Its entry sits exactly where v would be
        // merged; otherwise `lo` (the members before v) is v's insertion point.
        int lo = 0;
        if (enters) {
          int hi = size;
          while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            const bool bl = entry_less<DT>(keyc[mid], idc[mid] & kIdMask,
                                           f32 ? &dc[mid] : nullptr, kv, v, f32 ? &cand_d64 : nullptr, a,
                                           S.q, E, Eabs);
            if (bl) lo = mid + 1;
            else hi = mid;
          }
          if (lo < size && (idc[lo] & kIdMask) == v) enters = false;
        }
        const unsigned fm = __ballot_sync(0xffffffffu, enters);
        const int nf = __popc(fm);
        if (nf == 0) continue;
        // ---- the new members, compacted into lanes 0..nf-1
        if (enters) {
          const int r = __popc(fm & ((1u << lane) - 1u));
          S.ckey[r] = kv;
          S.cid[r] = v;
          S.clo[r] = lo;
          if (f32) S.cd64[r] = cand_d64;
        }
        __syncwarp();
        unsigned myk = 0xffffffffu, myid = 0xffffffffu;
        int mylo = 0x7fffffff;
        double myd = qnan;
        if (lane < nf) {
          myk = S.ckey[lane];
          myid = S.cid[lane];
          mylo = S.clo[lane];
          if (f32) myd = S.cd64[lane];
        }
        // ---- sort them: bitonic over the smallest power of two >= nf lanes
        // (empty lanes sort last).  Different insertion points order two new
        // members without a distance: a list member lies between them.
        if (nf > 1) {
          const int w = 1 << (32 - __clz(nf - 1));
          for (int kk = 2; kk <= w; kk <<= 1) {
            for (int j = kk >> 1; j > 0; j >>= 1) {
              const unsigned ok = __shfl_xor_sync(0xffffffffu, myk, j);
              const unsigned oi = __shfl_xor_sync(0xffffffffu, myid, j);
              const int olo = __shfl_xor_sync(0xffffffffu, mylo, j);
              // dec: 1 = my entry comes first, 0 = the partner's, -1 = undecided
              int dec;
              const bool me_empty = myid == 0xffffffffu, o_empty = oi == 0xffffffffu;
              if (me_empty && o_empty) dec = lane < (lane ^ j) ? 1 : 0;
              else if (me_empty) dec = 0;
              else if (o_empty) dec = 1;
              else if (mylo != olo) dec = mylo < olo ? 1 : 0;
              else if (DT == kU8) dec = (myk < ok || (myk == ok && myid < oi)) ? 1 : 0;
              else {
                const float fa = __uint_as_float(myk), fb = __uint_as_float(ok);
                dec = sure_less(fa, fb, E, Eabs) ? 1 : (sure_less(fb, fa, E, Eabs) ? 0 : -1);
              }
              double od = 0.0;
              if constexpr (DT == kF32) {
                // an undecided pair is undecided for both lanes: each brings its
                // own float-float distance, then (still undecided) its binary64
                // one, and both lanes compare the same pair of values
                const float* rowp = reinterpret_cast<const float*>(a.X + int64_t(myid) * a.row_bytes);
                if (dec < 0 && isnan(myd)) myd = -ff_d2(reinterpret_cast<const float*>(S.q), rowp, a.row_bytes);
                od = __shfl_xor_sync(0xffffffffu, myd, j);
                if (dec < 0) dec = slot_order(myd, od, ff_bound(a.d));
                if (dec < 0 && signbit(myd)) {
                  myd = canon_d2_f32(reinterpret_cast<const float*>(S.q), rowp, a.d);
                  atomicAdd(&a.status->fp64_search, 1ull);
                }
                od = __shfl_xor_sync(0xffffffffu, myd, j);
                if (dec < 0) dec = (myd < od || (myd == od && myid < oi)) ? 1 : 0;
              }
              const bool less_me = dec == 1;
              const bool up = (lane & kk) == 0;
              const bool lower = (lane & j) == 0;
              const bool take_partner = (lower == up) ? !less_me : less_me;
              if (take_partner) {
                myk = ok;
                myid = oi;
                mylo = olo;
                myd = od;
              }
            }
          }
          if (lane < nf) S.clo[lane] = mylo;
          __syncwarp();
        }
        // ---- merge in place, back to front: member i moves to i + #{r : clo[r] <= i}
        // and new member r to clo[r] + r; positions from L on are cut.  New
        // positions only grow and never meet, so a chunk read before any write
        // to its range is never clobbered.  Members before clo[0] stay.
        const int first = __shfl_sync(0xffffffffu, mylo, 0);
        for (int c0 = (size - 1) & ~31; c0 >= (first & ~31) && first < size; c0 -= 32) {
          const int i = c0 + lane;
          const bool mv = i >= first && i < size;
          unsigned bk = 0, bi = 0;
          double bd = 0.0;
          int np = L;
          if (mv) {
            bk = keyc[i];
            bi = idc[i];
            if (f32) bd = dc[i];
            int l2 = 1, h2 = nf;  // clo[0] = first <= i
            while (l2 < h2) {
              const int mid = (l2 + h2) >> 1;
              if (S.clo[mid] <= i) l2 = mid + 1;
              else h2 = mid;
            }
            np = i + l2;
          }
          __syncwarp();
          if (mv && np < L) {
            keyc[np] = bk;
            idc[np] = bi;
            if (f32) dc[np] = bd;
          }
          __syncwarp();
        }
        if (lane < nf && mylo + lane < L) {
          keyc[mylo + lane] = myk;
          idc[mylo + lane] = myid;
          if (f32) dc[mylo + lane] = myd;
        }
        __syncwarp();
        size = min(L, size + nf);
        f = min(f, first);
      }
    }
    if (a.visited_cnt && lane == 0) a.visited_cnt[qi] = int32_t(iters < INT32_MAX ? iters : INT32_MAX);
    // ---- the k closest members
    for (int j = lane; j < a.k; j += 32) {
      const bool have = j < size;
      a.out_ids[int64_t(qi) * a.k + j] = have ? int32_t(idc[j] & kIdMask) : -1;
      if (a.out_dists) {
        float dv;
        if (!have) dv = __int_as_float(0x7f800000);
        else if (DT == kU8) dv = float(keyc[j]);
        else dv = __uint_as_float(keyc[j]);
        a.out_dists[int64_t(qi) * a.k + j] = dv;
      }
    }
    __syncwarp();
  }
}

// ---------------------------------------------------------------------------
// the list in registers
// ---------------------------------------------------------------------------
constexpr int kRegL = 256;      // longest list of search_reg_kernel
constexpr int kNbr = 64;        // neighbours taken at a time
constexpr int kTeamQueriesPerSm = 3;
constexpr int kSmallTeam = 3;   // the same with two that read rows
constexpr int kSmallTeamCtas = 7;
constexpr int kSmallTeamQueriesPerSm = 8;
constexpr unsigned kEmptyId = 0xffffffffu;  // an empty slot: expanded, no point has its id

struct RegSmem {
  unsigned* cache;
  uint8_t* q;
  unsigned* cid;   // [kNbr] new ids
  unsigned* ckey;  // [kNbr] their distances
  int* ctl;        // team form: rows to read (-1: the query is done); [1] the query; [2] what is left of kFineBudget, [3] binary64 decisions
};

__host__ __device__ inline size_t reg_bytes(int64_t row_bytes, int cache_bits) {
  return ((size_t(4) << cache_bits) + size_t(row_bytes) + size_t(2 * kNbr) * 4 + 16 + 127) & ~size_t(127);
}
__device__ inline RegSmem reg_carve(unsigned char* p, int64_t row_bytes, int cache_bits) {
  RegSmem w;
  w.cache = reinterpret_cast<unsigned*>(p);
  p += size_t(4) << cache_bits;
  w.q = p;
  p += row_bytes;
  w.cid = reinterpret_cast<unsigned*>(p);
  p += kNbr * 4;
  w.ckey = reinterpret_cast<unsigned*>(p);
  p += kNbr * 4;
  w.ctl = reinterpret_cast<int*>(p);
  return w;
}

// Whether point `m` precedes point `c` in (distance, id) order, where their
// single-precision intervals overlap: by float-float distances, by id where those are
// exact or the rows the same, else by the canonical binary64 ones.  Called by a whole
// warp; out of line, since it is rare.  q lies in a RegSmem, whose ctl[2] is what the
// query may still spend: once that is negative, any answer does and rows of no
// dimensions are compared.  ctl[3] counts the binary64 decisions.  Where one is no
// number, so are most that follow: that costs the whole budget.
__device__ __noinline__ bool precedes_fine(const uint8_t* Xb, int64_t row_bytes, int d, const float* q, unsigned m,
                                           unsigned c) {
  int* left = reinterpret_cast<int*>(const_cast<uint8_t*>(reinterpret_cast<const uint8_t*>(q)) + row_bytes) +
              2 * kNbr + 2;
  const int nch = *left < 0 ? 0 : int(row_bytes / 16);
  const float* xm = reinterpret_cast<const float*>(Xb + int64_t(m) * row_bytes);
  const float* xc = reinterpret_cast<const float*>(Xb + int64_t(c) * row_bytes);
  // (every vote on the way of every call: one under a condition, or a return before
  // the end, and ptxas spills in the search's loop, 1.43 to 1.58 ms where it takes 0.95)
  bool differ = false;
#pragma unroll 1
  for (int i = threadIdx.x & 31; i < nch; i += 32) {
    const float4 a = __ldg(reinterpret_cast<const float4*>(xm) + i), b = __ldg(reinterpret_cast<const float4*>(xc) + i);
    differ |= a.x != b.x || a.y != b.y || a.z != b.z || a.w != b.w;
  }
  const bool same = !__any_sync(0xffffffffu, differ);
  bool em, ec;
  const double dm = ff_d2_exact(q, xm, nch, em), dc = ff_d2_exact(q, xc, nch, ec);
  int o = slot_order(-dm, -dc, ff_bound(d));
  if (em && ec) o = dm < dc || (dm == dc && m < c);
  if (same) o = m < c;
  const bool f64 = o < 0;
  // lane 0 of m, lane 1 of c; no steps in the others, or if float-float decided
  const float* x = reinterpret_cast<const float*>(Xb + int64_t((threadIdx.x & 31) ? c : m) * row_bytes);
  const int steps = f64 && (threadIdx.x & 31) < 2 ? d : 0;
  double v = 0.0;
#pragma unroll 1
  for (int i = 0; i < steps; ++i) {
    const double t = __dsub_rn(double(q[i]), double(__ldg(x + i)));
    v = __dadd_rn(v, __dmul_rn(t, t));
  }
  const double vm = __shfl_sync(0xffffffffu, v, 0), vc = __shfl_sync(0xffffffffu, v, 1);
  if (f64) o = vm < vc || (vm == vc && m < c);
  if ((threadIdx.x & 31) == 0) {
    const bool finite = vm + vc < __longlong_as_double(0x7ff0000000000000LL);
    *left -= !f64 ? 1 : finite ? kFineF64 : kFineBudget + 1;
    left[1] += f64;
  }
  __syncwarp();
  return o == 1;
}

// The list of one query, held by a warp: entry i in slot i % S of lane i / S,
// sorted by (distance, id), empty entries last (they have no point's id and
// count as expanded).  Entries from L on have been cut: they are never expanded
// or returned, and since nothing is ever taken out they cannot come back.
// Slots are only indexed by constants, so they stay in registers.
template <int DT, int S>
struct RegList {
  static constexpr unsigned kFull = 0xffffffffu;
  unsigned key[S], idv[S];
  unsigned inside;  // bit j: entry j of this lane lies before L

  __device__ __forceinline__ void clear(int L, int lane) {
    inside = 0;
#pragma unroll
    for (int j = 0; j < S; ++j) {
      key[j] = DT == kU8 ? 0xffffffffu : 0x7f800000u;  // behind every point
      idv[j] = kEmptyId;
      inside |= lane * S + j < L ? 1u << j : 0u;
    }
  }
  // Slot j of lane l: the key there, in every lane.
  __device__ __forceinline__ unsigned key_at(int l, int j) const {
    unsigned v = 0;
#pragma unroll
    for (int i = 0; i < S; ++i) v |= i == j ? key[i] : 0u;
    return __shfl_sync(kFull, v, l);
  }
  // This lane's unexpanded entries before L, as bits.
  __device__ __forceinline__ unsigned open_bits() const {
    unsigned v = 0;
#pragma unroll
    for (int j = 0; j < S; ++j) v |= (idv[j] >> 31) << j;
    return inside & ~v;
  }
  // The point at the lowest of `u`'s bits in the first lane that has any.
  __device__ __forceinline__ unsigned first_of(unsigned u, unsigned who) const {
    unsigned v = idv[S - 1];
#pragma unroll
    for (int j = S - 2; j >= 0; --j) v = (u >> j) & 1u ? idv[j] : v;
    return __shfl_sync(kFull, v, __ffs(who) - 1);
  }
  // The closest unexpanded member, marked expanded (kEmptyId: none is left), and
  // if `next` is asked for the one after it.
  template <bool NEXT>
  __device__ __forceinline__ unsigned pop(unsigned& next, int lane) {
    unsigned u = open_bits();
    const unsigned who = __ballot_sync(kFull, u != 0);
    if (!who) return kEmptyId;
    const unsigned p = first_of(u, who);
    const unsigned low = lane == __ffs(who) - 1 ? u & (0u - u) : 0u;
#pragma unroll
    for (int j = 0; j < S; ++j) idv[j] |= (low << (31 - j)) & kVisited;
    if constexpr (NEXT) {
      u &= ~low;
      const unsigned who2 = __ballot_sync(kFull, u != 0);
      next = who2 ? first_of(u, who2) : kEmptyId;
    }
    return p;
  }
  // Puts point c at distance kc in its place.  stay: bit j = this lane's entry j
  // precedes it; before: so does the entry before this lane's first.
  __device__ __forceinline__ void place(unsigned kc, unsigned c, unsigned stay, bool before, unsigned pk, unsigned pi) {
#pragma unroll
    for (int j = S - 1; j >= 0; --j) {
      const bool here = (stay >> j) & 1u;
      const bool prev = j > 0 ? (stay >> (j > 0 ? j - 1 : 0)) & 1u : before;
      const unsigned mk = j > 0 ? key[j > 0 ? j - 1 : 0] : pk, mi = j > 0 ? idv[j > 0 ? j - 1 : 0] : pi;
      key[j] = here ? key[j] : prev ? kc : mk;
      idv[j] = here ? idv[j] : prev ? c : mi;
    }
  }
  // Adds point c at distance kc unless it is a member.  An entry whose key lies
  // below kc (1 - E2) - A2 surely precedes it and one above kc (1 + E2) + A2
  // surely follows (E2 = 2 E and four ulps, A2 = 4 Eabs: the two intervals are
  // then apart); the rest, equal keys for uint8, are settled on ids or on finer
  // distances, and the point itself is among them if it is a member.
  __device__ __forceinline__ void add(unsigned kc, unsigned c, const SearchArgs& a, const uint8_t* q, float E2,
                                      float A2, int lane) {
    const unsigned pk = __shfl_up_sync(kFull, key[S - 1], 1), pi = __shfl_up_sync(kFull, idv[S - 1], 1);
    bool less[S];
    bool near = false, before;
    if constexpr (DT == kU8) {
#pragma unroll
      for (int j = 0; j < S; ++j) {
        less[j] = key[j] < kc;
        near |= key[j] == kc;
      }
      before = pk < kc || lane == 0;
    } else {
      const float f = __uint_as_float(kc);
      const float lo = f * (1.0f - E2) - A2, hi = f * (1.0f + E2) + A2;
#pragma unroll
      for (int j = 0; j < S; ++j) {
        less[j] = __uint_as_float(key[j]) < lo;
        near |= !less[j] && !(__uint_as_float(key[j]) > hi);
      }
      before = __uint_as_float(pk) < lo || lane == 0;
    }
    if (__any_sync(kFull, near)) {
      add_near(kc, c, a, q, E2, A2, lane, pk, pi);
      return;
    }
#pragma unroll
    for (int j = S - 1; j >= 0; --j) {
      const bool prev = j > 0 ? less[j > 0 ? j - 1 : 0] : before;
      const unsigned mk = j > 0 ? key[j > 0 ? j - 1 : 0] : pk, mi = j > 0 ? idv[j > 0 ? j - 1 : 0] : pi;
      key[j] = less[j] ? key[j] : prev ? kc : mk;
      idv[j] = less[j] ? idv[j] : prev ? c : mi;
    }
  }
  __device__ __forceinline__ void add_near(unsigned kc, unsigned c, const SearchArgs& a, const uint8_t* q, float E2,
                                           float A2, int lane, unsigned pk, unsigned pi) {
    unsigned stay = 0;
    // a float query without budget: nothing more is added
    bool have = DT == kF32 && reinterpret_cast<const int*>(q + a.row_bytes)[2 * kNbr + 2] < 0;
#pragma unroll
    for (int j = 0; j < S; ++j) have |= (idv[j] & kIdMask) == c;
    if (__any_sync(kFull, have)) return;
    if constexpr (DT == kU8) {
#pragma unroll
      for (int j = 0; j < S; ++j)
        stay |= key[j] < kc || (key[j] == kc && (idv[j] & kIdMask) < c) ? 1u << j : 0u;
    } else {
      const float f = __uint_as_float(kc);
      const float lo = f * (1.0f - E2) - A2, hi = f * (1.0f + E2) + A2;
      unsigned close = 0;  // this lane's entries to be settled
#pragma unroll
      for (int j = 0; j < S; ++j) {
        const float fj = __uint_as_float(key[j]);
        stay |= fj < lo ? 1u << j : 0u;
        close |= !(fj < lo) && !(fj > hi) && idv[j] != kEmptyId ? 1u << j : 0u;
      }
      while (const unsigned who = __ballot_sync(kFull, close != 0)) {
        const unsigned low = close & (0u - close);
        const unsigned m = first_of(close, who) & kIdMask;
        const bool first = precedes_fine(a.X, a.row_bytes, a.d, reinterpret_cast<const float*>(q), m, c);
        if (lane == __ffs(who) - 1) {
          close ^= low;
          stay |= first ? low : 0u;
        }
      }
    }
    const unsigned ps = __shfl_up_sync(kFull, stay, 1);
    place(kc, c, stay, lane == 0 || ((ps >> (S - 1)) & 1u), pk, pi);
  }
};

// One query per warp (W = 1, four warps per CTA), or per CTA of W warps: warp 0
// keeps the list and the others read the rows.
//
// What bounds it: with one warp per query, the instructions of an expansion (row
// distances, adding points); with a team, the chain row bounds -> ids -> rows of
// each expansion and the list's warp.  A team therefore knows the next member to
// be expanded before the current one is done (only a closer new point displaces
// it: 9 of 10 stay), loads its row bounds before the current rows are read and
// its ids before they are added.  Without a team other queries hide that chain,
// and the registers count for more.
//
// Measured, a list sorted in shared memory (32 neighbours at a time, one lane per
// row) -> this kernel: 400,000 x 96 floats, L = 100, one query 585 -> 142 us,
// 10,000 queries 2.57 -> 0.89 ms; 400,000 x 128 uint8, L = 128, 10,000 queries
// 2.11 -> 1.13 ms; 30,000 x 960 floats, L = 200, 1,000 queries 23.2 -> 4.6 ms (by
// the counters 37 GB from L2, 7.9 TB/s; the two before 4.1 and 7.3 GB).  Also
// measured: an unordered list with its minimum and maximum by warp reductions (one
// query 216 us, 10,000 1.84 ms).  Eight CTAs per SM of one-warp queries (64 registers)
// beat six and ten (0.89 against 0.98 and 1.09 ms on the float rows).
template <int DT, int S, int W>
__global__ void __launch_bounds__(W == 1 ? kWarps * 32 : W * 32, W == 1 ? 8 : W == kTeam ? 3 : kSmallTeamCtas)
    search_reg_kernel(SearchArgs a) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const RegSmem M = reg_carve(smem_raw + (W == 1 ? size_t(warp) * reg_bytes(a.row_bytes, a.cache_bits) : 0),
                              a.row_bytes, a.cache_bits);
  const int cshift = 32 - a.cache_bits;
  const int nch = int(a.row_bytes / 16);
  const unsigned full = 0xffffffffu;
  const float E2 = 2.0f * lane_rel_bound(nch) + 2.3841858e-07f, A2 = 4.0f * abs_bound(a.d);
  const int wthreads = W == 1 ? 32 : W * 32, wt = W == 1 ? lane : int(threadIdx.x);

  for (;;) {
    unsigned qi = 0;
    if constexpr (W == 1) {
      if (lane == 0) qi = atomicAdd(a.work, 1u);
      qi = __shfl_sync(full, qi, 0);
    } else {
      if (threadIdx.x == 0) M.ctl[1] = int(atomicAdd(a.work, 1u));
      __syncthreads();
      qi = unsigned(M.ctl[1]);
    }
    if (qi >= a.nq) break;
    const uint4* src = reinterpret_cast<const uint4*>(
        a.q_point ? a.X + int64_t(a.q_point[qi]) * a.row_bytes : a.Q + int64_t(qi) * a.row_bytes);
    for (int c = wt; c < nch; c += wthreads) reinterpret_cast<uint4*>(M.q)[c] = src[c];
    for (int c = wt; c < (1 << a.cache_bits); c += wthreads) M.cache[c] = kEmptyId;
    if constexpr (W == 1) __syncwarp();
    else __syncthreads();
    unsigned qn = 0;  // uint8: |q|^2
    if constexpr (DT == kU8) {
      for (int w4 = lane; w4 < 4 * nch; w4 += 32) {
        const unsigned qw = reinterpret_cast<const unsigned*>(M.q)[w4];
        qn = __dp4a(qw, qw, qn);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) qn += __shfl_xor_sync(full, qn, o);
    }
    if (W > 1 && warp > 0) {
      // the team: distances of the new rows, as warp 0 asks for them
      for (;;) {
        __syncthreads();
        const int nf = M.ctl[0];
        if (nf < 0) break;
        row_keys<DT, W>(a.X, a.row_bytes, M.q, M.cid, M.ckey, nf, warp - 1, W - 1, qn);
        __syncthreads();
      }
      __syncthreads();
      continue;
    }
    const int64_t* __restrict__ row_ptr = a.row_ptr;
    const int32_t* __restrict__ col = a.col;
    unsigned start = unsigned(a.start);
    if (a.q_graph) {
      const SearchGraph sg = a.graphs[a.q_graph[qi]];
      row_ptr = sg.row_ptr;
      col = sg.col;
      start = unsigned(sg.start);
    }
    RegList<DT, S> list;
    const int L = a.q_L ? a.q_L[qi] : a.L;
    list.clear(L, lane);
    if (lane == 0) {
      M.cid[0] = start;
      M.cache[(start * 0x9E3779B1u) >> cshift] = start;
      if (DT == kF32) M.ctl[2] = a.fine_budget, M.ctl[3] = 0;
    }
    __syncwarp();
    row_keys<DT, 1>(a.X, a.row_bytes, M.q, M.cid, M.ckey, 1, 0, 1, qn);
    __syncwarp();
    if (lane == 0) {
      list.key[0] = M.ckey[0];
      list.idv[0] = start;
    }
    __syncwarp();

    // the expected next expansion: its point, row and first ids
    unsigned nx = kEmptyId;
    const int32_t* nx_ids = col;
    int nx_deg = 0;
    unsigned nx_v0 = 0, nx_v1 = 0;
    int64_t iters = 0;
    for (;;) {
      unsigned after = kEmptyId;
      const unsigned ps = list.template pop<(W > 1)>(after, lane);
      if (ps == kEmptyId) break;
      if (++iters > a.n + 1) {  // cannot happen: each point is expanded at most once
        if (lane == 0) raise_status(a.status, kDevOverflow, qi);
        break;
      }
      if (a.visited && lane == 0 && iters <= a.visited_cap)
        a.visited[int64_t(qi) * a.visited_cap + iters - 1] = int32_t(ps);
      // row v: its first id and its degree
      auto bounds = [&](unsigned v, const int32_t*& ids, int& deg) {
        if (a.adj_deg) {
          ids = col + int64_t(v) * a.adj_stride;
          deg = a.adj_deg[v];
        } else {
          const int64_t b = row_ptr[v];
          ids = col + b;
          deg = int(row_ptr[v + 1] - b);
        }
      };
      const int32_t* ids;
      int deg;
      unsigned v0, v1;
      if (W > 1 && ps == nx) {
        ids = nx_ids;
        deg = nx_deg;
        v0 = nx_v0;
        v1 = nx_v1;
      } else {
        bounds(ps, ids, deg);
        v0 = lane < deg ? unsigned(ids[lane]) : 0u;
        v1 = 32 + lane < deg ? unsigned(ids[32 + lane]) : 0u;
      }
      nx = after;
      if (W > 1 && nx != kEmptyId) bounds(nx, nx_ids, nx_deg);
      bool first = true;
      for (int eb = 0; eb < deg || first; eb += kNbr) {
        if (!first) {
          v0 = eb + lane < deg ? unsigned(ids[eb + lane]) : 0u;
          v1 = eb + 32 + lane < deg ? unsigned(ids[eb + 32 + lane]) : 0u;
        }
        // ---- the neighbours that the cache does not hold.  A row holds
        // distinct ids, so lanes that share a cache entry hold different ids:
        // whichever write lands, no lane skips a new id.
        const unsigned below = (1u << lane) - 1u;
        int nf = 0;
        auto take = [&](unsigned v, bool in) {
          const unsigned h = (v * 0x9E3779B1u) >> cshift;
          const bool f = in && M.cache[h] != v;
          const unsigned m = __ballot_sync(full, f);
          if (f) {
            M.cache[h] = v;
            M.cid[nf + __popc(m & below)] = v;
          }
          nf += __popc(m);
        };
        take(v0, eb + lane < deg);
        if (eb + 32 < deg) take(v1, eb + 32 + lane < deg);
        if (nf > 0) {
          if constexpr (W == 1) {
            __syncwarp();
            row_keys<DT, 1>(a.X, a.row_bytes, M.q, M.cid, M.ckey, nf, 0, 1, qn);
          } else {
            if (lane == 0) M.ctl[0] = nf;
            __syncthreads();
          }
        }
        if (W > 1 && first && nx != kEmptyId) {  // its row bounds are here by now
          nx_v0 = lane < nx_deg ? unsigned(nx_ids[lane]) : 0u;
          nx_v1 = 32 + lane < nx_deg ? unsigned(nx_ids[32 + lane]) : 0u;
        }
        first = false;
        if (nf == 0) continue;
        if constexpr (W == 1) __syncwarp();
        else __syncthreads();
        // ---- those that may come before the L-th entry (an empty one: all of
        // them).  A distance that is no number, of a query that holds one, never
        // displaces a member.  None once the query's budget is spent: it then soon
        // runs out of members to expand.
        const unsigned kth = list.key_at((L - 1) / S, (L - 1) % S);
        const float last = __uint_as_float(kth) * (1.0f + E2) + A2;
        auto enters = [&](int i) {
          if (i >= nf || (W == 1 && DT == kF32 && M.ctl[2] < 0)) return false;
          if constexpr (DT == kU8) return M.ckey[i] <= kth;
          else return __uint_as_float(M.ckey[i]) <= last || kth == 0x7f800000u;
        };
#pragma unroll 1
        for (int base = 0; base < nf; base += 32) {
          unsigned todo = __ballot_sync(full, enters(base + lane));
          if (W > 1 && DT == kF32 && todo && M.ctl[2] < 0) break;
          while (todo) {
            const int at = base + __ffs(todo) - 1;
            todo &= todo - 1;
            list.add(M.ckey[at], M.cid[at], a, M.q, E2, A2, lane);
          }
        }
        __syncwarp();
      }
    }
    if constexpr (W > 1) {
      if (lane == 0) M.ctl[0] = -1;
      __syncthreads();
    }
    if (a.visited_cnt && lane == 0) a.visited_cnt[qi] = int32_t(iters < INT32_MAX ? iters : INT32_MAX);
    // ---- the k closest members
    const bool redo = DT == kF32 && M.ctl[2] < 0;  // given up for search_list_kernel
    if (DT == kF32 && lane == 0 && M.ctl[3] != 0) atomicAdd(&a.status->fp64_search, 2ull * unsigned(M.ctl[3]));
#pragma unroll
    for (int j = 0; j < S; ++j) {
      const int i = lane * S + j;
      if (redo) {
        if (i == 0) a.out_ids[int64_t(qi) * a.k] = kSearchRedo;
      } else if (i < a.k) {
        const bool have = list.idv[j] != kEmptyId;
        const int64_t at = int64_t(qi) * a.k + i;
        a.out_ids[at] = have ? int32_t(list.idv[j] & kIdMask) : -1;
        if (a.out_dists)
          a.out_dists[at] = !have ? __int_as_float(0x7f800000)
                                  : (DT == kU8 ? float(list.key[j]) : __uint_as_float(list.key[j]));
      }
    }
    if constexpr (W == 1) __syncwarp();
    else __syncthreads();
  }
}

__global__ void recall_kernel(const int32_t* __restrict__ found, int ld_found, const int32_t* __restrict__ truth,
                              int ld_truth, int64_t nq, int k, unsigned long long* hits) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t q = int64_t(blockIdx.x) * (blockDim.x >> 5) + w;
  if (q >= nq) return;
  const int32_t* f = found + q * ld_found;
  const int32_t* t = truth + q * ld_truth;
  unsigned long long h = 0;
  for (int i = lane; i < k; i += 32) {
    const int32_t v = f[i];
    if (v < 0) continue;
    for (int j = 0; j < k; ++j)
      if (t[j] == v) {
        ++h;
        break;
      }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) h += __shfl_down_sync(0xffffffffu, h, o);
  if (lane == 0 && h) atomicAdd(hits, h);
}

}  // namespace

// The CTAs per SM a configured plan may ask for.
constexpr int kMaxCtasPerSmCap = 16;
constexpr int kMinCacheBits = 8, kMaxCacheBits = 12;
// The default plan stops at 1,024 entries for one warp per query, whose caches
// share an SM with 31 others, and at the most for a team (L = 100 to 256, one pass of
// 512 / 1,024 / the default, in ms: 10,000 queries on 400,000 x 128 uint8 1.19 / 1.14 /
// 1.13, on 400,000 x 96 floats 1.04 / 0.93 / 0.93; by teams, 1,000 on 30,000 x 960
// floats 5.67 / 5.42 / 4.69, 333 on 200,000 x 128 uint8 0.57 / 0.52 / 0.45).
constexpr int kDefaultMaxCacheBits = 10;

using SearchKernel = void (*)(SearchArgs);

// The kernels of one data type: the list in registers in 4 or 8 slots, one
// warp or a team per query, and the list in shared memory.
template <int DT>
SearchKernel search_kernel_of(bool reg, int slots, int warps) {
  if (!reg) return search_list_kernel<DT, false>;
  if (warps == kTeam) return slots <= 4 ? search_reg_kernel<DT, 4, kTeam> : search_reg_kernel<DT, 8, kTeam>;
  if (warps == kSmallTeam) return slots <= 4 ? search_reg_kernel<DT, 4, kSmallTeam> : search_reg_kernel<DT, 8, kSmallTeam>;
  return slots <= 4 ? search_reg_kernel<DT, 4, 1> : search_reg_kernel<DT, 8, 1>;
}

// Every kernel may use all the shared memory a block can have, set once per
// device (which also loads them all, so that a later call inside a stream
// capture finds its kernel loaded).
cudaError_t prepare_kernels() {
  static std::mutex mu;
  static std::map<int, bool> done;
  int dev = 0, most = 0;
  cudaError_t err = cudaGetDevice(&dev);
  if (err != cudaSuccess) return err;
  std::lock_guard<std::mutex> g(mu);
  if (done.count(dev)) return cudaSuccess;
  if ((err = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess) return err;
  const int warps[4] = {1, kSmallTeam, kTeam, 0};
  for (int v = 0; v < 16; ++v) {
    const int slots = (v & 2) ? 8 : 4, w = warps[v >> 2];
    SearchKernel k = (v & 1) ? search_kernel_of<kF32>(w > 0, slots, w) : search_kernel_of<kU8>(w > 0, slots, w);
    if ((err = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, most)) != cudaSuccess) return err;
  }
  err = cudaFuncSetAttribute(search_list_kernel<kF32, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
  if (err != cudaSuccess) return err;
  done[dev] = true;
  return cudaSuccess;
}

// Default plan: the queries in flight hide the latency of each expansion, so
// the search first maximises the CTAs per SM, then takes the largest id cache
// (256 to 1,024 entries per query, a team's up to 4,096) that keeps that many.
// Plans are remembered per (kernel, L, row bytes); the occupancy queries run once for
// each.
struct SearchPlan {
  int bits = kMinCacheBits;
  int ctas = 1;
};

struct SearchForm {
  SearchKernel kern = nullptr;
  int threads = 0;
  int queries = 0;  // in flight per CTA
  bool reg = false, f32 = false;
  int L = 0;
  int64_t row_bytes = 0;
  size_t bytes(int bits) const {
    return size_t(queries) * (reg ? reg_bytes(row_bytes, bits) : warp_bytes(L, row_bytes, f32, bits));
  }
};

cudaError_t default_plan(const SearchForm& F, SearchPlan* plan) {
  static std::mutex mu;
  static std::map<std::tuple<SearchKernel, int, int64_t>, SearchPlan> memo;
  const auto key = std::make_tuple(F.kern, F.reg ? 0 : F.L, F.row_bytes);
  {
    std::lock_guard<std::mutex> g(mu);
    auto it = memo.find(key);
    if (it != memo.end()) {
      *plan = it->second;
      return cudaSuccess;
    }
  }
  SearchPlan best;
  int best_ctas = 0;
  for (int b = kMinCacheBits; b <= (F.queries == 1 ? kMaxCacheBits : kDefaultMaxCacheBits); ++b) {
    int nb = 0;
    cudaError_t err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, F.kern, F.threads, F.bytes(b));
    if (err != cudaSuccess) return err;
    if (nb >= best_ctas && nb > 0) {  // ties go to the larger cache
      best_ctas = nb;
      best.bits = b;
      best.ctas = nb;
    }
  }
  if (best_ctas == 0) return cudaErrorInvalidConfiguration;
  best.ctas = std::min(best.ctas, kMaxCtasPerSmCap);
  std::lock_guard<std::mutex> g(mu);
  memo[key] = best;
  *plan = best;
  return cudaSuccess;
}

cudaError_t launch_search(const SearchLaunch& L, cudaStream_t s, int* kernels) {
  SearchArgs a{};
  a.X = L.data.X;
  a.row_bytes = L.data.row_bytes;
  a.d = L.data.d;
  a.n = L.data.n;
  a.row_ptr = L.row_ptr;
  a.col = L.col;
  a.start = L.start;
  a.graphs = L.graphs;
  a.q_graph = L.q_graph;
  a.q_L = L.q_L;
  a.Q = L.Q;
  a.nq = L.nq;
  a.L = L.L;
  a.k = L.k;
  a.out_ids = L.out_ids;
  a.out_dists = L.out_dists;
  a.work = L.work;
  a.status = L.status;
  a.q_point = L.q_point;
  a.adj_deg = L.adj_deg;
  a.adj_stride = L.adj_stride;
  a.visited = L.visited;
  a.visited_cnt = L.visited_cnt;
  a.visited_cap = L.visited_cap;
  cudaError_t err = prepare_kernels();
  if (err != cudaSuccess) return err;
  SearchForm F;
  F.f32 = L.data.dtype == kF32;
  F.reg = L.L <= kRegL;
  F.L = L.L;
  F.row_bytes = L.data.row_bytes;
  // Few queries: a team per query.  400,000 x 96 floats, one warp / team of
  // three / team of five, in us: 152 queries 198 / 178 / 181, 456: 292 / 256 /
  // 241, 800: 370 / 321 / 450, 1,216: 382 / 342 / 624, 1,824: 399 / 495 / 858;
  // 128-byte uint8 rows alike.  The lines lie at 3 and 8 queries per SM: a team's
  // CTAs (3 and 7 per SM) then hold all or nearly all of them at once.
  const int warps = !F.reg ? 0
                    : L.nq <= int64_t(L.num_sms) * kTeamQueriesPerSm      ? kTeam
                    : L.nq <= int64_t(L.num_sms) * kSmallTeamQueriesPerSm ? kSmallTeam
                                                                          : 1;
  const int slots = (L.L + 31) / 32;
  F.kern = F.f32 ? search_kernel_of<kF32>(F.reg, slots, warps) : search_kernel_of<kU8>(F.reg, slots, warps);
  F.threads = (warps > 1 ? warps : kWarps) * 32;
  F.queries = warps > 1 ? 1 : kWarps;
  SearchPlan plan;
  if (L.cache_bits >= kMinCacheBits && L.cache_bits <= kMaxCacheBits) {  // a configured plan (rp_set_search_config)
    plan.bits = L.cache_bits;
    err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&plan.ctas, F.kern, F.threads, F.bytes(plan.bits));
    if (err != cudaSuccess) return err;
    plan.ctas = std::min(plan.ctas, kMaxCtasPerSmCap);
  } else if ((err = default_plan(F, &plan)) != cudaSuccess) {
    return err;
  }
  // Float queries that search_reg_kernel gives up (none, where the other kernel's
  // shared memory does not fit: long rows of few queries).
  SearchForm R = F;
  SearchPlan redo_plan;
  bool redo = F.f32 && F.reg;
  if (redo) {
    R.kern = search_list_kernel<kF32, true>;
    R.reg = false;
    R.threads = kWarps * 32;
    R.queries = kWarps;
    err = default_plan(R, &redo_plan);
    if (err != cudaSuccess && err != cudaErrorInvalidConfiguration) return err;
    redo = err == cudaSuccess;
  }
  a.fine_budget = redo ? kFineBudget : INT_MAX;
  if (L.pass == kSearchAgain && !redo) return cudaSuccess;
  auto run = [&](const SearchForm& G, const SearchPlan& p) {
    int base_ctas = p.ctas;
    if (L.ctas_per_sm > 0) base_ctas = std::min(base_ctas, L.ctas_per_sm);
    base_ctas = std::max(base_ctas, 1);
    a.cache_bits = p.bits;
    const int64_t want = int64_t(L.num_sms) * base_ctas;
    const int64_t need = (L.nq + G.queries - 1) / G.queries;
    const int grid = int(std::max<int64_t>(1, std::min(want, need)));
    G.kern<<<grid, G.threads, G.bytes(p.bits), s>>>(a);
    return cudaGetLastError();
  };
  const bool first = L.pass != kSearchAgain, again = redo && L.pass != kSearchOnce;
  if (kernels) *kernels = int(first) + int(again);
  err = first ? run(F, plan) : cudaSuccess;
  return err == cudaSuccess && again ? run(R, redo_plan) : err;
}

cudaError_t launch_recall(const int32_t* found, int ld_found, const int32_t* truth, int ld_truth, int64_t nq, int k,
                          unsigned long long* hits, cudaStream_t s) {
  const int per = 8;
  const int64_t blocks = (nq + per - 1) / per;
  recall_kernel<<<unsigned(blocks), per * 32, 0, s>>>(found, ld_found, truth, ld_truth, nq, k, hits);
  return cudaGetLastError();
}

}  // namespace rpk
