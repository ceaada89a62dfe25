// Exact k nearest neighbours by brute force, ordered by (distance, id): the
// ground truth of k-recall@k (§4) and the candidate lists of kNN-candidate
// base graphs.
//
// A CTA owns 32 queries and streams every base point past them in tiles of
// 128 points, one 128-byte slice of every row at a time (cp.async into padded
// shared rows).  Each thread accumulates a 4 x 4 block of squared distances.
// A distance enters the query's candidate buffer only if its (distance, id)
// key is below the query's current threshold (the KEEP-th best so far); when
// a buffer could overflow on the next tile, each warp sorts the buffers of
// its queries in shared memory and keeps the best KEEP.
//
// uint8 distances are exact.  float32 keys are summed per 128-byte slice (32
// dimensions, in index order) and the slice sums added in order, which keeps
// their rigorous error bound at (min(d, 32) + ceil(d / 32) + 8) ulps instead
// of (d + 8) for one running sum (the difference matters at d = 960, where
// the distances of the 128-th and 160-th neighbours can lie that close).  At
// the end, runs of keys whose intervals overlap are re-ordered by binary64
// distances, and the list is accepted only if the k-th entry's run ends
// strictly before the last kept entry (so no discarded point can belong to
// the true top k); otherwise the device status reports kDevTieUnresolved.
#include <cmath>
#include <cstring>

#include "internal.h"
#include "tc.cuh"

namespace rpk {

namespace {

constexpr int QB = 32;        // queries per CTA
constexpr int PB = 128;       // points per tile
constexpr int CAP = 512;      // candidate buffer per query
constexpr int kPitch = 144;   // shared row pitch for one 128-byte slice
constexpr int kThreads = 256;

struct KnnArgs {
  const uint8_t* X;
  int64_t row_bytes;
  int64_t n;
  int d;
  const uint8_t* Q;  // nullptr: queries are base points 0..nq-1 (self excluded)
  int64_t nq;
  int64_t q_base;    // this launch handles queries q_base .. q_end-1
  int64_t q_end;
  int k;
  int keep;  // entries kept per query between merges (k for exact data, k + 32 for float)
  int32_t* out_ids;
  float* out_dists;
  DevStatus* status;
};

struct KnnSmem {
  unsigned long long buf[QB][CAP];
  unsigned long long thr[QB];
  int cnt[QB];
  int flag;
  alignas(16) unsigned char qs[QB * kPitch];
  alignas(16) unsigned char ps[PB * kPitch];
};

template <int DT>
__device__ __forceinline__ void acc_pair(uint2 x, uint2 y, unsigned& acc) {
  if constexpr (DT == kU8) {
    acc = sqdiff4_u8(x.x, y.x, acc);
    acc = sqdiff4_u8(x.y, y.y, acc);
  } else {
    float f = __uint_as_float(acc);
    float t = __uint_as_float(x.x) - __uint_as_float(y.x);
    f = fmaf(t, t, f);
    t = __uint_as_float(x.y) - __uint_as_float(y.y);
    f = fmaf(t, t, f);
    acc = __float_as_uint(f);
  }
}

// Runs of single-precision keys in b[0, m) (sorted ascending) whose intervals
// overlap are re-ordered by (binary64 distance, id); lane 0 alone, runs are
// rare.  Returns the end of the run holding position k - 1 (or -1).
__device__ __forceinline__ int fix_near_ties(const uint8_t* Xb, int64_t row_bytes, int d, DevStatus* status,
                                             unsigned long long* b, int m, const float* qv, int64_t qg, int k = 0) {
  const float E = slice_rel_bound(d), Eabs = abs_bound(d);
  const float* X = reinterpret_cast<const float*>(Xb);
  const int64_t stride = row_bytes / 4;
  int i = 0;
  int kth_run_end = -1;
  while (i < m) {
    int e = i;
    while (e + 1 < m && !sure_less(__uint_as_float(unsigned(b[e] >> 32)), __uint_as_float(unsigned(b[e + 1] >> 32)), E,
                                   Eabs))
      ++e;
    if (e > i) {
      // insertion sort of b[i..e] by (binary64 distance, id)
      double dd[64];
      const int len = min(e - i + 1, 64);
      if (e - i + 1 > 64) raise_status(status, kDevTieUnresolved, qg);
      for (int r = 0; r < len; ++r) dd[r] = canon_d2_f32(qv, X + int64_t(unsigned(b[i + r])) * stride, d);
      atomicAdd(&status->fp64_sort_keys, static_cast<unsigned long long>(len));
      for (int r = 1; r < len; ++r) {
        const unsigned long long kv = b[i + r];
        const double dv = dd[r];
        int z = r - 1;
        while (z >= 0 && (dd[z] > dv || (dd[z] == dv && unsigned(b[i + z]) > unsigned(kv)))) {
          b[i + z + 1] = b[i + z];
          dd[z + 1] = dd[z];
          --z;
        }
        b[i + z + 1] = kv;
        dd[z + 1] = dv;
      }
    }
    if (i <= k - 1 && k - 1 <= e) kth_run_end = e;
    i = e + 1;
  }
  return kth_run_end;
}

// Sort the first `len` (padded to a power of two) keys of one buffer with one warp.
__device__ void warp_sort(unsigned long long* b, int len) {
  int P = 32;
  while (P < len) P <<= 1;
  const int lane = threadIdx.x & 31;
  for (int i = len + lane; i < P; i += 32) b[i] = ~0ull;
  __syncwarp();
  for (int k = 2; k <= P; k <<= 1) {
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int idx = lane; idx < P / 2; idx += 32) {
        const int i = (idx / j) * 2 * j + (idx % j);
        const int l = i + j;
        const bool up = (i & k) == 0;
        const unsigned long long x = b[i], y = b[l];
        if ((x > y) == up) {
          b[i] = y;
          b[l] = x;
        }
      }
      __syncwarp();
    }
  }
}

template <int DT>
__device__ void merge_buffers(KnnSmem& S, int keep) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int q = w; q < QB; q += kThreads / 32) {
    const int c = S.cnt[q];
    if (c > keep || (c == keep && S.thr[q] == ~0ull)) {
      warp_sort(S.buf[q], c);
      if (lane == 0) {
        const int nc = min(c, keep);
        S.cnt[q] = nc;
        if (nc == keep) S.thr[q] = S.buf[q][keep - 1];
      }
    }
    __syncwarp();
  }
}

template <int DT>
__global__ void __launch_bounds__(kThreads) knn_kernel(KnnArgs a) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  KnnSmem& S = *reinterpret_cast<KnnSmem*>(smem_raw);
  const int t = threadIdx.x;
  const int64_t q0 = a.q_base + int64_t(blockIdx.x) * QB;
  const int nqb = int(a.q_end - q0 < QB ? a.q_end - q0 : QB);
  for (int q = t; q < QB; q += kThreads) {
    S.cnt[q] = 0;
    S.thr[q] = ~0ull;
  }
  const int tq = t & 7, tp = t >> 3;  // thread rows: queries tq + 8j, points tp + 32i
  const int nslices = int(a.row_bytes / 128);
  __syncthreads();

  for (int64_t p0 = 0; p0 < a.n; p0 += PB) {
    const int npb = int(a.n - p0 < PB ? a.n - p0 : PB);
    unsigned acc[4][4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[j][i] = 0u;
    for (int s = 0; s < nslices; ++s) {
      unsigned part[4][4];  // this slice's sums
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int i = 0; i < 4; ++i) part[j][i] = 0u;
      for (int c = t; c < (QB + PB) * 8; c += kThreads) {
        const int r = c >> 3, part = c & 7;
        unsigned char* dst;
        const uint8_t* src = nullptr;
        if (r < QB) {
          dst = S.qs + r * kPitch + part * 16;
          if (r < nqb) {
            const int64_t qg = q0 + r;
            src = (a.Q ? a.Q + qg * a.row_bytes : a.X + qg * a.row_bytes) + s * 128 + part * 16;
          }
        } else {
          const int pr = r - QB;
          dst = S.ps + pr * kPitch + part * 16;
          if (pr < npb) src = a.X + (p0 + pr) * a.row_bytes + s * 128 + part * 16;
        }
        if (src) cp_async16(dst, src, 16);
        else *reinterpret_cast<uint4*>(dst) = make_uint4(0, 0, 0, 0);
      }
      cp_async_commit();
      cp_async_wait<0>();
      __syncthreads();
#pragma unroll 4
      for (int wd = 0; wd < 16; ++wd) {
        uint2 qv[4], pv[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) qv[j] = *reinterpret_cast<const uint2*>(S.qs + (tq + 8 * j) * kPitch + wd * 8);
#pragma unroll
        for (int i = 0; i < 4; ++i) pv[i] = *reinterpret_cast<const uint2*>(S.ps + (tp + 32 * i) * kPitch + wd * 8);
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int i = 0; i < 4; ++i) acc_pair<DT>(qv[j], pv[i], part[j][i]);
      }
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          if constexpr (DT == kU8) acc[j][i] += part[j][i];
          else acc[j][i] = __float_as_uint(__uint_as_float(acc[j][i]) + __uint_as_float(part[j][i]));
        }
      __syncthreads();
    }
    // candidates below the thresholds
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int ql = tq + 8 * j;
      if (ql >= nqb) continue;
      const int64_t self = a.Q ? -1 : q0 + ql;
      const unsigned long long thr = S.thr[ql];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int pl = tp + 32 * i;
        const int64_t pid = p0 + pl;
        if (pl >= npb || pid == self) continue;
        const unsigned long long key = (static_cast<unsigned long long>(acc[j][i]) << 32) | unsigned(pid);
        if (key < thr) {
          const int at = atomicAdd(&S.cnt[ql], 1);
          S.buf[ql][at] = key;  // at < CAP: buffers are merged while they hold <= CAP - PB entries
        }
      }
    }
    __syncthreads();
    if (t == 0) {
      int f = 0;
      for (int q = 0; q < QB; ++q) f |= S.cnt[q] > CAP - PB;
      S.flag = f;
    }
    __syncthreads();
    if (S.flag) {
      merge_buffers<DT>(S, a.keep);
      __syncthreads();
    }
  }
  // final ordering
  const int w = t >> 5, lane = t & 31;
  for (int q = w; q < nqb; q += kThreads / 32) {
    const int c = S.cnt[q];
    warp_sort(S.buf[q], c);
    const int nc = min(c, a.keep);
    const int64_t qg = q0 + q;
    unsigned long long* b = S.buf[q];
    if constexpr (DT == kF32) {
      // near-tie runs: re-order by binary64 distances (serial in lane 0; rare)
      if (lane == 0) {
        const float* X = reinterpret_cast<const float*>(a.X);
        const int64_t stride = a.row_bytes / 4;
        const float* qv = a.Q ? reinterpret_cast<const float*>(a.Q + qg * a.row_bytes) : X + qg * stride;
        const int kth_run_end = fix_near_ties(a.X, a.row_bytes, a.d, a.status, b, nc, qv, qg, a.k);
        // a full list whose k-th run reaches the last kept entry may miss points
        if (nc == a.keep && kth_run_end >= nc - 1 && a.keep > a.k) raise_status(a.status, kDevTieUnresolved, qg);
      }
      __syncwarp();
    }
    for (int j = lane; j < a.k; j += 32) {
      const bool have = j < nc;
      a.out_ids[qg * a.k + j] = have ? int32_t(unsigned(b[j])) : -1;
      if (a.out_dists) {
        const unsigned kb = unsigned(b[j] >> 32);
        a.out_dists[qg * a.k + j] = !have ? __int_as_float(0x7f800000) : (DT == kU8 ? float(kb) : __uint_as_float(kb));
      }
    }
  }
}

// ---------------------------------------------------------------------------
// tensor-core path: exact kNN with an f16 Gram filter
// ---------------------------------------------------------------------------
// Points and queries are packed once as f16 rows in tiles of 128 rows, each
// tile already in the core-matrix order of the tcgen05 operand layout: uint8
// values as they are (exact), float rows scaled by a power of two so that
// |x| <= 1 and split into two f16 operands, hi = f16(x) and lo =
// f16(2^11 (x - hi)), the tile holding hi then lo.  The split keeps the Gram
// error near 2^-22 |q||p| instead of f16's 2^-11, so the candidate window stays
// narrow on data whose neighbours lie close together.
//
// Scan (knn_scan_kernel): a step is one query tile against one point tile, D =
// Q P^T on tcgen05 (float rows: hi hi^T in one accumulator, hi lo^T + lo hi^T in
// a second, G~ = the first + 2^-11 the second).  The steps of a chunk of query
// tiles, in order, are cut evenly over the CTAs, so that 79 query tiles (10,000
// queries) keep every SM busy; a query tile's points are then scanned in a few
// parts by neighbouring CTAs.  One warp copies the tiles in (bulk copies, two or
// three in flight) and issues the MMAs one step ahead of the eight warps that
// read the accumulators: two threads per query (TMEM lane), half the columns each.
//
// From G~ a thread forms d2~ = |q|^2 + |p|^2 - 2 G~ (scaled units) and a rigorous
// error bound err (zero for uint8 rows of d <= 128, where every quantity is an
// exact integer below 2^24).  Point p is kept as a candidate, as {d2~, id}, when
// its lower bound may be at most tau, an upper bound of the k-th smallest
// distance met so far by any part of the query (the k-th smallest d2~ of a part
// plus the largest err of any point): at least k points have d2 <= tau, so every
// true k nearest neighbour passes when it is met (tau only decreases).  Eight
// columns at a time are tested branch-free (the sign of d2~ - threshold, shifted
// into a mask), and the few that pass are stored by predicated instructions, if
// any lane has one.  A query's candidates live in a global buffer per part, one
// thread's from its start up, the other's from its end down; when it gets long, a
// warp selects the k-th, lowers tau and drops the candidates above it.
//
// err grows with the square of p's norm, so that the largest err of all points says
// nothing about most of them once one has a large norm.  The test therefore takes
// each point's own, as a linear function of its squared norm (tc_err_linear: one
// multiply-add in place of an add).  A cut, and the ranking, take the largest while
// it is narrow against tau or leaves few; else every entry's own (from its norm):
// tau is then the k-th smallest d2~ + err, and an entry stays if its d2~ - err is
// not above it.
//
// Rank (knn_rank_kernel), one warp per query: the candidates of its parts are
// cut to the final tau and ranked by their exact keys (uint8: exact integers;
// float: sums per 32-dim slice with near-tie runs re-ordered in binary64), as
// the CUDA-core kernel ranks its lists.
//
// Redo (knn_redo_kernel): a part that met more than kTcCand - kTcP equal or nearly
// equal distances before any other part had a better tau has no room left, though
// the query as a whole has better points and needs few of them (a block of repeated
// rows does that).  Such a query is marked, not ranked, and scanned again: one CTA
// per query tile takes all points in order as one part, from the tau that the first
// scan came to, with exact cuts, and ranks the marked queries.  A query is refused
// only if that runs out of room.  With nothing marked, as good as always, it costs its
// launch.
//
// What bounds the scan: the threads' 64 columns a step, read, tested and now and
// then stored, about 2,400 of a step's 4,000 cycles (its products: 1,150 at d = 96),
// and the cuts, which hold the other warps up through the accumulators.  10,000
// queries x 400,000 points x 96 dims, k 100: 3.6 ms, of which the ranking 0.34; one
// CTA per query tile, a lane per query row and the tile's loads, products and cuts
// in turn took 47.6 (79 CTAs of 152, the tensor cores idle through every cut).  With
// the exact k-th in a cut, its entries read twice, and a vote per eight columns it
// took 5.4.  All 64 columns read at once, for one wait less, changed nothing.
constexpr int kTcQ = 128;     // queries per tile (rows of the MMA)
constexpr int kTcP = 128;     // points per tile (columns of the MMA)
constexpr int kTcCand = 512;  // candidates a part keeps per query
// A part's candidates are cut when they pass kTcCut (or what a cut left plus 96):
// more candidates pass an old tau than a cut costs.  A tile adds at most kTcP.
constexpr int kTcCut = 224;
constexpr int kTcThreads = 288;
constexpr int kTcNorms = 8;   // point-norm rows in shared memory
constexpr int kTcMinSteps = 8;  // a CTA takes at least this many point tiles (if there are as many)
constexpr int kRankCand = 1024;

struct KnnTcArgs {
  const uint8_t* X;          // raw rows (exact ranking)
  int64_t row_bytes;
  int64_t n;
  int d;
  const uint8_t* Qraw;       // raw query rows, or nullptr: queries are base points
  int64_t nq;
  int k;
  const uint8_t* qtiles;     // packed query tiles (the point tiles for base-point queries)
  const uint8_t* ptiles;     // packed point tiles
  int64_t tile_bytes;        // kTcP * dpad * 2 per operand: uint8 one (f16), float two (hi, lo)
  int ksteps;                // dpad / 16
  int nbuf;                  // point tiles in shared memory, 2 or 3
  const float* qnorm;        // |q'|^2 per query (scaled)
  const float* pnorm;        // |p'|^2 per point, padded to whole tiles with 0
  const float2* tmax;        // (max |p'|^2, max |p'|) over all points
  int exact;                 // 1: G~ and d2~ are exact
  float eps_ip, eps_n, sub_abs;  // sub_abs: the subnormal-rounding term per unit of |q| + |p|
  // this chunk: query tiles qt0 .. qt0 + nqt - 1, `per` steps per CTA.  The part
  // of CTA c on the chunk's query tile t is part c + t: each is met once, since
  // from one part to the next c or t or both grow.
  int64_t qt0, nqt, per;
  int kscan;                 // k, one more for base points, whose own row is met too
  uint2* cand;               // [part][query][kTcCand] {d2~, id}
  int* pcnt;                 // [part][query] candidates (from the start, << 16 from the end), zeroed: none
                             // of a part that could not finish
  unsigned* tauq;            // [chunk query] tau as an ordered key (fkey), lowered by every part
  int* marked;               // [chunk query] not 0: to be scanned again (zeroed before the scan)
  int32_t* out_ids;
  float* out_dists;
  DevStatus* status;
};

// Total order on floats as unsigned keys (negatives included).
__device__ __forceinline__ unsigned fkey(float f) {
  const unsigned b = __float_as_uint(f);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float fkey_inv(unsigned k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

// Bound on |d2~ - d2'| for one (query, point) pair in scaled units: twice the
// Gram error (eps_ip |q'||p'| plus the subnormal roundings, sub_abs (|q'| +
// |p'|) in all), the single-precision norms, and the roundings that form d2~
// and its two bounds (2^-21 (|q'|^2 + |p'|^2) covers them).
__device__ __forceinline__ float tc_err(const KnnTcArgs& a, float nq, float sq, float np, float sp) {
  return (2.f * a.eps_ip * sq * sp * 1.001f + a.sub_abs * (sq + sp) + (a.eps_n + 4.7683716e-07f) * (nq + np)) *
             1.0001f +
         1e-30f;
}

// tc_err as linear in np, for the scan's test: err <= (1 - f) np + c, since
// 2 sq sp <= nq + np and 2 sp <= np / s + s for any s > 0: sq, or 2^-20 for queries
// so small that sub_abs / sq would count.  Both also carry 2^-21 of nq and np for the
// roundings of the test.
__device__ __forceinline__ void tc_err_linear(const KnnTcArgs& a, float nq, float& f, float& c) {
  const float sq = sqrtf(nq), s = fmaxf(sq, 9.5367432e-07f);
  const float g = a.eps_ip * 1.001f + a.eps_n + 9.5367432e-07f;
  f = 1.f - (g + 0.5f * a.sub_abs / s) * 1.0002f;
  c = (g * nq + a.sub_abs * (sq + 0.5f * s)) * 1.0002f + 2e-30f;
}

// tc_err of point id (its norm read from global memory).
__device__ __forceinline__ float own_err(const KnnTcArgs& a, float nq, float sq, unsigned id) {
  const float np = __ldg(a.pnorm + id);
  return tc_err(a, nq, sq, np, sqrtf(np));
}

// Operands per tile: uint8 rows one f16 operand, float rows two (hi, lo).
__host__ __device__ constexpr int tc_nop(int dtype) { return dtype == kF32 ? 2 : 1; }

// Entry i of a buffer that holds `a` entries from its start and the rest from
// `gap` places on: gap = 0 for a plain list.
__device__ __forceinline__ int entry_at(int i, int a, int gap) { return i < a ? i : i + gap; }

// The k-th smallest value(entry) of the m >= k entries as a key, by bisection on
// its bits; the entries are read once, PER of them per lane.  One warp.
template <int PER, typename F>
__device__ __forceinline__ unsigned kth_of(const uint2* e, int m, int k, F value) {
  const int lane = threadIdx.x & 31;
  unsigned u[PER];
#pragma unroll
  for (int i = 0; i < PER; ++i) u[i] = 32 * i + lane < m ? fkey(value(e[32 * i + lane])) : 0xffffffffu;
  unsigned lo = 0xffffffffu, hi = 0;
#pragma unroll
  for (int i = 0; i < PER; ++i) {
    lo = min(lo, u[i]);
    if (32 * i + lane < m) hi = max(hi, u[i]);
  }
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  while (lo < hi) {  // the k-th smallest lies in [lo, hi]
    const unsigned mid = lo + (hi - lo) / 2;
    int c = 0;
#pragma unroll
    for (int i = 0; i < PER; ++i) c += u[i] <= mid;
    if (__reduce_add_sync(0xffffffffu, c) >= k) hi = mid;
    else lo = mid + 1;
  }
  return lo;
}

// An error bound as what is added to or taken from a d2~: e with the roundings of
// that sum.
__device__ __forceinline__ float cut_width(float e, float norms) { return e * 1.0001f + 4.7683716e-07f * norms; }

// Drops the entries whose lower bound, lower(entry), lies above tau and moves the
// rest to the start; returns how many are left.  One warp.
template <typename F>
__device__ __forceinline__ int cut_above(uint2* e, int m, float tau, F lower) {
  const int lane = threadIdx.x & 31;
  int kept = 0;
  for (int i0 = 0; i0 < m; i0 += 32) {
    const int i = i0 + lane;
    uint2 v = make_uint2(0, 0);
    if (i < m) v = e[i];  // never before the place it may be moved to
    const bool keep = i < m && lower(v) <= tau;
    const unsigned km = __ballot_sync(0xffffffffu, keep);
    __syncwarp();
    if (keep) e[kept + __popc(km & ((1u << lane) - 1))] = v;
    kept += __popc(km);
    __syncwarp();
  }
  return kept;
}

// A key that at least k of a warp's m entries do not exceed: the k-th smallest,
// or one that k to k + slack entries do not exceed.  u: the entries' keys, PER per
// lane, all ones past m.
template <int PER>
__device__ __forceinline__ unsigned kth_key(const unsigned (&u)[PER], int m, int k, int slack) {
  const int lane = threadIdx.x & 31;
  unsigned lo = 0xffffffffu, hi = 0;
#pragma unroll
  for (int i = 0; i < PER; ++i) {
    lo = min(lo, u[i]);
    if (32 * i + lane < m) hi = max(hi, u[i]);
  }
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  while (lo < hi) {  // the k-th smallest lies in [lo, hi]
    const unsigned mid = lo + (hi - lo) / 2;
    int c = 0;
#pragma unroll
    for (int i = 0; i < PER; ++i) c += u[i] <= mid;
    c = __reduce_add_sync(0xffffffffu, c);
    if (c >= k) hi = mid;
    else lo = mid + 1;
    if (c >= k && c <= k + slack) break;
  }
  return hi;
}

// The cut of a part by every entry's own bound: tau = the k-th smallest d2~ + err of
// the m entries (the first n0 from the start of e, the rest `gap` places on), those
// with d2~ - err above it dropped and the others moved to the start; returns how many.
// Out of line, since it is rare and a small call's scan runs cold (inlined, 4 us more).
// One warp.
__device__ __noinline__ int cut_own(const KnnTcArgs& a, uint2* e, int m, int k, float nq, int n0, int gap, float& tau) {
  const int lane = threadIdx.x & 31;
  const float sq = sqrtf(nq);
  auto err = [&](uint2 v) { return own_err(a, nq, sq, v.y); };
  unsigned u[kTcCand / 32];
#pragma unroll
  for (int i = 0; i < kTcCand / 32; ++i) {
    u[i] = 0xffffffffu;
    if (32 * i + lane < m) {
      const uint2 v = e[entry_at(32 * i + lane, n0, gap)];
      u[i] = fkey(__uint_as_float(v.x) + err(v));
    }
  }
  tau = fkey_inv(kth_key<kTcCand / 32>(u, m, k, 0));
  int kept = 0;
  for (int i0 = 0; i0 < m; i0 += 32) {
    const int i = i0 + lane;
    uint2 v = make_uint2(0, 0);
    if (i < m) v = e[entry_at(i, n0, gap)];  // never before the place it may be moved to
    const bool keep = i < m && __uint_as_float(v.x) - err(v) <= tau;
    const unsigned km = __ballot_sync(0xffffffffu, keep);
    __syncwarp();
    if (keep) e[kept + __popc(km & ((1u << lane) - 1))] = v;
    kept += __popc(km);
    __syncwarp();
  }
  return kept;
}

// A part's m >= k candidates (`n0` of them at the buffer's start, the rest up to its
// end), PER per lane, read once: tau = an upper bound of the k-th smallest d2~, plus
// w; the entries whose lower bound lies above it are dropped and the rest moved to
// the start.  Returns how many are left.  The bisection stops at a value that k to
// k + kCutSlack entries do not exceed, after 5 or 6 of its 25 steps; the few more
// that stay cost less.  If w is wide and leaves more than k + kOwnSlack, every entry's
// own bound takes its place (nq: the query's squared norm).  One warp.
constexpr int kCutSlack = 8;
constexpr int kOwnSlack = 64;
constexpr float kNarrow = 0.0009765625f;  // a bound below this part of tau is not looked into
template <int DT, int PER, bool REDO>
__device__ __forceinline__ int cut_part(const KnnTcArgs& a, uint2* e, int m, float w, float nq, int n0, float& tau) {
  const int lane = threadIdx.x & 31;
  const int gap = kTcCand - m, k = a.kscan;
  unsigned u[PER], id[PER];
#pragma unroll
  for (int i = 0; i < PER; ++i) {
    const uint2 v = 32 * i + lane < m ? e[entry_at(32 * i + lane, n0, gap)] : make_uint2(0x7fffffffu, 0);
    u[i] = fkey(__uint_as_float(v.x));  // past m: above every distance
    id[i] = v.y;
  }
  tau = fkey_inv(kth_key<PER>(u, m, k, REDO ? 0 : kCutSlack)) + w;
  if (DT == kF32 && (REDO || w > kNarrow * tau)) {
    int c = 0;
#pragma unroll
    for (int i = 0; i < PER; ++i) c += 32 * i + lane < m && fkey_inv(u[i]) - w <= tau;
    if (__reduce_add_sync(0xffffffffu, c) > k + kOwnSlack) return cut_own(a, e, m, k, nq, n0, gap, tau);
  }
  int kept = 0;
  __syncwarp();  // every entry has been read
#pragma unroll
  for (int i = 0; i < PER; ++i) {
    const float x = fkey_inv(u[i]);
    const bool keep = 32 * i + lane < m && x - w <= tau;
    const unsigned km = __ballot_sync(0xffffffffu, keep);
    if (keep) e[kept + __popc(km & ((1u << lane) - 1))] = make_uint2(__float_as_uint(x), id[i]);
    kept += __popc(km);
  }
  return kept;
}

// *at = {x, y} and at += step bytes if `yes`, by predicated instructions: a branch per column costs
// more than the stores it skips.
__device__ __forceinline__ void push_if(unsigned yes, uint2*& at, long long step, unsigned x, unsigned y) {
  unsigned long long p = reinterpret_cast<unsigned long long>(at);
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.u32 p, %1, 0;\n@p st.global.v2.u32 [%0], {%2, %3};\n@p add.s64 %0, %0, %4;\n}\n"
      : "+l"(p)
      : "r"(yes), "r"(x), "r"(y), "l"(step)
      : "memory");
  at = reinterpret_cast<uint2*>(p);
}

// A query tile, the point tiles, their norms, the barriers.  uint8: at least a
// third of an SM's shared memory, so that at most two CTAs (each holding 256 of
// the SM's 512 TMEM columns) share an SM; float: more than half, one CTA holding
// all 512 (two sets of two accumulators).
size_t knn_tc_smem(int dtype, int64_t tile_bytes, int nbuf) {
  const size_t need = size_t(tile_bytes) * size_t(1 + nbuf) + kTcNorms * kTcP * 4 + 256 + 3 * kTcQ * 4;
  return std::max(need, dtype == kF32 ? size_t(228 * 1024 / 2 + 1024) : size_t(228 * 1024 / 3 + 1024));
}

// The steps of one CTA.  REDO: of the marked queries only, its query tile's points as one part.
template <int DT, bool REDO>
__device__ __forceinline__ void scan_steps(const KnnTcArgs& a, unsigned char* smem_raw) {
  // float rows: hi and lo operands, two accumulators per set (acc0 at column
  // 0 of the set, acc1 at 128)
  constexpr bool kSplit = DT == kF32;
  constexpr uint32_t kSetCols = kSplit ? 256u : 128u;
  constexpr int kWait = 1 << 20;
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  unsigned char* sA = smem_raw;
  unsigned char* sB = smem_raw + a.tile_bytes;
  float* sPn = reinterpret_cast<float*>(smem_raw + (1 + a.nbuf) * a.tile_bytes);  // [kTcNorms][kTcP]
  uint64_t* bars = reinterpret_cast<uint64_t*>(sPn + kTcNorms * kTcP);
  uint64_t* full = bars;           // [3] point tile landed
  uint64_t* afull = bars + 3;      // query tile landed
  uint64_t* mma_done = bars + 4;   // [2] accumulator set written
  uint64_t* acc_free = bars + 6;   // [2] accumulator set read (8 warps)
  uint64_t* nfull = bars + 8;      // [kTcNorms] point norms landed
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 8 + kTcNorms);
  int* sCnt = reinterpret_cast<int*>(bars + 32);               // [2][kTcQ] candidates, by half
  float* sTau = reinterpret_cast<float*>(sCnt + 2 * kTcQ);     // [kTcQ] tau after a cut
  const int64_t npt = (a.n + kTcP - 1) / kTcP;
  const int64_t s0 = int64_t(blockIdx.x) * a.per;
  const int64_t total = a.nqt * npt;
  const int64_t s1 = s0 + a.per < total ? s0 + a.per : total;
  const int steps = int(s1 > s0 ? s1 - s0 : 0);
  const int q_first = int(s0 / npt), j_first = int(s0 - q_first * npt), ntile = int(npt);

  if (warp == 0) tmem_alloc(tmem_slot, 2 * kSetCols);  // two accumulator sets
  if (t == 0) {
    for (int i = 0; i < 4; ++i) mbar_init(&full[i], 1);  // full[0..2], afull
    for (int i = 0; i < 2; ++i) mbar_init(&mma_done[i], 1);
    for (int i = 0; i < 2; ++i) mbar_init(&acc_free[i], 8);
    for (int i = 0; i < kTcNorms; ++i) mbar_init(&nfull[i], 1);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 8) {
    // ---------------- copies and MMAs, one lane ----------------
    if (lane == 0 && steps > 0) {
      constexpr uint32_t idesc = umma_idesc_f16(128, 128);
      constexpr uint32_t lbo = 16u * 128u;  // 16 row-groups of 128 bytes per k-chunk
      const uint32_t lo_off = uint32_t(a.tile_bytes / 2);  // float tiles: lo after hi
      // A point tile goes into buffer (step % nbuf) once the MMA of the step
      // that used it is done, its norms into row (step % kTcNorms): step s is
      // loaded after the MMA of step s - 2 was issued, which waited until the
      // accumulators of step s - 4 were read; whoever has read those is done with
      // the norms of every step before, s - kTcNorms among them.
      int loaded = 0, lj = j_first, lb = 0;
      auto load_point_tile = [&]() {  // step `loaded` of this CTA
        const int nb = loaded % kTcNorms;
        mbar_expect(&full[lb], uint32_t(a.tile_bytes));
        bulk_load(sB + lb * a.tile_bytes, a.ptiles + lj * a.tile_bytes, uint32_t(a.tile_bytes), &full[lb]);
        mbar_expect(&nfull[nb], kTcP * 4u);
        bulk_load(sPn + nb * kTcP, a.pnorm + int64_t(lj) * kTcP, kTcP * 4u, &nfull[nb]);
        ++loaded;
        if (++lj == ntile) lj = 0;
        if (++lb == a.nbuf) lb = 0;
      };
      for (int i = 0; i < a.nbuf - 1 && loaded < steps; ++i) load_point_tile();
      bool ok = true;
      uint32_t aphase = 0, pphase = 0;
      int q = q_first, j = j_first, pb = 0;
      for (int it = 0; it < steps && ok; ++it) {
        const int b = it & 1;
        if (it == 0 || j == 0) {  // the next query tile, once the last MMA has read the old one
          if (it > 0) ok = mbar_wait(&mma_done[b ^ 1], uint32_t((it - 1) >> 1) & 1u, kWait);
          if (!ok) break;
          mbar_expect(afull, uint32_t(a.tile_bytes));
          bulk_load(sA, a.qtiles + (a.qt0 + q) * a.tile_bytes, uint32_t(a.tile_bytes), afull);
          ok = mbar_wait(afull, aphase, kWait);
          aphase ^= 1u;
          if (!ok) break;
        }
        ok = mbar_wait(&full[pb], pphase, kWait);
        if (ok && it >= 2) ok = mbar_wait(&acc_free[b], uint32_t((it >> 1) - 1) & 1u, kWait);
        if (!ok) break;
        tc_fence_after();
        const uint32_t acc = tmem + uint32_t(b) * kSetCols;
        const unsigned char* B = sB + pb * a.tile_bytes;
        for (int kk = 0; kk < a.ksteps; ++kk) {
          const uint64_t da = umma_desc(smem_addr(sA) + uint32_t(kk) * 2u * lbo, lbo, 128u);
          const uint64_t db = umma_desc(smem_addr(B) + uint32_t(kk) * 2u * lbo, lbo, 128u);
          umma_f16(acc, da, db, idesc, kk > 0);
          if constexpr (kSplit) {  // the cross terms with the low halves
            const uint64_t dal = umma_desc(smem_addr(sA) + lo_off + uint32_t(kk) * 2u * lbo, lbo, 128u);
            const uint64_t dbl = umma_desc(smem_addr(B) + lo_off + uint32_t(kk) * 2u * lbo, lbo, 128u);
            umma_f16(acc + 128u, da, dbl, idesc, kk > 0);
            umma_f16(acc + 128u, dal, db, idesc, true);
          }
        }
        umma_commit(&mma_done[b]);
        if (loaded < steps) {  // into the buffer that step it - 1 has read
          if (it > 0) ok = mbar_wait(&mma_done[b ^ 1], uint32_t((it - 1) >> 1) & 1u, kWait);
          if (ok) load_point_tile();
        }
        if (++j == ntile) {
          j = 0;
          ++q;
        }
        if (++pb == a.nbuf) {
          pb = 0;
          pphase ^= 1u;
        }
      }
      if (!ok) {  // a wait ran out: report, let the copies in flight land, stop
        raise_status(a.status, kDevOverflow, -3);
        for (int s = loaded > a.nbuf ? loaded - a.nbuf : 0; s < loaded; ++s) {
          mbar_wait(&full[s % a.nbuf], uint32_t(s / a.nbuf) & 1u, kWait);
          mbar_wait(&nfull[s % kTcNorms], uint32_t(s / kTcNorms) & 1u, kWait);
        }
      }
    }
  } else {
    // ---------------- candidates: threads tl and 128 + tl, query tl of the tile ----------------
    const int tl = t & (kTcQ - 1), half = t >> 7, quad = warp & 3;
    const long long dir = half ? -8 : 8;
    const float inf = __int_as_float(0x7f800000);
    float tau = inf, nqq = 0.f, width = 0.f, lin_f = 1.f, lin_c = 0.f;  // width: cut_width of any point
    int cnt = 0, limit = kTcCut;
    int q = q_first, j = j_first;
    int64_t qi = 0;
    bool qlive = false;
    uint2 *cbuf = nullptr, *cnext = nullptr;
    unsigned* tq = nullptr;
    bool ok = true;
    float shared_tau = inf;  // of the query's other parts, loaded a step ahead
    const float2 tm = *a.tmax;
    // A warp whose wait runs out takes no more candidates, but stays with its
    // partner's barriers to the end.
    for (int it = 0; it < steps; ++it) {
      const int b = it & 1;
      if (it == 0 || j == 0) {  // a new part
        qi = (a.qt0 + q) * kTcQ + tl;
        qlive = qi < a.nq && (!REDO || a.marked[q * kTcQ + tl] != 0);
        nqq = qlive ? a.qnorm[qi] : 0.f;
        if constexpr (kSplit) {
          tc_err_linear(a, nqq, lin_f, lin_c);
          width = cut_width(tc_err(a, nqq, sqrtf(nqq), tm.x, tm.y), nqq + tm.x);
        }
        cbuf = a.cand + (int64_t(blockIdx.x + q) * kTcQ + tl) * kTcCand;
        tq = a.tauq + int64_t(q) * kTcQ + tl;
        if (half) cbuf += kTcCand - 1;  // this thread's own start
        cnext = cbuf;
        cnt = 0;
        limit = kTcCut;
        tau = inf;
        shared_tau = fkey_inv(__ldcg(tq));
      }
      // tau as lowered meanwhile by the query's other parts (any value that was
      // ever there is a valid one; not a number: none yet)
      tau = fminf(tau, shared_tau);
      // passes: |q'|^2 + f |p'|^2 - 2 G~ below thr
      const float thr = kSplit ? tau * 1.000001f + lin_c : tau + 1.f;  // integers: d2 <= tau as d2 - (tau + 1) < 0
      const bool tail = int64_t(j + 1) * kTcP > a.n;
      const float base = nqq - thr;
      const float* pnb = sPn + (it % kTcNorms) * kTcP;
      ok = ok && mbar_wait(&nfull[it % kTcNorms], uint32_t(it / kTcNorms) & 1u, kWait);
      ok = ok && mbar_wait(&mma_done[b], uint32_t(it >> 1) & 1u, kWait);
      ok = __all_sync(0xffffffffu, ok);
      tc_fence_after();
      shared_tau = fkey_inv(__ldcg(tq));
      const int64_t p0 = int64_t(j) * kTcP;
#pragma unroll 1
      for (int c0 = half * (kTcP / 2); ok && c0 < (half + 1) * (kTcP / 2); c0 += 32) {
        uint32_t v[32], v2[kSplit ? 32 : 1];
        const uint32_t acc = tmem + (uint32_t(32 * quad) << 16) + uint32_t(b) * kSetCols + uint32_t(c0);
        tmem_ld32(acc, v);
        if constexpr (kSplit) tmem_ld32(acc + 128u, *reinterpret_cast<uint32_t(*)[32]>(v2));
        tmem_ld_wait();
        if (c0 + 32 == (half + 1) * (kTcP / 2)) {  // the last read of this set
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&acc_free[b]);
        }
        // float rows: hi hi^T + 2^-11 (hi lo^T + lo hi^T), scaled units
        if constexpr (kSplit) {
#pragma unroll
          for (int jj = 0; jj < 32; ++jj)
            v[jj] = __float_as_uint(fmaf(__uint_as_float(v2[jj]), 4.8828125e-04f, __uint_as_float(v[jj])));
        }
        unsigned m = 0;  // bit e: column c0 + e
#pragma unroll
        for (int g = 0; g < 32; g += 8) {
          const float4 pa = *reinterpret_cast<const float4*>(pnb + c0 + g);
          const float4 pb = *reinterpret_cast<const float4*>(pnb + c0 + g + 4);
          const float pn[8] = {pa.x, pa.y, pa.z, pa.w, pb.x, pb.y, pb.z, pb.w};
          unsigned mg = 0;
#pragma unroll
          for (int e = 7; e >= 0; --e)
            mg = __funnelshift_l(__float_as_uint(fmaf(-2.f, __uint_as_float(v[g + e]),
                                                      kSplit ? fmaf(pn[e], lin_f, base) : base + pn[e])), mg, 1);
          m |= mg << g;
        }
        if (!qlive) m = 0;
        if (tail) {  // the last tile: columns past n
          const int64_t left = a.n - (p0 + c0);
          m &= left >= 32 ? 0xffffffffu : left > 0 ? (1u << int(left)) - 1u : 0u;
        }
        const unsigned any = __reduce_or_sync(0xffffffffu, m);
        if (any == 0) continue;
#pragma unroll
        for (int g = 0; g < 32; g += 4) {
          if (((any >> g) & 0xfu) == 0) continue;
          const float4 pa = *reinterpret_cast<const float4*>(pnb + c0 + g);
          const float pn[4] = {pa.x, pa.y, pa.z, pa.w};
          const unsigned id0 = unsigned(p0) + unsigned(c0 + g);
#pragma unroll
          for (int e = 0; e < 4; ++e)  // at most kTcP more a tile: the buffer has room
            push_if((m >> (g + e)) & 1u, cnext, dir, __float_as_uint(fmaf(-2.f, __uint_as_float(v[g + e]), nqq + pn[e])),
                    id0 + unsigned(e));
        }
      }
      // ---- both threads of a query know its length
      cnt = half ? int(cbuf - cnext) : int(cnext - cbuf);
      sCnt[half * kTcQ + tl] = cnt;
      named_sync(1 + quad, 64);  // and what either has stored
      const int other = sCnt[(half ^ 1) * kTcQ + tl];
      // ---- long buffers: lower tau, drop what lies above it; every other one of
      // the quadrant's by either warp
      const unsigned need = __ballot_sync(0xffffffffu, cnt + other > limit);
      if (need) {  // the same in both warps
        named_sync(1 + quad, 64);  // sCnt read
        int nth = 0;
        for (unsigned todo = need; todo; todo &= todo - 1, ++nth) {
          if ((nth & 1) != half) continue;
          const int L = __ffs(int(todo)) - 1;
          const int own = __shfl_sync(0xffffffffu, cnt, L), oth = __shfl_sync(0xffffffffu, other, L);
          const float wL = __shfl_sync(0xffffffffu, width, L), nL = __shfl_sync(0xffffffffu, nqq, L);
          const int nA = half ? oth : own, cL = own + oth, ql = quad * 32 + L;
          uint2* bL = a.cand + (int64_t(blockIdx.x + q) * kTcQ + ql) * kTcCand;
          // cL > kTcCut >= kscan
          float tnew;
          const int w = cL <= 256 ? cut_part<DT, 8, REDO>(a, bL, cL, wL, nL, nA, tnew)
                                  : cut_part<DT, kTcCand / 32, REDO>(a, bL, cL, wL, nL, nA, tnew);
          if (lane == 0) {
            sCnt[ql] = w;
            sTau[ql] = tnew;
            atomicMin(a.tauq + int64_t(q) * kTcQ + ql, fkey(tnew));
            if (w > kTcCand - kTcP) {
              if (REDO) raise_status(a.status, kDevOverflow, (a.qt0 + q) * kTcQ + ql);
              else a.marked[q * kTcQ + ql] = 1;
            }
          }
          __syncwarp();
        }
        named_sync(1 + quad, 64);
        if ((need >> lane) & 1u) {
          const int w = sCnt[tl];
          cnt = half ? 0 : w;
          cnext = half ? cbuf : cbuf + w;
          tau = fminf(tau, sTau[tl]);
          limit = min(max(kTcCut, w + 96), kTcCand - kTcP);
          if (w > kTcCand - kTcP) qlive = false;  // no room for the next tile: marked or reported, take no more
        }
      }
      if (it + 1 == steps || j + 1 == ntile) {
        // the part's candidates; `other` as it stands after a cut
        const int second = half ? cnt : (need >> lane) & 1u ? 0 : other;
        if (!half) a.pcnt[int64_t(blockIdx.x + q) * kTcQ + tl] = cnt | (second << 16);
      }
      named_sync(1 + quad, 64);  // sCnt and sTau read before the next step writes them
      if (++j == ntile) {
        j = 0;
        ++q;
      }
    }
    if (!ok && lane == 0) raise_status(a.status, kDevOverflow, -4);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0) tmem_dealloc(tmem, 2 * kSetCols);
}

// Query ql of the chunk, by one warp with kRankCand entries of shared memory at e.
template <int DT, bool REDO>
__device__ __forceinline__ void rank_query(const KnnTcArgs& a, int64_t ql, uint2* e) {
  const int lane = threadIdx.x & 31;
  const int64_t qg = a.qt0 * kTcQ + ql;
  const int64_t npt = (a.n + kTcP - 1) / kTcP, qt = ql / kTcQ;
  const int t = int(ql % kTcQ);
  const float inf = __int_as_float(0x7f800000);
  float tau = fminf(inf, fkey_inv(__ldcg(a.tauq + ql)));  // never lowered: all ones, not a number
  float w = 0.f, nqq = 0.f;
  if (!a.exact) {
    nqq = a.qnorm[qg];
    const float2 tm = *a.tmax;
    w = cut_width(tc_err(a, nqq, sqrtf(nqq), tm.x, tm.y), nqq + tm.x);
  }
  // ---- the candidates of the query's parts, cut to the smallest tau
  int m = 0;
  bool over = false;
  auto lower = [&]() {  // tau from what is held
    if (m < a.k) return;
    const float tnew =
        fkey_inv(kth_of<kRankCand / 32>(e, m, a.k, [](uint2 v) { return __uint_as_float(v.x); })) + w;
    tau = fminf(tau, tnew);
    m = cut_above(e, m, tau, [&](uint2 v) { return __uint_as_float(v.x) - w; });
    if constexpr (DT == kF32) {
      if (!REDO && m <= a.k + kOwnSlack) return;
      const float sq = sqrtf(nqq);
      const float own = fkey_inv(kth_of<kRankCand / 32>(
          e, m, a.k, [&](uint2 v) { return __uint_as_float(v.x) + own_err(a, nqq, sq, v.y); }));
      tau = fminf(tau, own);
      m = cut_above(e, m, tau, [&](uint2 v) { return __uint_as_float(v.x) - own_err(a, nqq, sq, v.y); });
    }
  };
  const int64_t c1 = ((qt + 1) * npt - 1) / a.per;
  for (int64_t c = qt * npt / a.per; c <= c1; ++c) {
    const int64_t part = (c + qt) * kTcQ + t;
    const int nA = a.pcnt[part] & 0xffff, cn = nA + (a.pcnt[part] >> 16), gap = kTcCand - cn;
    const uint2* src = a.cand + part * kTcCand;
    for (int i0 = 0; i0 < cn; i0 += 32) {
      if (m > kRankCand - 32) {
        __syncwarp();
        lower();
        if (m > kRankCand - 32) {
          over = true;
          break;
        }
      }
      const int i = i0 + lane;
      uint2 v = make_uint2(0, 0);
      if (i < cn) v = src[entry_at(i, nA, gap)];
      const bool self = !a.Qraw && int64_t(v.y) == qg;
      const bool keep = i < cn && !self && __uint_as_float(v.x) - w <= tau;
      const unsigned km = __ballot_sync(0xffffffffu, keep);
      if (keep) e[m + __popc(km & ((1u << lane) - 1))] = v;
      m += __popc(km);
      __syncwarp();
    }
  }
  if (!REDO && over) {
    if (lane == 0) a.marked[ql] = 1;
    return;
  }
  lower();
  // ---- exact keys: four lanes per row
  unsigned long long* keys = reinterpret_cast<unsigned long long*>(e);
  const uint8_t* qrow = a.Qraw ? a.Qraw + qg * a.row_bytes : a.X + qg * a.row_bytes;
  const int ns = int(a.row_bytes / 128);  // at most four slices of 128 bytes
  const int sub = lane & 3;
  for (int i0 = 0; i0 < m; i0 += 8) {
    const int i = i0 + (lane >> 2);
    const unsigned id = e[i < m ? i : m - 1].y;
    const uint4* x = reinterpret_cast<const uint4*>(qrow);
    const uint4* y = reinterpret_cast<const uint4*>(a.X + int64_t(id) * a.row_bytes);
    unsigned key;
    if constexpr (DT == kU8) {
      unsigned part = 0;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const uint4 p = __ldg(x + sub + 4 * h), q = __ldg(y + sub + 4 * h);
        acc_pair<DT>(make_uint2(p.x, p.y), make_uint2(q.x, q.y), part);
        acc_pair<DT>(make_uint2(p.z, p.w), make_uint2(q.z, q.w), part);
      }
      part += __shfl_xor_sync(0xffffffffu, part, 1);
      part += __shfl_xor_sync(0xffffffffu, part, 2);
      key = part;
    } else {
      // a lane sums one slice in index order; the slice sums are added in order,
      // as the CUDA-core kernel does
      unsigned part = 0;
      if (sub < ns) {
        uint4 p[8], q[8];
#pragma unroll
        for (int h = 0; h < 8; ++h) {
          p[h] = __ldg(x + 8 * sub + h);
          q[h] = __ldg(y + 8 * sub + h);
        }
#pragma unroll
        for (int h = 0; h < 8; ++h) {
          acc_pair<DT>(make_uint2(p[h].x, p[h].y), make_uint2(q[h].x, q[h].y), part);
          acc_pair<DT>(make_uint2(p[h].z, p[h].w), make_uint2(q[h].z, q[h].w), part);
        }
      }
      float acc = 0.f;
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        const float ps = __uint_as_float(__shfl_sync(0xffffffffu, part, (lane & ~3) + s));
        if (s < ns) acc += ps;
      }
      key = __float_as_uint(acc);
    }
    __syncwarp();
    if (sub == 0 && i < m) keys[i] = (static_cast<unsigned long long>(key) << 32) | id;
    __syncwarp();
  }
  warp_sort(keys, m);
  const int nc = min(m, a.k);
  if constexpr (DT == kF32) {
    // near-tie runs are rare: one lane walks the list only if there is any
    const float E = slice_rel_bound(a.d), Eabs = abs_bound(a.d);
    bool near = false;
    for (int i = lane; i + 1 < m; i += 32)
      near |= !sure_less(__uint_as_float(unsigned(keys[i] >> 32)), __uint_as_float(unsigned(keys[i + 1] >> 32)), E, Eabs);
    if (__any_sync(0xffffffffu, near)) {
      if (lane == 0) fix_near_ties(a.X, a.row_bytes, a.d, a.status, keys, m, reinterpret_cast<const float*>(qrow), qg);
      __syncwarp();
    }
  }
  for (int j = lane; j < a.k; j += 32) {
    const bool have = j < nc;
    a.out_ids[qg * a.k + j] = have ? int32_t(unsigned(keys[j])) : -1;
    if (a.out_dists) {
      const unsigned kb = unsigned(keys[j] >> 32);
      a.out_dists[qg * a.k + j] = !have ? inf : (DT == kU8 ? float(kb) : __uint_as_float(kb));
    }
  }
}

// uint8 rows: registers for two CTAs on an SM, as its memory and TMEM allow (10,000
// queries x 400,000 points x 128, k 100: one CTA's 130 registers 3.7 ms, 96 3.4; 500
// queries x 200,000 x 96, k 10: 0.47 and 0.40).
template <int DT>
__global__ void __launch_bounds__(kTcThreads, DT == kU8 ? 2 : 1) knn_scan_kernel(KnnTcArgs a) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  scan_steps<DT, false>(a, smem_raw);
}

template <int DT>
__global__ void __launch_bounds__(128) knn_rank_kernel(KnnTcArgs a) {
  __shared__ uint2 sbuf[4][kRankCand];
  const int warp = threadIdx.x >> 5;
  const int64_t ql = int64_t(blockIdx.x) * 4 + warp;
  if (ql >= a.nqt * kTcQ || a.qt0 * kTcQ + ql >= a.nq || a.marked[ql] != 0) return;
  rank_query<DT, false>(a, ql, sbuf[warp]);
}

// The marked queries of query tile blockIdx.x of the chunk: a.per = all its points.
template <int DT>
__global__ void __launch_bounds__(kTcThreads, 1) knn_redo_kernel(KnnTcArgs a) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int64_t q0 = int64_t(blockIdx.x) * kTcQ;
  if (!__syncthreads_or(threadIdx.x < kTcQ && a.marked[q0 + threadIdx.x] != 0)) return;
  scan_steps<DT, true>(a, smem_raw);
  __syncthreads();  // the candidates; shared memory is free
  const int warp = threadIdx.x >> 5;
  for (int q = warp; warp < 8 && q < kTcQ; q += 8)  // a query past nq is never marked
    if (a.marked[q0 + q] != 0) rank_query<DT, true>(a, q0 + q, reinterpret_cast<uint2*>(smem_raw) + warp * kRankCand);
}
static_assert(8 * kRankCand * sizeof(uint2) <= 228 * 1024 / 3, "the redo's ranking fits in what every scan has");

// ---- packing: f16 operand tiles, scaled squared norms, their maximum

// max |x| over n rows of float data (bits of a non-negative float, atomicMax)
__global__ void maxabs_kernel(const uint8_t* __restrict__ X, int64_t row_bytes, int64_t n, int d,
                              unsigned* __restrict__ out) {
  float m = 0.f;
  const int64_t total = n * d;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < total; i += int64_t(gridDim.x) * blockDim.x) {
    const int64_t r = i / d, c = i % d;
    m = fmaxf(m, fabsf(reinterpret_cast<const float*>(X + r * row_bytes)[c]));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(out, __float_as_uint(m));
}

// Row i -> tile i / 128, row i % 128 of the core-matrix layout: uint8 values
// as f16 (exact); float rows scaled by s (a power of two: exact) and split
// into f16 hi and lo (split_f16x2), lo kTcP * dpad * 2 bytes after hi; the
// norm |x'|^2 in single precision in index order.
template <int DT>
__global__ void pack_f16_kernel(const uint8_t* __restrict__ X, int64_t row_bytes, int64_t n, int d, int dpad,
                                float s, uint8_t* __restrict__ tiles, float* __restrict__ norms) {
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  const int64_t ntile = (n + kTcP - 1) / kTcP;
  if (i >= ntile * kTcP) return;
  const int64_t tile = i / kTcP;
  const int r = int(i % kTcP);
  const int64_t op_bytes = int64_t(kTcP) * dpad * 2;
  uint8_t* tb = tiles + tile * op_bytes * tc_nop(DT);
  float acc = 0.f;
  const uint8_t* row = X + i * row_bytes;  // padded with zeros past d, and row_bytes covers dpad
  for (int kc = 0; kc < dpad / 8; ++kc) {
    float v[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (i < n) {
      if constexpr (DT == kU8) {
        const uint2 w = *reinterpret_cast<const uint2*>(row + kc * 8);
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = float(((e < 4 ? w.x : w.y) >> (8 * (e & 3))) & 0xffu);
      } else {
        const float4 p = *reinterpret_cast<const float4*>(row + kc * 32);
        const float4 q = *reinterpret_cast<const float4*>(row + kc * 32 + 16);
        const float x[8] = {p.x, p.y, p.z, p.w, q.x, q.y, q.z, q.w};
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = x[e] * s;
      }
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) acc = fmaf(v[e], v[e], acc);
    const int64_t at = (int64_t(kc) * 16 + r / 8) * 128 + (r % 8) * 16;
    if constexpr (DT == kF32) {
      uint4 hi, lo;
      split_f16x2(v[0], v[1], hi.x, lo.x);
      split_f16x2(v[2], v[3], hi.y, lo.y);
      split_f16x2(v[4], v[5], hi.z, lo.z);
      split_f16x2(v[6], v[7], hi.w, lo.w);
      *reinterpret_cast<uint4*>(tb + at) = hi;
      *reinterpret_cast<uint4*>(tb + op_bytes + at) = lo;
    } else {
      *reinterpret_cast<uint4*>(tb + at) = make_uint4(pack_f16x2(v[0], v[1]), pack_f16x2(v[2], v[3]),
                                                      pack_f16x2(v[4], v[5]), pack_f16x2(v[6], v[7]));
    }
  }
  norms[i] = acc;
}

// *out, zeroed before: (max |x'|^2, max |x'|), the latter rounded up
__global__ void norm_max_kernel(const float* __restrict__ norms, int64_t ntile, float2* __restrict__ out) {
  const int64_t tile = int64_t(blockIdx.x) * (blockDim.x / 32) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (tile >= ntile) return;
  float m = 0.f;
  for (int r = lane; r < kTcP; r += 32) m = fmaxf(m, norms[tile * kTcP + r]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) {
    unsigned* bits = reinterpret_cast<unsigned*>(out);  // of non-negative floats
    atomicMax(bits, __float_as_uint(m));
    atomicMax(bits + 1, __float_as_uint(sqrtf(m) * 1.000001f));
  }
}

}  // namespace

cudaError_t launch_knn(const KnnLaunch& K, cudaStream_t s) {
  KnnArgs a{};
  a.X = K.data.X;
  a.row_bytes = K.data.row_bytes;
  a.n = K.data.n;
  a.d = K.data.d;
  a.Q = K.Q;
  a.nq = K.nq;
  a.k = K.k;
  a.keep = K.data.dtype == kF32 ? K.k + 32 : K.k;
  a.out_ids = K.out_ids;
  a.out_dists = K.out_dists;
  a.status = K.status;
  if (a.keep > CAP - PB) return cudaErrorInvalidValue;
  const size_t bytes = sizeof(KnnSmem);
  cudaError_t err = cudaFuncSetAttribute(knn_kernel<kF32>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(bytes));
  if (err == cudaSuccess)
    err = cudaFuncSetAttribute(knn_kernel<kU8>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(bytes));
  if (err != cudaSuccess) return err;
  // launches of at most kChunk queries each, so that long scans proceed in bounded steps
  constexpr int64_t kChunk = 65536;
  for (int64_t c0 = 0; c0 < K.nq; c0 += kChunk) {
    a.q_base = c0;
    a.q_end = std::min(K.nq, c0 + kChunk);
    const unsigned grid = unsigned((a.q_end - c0 + QB - 1) / QB);
    if (K.data.dtype == kF32) knn_kernel<kF32><<<grid, kThreads, bytes, s>>>(a);
    else knn_kernel<kU8><<<grid, kThreads, bytes, s>>>(a);
    if ((err = cudaGetLastError()) != cudaSuccess) return err;
  }
  return cudaGetLastError();
}

cudaError_t launch_maxabs_f32(const uint8_t* X, int64_t row_bytes, int64_t n, int d, unsigned* out, cudaStream_t s) {
  if (n > 0) maxabs_kernel<<<1024, 256, 0, s>>>(X, row_bytes, n, d, out);
  return cudaGetLastError();
}

bool knn_tc_eligible(int dtype, int d, int k) {
  if (k < 1 || k > 128) return false;
  const int dpad = (d + 15) / 16 * 16;
  return dtype == kU8 ? d <= 128 : dpad <= 128;  // float: three split tiles fit in shared memory
}

namespace {
struct TcPlan {
  int dpad, nbuf, ctas, grid;
  int64_t ntile, nqtile, chunk, tile_bytes;
  size_t off_ptiles, off_pnorm, off_tmax, off_qtiles, off_qnorm, off_cand, off_pcnt, off_marked, off_tauq, total;
};

size_t align256(size_t x) { return (x + 255) / 256 * 256; }

TcPlan tc_plan(int dtype, int d, int64_t n, int64_t nq_ext, int num_sms) {
  TcPlan P{};
  P.dpad = (d + 15) / 16 * 16;
  P.tile_bytes = int64_t(kTcP) * P.dpad * 2 * tc_nop(dtype);
  P.nbuf = knn_tc_smem(dtype, P.tile_bytes, 3) <= size_t(227) * 1024 ? 3 : 2;  // float rows past 112 dimensions: 2
  if (dtype == kU8) P.nbuf = 2;                                              // two CTAs share an SM
  const size_t smem = knn_tc_smem(dtype, P.tile_bytes, P.nbuf);
  P.ctas = int(std::max<size_t>(1, std::min<size_t>(2, size_t(228 * 1024) / (smem + 1024))));
  P.grid = num_sms * P.ctas;
  // query tiles per launch: as many as there are CTAs, less four, which makes up
  // to 2 grid - 4 parts of 512 KB
  P.chunk = std::max(P.grid - 4, 1);
  P.ntile = (n + kTcP - 1) / kTcP;
  P.nqtile = (nq_ext + kTcQ - 1) / kTcQ;
  const size_t parts = size_t(P.grid) + size_t(P.chunk);
  size_t o = 256;  // header: max |x| bits at 0
  P.off_ptiles = o;
  o = align256(o + size_t(P.ntile) * P.tile_bytes);
  P.off_pnorm = o;
  o = align256(o + size_t(P.ntile) * kTcP * 4);
  P.off_tmax = o;
  o = align256(o + sizeof(float2));
  P.off_qtiles = o;
  o = align256(o + size_t(P.nqtile) * P.tile_bytes);
  P.off_qnorm = o;
  o = align256(o + size_t(P.nqtile) * kTcQ * 4);
  P.off_cand = o;
  o = align256(o + parts * kTcQ * kTcCand * 8);
  P.off_pcnt = o;
  o = o + parts * kTcQ * 4;
  P.off_marked = o;  // right behind: one fill for both
  o = align256(o + size_t(P.chunk) * kTcQ * 4);
  P.off_tauq = o;
  o = align256(o + size_t(P.chunk) * kTcQ * 4);
  P.total = o;
  return P;
}

template <int DT>
cudaError_t scan_and_rank(KnnTcArgs a, const TcPlan& P, cudaStream_t s) {
  const size_t smem = knn_tc_smem(DT, P.tile_bytes, P.nbuf);
  cudaError_t err = cudaFuncSetAttribute(knn_scan_kernel<DT>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
  if (err == cudaSuccess)
    err = cudaFuncSetAttribute(knn_redo_kernel<DT>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
  if (err != cudaSuccess) return err;
  const int64_t nqt = (a.nq + kTcQ - 1) / kTcQ;
  for (a.qt0 = 0; a.qt0 < nqt; a.qt0 += P.chunk) {
    a.nqt = std::min(P.chunk, nqt - a.qt0);
    const int64_t total = a.nqt * P.ntile;
    a.per = std::max<int64_t>((total + P.grid - 1) / P.grid, std::min<int64_t>(P.ntile, kTcMinSteps));
    if ((err = cudaMemsetAsync(a.tauq, 0xff, size_t(a.nqt) * kTcQ * 4, s)) != cudaSuccess) return err;
    if ((err = cudaMemsetAsync(a.pcnt, 0, size_t(P.grid + 2 * P.chunk) * kTcQ * 4, s)) != cudaSuccess) return err;
    knn_scan_kernel<DT><<<unsigned((total + a.per - 1) / a.per), kTcThreads, smem, s>>>(a);
    knn_rank_kernel<DT><<<unsigned(a.nqt * kTcQ / 4), 128, 0, s>>>(a);
    a.per = P.ntile;
    knn_redo_kernel<DT><<<unsigned(a.nqt), kTcThreads, smem, s>>>(a);
    if ((err = cudaGetLastError()) != cudaSuccess) return err;
  }
  return cudaSuccess;
}
}  // namespace

size_t knn_tc_scratch_bytes(int dtype, int d, int64_t n, int64_t nq_ext, int num_sms) {
  return tc_plan(dtype, d, n, nq_ext, num_sms).total;
}

cudaError_t launch_knn_tc(const KnnTcLaunch& K, cudaStream_t s, int64_t* kernels) {
  const bool f32 = K.data.dtype == kF32;
  const TcPlan P = tc_plan(K.data.dtype, K.data.d, K.data.n, K.Q ? K.nq : 0, K.num_sms);
  uint8_t* base = K.scratch;
  unsigned* maxbits = reinterpret_cast<unsigned*>(base);
  cudaError_t err = cudaMemsetAsync(base, 0, 256, s);
  if (err != cudaSuccess) return err;
  // the scale: a power of two that brings max |x| (points, known since their
  // load, and queries) to at most 1
  float scale = f32 ? K.data.scale : 1.f;
  if (f32 && K.Q) {
    maxabs_kernel<<<256, 256, 0, s>>>(K.Q, K.data.row_bytes, K.nq, K.data.d, maxbits);
    unsigned mb = 0;
    if ((err = cudaMemcpyAsync(&mb, maxbits, 4, cudaMemcpyDeviceToHost, s)) != cudaSuccess) return err;
    if ((err = cudaStreamSynchronize(s)) != cudaSuccess) return err;
    float mx = 0.f;
    memcpy(&mx, &mb, 4);
    int e = 0;
    if (mx > 0.f && std::isfinite(mx)) {
      std::frexp(mx, &e);  // mx < 2^e
      scale = std::min(scale, std::ldexp(1.f, -e));
    }
  }
  uint8_t* ptiles = base + P.off_ptiles;
  float* pnorm = reinterpret_cast<float*>(base + P.off_pnorm);
  float2* tmax = reinterpret_cast<float2*>(base + P.off_tmax);
  const int64_t rows = P.ntile * kTcP;
  if (f32)
    pack_f16_kernel<kF32><<<unsigned((rows + 255) / 256), 256, 0, s>>>(K.data.X, K.data.row_bytes, K.data.n, K.data.d,
                                                                      P.dpad, scale, ptiles, pnorm);
  else
    pack_f16_kernel<kU8><<<unsigned((rows + 255) / 256), 256, 0, s>>>(K.data.X, K.data.row_bytes, K.data.n, K.data.d,
                                                                     P.dpad, 1.f, ptiles, pnorm);
  if ((err = cudaMemsetAsync(tmax, 0, sizeof(float2), s)) != cudaSuccess) return err;
  norm_max_kernel<<<unsigned((P.ntile + 7) / 8), 256, 0, s>>>(pnorm, P.ntile, tmax);
  const uint8_t* qtiles = ptiles;
  const float* qnorm = pnorm;
  if (K.Q) {
    uint8_t* qt = base + P.off_qtiles;
    float* qn = reinterpret_cast<float*>(base + P.off_qnorm);
    const int64_t qrows = P.nqtile * kTcQ;
    if (f32)
      pack_f16_kernel<kF32><<<unsigned((qrows + 255) / 256), 256, 0, s>>>(K.Q, K.data.row_bytes, K.nq, K.data.d,
                                                                         P.dpad, scale, qt, qn);
    else
      pack_f16_kernel<kU8><<<unsigned((qrows + 255) / 256), 256, 0, s>>>(K.Q, K.data.row_bytes, K.nq, K.data.d,
                                                                        P.dpad, 1.f, qt, qn);
    qtiles = qt;
    qnorm = qn;
  }
  if ((err = cudaGetLastError()) != cudaSuccess) return err;
  KnnTcArgs a{};
  a.X = K.data.X;
  a.row_bytes = K.data.row_bytes;
  a.n = K.data.n;
  a.d = K.data.d;
  a.Qraw = K.Q;
  a.nq = K.nq;
  a.k = K.k;
  a.qtiles = qtiles;
  a.ptiles = ptiles;
  a.tile_bytes = P.tile_bytes;
  a.ksteps = P.dpad / 16;
  a.nbuf = P.nbuf;
  a.qnorm = qnorm;
  a.pnorm = pnorm;
  a.tmax = tmax;
  a.exact = f32 ? 0 : 1;
  a.kscan = K.Q ? K.k : K.k + 1;
  // Split Gram of scaled rows: |G~ - G| <= eps_ip |q'||p'| + 2^-36 sqrt(d) (|q'| + |p'|):
  // 2^-22 left by the split of each operand, 2^-22 for the dropped lo lo^T, 2^-23 for
  // the last sum, f32 accumulation d 2^-24 with a factor 4 allowance; the lo halves
  // that fall below f16's normal range round to 2^-25 in their units, 2^-36 here.
  a.eps_ip = 4.f * 2.384185791015625e-07f + 1.1920929e-07f + float(K.data.d) * 2.384185791015625e-07f;
  a.eps_n = float(K.data.d + 2) * 5.9604645e-08f;
  a.sub_abs = std::sqrt(float(K.data.d)) * 1.001f * 2.910383e-11f;  // twice 2^-36 sqrt(d)
  a.cand = reinterpret_cast<uint2*>(base + P.off_cand);
  a.pcnt = reinterpret_cast<int*>(base + P.off_pcnt);
  a.marked = reinterpret_cast<int*>(base + P.off_marked);
  a.tauq = reinterpret_cast<unsigned*>(base + P.off_tauq);
  a.out_ids = K.out_ids;
  a.out_dists = K.out_dists;
  a.status = K.status;
  const int64_t chunks = ((K.nq + kTcQ - 1) / kTcQ + P.chunk - 1) / P.chunk;
  *kernels = 2 + (K.Q ? (f32 ? 2 : 1) : 0) + 3 * chunks;
  return f32 ? scan_and_rank<kF32>(a, P, s) : scan_and_rank<kU8>(a, P, s);
}

}  // namespace rpk
