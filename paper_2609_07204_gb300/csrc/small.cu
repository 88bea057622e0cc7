// small.cu -- graphs of up to kSmMaxN vertices solved by one thread block
// each, all rounds of Algorithm 2 in one launch: a batch's graphs (a work
// queue, largest first) and the small graphs of single solves (also what is
// left of a large graph after its first rounds).
//
// A round is the degree bound, the certificate forests of forest.cu (same
// certificate, same batches of highest r; the union-finds are in shared
// memory) and the contraction.  The graph is a list of undirected edges (both
// ends in one word, and the weight): a round relabels the ends and drops the
// loops, and that is all of the contraction -- the forests take parallel edges
// as they come, so nothing is sorted or summed.  Every pass of a round is a
// stream over that list; an edge is inserted in the batch that scans its first
// end.
//
// A round that joins next to nothing (kSmSlow) and lowers nothing first drops the
// soft quantum (weights in units of up to half their mean, for few levels), then
// leaves the graph to the caller's other rounds (bail): Algorithm 2's progress guarantee
// needs an exact maximum-adjacency order.  Counted on the CPU on the batched
// workload (n 20 to 2,000, average degree 3 to 12, weights 1 to 100): 6 levels
// with PR1 / PR2 take 2.85 rounds per graph and no graph is left, 16 levels
// 2.7, without the PR tests 3.5 rounds and one graph in six needs the fine
// quantum.
//
// Bound by instruction issue and shared-memory latency of the links (some
// n x levels of them per round) and by block barriers (7-10 batches per round),
// against one dependent visit per vertex (~0.8 us) of the one-warp solver and
// the whole-graph passes.  Measured (whole calls, one GB300): G(2000, 16000)
// 2.16 -> 0.42 ms, a 256-vertex graph created and solved 0.90 -> 0.21 ms,
// 4,096 graphs (6.3 M edges) 5.44 -> 1.45 ms.
#include <algorithm>
#include <climits>

#include "common.cuh"
#include "kernels.h"
#include "launch.h"

namespace mc {

namespace {

constexpr int kSmMaxK = 254;
constexpr int kSmUnroll = 4;    // edges per lane loaded ahead
constexpr int kSmLevels = 6;    // levels wanted (soft quantum)
constexpr int kSmFast = 8;      // levels inserted at once
constexpr int kSmFrac = 4;      // a batch takes at least 1 / kSmFrac of the vertices left
// Joining less than this a round is left to the other rounds, whose many
// whole-graph passes join up to one vertex each: cycles whose weights are all
// equal by now lose one vertex a round here (a cycle of 50,000 vertices with
// weights of 1 to 100 57.4 -> 3.2 ms, a ring of 3,000 cliques of 8 141 -> 22; with
// 1 / 32 a cycle of 5,000 4.3 instead of 2.8).  Two such rounds in a row: what
// little the first joins may lower the next degree bound (a random 3-regular graph of
// 1,500 with a few doubled edges 0.47 ms, 2.6 when one was enough).
constexpr int kSmSlow = 8;      // one of two rounds joins at least 1 / kSmSlow of the vertices,
constexpr int kSmSlowBatch = 32;  // in a batch, where the warp solver comes after, of them,
constexpr int kSmSlowMin = 64;  // of fewer than kSmSlowMin any
constexpr int kSmThin = 32;     // twice in a row fewer vertices queued, and less than half as many
                                // again as before: everything left is one batch (see kFoThin;
                                // wheel of 1,025 766 -> 429 us, with both 380)
constexpr int kSmThinLate = 6;  // (six times once it has been wider)
constexpr int kSmBatches = 32;  // from this batch on, everything left is one batch

// Shared memory of a block, for graphs of up to `cap` vertices.
struct SmMem {
  int* deg;              // cap
  int* r;                // cap (with deg: the row offsets while the edges are listed)
  unsigned short* lab;   // cap
  unsigned short* map;   // cap: current vertex of each input vertex
  uint8_t* tag;          // cap: batch of each vertex
  uint8_t* side;         // cap: best witness, per input vertex
  int* F;                // fcap union-find words (-1: root)
  int fcap;
};

constexpr int kSmVertexBytes = 4 + 4 + 2 + 2 + 1 + 1;

__device__ __forceinline__ SmMem sm_mem(unsigned char* p, int cap, int fcap) {
  SmMem m;
  m.deg = reinterpret_cast<int*>(p);
  m.r = m.deg + cap;
  m.F = m.r + cap + 4;
  m.lab = reinterpret_cast<unsigned short*>(m.F + fcap);
  m.map = m.lab + cap;
  m.tag = reinterpret_cast<uint8_t*>(m.map + cap);
  m.side = m.tag + cap;
  m.fcap = fcap;
  return m;
}

size_t sm_bytes(int cap, int fcap) {
  return (size_t)cap * kSmVertexBytes + 16 + (size_t)fcap * 4;
}

template <int T>
struct SmShared {
  unsigned long long red[T / 32];
  int warp_cnt[T / 32];
  long long part[T / 32];  // sum: the scanned set's cut weight (see sm_total)
  unsigned long long key;
  int cnt, item;
  unsigned hist[T / 32][5];
  uint2 q[T / 32][64];
};

// Undirected edges: both ends in one word (u | v << 16), weights apart, since
// most passes need the ends alone.
struct SmEdges {
  unsigned* ends;
  int* w;
};

// (see fo_root, fo_joined, fo_join)
__device__ __forceinline__ int sm_root(volatile int* F, int k, int x, int& val) {
  for (;;) {
    const int p = F[x * k];
    if (p < 0) {
      val = p;
      return x;
    }
    const int g = F[p * k];
    if (g < 0) {
      val = g;
      return p;
    }
    F[x * k] = g;
    x = g;
  }
}

__device__ __forceinline__ bool sm_joined(volatile int* F, int k, int x, int y) {
  const int a = F[x * k], b = F[y * k];
  const int a1 = a < 0 ? x : a, b1 = b < 0 ? y : b;
  if (a1 == b1) return true;
  if (a < 0 && b < 0) return false;
  int v;
  return sm_root(F, k, x, v) == sm_root(F, k, y, v);
}

__device__ __forceinline__ bool sm_join(int* F, int k, int x, int y) {
  int vx, vy;
  x = sm_root(F, k, x, vx);
  y = sm_root(F, k, y, vy);
  for (;;) {
    if (x == y) return false;
    if (vx < vy || (vx == vy && x > y)) {  // x: the lesser of the two
      int t = x;
      x = y;
      y = t;
      t = vx;
      vx = vy;
      vy = t;
    }
    const int p = atomicCAS(F + x * k, vx, y);
    if (p == vx) {
      if (vx == vy) atomicCAS(F + y * k, vy, vy - 1);
      return true;
    }
    if (p < 0) vx = p;
    else x = sm_root(F, k, p, vx);
  }
}

// At most kSmFast levels: a lane per (edge, level), 32 / k of the queued edges
// {x, y | units} at a time.  Each lane compares the words of its level (paths
// are short, so most joined levels show), then the lanes of an edge's first
// `units` levels above the last one so joined link them: where y is alone
// (fo_scanned), which is most, by one CAS, else by sm_join.  A lane per edge
// that walked its levels in turn (sm_insert_fast) took ~8 K cycles a call at any
// fill; 4,096 graphs took 2.15 ms with it and take 1.80 with this (1.64 with the
// rest of the change), a G(2000, 16000) round of 32 warps, which is bound by
// issue rather than by that latency, 200 and 255 us: so blocks of few warps and
// rounds of few edges.
__device__ __forceinline__ void sm_insert_wide(int* F, int k, int take, const uint2* q) {
  const int lane = threadIdx.x & 31;
  const int g = lane / k, i = lane - g * k;
  const bool act = g < take;
  const uint2 it = q[act ? g : 0];
  const int x = it.x & 0xffff, y = it.x >> 16, units = (int)it.y;
  const int a = *(volatile int*)&F[x * k + i], b = *(volatile int*)&F[y * k + i];
  const int px = a < 0 ? x : a;
  const unsigned field = ((1u << k) - 1u);
  const int at = act ? g * k : 0;
  const unsigned closed = __ballot_sync(FULL, act && px == (b < 0 ? y : b)) >> at & field;
  int lo = 32 - __clz(closed), want = act ? min(units, k - lo) : 0;
  bool alone = b == -1;
  for (;;) {
    bool ok = false;
    if (i >= lo && i < lo + want)
      ok = (alone && atomicCAS(&F[y * k + i], -1, px) == -1) || sm_join(F + i, k, x, y);
    const int got = __popc(__ballot_sync(FULL, ok) >> at & field);
    lo += want;  // units whose level was joined meanwhile go on above
    want = max(0, min(want - got, k - lo));
    if (!__any_sync(FULL, want > 0)) return;
    alone = false;
  }
}

// At most kSmFast levels: the levels that join x and y by their words alone
// (paths are short, so most), then the units into those above the last one;
// where y is alone (fo_scanned), which is most, by one CAS.  Returns the units
// inserted, -1 if the last level joins the ends already.
__device__ __forceinline__ int sm_insert_fast(int* F, int k, int x, int y, int units) {
  int a[kSmFast], b[kSmFast];
  unsigned closed = 0;
#pragma unroll
  for (int i = 0; i < kSmFast; ++i) {
    a[i] = b[i] = 0;
    if (i < k) {
      const int p = *(volatile int*)&F[x * k + i];
      b[i] = *(volatile int*)&F[y * k + i];
      a[i] = p < 0 ? x : p;
      if (a[i] == (b[i] < 0 ? y : b[i])) closed |= 1u << i;
    }
  }
  if (closed >> (k - 1)) return -1;
  const int lo = 32 - __clz(closed);
  int got = 0, tried = 0;
  unsigned rest = 0;  // tried levels left to sm_join
#pragma unroll
  for (int i = 0; i < kSmFast; ++i)
    if (i >= lo && i < k && tried < units) {
      ++tried;
      if (b[i] == -1 && atomicCAS(&F[y * k + i], -1, a[i]) == -1) ++got;
      else rest |= 1u << i;
    }
  for (int i = lo + tried; rest || (got < units && i < k);) {
    int l = i;
    if (rest) {
      l = __ffs(rest) - 1;
      rest &= rest - 1;
    } else {
      ++i;  // units whose level was joined meanwhile go on above
    }
    if (sm_join(F + l, k, x, y)) ++got;
  }
  return got;
}

// First level that does not join x and y (k: none), level `guess` tried first
// (see fo_insert).
__device__ __forceinline__ int sm_level(int* F, int k, int x, int y, int guess) {
  int lo = 0, hi = guess;
  if (sm_joined(F + guess, k, x, y)) {
    lo = guess + 1;
    hi = k;
    for (int st = 1; lo < hi; st *= 2) {
      const int m = min(hi - 1, lo + st - 1);
      if (!sm_joined(F + m, k, x, y)) {
        hi = m;
        break;
      }
      lo = m + 1;
    }
  } else {
    for (int st = 1; lo < hi; st *= 2) {
      const int m = max(lo, hi - st);
      if (sm_joined(F + m, k, x, y)) {
        lo = m + 1;
        break;
      }
      hi = m;
    }
  }
  while (lo < hi) {
    const int m = (lo + hi) >> 1;
    if (sm_joined(F + m, k, x, y)) lo = m + 1;
    else hi = m;
  }
  return lo;
}

// Insert a warp's edges {x, y} from level lo up (units = 0: none), a lane per
// (edge, level): a lane that walked its own edge's levels would hold the warp
// up for its longest.
__device__ __forceinline__ void sm_insert(int* F, int k, int x, int y, int lo, int units) {
  const int lane = threadIdx.x & 31;
  int want = min(units, k - lo);
  for (;;) {
    int incl = want;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(FULL, incl, o);
      if (lane >= o) incl += u;
    }
    const int total = __shfl_sync(FULL, incl, 31);
    if (total == 0) return;
    const int excl = incl - want;
    int got = 0;
    for (int p0 = 0; p0 < total; p0 += 32) {
      const int p = p0 + lane;
      int o = 0;  // the edge of position p
#pragma unroll
      for (int stp = 16; stp > 0; stp >>= 1) {
        const int v = __shfl_sync(FULL, incl, o + stp - 1);
        if (v <= p) o += stp;
      }
      const int ex = __shfl_sync(FULL, x, o), ey = __shfl_sync(FULL, y, o);
      const int level = __shfl_sync(FULL, lo - excl, o) + p;
      const bool ok = p < total && sm_join(F + level, k, ex, ey);
      const unsigned bal = __ballot_sync(FULL, ok);
      const int b0 = max(excl - p0, 0), b1 = min(incl - p0, 32);
      if (b0 < b1) got += __popc(bal & (FULL >> (32 - (b1 - b0)) << b0));
    }
    lo += want;  // units whose level was joined meanwhile go on above
    want = max(0, min(want - got, k - lo));
  }
}

template <int T>
__device__ __forceinline__ unsigned long long sm_min(unsigned long long v, SmShared<T>& s) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = min(v, __shfl_xor_sync(FULL, v, o));
  if ((threadIdx.x & 31) == 0) s.red[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    unsigned long long u = threadIdx.x < T / 32 ? s.red[threadIdx.x] : ~0ull;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) u = min(u, __shfl_xor_sync(FULL, u, o));
    if (threadIdx.x == 0) s.key = u;
  }
  __syncthreads();
  return s.key;
}

// Sum of the warps' parts (each warp adds to its own: 64-bit atomics on one
// shared word spin, ~2 K cycles a batch with 32 warps).
template <int T>
__device__ __forceinline__ long long sm_total(const SmShared<T>& s) {
  const int lane = threadIdx.x & 31;
  return warp_sum(lane < T / 32 ? s.part[lane] : 0ll);
}

// Unscanned vertices with at least t units.
template <int T>
__device__ __forceinline__ int sm_count(const SmMem& sm, int n, int t) {
  int c = 0;
  for (int v0 = 0; v0 < n; v0 += T) {
    const int v = v0 + (int)threadIdx.x;
    c += __syncthreads_count(v < n && sm.tag[v] == 0 && sm.r[v] >= t);
  }
  return c;
}

// The batch threshold at most kSmFast levels: the largest t that `need` of the
// vertices left have (1 if none), 0 where no vertex left has a unit or `all`.
// Returns the vertices left; queued: those of them with any unit.  One pass and one barrier: each warp's counts per
// key, 16 bits each (a graph has at most kSmMaxN vertices), added up by every
// warp for itself.  The bisection over block-wide counts that more levels take
// took 12 K cycles of each batch of a
// G(2000, 16000) round, this 9 K (most of it the new tags); with the loads of
// the edge list four at a time that solve went from 455 to 418 us.
template <int T>
__device__ __forceinline__ int sm_select(const SmMem& sm, SmShared<T>& s, int n, int k, bool all,
                                         int& t, int& queued) {
  static_assert(kSmFast <= 9 && kSmMaxN < 65536, "counts per key");
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  unsigned long long h[3] = {0, 0, 0};
  for (int v = threadIdx.x; v < n; v += T)
    if (sm.tag[v] == 0) {
      const int key = min(sm.r[v], k);
      const unsigned long long one = 1ull << (16 * (key & 3));
      if (key < 4) h[0] += one;
      else if (key < 8) h[1] += one;
      else h[2] += one;
    }
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    const unsigned x = __reduce_add_sync(FULL, (unsigned)(h[i / 2] >> (32 * (i & 1))));
    if (lane == 0) s.hist[wp][i] = x;
  }
  __syncthreads();
  unsigned c[5];
  int left = 0;
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    c[i] = __reduce_add_sync(FULL, lane < T / 32 ? s.hist[lane][i] : 0u);
    left += (int)(c[i] & 0xffff) + (int)(c[i] >> 16);
  }
  t = 0;
  queued = left - (int)(c[0] & 0xffff);
  if (queued > 0 && !all) {
    const int need = max(1, left / kSmFrac);
    int have = 0;
    t = 1;
#pragma unroll
    for (int key = 9; key >= 1; --key) {
      have += (int)(c[key / 2] >> (16 * (key & 1)) & 0xffff);
      if (have >= need) t = max(t, key);
    }
  }
  return left;
}

// Lists the undirected edges of rows [v0, v0 + n) in `ed` (ends relative to
// v0; weights are positive, rows hold no loops); returns their number, -1 if
// there are more than ecap (only an input that is not symmetric has).
template <int T>
__device__ int sm_load(const SmMem& sm, SmShared<T>& s, const int64_t* rp, const int* col,
                       const int* w, int v0, int n, SmEdges ed, int ecap) {
  const int tid = threadIdx.x, lane = tid & 31;
  const long long base = rp[v0];
  int* srp = sm.deg;  // n + 1 words over deg and r
  for (int i = tid; i <= n; i += T) srp[i] = (int)(rp[v0 + i] - base);
  if (tid == 0) s.cnt = 0;
  __syncthreads();
  const int M = srp[n];
  // (kSmUnroll entries per lane at a time: their loads and row searches overlap)
  for (int e0 = tid; e0 - lane < M; e0 += T * kSmUnroll) {
    int u[kSmUnroll], v[kSmUnroll], c[kSmUnroll];
    int lo[kSmUnroll], hi[kSmUnroll];
#pragma unroll
    for (int j = 0; j < kSmUnroll; ++j) {
      const int e = e0 + j * T;
      v[j] = e < M ? col[base + e] - v0 : -1;
      c[j] = e < M ? w[base + e] : 0;
      lo[j] = 0;
      hi[j] = n;
    }
    // the row with srp[row] <= e < srp[row + 1]
    for (int half = n; half > 1; half = (half + 1) >> 1) {
#pragma unroll
      for (int j = 0; j < kSmUnroll; ++j) {
        const int mid = (lo[j] + hi[j]) >> 1;
        if (hi[j] - lo[j] > 1) {
          if (srp[mid] <= e0 + j * T) lo[j] = mid;
          else hi[j] = mid;
        }
      }
    }
    unsigned bal[kSmUnroll];
    int cnt = 0;
#pragma unroll
    for (int j = 0; j < kSmUnroll; ++j) {
      u[j] = lo[j];
      bal[j] = __ballot_sync(FULL, u[j] < v[j]);
      cnt += __popc(bal[j]);
    }
    int at = 0;
    if (lane == 0 && cnt) at = atomicAdd(&s.cnt, cnt);
    at = __shfl_sync(FULL, at, 0);
#pragma unroll
    for (int j = 0; j < kSmUnroll; ++j) {
      const int o = at + __popc(bal[j] & lanemask_lt());
      if (u[j] < v[j] && o < ecap) {
        ed.ends[o] = (unsigned)u[j] | ((unsigned)v[j] << 16);
        ed.w[o] = c[j];
      }
      at += __popc(bal[j]);
    }
  }
  __syncthreads();
  return s.cnt <= ecap ? s.cnt : -1;
}

// All rounds on the n0-vertex graph of the m edges in ed[0].  lam_io: the
// bound so far, lowered to the smallest cut found (its witness then in
// sm.side and source 1: a degree, 3: a prefix cut; else 0).  False: some round could
// not go on (bail); limited: with more levels, which the grid-wide forests have, it might.
template <int T>
__device__ bool sm_solve(const SmMem& sm, SmShared<T>& s, SmEdges ed0, SmEdges ed1, int m, int n0,
                         uint32_t pr_mask, long long& lam_io, int& source, int& rounds,
                         bool& limited) {
  const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
  long long lam = lam_io;
  int n = n0, cur = 0;
  bool soft = true, slow = false;
  source = 0;
  rounds = 0;
  limited = false;
  for (int i = tid; i < n0; i += T) sm.map[i] = (unsigned short)i;
  bool ok = false;
  for (int round = 0; round < 2 * n0 + 8; ++round) {
    const SmEdges ed = cur ? ed1 : ed0;
    // ---- degree bound
    for (int v = tid; v < n; v += T) sm.deg[v] = 0;
    __syncthreads();
    long long wsum = 0;
    for (int e = tid; e < m; e += T) {
      const unsigned d = ed.ends[e];
      const int c = ed.w[e];
      atomicAdd(&sm.deg[d & 0xffff], c);
      atomicAdd(&sm.deg[d >> 16], c);
      wsum += c;
    }
    wsum = warp_sum(wsum);
    if (lane == 0) s.part[wp] = wsum;
    __syncthreads();
    wsum = sm_total<T>(s);
    unsigned long long best = ~0ull;
    for (int v = tid; v < n; v += T)
      best = min(best, ((unsigned long long)(unsigned)sm.deg[v] << 32) | (unsigned)v);
    best = sm_min<T>(best, s);
    if (n >= 2 && (long long)(best >> 32) < lam) {
      lam = (long long)(best >> 32);
      const int x = (int)(best & 0xffffffffull);
      for (int i = tid; i < n0; i += T) sm.side[i] = sm.map[i] == x ? 1 : 0;
      source = 1;
    }
    if (n <= 2 || lam == 0) {
      ok = true;
      break;
    }
    ++rounds;
    const long long mean = wsum / max(m, 1);
    const int kcap = min(kSmMaxK, sm.fcap / n);
    if (kcap < 1) break;
    const long long qmin = (lam + kcap - 1) / kcap;
    // too few levels for the weights: in a batch hardly an edge has a unit, in a
    // single solve, which has the grid-wide forests behind it, the mean edge has none
    // (500 vertices of degree 200 and weights 1 to 20: 4.4 -> 1.6 ms with what follows)
    if (qmin >= (T > 256 ? mean + 1 : 2 * max(mean, 1ll))) {
      limited = true;
      break;  // bail
    }
    // soft quantum: as few levels as the size asks for, at most half the mean
    // weight
    const long long qw = max(qmin, soft ? min((mean + 1) / 2, (lam + kSmLevels - 1) / kSmLevels) : 1ll);
    const int q = (int)qw;  // (at most the bound, a degree)
    const int k = (int)((lam + qw - 1) / qw);
    __syncthreads();  // (the parts are read above)
    const bool fast = k <= kSmFast;
    const bool wide = fast && (T <= 256 || m <= T);
    const int group = wide ? 32 / k : 32;  // edges inserted together
    // ---- all roots, nothing scanned, the first batch is vertex 0
    for (int i = tid; i < n * k; i += T) sm.F[i] = i < k ? -2 : -1;
    for (int v = tid; v < n; v += T) {
      sm.r[v] = 0;
      sm.tag[v] = v == 0 ? 1 : 0;
    }
    if (lane == 0) s.part[wp] = wp == 0 ? sm.deg[0] : 0;
    __syncthreads();
    long long best_alpha = kInf;
    int thin = 0, queued_before = 1, widest = 0;
    int best_batch = 0;
    for (int b = 1;; ++b) {
      if (b > 1) {
        // the largest t that takes 1 / kSmFrac of the vertices left, by
        // bisection over block-wide counts (a shared histogram would serialise
        // its few hot words); t = 1 where the queue is smaller than that
        int t = 0, left;
        int queued;
        if (fast) {
          left = sm_select<T>(sm, s, n, k, b >= kSmBatches, t, queued);
        } else {
          left = sm_count<T>(sm, n, 0);
          queued = sm_count<T>(sm, n, 1);
        }
        widest = max(widest, queued);
        thin = queued < kSmThin && 2 * queued < 3 * queued_before ? thin + 1 : 0;
        queued_before = queued;
        if (thin >= (widest < kSmThin ? 2 : kSmThinLate)) {
          t = 0;
        } else if (!fast) {
          if (left > 0 && b < kSmBatches && queued > 0) {
            const int need = max(1, left / kSmFrac);
            int lo = 1, hi = k;
            while (lo < hi) {
              const int mid = (lo + hi + 1) >> 1;
              if (sm_count<T>(sm, n, mid) >= need) lo = mid;
              else hi = mid - 1;
            }
            t = lo;
          }
        }
        const long long al = sm_total<T>(s);
        if (left > 0 && al < best_alpha) {
          best_alpha = al;
          best_batch = b - 1;
        }
        if (left <= 0) break;
        __syncthreads();
        long long add = 0;
        for (int v = tid; v < n; v += T)
          if (sm.tag[v] == 0) {
            const int key = min(sm.r[v], k);
            if (key >= t) {
              sm.tag[v] = (uint8_t)b;
              for (int i = 0; i < k; ++i)
                if (sm.F[v * k + i] == -1) sm.F[v * k + i] = -2;
              add += sm.deg[v];
            }
          }
        add = warp_sum(add);
        if (lane == 0) s.part[wp] += add;
        __syncthreads();
      }
      // ---- the edges whose first end is in this batch
      long long sub = 0;
      int qn = 0;
      // few edges are dealt out one by one, so that every warp has some
      const bool spread = m <= 2 * T;
      for (int i0 = 0; i0 < m; i0 += T * kSmUnroll) {
        const int e0 = i0 + (spread ? lane * (T / 32) + wp : wp * (32 * kSmUnroll) + lane);
        const int stp = spread ? T : 32;
        const bool last = i0 + T * kSmUnroll >= m;
        unsigned d[kSmUnroll];
        int c[kSmUnroll];
        bool keep[kSmUnroll];
#pragma unroll
        for (int j = 0; j < kSmUnroll; ++j) d[j] = e0 + j * stp < m ? ed.ends[e0 + j * stp] : 0u;
#pragma unroll
        for (int j = 0; j < kSmUnroll; ++j) {
          const int e = e0 + j * stp;
          const int tu = sm.tag[d[j] & 0xffff], tv = sm.tag[d[j] >> 16];
          const bool now = e < m && (tu == b || tv == b);
          c[j] = now ? ed.w[e] : 0;
          keep[j] = now && (tu == b || tu == 0) && (tv == b || tv == 0);
          if (now && tu != 0 && tv != 0) sub += c[j];  // now inside the scanned set
          if (tu != b) d[j] = d[j] >> 16 | d[j] << 16;  // x scanned, y the far end
        }
#pragma unroll
        for (int j = 0; j < kSmUnroll; ++j) {
          const int units = !keep[j] ? 0 : min(k, q == 1 ? c[j] : c[j] / q);
          const unsigned bal = __ballot_sync(FULL, units > 0);
          if (units > 0) {
            if (fast && sm.r[d[j] >> 16] < k) atomicAdd(&sm.r[d[j] >> 16], units);
            s.q[wp][qn + __popc(bal & lanemask_lt())] = make_uint2(d[j], (unsigned)units);
          }
          qn += __popc(bal);
          const bool end = j == kSmUnroll - 1 && last;  // the warp's last edges
          while (qn >= group || (end && qn > 0)) {
            __syncwarp();
            const int take = min(qn, group);
            qn -= take;
            if (wide) {
              sm_insert_wide(sm.F, k, take, &s.q[wp][qn]);
            } else if (fast) {
              if (lane < take) {
                const uint2 it = s.q[wp][qn + lane];
                sm_insert_fast(sm.F, k, it.x & 0xffff, it.x >> 16, (int)it.y);
              }
            } else {
              int x = 0, y = 0, u = 0, lo = 0;
              if (lane < take) {
                const uint2 it = s.q[wp][qn + lane];
                x = it.x & 0xffff;
                y = it.x >> 16;
                u = (int)it.y;
                int g = sm.r[y];
                if (g < k) g = atomicAdd(&sm.r[y], u);
                lo = sm_level(sm.F, k, x, y, min(g, k - 1));
                if (lo == k) u = 0;
              }
              __syncwarp();
              sm_insert(sm.F, k, x, y, lo, u);
            }
            __syncwarp();
          }
        }
      }
      sub = warp_sum(sub);
      if (lane == 0) s.part[wp] -= 2 * sub;
      __syncthreads();
    }
    __syncthreads();
    bool lowered = false;
    if (best_alpha < lam) {
      lam = best_alpha;
      for (int i = tid; i < n0; i += T) sm.side[i] = sm.tag[sm.map[i]] <= best_batch ? 1 : 0;
      lowered = true;
      source = 3;
      if (lam == 0) {
        ok = true;
        break;
      }
    }
    // the last level that the bound still asks for
    int* top = sm.F + (int)((lam + q - 1) / q) - 1;
    // ---- PR1 / PR2 (Sec. 2.1) join in it too: of parallel edges each alone,
    // which is a weaker test of the same edge
    if (pr_mask) {
      for (int e = tid; e < m; e += T) {
        const unsigned d = ed.ends[e];
        const long long c = ed.w[e];
        const int u = d & 0xffff, v = d >> 16;
        if (((pr_mask & 1u) && c >= lam) ||
            ((pr_mask & 2u) && (sm.deg[u] < 2 * c || sm.deg[v] < 2 * c)))
          sm_join(top, k, u, v);
      }
      __syncthreads();
    }
    // ---- labels: the rank of the root
    int n2 = 0;
    for (int v0 = 0; v0 < n; v0 += T) {
      const int v = v0 + tid;
      const bool root = v < n && top[v * k] < 0;
      const unsigned bal = __ballot_sync(FULL, root);
      if (lane == 0) s.warp_cnt[wp] = __popc(bal);
      __syncthreads();
      int before = n2, total = 0;
      for (int i = 0; i < T / 32; ++i) {
        const int c = s.warp_cnt[i];
        if (i < wp) before += c;
        total += c;
      }
      if (root) sm.r[v] = before + __popc(bal & lanemask_lt());
      n2 += total;
      __syncthreads();
    }
    const int least = n < kSmSlowMin ? 1 : n / (T > 256 ? kSmSlow : kSmSlowBatch);
    if (lowered || n - n2 >= least) {
      slow = false;
    } else if (n2 < n && !slow) {
      slow = true;  // (what little it joined may lower the next degree bound)
    } else {
      // (a finer quantum does not help where a thin frontier and PR joined nothing)
      if (!soft || q == qmin || (widest < kSmThin && thin >= 2 && pr_mask && n2 == n)) {
        limited = qmin > (mean + 1) / 2;
        break;  // bail
      }
      soft = false;
    }
    if (n2 == n) continue;  // again, from the lower bound or with the finer quantum
    for (int v = tid; v < n; v += T) {
      int x = v;
      while (top[x * k] >= 0) x = top[x * k];
      sm.lab[v] = (unsigned short)sm.r[x];
    }
    if (tid == 0) s.cnt = 0;
    __syncthreads();
    // ---- contraction
    for (int i = tid; i < n0; i += T) sm.map[i] = sm.lab[sm.map[i]];
    const SmEdges out = cur ? ed0 : ed1;
    // few vertices left: parallel edges are summed in a matrix (over F, which
    // is done with); else the list keeps them
    const bool dense = n2 * n2 <= sm.fcap;
    if (dense) {
      __syncthreads();
      for (int i = tid; i < n2 * n2; i += T) sm.F[i] = 0;
      __syncthreads();
      for (int e = tid; e < m; e += T) {
        const unsigned d = ed.ends[e];
        const int u = sm.lab[d & 0xffff], v = sm.lab[d >> 16];
        if (u != v) atomicAdd(&sm.F[min(u, v) * n2 + max(u, v)], ed.w[e]);
      }
      __syncthreads();
    }
    const int items = dense ? n2 * n2 : m;
    for (int e0 = wp * 32; e0 < items; e0 += T) {
      const int e = e0 + lane;
      bool keep = false;
      unsigned d = 0;
      int c = 0;
      if (e < items) {
        if (dense) {
          c = sm.F[e];
          keep = c != 0;
          d = keep ? (unsigned)(e / n2) | ((unsigned)(e % n2) << 16) : 0u;
        } else {
          d = ed.ends[e];
          const unsigned u = sm.lab[d & 0xffff], v = sm.lab[d >> 16];
          keep = u != v;
          if (keep) c = ed.w[e];
          d = u | (v << 16);
        }
      }
      const unsigned bal = __ballot_sync(FULL, keep);
      int at = 0;
      if (lane == 0 && bal) at = atomicAdd(&s.cnt, __popc(bal));
      at = __shfl_sync(FULL, at, 0) + __popc(bal & lanemask_lt());
      if (keep) {
        out.ends[at] = d;
        out.w[at] = c;
      }
    }
    __syncthreads();
    m = s.cnt;
    n = n2;
    cur ^= 1;
    if (n <= 1) {
      ok = true;
      break;
    }
  }
  __syncthreads();
  lam_io = lam;
  return ok;
}

// The current graph of a single solve (n <= kSmMaxN; or, with `count`, the
// st->n_next vertices and *count edges in ed0): its minimum cut below
// st->lambda.  st->small_status: 1 solved, 2 bail (too many entries, or too few
// levels for a round), 3 bail and no use for the grid-wide forests; st->small_improved: what lowered the bound
// (0: nothing), its witness per vertex of the graph in cur_side.
template <int T>
__global__ void __launch_bounds__(T, 1)
    small_solve_kernel(int n, const int64_t* rp, const int* col, const int* w, SmEdges ed0,
                       SmEdges ed1, long long mcap, int fcap, uint32_t pr_mask, uint8_t* cur_side,
                       const int* count, DevState* st) {
  extern __shared__ __align__(16) unsigned char sm_dyn[];
  __shared__ SmShared<T> s;
  const SmMem sm = sm_mem(sm_dyn, kSmMaxN, fcap);
  if (count) n = st->n_next;
  if (count ? *count > mcap / 2 || n > kSmMaxN : rp[n] > mcap) {
    if (threadIdx.x == 0) {
      st->small_status = 2;
      st->small_improved = 0;
    }
    return;
  }
  long long lam = (long long)*(volatile unsigned long long*)&st->lambda;
  int source, rounds;
  bool limited = true;
  const int m = count ? *count : sm_load<T>(sm, s, rp, col, w, 0, n, ed0, (int)(mcap / 2));
  source = rounds = 0;
  const bool ok = m >= 0 && sm_solve<T>(sm, s, ed0, ed1, m, n, pr_mask, lam, source, rounds, limited);
  if (source)
    for (int i = threadIdx.x; i < n; i += T) cur_side[i] = sm.side[i];
  if (threadIdx.x == 0) {
    st->lambda = (unsigned long long)lam;
    st->small_status = ok ? 1 : limited ? 2 : 3;
    st->small_improved = source;
    st->small_rounds = rounds;
  }
}

// A batch's graphs list[0 .. nlist) (largest first), a block per graph at a
// time: lam_g and side0 of each; those that bail go to left[0 .. *nleft).
// Block b's edges: `words` words at scratch + b * slot_words.
template <int T>
__global__ void __launch_bounds__(T, 3)
    small_batch_kernel(const int* __restrict__ list, int nlist, int* cursor,
                       const int* __restrict__ voff0, const int64_t* rp0, const int* col0,
                       const int* w0, int* scratch, long long slot_words, int mmax, int cap,
                       int fcap, uint32_t pr_mask, unsigned long long* lam_g, uint8_t* side0,
                       int* left, int* nleft) {
  extern __shared__ __align__(16) unsigned char sm_dyn[];
  __shared__ SmShared<T> s;
  const SmMem sm = sm_mem(sm_dyn, cap, fcap);
  int* base = scratch + (long long)blockIdx.x * slot_words;
  const int half = mmax / 2 + 1;
  const SmEdges ed0{reinterpret_cast<unsigned*>(base), base + half};
  const SmEdges ed1{reinterpret_cast<unsigned*>(base + 2 * half), base + 3 * half};
  for (;;) {
    if (threadIdx.x == 0) s.item = atomicAdd(cursor, 1);
    __syncthreads();
    const int item = s.item;
    if (item >= nlist) return;
    const int gi = list[item];
    const int v0 = voff0[gi], n = voff0[gi + 1] - v0;
    long long lam = kInf;
    int source, rounds;
    bool limited = true;
    const int m = sm_load<T>(sm, s, rp0, col0, w0, v0, n, ed0, half);
    const bool ok = m >= 0 && sm_solve<T>(sm, s, ed0, ed1, m, n, pr_mask, lam, source, rounds, limited);
    if (ok)
      for (int i = threadIdx.x; i < n; i += T) side0[v0 + i] = sm.side[i];
    if (threadIdx.x == 0) {
      if (ok) lam_g[gi] = (unsigned long long)lam;
      else left[atomicAdd(nleft, 1)] = gi;
    }
    __syncthreads();  // (the next graph reuses the block's shared memory)
  }
}

__global__ void side_if_improved_kernel(uint8_t* side0, const int* __restrict__ map0,
                                        const int* __restrict__ L, int n0,
                                        const uint8_t* __restrict__ cur, const DevState* st) {
  if (!st->small_improved) return;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n0; i += gridDim.x * blockDim.x)
    side0[i] = cur[L ? L[map0[i]] : map0[i]];
}

}  // namespace

constexpr int kSmThreads = 1024;
constexpr int kSmFcap = 40 * 1024;  // union-find words of the single solves: 160 KB

static SmEdges sm_edges(void* p, long long mcap) {  // mcap / 2 edges
  return SmEdges{static_cast<unsigned*>(p), static_cast<int*>(p) + (mcap / 2 + 1)};
}

static bool sm_solve_attr() {
  static OncePerDevice once;
  return once([] {
    return cudaFuncSetAttribute(small_solve_kernel<kSmThreads>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)sm_bytes(kSmMaxN, kSmFcap)) == cudaSuccess;
  });
}

cudaError_t small_solve(int n, const int64_t* rp, const int* col, const int* w, void* ed0,
                        void* ed1, long long mcap, uint32_t pr_mask, uint8_t* cur_side,
                        const int* map0, int n0, uint8_t* side0, int sms, DevState* st,
                        cudaStream_t s, int* launches) {
  if (n < 1 || n > kSmMaxN || !sm_solve_attr()) return cudaErrorInvalidValue;
  small_solve_kernel<kSmThreads><<<1, kSmThreads, sm_bytes(kSmMaxN, kSmFcap), s>>>(
      n, rp, col, w, sm_edges(ed0, mcap), sm_edges(ed1, mcap), mcap, kSmFcap, pr_mask, cur_side,
      nullptr, st);
  ++*launches;
  return small_side(cur_side, map0, nullptr, n0, side0, sms, st, s, launches);
}

cudaError_t small_side(const uint8_t* cur_side, const int* map0, const int* L, int n0,
                       uint8_t* side0, int sms, const DevState* st, cudaStream_t s,
                       int* launches) {
  side_if_improved_kernel<<<std::max(1, std::min((n0 + 255) / 256, sms * 8)), 256, 0, s>>>(
      side0, map0, L, n0, cur_side, st);
  ++*launches;
  return cudaGetLastError();
}

SmallList small_list(void* ed0, void* mat, long long mat_words, long long mcap) {
  const SmEdges e = sm_edges(ed0, mcap);
  return SmallList{e.ends, e.w, (int)(mcap / 2), static_cast<int*>(mat), mat_words};
}

cudaError_t small_rest(void* ed0, void* ed1, long long mcap, const int* count, uint32_t pr_mask,
                       uint8_t* cur_side, DevState* st, cudaStream_t s, int* launches) {
  if (!sm_solve_attr()) return cudaErrorInvalidValue;
  small_solve_kernel<kSmThreads><<<1, kSmThreads, sm_bytes(kSmMaxN, kSmFcap), s>>>(
      0, nullptr, nullptr, nullptr, sm_edges(ed0, mcap), sm_edges(ed1, mcap), mcap, kSmFcap,
      pr_mask, cur_side, count, st);
  ++*launches;
  return cudaGetLastError();
}

// Shared memory of the batch kernel by its largest graph: as many union-find
// words as let three blocks share an SM (at least 5 levels of the largest).
constexpr int kSmBatchThreads = 256;
static int sm_batch_cap(int nmax) { return (nmax + 63) / 64 * 64; }
static int sm_batch_fcap(int nmax) { return std::max(4096, std::min(10240, 16 * sm_batch_cap(nmax))); }

cudaError_t small_batch(const int* list, int nlist, int* cursor, const int* voff0,
                        const int64_t* rp0, const int* col0, const int* w0, int* scratch,
                        long long slot_words, int slots, int nmax, int mmax, uint32_t pr_mask,
                        unsigned long long* lam_g, uint8_t* side0, int* left, int* nleft, int sms,
                        cudaStream_t s, int* launches) {
  if (nlist <= 0) return cudaSuccess;
  if (nmax > kSmMaxN || slots < 1) return cudaErrorInvalidValue;
  const int cap = sm_batch_cap(nmax), fcap = sm_batch_fcap(nmax);
  const size_t bytes = sm_bytes(cap, fcap);
  static OncePerDevice once;
  const auto set_up = [] {
    return cudaFuncSetAttribute(small_batch_kernel<kSmBatchThreads>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)sm_bytes(sm_batch_cap(kSmMaxN), sm_batch_fcap(kSmMaxN))) ==
           cudaSuccess;
  };
  if (!once(set_up)) return cudaErrorInvalidValue;
  int per_sm = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
      &per_sm, small_batch_kernel<kSmBatchThreads>, kSmBatchThreads, bytes);
  if (e != cudaSuccess) return e;
  const int blocks = std::min({nlist, slots, sms * std::max(1, per_sm)});
  e = cudaMemsetAsync(cursor, 0, sizeof(int), s);
  if (e == cudaSuccess) e = cudaMemsetAsync(nleft, 0, sizeof(int), s);
  if (e != cudaSuccess) return e;
  small_batch_kernel<kSmBatchThreads><<<blocks, kSmBatchThreads, bytes, s>>>(
      list, nlist, cursor, voff0, rp0, col0, w0, scratch, slot_words, mmax, cap, fcap, pr_mask, lam_g,
      side0, left, nleft);
  ++*launches;
  return cudaGetLastError();
}

}  // namespace mc
