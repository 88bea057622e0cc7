// forest.cu -- certificate forests: the marking step of a round as one
// edge-parallel pass over the whole graph, in one cooperative kernel with the
// rest of the round's head: degree bound before, labels and the list of what is
// left after (22 launches of 2 to 5 us each otherwise, and as many gaps: R-MAT
// scale 16 core 473 -> 394 us, 64 served requests 11.9 -> 8.4 ms).
//
// Certificate.  Let lam be the round's bound, q a quantum and k = ceil(lam/q).
// An edge of weight c has floor(c/q) units.  Every edge puts its units into
// k edge sets F_0 .. F_{k-1}: into the lowest levels whose components do not
// yet join its ends, at most one unit per level, level i only once its ends
// are joined in F_{i-1}.  Components of F_i therefore refine those of F_{i-1}
// (the forest decomposition of Nagamochi and Ibaraki, with forests that need
// not come from a maximum-adjacency order), so two vertices joined in F_{k-1}
// are joined in each of the k edge-disjoint sets: their connectivity is at
// least k q >= lam and they may be contracted.  This holds for every order of
// the edges and every interleaving of threads: a level's union-find only ever
// merges, and "joined in F_{i-1}" once read stays true.
//
// Order.  How much F_{k-1} joins does depend on the order.  A maximum-
// adjacency order is the best known and strictly sequential; here the vertices
// are scanned in a few batches, each the unscanned vertices of highest r (the
// units that met them), at least 1 / kFoFrac of the vertices left and 1 / kFoTail
// of all where so many are queued.  Counted on the CPU on the planted cut (2 x 2^13 vertices,
// the entries of a batch in random order), the vertices F_{k-1} leaves: exact
// order 0.80 n, batches of 1/50 0.80 n, 1/20 0.81 n, 1/10 0.83 n, 1/4 0.93 n:
// ~30 grid-wide steps replace one dependent step per vertex (1/16 without the
// 1/64 of all, ~50 steps: 6% slower on both planted cuts; 1/8 as fast, but now
// and then a round too weak).
//
// The prefix cuts of the batches (alpha, as in a CAPFOREST pass) are cuts of
// the graph: the smallest lowers the bound, the scanned batches up to it its
// witness, and the marks are taken from the level that the lowered bound asks
// for.  A batch does not reach below half the highest r, so one ends where a
// region ends (planted cut 2 x 2^19: the cut of 25 is found in the first round,
// which joins 0.43 n instead of 0.22 n; 16.0 -> 9.1 ms, 2 x 2^15 6.3 -> 3.9).
//
// Cost.  An entry is read once, with its vertex: a stream read of (col, w) and
// the far end's tag byte (scanned before: done).  The rest queue per warp, so
// that the divergent part runs with full warps: the far end's r (the level to
// try first), usually two adjacent levels of each end's row of parent words
// (vertex-major: one 32-byte sector) and one CAS per unit, all random accesses
// to L1 and L2 in a dependent chain of ~2 us.  Bound by that latency and by
// what makes the chain longer, hence (each measured on whole solves): cached
// reads everywhere and queues (2.4x), links by rank instead of by id and the
// far end's count raised before the insertion (together 1.2x on the planted
// cuts, 1.3x on R-MAT), up to four levels' CAS in flight, long rows in pieces
// of 64 (against 256: 1.2x on the 2 x 2^19 cut, whose merged regions become
// rows of 10^5 entries), pieces fetched by whichever warp is free.
//
// Measured against the whole-graph CAPFOREST passes that such rounds needed
// before (whole solves, one GB300): planted cut 2 x 2^19 (n = 1.02 M, m = 21 M)
// 1,340 ms -> 8.8 ms, 2 x 2^15 83 -> 3.3 ms; against PR tests, label
// propagation and concurrent passes: R-MAT scale 20 10-core 3.69 -> 0.87 ms
// (0.73 ms of it here), scale 16 1.13 -> 0.39 ms, random weighted n = 150,001
// (with its creation) 2.25 -> 0.68 ms.
//
// What is left: up to kFoMatrix labels it is summed in a matrix, above that
// listed as it comes.  Measured on the R-MAT scale 20 core (386 labels of 247 K
// vertices): 57 us as four launches of its own, against ~450 us of contraction
// and two host synchronisations; long rows (a first hub stays a vertex of its
// own) go in pieces: by one warp each they took 346 us.
#include <algorithm>
#include <atomic>
#include <climits>

#include "common.cuh"
#include "grid_barrier.cuh"
#include "kernels.h"
#include "launch.h"

namespace mc {

namespace {

constexpr int kFoThreads = 512;
constexpr int kFoPerThread = 32;  // entries per thread that a grid is sized for: more blocks make
                                  // the barriers dearer (2 x 2^15 cut: 3.7 ms, 4.0 with the
                                  // whole GPU) and keep other streams' solves waiting
// Up to kFoFew blocks, whose barriers are cheap, are sized for kFoFewPerThread
// entries a thread on graphs of at most kFoSparse entries per vertex, else one
// block's while they are small: wheel of 4,097 and unit weights 523 -> 415 us
// whole, torus of 60 x 60 656 -> 335, random n = 20,000 of degree 3 553 -> 390;
// 16 blocks or 8 entries 0-10% slower.  Not on denser ones: more warps insert
// more out of order, and a small planted cut (2 x 2^10) loses its joins (2.5 -> 3.1 ms).
constexpr int kFoFewPerThread = 4;
constexpr int kFoFew = 32;
constexpr int kFoSparse = 8;
constexpr int kFoChunk = 64;      // entries of a row handled by one warp at a time
constexpr int kFoOwnPieces = 4;  // pieces of a row that its own thread lists
constexpr int kFoMaxK = 254;      // levels (histogram bins: k + 1)
constexpr int kFoLevels = 8;      // levels wanted where the weights allow it (qsoft): fewer
                                  // unions, and on random weights 1..100 all of the joins
constexpr int kFoBatches = 100;   // from this batch on, everything left is one batch
constexpr int kFoFrac = 12;       // a batch takes at least 1 / kFoFrac of the vertices left,
constexpr int kFoTail = 64;       // and at least 1 / kFoTail of all
// A frontier that hardly grows (a cycle's, a wheel's rim, a grid's, a ball's in the
// plane or in space) pays 12 to 20 us a batch for a few vertices until kFoBatches;
// all at once, the forests of such graphs join as much.  So everything left is one batch
// after two in a row that queue less than half as many again as the one before,
// until the queue has once held a kFoWideDiv-th of the vertices (at least kFoThin,
// at most kFoWide).  Whole solves: torus of 300 x 300 and weights 1 to 50 2.64 -> 0.79 ms
// (0.86 without forests), grid of 300 x 300 2.37 -> 0.86 (1.77), grid of 40^3 and
// weights 1 to 20 1.8 -> 0.73 (1.07), 50,000 points of degree 12 2.4 -> 0.65 (0.82),
// 3,000 points 0.84 -> 0.32 (0.43; with a 16th for the 8th 0.84).  Scanning a 64th, a
// 16th or a quarter of the vertices first, to go on from many places, is slower
// (that 300 x 300 grid 1.41, 1.29 and 1.13).  With one level there is no order to
// keep: a tree of 50,000 0.89 -> 0.29.
// Once the queue has been wide it takes kFoThinLate in a row below kFoThin: a scanned
// region's last vertices come in small batches, too, and their prefix cuts lower
// the bound (planted cut 2 x 5,000 with Pareto 1.5 weights 0.80 ms, 1.54 when two were
// enough).  Nor is a larger kFoThin of use: with 256 and 512 the forests of small planted
// cuts (2 x 2^11, 2 x 2^12) join 0.09 instead of 0.2 and need whole-graph passes.
constexpr int kFoThin = 64;
constexpr int kFoThinLate = 6;
constexpr int kFoWideDiv = 8;
constexpr int kFoWide = 2048;
// Vertices sampled, and entries of each; fewer than 1 / kFoAble of them with a
// unit for every level, which a vertex that the last level joins has: no batch is
// scanned (a wheel, whose spokes have no units and whose rim edges have three for
// eight levels: 4,097 vertices 0.65 -> 0.36 ms, 40,001 0.91 -> 0.61; elsewhere no
// change, the sample is taken beside the clearing).  Not "more than a unit for
// every level", which would also spare a wheel of unit weights: that gives up
// R-MAT graphs whose many leaves have just enough (scale 18 with a cycle through
// all 2.4 -> 4.3 ms).
constexpr int kFoSample = 512;
constexpr int kFoSampleRow = 256;
constexpr int kFoAble = 16;
// None either where at least kFoManyLevels levels are asked for and there are
// (by the sampled weights) units per vertex for fewer than kFoUnits / 10 of them: every level
// takes nearly one per vertex before the next gets any, the last joins next to nothing,
// and many levels cost milliseconds (5,000 vertices of degree 200 and weights 1
// to 100 16.4 -> 13.6 ms).  Not with few levels: on graphs as near to regular whose
// minimum cut is a prefix cut, that lowers the bound and the forests join nearly all
// (two random 30-regular graphs of 50,000 vertices joined by 9 edges: 2.5 ms, 108 without).
constexpr int kFoManyLevels = 128;
constexpr int kFoUnits = 6;
constexpr unsigned kFoMain = 128; // tag bit: known to be in the main component of F_{k-1}

constexpr int kFoMaxBlocks = 1024;

struct FoCtl {
  GridBar bar;
  unsigned items;      // work items listed so far
  unsigned main;       // 1 + a vertex of the main component of F_{k-1} (0: none yet)
  int count;           // edges listed of what is left; INT_MAX: not listed
  int able;            // sampled vertices that the last level can join
  unsigned pieces;     // pieces of long rows listed for that
  unsigned long long deg_inv;  // ~(minimum degree)
  int deg_arg_inv;     // INT_MAX - (its smallest vertex)
  int roots[kFoMaxBlocks];     // components by the block that holds their smallest member
  long long alpha;     // cut of the scanned set
  unsigned next[2];    // items fetched in a batch beyond the first deal (by its parity)
  int hist[256];       // unscanned vertices by min(r, k)
};

struct FoArgs {
  int n;
  const int64_t* rp;
  const int* col;
  const void* w;
  const void* deg;
  int* F;              // n * k parent words, vertex-major; -1: root
  long long fcap;      // ints in F
  uint8_t* tag;        // per vertex: the batch it was scanned in (0: not yet), kFoMain
  int* r;              // per vertex: units that met it while unscanned
  int2* items;         // (vertex, chunk of its row)
  int* parent;
  int *L, *flags, *rank;  // labels, 1 per root, its exclusive prefix sum
  // the rest (what the labels leave), when it is asked for: edges listed in
  // (ends, ew), at most ecap; mat: mat_words ints of scratch
  int rest;
  unsigned* ends;
  int* ew;
  int ecap;
  int* mat;
  long long mat_words;
  FoCtl* ctl;
  DevState* st;
  long long spin;
  long long qsoft;     // half the mean weight of the input
};

// A level's union-find, linked by rank: a root's word is -1 - rank, another's
// its parent, and (rank, id) grows from child to parent, so concurrent links
// close no cycle.  (Linked by id instead, the links of one batch build random
// recursive trees, ~ln n deep, and every walk pays their depth.)  All reads
// are cached: a stale word names an ancestor all the same, or an older rank of
// a root; a root's word is read by every thread, and in L2 its one line would
// serve them in turn.  Only the CAS has to see the present.

// Top of x's tree, halving the path: an ancestor and, but for merges this SM
// has not seen yet, the root; val: its word.  Only words that are no root's
// are written, with an ancestor.  F points at vertex 0's word of the level.
__device__ __forceinline__ int fo_root(int* F, int k, int x, int& val) {
  for (;;) {
    int* px = F + (long long)x * k;
    const int p = *px;
    if (p < 0) {
      val = p;
      return x;
    }
    const int g = F[(long long)p * k];
    if (g < 0) {
      val = g;
      return p;
    }
    *px = g;
    x = g;
  }
}

__device__ __forceinline__ int fo_root(int* F, int k, int x) {
  int val;
  return fo_root(F, k, x, val);
}

// Whether x and y are known to be joined at the level (false may be stale).
__device__ __forceinline__ bool fo_joined(int* F, int k, int x, int y) {
  const int a = F[(long long)x * k], b = F[(long long)y * k];
  const int a1 = a < 0 ? x : a, b1 = b < 0 ? y : b;
  if (a1 == b1) return true;
  if (a < 0 && b < 0) return false;
  return fo_root(F, k, x) == fo_root(F, k, y);
}

// Join the trees whose tops x and y (words vx, vy) are, or were when read:
// true when they were separate.
__device__ __forceinline__ bool fo_link(int* F, int k, int x, int vx, int y, int vy) {
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
    const int p = atomicCAS(F + (long long)x * k, vx, y);
    if (p == vx) {
      if (vx == vy) atomicCAS(F + (long long)y * k, vy, vy - 1);
      return true;
    }
    if (p < 0) {  // still a root, of a higher rank
      vx = p;
    } else {
      // this SM held an old word: the store brings the new one into its cache
      // (else every thread that meets it sends its own failing CAS)
      F[(long long)x * k] = p;
      x = fo_root(F, k, p, vx);
    }
  }
}

__device__ __forceinline__ bool fo_join(int* F, int k, int x, int y) {
  int vx, vy;
  x = fo_root(F, k, x, vx);
  y = fo_root(F, k, y, vy);
  return fo_link(F, k, x, vx, y, vy);
}

// Pieces of a row of `len` entries (at least one: it carries the degree).
__device__ __forceinline__ int fo_pieces(long long len) {
  return max(1, (int)((len + kFoChunk - 1) / kFoChunk));
}

// A vertex about to be scanned takes rank 1 where it is still alone.  Of an
// edge's two trees the scanned end's has a top of rank 1 and more then, and an
// unscanned vertex alone is the lesser: it goes under the scanned end's parent
// (or the end itself) without a look at its rank, which a first link need not
// raise either -- all neighbours' links would do that, on one word.  For the
// same reason a long row starts higher, by its length.
__device__ __forceinline__ void fo_scanned(int* F, int k, int v, long long len) {
  int* f = F + (long long)v * k;
  const int word = len > 64 ? -2 - (58 - __clzll(len)) : -2;  // rank 1, + log2(len) - 5
  for (int i0 = 0; i0 < k; i0 += 8) {
    int w[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) w[j] = i0 + j < k ? f[i0 + j] : 0;
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (w[j] == -1) f[i0 + j] = word;
  }
}

// atomicCAS where `on` (0 elsewhere), predicated: under a branch of its own each
// of several waits for the one before (a batch of 2,392 edges of 25 units, 57 us
// with branches, takes 30; one of 293,570 such edges 102 and 64).
__device__ __forceinline__ int fo_cas_if(bool on, int* p, int old, int to) {
  int r = 0;
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.s32 q, %4, 0;\n\t"
      "@q atom.relaxed.gpu.global.cas.b32 %0, [%1], %2, %3;\n\t}"
      : "+r"(r)
      : "l"(p), "r"(old), "r"(to), "r"((int)on)
      : "memory");
  return r;
}

// Insert `units` units of the edge {x, y}, level `guess` tried first; returns
// the units inserted, or -1 if the last level joins x and y already.
__device__ __forceinline__ int fo_insert(int* F, int k, int x, int y, int units, int guess) {
  int lo = 0, hi = guess;  // first level that does not join x and y, in [lo, hi]
  if (fo_joined(F + guess, k, x, y)) {
    if (guess == k - 1) return -1;
    lo = guess + 1;
    hi = k;
    for (int st = 1; lo < hi; st *= 2) {
      const int m = min(hi - 1, lo + st - 1);
      if (!fo_joined(F + m, k, x, y)) {
        hi = m;
        break;
      }
      lo = m + 1;
    }
    if (lo >= k) return -1;
  } else {
    for (int st = 1; lo < hi; st *= 2) {
      const int m = max(lo, hi - st);
      if (fo_joined(F + m, k, x, y)) {
        lo = m + 1;
        break;
      }
      hi = m;
    }
  }
  while (lo < hi) {
    const int m = (lo + hi) >> 1;
    if (fo_joined(F + m, k, x, y)) lo = m + 1;
    else hi = m;
  }
  // up to four levels at a time: where y is alone (fo_scanned), which is most,
  // the levels' round trips go side by side
  const int asked = units;
  int* px = F + (long long)x * k;
  int* py = F + (long long)y * k;
  while (lo < k && units > 0) {
    const int cnt = min(min(units, k - lo), 4);
    int a[4], b[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      a[j] = j < cnt ? px[lo + j] : 0;
      b[j] = j < cnt ? py[lo + j] : 0;
    }
    int p[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) p[j] = fo_cas_if(b[j] == -1, &py[lo + j], -1, a[j] < 0 ? x : a[j]);
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (j < cnt && (p[j] == -1 || fo_join(F + lo + j, k, x, y))) --units;
    lo += cnt;
  }
  return asked - units;
}

// Batch b: the unscanned vertices with min(r, k) >= t are tagged, take their
// ranks and are listed.  (A function of its own: inlined, its loads push the
// scan's registers out.)
__device__ __noinline__ void fo_select(const FoArgs& a, int k, int b, int t, int* s_hist,
                                       unsigned* s_scan, unsigned* s_base) {
  const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
  const int n = a.n;
  int* F = a.F;
  uint8_t* tag = a.tag;
  const int* ru = a.r;
  FoCtl* ctl = a.ctl;
        // (four vertices a thread: a pass over all of them costs its dependent
        // loads and block-wide sums once per 2,048)
        for (long long v0 = (long long)blockIdx.x * (4 * kFoThreads); v0 < n;
             v0 += (long long)gridDim.x * (4 * kFoThreads)) {
          const int v = (int)v0 + 4 * tid;
          int mine = 0;
          unsigned take = 0;
          if (v < n) {
            // (the arrays end on 256-byte boundaries; vertices from n on are ignored)
            const unsigned tg4 = *reinterpret_cast<const unsigned*>(tag + v);
            const int4 r4 = *reinterpret_cast<const int4*>(ru + v);
            if ((tg4 & 127u) == 0 && min(r4.x, k) >= t) take |= 1u;
            if ((tg4 & 0x7f00u) == 0 && min(r4.y, k) >= t) take |= 2u;
            if ((tg4 & 0x7f0000u) == 0 && min(r4.z, k) >= t) take |= 4u;
            if ((tg4 & 0x7f000000u) == 0 && min(r4.w, k) >= t) take |= 8u;
            if (n - v < 4) take &= (1u << (n - v)) - 1u;
            for (unsigned rest = take; rest; rest &= rest - 1) {
              const int x = v + __ffs(rest) - 1;
              const long long len = a.rp[x + 1] - a.rp[x];
              tag[x] = (uint8_t)(tag[x] | (unsigned)b);
              atomicSub(&s_hist[min(ru[x], k)], 1);
              mine += fo_pieces(len);
              fo_scanned(F, k, x, len);
            }
          }
          int incl = mine;
  #pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(FULL, incl, o);
            if (lane >= o) incl += u;
          }
          if (lane == 31) s_scan[wp] = incl;
          __syncthreads();
          unsigned before = 0, total = 0;
  #pragma unroll
          for (int i = 0; i < kFoThreads / 32; ++i) {
            if (i < wp) before += s_scan[i];
            total += s_scan[i];
          }
          if (total) {  // (the same for the whole block)
            if (tid == 0) *s_base = atomicAdd(&ctl->items, total);
            __syncthreads();
            unsigned at = *s_base + before + (unsigned)(incl - mine);
            // (a warp writes a long row's pieces together: by the row's own thread the
            // 4,600 of a contracted vertex took 320 us, and the grid waited)
            for (unsigned any = __ballot_sync(FULL, take != 0); any;
                 any = __ballot_sync(FULL, take != 0)) {
              const int x = v + __ffs(take) - 1;
              const int pieces = take ? fo_pieces(a.rp[x + 1] - a.rp[x]) : 0;
              if (pieces <= kFoOwnPieces)
                for (int c = 0; c < pieces; ++c) __stcg(&a.items[at + c], make_int2(x, c));
              for (unsigned big = __ballot_sync(FULL, pieces > kFoOwnPieces); big; big &= big - 1) {
                const int src = __ffs(big) - 1;
                const int bx = __shfl_sync(FULL, x, src), bp = __shfl_sync(FULL, pieces, src);
                const unsigned ba = __shfl_sync(FULL, at, src);
                for (int c = lane; c < bp; c += 32) __stcg(&a.items[ba + c], make_int2(bx, c));
              }
              at += pieces;
              take &= take - 1;
            }
          }
          __syncthreads();
        }
}

// The quantum that loses little of the weights: half the mean (`half`).  Just
// above half of weights that are nearly all alike, as half their mean is with a few
// heavier ones among them, that drops half of each and the last level joins
// nothing; so where most of a sample (the same in every block) lose 3 tenths and more
// of themselves, the quantum divides the median of it evenly instead, if that is
// larger: planted cut 2 x 2^13 with weights of 10^5 (64-bit) 24.8 -> 2.4 ms.  Not
// always: finer quanta mean more units to insert for the same joins (two 10-regular
// graphs of 20,000 with weights 1 to 5 0.97 -> 1.34 ms so; Pareto 1.2 weights on the
// planted cut 1.5 -> 2.6 ms by half the median).
__device__ __forceinline__ long long fo_quantum(unsigned long long x, long long half,
                                                unsigned* s_scan) {
  const int tid = threadIdx.x;
  if (__syncthreads_count((x % (unsigned long long)half) * 10 >= 3 * x) * 10 < 6 * kFoThreads)
    return half;
  int bits = __reduce_max_sync(FULL, 64 - __clzll((long long)x));
  if ((tid & 31) == 0) s_scan[tid >> 5] = (unsigned)bits;
  __syncthreads();
  for (int i = 0; i < kFoThreads / 32; ++i) bits = max(bits, (int)s_scan[i]);
  // the largest value that half of the sample reaches, bit by bit
  unsigned long long v = 0;
  for (int b = bits - 1; b >= 0; --b)
    if (__syncthreads_count(x >= (v | 1ull << b)) * 2 >= kFoThreads) v |= 1ull << b;
  __syncthreads();
  const long long typical = (long long)v;
  return typical > half ? typical / ((typical + half - 1) / half) : half;
}

constexpr int kFoMatrix = 1024;  // labels that are summed in a matrix
constexpr int kFoPiece = 512;    // entries of a long row that one warp lists

// Entries [b, e) of a vertex of label u, by one warp.
template <typename WT>
__device__ __noinline__ void fo_collect(const FoArgs& a, int u, long long b, long long e, int skip,
                                        bool matrix, int n2, const WT* w) {
  const int lane = threadIdx.x & 31;
  for (long long p0 = b; p0 < e; p0 += 32) {
    int x = u;
    if (p0 + lane < e) x = a.L[a.col[p0 + lane]];
    const bool keep = x == skip || u < x;  // between two others: from the smaller label
    if (matrix) {
      if (keep) atomicAdd(&a.mat[min(u, x) * n2 + max(u, x)], (int)w[p0 + lane]);
      continue;
    }
    const unsigned bal = __ballot_sync(FULL, keep);
    if (!bal) continue;
    int at = 0;
    if (lane == 0) at = atomicAdd(&a.ctl->count, __popc(bal));
    at = __shfl_sync(FULL, at, 0) + __popc(bal & lanemask_lt());
    if (keep && at < a.ecap) {
      a.ends[at] = (unsigned)u | ((unsigned)x << 16);
      a.ew[at] = (int)w[p0 + lane];
    }
  }
}

// (two blocks per SM, stated: without the 2 the compiler takes the same 64
// registers and spills 664 bytes, with it 8, or 12 for 64-bit weights)
template <typename WT>
__global__ void __launch_bounds__(kFoThreads, 2) forest_kernel(FoArgs a) {
  __shared__ int s_hist[256];   // this block's changes since the last flush
  __shared__ int s_all[256];
  __shared__ unsigned s_scan[kFoThreads / 32];
  __shared__ unsigned s_base;
  __shared__ int s_ok, s_t, s_left, s_main;
  __shared__ int2 s_q[kFoThreads / 32][64];      // queued edges of each warp
  __shared__ uint8_t s_qu[kFoThreads / 32][64];  // and their units
  __shared__ long long s_alpha[kFoThreads / 32];
  // the block's view of the round (the same in all of them): bound, minimum
  // degree, smallest prefix cut and the batch it ends with
  __shared__ long long s_lam, s_best;
  __shared__ unsigned long long s_dmin;
  __shared__ int s_best_batch;
  const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
  const int n = a.n;
  const int gtid = blockIdx.x * kFoThreads + tid, gsize = gridDim.x * kFoThreads;
  const WT* __restrict__ w = reinterpret_cast<const WT*>(a.w);
  const WT* __restrict__ deg = reinterpret_cast<const WT*>(a.deg);
  FoCtl* ctl = a.ctl;
  unsigned gen = 0;
  const long long M = a.rp[n];
  const unsigned long long sample = M > 0 ? (unsigned long long)w[tid * M / kFoThreads] : 0;
  const long long qsoft = fo_quantum(sample, a.qsoft, s_scan);
  // ---- degree bound (Sec. 2.1), and a clean round state
  const long long lam_in = (long long)*(volatile unsigned long long*)&a.st->lambda;
  unsigned long long dmin = ~0ull;
  for (int v = gtid; v < n; v += gsize) {
    a.parent[v] = v;  // nothing joined, however this ends
    dmin = min(dmin, (unsigned long long)(long long)deg[v]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) dmin = min(dmin, __shfl_xor_sync(FULL, dmin, o));
  if (lane == 0) s_alpha[wp] = (long long)dmin;
  __syncthreads();
  if (tid == 0) {
    for (int i = 1; i < kFoThreads / 32; ++i) dmin = min(dmin, (unsigned long long)s_alpha[i]);
    atomicMax(&ctl->deg_inv, ~dmin);
    if (blockIdx.x == 0) {
      DevState* st = a.st;
      st->marks_pr = 0;
      st->marks_cf = 0;
      st->emit_count = 0;
      st->lp_val = ~0ull;
      st->lp_label = -1;
      st->cf_val = ~0ull;
      st->cf_pass = -1;
      st->cf_len = 0;
      st->cf_nscanned = 0;
      st->cf_nmarks = 0;
      st->claimed = 0;
      ctl->count = INT_MAX;
    }
  }
  if (!grid_barrier(&ctl->bar, ++gen, a.spin, &s_ok, a.st)) return;
  dmin = ~__ldcg(&ctl->deg_inv);
  const long long lam = min(lam_in, (long long)dmin);
  {
    int arg = INT_MAX;
    for (int v = gtid; v < n && arg == INT_MAX; v += gsize)
      if ((unsigned long long)(long long)deg[v] == dmin) arg = v;
    arg = __reduce_min_sync(FULL, arg);
    if (lane == 0) s_scan[wp] = (unsigned)arg;
    __syncthreads();
    if (tid == 0) {
      for (int i = 1; i < kFoThreads / 32; ++i) arg = min(arg, (int)s_scan[i]);
      if (arg != INT_MAX) atomicMax(&ctl->deg_arg_inv, INT_MAX - arg);
    }
  }
  if (tid == 0) {
    s_lam = lam;
    s_dmin = dmin;
    s_best = kInf;
    s_best_batch = 0;
  }
  const int kcap = (int)min((long long)kFoMaxK, a.fcap / n);
  bool scan = n > 2 && lam > 0 && kcap >= 1;  // (else the round stops)
  // (the quantum, like the bound, fits the weight type)
  const WT q = scan ? (WT)max((lam + kcap - 1) / kcap,
                              min(qsoft, (lam + kFoLevels - 1) / kFoLevels))
                    : (WT)1;
  const int k = scan ? (int)((lam + q - 1) / q) : 1;
  if (scan && k >= kFoManyLevels) {
    // units per vertex: M / 2 edges of the sample's mean
    const int units = __reduce_add_sync(FULL, (int)min((unsigned long long)k, sample / (unsigned long long)q));
    if (lane == 0) s_all[wp] = units;  // (s_scan is still read)
    __syncthreads();
    long long sum = 0;
    for (int i = 0; i < kFoThreads / 32; ++i) sum += s_all[i];
    scan = 10 * sum * M >= 2ll * kFoThreads * kFoUnits * k * n;
  }
  if (!scan) {
    if (!grid_barrier(&ctl->bar, ++gen, a.spin, &s_ok, a.st)) return;
    if (gtid == 0) {
      a.st->deg_val = dmin;
      a.st->deg_arg = INT_MAX - ctl->deg_arg_inv;
      a.st->lambda = (unsigned long long)lam;
    }
    return;
  }
  int* F = a.F;
  uint8_t* tag = a.tag;
  int* ru = a.r;
  // ---- vertices with a unit for every level, of a sample
  for (int i = gtid >> 5; i < kFoSample; i += gsize >> 5) {
    const int v = (int)((long long)i * n / kFoSample);
    const long long rb = a.rp[v], re = min((long long)a.rp[v + 1], rb + kFoSampleRow);
    int units = 0;
    for (long long e0 = rb; e0 < re && units < k; e0 += 32) {
      const WT c = e0 + lane < re ? w[e0 + lane] : WT(0);
      units += __reduce_add_sync(FULL, (int)min((WT)k, q == 1 ? c : c / q));
    }
    if (lane == 0 && units >= k) atomicAdd(&ctl->able, 1);
  }
  // ---- every vertex a root at every level, nothing scanned; the first batch
  // is vertex 0
  {
    const long long words = (long long)n * k, quads = words / 4;
    const int4 r4 = make_int4(-1, -1, -1, -1);
    const long long own = (k + 3) / 4;  // (vertex 0's words are set below)
    for (long long i = own + gtid; i < quads; i += gsize) reinterpret_cast<int4*>(F)[i] = r4;
    for (long long i = max(quads, own) * 4 + gtid; i < words; i += gsize) F[i] = -1;
    for (int i = gtid; i < min(own * 4, words); i += gsize) F[i] = i < k ? -2 : -1;
    for (int v = gtid; v < n; v += gsize) {
      tag[v] = v == 0 ? 1 : 0;
      ru[v] = 0;
    }
    for (int i = tid; i < 256; i += kFoThreads) s_hist[i] = 0;
    if (blockIdx.x == 0) {
      const int chunks = fo_pieces(a.rp[1] - a.rp[0]);
      for (int c = tid; c < chunks; c += kFoThreads) __stcg(&a.items[c], make_int2(0, c));
      if (tid == 0) {
        atomicExch(&ctl->items, (unsigned)chunks);
        ctl->hist[0] = n - 1;
      }
    }
  }
  if (!grid_barrier(&ctl->bar, ++gen, a.spin, &s_ok, a.st)) return;
  if (__ldcg(&ctl->able) * kFoAble < kFoSample) {
    if (gtid == 0) {
      a.st->deg_val = dmin;
      a.st->deg_arg = INT_MAX - ctl->deg_arg_inv;
      a.st->lambda = (unsigned long long)lam;
    }
    return;
  }
  unsigned start = 0;
  // (of the thread that chooses the batch)
  int thin = 0, queued_before = 1, wide = 0;
  const int wide_from = min(max(n / kFoWideDiv, kFoThin), kFoWide);
  int rep = -1, main_root = -1;  // a vertex of the main component of the last level, its root
  for (int b = 1;; ++b) {
    if (b > 1) {
      // ---- the batch: the highest r until 1 / kFoFrac of the vertices left
      // are taken; the whole queue if it is smaller; everything left when
      // nothing is queued (another component) or after kFoBatches batches
      for (int i = tid; i < 256; i += kFoThreads) s_all[i] = i <= k ? __ldcg(&ctl->hist[i]) : 0;
      __syncthreads();
      if (wp == 0) {
        int left = 0;
        for (int i = lane; i <= k; i += 32) left += s_all[i];
        left = warp_sum(left);
        if (lane == 0) {
          const int need = max(left / kFoFrac, max(n / kFoTail, 32));
          // (not below half the highest r: a batch that ends where a
          // region ends has that region's cut as its alpha)
          int t = k, acc = s_all[k], low = max(1, k / 2);
          while (t > 1 && acc < need && (acc == 0 || t > low)) {
            const int c = s_all[--t];
            if (acc == 0 && c > 0) low = max(1, t / 2);
            acc += c;
          }
          // a frontier that stays thin never fills a batch: everything left
          const int queued = left - s_all[0];
          wide = max(wide, queued);
          const bool narrow = wide < wide_from;
          thin = queued < (narrow ? wide_from : kFoThin) && 2 * queued < 3 * queued_before ? thin + 1 : 0;
          queued_before = queued;
          if (acc == 0 || thin >= (narrow ? 2 : kFoThinLate) || k == 1 || b >= kFoBatches) t = 0;
          s_t = t;
          s_left = left;
        }
      }
      __syncthreads();
      const int left = s_left, t = s_t;
      rep = (int)*(volatile unsigned*)&ctl->main - 1;
      main_root = rep >= 0 ? fo_root(F + (k - 1), k, rep) : -1;
      // the batches before this one are a proper subset while anything is left
      const long long al = *(volatile long long*)&ctl->alpha;
      if (tid == 0 && left > 0 && al < s_best) {
        s_best = al;
        s_best_batch = b - 1;
      }
      if (left <= 0) break;
      fo_select(a, k, b, t, s_hist, s_scan, &s_base);
      if (!grid_barrier(&ctl->bar, ++gen, a.spin, &s_ok, a.st)) return;
    }
    // ---- scan the batch: a warp walks the entries of a few items (short rows,
    // pieces of long ones) as one list, fetched as warps get free (dealt in
    // turn: 1.15-1.4x the time); the entries that may change a forest queue up in
    // shared memory until a full warp of them can be inserted together
    const unsigned end = *(volatile unsigned*)&ctl->items;
    const unsigned nitems = end - start;
    const unsigned warps = gridDim.x * (kFoThreads / 32);
    unsigned per = 1;
    while (per < 32 && per * 8 * warps <= nitems) per *= 2;
    if (tid == 0) s_main = rep >= 0;
    long long alpha = 0;
    int qn = 0;  // queued edges of this warp
    __syncthreads();
    // (the first ones dealt over the blocks before the warps of a block: the few
    // items of a small batch spread over the SMs, 39 of them 57 -> 53 us)
    unsigned i0 = ((unsigned)wp * gridDim.x + blockIdx.x) * per;
    while (i0 < nitems || qn > 0) {
      int x = -1, len = 0;
      unsigned eb = 0;
      if (lane < (int)per && i0 + lane < nitems) {
        const int2 it = __ldcg(&a.items[start + i0 + lane]);
        x = it.x;
        const unsigned rb = (unsigned)a.rp[x], re = (unsigned)a.rp[x + 1];
        eb = rb + (unsigned)it.y * kFoChunk;
        len = (int)min((unsigned)kFoChunk, re - eb);
        if (it.y == 0) alpha += (long long)deg[x];
      }
      const bool last = i0 >= nitems;
      if (!last && lane == 0) i0 = warps * per + atomicAdd(&ctl->next[b & 1], per);
      i0 = __shfl_sync(FULL, i0, 0);
      int incl = len;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += u;
      }
      const int total = __shfl_sync(FULL, incl, 31);
      const unsigned e_first = eb - (unsigned)(incl - len);  // position 0, as if it were x's
      for (int p0 = 0; p0 < total || last; p0 += 32) {
        if (!last) {
          const int p = p0 + lane;
          int o = 0;  // the item of position p: the first whose inclusive end is above p
#pragma unroll
          for (int stp = 16; stp > 0; stp >>= 1) {
            const int v = __shfl_sync(FULL, incl, o + stp - 1);
            if (v <= p) o += stp;
          }
          const int xx = __shfl_sync(FULL, x, o);
          const unsigned e = __shfl_sync(FULL, e_first, o) + (unsigned)p;
          bool keep = false;
          int y = 0, u = 0;
          if (p < total) {
            y = a.col[e];
            const WT c = w[e];
            const unsigned ty = tag[y], tx = tag[xx];
            const int by = (int)(ty & 127u);
            u = (int)min((WT)k, q == 1 ? c : c / q);
            if (by != 0 && by < b) {  // inserted when y was scanned
              alpha -= 2 * (long long)c;
            } else {
              // both ends in this batch: the smaller id inserts
              if (by == b) alpha -= c;
              keep = u > 0 && !(by == b && xx > y) && !(ty & tx & kFoMain);
            }
          }
          const unsigned bal = __ballot_sync(FULL, keep);
          if (keep) {
            const int at = qn + __popc(bal & lanemask_lt());
            s_q[wp][at] = make_int2(xx, y);
            s_qu[wp][at] = (uint8_t)u;
          }
          qn += __popc(bal);
          __syncwarp();
          if (qn < 32) continue;
        }
        // insert up to 32 queued edges (the last ones of the queue)
        const int take = min(qn, 32);
        qn -= take;
        int from = 0, to = 0;  // y's key before and after, if it changed
        if (lane < take) {
          const int2 xy = s_q[wp][qn + lane];
          const int u = s_qu[wp][qn + lane];
          const int y = xy.y;
          const unsigned ty = tag[y];
          const bool out = (ty & 127u) == 0;
          // y's count goes up first: the edges that meet at y get levels of
          // their own to try (from a count raised after the insertion each
          // would climb past all those in flight: 60 us a batch)
          int g = ru[y];
          if (g < k) {
            g = atomicAdd(&ru[y], u);
            if (out && g < k) {
              from = g;
              to = min(k, g + u);
              if (to == k && !*(volatile int*)&s_main) {
                *(volatile int*)&s_main = 1;
                atomicCAS(&ctl->main, 0u, (unsigned)y + 1u);
              }
            }
            if (g >= k) ru[y] = k;  // (this SM's old copy would bring every edge here)
          }
          if (fo_insert(F, k, xy.x, y, u, min(g, k - 1)) < 0 && main_root >= 0 &&
              fo_root(F + (k - 1), k, y) == main_root) {
            tag[y] = (uint8_t)(ty | kFoMain);
            tag[xy.x] = (uint8_t)(tag[xy.x] | kFoMain);
          }
        }
        // one shared atomic per distinct change, not per lane
        const unsigned change = from < to ? ((unsigned)from << 8) | (unsigned)to : 0u;
        const unsigned same = __match_any_sync(FULL, change);
        if (change && (same & lanemask_lt()) == 0) {
          atomicSub(&s_hist[from], __popc(same));
          atomicAdd(&s_hist[to], __popc(same));
        }
        __syncwarp();
        if (last && qn == 0) break;
      }
    }
    if (blockIdx.x == 0 && tid == 0) ctl->next[(b + 1) & 1] = 0;
    alpha = warp_sum(alpha);
    if (lane == 0) s_alpha[wp] = alpha;
    __syncthreads();
    if (tid == 0) {
      long long sum = 0;
      for (int i = 0; i < kFoThreads / 32; ++i) sum += s_alpha[i];
      if (sum) atomicAdd(reinterpret_cast<unsigned long long*>(&ctl->alpha), (unsigned long long)sum);
    }
    for (int i = tid; i <= k; i += kFoThreads) {
      const int d = s_hist[i];
      if (d) {
        atomicAdd(&ctl->hist[i], d);
        s_hist[i] = 0;
      }
    }
    start = end;
    if (!grid_barrier(&ctl->bar, ++gen, a.spin, &s_ok, a.st)) return;
  }
  // ---- the round's marks: the components of the last level (the last that
  // the bound still asks for: a prefix cut may have lowered it), each under its
  // smallest member (r, done with, holds it per root; a warp's vertices of one
  // root send one atomic)
  const long long best = s_best, lam_end = min(s_lam, best);
  int* Fe = F + (lam_end > 0 ? (int)((lam_end + q - 1) / q) - 1 : 0);
  for (int v = gtid; v < n; v += gsize) ru[v] = INT_MAX;
  if (!grid_barrier(&ctl->bar, ++gen, a.spin, &s_ok, a.st)) return;
  unsigned joined = 0;
  for (int v0 = gtid - lane; v0 < n; v0 += gsize) {
    const int v = v0 + lane;
    const int r = v < n ? fo_root(Fe, k, v) : -1;
    const unsigned same = __match_any_sync(FULL, r);
    if (r >= 0 && (same & lanemask_lt()) == 0) atomicMin(&ru[r], v);
    joined += r >= 0 && r != v;
  }
  if (!grid_barrier(&ctl->bar, ++gen, a.spin, &s_ok, a.st)) return;
  // ---- labels: the components by smallest member; a block counts those of its
  // own run of vertices, then numbers them
  const int per = (int)(((long long)n + gridDim.x - 1) / gridDim.x);
  const int vb = (int)min((long long)n, (long long)blockIdx.x * per), ve = min(n, vb + per);
  int mine = 0;
  for (int v = vb + tid; v < ve; v += kFoThreads) {
    const int p = ru[fo_root(Fe, k, v)];
    a.parent[v] = p;
    mine += p == v;
  }
  mine = __reduce_add_sync(FULL, mine);
  if (lane == 0) s_scan[wp] = (unsigned)mine;
  joined = warp_sum(joined);
  if (lane == 0) s_alpha[wp] = joined;
  __syncthreads();
  if (tid == 0) {
    int sum = 0;
    long long j = 0;
    for (int i = 0; i < kFoThreads / 32; ++i) {
      sum += (int)s_scan[i];
      j += s_alpha[i];
    }
    __stcg(&ctl->roots[blockIdx.x], sum);
    if (j) atomicAdd(&a.st->marks_cf, (unsigned long long)j);
    if (blockIdx.x == 0) {
      a.st->deg_val = s_dmin;
      a.st->deg_arg = INT_MAX - ctl->deg_arg_inv;
      a.st->lambda = (unsigned long long)lam_end;
      if (best < s_lam) {
        a.st->cf_val = (unsigned long long)best;
        a.st->cf_pass = kForestPass;
        a.st->cf_len = s_best_batch;
      }
    }
  }
  if (!grid_barrier(&ctl->bar, ++gen, a.spin, &s_ok, a.st)) return;
  int n2 = 0, base = 0;
  for (int i = tid; i < (int)gridDim.x; i += kFoThreads) {
    const int c = __ldcg(&ctl->roots[i]);
    n2 += c;
    if (i < (int)blockIdx.x) base += c;
  }
  n2 = __reduce_add_sync(FULL, n2);
  base = __reduce_add_sync(FULL, base);
  __syncthreads();
  if (lane == 0) {
    s_all[wp] = n2;
    s_hist[wp] = base;
  }
  __syncthreads();
  n2 = base = 0;
  for (int i = 0; i < kFoThreads / 32; ++i) {
    n2 += s_all[i];
    base += s_hist[i];
  }
  if (gtid == 0) a.st->n_next = n2;
  for (int v0 = vb; v0 < ve; v0 += kFoThreads) {
    const int v = v0 + tid;
    const bool root = v < ve && a.parent[v] == v;
    const unsigned bal = __ballot_sync(FULL, root);
    __syncthreads();
    if (lane == 0) s_scan[wp] = (unsigned)__popc(bal);
    __syncthreads();
    int before = base, total = 0;
    for (int i = 0; i < kFoThreads / 32; ++i) {
      if (i < wp) before += (int)s_scan[i];
      total += (int)s_scan[i];
    }
    if (v < ve) {
      a.flags[v] = root;
      a.rank[v] = before + __popc(bal & lanemask_lt());
    }
    base += total;
  }
  const bool rest = a.rest && n2 >= 2 && n2 <= kSmMaxN;
  const bool matrix = n2 <= kFoMatrix && (long long)n2 * n2 <= a.mat_words;
  if (rest && matrix)
    for (int i = gtid; i < n2 * n2; i += gsize) a.mat[i] = 0;
  if (rest && gtid == 0) ctl->count = 0;
  if (!grid_barrier(&ctl->bar, ++gen, a.spin, &s_ok, a.st)) return;
  for (int v = gtid; v < n; v += gsize) a.L[v] = a.rank[a.parent[v]];
  if (!rest) return;
  if (!grid_barrier(&ctl->bar, ++gen, a.spin, &s_ok, a.st)) return;
  // ---- what is left: the edges between different labels.  Up to kFoMatrix
  // labels they are summed in a matrix, above that listed as they come (count
  // ends above ecap when they do not fit).  Every edge of the largest group also
  // stands in its other end's row, so that group's rows, most of the graph where
  // the forests join nearly everything, are not read: it is estimated from a
  // sample, and any other choice is as correct.
  int* s_cnt = reinterpret_cast<int*>(s_q);
  static_assert(sizeof(s_q) >= kSmMaxN * sizeof(int), "label counts");
  for (int i = tid; i < n2; i += kFoThreads) s_cnt[i] = 0;
  if (tid == 0) s_base = 0;
  __syncthreads();
  // (the same sample in every block, hence the same choice)
  atomicAdd(&s_cnt[a.L[(long long)tid * n / kFoThreads]], 1);
  __syncthreads();
  for (int i = tid; i < n2; i += kFoThreads)
    if (s_cnt[i]) atomicMax(&s_base, ((unsigned)s_cnt[i] << 16) | (unsigned)i);
  __syncthreads();
  const int skip = (int)(s_base & 0xffffu);
  const int gwarp = gtid >> 5, nwarps = gsize >> 5;
  for (long long v0 = (long long)gwarp * 32; v0 < n; v0 += (long long)nwarps * 32) {
    const int v = (int)v0 + lane;
    const int lv = v < n ? a.L[v] : skip;
    unsigned todo = __ballot_sync(FULL, lv != skip);
    if (!matrix && __shfl_sync(FULL, todo ? *(volatile int*)&ctl->count : 0, 0) > a.ecap) break;
    while (todo) {
      const int src = __ffs(todo) - 1;
      todo &= todo - 1;
      const int u = __shfl_sync(FULL, lv, src);
      const long long rb = a.rp[v0 + src], re = a.rp[v0 + src + 1];
      if (re - rb > kFoPiece) {  // a long row goes in pieces, below
        const int np = (int)((re - rb + kFoPiece - 1) / kFoPiece);
        unsigned at = 0;
        if (lane == 0) at = atomicAdd(&ctl->pieces, (unsigned)np);
        at = __shfl_sync(FULL, at, 0);
        for (int i = lane; i < np; i += 32) __stcg(&a.items[at + i], make_int2((int)v0 + src, i));
      } else {
        fo_collect<WT>(a, u, rb, re, skip, matrix, n2, w);
      }
    }
  }
  if (!grid_barrier(&ctl->bar, ++gen, a.spin, &s_ok, a.st)) return;
  const int np = (int)__ldcg(&ctl->pieces);
  for (int i = gwarp; i < np; i += nwarps) {
    if (!matrix && __shfl_sync(FULL, *(volatile int*)&ctl->count, 0) > a.ecap) break;
    const int2 p = __ldcg(&a.items[i]);
    const long long rb = a.rp[p.x] + (long long)p.y * kFoPiece;
    fo_collect<WT>(a, a.L[p.x], rb, min(rb + kFoPiece, (long long)a.rp[p.x + 1]), skip, matrix, n2,
                   w);
  }
  if (!matrix) return;
  if (!grid_barrier(&ctl->bar, ++gen, a.spin, &s_ok, a.st)) return;
  for (int i0 = gtid - lane; i0 < n2 * n2; i0 += gsize) {
    const int i = i0 + lane;
    const int c = i < n2 * n2 ? __ldcg(&a.mat[i]) : 0;
    const unsigned bal = __ballot_sync(FULL, c != 0);
    if (!bal) continue;
    int at = 0;
    if (lane == 0) at = atomicAdd(&ctl->count, __popc(bal));
    at = __shfl_sync(FULL, at, 0) + __popc(bal & lanemask_lt());
    if (c != 0 && at < a.ecap) {
      a.ends[at] = (unsigned)(i / n2) | ((unsigned)(i % n2) << 16);
      a.ew[at] = c;
    }
  }
}

__global__ void side_batch_kernel(uint8_t* side0, const int* __restrict__ map0, int n0,
                                  const uint8_t* __restrict__ tag, int last) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n0; i += gridDim.x * blockDim.x) {
    const int b = (int)(tag[map0[i]] & 127u);
    side0[i] = b >= 1 && b <= last ? 1 : 0;
  }
}

}  // namespace

long long forest_item_cap(long long n, long long M) { return n + M / kFoChunk + 1; }
size_t forest_ctl_bytes() { return sizeof(FoCtl); }

template <typename WT>
cudaError_t forest_marks(const ForestScratch& f, int n, long long M, const int64_t* rp,
                         const int* col, const WT* w, const WT* deg, int* parent, int* L,
                         int* flags, int* rank, long long qsoft, const SmallList* rest, int sms,
                         long long spin, DevState* st, cudaStream_t s, int* launches) {
  static std::atomic<int> known{0};  // (the kernel's, on any sm_103a device)
  int per_sm = known.load(std::memory_order_relaxed);
  if (!per_sm) {
    const cudaError_t e =
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, forest_kernel<WT>, kFoThreads, 0);
    if (e != cudaSuccess) return e;
    per_sm = std::max(1, per_sm);
    known.store(per_sm, std::memory_order_relaxed);
  }
  cudaError_t e = cudaMemsetAsync(f.ctl, 0, sizeof(FoCtl), s);
  if (e != cudaSuccess) return e;
  FoArgs a{};
  a.n = n;
  a.rp = rp;
  a.col = col;
  a.w = w;
  a.deg = deg;
  a.F = f.F;
  a.fcap = f.fcap;
  a.tag = f.tag;
  a.r = f.r;
  a.qsoft = qsoft;
  a.items = f.items;
  a.parent = parent;
  a.L = L;
  a.flags = flags;
  a.rank = rank;
  if (rest) {
    a.rest = 1;
    a.ends = rest->ends;
    a.ew = rest->w;
    a.ecap = rest->cap;
    a.mat = rest->mat;
    a.mat_words = rest->mat_words;
  }
  a.ctl = static_cast<FoCtl*>(f.ctl);
  a.st = st;
  a.spin = spin;
  const long long want =
      (std::max<long long>(M, n) + kFoPerThread * kFoThreads - 1) / (kFoPerThread * kFoThreads);
  const long long few =
      M > (long long)kFoSparse * n
          ? 1
          : std::min<long long>(kFoFew,
                                (std::max<long long>(M, n) + kFoFewPerThread * kFoThreads - 1) /
                                    (kFoFewPerThread * kFoThreads));
  const int blocks = (int)std::max<long long>(
      1, std::min<long long>({std::max(want, few), (long long)sms * per_sm, (long long)kFoMaxBlocks}));
  void* params[] = {&a};
  e = launch_fitting(blocks, [&](int fitting) {
    return cudaLaunchCooperativeKernel((const void*)forest_kernel<WT>, dim3(fitting),
                                       dim3(kFoThreads), params, 0, s);
  });
  if (e != cudaSuccess) return e;
  ++*launches;
  return cudaGetLastError();
}

const int* forest_count(const ForestScratch& f) { return &static_cast<const FoCtl*>(f.ctl)->count; }

cudaError_t side_from_batches(uint8_t* side0, const int* map0, int n0, const uint8_t* tag, int last,
                              int sms, cudaStream_t s, int* launches) {
  side_batch_kernel<<<std::max(1, std::min((n0 + 255) / 256, sms * 8)), 256, 0, s>>>(
      side0, map0, n0, tag, last);
  ++*launches;
  return cudaGetLastError();
}

#define MC_FO_INST(WT)                                                                           \
  template cudaError_t forest_marks<WT>(const ForestScratch&, int, long long, const int64_t*,    \
                                        const int*, const WT*, const WT*, int*, int*, int*,      \
                                        int*, long long, const SmallList*, int, long long,       \
                                        DevState*, cudaStream_t, int*);
MC_FO_INST(int32_t)
MC_FO_INST(int64_t)

}  // namespace mc
