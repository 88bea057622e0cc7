// matrix.cu -- contraction to few vertices through a dense matrix.
//
// When the contracted graph has so few vertices that the upper triangle of
// its weight matrix has at most half as many cells as the graph has entries,
// the entries are added into that triangle (each undirected edge once, from the row of
// its smaller vertex) and the CSR is read off it: two passes over the triangle,
// no pairs, no sort, no per-group accumulators and no host read
// between.  Sorted rows, summed parallel edges, dropped self-loops and zero
// weights come by construction.
#include <algorithm>

#include "common.cuh"
#include "kernels.h"
#include "tiles.cuh"

namespace mc {
namespace {

constexpr int kMatThreads = 256;
// Bytes of a block's own triangles: what the default 48 KB leave beside the
// tile's rows (16,416 bytes), in whole 256.
constexpr int kMatShared = (48 * 1024 - (int)sizeof(TileRowsSmem)) / 256 * 256;
static_assert(kMatShared >= 32000 && kMatShared + sizeof(TileRowsSmem) <= 48 * 1024,
              "own triangles and tile rows share a block's default shared memory");
constexpr size_t kMatHead = 256;   // the ticket, then the row counts

__device__ __forceinline__ int tri(int i, int j) {  // i < j
  return (int)((long long)j * (j - 1) / 2) + i;
}

// mat[c] += x for the lanes with c >= 0.  Where one cell takes much of a warp
// (two large groups), its sum goes out as one atomic: same-word atomics come
// one after another, ~0.5 ns each over the whole chip.  `hot`: the cell last
// found so, looked for first.
template <typename WT>
__device__ __forceinline__ void mat_add(WT* mat, int c, WT x, int& hot) {
  const unsigned act = __ballot_sync(FULL, c >= 0);
  if (!act) return;
  unsigned same = __ballot_sync(FULL, c == hot) & act;
  if (__popc(same) <= 2) {
    hot = __shfl_sync(FULL, c, __ffs(act) - 1);
    same = __ballot_sync(FULL, c == hot);
  }
  if (__popc(same) > 2) {
    const WT t = warp_sum(c == hot ? x : WT(0));
    if ((threadIdx.x & 31) == __ffs(same) - 1) atomic_add_w(&mat[hot], t);
    if (c == hot) c = -1;
  }
  if (c >= 0) atomic_add_w(&mat[c], x);
}

// Adds the entries to the triangle.  Bound by its atomics and by the gathers of
// the far labels, both one L2 sector each (~120 G/s): taking each edge from one
// of its two entries halves both.  Small triangles (copies > 0) are summed per block in
// shared memory first, in up to 32 copies by lane, so that a handful of cells
// does not serialise the chip on a few words; those blocks take several tiles
// each and flush once.
// 65 K vertices, 6.9 M entries to 300: 39 us, against 56 for the accumulator
// rows with twice the atomics.
template <typename WT>
__global__ void __launch_bounds__(kETThreads)
    mat_acc_kernel(int n, long long M, const int64_t* __restrict__ rp, const int* __restrict__ col,
                   const WT* __restrict__ w, const int* __restrict__ L,
                   const int* __restrict__ tile_row, int ntiles, int cells, int copies,
                   WT* __restrict__ mat) {
  __shared__ TileRowsSmem tr;
  extern __shared__ __align__(16) unsigned char s_raw[];
  WT* own = reinterpret_cast<WT*>(s_raw);
  for (int c = threadIdx.x; c < cells * copies; c += kETThreads) own[c] = WT(0);
  const int slot = threadIdx.x & (copies - 1);
  int hot = -1;
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
    __syncthreads();
    tile_rows_load(tr, rp, n, tile_row, ntiles, t);
    const long long e0 = (long long)t * kET;
    int u[kETItems], v[kETItems];
    WT x[kETItems];
#pragma unroll
    for (int k = 0; k < kETItems; ++k) {
      const long long e = e0 + k * kETThreads + threadIdx.x;
      v[k] = e < M ? col[e] : -1;
      u[k] = e < M ? tile_row_of(tr, rp, e) : 0;
    }
#pragma unroll
    for (int k = 0; k < kETItems; ++k) {
      const bool use = v[k] > u[k];
      x[k] = use ? w[e0 + k * kETThreads + threadIdx.x] : WT(0);
      u[k] = use ? L[u[k]] : 0;
      v[k] = use ? L[v[k]] : 0;
    }
#pragma unroll
    for (int k = 0; k < kETItems; ++k) {
      const int c = u[k] == v[k] ? -1 : tri(min(u[k], v[k]), max(u[k], v[k]));
      if (copies) {
        if (c >= 0) atomic_add_w(&own[c * copies + slot], x[k]);
      } else {
        mat_add(mat, c, x[k], hot);
      }
    }
  }
  if (!copies) return;
  __syncthreads();
  for (int c = threadIdx.x; c < cells; c += kETThreads) {
    WT x = 0;
    for (int k = 0; k < copies; ++k) x += own[c * copies + ((k + threadIdx.x) & (copies - 1))];
    if (x != 0) atomic_add_w(&mat[c], x);
  }
}

// The weight between i and j (0 on the diagonal).
template <typename WT>
__device__ __forceinline__ WT mat_at(const WT* mat, int i, int j) {
  if (i == j) return WT(0);
  return i < j ? mat[tri(i, j)] : mat[tri(j, i)];
}

// Neighbours and weighted degree of each row (a block per row); the last block
// done turns the counts into row offsets.
template <typename WT>
__global__ void __launch_bounds__(kMatThreads)
    mat_count_kernel(int n2, const WT* __restrict__ mat, unsigned* ticket, int* cnt,
                     int64_t* __restrict__ rp, WT* __restrict__ deg, int* total) {
  __shared__ int s_warp[kMatThreads / 32];
  __shared__ long long s_sum[kMatThreads / 32];
  __shared__ int s_last;
  const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5, i = blockIdx.x;
  int c = 0;
  long long d = 0;
  for (int j = tid; j < n2; j += kMatThreads) {
    const WT x = mat_at(mat, i, j);
    c += x != 0;
    d += (long long)x;
  }
  c = __reduce_add_sync(FULL, c);
  d = warp_sum(d);
  if (lane == 0) {
    s_warp[wp] = c;
    s_sum[wp] = d;
  }
  __syncthreads();
  if (tid == 0) {
    c = 0;
    d = 0;
    for (int k = 0; k < kMatThreads / 32; ++k) {
      c += s_warp[k];
      d += s_sum[k];
    }
    __stcg(&cnt[i], c);
    deg[i] = (WT)d;
    __threadfence();
    s_last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  int base = 0;
  for (int i0 = 0; i0 < n2; i0 += kMatThreads) {
    const int v = i0 + tid < n2 ? __ldcg(&cnt[i0 + tid]) : 0;
    int incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(FULL, incl, o);
      if (lane >= o) incl += u;
    }
    __syncthreads();
    if (lane == 31) s_warp[wp] = incl;
    __syncthreads();
    int before = base;
    for (int k = 0; k < kMatThreads / 32; ++k) {
      if (k < wp) before += s_warp[k];
      base += s_warp[k];
    }
    if (i0 + tid < n2) rp[i0 + tid] = before + incl - v;
  }
  if (tid == 0) {
    rp[n2] = base;
    *total = base;
  }
}

template <typename WT>
__global__ void __launch_bounds__(kMatThreads)
    mat_write_kernel(int n2, const WT* __restrict__ mat, const int64_t* __restrict__ rp,
                     int* __restrict__ col, WT* __restrict__ w) {
  __shared__ int s_warp[kMatThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5, i = blockIdx.x;
  long long base = rp[i];
  for (int j0 = 0; j0 < n2; j0 += kMatThreads) {
    const int j = j0 + tid;
    const WT x = j < n2 ? mat_at(mat, i, j) : WT(0);
    const unsigned bal = __ballot_sync(FULL, x != 0);
    __syncthreads();
    if (lane == 0) s_warp[wp] = __popc(bal);
    __syncthreads();
    long long at = base + __popc(bal & lanemask_lt());
    for (int k = 0; k < kMatThreads / 32; ++k) {
      if (k < wp) at += s_warp[k];
      base += s_warp[k];
    }
    if (x != 0) {
      col[at] = j;
      w[at] = x;
    }
  }
}

}  // namespace

long long matrix_limit(long long M) { return M < 1024 ? 0 : M; }

template <typename WT>
cudaError_t matrix_contract(int n, long long M, int n2, const int64_t* rp, const int* col,
                            const WT* w, const int* L, const int* tile_row, void* scratch,
                            int64_t* rp2, int* col2, WT* w2, WT* deg2, int* total,
                            cudaStream_t s, int* launches) {
  unsigned char* base = static_cast<unsigned char*>(scratch);
  unsigned* ticket = reinterpret_cast<unsigned*>(base);
  int* cnt = reinterpret_cast<int*>(base + kMatHead);
  const size_t off = kMatHead + ((size_t)n2 * 4 + 255) / 256 * 256;
  WT* mat = reinterpret_cast<WT*>(base + off);
  const int cells = (int)((long long)n2 * (n2 - 1) / 2);
  cudaError_t err = cudaMemsetAsync(base, 0, off + (size_t)cells * sizeof(WT), s);
  if (err != cudaSuccess) return err;
  const int ntiles = (int)((M + kET - 1) / kET);
  // own triangles when they fit and their flush costs at most half an atomic per
  // entry; otherwise one tile per block, straight to the triangle in L2.
  // 4.8 M entries to 45 vertices: 250 us by own triangles, 410 straight; 24 M to
  // 60: 644 and 967; with 90% of the vertices in two groups 717 and 1,943
  int copies = 0, grid = ntiles;
  const int blocks = std::min(ntiles, 4 * num_sms());
  if ((size_t)cells * sizeof(WT) <= kMatShared && (long long)cells * blocks <= M / 2) {
    for (copies = 1; copies < 32 && (size_t)cells * copies * 2 * sizeof(WT) <= kMatShared;)
      copies *= 2;
    grid = blocks;
  }
  if (cells > 0) {
    mat_acc_kernel<WT><<<grid, kETThreads, (size_t)cells * copies * sizeof(WT), s>>>(
        n, M, rp, col, w, L, tile_row, ntiles, cells, copies, mat);
    ++*launches;
    if ((err = cudaGetLastError()) != cudaSuccess) return err;
  }
  mat_count_kernel<WT><<<n2, kMatThreads, 0, s>>>(n2, mat, ticket, cnt, rp2, deg2, total);
  mat_write_kernel<WT><<<n2, kMatThreads, 0, s>>>(n2, mat, rp2, col2, w2);
  *launches += 2;
  return cudaGetLastError();
}

#define MC_INST(WT)                                                                               \
  template cudaError_t matrix_contract<WT>(int, long long, int, const int64_t*, const int*,       \
                                           const WT*, const int*, const int*, void*, int64_t*,    \
                                           int*, WT*, WT*, int*, cudaStream_t, int*);
MC_INST(int32_t)
MC_INST(int64_t)
#undef MC_INST

}  // namespace mc
