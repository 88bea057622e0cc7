// noalloc.cu -- contraction of a small device CSR that allocates no memory.
//
// Some callers cannot allocate device memory: a plug-in running inside a
// host application that owns the whole device pool and forbids other
// allocations, or a latency-critical loop where cudaMalloc's implicit
// synchronisation and latency are not acceptable.  For them this file offers
// mincut_contract_csr_noalloc(): the caller passes the input CSR, the labels
// and the output buffers; every intermediate buffer (offsets and
// counters per label, the entries by label, scan partials, the device status
// block) lives in one file-scope __device__ array of fixed size, which every
// GPU that loads the library keeps until the process exits.
//
// The host cannot use the array's name as a device address, so the first
// call on each device looks the address up with cudaGetSymbolAddress (with
// that device current) and caches it.  Every call shares the one array:
// calls whose work overlaps on the GPU (two streams, two threads) race and
// must be serialised by the caller.
#include <algorithm>
#include <cstring>
#include <mutex>

#include "../../include/mincut.h"
#include "common.cuh"
#include "grid_barrier.cuh"
#include "kernels.h"
#include "launch.h"

using namespace mc;

namespace {

constexpr long long kNaMaxEntries = 1ll << 18;   // directed CSR entries
constexpr long long kNaMaxVertices = 1ll << 18;  // vertices

constexpr size_t a256(size_t x) { return (x + 255) / 256 * 256; }
// Labels of more than kNaWarpRow entries; far labels a block sums at a time.
constexpr int kNaThreads = 512;
constexpr int kNaWarps = kNaThreads / 32;
constexpr int kNaMaxBlocks = 512;
constexpr int kNaWarpRow = 256;                // a label's entries that one warp sorts
constexpr int kNaRow = kNaWarpRow * kNaWarps;  // that a block sorts
constexpr int kNaChunk = 2 * kNaRow;           // far labels of one dense sum
constexpr int kNaMids = (int)(kNaMaxEntries / kNaWarpRow);
constexpr int kNaChunks = (int)(kNaMaxVertices / kNaChunk);

struct NaHead {  // zeroed before the launch, read back after it
  GridBar bar;
  unsigned long long wsum;
  unsigned bad;  // a malformed input
  int nmid;      // labels of more than kNaWarpRow entries, listed in mid
  int m2;
};

struct NaCtl {
  NaHead h;
  int tot[2][kNaMaxBlocks];
  int mid[kNaMids];
  int cnt[kNaMids * kNaChunks];  // distinct far labels of a listed label and chunk
};

constexpr size_t kRow = a256((kNaMaxVertices + 1) * 4);
constexpr size_t kOffOff = 0;
constexpr size_t kOffUoff = kOffOff + kRow;
constexpr size_t kOffCur = kOffUoff + kRow;
constexpr size_t kOffUcnt = kOffCur + kRow;
constexpr size_t kOffSegL = kOffUcnt + kRow;
constexpr size_t kOffSegW = kOffSegL + a256(kNaMaxEntries * 4);
constexpr size_t kOffState = kOffSegW + a256(kNaMaxEntries * 4);
constexpr size_t kOffCtl = kOffState + a256(sizeof(DevState));
constexpr size_t kScratchBytes = kOffCtl + a256(sizeof(NaCtl));  // about 6.4 MB

static __device__ __align__(256) unsigned char g_noalloc_scratch[kScratchBytes];

std::mutex g_mu;
unsigned char* g_scratch_ptr[128] = {};

int na_fail(int status, const char* msg) {
  set_last_error(msg);
  return status;
}

// ---- the whole contraction as one cooperative kernel: check, count per label,
// offsets, scatter by label, sort and sum of each label's row, offsets, copy.
// Bound by its seven barriers (~3 us each), the gathers between them, the launch
// and the one read back: the input is read three times from L2 and the DRAM
// floor is below a microsecond.  The form before it (a pass of checks, then
// relabelled pairs through the radix sort and the CSR builder: 13 launches and
// three host reads in turn) took 212 us on 15,001 vertices, 240 K entries
// and 3,750 labels; this one takes 90.
//
// A row of up to kNaWarpRow entries is sorted by one warp in shared memory, a
// longer one by a block's dense sum over the far labels, kNaChunk at a time
// (at most 64 rows can exceed kNaRow entries, so many chunks stay cheap), run
// twice: to count, then to write.  With several chunks and a row that a block
// can sort, the block sorts it: the chunks' scans would cost more than the row.
struct NaArgs {
  int n, n2, M;
  const int64_t* rp;
  const int32_t *col, *w, *lab;
  int *off, *cur, *ucnt, *uoff;  // n2 + 1 each
  int *seg_l, *seg_w;            // M each: entries by label (far label, weight)
  int64_t* rp_out;
  int32_t *col_out, *w_out;
  NaCtl* ctl;
  DevState* st;
  long long spin;
};

// Exclusive prefix sums of in[0 .. n) to out[0 .. n], each block over its own
// run [beg, end); one barrier between the totals and the sums.  A block may use
// its own run's sums at once.
__device__ __forceinline__ bool na_scan(const NaArgs& a, const int* in, int* out, int n, int* tot, unsigned& gen,
                        int* s_ok, int* s_warp, int* beg, int* end) {
  const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
  const int per = (n + gridDim.x - 1) / gridDim.x;
  const int b = min(n, (int)blockIdx.x * per), e = min(n, b + per);
  *beg = b;
  *end = e;
  int sum = 0;
  for (int i = b + tid; i < e; i += kNaThreads) sum += __ldcg(in + i);
  sum = __reduce_add_sync(FULL, sum);
  if (lane == 0) s_warp[wp] = sum;
  __syncthreads();
  if (tid == 0) {
    int t = 0;
    for (int i = 0; i < kNaWarps; ++i) t += s_warp[i];
    __stcg(&tot[blockIdx.x], t);
  }
  if (!grid_barrier(&a.ctl->h.bar, ++gen, a.spin, s_ok, a.st)) return false;
  int base = 0;
  for (int i = tid; i < (int)blockIdx.x; i += kNaThreads) base += __ldcg(&tot[i]);
  base = __reduce_add_sync(FULL, base);
  __syncthreads();
  if (lane == 0) s_warp[wp] = base;
  __syncthreads();
  base = 0;
  for (int i = 0; i < kNaWarps; ++i) base += s_warp[i];
  for (int i0 = b; i0 < e; i0 += kNaThreads) {
    const int i = i0 + tid;
    const int v = i < e ? __ldcg(in + i) : 0;
    int incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(FULL, incl, o);
      if (lane >= o) incl += u;
    }
    __syncthreads();
    if (lane == 31) s_warp[wp] = incl;
    __syncthreads();
    int before = base, total = 0;
    for (int k = 0; k < kNaWarps; ++k) {
      if (k < wp) before += s_warp[k];
      total += s_warp[k];
    }
    if (i < e) out[i] = before + incl - v;
    base += total;
  }
  if (e == n && b < e && tid == 0) out[n] = base;
  __syncthreads();
  return true;
}

// Sort the len (key, value) pairs by key and sum equal keys, by the threads
// t of a group of G (one warp, or the block); returns the distinct keys.
template <int G>
__device__ __forceinline__ int na_sort_sum(int* key, int* val, int len, int t, int* s_warp) {
  auto sync = [] {
    if (G == 32) __syncwarp();
    else __syncthreads();
  };
  int p2 = 1;
  while (p2 < len) p2 *= 2;
  for (int i = len + t; i < p2; i += G) key[i] = 0x7fffffff;  // (behind every label)
  sync();
  for (int k = 2; k <= p2; k *= 2)
    for (int j = k / 2; j > 0; j /= 2) {
      for (int i = t; i < p2 / 2; i += G) {
        const int x = ((i & ~(j - 1)) << 1) | (i & (j - 1)), y = x + j;
        const int kx = key[x], ky = key[y];
        if ((kx > ky) == ((x & k) == 0)) {
          const int vx = val[x];
          key[x] = ky;
          key[y] = kx;
          val[x] = val[y];
          val[y] = vx;
        }
      }
      sync();
    }
  // runs of equal keys: the head keeps the run, its index is the heads before
  int run = 0;
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  for (int i0 = 0; i0 < len; i0 += G) {
    const int i = i0 + t;
    const int x = i < len ? key[i] : -1, c = i < len ? val[i] : 0;
    const bool head = i < len && (i == 0 || key[i - 1] != x);
    const unsigned bal = __ballot_sync(FULL, head);
    int before = run, total = __popc(bal);
    if (G > 32) {
      if (lane == 0) s_warp[wp] = total;
      __syncthreads();
      total = 0;
      for (int k = 0; k < G / 32; ++k) {
        if (k < wp) before += s_warp[k];
        total += s_warp[k];
      }
    }
    const int at = before + __popc(bal & (lanemask_lt() << 1 | 1u)) - 1;
    sync();  // (all of this stretch is read: at <= i)
    if (head) {
      key[at] = x;
      val[at] = c;
    }
    sync();
    if (i < len && !head) atomicAdd(&val[at], c);
    run += total;
    // the next stretch's first entry looks at its left neighbour's key, which
    // may have been overwritten: keep it where that entry will look
    sync();
    if (t == G - 1 && i < len) key[i] = x;
    sync();
  }
  return run;
}

// Whether a row of len > kNaWarpRow entries is summed over all far labels.
__device__ __forceinline__ bool na_dense(int len, int chunks) {
  return chunks == 1 || len > kNaRow;
}

// s_buf[x] = the weight between the row and far label ch * kNaChunk + x (below
// 2^31: the input's total is).
__device__ void na_dense_sum(const NaArgs& a, int b, int len, int ch, int* s_buf) {
  const int tid = threadIdx.x;
  for (int i = tid; i < kNaChunk; i += kNaThreads) s_buf[i] = 0;
  __syncthreads();
  for (int i = tid; i < len; i += kNaThreads) {
    const unsigned x = (unsigned)(__ldcg(&a.seg_l[b + i]) - ch * kNaChunk);
    if (x < (unsigned)kNaChunk) atomicAdd(&s_buf[x], __ldcg(&a.seg_w[b + i]));
  }
  __syncthreads();
}

__global__ void __launch_bounds__(kNaThreads) noalloc_kernel(NaArgs a) {
  __shared__ int s_buf[kNaChunk];
  __shared__ int s_warp[kNaWarps], s_ok;
  const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
  const int gtid = blockIdx.x * kNaThreads + tid, gsize = gridDim.x * kNaThreads;
  const int gwarp = gtid >> 5, nwarps = gsize >> 5;
  NaCtl* ctl = a.ctl;
  unsigned gen = 0;
  int l_beg, l_end;  // this block's labels in the scans
  // ---- the whole input before anything relies on it
  {
    unsigned long long sum = 0;
    bool bad = false;
    if (a.rp[0] != 0 || a.rp[a.n] != a.M) {  // (every block: M entries may not be there)
      if (gtid == 0) atomicOr(&ctl->h.bad, 2u);
      return;
    }
    for (int v = gtid; v < a.n; v += gsize) {
      const int l = a.lab[v];
      if (l < 0 || l >= a.n2 || a.rp[v] > a.rp[v + 1]) bad = true;
    }
    for (int e = gtid; e < a.M; e += gsize) {
      const int c = a.col[e], x = a.w[e];
      if (c < 0 || c >= a.n || x < 0) bad = true;
      else sum += (unsigned long long)x;
    }
    sum = warp_sum(sum);
    if (lane == 0 && sum) atomicAdd(&ctl->h.wsum, sum);
    if (bad) atomicOr(&ctl->h.bad, 1u);
    for (int l = gtid; l < a.n2; l += gsize) a.cur[l] = 0;
  }
  if (!grid_barrier(&ctl->h.bar, ++gen, a.spin, &s_ok, a.st)) return;
  if (__ldcg(&ctl->h.bad) || __ldcg(&ctl->h.wsum) > 0x7fffffffull) return;
  // ---- entries per label, then their places: a warp takes a run of entries and
  // sends one atomic per label it meets
  const int run = (int)(((long long)a.M + (long long)nwarps * 32 - 1) / ((long long)nwarps * 32)) * 32;
  const int e_beg = (int)min((long long)a.M, (long long)gwarp * run), e_end = min(a.M, e_beg + run);
  for (int pass = 0; pass < 2; ++pass) {
    int row = e_beg < e_end ? row_of(a.rp, 0, a.n, e_beg) : 0;
    for (int e0 = e_beg; e0 < e_end; e0 += 32) {
      const int e = e0 + lane;
      int lu = -1, lv = -1, c = 0;
      if (e < e_end) {
        int lo = row, hi = row + 1;  // the row of e: doubling from the last one, then bisection
        for (int st = 1; hi < a.n && a.rp[hi] <= e; st *= 2) {
          lo = hi;
          hi = min(a.n, hi + st);
        }
        row = row_of(a.rp, lo, hi, e);
        lu = a.lab[row];
        lv = a.lab[a.col[e]];
        c = a.w[e];
      }
      row = __shfl_sync(FULL, row, min(31, e_end - 1 - e0));
      const bool keep = lu != lv && c > 0;
      const unsigned same = __match_any_sync(FULL, keep ? lu : -1);
      const int rank = __popc(same & lanemask_lt());
      int at = 0;
      if (keep && rank == 0) at = atomicAdd(&a.cur[lu], __popc(same));
      if (pass == 0) continue;
      at = __shfl_sync(FULL, at, __ffs(same) - 1) + rank;
      if (keep) {
        __stcg(&a.seg_l[at], lv);
        __stcg(&a.seg_w[at], c);
      }
    }
    if (!grid_barrier(&ctl->h.bar, ++gen, a.spin, &s_ok, a.st)) return;
    if (pass == 0) {
      if (!na_scan(a, a.cur, a.off, a.n2, ctl->tot[0], gen, &s_ok, s_warp, &l_beg,
                   &l_end))
        return;
      for (int l = l_beg + tid; l < l_end; l += kNaThreads) {
        if (__ldcg(&a.cur[l]) > kNaWarpRow) {
          ctl->mid[atomicAdd(&ctl->h.nmid, 1)] = l;
          a.ucnt[l] = 0;
        }
        a.cur[l] = a.off[l];
      }
      if (!grid_barrier(&ctl->h.bar, ++gen, a.spin, &s_ok, a.st)) return;
    }
  }
  // ---- each label's row sorted by the far label, equal ones summed, in place:
  int* wk = s_buf + wp * kNaWarpRow;
  int* wv = wk + kNaRow;
  for (int l = gwarp; l < a.n2; l += nwarps) {
    const int b = __ldcg(&a.off[l]), len = __ldcg(&a.off[l + 1]) - b;
    if (len > kNaWarpRow) continue;
    for (int i = lane; i < len; i += 32) {
      wk[i] = __ldcg(&a.seg_l[b + i]);
      wv[i] = __ldcg(&a.seg_w[b + i]);
    }
    __syncwarp();
    const int u = na_sort_sum<32>(wk, wv, len, lane, s_warp);
    __syncwarp();
    for (int i = lane; i < u; i += 32) {
      __stcg(&a.seg_l[b + i], wk[i]);
      __stcg(&a.seg_w[b + i], wv[i]);
    }
    if (lane == 0) __stcg(&a.ucnt[l], u);
    __syncwarp();
  }
  __syncthreads();
  const int chunks = (a.n2 + kNaChunk - 1) / kNaChunk;
  const int items = __ldcg(&ctl->h.nmid) * chunks;
  for (int it = blockIdx.x; it < items; it += gridDim.x) {
    const int l = __ldcg(&ctl->mid[it / chunks]), ch = it % chunks;
    const int b = __ldcg(&a.off[l]), len = __ldcg(&a.off[l + 1]) - b;
    if (!na_dense(len, chunks)) {
      if (ch) continue;
      for (int i = tid; i < len; i += kNaThreads) {
        s_buf[i] = __ldcg(&a.seg_l[b + i]);
        s_buf[kNaRow + i] = __ldcg(&a.seg_w[b + i]);
      }
      __syncthreads();
      const int u = na_sort_sum<kNaThreads>(s_buf, s_buf + kNaRow, len, tid, s_warp);
      for (int i = tid; i < u; i += kNaThreads) {
        __stcg(&a.seg_l[b + i], s_buf[i]);
        __stcg(&a.seg_w[b + i], s_buf[kNaRow + i]);
      }
      if (tid == 0) __stcg(&a.ucnt[l], u);
      __syncthreads();
      continue;
    }
    na_dense_sum(a, b, len, ch, s_buf);
    int c = 0;
    for (int i = tid; i < kNaChunk; i += kNaThreads) c += s_buf[i] != 0;
    c = __reduce_add_sync(FULL, c);
    if (lane == 0) s_warp[wp] = c;
    __syncthreads();
    if (tid == 0) {
      c = 0;
      for (int k = 0; k < kNaWarps; ++k) c += s_warp[k];
      __stcg(&ctl->cnt[it], c);
      if (c) atomicAdd(&a.ucnt[l], c);
    }
    __syncthreads();
  }
  if (!grid_barrier(&ctl->h.bar, ++gen, a.spin, &s_ok, a.st)) return;
  if (!na_scan(a, a.ucnt, a.uoff, a.n2, ctl->tot[1], gen, &s_ok, s_warp, &l_beg, &l_end))
    return;
  // ---- the contracted CSR (the first write to the caller's arrays)
  for (int l = l_beg + wp; l < l_end; l += kNaWarps) {
    const int b = __ldcg(&a.off[l]), len = __ldcg(&a.off[l + 1]) - b;
    const int o = a.uoff[l], u = __ldcg(&a.ucnt[l]);
    if (len <= kNaWarpRow || !na_dense(len, chunks))
      for (int i = lane; i < u; i += 32) {
        a.col_out[o + i] = __ldcg(&a.seg_l[b + i]);
        a.w_out[o + i] = __ldcg(&a.seg_w[b + i]);
      }
    if (lane == 0) a.rp_out[l] = o;
  }
  if (l_end == a.n2 && l_beg < l_end && tid == 0) {
    const int m2 = a.uoff[a.n2];
    a.rp_out[a.n2] = m2;
    ctl->h.m2 = m2;
  }
  if (items == 0 || !grid_barrier(&ctl->h.bar, ++gen, a.spin, &s_ok, a.st)) return;
  for (int it = blockIdx.x; it < items; it += gridDim.x) {
    const int l = __ldcg(&ctl->mid[it / chunks]), ch = it % chunks;
    const int b = __ldcg(&a.off[l]), len = __ldcg(&a.off[l + 1]) - b;
    if (!na_dense(len, chunks)) continue;
    int o = __ldcg(&a.uoff[l]);
    for (int k = 0; k < ch; ++k) o += __ldcg(&ctl->cnt[it - ch + k]);
    na_dense_sum(a, b, len, ch, s_buf);
    for (int i0 = 0; i0 < kNaChunk; i0 += kNaThreads) {
      const int x = s_buf[i0 + tid];
      const unsigned bal = __ballot_sync(FULL, x != 0);
      if (lane == 0) s_warp[wp] = __popc(bal);
      __syncthreads();
      int before = o;
      for (int k = 0; k < kNaWarps; ++k) {
        if (k < wp) before += s_warp[k];
        o += s_warp[k];
      }
      if (x) {
        const int at = before + __popc(bal & lanemask_lt());
        a.col_out[at] = ch * kNaChunk + i0 + tid;
        a.w_out[at] = x;
      }
      __syncthreads();
    }
  }
}

}  // namespace

extern "C" {

int mincut_contract_csr_noalloc(int64_t n, const int64_t* row_ptr, const int32_t* col,
                                const int32_t* w, int64_t m_directed, const int32_t* labels,
                                int64_t n2, int64_t* row_ptr_out, int32_t* col_out,
                                int32_t* w_out, int64_t* m_out, void* cuda_stream) {
  set_last_error("");
  if (!row_ptr || !labels || !row_ptr_out || !m_out || (m_directed > 0 && (!col || !w)) ||
      (m_directed > 0 && (!col_out || !w_out)))
    return na_fail(MINCUT_ERR_INVALID, "NULL pointer argument");
  if (n < 1 || n2 < 1 || n2 > n || m_directed < 0)
    return na_fail(MINCUT_ERR_INVALID, "need 1 <= n2 <= n and m_directed >= 0");
  if (n > kNaMaxVertices || m_directed > kNaMaxEntries)
    return na_fail(MINCUT_ERR_OVERFLOW,
                   "graph exceeds the fixed scratch: at most 262144 vertices and 262144 "
                   "directed entries");
  cudaStream_t s = (cudaStream_t)cuda_stream;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 128)
    return na_fail(MINCUT_ERR_CUDA, "cudaGetDevice failed");
  unsigned char* base;
  {
    std::lock_guard<std::mutex> lk(g_mu);
    if (!g_scratch_ptr[dev]) {
      void* p = nullptr;
      const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
      if (e != cudaSuccess || !p) return na_fail(MINCUT_ERR_CUDA, "cudaGetSymbolAddress failed");
      g_scratch_ptr[dev] = static_cast<unsigned char*>(p);
    }
    base = g_scratch_ptr[dev];
  }
  // the status block and the kernel's state keep the previous call's contents:
  // clear them; the kernel checks the whole input before it relies on it
  DevState* st = reinterpret_cast<DevState*>(base + kOffState);
  NaCtl* ctl = reinterpret_cast<NaCtl*>(base + kOffCtl);
  NaArgs a{};
  a.n = (int)n;
  a.n2 = (int)n2;
  a.M = (int)m_directed;
  a.rp = row_ptr;
  a.col = col;
  a.w = w;
  a.lab = labels;
  a.off = reinterpret_cast<int*>(base + kOffOff);
  a.uoff = reinterpret_cast<int*>(base + kOffUoff);
  a.cur = reinterpret_cast<int*>(base + kOffCur);
  a.ucnt = reinterpret_cast<int*>(base + kOffUcnt);
  a.seg_l = reinterpret_cast<int*>(base + kOffSegL);
  a.seg_w = reinterpret_cast<int*>(base + kOffSegW);
  a.rp_out = row_ptr_out;
  a.col_out = col_out;
  a.w_out = w_out;
  a.ctl = ctl;
  a.st = st;
  a.spin = 1ll << 22;
  int sms = 0, per_sm = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, noalloc_kernel, kNaThreads, 0) !=
          cudaSuccess)
    return na_fail(MINCUT_ERR_CUDA, "device query failed");
  // two entries a thread: 85 us on the size above in one run; with one 96 (more blocks to
  // wait for at each barrier), with four 90 (longer runs of gathers per warp)
  const long long work = std::max({(long long)n, (long long)m_directed, (long long)1});
  const int blocks = (int)std::min<long long>(
      {(work + 2 * kNaThreads - 1) / (2 * kNaThreads), (long long)sms * std::max(1, per_sm),
       (long long)kNaMaxBlocks});
  void* params[] = {&a};
  struct {  // what comes back: the status block up to the kernel's own totals
    unsigned char bytes[kOffCtl - kOffState + sizeof(NaHead)];
  } back;
  if (cudaMemsetAsync(st, 0, kOffCtl - kOffState + sizeof(NaHead), s) != cudaSuccess ||
      launch_fitting(blocks, [&](int fitting) {
        return cudaLaunchCooperativeKernel((const void*)noalloc_kernel, dim3(fitting),
                                           dim3(kNaThreads), params, 0, s);
      }) != cudaSuccess ||
      cudaMemcpyAsync(&back, st, sizeof(back), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return na_fail(MINCUT_ERR_CUDA, "contraction failed");
  DevState h;
  NaHead hc;
  memcpy(&h, back.bytes, sizeof(h));
  memcpy(&hc, back.bytes + (kOffCtl - kOffState), sizeof(NaHead));
  if (hc.bad & 2u)
    return na_fail(MINCUT_ERR_INVALID, "need row_ptr[0] = 0 and row_ptr[n] = m_directed");
  if (hc.bad)
    return na_fail(MINCUT_ERR_INVALID,
                   "row_ptr decreasing, or column index, weight or label out of range");
  if (hc.wsum > 0x7fffffffull)
    return na_fail(MINCUT_ERR_OVERFLOW,
                   "total weight of the directed entries exceeds 2^31 - 1 (32-bit sums)");
  if (h.error & ERR_TIMEOUT) return na_fail(MINCUT_ERR_DEVICE_TIMEOUT, "a bounded wait ran out");
  if (h.error) return na_fail(MINCUT_ERR_INTERNAL, "device check failed");
  *m_out = hc.m2;
  return MINCUT_OK;
}

}  // extern "C"
