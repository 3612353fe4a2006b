// Optional canonical output order (pc_options.canonical).
//
// The extraction numbers vertices in creation order and emits intersecting
// edges in the order the pairings complete, which varies from run to run.
// With canonical order the result is put in one fixed order after the last
// step: vertices sorted by their packed sign vectors (word 0 most
// significant, each 64-bit word compared as an unsigned number; sign vectors
// are unique under genericity, Section 4.1; equal ones keep their creation
// order), edges renumbered to the new vertex ids and sorted by (smaller
// endpoint, larger endpoint).  Two extractions of the same network and box
// then return identical arrays.
//
// Vertices, up to kRankMax of them: the rank of a vertex is the number of
// vertices that sort before it, counted directly (k_rank_count; n^2 word
// comparisons over the whole chip, no passes).
// More vertices: sign vectors differ early, so the keys are taken from the
// most significant end and only as far as needed.  A level turns the next
// entries of every vertex into a 64-bit key (position of its group of equal
// prefixes, then up to 40 entries in base 3: a code has three values, so 8
// bits hold 5 entries where the packed words hold 4) and radix-sorts (key,
// vertex) with 8-bit digits; equal keys form the next groups.  As soon as no
// group is larger than kGroupMax, each vertex counts the smaller ones of its
// group (k_group_rank).  A pass is three launches over tiles of kTile items:
// digit counts (k_digit_count), one CTA per digit scans its row of tile
// counts (k_digit_scan), and the items move to their places (k_digit_move;
// a warp ranks 32 items at a time with match.any, which keeps the order).
// It moves 12 bytes per item and is bound by launches up to ~1e6 items and by
// the scattered writes beyond.
// Edges: a generic vertex has at most 2D edges, so they are counted per
// smaller endpoint, scattered to its row, and each row is sorted by one
// thread.
// Measured on GB300 (whole pc_canonicalize): 314,640 vertices with 9 words
// and 938,105 edges 54 -> 0.95 ms; 1,813 vertices with 6 words 14.4 -> 0.07 ms
// (an 8-bit sort of every word with one thread per 1024 items before).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <string>

#include "pc_ctx.h"
#include "pc_device.cuh"

namespace pc {

constexpr int kRankMax = 16384;    // counting n^2 pairs beats ~20 radix passes of three launches below this
constexpr int kRankThreads = 256;
constexpr int kTileThreads = 256;
constexpr int kTileRounds = 16;    // items per thread of a radix tile
constexpr int kTile = kTileThreads * kTileRounds;
constexpr size_t kCanonKeep = 16 << 20;  // bytes of scratch a context keeps between calls
constexpr int kGroupMax = 64;      // groups up to this size are ranked by counting

// Exclusive prefix sum of counts[0..m) in place, one CTA of 1024 threads.
__global__ void __launch_bounds__(1024) k_scan_counts(int* counts, long long m) {
  __shared__ int warp_sum[32];
  __shared__ long long carry;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (long long base = 0; base < m; base += 1024) {
    const long long i = base + threadIdx.x;
    const int v = i < m ? counts[i] : 0;
    int x = v;
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) warp_sum[warp] = x;
    __syncthreads();
    if (warp == 0) {
      int w = warp_sum[lane], xx = w;
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, xx, o);
        if (lane >= o) xx += y;
      }
      warp_sum[lane] = xx - w;
    }
    __syncthreads();
    const long long excl = carry + warp_sum[warp] + (x - v);
    if (i < m) counts[i] = static_cast<int>(excl);
    __syncthreads();
    if (threadIdx.x == 1023) carry = excl + v;
    __syncthreads();
  }
}

// Whether vertex u sorts before vertex v by words w0..S-1; equal words: eq.
__device__ __forceinline__ bool words_before(const uint64_t* SIG, long long ld, int w0, int S, long long u,
                                             long long v, bool eq) {
  for (int w = w0; w < S; ++w) {
    const uint64_t a = SIG[(long long)w * ld + u], b = SIG[(long long)w * ld + v];
    if (a != b) return a < b;
  }
  return eq;
}

// rank[v] += vertices of this block's range (blockIdx.y) that sort before v.
__global__ void __launch_bounds__(kRankThreads) k_rank_count(const uint64_t* SIG, long long ld, int S, int n,
                                                             int range, int* rank) {
  __shared__ uint64_t first[kRankThreads];
  const int v = blockIdx.x * kRankThreads + threadIdx.x;
  const int u0 = blockIdx.y * range, u1 = n < u0 + range ? n : u0 + range;
  const uint64_t mine = v < n ? SIG[v] : 0ull;
  int before = 0;
  for (int base = u0; base < u1; base += kRankThreads) {
    if (base + (int)threadIdx.x < u1) first[threadIdx.x] = SIG[base + threadIdx.x];
    __syncthreads();
    const int cnt = u1 - base < kRankThreads ? u1 - base : kRankThreads;
    if (v < n)
      for (int k = 0; k < cnt; ++k) {
        const uint64_t a = first[k];
        if (a < mine) ++before;
        else if (a == mine && base + k != v) before += words_before(SIG, ld, 1, S, base + k, v, base + k < v);
      }
    __syncthreads();
  }
  if (v < n && before) atomicAdd(&rank[v], before);
}

// perm[rank[v]] = v
__global__ void k_inverse(const int* rank, long long n, int* perm) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    perm[rank[i]] = static_cast<int>(i);
}

// Keys of one level: the group's position shifted above the entries
// [k0, k0 + cnt) of the sign vector in order of significance, in base 3.
// Entry k of that order is entry 32 w + (valid entries of word w) - 1 - (k -
// 32 w) of the vector, w = k / 32.  perm == nullptr: the first level (vertex
// i at place i, no groups).
__global__ void k_level_keys(const uint64_t* SIG, long long ld, int P, long long n, int k0, int cnt, int bits,
                             int* perm, const int* group, bool first, uint64_t* key) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    if (first) perm[i] = static_cast<int>(i);
    const long long v = first ? i : perm[i];
    uint64_t trits = 0, word = 0;
    int cw = -1;
    for (int k = k0; k < k0 + cnt; ++k) {
      const int w = k >> 5;
      if (w != cw) {
        word = SIG[(long long)w * ld + v];
        cw = w;
      }
      const int valid = P - 32 * w < 32 ? P - 32 * w : 32;
      trits = 3 * trits + ((word >> (2 * (valid - 1 - (k & 31)))) & 3ull);
    }
    key[i] = first ? trits : ((static_cast<uint64_t>(group[i]) << bits) | trits);
  }
}

// counts[d * ntiles + t] = items of tile t whose digit is d.
__global__ void __launch_bounds__(kTileThreads) k_digit_count(const uint64_t* key, long long n, int shift, int* counts,
                                                              int ntiles) {
  __shared__ int c[256];
  c[threadIdx.x] = 0;
  __syncthreads();
  const long long i0 = (long long)blockIdx.x * kTile + threadIdx.x;
#pragma unroll 4
  for (int r = 0; r < kTileRounds; ++r) {
    const long long i = i0 + r * kTileThreads;
    if (i < n) atomicAdd(&c[(key[i] >> shift) & 255u], 1);
  }
  __syncthreads();
  counts[(long long)threadIdx.x * ntiles + blockIdx.x] = c[threadIdx.x];
}

// One CTA per digit: exclusive scan of its row of tile counts, and its total.
__global__ void __launch_bounds__(256) k_digit_scan(int* counts, int ntiles, int* totals) {
  __shared__ int ws[8];
  int* row = counts + (long long)blockIdx.x * ntiles;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int carry = 0;
  for (int base = 0; base < ntiles; base += 256) {
    const int i = base + threadIdx.x;
    const int v = i < ntiles ? row[i] : 0;
    int x = v;
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) ws[warp] = x;
    __syncthreads();
    int below = 0, all = 0;
    for (int w = 0; w < 8; ++w) {
      if (w < warp) below += ws[w];
      all += ws[w];
    }
    if (i < ntiles) row[i] = carry + below + x - v;
    carry += all;
    __syncthreads();
  }
  if (threadIdx.x == 0) totals[blockIdx.x] = carry;
}

// Moves the tile's items to their places, equal digits in their order.
__global__ void __launch_bounds__(kTileThreads) k_digit_move(const uint64_t* key, const int* val, long long n,
                                                             int shift, const int* offsets, const int* totals,
                                                             int ntiles, uint64_t* key_out, int* val_out) {
  __shared__ int cnt[kTileThreads / 32][256];
  __shared__ int ws[8];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int w = 0; w < 8; ++w) cnt[w][tid] = 0;
  __syncthreads();
  const long long i0 = (long long)blockIdx.x * kTile + warp * (32 * kTileRounds) + lane;
  uint64_t kk[kTileRounds];
  int rk[kTileRounds];
#pragma unroll
  for (int r = 0; r < kTileRounds; ++r) kk[r] = i0 + 32 * r < n ? key[i0 + 32 * r] : 0ull;
#pragma unroll
  for (int r = 0; r < kTileRounds; ++r) {  // rank among the warp's items of the same digit
    const bool in = i0 + 32 * r < n;
    const int d = in ? static_cast<int>((kk[r] >> shift) & 255u) : 256;
    const unsigned peers = __match_any_sync(0xffffffffu, d);
    int base = 0;
    if (in) base = cnt[warp][d];
    __syncwarp();
    rk[r] = base + __popc(peers & ((1u << lane) - 1u));
    if (in && lane == __ffs(peers) - 1) cnt[warp][d] = base + __popc(peers);
    __syncwarp();
  }
  __syncthreads();
  {  // start of (digit tid, warp w): digits below, this digit's earlier tiles, earlier warps
    int x = totals[tid];
    const int v = x;
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) ws[warp] = x;
    __syncthreads();
    int at = x - v + offsets[(long long)tid * ntiles + blockIdx.x];
    for (int w = 0; w < warp; ++w) at += ws[w];
    for (int w = 0; w < 8; ++w) {
      const int c = cnt[w][tid];
      cnt[w][tid] = at;
      at += c;
    }
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kTileRounds; ++r)
    if (i0 + 32 * r < n) {
      const int at = cnt[warp][(kk[r] >> shift) & 255u] + rk[r];
      key_out[at] = kk[r];
      val_out[at] = val[i0 + 32 * r];
    }
}

// Device-wide scans over tiles of 1024 items: an inclusive maximum of the
// group heads' positions (heads of the sorted keys), or an exclusive sum.
// Tile totals first, then the totals' scan (one CTA), then the items.
__device__ __forceinline__ int block_scan_max(int x, int* ws) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o && y > x) x = y;
  }
  if (lane == 31) ws[warp] = x;
  __syncthreads();
  for (int w = 0; w < warp; ++w)
    if (ws[w] > x) x = ws[w];
  __syncthreads();
  return x;
}

__device__ __forceinline__ int head_at(const uint64_t* key, long long i, long long n) {
  return i < n && (i == 0 || key[i] != key[i - 1]) ? static_cast<int>(i) : 0;
}

__global__ void __launch_bounds__(1024) k_head_tiles(const uint64_t* key, long long n, int* last) {
  __shared__ int ws[32];
  const int x = block_scan_max(head_at(key, (long long)blockIdx.x * 1024 + threadIdx.x, n), ws);
  if (threadIdx.x == 1023) last[blockIdx.x] = x;
}

__global__ void __launch_bounds__(1024) k_head_scan(int* last, int ntiles) {  // exclusive maximum, one CTA
  __shared__ int ws[32];
  __shared__ int s_top;
  int carry = 0;
  for (int base = 0; base < ntiles; base += 1024) {
    const int t = base + threadIdx.x;
    const int v = t < ntiles ? last[t] : 0;
    int x = block_scan_max(v, ws);
    if (threadIdx.x == 1023) s_top = x;
    // exclusive: the inclusive value of the thread before
    __shared__ int incl[1024];
    incl[threadIdx.x] = x;
    __syncthreads();
    const int before = threadIdx.x ? incl[threadIdx.x - 1] : 0;
    if (t < ntiles) last[t] = before > carry ? before : carry;
    carry = s_top > carry ? s_top : carry;
    __syncthreads();
  }
}

// group[i] = the place of the first item with item i's key; largest = the
// size of the largest group.
__global__ void __launch_bounds__(1024) k_groups(const uint64_t* key, long long n, const int* last, int* group,
                                                 int* largest) {
  __shared__ int ws[32];
  const long long i = (long long)blockIdx.x * 1024 + threadIdx.x;
  int x = block_scan_max(head_at(key, i, n), ws);
  const int before = last[blockIdx.x];
  if (before > x) x = before;
  int size = 0;
  if (i < n) {
    group[i] = x;
    if (i == n - 1 || key[i + 1] != key[i]) size = static_cast<int>(i) + 1 - x;
  }
  size = __reduce_max_sync(0xffffffffu, size);
  if ((threadIdx.x & 31) == 0 && size > 1) atomicMax(largest, size);
}

// Within a group of equal prefixes (the words before w0 are equal): the
// place of each vertex by counting the group's smaller ones.
__global__ void k_group_rank(const uint64_t* SIG, long long ld, int w0, int S, long long n, const int* perm,
                             const int* group, int* out) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const int g = group[i], v = perm[i];
    int before = 0;
    for (long long j = g; j < n && group[j] == g; ++j)
      if (j != i) before += words_before(SIG, ld, w0, S, perm[j], v, j < i);
    out[g + before] = v;
  }
}

// rank[perm[i]] = i
__global__ void k_rank_of(const int* perm, long long n, int* rank) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    rank[perm[i]] = static_cast<int>(i);
}

// dst[r * n + i] = src[r * ld + perm[i]] for rows r < rows
template <typename T>
__global__ void k_gather_rows(const T* src, long long ld, const int* perm, long long n, int rows, T* dst) {
  const long long total = n * rows;
  for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < total;
       k += (long long)gridDim.x * blockDim.x) {
    const long long r = k / n, i = k % n;
    dst[k] = src[r * ld + perm[i]];
  }
}

template <typename T>
__global__ void k_store_rows(const T* src, long long n, int rows, T* dst, long long ld) {
  const long long total = n * rows;
  for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < total;
       k += (long long)gridDim.x * blockDim.x) {
    const long long r = k / n, i = k % n;
    dst[r * ld + i] = src[k];
  }
}

// The values' rows: dst[i][j] = src[perm[i]][j], j < H.
template <typename T>
__global__ void k_gather_items(const T* src, const int* perm, long long n, int H, T* dst) {
  const long long total = n * H;
  for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < total;
       k += (long long)gridDim.x * blockDim.x)
    dst[k] = src[(long long)perm[k / H] * H + k % H];
}

// Edges renumbered to the vertex ranks, counted per smaller endpoint.
__global__ void k_edge_count(int32_t* EU, int32_t* EW, const int* rank, long long nE, int* count) {
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < nE; e += (long long)gridDim.x * blockDim.x) {
    const int a = rank[EU[e]], b = rank[EW[e]];
    const int lo = a < b ? a : b;
    EU[e] = lo;
    EW[e] = a < b ? b : a;
    atomicAdd(&count[lo], 1);
  }
}

// Exclusive sum over tiles of 1024: tile totals ...
__global__ void __launch_bounds__(1024) k_sum_tiles(const int* count, long long n, int* total) {
  const long long i = (long long)blockIdx.x * 1024 + threadIdx.x;
  __shared__ int ws[32];
  int x = __reduce_add_sync(0xffffffffu, i < n ? count[i] : 0);
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = x;
  __syncthreads();
  if (threadIdx.x < 32) {
    x = __reduce_add_sync(0xffffffffu, ws[threadIdx.x]);
    if (threadIdx.x == 0) total[blockIdx.x] = x;
  }
}

// ... and, after the totals' scan, the items.
__global__ void __launch_bounds__(1024) k_sum_items(int* count, long long n, const int* total) {
  const long long i = (long long)blockIdx.x * 1024 + threadIdx.x;
  __shared__ int ws[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int v = i < n ? count[i] : 0;
  int x = v;
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) ws[warp] = x;
  __syncthreads();
  int at = total[blockIdx.x] + x - v;
  for (int w = 0; w < warp; ++w) at += ws[w];
  if (i < n) count[i] = at;
}

// Each edge's larger endpoint to its row (rows of start; start[v] becomes the
// row's end).
__global__ void k_edge_rows(const int32_t* EU, const int32_t* EW, long long nE, int* start, int32_t* row) {
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < nE; e += (long long)gridDim.x * blockDim.x)
    row[atomicAdd(&start[EU[e]], 1)] = EW[e];
}

// One thread per row: insertion sort (a generic vertex has at most 2D edges),
// and the edges back in order.
__global__ void k_edge_sort(const int* end, long long nV, int32_t* row, int32_t* EU, int32_t* EW) {
  for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < nV; v += (long long)gridDim.x * blockDim.x) {
    const int b = v ? end[v - 1] : 0, e = end[v];
    for (int i = b; i < e; ++i) {
      const int32_t x = row[i];
      int j = i;
      for (; j > b && row[j - 1] > x; --j) row[j] = row[j - 1];
      row[j] = x;
    }
    for (int i = b; i < e; ++i) {
      EU[i] = static_cast<int32_t>(v);
      EW[i] = row[i];
    }
  }
}

}  // namespace pc

using namespace pc;

namespace {

int grid_for(long long n) { return static_cast<int>(std::max<long long>(1, std::min<long long>(4096, (n + 255) / 256))); }

long long tiles_of(long long n) { return (n + kTile - 1) / kTile; }

// Scratch of the vertex sort: two key buffers, a second permutation, tile
// counts, digit totals (also the tiles of the group scan) and one flag.
size_t sort_scratch(long long n) {
  if (n <= kRankMax) return 256;
  return 20ull * n + 4ull * (256 * tiles_of(n) + 256 + 64) + 4ull * ((n + 1023) / 1024);
}

}  // namespace

// Puts the context's result (coordinates, sign words, last-layer values,
// error estimates, edges) in canonical order.  Throws PcError on failure.
void pc_canonicalize(pc_ctx* c) {
  const long long nV = c->nV, nE = c->nE;
  if (nV <= 0) return;
  cudaStream_t s = c->stream;
  const int H = c->net.w[c->net.L], S = c->net.S, Pn = c->net.P;
  const size_t zs = c->net.precision == PC_PREC_FP64 ? 8 : 4;
  const size_t row_bytes = std::max<size_t>({8 * (size_t)c->net.D, 8 * (size_t)S, zs * H, 8});
  const long long vtiles = (nV + 1023) / 1024;
  // one scratch for the three phases: the sort, the rows on their way, the edges' rows
  const size_t edge_bytes = 4ull * nE + 4ull * nV + 4ull * vtiles;
  // perm, rank and the scratch in one buffer, which a context keeps while it is
  // small: the small results are where an allocation per call would show
  auto up = [](size_t x) { return (x + 255) / 256 * 256; };
  const size_t index_bytes = up(sizeof(int) * (size_t)nV);
  const size_t bytes = 2 * index_bytes + std::max<size_t>({sort_scratch(nV), row_bytes * (size_t)nV, edge_bytes});
  if (c->canon_cap < bytes) {
    ctx_free(c, c->canon_buf);
    c->canon_buf = ctx_alloc(c, bytes);
    c->canon_cap = c->canon_buf ? bytes : 0;
    if (!c->canon_buf) throw PcError(PC_ERR_OOM, "canonical order: device allocation failed");
  }
  void* perm = c->canon_buf;
  void* rank = static_cast<char*>(perm) + index_bytes;
  void* work = static_cast<char*>(rank) + index_bytes;
  auto release = [&]() {
    if (c->canon_cap <= kCanonKeep) return;
    ctx_free(c, c->canon_buf);
    c->canon_cap = 0;
  };
  auto check = [&](cudaError_t e) {
    if (e != cudaSuccess) {
      release();
      throw PcError(PC_ERR_CUDA, std::string("canonical order: ") + cudaGetErrorString(e));
    }
  };
  int* P = static_cast<int*>(perm);
  int* R = static_cast<int*>(rank);
  const long long ld = c->Vcap;
  const uint64_t* SIG = static_cast<const uint64_t*>(c->bufs.SIG);
  if (nV <= kRankMax) {
    const int n = static_cast<int>(nV);
    const int gx = (n + kRankThreads - 1) / kRankThreads;
    const int gy = std::max(1, std::min(gx, 8 * c->num_sms / gx));
    const int range = (n + gy - 1) / gy;
    check(cudaMemsetAsync(R, 0, sizeof(int) * nV, s));
    k_rank_count<<<dim3(gx, gy), kRankThreads, 0, s>>>(SIG, ld, S, n, range, R);
    k_inverse<<<grid_for(nV), 256, 0, s>>>(R, nV, P);
    c->launches += 2;
  } else {
    uint64_t* K[2] = {static_cast<uint64_t*>(work), static_cast<uint64_t*>(work) + nV};
    int* V[2] = {P, reinterpret_cast<int*>(K[1] + nV)};
    const int ntiles = static_cast<int>(tiles_of(nV));
    int* counts = V[1] + nV;
    int* totals = counts + 256ll * ntiles;
    int* largest = totals + 256;
    int* last = largest + 64;
    int* group = R;  // the ranks are written at the end
    int gbits = 0, in = 0, w0 = 0;
    while ((1ll << gbits) < nV) ++gbits;
    bool grouped = false;
    for (int k0 = 0; k0 < Pn;) {
      // entries of this level: as many as fit below the group's bits
      const bool first = k0 == 0;
      const int room = first ? 64 : 64 - gbits;
      int cnt = 0, bits = 0;
      for (double v = 1.0; cnt < Pn - k0;) {
        v *= 3.0;
        int b = 0;
        while (b < 64 && std::ldexp(1.0, b) < v) ++b;  // 3^cnt - 1 fits in b bits
        if (b > room || cnt >= 40) break;
        ++cnt;
        bits = b;
      }
      k_level_keys<<<grid_for(nV), 256, 0, s>>>(SIG, ld, Pn, nV, k0, cnt, bits, V[in], group, first, K[in]);
      const int total_bits = bits + (first ? 0 : gbits);
      for (int shift = 0; shift < total_bits; shift += 8) {
        k_digit_count<<<ntiles, kTileThreads, 0, s>>>(K[in], nV, shift, counts, ntiles);
        k_digit_scan<<<256, 256, 0, s>>>(counts, ntiles, totals);
        k_digit_move<<<ntiles, kTileThreads, 0, s>>>(K[in], V[in], nV, shift, counts, totals, ntiles, K[in ^ 1],
                                                     V[in ^ 1]);
        in ^= 1;
        c->launches += 3;
      }
      k0 += cnt;
      w0 = k0 / 32;
      check(cudaMemsetAsync(largest, 0, sizeof(int), s));
      k_head_tiles<<<vtiles, 1024, 0, s>>>(K[in], nV, last);
      k_head_scan<<<1, 1024, 0, s>>>(last, static_cast<int>(vtiles));
      k_groups<<<vtiles, 1024, 0, s>>>(K[in], nV, last, group, largest);
      c->launches += 4;
      check(cudaGetLastError());
      int most = 0;
      check(cudaMemcpyAsync(&most, largest, sizeof(int), cudaMemcpyDeviceToHost, s));
      check(cudaStreamSynchronize(s));
      grouped = most > 1 && k0 < Pn;
      if (!grouped || most <= kGroupMax) break;
    }
    if (grouped) {  // small groups are left (or the entries ran out: equal vertices keep their order)
      k_group_rank<<<grid_for(nV), 256, 0, s>>>(SIG, ld, w0, S, nV, V[in], group, V[in ^ 1]);
      in ^= 1;
      c->launches += 1;
    }
    if (in != 0) check(cudaMemcpyAsync(P, V[1], sizeof(int) * nV, cudaMemcpyDeviceToDevice, s));
    k_rank_of<<<grid_for(nV), 256, 0, s>>>(P, nV, R);
    c->launches += 1;
  }
  check(cudaGetLastError());
  // permute the per-vertex rows
  auto permute = [&](void* base, size_t elem, int nrows) {
    if (!base || nrows <= 0) return;
    const int g = grid_for(nV * nrows);
    if (elem == 8) {
      k_gather_rows<uint64_t><<<g, 256, 0, s>>>(static_cast<const uint64_t*>(base), ld, P, nV, nrows,
                                               static_cast<uint64_t*>(work));
      k_store_rows<uint64_t><<<g, 256, 0, s>>>(static_cast<const uint64_t*>(work), nV, nrows,
                                              static_cast<uint64_t*>(base), ld);
    } else {
      k_gather_rows<uint32_t><<<g, 256, 0, s>>>(static_cast<const uint32_t*>(base), ld, P, nV, nrows,
                                               static_cast<uint32_t*>(work));
      k_store_rows<uint32_t><<<g, 256, 0, s>>>(static_cast<const uint32_t*>(work), nV, nrows,
                                              static_cast<uint32_t*>(base), ld);
    }
  };
  permute(c->bufs.X, 8, c->net.D);
  permute(c->bufs.SIG, 8, c->net.S);
  void* Z = pc_make_state(c).Z[c->net.L - 1];
  if (zs == 8)
    k_gather_items<uint64_t><<<grid_for(nV * H), 256, 0, s>>>(static_cast<const uint64_t*>(Z), P, nV, H,
                                                             static_cast<uint64_t*>(work));
  else
    k_gather_items<uint32_t><<<grid_for(nV * H), 256, 0, s>>>(static_cast<const uint32_t*>(Z), P, nV, H,
                                                             static_cast<uint32_t*>(work));
  check(cudaMemcpyAsync(Z, work, zs * H * nV, cudaMemcpyDeviceToDevice, s));
  if (c->net.precision != PC_PREC_FP64) {
    permute(c->bufs.esc, 4, 1);
    permute(c->bufs.exc, 4, 1);
  }
  check(cudaGetLastError());
  // edges: renumber, then sort by (smaller, larger)
  if (nE > 0) {
    int32_t* EU = static_cast<int32_t*>(c->bufs.E);
    int32_t* EW = EU + c->Ecap;
    int32_t* row = static_cast<int32_t*>(work);
    int* start = row + nE;
    int* total = start + nV;
    check(cudaMemsetAsync(start, 0, sizeof(int) * nV, s));
    k_edge_count<<<grid_for(nE), 256, 0, s>>>(EU, EW, R, nE, start);
    k_sum_tiles<<<vtiles, 1024, 0, s>>>(start, nV, total);
    k_scan_counts<<<1, 1024, 0, s>>>(total, vtiles);
    k_sum_items<<<vtiles, 1024, 0, s>>>(start, nV, total);
    k_edge_rows<<<grid_for(nE), 256, 0, s>>>(EU, EW, nE, start, row);
    k_edge_sort<<<grid_for(nV), 256, 0, s>>>(start, nV, row, EU, EW);
    c->launches += 6;
    check(cudaGetLastError());
  }
  c->launches += 2 * (3 + 2 * (c->net.precision != PC_PREC_FP64));
  const cudaError_t e = cudaStreamSynchronize(s);
  release();
  if (e != cudaSuccess) throw PcError(PC_ERR_CUDA, std::string("canonical order: ") + cudaGetErrorString(e));
}
