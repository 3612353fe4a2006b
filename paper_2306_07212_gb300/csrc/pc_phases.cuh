// The per-neuron steps of edge subdivision (Section 4.2) as device functions.
//
// A layer l (neurons i = 0 .. H-1, global index n = off_l + i, sign entry
// e = m + n) runs as
//
//   phase_decide   (layer start, once) every value z_j of every current
//       vertex gets its final sign: an exact zero is a genericity violation
//       (counted, taken as +); in mixed precision a |z_j| within kappa times
//       its FP32 error estimate is re-decided in FP64 at the exact vertex.
//       The layer's sign codes go into the vertices' sign words.
//   phase_scan0    (layer start, once) step (3) for the whole layer: the
//       neurons that cross an edge are the entries in which its endpoints'
//       sign words are opposite.  nx[e] = the first of them; the edges that
//       neuron 0 crosses are listed as (edge, V+, V-).
//   phase_step     (once per neuron, one grid-wide synchronisation each)
//       steps (4) + (5) for the listed splitting edges of neuron i: new
//       vertex by interpolation (FP64 t and coordinates), the edge split into
//       E+ and E-, the parent 2-faces paired in a hash table; and, looking
//       ahead, step (3) for neuron i + 1: the warp that splits an edge finds
//       the next crossing of its two halves (and lists those that neuron
//       i + 1 crosses), and the edge scan lists every other edge with nx =
//       i + 1.  So each step starts with its splitting edges listed and
//       counted, and the capacity check happens before any write.
//
// The scan of a step reads two bytes per edge.  (Reading every edge's two
// endpoints and gathering their values instead, step after step, was 40 % of
// the loop's time on a net of 1e7 vertices and 5e7 edges: it moved 8 bytes
// per edge from HBM and two 32-byte sectors per edge from L2.)  The
// intersecting edges of a step get their nx one step later (kFresh until
// then): their endpoints' sign words are visible to every CTA only after the
// grid-wide synchronisation; whether neuron i + 1 crosses them is known at
// once from one sign bit in the hash payload.
//
// A new vertex's sign words are written complete when it is created: earlier
// entries from its edge's endpoints, the later neurons of the layer from the
// signs of its interpolated values.  During a layer the sign of a vertex
// w.r.t. a neuron j of the layer is the sign of its stored value z_j (0
// exactly on the folded hyperplane); values and codes are made consistent
// when they are created.
//
// A new vertex whose value for a later neuron of the layer is within the FP32
// filter is queued when it is created and re-decided in FP64 at the step's end
// by its CTA (all its queued vertices together), before anything reads that
// sign: its split's pairing and look-ahead wait for it.
#pragma once

#include "pc_device.cuh"
#include "pc_newton.cuh"

namespace pc {

constexpr int kPairCap = 64;           // intersecting edges a warp buffers before it appends them
constexpr int kLaCap = 64;             // list entries a warp buffers
constexpr int kPendCap = 2048;         // splits a CTA queues for an FP64 re-decision
constexpr int kDecideCap = 2 * kPendCap;  // vertices it queues at the layer start
constexpr int kGroup = 16;             // lanes of a split
constexpr int kSplits = 2 * kWarps;    // splits a CTA works on at a time
constexpr int kPendRounds = 32;        // rounds of splits between two looks at the queue
constexpr int kScanTile = 1024;        // edges a warp scans at a time (4 x 16 bytes of nx per lane)

// nx[e]: the next neuron of the layer (local index) that crosses edge e, or
constexpr uint16_t kNxNone = 0x7fff;    // no neuron left
constexpr uint16_t kNxFresh = 0x7ffe;   // made by the last step's pairing, not known yet
constexpr uint16_t kNxListed = 0x8000;  // in the next step's list already

struct ListEntry {
  int e, p, q;                         // splitting edge, V+, V-
};

struct Smem {
  union {
    int verts[kDecideCap];             // layer start: vertices with a value within the filter
    struct {
      int v0[kPendCap], k[kPendCap];   // splits: new vertex, list position
    } split;
  } pend;
  int4 pairs[kWarps][kPairCap];        // (v_a, v_b, zero ordinals, signs at the next neuron: bit 0 v_a -, bit 1 v_b -)
  ListEntry la[kWarps][kLaCap];        // the warps' list entries for the next neuron
  int lac[kWarps], pc[kWarps], pla[kWarps];
  int npend;
  int tile;                            // next scan tile of this CTA
  long long pbase, lbase;
  int zlist[kSplits][16];
  float nrl[3 * kMaxWidth];            // the layer's per-neuron norms (NetDesc::nrm)
  int nrl_layer;                       // layer staged in nrl, -1: none
  long long acc[4];
};

template <typename ZT>
__device__ __forceinline__ ZT tiny_value() {
  return ZT(1e-30);
}

// bit 2k of the result = bit k of m
__device__ __forceinline__ uint64_t spread_even(uint32_t m) {
  uint64_t x = m;
  x = (x | (x << 16)) & 0x0000FFFF0000FFFFull;
  x = (x | (x << 8)) & 0x00FF00FF00FF00FFull;
  x = (x | (x << 4)) & 0x0F0F0F0F0F0F0F0Full;
  x = (x | (x << 2)) & 0x3333333333333333ull;
  x = (x | (x << 1)) & 0x5555555555555555ull;
  return x;
}

// Bits of word w that hold entries < e_end.
__device__ __forceinline__ uint64_t entries_below(int w, int e_end) {
  const int cnt = e_end - 32 * w;
  if (cnt <= 0) return 0ull;
  if (cnt >= 32) return ~0ull;
  return (1ull << (2 * cnt)) - 1ull;
}

// Vertex and edge counts at the start of step n.
__device__ __forceinline__ bool step_counts(const State& st, int n, long long& nV, long long& nE) {
  const Counters* prev = st.cnt + n;
  nV = prev->nV_before + prev->nsplit;
  nE = prev->pruned_e1 > 0 ? prev->pruned_e1 - 1 : prev->nE_before + prev->nsplit + prev->npairs;
  return nV >= 0 && nV <= st.Vcap && nE >= 0 && nE <= st.Ecap;
}

__device__ __forceinline__ void list_store(int32_t* list, long long Ecap, long long k, const ListEntry& x) {
  list[k] = x.e;
  list[Ecap + k] = x.p;
  list[2 * Ecap + k] = x.q;
}

// Appends the warp's buffered entries to the list with one atomic.
__device__ __forceinline__ void warp_flush(const State& st, const ListEntry* la, int& lac, int32_t* list,
                                           long long* counter) {
  const int lane = threadIdx.x & 31;
  __syncwarp();
  long long base = 0;
  if (lane == 0) base = atomic_add_ll(counter, (long long)lac);
  base = __shfl_sync(0xffffffffu, base, 0);
  if (base + lac <= st.Ecap)  // see warp_flush_pairs
    for (int t = lane; t < lac; t += 32) list_store(list, st.Ecap, base + t, la[t]);
  __syncwarp();
  lac = 0;
}

// One entry (hit) per lane into the warp's buffer, appended when it fills
// (lac: entries held, warp-uniform).  All lanes call it.
__device__ __forceinline__ void warp_list(const State& st, bool hit, const ListEntry& x, ListEntry* la, int& lac,
                                          int32_t* list, long long* counter) {
  const unsigned b = __ballot_sync(0xffffffffu, hit);
  if (!b) return;
  const int n = __popc(b);
  if (lac + n > kLaCap) warp_flush(st, la, lac, list, counter);
  if (hit) la[lac + __popc(b & ((1u << (threadIdx.x & 31)) - 1u))] = x;
  lac += n;
}

// Bit 2r of the result is set iff entry 32 w + r is + in one word and - in
// the other: neuron r separates the two vertices.
__device__ __forceinline__ uint64_t opposite(uint64_t a, uint64_t b) {
  return ((a & (b >> 1)) | (b & (a >> 1))) & kEvenBits;
}

// The first entry in [e_from, e_end) that separates vertices u and v (their
// stored sign words), or -1.
__device__ __forceinline__ int first_opposite(const State& st, long long u, long long v, int e_from, int e_end) {
  for (int w = e_from >> 5; 32 * w < e_end; ++w) {
    uint64_t c = opposite(st.SIG[(long long)w * st.Vcap + u], st.SIG[(long long)w * st.Vcap + v]);
    c &= entries_below(w, e_end) & ~entries_below(w, e_from);
    if (c) return 32 * w + (__ffsll((long long)c) - 1) / 2;
  }
  return -1;
}

// ---------------------------------------------------------------------------
// FP64 re-decision of the values z_j, j >= j_from, of layer l that lie within
// the FP32 filter, for a batch of P vertices at once (the CTA's queued
// vertices).  Each vertex's values are evaluated at its exact position: a
// forward pass in float64 from its stored coordinates through layers 0..l on
// its own piece (activation pattern = its sign words; gradients in float32,
// forward mode), then one Newton step on its zero set moves every value to
// the exact vertex, z + grad . dx (the step is small, so the float32 gradient
// adds only ~1e-7 of it).  Each filtered value is written back with its FP64
// sign.
//
// Bound by GB300's FP64 rate (2 multiply-adds per clock and SM, conversions
// at the same rate) and by the latency of the weights' loads, and it sits on
// the step's critical path, so only what is needed is computed: the inputs of
// a layer are the vertex's active neurons (the others contribute an exact
// zero), its outputs the active neurons and the neurons of the vertex's zero
// set, in layer l only the filtered neurons and the zero set (about a quarter
// of a dense pass; lists per vertex, values stored by list position).  Eight
// lanes share an output, a fixed number, so that each value's summation order
// does not depend on how vertices are batched; the batch pays one chain of
// per-layer latency.  The D x D Newton system is solved by one warp per
// vertex, a row per lane (newton_warp).
// Measured on GB300, what the re-decisions add to the neuron loop: 1.9 -> 1.6
// ms on a 3-64x4-1 net (88 steps with re-decisions), 7.7 -> 4.3 ms on a
// 2-128x4-1 net (236 such steps), dense pass -> this.
// Workspace (dynamic shared memory), rd_layout(P, mw, D, S) bytes:
struct RdLayout {
  size_t a, an, A, gv, dlt, sig, J, Jn, sc, zl, nz, ok, li, cnt, total;
};
// Neurons in a vertex's lists over all layers: the net's neurons (at most 32 S).
__host__ __device__ inline RdLayout rd_layout(int P, int mw, int D, int S) {
  RdLayout r{};
  size_t o = 0;
  auto take = [&](size_t bytes) {
    const size_t at = o;
    o += (bytes + 15) / 16 * 16;
    return at;
  };
  r.a = take((size_t)P * mw * 8);       // activations (float64) [P][mw], by list position
  r.an = take((size_t)P * mw * 8);      // next layer's
  r.A = take((size_t)P * D * D * 8);    // Newton rows [P][D][D]
  r.gv = take((size_t)P * D * 8);       // their values [P][D]
  r.dlt = take((size_t)P * D * 8);      // Newton steps [P][D]
  r.sig = take(0);                      // sign words: none, they become the lists below
  r.J = take((size_t)P * mw * D * 4);   // gradients (float) [P][mw][D], by list position
  r.Jn = take((size_t)P * mw * D * 4);
  r.sc = take((size_t)P * mw * 4);      // sums of |terms| of layer l [P][mw]
  r.zl = take((size_t)P * D * 4);       // zero entries [P][D]
  r.nz = take((size_t)P * 4);           // zero entries found
  r.ok = take((size_t)P * 4);           // Newton step taken
  r.li = take((size_t)P * 32 * S * 2);  // outputs of each layer from off_k on: active (filtered) ones, then the zero set's
  r.cnt = take((size_t)P * kMaxL * 4);  // per layer: active (filtered) outputs, and 16 bits up all outputs
  r.total = o;
  return r;
}
constexpr int kRdSmemBudget = 48 * 1024;  // shared memory for a batch
constexpr int kRdSmemMax = 64 * 1024;     // launch attribute of the kernels that hold it
constexpr int kRdLanes = 8;               // lanes per output

// Vertices per batch: half the CTA's warps (a queue rarely holds more), fewer
// when the workspace would exceed the budget (wide layers, large D).
__host__ inline int rd_batch_size(int mw, int D, int S) {
  int P = kWarps / 2;
  while (P > 1 && rd_layout(P, mw, D, S).total > (size_t)kRdSmemBudget) --P;
  return P;
}

template <typename ZT>
__device__ __noinline__ void redecide_batch(const NetDesc& net, const State& st, const int* vs, int P, int l,
                                            int e_end, int j_from, int mw, unsigned char* ws) {
  const int D = net.D, S = net.S, m = net.m;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long Vcap = st.Vcap;
  const RdLayout L = rd_layout(P, mw, D, S);
  double* a = reinterpret_cast<double*>(ws + L.a);
  double* an = reinterpret_cast<double*>(ws + L.an);
  double* A = reinterpret_cast<double*>(ws + L.A);
  double* gv = reinterpret_cast<double*>(ws + L.gv);
  double* dlt = reinterpret_cast<double*>(ws + L.dlt);
  float* J = reinterpret_cast<float*>(ws + L.J);
  float* Jn = reinterpret_cast<float*>(ws + L.Jn);
  float* sc = reinterpret_cast<float*>(ws + L.sc);
  int* zl = reinterpret_cast<int*>(ws + L.zl);
  int* nzs = reinterpret_cast<int*>(ws + L.nz);
  int* oks = reinterpret_cast<int*>(ws + L.ok);
  uint16_t* lists = reinterpret_cast<uint16_t*>(ws + L.li);  // [P][32 S]
  int* cnt = reinterpret_cast<int*>(ws + L.cnt);             // [P][kMaxL]
  const int ln = 32 * S;
  ZT* Z = static_cast<ZT*>(st.Z[l]);
  const int HL = net.w[l + 1];
  // Sign words, zero set, coordinates and the layers' output lists of each
  // vertex: one warp for a (vertex, layer), all at once (a layer's list does
  // not depend on the layers before it).
  for (int x = warp; x < P * (l + 1); x += kWarps) {
    const int q = x / (l + 1), k = x - q * (l + 1);
    const long long v = vs[q];
    const int H = net.w[k + 1], nk = net.off[k], ebase = m + nk;
    uint64_t word = lane < S ? __ldcg(st.SIG + (long long)lane * Vcap + v) : 0ull;
    double xd = 0.0;
    if (k == 0 && lane < D) xd = st.X[(long long)lane * Vcap + v];
    const float esc = k == l ? st.esc[v] : 0.f;
    uint16_t* out = lists + q * ln + nk;
    int n = 0;
    unsigned zeros[kMaxWidth / 32];
#pragma unroll
    for (int h = 0; h < kMaxWidth / 32; ++h) {
      if (32 * h >= H) break;
      const int r = 32 * h + lane, entry = ebase + r;
      const uint64_t w0 = __shfl_sync(0xffffffffu, word, (entry >> 5) & 31);
      const uint64_t code = r < H ? (w0 >> (2 * (entry & 31))) & 3ull : 3ull;
      bool first = code == kPlus;
      if (k == l) {
        first = false;
        if (r >= j_from && r < H) {
          const float z32 = static_cast<float>(Z[v * HL + r]);
          first = fabsf(z32) <= net.kappa_sel * (net.nrm[3 * (nk + r)] * esc + 2.9802322e-8f * net.nrm[3 * (nk + r) + 1]);
        }
      }
      const unsigned bf = __ballot_sync(0xffffffffu, first);
      zeros[h] = __ballot_sync(0xffffffffu, code == 0 && entry < e_end);
      if (first) out[n + __popc(bf & ((1u << lane) - 1u))] = (uint16_t)r;
      n += __popc(bf);
    }
    int nn = n;
#pragma unroll
    for (int h = 0; h < kMaxWidth / 32; ++h) {
      if (32 * h >= H) break;
      if ((zeros[h] >> lane) & 1u) out[nn + __popc(zeros[h] & ((1u << lane) - 1u))] = (uint16_t)(32 * h + lane);
      nn += __popc(zeros[h]);
    }
    if (lane == 0) cnt[q * kMaxL + k] = n | (nn << 16);
    if (k == 0) {
      uint64_t zm = lane < S ? zero_mask(word, lane, e_end) : 0ull;
      const int c = __popcll(zm);
      int y = c;
      for (int o = 1; o < 32; o <<= 1) {
        const int z = __shfl_up_sync(0xffffffffu, y, o);
        if (lane >= o) y += z;
      }
      int nz = y - c;
      for (; zm; zm &= zm - 1, ++nz)
        if (nz < D) zl[q * D + nz] = lane * 32 + (__ffsll((long long)zm) - 1) / 2;
      if (lane == 31) nzs[q] = y;
      if (lane < D) {
        a[q * mw + lane] = xd;
        for (int dd = 0; dd < D; ++dd) J[(q * mw + lane) * D + dd] = lane == dd ? 1.f : 0.f;
      }
    }
  }
  __syncthreads();
  int in = D;
  for (int k = 0; k <= l; ++k) {
    const int nk = net.off[k], ebase = m + nk;
    const double* W = net.W64 + net.wofs[k];  // [H][in]
    const float* W32 = net.W32 + net.wofs[k];
    const double* b = net.W64 + net.bofs[k];
    int pairs = 0;
    for (int q = 0; q < P; ++q) pairs += cnt[q * kMaxL + k] >> 16;
    for (int p0 = 0; p0 < pairs; p0 += kBlock / kRdLanes) {
      int x = p0 + threadIdx.x / kRdLanes, q = 0;
      const int s = threadIdx.x % kRdLanes;
      const bool valid = x < pairs;
      if (valid)
        while (x >= (cnt[q * kMaxL + k] >> 16)) x -= cnt[q++ * kMaxL + k] >> 16;  // output x of vertex q
      const int n1 = valid ? cnt[q * kMaxL + k] & 0xffff : 0;
      double acc = 0.0;
      float scl = 0.f, jd[kMaxD];
#pragma unroll
      for (int dd = 0; dd < kMaxD; ++dd) jd[dd] = 0.f;
      const int r = valid ? lists[q * ln + nk + x] : 0;
      double br = 0.0;
      if (valid) {
        if (s == 0) br = b[r];
        const double* wr = W + (long long)r * in;
        const float* wr32 = W32 + (long long)r * in;
        const double* aq = a + q * mw;
        const float* Jq = J + q * mw * D;
        const uint16_t* lq = lists + q * ln + (k > 0 ? net.off[k - 1] : 0);
        const int ci = k > 0 ? cnt[q * kMaxL + k - 1] & 0xffff : D;
#pragma unroll 4
        for (int t = s; t < ci; t += kRdLanes) {
          const int c = k > 0 ? lq[t] : t;
          acc = fma(wr[c], aq[t], acc);
          const float w32 = wr32[c];
          if (k == l) scl = fmaf(fabsf(w32), fabsf(static_cast<float>(aq[t])), scl);
#pragma unroll
          for (int dd = 0; dd < kMaxD; ++dd)
            if (dd < D) jd[dd] = fmaf(w32, Jq[t * D + dd], jd[dd]);
        }
      }
#pragma unroll
      for (int o = kRdLanes >> 1; o > 0; o >>= 1) {  // the lanes of an output are aligned
        acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (k == l) scl += __shfl_xor_sync(0xffffffffu, scl, o);
#pragma unroll
        for (int dd = 0; dd < kMaxD; ++dd)
          if (dd < D) jd[dd] += __shfl_xor_sync(0xffffffffu, jd[dd], o);
      }
      if (valid && s == 0) {
        const double z = acc + br;
        const int entry = ebase + r;
        const int nzc = nzs[q] < D ? nzs[q] : D;
        if (x >= n1)  // a neuron of the zero set
          for (int qq = 0; qq < nzc; ++qq)
            if (zl[q * D + qq] == entry) {
              gv[q * D + qq] = z;
#pragma unroll
              for (int dd = 0; dd < kMaxD; ++dd)
                if (dd < D) A[(q * D + qq) * D + dd] = jd[dd];
            }
        if (x < n1) {
          an[q * mw + x] = z;
          if (k == l) sc[q * mw + x] = scl + fabsf(static_cast<float>(br));
#pragma unroll
          for (int dd = 0; dd < kMaxD; ++dd)
            if (dd < D) Jn[(q * mw + x) * D + dd] = jd[dd];
        }
      }
    }
    __syncthreads();
    double* t0 = a; a = an; an = t0;
    float* t1 = J; J = Jn; Jn = t1;
    in = net.w[k + 1];
  }
  for (int q = warp; q < P; q += kWarps) {  // the Newton step of each vertex
    int* zq = zl + q * D;
    const int nzc = nzs[q] < D ? nzs[q] : D;
    if (net.fA != nullptr) {
      domain_facet_rows(net, st, vs[q], zq, nzc, lane, A + q * D * D, gv + q * D);
      __syncwarp();
    }
    double dl = 0.0;
    const bool ok = nzs[q] == D && newton_warp(net, st, vs[q], zq, A + q * D * D, gv + q * D, dl);
    if (lane == 0) oks[q] = ok;
    if (lane < D) dlt[q * D + lane] = ok ? dl : 0.0;
    __syncwarp();
  }
  __syncthreads();
  // layer l's filtered values (a), gradients (J) and sums of |terms| (sc): decide
  const int n0 = net.off[l];
  for (int q = warp; q < P; q += kWarps) {
    const long long v = vs[q];
    for (int x = lane; x < (cnt[q * kMaxL + l] & 0xffff); x += 32) {
      const int j = lists[q * ln + n0 + x];
      const float z32 = static_cast<float>(Z[v * HL + j]);
      const float est = net.nrm[3 * (n0 + j)] * st.esc[v] + 2.9802322e-8f * net.nrm[3 * (n0 + j) + 1];
      double zs = a[q * mw + x];
      if (oks[q])
        for (int d = 0; d < D; ++d) zs += static_cast<double>(J[(q * mw + x) * D + d]) * dlt[q * D + d];
      const bool und = !oks[q] || fabs(zs) <= 1e-12 * sc[q * mw + x];
      const bool minus = zs < 0.0;
      if (!(fabsf(z32) <= net.kappa * est)) {  // audit band: record a wrong FP32 sign, change nothing
        if ((z32 < 0.f) != minus && !und) {
          atomicAdd(&st.g->missed, 1);
          atomicMax(&st.g->missed_margin_bits, __float_as_int(fabsf(z32) / est));
        }
        continue;
      }
      ZT zz = static_cast<ZT>(zs);
      if (!minus && !(zz > ZT(0))) zz = tiny_value<ZT>();
      if (minus && !(zz < ZT(0))) zz = -tiny_value<ZT>();
      Z[v * HL + j] = zz;
      atomic_add_ll(&st.cnt[n0 + j + 1].nfilter, 1ll);
      if (und) atomic_add_ll(&st.cnt[n0 + j + 1].nundecided, 1ll);
      if ((z32 < 0.f) != minus) {  // the FP32 sign was wrong: its code 01 <-> 10; how close to the filter's edge was it?
        const int entry = m + n0 + j;
        atomicXor(reinterpret_cast<unsigned long long*>(st.SIG) + (long long)(entry >> 5) * Vcap + v,
                  3ull << (2 * (entry & 31)));
        atomicAdd(&st.g->flips, 1);
        atomicMax(&st.g->flip_margin_bits, __float_as_int(est > 0.f ? fabsf(z32) / est : 0.f));
      }
    }
  }
  __syncthreads();
}

// Re-decides np queued vertices in batches of net.rd_batch.
template <typename ZT>
__device__ void drain_pending(const NetDesc& net, const State& st, const int* vs, int np, int l, int e_end, int j_from,
                              int mw, double* ws) {
  for (int q0 = 0; q0 < np; q0 += net.rd_batch) {
    const int P = np - q0 < net.rd_batch ? np - q0 : net.rd_batch;
    redecide_batch<ZT>(net, st, vs + q0, P, l, e_end, j_from, mw, reinterpret_cast<unsigned char*>(ws));
  }
}

// ---------------------------------------------------------------------------
// Sixteen lanes per vertex or split: lane gl of the group holds the values of
// the neurons 64 c + 16 t + gl (t < 4) of a 64-neuron chunk, so that a group
// reads 64 consecutive bytes of a vertex's row at a time, and the sign words
// gl and gl + 16.
__device__ __forceinline__ unsigned group_ballot(bool x) {
  return (__ballot_sync(0xffffffffu, x) >> (threadIdx.x & 16)) & 0xffffu;
}

// The 32 neurons of sign word w among the 64 of chunk c, as bits of mask
// (neuron 64 c + b at bit b); e0: the layer's first entry.
__device__ __forceinline__ uint32_t word_window(uint64_t mask, int w, int c, int e0) {
  const int s = 32 * w - e0 - 64 * c;
  if (s <= -32 || s >= 64) return 0u;
  return static_cast<uint32_t>(s >= 0 ? mask >> s : mask << -s);
}

// The codes of a word's entries from their minus bits.
__device__ __forceinline__ uint64_t codes_of(uint32_t minus) {
  const uint64_t x = spread_even(minus);
  return (x << 1) | (kEvenBits ^ x);
}

// Layer start, step (2) for every current vertex and every neuron of the
// layer (values from the layer-start product, step (1)): one group per
// vertex, or one thread for layers of up to kThinWidth neurons (an output
// layer), where a group would leave most lanes idle (1e7 vertices, one
// neuron: 3.8 ms with a group, 0.95 ms with a thread).
constexpr int kThinWidth = 4;

// The final sign of the layer-start value z of neuron j: exact zeros count as
// degenerate and become tiny (+).  Returns whether it is -; filt: within the
// filter.
template <typename ZT, bool MIXED>
__device__ __forceinline__ bool decide_value(const NetDesc& net, const State& st, int n0, int j, ZT* at, float esc,
                                             bool& filt) {
  ZT z = *at;
  if (z == ZT(0)) {  // on a folded hyperplane it was not created on: not generic
    z = tiny_value<ZT>();
    *at = z;
    atomic_add_ll(&st.cnt[n0 + j + 1].ndegenerate, 1ll);
  }
  if (MIXED)
    filt = filt || fabsf(static_cast<float>(z)) <=
                       net.kappa_sel * (net.nrm[3 * (n0 + j)] * esc + 2.9802322e-8f * net.nrm[3 * (n0 + j) + 1]);
  return z < ZT(0);
}

template <typename ZT, bool MIXED>
__device__ __noinline__ void phase_decide(const NetDesc& net, const State& st, int l, Smem& sm, double* ws, int mw) {
  const int n0 = net.off[l], H = net.w[l + 1];
  long long nV, nE;
  if (!step_counts(st, n0, nV, nE)) {
    if (threadIdx.x == 0) report_corrupt(st.g, 2, n0, nV, nE, st.Vcap);
    return;
  }
  const long long Vcap = st.Vcap;
  ZT* Z = static_cast<ZT*>(st.Z[l]);
  if (threadIdx.x == 0) sm.npend = 0;
  __syncthreads();
  const bool thin = H <= kThinWidth;
  const int gl = threadIdx.x & (kGroup - 1), grp = threadIdx.x / kGroup;
  const int per = thin ? kBlock : kSplits;  // vertices of a CTA's round
  const int looks = kDecideCap / (2 * per);  // rounds between two looks at the queue
  const long long span = (long long)gridDim.x * per;
  const int e0 = net.m + n0, wf = e0 >> 5, wl = (e0 + H - 1) >> 5;
  const long long rounds = (nV + span - 1) / span;
  for (long long rd = 0; rd < rounds; ++rd) {
    const long long v = rd * span + (long long)blockIdx.x * per + (thin ? (int)threadIdx.x : grp);
    const bool in = v < nV;
    bool filt = false;
    const float esc = MIXED && in ? st.esc[v] : 0.f;
    uint32_t minus = 0u;  // of the word w
    const int w = thin ? wf : wf + gl;
    if (thin) {
      uint32_t mask = 0;
      if (in)
        for (int j = 0; j < H; ++j)
          if (decide_value<ZT, MIXED>(net, st, n0, j, Z + v * H + j, esc, filt)) mask |= 1u << j;
      minus = word_window(mask, wf, 0, e0);
      if (in && wl > wf) {  // the entries straddle two words
        const uint32_t m1 = word_window(mask, wl, 0, e0);
        st.SIG[(long long)wl * Vcap + v] = codes_of(m1) & entries_below(wl, e0 + H);
      }
    } else {
      for (int c = 0; 64 * c < H; ++c) {
        uint64_t mask = 0;
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const int j = 64 * c + 16 * t + gl;
          bool mi = false;
          if (in && j < H) mi = decide_value<ZT, MIXED>(net, st, n0, j, Z + v * H + j, esc, filt);
          mask |= static_cast<uint64_t>(group_ballot(mi)) << (16 * t);
        }
        minus |= word_window(mask, w, c, e0);  // at most 9 words hold a layer's entries
      }
    }
    if (in && w <= wl) {
      const uint64_t below = entries_below(w, e0);
      const uint64_t old = below ? st.SIG[(long long)w * Vcap + v] & below : 0ull;
      st.SIG[(long long)w * Vcap + v] = old | (codes_of(minus) & entries_below(w, e0 + H) & ~below);
    }
    if (MIXED) {
      const bool any = thin ? filt : group_ballot(filt) != 0 && gl == 0;
      if (any) sm.pend.verts[atomicAdd(&sm.npend, 1)] = int(v);
      const bool last = rd + 1 == rounds;
      if (last || rd % looks == looks - 1) {
        __syncthreads();
        const int np = sm.npend;
        if (np > 0 && (last || np > kDecideCap / 2)) {
          drain_pending<ZT>(net, st, sm.pend.verts, np, l, e0, 0, mw, ws);
          __syncthreads();
          if (threadIdx.x == 0) sm.npend = 0;
        }
        __syncthreads();
      }
    }
  }
}

// ---------------------------------------------------------------------------
// The code of vertex v at an entry is - (it has a code there).
__device__ __forceinline__ bool minus_at(const State& st, long long v, int entry) {
  return ((st.SIG[(long long)(entry >> 5) * st.Vcap + v] >> (2 * (entry & 31))) & 3ull) == kMinus;
}

// Step (3) for neuron i + 1 (entry e + 1) during step i: lists the edges with
// nx = i + 1 among the first nA, whose nx is known, and finds nx of the
// others (made by the last step's pairing).  The warps of a CTA take its
// tiles (kScanTile known edges or 32 fresh ones; tiles dealt to the CTAs
// round-robin) until none is left, so the scan runs beside the splits.  An
// edge that splits in this step has another nx before and after its warp
// rewrites it, so it is never listed here.
__device__ __forceinline__ void scan_tiles(const State& st, int i, int e, int e_end, long long nA, long long nE,
                                           long long nV, int n, Smem& sm, ListEntry* la, int& lac, int32_t* lnext,
                                           long long* counter) {
  const int lane = threadIdx.x & 31;
  const long long G = gridDim.x;
  const long long TA = (nA + kScanTile - 1) / kScanTile, TB = (nE - nA + 31) / 32;
  const uint32_t want = uint32_t(i + 1) * 0x10001u;
  for (;;) {
    int k = 0;
    if (lane == 0) k = atomicAdd(&sm.tile, 1);
    k = __shfl_sync(0xffffffffu, k, 0);
    const long long t = (long long)k * G + blockIdx.x;
    if (t >= TA + TB) return;
    if (t < TA) {
      const long long base = t * kScanTile + 8 * lane;
      uint4 x[4];
#pragma unroll
      for (int h = 0; h < 4; ++h)
        x[h] = base + 256 * h < nA ? *reinterpret_cast<const uint4*>(st.nx + base + 256 * h)
                                   : make_uint4(~0u, ~0u, ~0u, ~0u);
      uint32_t hits = 0;  // bit 8 h + q: edge base + 256 h + q
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        const uint32_t w[4] = {x[h].x, x[h].y, x[h].z, x[h].w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const uint32_t m = __vcmpeq2(w[q], want);
          if (m) hits |= ((m & 1u) | ((m >> 15) & 2u)) << (8 * h + 2 * q);
        }
      }
      while (__any_sync(0xffffffffu, hits != 0)) {
        bool hit = false;
        ListEntry ent{};
        if (hits) {
          const int bit = __ffs(hits) - 1;
          hits &= hits - 1;
          const long long ed = base + 256 * (bit >> 3) + (bit & 7);
          if (ed < nA) {
            const int u = st.EU[ed], w = st.EW[ed];
            if (u < 0 || u >= nV || w < 0 || w >= nV) {
              report_corrupt(st.g, 6, n, ed, u, w);  // never index with it
            } else {
              const bool su = minus_at(st, u, e + 1);
              ent = ListEntry{int(ed), su ? w : u, su ? u : w};
              hit = true;
            }
          }
        }
        warp_list(st, hit, ent, la, lac, lnext, counter);
      }
    } else {
      const long long ed = nA + (t - TA) * 32 + lane;
      bool hit = false;
      ListEntry ent{};
      if (ed < nE && *(volatile const uint16_t*)(st.nx + ed) == kNxFresh) {
        const int u = st.EU[ed], w = st.EW[ed];
        if (u < 0 || u >= nV || w < 0 || w >= nV) {
          report_corrupt(st.g, 7, n, ed, u, w);
        } else {
          const int f = first_opposite(st, u, w, e + 1, e_end);
          hit = f == e + 1;
          if (hit) {
            const bool su = minus_at(st, u, e + 1);
            ent = ListEntry{int(ed), su ? w : u, su ? u : w};
          }
          st.nx[ed] = f < 0 ? kNxNone : (hit ? kNxListed : uint16_t(f - e + i));
        }
      }
      warp_list(st, hit, ent, la, lac, lnext, counter);
    }
  }
}

__device__ void flush_cta(const State& st, Counters* cur, long long* cnext, int32_t* lnext, long long ebase, int n,
                          bool ahead, int lac, int pc, int pla, Smem& sm);

// Layer start: nx of every edge, and the list of neuron 0 of layer l.
__device__ inline void phase_scan0(const NetDesc& net, const State& st, int l, Smem& sm) {
  const int n0 = net.off[l], H = net.w[l + 1], e0 = net.m + n0;
  long long nV, nE;
  if (!step_counts(st, n0, nV, nE)) {
    if (threadIdx.x == 0) report_corrupt(st.g, 2, n0, nV, nE, st.Vcap);
    return;
  }
  const int warp = threadIdx.x >> 5;
  int32_t* list = st.list[n0 & 1];
  long long* counter = &st.cnt[n0 + 1].nsplit;
  int lac = 0;
  const long long step = (long long)gridDim.x * kBlock;
  for (long long base = (long long)blockIdx.x * kBlock; base < nE; base += step) {
    const long long ed = base + threadIdx.x;
    bool hit = false;
    ListEntry ent{};
    if (ed < nE) {
      const int u = st.EU[ed], w = st.EW[ed];
      if (u < 0 || u >= nV || w < 0 || w >= nV) {
        report_corrupt(st.g, 6, n0, ed, u, w);
      } else {
        const int f = first_opposite(st, u, w, e0, e0 + H);
        hit = f == e0;
        if (hit) {
          const bool su = minus_at(st, u, e0);
          ent = ListEntry{int(ed), su ? w : u, su ? u : w};
        }
        st.nx[ed] = f < 0 ? kNxNone : (hit ? kNxListed : uint16_t(f - e0));
      }
    }
    warp_list(st, hit, ent, sm.la[warp], lac, list, counter);
  }
  flush_cta(st, nullptr, counter, list, 0, n0, true, lac, 0, 0, sm);
}

// ---------------------------------------------------------------------------
// Whole-warp check (inline pairing) that the 2-face key of the new vertex
// nV + k2 (payload r2 = 2 * zero ordinal + minus) equals F, where lane w holds word w of this
// splitting edge's sign vector s0 and F is s0 with word wj replaced by Fw.
// The partner's face is rebuilt from its new vertex's sign words, which the
// partner wrote (and fenced) before it inserted its key.  All lanes call it.
__device__ __forceinline__ bool warp_face_matches(const State& st, long long k2, int r2, int e, int S, uint64_t s0,
                                                  int wj, uint64_t Fw, long long nV, long long total, int n) {
  const int lane = threadIdx.x & 31;
  if (k2 < 0 || k2 >= total) {  // a payload that no new vertex of this step wrote
    if (lane == 0) report_corrupt(st.g, 5, n, k2, total, r2);
    return false;
  }
  const long long v2 = nV + k2;
  uint64_t w2 = 0, zm = 0;
  if (lane < S) {
    w2 = __ldcg(st.SIG + (long long)lane * st.Vcap + v2) & entries_below(lane, e);
    zm = zero_mask(w2, lane, e);
  }
  const int c = __popcll(zm);
  int x = c;
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  const int o2 = r2 >> 1;
  int j2 = -1;
  if (o2 >= x - c && o2 < x) {
    uint64_t mm = zm;
    for (int q = x - c; q < o2; ++q) mm &= mm - 1;
    j2 = lane * 32 + (__ffsll((long long)mm) - 1) / 2;
  }
  const unsigned owner = __ballot_sync(0xffffffffu, j2 >= 0);
  if (!owner) return false;
  j2 = __shfl_sync(0xffffffffu, j2, __ffs(owner) - 1);
  if (lane == (j2 >> 5)) {
    const int sj = 2 * (j2 & 31);
    w2 = (w2 & ~(3ull << sj)) | (((r2 & 1) ? kMinus : kPlus) << sj);
  }
  const uint64_t f1 = (lane == wj) ? Fw : s0;
  return __all_sync(0xffffffffu, lane >= S || f1 == w2);
}

// ---------------------------------------------------------------------------
// One intersecting edge to position x: its record, and its nx (listed at lb
// + its rank among the listed ones if the next neuron crosses it).
__device__ __forceinline__ bool pair_splits(const int4& rec) { return (rec.w ^ (rec.w >> 1)) & 1; }

__device__ __forceinline__ void pair_store(const State& st, long long x, const int4& rec, int n, bool ahead,
                                           int32_t* lnext, long long at) {
  st.EU[x] = rec.x;
  st.EW[x] = rec.y;
  if (st.deferred) st.vlist[x] = make_int4(rec.x, rec.y, rec.z, n + 1);
  if (!ahead) return;
  const bool hit = pair_splits(rec);
  st.nx[x] = hit ? kNxListed : kNxFresh;
  if (hit)
    list_store(lnext, st.Ecap, at, (rec.w & 1) ? ListEntry{int(x), rec.y, rec.x} : ListEntry{int(x), rec.x, rec.y});
}

// Appends the warp's buffered intersecting edges (pc, of them pla that split
// at the next neuron) with one atomic each.
// The capacity check of a step counts two arrivals at a 2-face, as a generic
// input has them.  When signs are rounding noise a 2-face can be met more often
// and every later arrival pairs too (and raises kErrPairing), so the edges can
// pass the capacity, and with them the list (each edge is listed at most once).
// Entries whose places are not all inside are counted but not stored, and the
// next kernel that reads the counters finds them above the capacity and stops.
__device__ __forceinline__ void warp_flush_pairs(const State& st, const int4* pairs, int& pc, int& pla, Counters* cur,
                                                 long long* cnext, int32_t* lnext, long long ebase, int n,
                                                 bool ahead) {
  const int lane = threadIdx.x & 31;
  __syncwarp();
  long long pb = 0, lb = 0;
  if (lane == 0) pb = atomic_add_ll(&cur->npairs, (long long)pc);
  if (lane == 1 && ahead && pla) lb = atomic_add_ll(cnext, (long long)pla);
  pb = ebase + __shfl_sync(0xffffffffu, pb, 0);
  lb = __shfl_sync(0xffffffffu, lb, 1);
  const int np = pb + pc <= st.Ecap && lb + pla <= st.Ecap ? pc : 0;
  for (int t0 = 0; t0 < np; t0 += 32) {
    const bool in = t0 + lane < np;
    const int4 rec = in ? pairs[t0 + lane] : make_int4(0, 0, 0, 0);
    const unsigned b = __ballot_sync(0xffffffffu, in && ahead && pair_splits(rec));
    if (in) pair_store(st, pb + t0 + lane, rec, n, ahead, lnext, lb + __popc(b & ((1u << lane) - 1u)));
    lb += __popc(b);
  }
  __syncwarp();
  pc = 0;
  pla = 0;
}

// The step's end: the warps' buffered intersecting edges (pc, of them pla
// that split at the next neuron) and list entries (lac), one atomic each for
// the CTA.  All threads call it.
__device__ void flush_cta(const State& st, Counters* cur, long long* cnext, int32_t* lnext, long long ebase, int n,
                          bool ahead, int lac, int pc, int pla, Smem& sm) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) {
    sm.lac[warp] = lac;
    sm.pc[warp] = pc;
    sm.pla[warp] = pla;
  }
  __syncthreads();
  // warp sums and this warp's places, a warp's counts per lane
  int a = lane < kWarps ? sm.pc[lane] : 0, b = lane < kWarps ? sm.lac[lane] + (ahead ? sm.pla[lane] : 0) : 0;
  const int na = __reduce_add_sync(0xffffffffu, a), nb = __reduce_add_sync(0xffffffffu, b);
  if (na + nb == 0) return;  // uniform
  const int fa = __reduce_add_sync(0xffffffffu, lane < warp ? a : 0);
  const int fb = __reduce_add_sync(0xffffffffu, lane < warp ? b : 0);
  if (threadIdx.x == 0) {  // both places in flight at once
    long long x = 0, y = 0;
    if (na) x = atomic_add_ll(&cur->npairs, (long long)na);
    if (ahead && nb) y = atomic_add_ll(cnext, (long long)nb);
    if (ebase + x + na > st.Ecap || y + nb > st.Ecap) x = -1;  // nothing stored (see warp_flush_pairs)
    sm.pbase = x;
    sm.lbase = y;
  }
  __syncthreads();
  long long pb = sm.pbase;
  if (pb < 0) return;  // uniform
  pb += ebase + fa;
  long long lb = sm.lbase + fb;
  if (ahead)
    for (int t = lane; t < lac; t += 32) list_store(lnext, st.Ecap, lb + t, sm.la[warp][t]);
  lb += lac;
  for (int t0 = 0; t0 < pc; t0 += 32) {
    const bool in = t0 + lane < pc;
    const int4 rec = in ? sm.pairs[warp][t0 + lane] : make_int4(0, 0, 0, 0);
    const unsigned hb = __ballot_sync(0xffffffffu, in && ahead && pair_splits(rec));
    if (in) pair_store(st, pb + t0 + lane, rec, n, ahead, lnext, lb + __popc(hb & ((1u << lane) - 1u)));
    lb += __popc(hb);
  }
}

// One neuron step: steps (4)+(5) for the listed splitting edges, step (3) for
// the next neuron.  Returns true when the step must not run (capacity ran out
// -- nothing has been written -- or a counter is corrupt); the caller exits.
//
// A split is a chain of dependent memory round trips (the list entry, its two
// vertices, the hash table) and reductions over a vertex's neurons and sign
// words; the step's time is that chain, and on large nets the number of
// chains in flight.  So half a warp takes a split: the values lie vertex by
// vertex, 16 lanes read a row of 64 floats with four coalesced loads, every
// reduction has four shuffle steps for two splits at once, and 16 warps with
// up to 128 registers a thread keep 32 splits per SM in flight.  The mixed form,
// which also carries the queue of re-decisions, spills at that (k_layer: 358 bytes
// of stores and 560 of loads a thread), the others less (up to 48 of stores).
// Measured on GB300 against a warp per split, values neuron by neuron and two
// CTAs of 512 threads with 64 registers: neuron loop of a 5-40x4-1 net (1e7
// vertices) 63.4 -> 36.5 ms, of an 8-10x4-1 net 2.8 -> 1.9 ms, of a 3-64x4-1
// net 6.8 -> 5.3 ms (both including the re-decisions).
// WORDS: sign words per lane, 2 when a sign vector has more than 16.
template <typename ZT, bool MIXED, int WORDS>
__device__ bool phase_step(const NetDesc& net, const State& st, int l, int i, Smem& sm, double* ws, int mw) {
  constexpr bool TRACK = sizeof(ZT) == 4;  // FP32 values carry error estimates
  const int n = net.off[l] + i;
  const int H = net.w[l + 1];
  const bool ahead = i + 1 < H;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int gl = lane & (kGroup - 1), grp = lane / kGroup;
  const long long G = gridDim.x;
  const int32_t* lcur = st.list[n & 1];
  // this group's first splitting edge, loaded together with the counters
  const int slot0 = grp * kWarps + warp;  // the first half warps of all CTAs come first
  const long long k_first = (long long)slot0 * G + blockIdx.x;
  ListEntry sg_next{-1, -1, -1};
  if (k_first < st.Ecap) sg_next = ListEntry{lcur[k_first], lcur[st.Ecap + k_first], lcur[2 * st.Ecap + k_first]};
  Counters* cur = st.cnt + n + 1;
  const long long total = cur->nsplit;
  // edges whose nx is known: all but those of the last step's pairing
  const long long nA0 = st.cnt[n].nE_before + st.cnt[n].nsplit, tprev = 2 * st.cnt[n].tsize;
  long long nV, nE;
  if (!step_counts(st, n, nV, nE)) {
    if (threadIdx.x == 0) report_corrupt(st.g, 2, n, nV, nE, st.Vcap);
    return true;
  }
  if (total < 0 || total > nE) {
    if (threadIdx.x == 0) report_corrupt(st.g, 3, n, total, nV, nE);
    return true;
  }
  const int D = net.D, m = net.m, S = net.S;
  const int R = D > 1 ? 2 * (D - 1) : 1;
  // a 2-face key occurs twice, so the table is at most 2/5 full (4/5 if no face
  // found its partner)
  const long long kmax = total * (long long)(D - 1) * 2, tmin = kmax + kmax / 4;
  const long long tneed = tmin <= 64 ? 64 : 1ll << (64 - __clzll(tmin - 1));
  const long long eneed = nE + total * (long long)D;
  const long long vneed = nV + total;
  const bool overV = vneed > st.Vcap || vneed >= (1ll << 31) || total * R >= (1ll << 31);
  const bool overE = eneed > st.Ecap || eneed >= (1ll << 31);
  const bool overT = tneed > st.Tcap;
  const bool overTape = st.keep_tape && vneed > st.tape_cap;
  if (overV || overE || overT || overTape) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      Global* g = st.g;
      if (atomicCAS(&g->halted_at, -1, n) == -1) {
        g->halt_reason = (overV ? kHaltV : 0) | (overE ? kHaltE : 0) | (overT ? kHaltT : 0) | (overTape ? kHaltTape : 0);
        g->need_v = vneed;
        g->need_e = eneed;
        g->need_t = tneed;
      }
    }
    return true;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    cur->nV_before = nV;
    cur->nE_before = nE;
    cur->tsize = tneed;
  }
  if (threadIdx.x == 0) {
    sm.npend = 0;
    sm.tile = 0;
    sm.acc[0] = sm.acc[1] = 0;
  }
  if (sm.nrl_layer != l) {  // uniform: set by the previous step of this launch, or -1
    for (int t = threadIdx.x; t < 3 * H; t += kBlock) sm.nrl[t] = net.nrm[3 * net.off[l] + t];
  }
  __syncthreads();
  if (threadIdx.x == 0) sm.nrl_layer = l;
  // all counts are below 2^31 from here on
  const int nsp = int(total), nV32 = int(nV), nE32 = int(nE);
  const long long Vcap = st.Vcap;
  ZT* Z = static_cast<ZT*>(st.Z[l]);
  const int e = m + n;
  const int e0 = m + net.off[l];
  const int e_end = e0 + H;
  const long long nA = i > 0 ? nA0 : nE;
  int32_t* lnext = st.list[(n + 1) & 1];
  ListEntry* la = sm.la[warp];
  int4* pairs = sm.pairs[warp];
  int lac = 0, pc = 0, pla = 0;  // entries in la and pairs, and those of pairs that split at the next neuron
  bool scan = ahead;
  long long* cnext = ahead ? &st.cnt[n + 2].nsplit : nullptr;
  uint64_t* table = st.table + (long long)(n & 1) * 2 * st.Tcap;
  const uint32_t tmask = uint32_t(tneed - 1);
  const float* nrl = sm.nrl;
  int* zlist = sm.zlist[2 * warp + grp];
  int nkeys_w = 0, ndeg_w = 0;  // this group's (its first lane adds them up)
  int err_w = 0;
  unsigned long long paired_seen = 0;  // paired flags found by this lane's second arrivals
  // entries of this lane's words gl, gl + 16: before this neuron, later ones of the layer
  uint64_t m_below[WORDS], m_later[WORDS];
#pragma unroll
  for (int x = 0; x < WORDS; ++x) {
    const int w = gl + 16 * x;
    m_below[x] = w < S ? entries_below(w, e) : 0ull;
    m_later[x] = w < S ? entries_below(w, e_end) & ~entries_below(w, e + 1) : 0ull;
  }

  // Part B of a split: the next crossings of its halves, the parent 2-faces
  // (step (5)) and their pairing.  All lanes call it, act: the group has a
  // split.  Sign words of the new vertex, V+ and V- by lane (this layer's
  // entries complete).
  auto part_b = [&](bool act, uint64_t (&s0)[WORDS], const uint64_t (&sp)[WORDS], const uint64_t (&sq)[WORDS], int ed, int p, int q,
                    int v0, int k, bool bad) {
    if (pc > kPairCap - 2 * R) warp_flush_pairs(st, pairs, pc, pla, cur, cnext, lnext, nE + total, n, ahead);
    const uint32_t voff = act ? uint32_t(v0 - nV32) : 0;
    // the sign at the next neuron, and the next crossings of the two halves
    bool m0n = false;
    if (ahead) {
      const int wn = (e + 1) >> 5;
      const uint64_t x = __shfl_sync(0xffffffffu, wn < 16 ? s0[0] : s0[WORDS - 1], wn & 15, kGroup);
      m0n = ((x >> (2 * ((e + 1) & 31))) & 3ull) == kMinus;
      int j[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const uint64_t (&s)[WORDS] = h ? sq : sp;
        const uint64_t x0 = opposite(s[0], s0[0]) & m_later[0];
        unsigned b = group_ballot(x0 != 0);
        int f0 = 32 * gl + ((__ffsll((long long)x0) - 1) >> 1);
        if (WORDS == 2) {
          const uint64_t x1 = opposite(s[WORDS - 1], s0[WORDS - 1]) & m_later[WORDS - 1];
          const unsigned b1 = group_ballot(x1 != 0);
          if (!b) {
            b = b1;
            f0 = 512 + 32 * gl + ((__ffsll((long long)x1) - 1) >> 1);
          }
        }
        const int f = __shfl_sync(0xffffffffu, f0, __ffs(b) - 1, kGroup);
        j[h] = b ? f - e0 : int(kNxNone);
      }
      // E+ = (p, v0) keeps the edge's id, E- = (q, v0) is nE + k
      const int ju = gl == 0 ? j[0] : j[1];
      const int ex = gl == 0 ? ed : nE32 + k;
      const int u = gl == 0 ? p : q;
      const bool mine = act && gl < 2, hit = mine && ju == i + 1;
      if (mine) st.nx[ex] = hit ? kNxListed : uint16_t(ju);
      warp_list(st, hit, m0n ? ListEntry{ex, u, v0} : ListEntry{ex, v0, u}, la, lac, lnext, cnext);
    }
    // the 2-faces are named by the entries before this neuron
    uint64_t hb = 0;
#pragma unroll
    for (int x = 0; x < WORDS; ++x) {
      s0[x] &= m_below[x];
      if (gl + 16 * x < S) hb ^= word_hash(gl + 16 * x, s0[x]);
    }
#pragma unroll
    for (int o = kGroup / 2; o > 0; o >>= 1) hb ^= __shfl_xor_sync(0xffffffffu, hb, o);
    // the zero entries in order: a lane's place is the number of lower lanes'
    // zeros, counted by one ballot per multiplicity (most lanes hold 0 or 1)
    int nz = 0;
#pragma unroll
    for (int x = 0; x < WORDS; ++x) {
      const int w = gl + 16 * x;
      uint64_t mm = act && w < S ? zero_mask(s0[x], w, e) : 0ull;
      const int c0 = __popcll(mm);
      int at = nz;
      for (int y = 1; __any_sync(0xffffffffu, c0 >= y); ++y) {
        const unsigned b = group_ballot(c0 >= y);
        at += __popc(b & ((1u << gl) - 1u));
        nz += __popc(b);
      }
      for (; mm; mm &= mm - 1, ++at)
        if (at < 16) zlist[at] = w * 32 + ((__ffsll((long long)mm) - 1) >> 1);
    }
    __syncwarp();
    if (nz != D - 1) bad = true;
    if (bad && act) ndeg_w += 1;
    for (int r0 = 0; r0 < R; r0 += kGroup) {
      // this lane's key: zero ordinal r / 2, sign + (even r) or - (odd)
      const int r = r0 + gl, o = r >> 1;
      const bool minus = r & 1;
      const bool zero = act && nz == D - 1 && o < nz;
      const int jz = zero ? zlist[o] : 0;
      const int wj = jz >> 5, shj = 2 * (jz & 31);
      uint64_t s0w = __shfl_sync(0xffffffffu, s0[0], wj & 15, kGroup);
      if (WORDS == 2) {
        const uint64_t x = __shfl_sync(0xffffffffu, s0[WORDS - 1], wj & 15, kGroup);
        if (wj >= 16) s0w = x;
      }
      const bool has_key = zero && !(minus && jz < m);
      nkeys_w += __popc(group_ballot(has_key));
      bool paired = false;  // this lane's 2-face met its partner: rec
      int4 rec = make_int4(0, 0, 0, 0);
      uint64_t Fw = 0, h = 0;
      uint32_t slot = 0;
      if (has_key) {
        Fw = (s0w & ~(3ull << shj)) | ((minus ? kMinus : kPlus) << shj);
        h = hb ^ word_hash(wj, s0w) ^ word_hash(wj, Fw);
        slot = uint32_t(h) & tmask;
      }
      if (st.deferred) {
        // Full 64-bit fingerprint and payload in one 16-byte slot: the first
        // arrival inserts both with one 128-bit CAS, the second finds the
        // partner (and its sign at the next neuron, bit 62) in the same
        // atomic and pairs at once; the paired flag it sets is checked at the
        // end.  Every pairing is re-checked exactly after the extraction
        // (k_verify_pairs) from the two new vertices' sign vectors.
        if (has_key) {
          if (h == kEmpty) h = kEmpty - 1;
          const unsigned long long mine = (voff * uint32_t(R) + uint32_t(r)) | (m0n ? (1ull << 62) : 0ull);
          unsigned long long* tb = reinterpret_cast<unsigned long long*>(table);
          for (uint32_t probes = 0;; ++probes) {
            if (probes > tmask) {
              err_w |= kErrProbe;
              break;
            }
            unsigned long long ok, ov;
            cas128(tb + 2ull * slot, kEmpty, kEmpty, h, mine, ok, ov);
            if (ok == kEmpty) break;  // first arrival
            if (ok == h) {
              paired_seen |= atomicOr(tb + 2ull * slot + 1, kPaired64);
              const uint32_t pay = uint32_t(ov & ~(kPaired64 | (1ull << 62)));  // < total R < 2^31
              const uint32_t k2 = pay / uint32_t(R), r2 = pay - k2 * uint32_t(R);
              rec = make_int4(nV32 + int(k2), v0, int(r2 << 16) | r, ((ov >> 62) & 1ull ? 1 : 0) | (m0n ? 2 : 0));
              paired = true;
              break;
            }
            slot = (slot + 1) & tmask;
          }
        }
      } else {
        // Inline: a 32-bit tag; the second arrival compares the full faces
        // before it pairs, the whole warp for one candidate.  The partner's
        // sign words are read from memory, so they are fenced before the
        // insert.
        __threadfence();
        __syncwarp();
        const uint32_t tag = uint32_t(h >> 32);
        const uint64_t mine = has_key ? ((uint64_t(tag) << 32) | (voff * uint32_t(R) + uint32_t(r))) : 0ull;
        bool active = has_key;
        uint32_t probes = 0;
        while (__any_sync(0xffffffffu, active)) {
          bool cand = false;
          uint64_t old = 0;
          if (active) {
            old = atomicCAS(reinterpret_cast<unsigned long long*>(table + slot), (unsigned long long)kEmpty,
                            (unsigned long long)mine);
            if (old == kEmpty) {
              active = false;  // first arrival: the partner will pair with it
            } else if (uint32_t(old >> 32) == tag) {
              cand = true;
            } else {
              slot = (slot + 1) & tmask;
              if (++probes > tmask) {
                err_w |= kErrProbe;
                active = false;
              }
            }
          }
          __threadfence();
          unsigned cm = __ballot_sync(0xffffffffu, cand);
          while (cm) {
            const int Ld = __ffs(cm) - 1;
            cm &= cm - 1;
            const uint64_t pp = __shfl_sync(0xffffffffu, old, Ld) & 0x7fffffffull;
            const int wjL = __shfl_sync(0xffffffffu, wj, Ld);
            const uint64_t FwL = __shfl_sync(0xffffffffu, Fw, Ld);
            // word `lane` of the candidate's split: in its group's lane (lane & 15)
            const uint64_t a0 = __shfl_sync(0xffffffffu, s0[0], (Ld & kGroup) + (lane & 15));
            const uint64_t a1 = WORDS == 2 ? __shfl_sync(0xffffffffu, s0[WORDS - 1], (Ld & kGroup) + (lane & 15)) : 0ull;
            const bool eq = warp_face_matches(st, (long long)(pp / R), int(pp % R), e, S, lane < 16 ? a0 : a1, wjL, FwL,
                                              nV, total, n);
            if (lane == Ld) {
              if (eq) {
                const uint64_t prev = atomicOr(reinterpret_cast<unsigned long long*>(table + slot),
                                               (unsigned long long)kPaired);
                if (prev & kPaired) {
                  err_w |= kErrPairing;
                } else {
                  const int v2 = int(nV + (long long)(pp / R));
                  const bool m2 = ahead && __ldcg(Z + (long long)v2 * H + i + 1) < ZT(0);
                  rec = make_int4(v2, v0, 0, (m2 ? 1 : 0) | (m0n ? 2 : 0));
                  paired = true;
                }
                active = false;
              } else {
                slot = (slot + 1) & tmask;
                if (++probes > tmask) {
                  err_w |= kErrProbe;
                  active = false;
                }
              }
            }
          }
        }
      }
      const unsigned pb = __ballot_sync(0xffffffffu, paired);
      if (paired) pairs[pc + __popc(pb & ((1u << lane) - 1u))] = rec;
      pc += __popc(pb);
      pla += __popc(__ballot_sync(0xffffffffu, paired && ahead && pair_splits(rec)));
    }
    __syncwarp();
  };

  // Rounds of splits, two per warp, without synchronisation.  In mixed
  // precision a split whose new vertex has a value within the filter is
  // queued after part A; once in kPendRounds rounds if the queue could fill,
  // and after the last round, the CTA re-decides the queued vertices together
  // and finishes their part B with the state read back.
  const int Wt = int(G) * kSplits;
  const int rounds = (nsp + Wt - 1) / Wt;
  int rd = 0;
  bool looked = false;  // the queue was looked at before round rd
  int pn = 0, pt = 0;   // queued splits to finish, those done (uniform per CTA)
  for (;;) {
    const bool over = rd >= rounds;  // uniform
    if (over && scan) {  // the scan beside the last splits of other warps
      scan_tiles(st, i, e, e_end, nA, nE, nV, n, sm, la, lac, lnext, cnext);
      scan = false;
    }
    if (MIXED && !looked && (over || rd % kPendRounds == kPendRounds - 1)) {
      looked = true;
      __syncthreads();
      const int np = sm.npend;
      if (np > 0 && (over || np > kPendCap - kPendRounds * kSplits)) {
        drain_pending<ZT>(net, st, sm.pend.split.v0, np, l, e + 1, i + 1, mw, ws);
        pn = np;
        pt = 0;
      } else {
        __syncthreads();
      }
    }
    bool ready = false, bad = false;  // this group's split goes to part B
    int ed = 0, p = 0, q = 0, v0 = 0;
    int k = 0;
    uint64_t s0[WORDS], sp[WORDS], sq[WORDS];  // sign words of the new vertex and its parents
#pragma unroll
    for (int x = 0; x < WORDS; ++x) s0[x] = sp[x] = sq[x] = 0;
    if (MIXED && pn > 0) {
      const int t = pt + slot0;
      ready = t < pn;
      if (ready) {
        const int x = sm.pend.split.k[t];
        v0 = sm.pend.split.v0[t];
        bad = x < 0;  // complemented: not a regular crossing (counted)
        k = bad ? ~x : x;
        ed = lcur[k];
        p = st.EU[ed];
        q = st.EU[nE32 + k];
#pragma unroll
        for (int x = 0; x < WORDS; ++x) {
          const int w = gl + 16 * x;
          if (w < S) {
            s0[x] = __ldcg(st.SIG + (long long)w * Vcap + v0);
            sp[x] = st.SIG[(long long)w * Vcap + p];
            sq[x] = st.SIG[(long long)w * Vcap + q];
          }
        }
      }
      pt += kSplits;
    } else {
      if (over) break;
      k = rd * Wt + slot0 * int(G) + int(blockIdx.x);  // splits dealt over the CTAs first
      const ListEntry sg = sg_next;
      if (k + Wt < nsp)  // the next round's, loaded during this one
        sg_next = ListEntry{lcur[k + Wt], lcur[st.Ecap + k + Wt], lcur[2 * st.Ecap + k + Wt]};
      // The round's new vertices are numbered CTA by CTA: CTA b holds entries
      // w G + b of the round (w < n_b = rq + [b < rr]) and gives them the
      // consecutive offsets b rq + min(b, rr) + w, a bijection onto the
      // round's [0, rem), so each CTA writes whole sectors of the coordinate and
      // sign rows.
      const int rem = nsp - rd * Wt < Wt ? nsp - rd * Wt : Wt;
      const int rq = rem / int(G), rr = rem - rq * int(G), cta = int(blockIdx.x);
      const int voff = rd * Wt + cta * rq + (cta < rr ? cta : rr) + slot0;
      // ---- part A: the new vertex (step (4)) ----
      v0 = nV32 + voff;
      bool okA = k < nsp;
      if (okA) {
        ed = sg.e;
        p = sg.p;  // V+
        q = sg.q;  // V-
        okA = !(ed < 0 || ed >= nE32 || p < 0 || p >= nV32 || q < 0 || q >= nV32);
        if (!okA && gl == 0) report_corrupt(st.g, 4, n, ed, p, q);
      }
      if (__any_sync(0xffffffffu, okA)) {
        // every load of the endpoints is issued before any of them is used
        const ZT* Zp = Z + (long long)p * H;
        const ZT* Zq = Z + (long long)q * H;
        ZT* Z0 = Z + (long long)v0 * H;
        ZT za0 = ZT(0), zb0 = ZT(0);
        if (okA) {
          za0 = Zp[i];
          zb0 = Zq[i];
        }
        double xp = 0.0, xq = 0.0;
        if (okA && gl < D) {
          xp = st.X[(long long)gl * Vcap + p];
          xq = st.X[(long long)gl * Vcap + q];
        }
#pragma unroll
        for (int x = 0; x < WORDS; ++x) {
          const int w = gl + 16 * x;
          if (okA && w < S) {
            sp[x] = st.SIG[(long long)w * Vcap + p];
            sq[x] = st.SIG[(long long)w * Vcap + q];
          }
        }
        ZT zp[4], zq[4];  // neurons 16 t + gl of the chunk
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const int j = 16 * t + gl;
          const bool in = okA && j < H;
          zp[t] = in ? Zp[j] : ZT(0);
          zq[t] = in ? Zq[j] : ZT(0);
        }
        float rp = 0.f, rq_ = 0.f, xep = 0.f, xeq = 0.f;
        if (TRACK && okA && gl == 0) {
          rp = st.esc[p];
          rq_ = st.esc[q];
          xep = st.exc[p];
          xeq = st.exc[q];
        }
        const double a = static_cast<double>(za0);
        const double b = static_cast<double>(zb0);
        // t in float64 on one lane (the FP64 units are few), then broadcast
        double t_ = 0.0;
        int out_of_range = 0;
        if (okA && gl == 0) {
          t_ = a / (a - b);
          if (!(t_ >= 0.0 && t_ <= 1.0)) {
            t_ = t_ < 0.0 ? 0.0 : 1.0;
            out_of_range = 1;
          }
          if (!(a > 0.0 && b < 0.0)) out_of_range = 1;
        }
        const double tt = __shfl_sync(0xffffffffu, t_, 0, kGroup);
        bad = __shfl_sync(0xffffffffu, out_of_range, 0, kGroup);
        if (okA && gl < D) st.X[(long long)gl * Vcap + v0] = fma(tt, xq - xp, xp);
        const ZT tz = static_cast<ZT>(tt);
        // earlier entries: the join of the endpoints' words
#pragma unroll
        for (int x = 0; x < WORDS; ++x)
          if (opposite(sp[x], sq[x]) & m_below[x]) err_w |= kErrConflict;
        float amax = 0.f;
        float zk[4];  // the first chunk's new values (filter)
        uint32_t minus[WORDS];
#pragma unroll
        for (int x = 0; x < WORDS; ++x) minus[x] = 0u;
        for (int c = 0; 64 * c < H; ++c) {
          uint64_t mask = 0;
          ZT np4[4], nq4[4];  // the next chunk, loaded during this one
          if (64 * (c + 1) < H) {
#pragma unroll
            for (int t = 0; t < 4; ++t) {
              const int j = 64 * (c + 1) + 16 * t + gl;
              const bool in = okA && j < H;
              np4[t] = in ? Zp[j] : ZT(0);
              nq4[t] = in ? Zq[j] : ZT(0);
            }
          }
#pragma unroll
          for (int t = 0; t < 4; ++t) {
            const int j = 64 * c + 16 * t + gl;
            ZT zj = ZT(0);
            bool mi = false;
            if (okA && j < H) {
              if (j < i) {  // processed: the join of the endpoints' signs, value made consistent
                const bool pl = zp[t] > ZT(0) || zq[t] > ZT(0);
                mi = zp[t] < ZT(0) || zq[t] < ZT(0);
                if (pl && mi) err_w |= kErrConflict;
                zj = zp[t] + tz * (zq[t] - zp[t]);
                if (pl && !(zj > ZT(0))) zj = tiny_value<ZT>();
                if (mi && !(zj < ZT(0))) zj = -tiny_value<ZT>();
                if (!pl && !mi) zj = ZT(0);
              } else if (j > i) {
                zj = zp[t] + tz * (zq[t] - zp[t]);
                if (zj == ZT(0)) {  // on a later folded hyperplane: not generic
                  zj = tiny_value<ZT>();
                  atomic_add_ll(&st.cnt[net.off[l] + j + 1].ndegenerate, 1ll);
                }
                mi = zj < ZT(0);
              }
              Z0[j] = zj;  // row i: exactly 0
              if (TRACK) amax = fmaxf(amax, fabsf(static_cast<float>(zj)) * nrl[3 * j + 2]);
            }
            if (c == 0) zk[t] = static_cast<float>(zj);
            mask |= static_cast<uint64_t>(group_ballot(mi)) << (16 * t);
          }
#pragma unroll
          for (int x = 0; x < WORDS; ++x) minus[x] |= word_window(mask, gl + 16 * x, c, e0);
          if (64 * (c + 1) >= H) break;
#pragma unroll
          for (int t = 0; t < 4; ++t) {
            zp[t] = np4[t];
            zq[t] = nq4[t];
          }
        }
        // sign words: the join before this neuron, 0 at it, the values' signs after it
#pragma unroll
        for (int x = 0; x < WORDS; ++x) {
          s0[x] = ((sp[x] | sq[x]) & m_below[x]) | (codes_of(minus[x]) & m_later[x]);
          const int w = gl + 16 * x;
          if (okA && w < S) st.SIG[(long long)w * Vcap + v0] = s0[x];
        }
        bool pend = false;
        if (TRACK) {
          float dx = gl < D ? static_cast<float>(fabs(xq - xp)) : 0.f;
#pragma unroll
          for (int o = kGroup / 2; o > 0; o >>= 1) {
            amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
            dx = fmaxf(dx, __shfl_xor_sync(0xffffffffu, dx, o));
          }
          float esc0 = 0.f;
          if (okA && gl == 0) {
            // rms estimates, independent errors adding in quadrature: the value
            // scale takes the endpoints' (a convex combination does not amplify
            // them) and the interpolation's rounding (u |z_j|, in units of
            // ||W_j||_2); the position takes the endpoints' estimates and the
            // shift along the edge that the errors of a and b cause in t (all in
            // float32: estimates).
            const float rm = fmaxf(rp, rq_), rr_ = 5.9604645e-8f * amax;
            esc0 = sqrtf(rm * rm + rr_ * rr_);
            st.esc[v0] = esc0;
          }
          if (MIXED) {  // the later neurons' new values within the filter
            const float es = __shfl_sync(0xffffffffu, esc0, 0, kGroup);
            bool f = false;
#pragma unroll
            for (int t = 0; t < 4; ++t) {
              const int j = 16 * t + gl;
              if (j > i && j < H)
                f = f || fabsf(zk[t]) <= net.kappa_sel * (nrl[3 * j] * es + 2.9802322e-8f * nrl[3 * j + 1]);
            }
            for (int j = 64 + gl; j < H; j += kGroup)
              if (okA && j > i)
                f = f || fabsf(static_cast<float>(Z0[j])) <= net.kappa_sel * (nrl[3 * j] * es + 2.9802322e-8f * nrl[3 * j + 1]);
            pend = group_ballot(f && okA) != 0;
          }
          if (okA && gl == 0) {
            const float ep = nrl[3 * i] * rp + 2.9802322e-8f * nrl[3 * i + 1];
            const float eq = nrl[3 * i] * rq_ + 2.9802322e-8f * nrl[3 * i + 1];
            const float shift = (ep + eq) / static_cast<float>(za0 - zb0) * dx;
            const float xe = fmaxf(xep, xeq);
            st.exc[v0] = sqrtf(xe * xe + shift * shift);
          }
        }
        if (okA && gl == 0) {
          st.EU[ed] = p;
          st.EW[ed] = v0;
          st.EU[nE32 + k] = q;
          st.EW[nE32 + k] = v0;
          if (st.deferred) st.vlist[nE32 + k] = make_int4(0, 0, 0, 0);  // not a pairing edge
          if (st.keep_tape) {
            st.tape_pq[v0] = p;
            st.tape_pq[st.tape_cap + v0] = q;
            st.tape_t[v0] = tt;
          }
          if (MIXED && pend) {
            const int x = atomicAdd(&sm.npend, 1);  // < kPendCap: looked at every kPendRounds rounds
            sm.pend.split.v0[x] = v0;
            sm.pend.split.k[x] = bad ? ~k : k;
          }
        }
        ready = okA && !pend;
      } else if (scan) {  // a warp without a split: the scan, beside the others' splits
        scan_tiles(st, i, e, e_end, nA, nE, nV, n, sm, la, lac, lnext, cnext);
        scan = false;
      }
      rd += 1;
      looked = false;
    }
    if (__any_sync(0xffffffffu, ready)) part_b(ready, s0, sp, sq, ed, p, q, v0, k, bad);
    if (MIXED && pn > 0 && pt >= pn) {
      __syncthreads();
      if (threadIdx.x == 0) sm.npend = 0;
      __syncthreads();
      pn = 0;
    }
  }
  // the table of the previous step: emptied for the step after this one
  {
    uint4* told = reinterpret_cast<uint4*>(st.table + (long long)((n + 1) & 1) * 2 * st.Tcap);
    const uint4 ff4 = make_uint4(~0u, ~0u, ~0u, ~0u);
    for (long long t = (long long)blockIdx.x * kBlock + threadIdx.x; 2 * t < tprev; t += G * kBlock) told[t] = ff4;
  }
  if (paired_seen & kPaired64) err_w |= kErrPairing;  // a third arrival at a 2-face
  err_w = __reduce_or_sync(0xffffffffu, err_w);
  if (gl == 0) {
    if (nkeys_w) atomicAdd(reinterpret_cast<unsigned long long*>(&sm.acc[0]), (unsigned long long)nkeys_w);
    if (ndeg_w) atomicAdd(reinterpret_cast<unsigned long long*>(&sm.acc[1]), (unsigned long long)ndeg_w);
  }
  if (lane == 0 && err_w) atomicOr(&st.g->error, err_w);
  flush_cta(st, cur, cnext, lnext, nE + total, n, ahead, lac, pc, pla, sm);
  if (threadIdx.x == 0) {
    if (sm.acc[0]) atomic_add_ll(&cur->nkeys, sm.acc[0]);
    if (sm.acc[1]) atomic_add_ll(&cur->ndegenerate, sm.acc[1]);
  }
  return false;
}

}  // namespace pc
