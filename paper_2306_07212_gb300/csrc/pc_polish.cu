// Coordinate polish: every vertex whose coordinate error estimate exceeds the
// threshold moves to the exact intersection of its D zero sets (the vertex of
// Section 4.2's complex: D entries of its sign vector are zero, each affine on
// the vertex's own piece, Eq. 4 with the stored activation pattern).  One
// Newton step from the stored coordinates solves the D x D system A dx = -g,
// with the values g in float-float and the gradients A in float32 (the step is
// small, so float32 gradients add only ~1e-7 of the step; see pc_newton.cuh).
//
// The forward pass that gives g and A is a chain of matrix products with a mask
// per vertex: about half of a layer's inputs are inactive (exact zeros) and
// half of its outputs are not needed by the next layer, and in the vertex's
// last layer only its zero entries are.  So a vertex is worked on by itself, by
// 8 or 16 lanes, over lists: inputs are its active neurons, outputs its active
// neurons and the neurons of its zero set, about a fifth of the dense
// multiply-adds.  Every lane holds up to kPtRows outputs (the layer's list, 8 or
// 16 apart), so that an input's record (head, remainder and D gradient entries,
// one or two 16-byte broadcasts from shared memory) serves up to 64 outputs,
// and pairs of outputs run on packed FP32 instructions (each rounded as the
// scalar form).  Weight heads are staged in shared memory when they fit; their
// remainders are read only for networks that have any (NetDesc::rem); such a
// network's pairs come from global memory: 3-64x3-1 net (8.9e5 vertices) 1.69 ms
// staged and 1.93 as pairs, 5-30x3-1 (2.1e6) 2.66 and 3.31.
//
// The dot products follow Ogita-Rump-Oishi Dot2 (exact products by FMA, TwoSum
// of the running sum, error terms summed in a float), about 44 bits; a skipped
// zero input changes no bit of them, so every sum is the dense one's in its
// order.
//
// Bound by FP32 issue.  The instances take all 128 registers of the launch bound
// and spill, more with D: 84 bytes of stores and 172 of loads a thread at D = 3,
// 352 and 500 at D = 5, 404 and 1180 at D = 8 (8 lanes).  Measured on GB300 against a dense product over tiles
// of 32 vertices (D <= 5) and a dense pass of a warp per vertex (D > 5):
// 3-64x4-1 (314k vertices) 2.57 -> 0.77 ms, 5-40x4-1 (1e7) 39 -> 15.7 ms,
// 4-128x3-1 (212k) 3.8 -> 1.35 ms, 8-10x4-1 (369k) 7.7 -> 0.93 ms.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "pc_ctx.h"
#include "pc_device.cuh"
#include "pc_newton.cuh"

namespace pc {

constexpr int kPtThreads = 512;  // at most
constexpr int kPtRows = 8;       // outputs of a lane in one pass over the inputs, at most
constexpr int kPtMaxD = kMaxD;
constexpr int kPtSmemMax = 200 * 1024;  // vertices' workspace
constexpr int kPtSmemAll = 224 * 1024;  // and the staged weights

// Lanes of a vertex: 8 where they hold a layer's outputs in one pass and the
// Newton system's rows (what is not the products -- lists, the solve, the few
// outputs of the last layer -- then serves four vertices per instruction),
// else 16.  With 16 lanes throughout: 0.97 and 24.3 ms instead of 0.77 and 15.7
// on the two first nets above.
__host__ __device__ constexpr int pt_lanes(int mw, int D) { return mw <= 8 * kPtRows && D <= 8 ? 8 : 16; }

struct PtLayout {
  int TV, rows;
  size_t A, gv, sig, ahi, alo, J, zl, nz, total;
};

// Floats of an input's record: head, remainder, D gradient entries, padded to
// 16 bytes.
__host__ __device__ constexpr int pt_record(int D) { return (2 + D + 3) / 4 * 4; }

// Shared-memory layout of a CTA's TV vertices (byte offsets, each 16-aligned).
// rows: records held per vertex (the widest layer, and D for the coordinates).
__host__ __device__ inline PtLayout pt_layout(int TV, int mw, int S, int D) {
  PtLayout p{};
  p.TV = TV;
  p.rows = mw > D ? mw : D;
  size_t o = 0;
  auto take = [&](size_t bytes) {
    const size_t at = o;
    o += (bytes + 15) / 16 * 16;
    return at;
  };
  const size_t rec = (size_t)TV * p.rows * pt_record(D) * 4;
  p.A = take((size_t)TV * D * D * 4);                 // Newton rows [TV][D][D] (float)
  p.gv = take((size_t)TV * D * 8);                    // their values [TV][D] (double)
  p.sig = take(0);                                    // sign words: none, they stay in registers
  p.ahi = take(rec);                                  // records by list position [TV][rows][pt_record]
  // the next layer's, when one pass does not hold all outputs
  p.alo = take(p.rows > kPtRows * pt_lanes(mw, D) ? rec : 0);
  p.J = take((size_t)TV * p.rows * 2 * 2);            // lists [TV][2][rows]: inputs (offsets of weight rows), outputs
  p.zl = take((size_t)TV * D * 4);                    // zero entries [TV][D]
  p.nz = take((size_t)pt_record(D) * 4);              // a record of zeros
  p.total = o;
  return p;
}

// Vertices per CTA, fewer when their records do not fit.
static int pt_tile_vertices(int mw, int S, int D) {
  int TV = kPtThreads / pt_lanes(mw, D);
  while (TV > 4 && pt_layout(TV, mw, S, D).total > (size_t)kPtSmemMax) TV -= 4;
  return TV;
}

// One Dot2 step of two outputs: s + e += w * (hi + lo), w = head + rem; nhi =
// -hi.  Differences are FMAs with -1 (the packed instructions take no negated
// operands; the rounding is the subtraction's).
template <bool REM>
__device__ __forceinline__ void dot2_step(float2 w, float2 rem, float2 hi, float2 nhi, float2 lo, float2& s, float2& e) {
  const float2 m1 = make_float2(-1.f, -1.f);
  const float2 np = __fmul2_rn(w, nhi);                // -(w hi)
  float2 er = __ffma2_rn(w, hi, np);                   // exact low part of the product
  er = __ffma2_rn(w, lo, er);                          // cross terms of the low parts
  if (REM) er = __ffma2_rn(rem, hi, er);
  const float2 t = __ffma2_rn(np, m1, s);              // TwoSum: t + its error is exact
  const float2 bb = __ffma2_rn(s, m1, t);
  const float2 ts = __ffma2_rn(__ffma2_rn(bb, m1, t), m1, s);
  const float2 tp = __fadd2_rn(np, bb);
  e = __fadd2_rn(e, __fadd2_rn(__ffma2_rn(tp, m1, ts), er));
  s = t;
}

// Weight (head, remainder) of neuron r for input c: staged heads, or the
// pairs in global memory.
template <bool STAGED>
__device__ __forceinline__ float2 weight(const float* Ws, const float2* Wg, int at) {
  if (STAGED) return make_float2(Ws[at], 0.f);
  return __ldg(Wg + at);
}

// The scalar form.
template <bool REM>
__device__ __forceinline__ void dot2_step(float w, float rem, float hi, float lo, float& s, float& e) {
  const float pr = __fmul_rn(w, hi);
  float er = fmaf(w, hi, -pr);
  er = fmaf(w, lo, er);
  if (REM) er = fmaf(rem, hi, er);
  const float t = __fadd_rn(s, pr);
  const float bb = __fsub_rn(t, s);
  const float ts = __fsub_rn(s, __fsub_rn(t, bb));
  e = __fadd_rn(e, __fadd_rn(__fadd_rn(ts, __fsub_rn(pr, bb)), er));
  s = t;
}

// A lane's gradients of one output: pairs of components, then an odd one, as
// they lie in the records.
template <int DT>
struct Grad {
  float2 p[DT / 2 > 0 ? DT / 2 : 1];
  float o;
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int d = 0; d < DT / 2; ++d) p[d] = make_float2(0.f, 0.f);
    o = 0.f;
  }
  __device__ __forceinline__ void add(float w, const float* r) {  // r: the record's gradient
#pragma unroll
    for (int d = 0; d < DT / 2; ++d)
      p[d] = __ffma2_rn(make_float2(w, w), make_float2(r[2 * d], r[2 * d + 1]), p[d]);
    if (DT & 1) o = fmaf(w, r[DT - 1], o);
  }
  __device__ __forceinline__ float at(int d) const {
    return (DT & 1) && d == DT - 1 ? o : ((d & 1) ? p[d / 2].y : p[d / 2].x);
  }
};

// NR outputs per lane (value sums of pairs of outputs packed, then an odd one)
// over the vertex's inputs [0, cmax) (its own count is ci; the other half warp
// may have more, past its own it reads a record of zeros, which changes
// nothing): (s, e) and the gradients of the outputs row[0 .. NR).  li: offsets
// of the inputs' weight rows.
template <int DT, int NR, bool STAGED, bool REM>
__device__ __forceinline__ void rows_pass(const float* rec, const float* none, const uint16_t* li, int ci, int cmax,
                                          const float* Ws, const float2* Wg, const int (&row)[kPtRows],
                                          float2 (&s)[kPtRows / 2], float2 (&e)[kPtRows / 2], Grad<DT> (&g)[kPtRows]) {
  constexpr int PS = pt_record(DT), NP = NR / 2;
#pragma unroll 2
  for (int t = 0; t < cmax; ++t) {
    const bool in = t < ci;
    const int c = in ? li[t] : 0;
    const float* at = in ? rec + t * PS : none;
    float x[PS];
#pragma unroll
    for (int h = 0; h < PS / 4; ++h) {
      const float4 f = *reinterpret_cast<const float4*>(at + 4 * h);
      x[4 * h] = f.x;
      x[4 * h + 1] = f.y;
      x[4 * h + 2] = f.z;
      x[4 * h + 3] = f.w;
    }
    const float hi = x[0], lo = x[1];
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      const float2 wa = weight<STAGED>(Ws, Wg, c + row[2 * p]), wb = weight<STAGED>(Ws, Wg, c + row[2 * p + 1]);
      dot2_step<REM>(make_float2(wa.x, wb.x), make_float2(wa.y, wb.y), make_float2(hi, hi), make_float2(-hi, -hi),
                     make_float2(lo, lo), s[p], e[p]);
      g[2 * p].add(wa.x, x + 2);
      g[2 * p + 1].add(wb.x, x + 2);
    }
    if (NR & 1) {
      const float2 w = weight<STAGED>(Ws, Wg, c + row[2 * NP]);
      dot2_step<REM>(w.x, w.y, hi, lo, s[NP].x, e[NP].x);
      g[2 * NP].add(w.x, x + 2);
    }
  }
}

// The D x D system of a vertex by its LN lanes (lane r < D holds row r of M and
// the right-hand side; all lanes of the warp call it): Gaussian elimination
// with partial pivoting and back substitution in float32, rows in parallel.
// Component d in lane d; ok false when singular.
template <int DT, int LN>
__device__ __forceinline__ float solve_group(float (&M)[DT], float rhs, bool& ok) {
  const int gl = threadIdx.x & (LN - 1);
  int pos = gl;      // the row's place in the elimination order
  int piv[DT];       // lane of the c-th pivot row
#pragma unroll
  for (int c = 0; c < DT; ++c) {
    const unsigned key = gl < DT && pos >= c ? __float_as_uint(fabsf(M[c])) + 1u : 0u;
    unsigned top = 0;
    int best = 0, at = 0;
#pragma unroll
    for (int r = 0; r < DT; ++r) {  // the largest; the first of equal ones
      const unsigned k = __shfl_sync(0xffffffffu, key, r, LN);
      const int p = __shfl_sync(0xffffffffu, pos, r, LN);
      if (k > top || (k == top && p < at)) {
        top = k;
        best = r;
        at = p;
      }
    }
    if (top <= 1u) ok = false;
    piv[c] = best;
    const bool mine = gl == best;
    if (!mine && pos == c) pos = at;  // the rows change places
    if (mine) pos = c;
    const float f = M[c] / __shfl_sync(0xffffffffu, M[c], best, LN);
#pragma unroll
    for (int k = c + 1; k < DT; ++k) {
      const float x = __shfl_sync(0xffffffffu, M[k], best, LN);
      if (pos > c) M[k] = fmaf(-f, x, M[k]);
    }
    const float x = __shfl_sync(0xffffffffu, rhs, best, LN);
    if (pos > c) rhs = fmaf(-f, x, rhs);
  }
  float sol[DT], out = 0.f;
#pragma unroll
  for (int r = DT - 1; r >= 0; --r) {
    float acc = rhs;
#pragma unroll
    for (int k = r + 1; k < DT; ++k) acc = fmaf(-M[k], sol[k], acc);
    sol[r] = __shfl_sync(0xffffffffu, acc / M[r], piv[r], LN);
    if (gl == r) out = sol[r];
  }
  return out;
}

template <int N>
struct Int {
  static constexpr int value = N;
};

// STAGED: heads in shared memory (a network without remainders), or
// pairs from global memory.
template <int DT, int LN, bool STAGED>
__device__ __forceinline__ void polish_vertices(const NetDesc& net, const State& st, float thr, int mw, int TV,
                                                unsigned char* sm, const float* Ps, long long nV, int& npol) {
  constexpr int NW = kMaxWords / LN;        // sign words per lane: gl, gl + LN, ...
  constexpr unsigned kMask = (1u << LN) - 1u;
  constexpr int kPass = LN * kPtRows;
  constexpr bool REM = !STAGED;
  const int lane = threadIdx.x & 31, gl = lane & (LN - 1), gsh = lane & ~(LN - 1), g = threadIdx.x / LN;
  const int S = net.S, m = net.m;
  const long long Vcap = st.Vcap;
  constexpr int PS = pt_record(DT);
  const PtLayout lay = pt_layout(TV, mw, S, DT);
  float* A = reinterpret_cast<float*>(sm + lay.A) + g * DT * DT;
  double* gv = reinterpret_cast<double*>(sm + lay.gv) + g * DT;
  float* rec = reinterpret_cast<float*>(sm + lay.ahi) + (size_t)g * lay.rows * PS;
  float* next = lay.rows > kPass ? reinterpret_cast<float*>(sm + lay.alo) + (size_t)g * lay.rows * PS : rec;
  uint16_t* li = reinterpret_cast<uint16_t*>(sm + lay.J) + (size_t)g * 2 * lay.rows;
  uint16_t* lo_ = li + lay.rows;
  int* zl = reinterpret_cast<int*>(sm + lay.zl) + g * DT;
  const float* none = reinterpret_cast<const float*>(sm + lay.nz);  // a record of zeros
  auto gballot = [&](bool x) { return (__ballot_sync(0xffffffffu, x) >> gsh) & kMask; };
  auto most = [&](int x) {  // over the warp's groups
#pragma unroll
    for (int o = LN; o < 32; o <<= 1) x = max(x, __shfl_xor_sync(0xffffffffu, x, o));
    return x;
  };
  const long long stride = (long long)gridDim.x * TV;
  for (long long base = (long long)blockIdx.x * TV; base < nV; base += stride) {
    const long long v = base + g;
    bool act = v < nV && !(st.exc[v] <= thr);
    if (!__any_sync(0xffffffffu, act)) continue;
    uint64_t word[NW];
#pragma unroll
    for (int x = 0; x < NW; ++x)
      word[x] = act && gl + LN * x < S ? st.SIG[(long long)(gl + LN * x) * Vcap + v] : 0ull;
    double xd = 0.0;
    if (act && gl < DT) xd = st.X[(long long)gl * Vcap + v];
    // the zero entries in order
    int nz = 0;
#pragma unroll
    for (int x = 0; x < NW; ++x) {
      if (LN * x >= S) break;
      const int w = gl + LN * x;
      uint64_t mm = act && w < S ? zero_mask(word[x], w, net.P) : 0ull;
      const int c0 = __popcll(mm);
      int at = nz;
      for (int y = 1; __any_sync(0xffffffffu, c0 >= y); ++y) {
        const unsigned b = gballot(c0 >= y);
        at += __popc(b & ((1u << gl) - 1u));
        nz += __popc(b);
      }
      for (; mm; mm &= mm - 1, ++at)
        if (at < DT) zl[at] = w * 32 + ((__ffsll((long long)mm) - 1) >> 1);
    }
    act = act && nz == DT;  // else not a vertex of the generic complex: left as it is
    __syncwarp();
    // the highest layer among the zero entries
    int lmax = -1;
    const int mine = act && gl < DT ? zl[gl] : 0;
    for (int l = 0; l < net.L; ++l)
      if (act && gl < DT && mine - m >= net.off[l]) lmax = l;
#pragma unroll
    for (int o = LN / 2; o > 0; o >>= 1) lmax = max(lmax, __shfl_xor_sync(0xffffffffu, lmax, o));
    const int lall = most(lmax);
    // the coordinates (float-float) with the identity as their gradient
    if (gl < DT) {
      const float h = static_cast<float>(xd);
      float* r = rec + gl * PS;
      r[0] = h;
      r[1] = static_cast<float>(xd - static_cast<double>(h));
#pragma unroll
      for (int d = 0; d < DT; ++d) r[2 + d] = d == gl ? 1.f : 0.f;
      li[gl] = static_cast<uint16_t>(gl * net.w[1]);
    }
    int ci = act ? DT : 0;
    for (int k = 0; k <= lall; ++k) {
      const int H = net.w[k + 1], e0 = m + net.off[k];
      // outputs: the active neurons (not in the vertex's last layer), then the
      // zero set's
      const bool need = act && k <= lmax, last = k >= lmax;
      int n = 0;
      for (int h = 0; h * LN < H && __any_sync(0xffffffffu, need && !last); ++h) {
        const int r = h * LN + gl, entry = e0 + r, w = entry >> 5;
        uint64_t x = __shfl_sync(0xffffffffu, word[0], w & (LN - 1), LN);
#pragma unroll
        for (int y = 1; y < NW; ++y) {
          if (LN * y >= S) break;
          const uint64_t z = __shfl_sync(0xffffffffu, word[y], w & (LN - 1), LN);
          if (w / LN == y) x = z;
        }
        const bool take = need && !last && r < H && ((x >> (2 * (entry & 31))) & 3ull) == kPlus;
        const unsigned b = gballot(take);
        if (take) lo_[n + __popc(b & ((1u << gl) - 1u))] = static_cast<uint16_t>(r);
        n += __popc(b);
      }
      int nn = n;
#pragma unroll
      for (int q0 = 0; q0 < DT; q0 += LN) {  // the vertex's zero entries of this layer
        const bool here = need && q0 + gl < DT && mine >= e0 && mine < e0 + H;
        const unsigned b = gballot(here);
        if (here) lo_[nn + __popc(b & ((1u << gl) - 1u))] = static_cast<uint16_t>(mine - e0);
        nn += __popc(b);
      }
      __syncwarp();
      const int nmax = most(nn), cmax = most(ci);
      const float* Ws = Ps + net.wofs[k];       // [in][H] heads
      const float2* Wg = net.WT2 + net.wofs[k];  // [in][H] (head, remainder)
      const float2* bk = net.WT2 + net.bofs[k];
      float2 s[kPtRows / 2], e[kPtRows / 2];
      Grad<DT> gr[kPtRows];
      int row[kPtRows];
      // An output's value z and gradient: to the next layer's records, or to
      // the Newton system if it is one of the zero entries.
      auto store = [&](int x, int r, float sv, float ev, const Grad<DT>& gd) {
        const ff z = ff_fast_two_sum(sv, ev);
        if (x < n) {
          float o[PS] = {z.hi, z.lo};
#pragma unroll
          for (int d = 0; d < DT; ++d) o[2 + d] = gd.at(d);
#pragma unroll
          for (int h = 0; h < PS / 4; ++h)
            *reinterpret_cast<float4*>(next + x * PS + 4 * h) = make_float4(o[4 * h], o[4 * h + 1], o[4 * h + 2], o[4 * h + 3]);
        } else if (x < nn) {
#pragma unroll
          for (int q = 0; q < DT; ++q)
            if (zl[q] == e0 + r) {
              gv[q] = static_cast<double>(z.hi) + static_cast<double>(z.lo);
#pragma unroll
              for (int d = 0; d < DT; ++d) A[q * DT + d] = gd.at(d);
            }
        }
      };
      for (int b0 = 0; b0 < nmax; b0 += kPass) {
        const int left = nmax - b0;
#pragma unroll
        for (int j = 0; j < kPtRows; ++j) {
          const int x = b0 + LN * j + gl;
          row[j] = x < nn ? lo_[x] : 0;
        }
#pragma unroll
        for (int p = 0; p < kPtRows / 2; ++p) {
          const float2 ba = bk[row[2 * p]], bb = bk[row[2 * p + 1]];
          s[p] = make_float2(ba.x, bb.x);
          e[p] = make_float2(ba.y, bb.y);
          gr[2 * p].zero();
          gr[2 * p + 1].zero();
        }
        auto pass = [&](auto nr) {
          rows_pass<DT, decltype(nr)::value, STAGED, REM>(rec, none, li, ci, cmax, Ws, Wg, row, s, e, gr);
        };
        switch ((left + LN - 1) / LN) {
          case 0:
          case 1: pass(Int<1>()); break;
          case 2: pass(Int<2>()); break;
          case 3: pass(Int<3>()); break;
          case 4: pass(Int<4>()); break;
          case 5: pass(Int<5>()); break;
          case 6: pass(Int<6>()); break;
          default: pass(Int<8>()); break;
        }
        __syncwarp();  // one pass: every input has been read (next may be rec)
#pragma unroll
        for (int j = 0; j < kPtRows; ++j) {
          const int x = b0 + LN * j + gl;
          if (x < nn) store(x, row[j], (j & 1) ? s[j >> 1].y : s[j >> 1].x, (j & 1) ? e[j >> 1].y : e[j >> 1].x, gr[j]);
        }
      }
      __syncwarp();
      // this layer's outputs are the next one's inputs
      ci = n;
      if (k < lall) {
        const int Hn = net.w[k + 2];
        for (int x = gl; x < n; x += LN) li[x] = static_cast<uint16_t>(lo_[x] * Hn);  // < 2^16
      }
      float* t1 = rec;
      rec = next;
      next = t1;
    }
    // the Newton step
    float M[DT];
#pragma unroll
    for (int d = 0; d < DT; ++d) M[d] = 0.f;
    float rhs = 0.f;
    if (act && gl < DT) {
      if (mine >= m) {
#pragma unroll
        for (int d = 0; d < DT; ++d) M[d] = A[gl * DT + d];
        rhs = static_cast<float>(-gv[gl]);
      }
    }
    // box facet 2d: x_d - lo_d, 2d + 1: hi_d - x_d; a polyhedral domain's facet
    // j: c_j - A_j x; values in float64 from the stored coordinates
    if (net.fA != nullptr) {
      double f = 0.0;
      const bool facet = act && gl < DT && mine < m;
      if (facet) f = net.fc[mine];
#pragma unroll
      for (int d = 0; d < DT; ++d) {
        const double x = __shfl_sync(0xffffffffu, xd, d, LN);
        if (facet) {
          const double a = net.fA[(long long)mine * DT + d];
          f -= a * x;
          M[d] = static_cast<float>(-a);
        }
      }
      if (facet) rhs = static_cast<float>(-f);
    } else {
      const int fd = mine >> 1;
      const double x = __shfl_sync(0xffffffffu, xd, mine < m ? fd : 0, LN);
      if (act && gl < DT && mine < m) {
#pragma unroll
        for (int d = 0; d < DT; ++d)
          if (d == fd) M[d] = (mine & 1) ? -1.f : 1.f;
        rhs = static_cast<float>(-((mine & 1) ? (net.hi[fd] - x) : (x - net.lo[fd])));
      }
    }
    bool ok = act;
    const float dx = solve_group<DT, LN>(M, rhs, ok);
    if (ok && gl < DT) st.X[(long long)gl * Vcap + v] = xd + static_cast<double>(dx);
    if (ok && gl == 0) npol += 1;
    __syncwarp();
  }
}

// staged: the weights' heads fit in shared memory behind the vertices'
// workspace (they are used if the network has no remainders).
template <int DT, int LN>
__global__ void __launch_bounds__(kPtThreads, 1) k_polish_rows(NetDesc net, State st, float thr, int mw, int TV,
                                                               long long n_params, int staged) {
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ unsigned long long s_pol;
  if (cta_stopped(st)) return;
  const Counters* last = st.cnt + net.N;
  const long long nV = last->nV_before + last->nsplit;
  if ((long long)blockIdx.x * TV >= nV || nV > st.Vcap) return;
  const bool heads = staged && *net.rem == 0;
  const PtLayout lay = pt_layout(TV, mw, net.S, DT);
  float* Ps = reinterpret_cast<float*>(sm + lay.total);
  if (threadIdx.x == 0) s_pol = 0;
  if (threadIdx.x < pt_record(DT)) reinterpret_cast<float*>(sm + lay.nz)[threadIdx.x] = 0.f;
  if (heads)
    for (long long t = threadIdx.x; t < n_params; t += blockDim.x) Ps[t] = net.WT2[t].x;
  __syncthreads();
  int npol = 0;
  if (heads) polish_vertices<DT, LN, true>(net, st, thr, mw, TV, sm, Ps, nV, npol);
  else polish_vertices<DT, LN, false>(net, st, thr, mw, TV, sm, Ps, nV, npol);
  if (npol) atomicAdd(&s_pol, (unsigned long long)npol);
  __syncthreads();
  if (threadIdx.x == 0 && s_pol) atomic_add_ll(&st.g->polished, static_cast<long long>(s_pol));
}

// Vertices of a CTA, whether the weights' heads are staged, shared memory and
// threads of a launch.
struct PtShape {
  int TV;
  bool staged;
  size_t smem;
  int threads;
};
static PtShape pt_shape(int mw, int S, int D, long long n_params) {
  PtShape p{};
  p.TV = pt_tile_vertices(mw, S, D);
  // the weights' heads beside at least half the vertices, or none
  const size_t heads = (size_t)(n_params + 3) / 4 * 16;
  const int least = std::max(4, p.TV / 2);
  int tv = p.TV;
  while (tv > least && pt_layout(tv, mw, S, D).total + heads > (size_t)kPtSmemAll) tv -= 4;
  p.staged = pt_layout(tv, mw, S, D).total + heads <= (size_t)kPtSmemAll;
  if (p.staged) p.TV = tv;
  p.smem = pt_layout(p.TV, mw, S, D).total + (p.staged ? heads : 0);
  p.threads = p.TV * pt_lanes(mw, D);  // whole warps: TV is a multiple of 4
  return p;
}

template <int DT, int LN>
static cudaError_t pt_launch_d(const NetDesc& net, const State& st, float thr, int mw, int num_sms, long long n_params,
                               cudaStream_t stream) {
  const PtShape shape = pt_shape(mw, net.S, DT, n_params);
  const int TV = shape.TV, threads = shape.threads, staged = shape.staged;
  const size_t smem = shape.smem;
  int per_sm = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_polish_rows<DT, LN>, threads, smem);
  if (e != cudaSuccess) return e;
  const long long tiles = (st.Vcap + TV - 1) / TV;  // persistent: vertices dealt round-robin
  const int grid = (int)std::max<long long>(1, std::min<long long>((long long)num_sms * std::max(1, per_sm), tiles));
  k_polish_rows<DT, LN><<<grid, threads, smem, stream>>>(net, st, thr, mw, TV, n_params, staged);
  return cudaGetLastError();
}

template <int DT>
static cudaError_t pt_attributes() {
  cudaError_t e = cudaFuncSetAttribute(k_polish_rows<DT, 16>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPtSmemAll);
  if constexpr (DT <= 8) {
    const cudaError_t r = cudaFuncSetAttribute(k_polish_rows<DT, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPtSmemAll);
    if (e == cudaSuccess) e = r;
  }
  if constexpr (DT > 1) {
    const cudaError_t r = pt_attributes<DT - 1>();
    if (e == cudaSuccess) e = r;
  }
  return e;
}

template <int DT>
static cudaError_t pt_launch(const NetDesc& net, const State& st, float thr, int mw, int num_sms, long long n_params,
                             cudaStream_t stream) {
  if (net.D == DT) {
    if constexpr (DT <= 8)
      if (pt_lanes(mw, DT) == 8) return pt_launch_d<DT, 8>(net, st, thr, mw, num_sms, n_params, stream);
    return pt_launch_d<DT, 16>(net, st, thr, mw, num_sms, n_params, stream);
  }
  if constexpr (DT > 1) return pt_launch<DT - 1>(net, st, thr, mw, num_sms, n_params, stream);
  return cudaErrorInvalidValue;
}

}  // namespace pc

using namespace pc;

cudaError_t pc_polish_set_attributes() { return pt_attributes<kPtMaxD>(); }

cudaError_t pc_polish_launch(const NetDesc& net, const State& st, float thr, int mw, int num_sms, long long n_params,
                             cudaStream_t stream) {
  return pt_launch<kPtMaxD>(net, st, thr, mw, num_sms, n_params, stream);
}
