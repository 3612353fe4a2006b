// The Newton step to the exact vertex.
//
// A vertex lies on D zero entries (box facets or neuron pre-activations), all
// affine on the vertex's own piece: the activation pattern is its stored sign
// vector (a neuron is active iff its entry is +).  A forward pass from the
// stored coordinates gives the value g and gradient (float32, forward mode,
// D columns) of each zero entry; one Newton step on the D x D system
// A dx = -g lands on the exact vertex: the system is affine, and the step is
// small (the stored coordinates are FP32-accurate), so the float32 gradient
// adds only (1e-7 relative) x (step) to the result.  Used for
//   * the filtered sign predicate, values in float64 (redecide_batch,
//     pc_phases.cuh): the values of layer l at the exact vertex;
//   * the coordinate polish, values in float-float (pc_polish.cu): the exact
//     vertex itself.
#pragma once

#include "pc_device.cuh"

namespace pc {

// Added to a polyhedral domain's facet entry in a zero list once its row is
// in A / gv: the solve then takes it like a neuron's row.
constexpr int kFacetRow = 1 << 20;

// Rows of a polyhedral domain's facets among the zero entries s_zl[0, nzc)
// of vertex v: facet j has the value c_j - A_j x (x the stored coordinates)
// and the gradient -A_j; they go to the same rows A (q * D + d) and values
// gv[q] as the neurons', and the entry becomes j + kFacetRow (thread q of
// the group handles entry q).
__device__ inline void domain_facet_rows(const NetDesc& net, const State& st, long long v, int* s_zl, int nzc,
                                         int q, double* A, double* gv) {
  if (net.fA == nullptr || q >= nzc) return;
  const int j = s_zl[q];
  if (j >= net.m) return;
  const int D = net.D;
  const double* a = net.fA + (long long)j * D;
  double f = net.fc[j];
  for (int dd = 0; dd < D; ++dd) {
    f -= a[dd] * st.X[(long long)dd * st.Vcap + v];
    A[q * D + dd] = -a[dd];
  }
  gv[q] = f;
  s_zl[q] = j + kFacetRow;
}

// The inverse of M in float32 by one warp (lane r < D: row r of M; all lanes call
// it): Gauss-Jordan elimination of [M | I] with partial pivoting.  Row c of the
// inverse in lane c.  False when singular.
__device__ inline bool invert_warp(int D, const float (&A)[kMaxD], float (&V)[kMaxD]) {
  const int lane = threadIdx.x & 31;
  float M[kMaxD];
#pragma unroll
  for (int c = 0; c < kMaxD; ++c) {
    M[c] = A[c];
    V[c] = lane == c ? 1.f : 0.f;
  }
  int var = -1;  // the column whose pivot this lane's row is
  float diag = 1.f;
#pragma unroll
  for (int c = 0; c < kMaxD; ++c) {
    if (c >= D) break;
    const unsigned key = lane < D && var < 0 ? __float_as_uint(fabsf(M[c])) : 0u;
    const unsigned top = __reduce_max_sync(0xffffffffu, key);
    if (top == 0u) return false;  // uniform
    const int piv = __ffs(__ballot_sync(0xffffffffu, key == top)) - 1;
    const float pv = __shfl_sync(0xffffffffu, M[c], piv);
    if (lane == piv) {
      var = c;
      diag = pv;
    }
    const float f = lane == piv ? 0.f : M[c] / pv;
#pragma unroll
    for (int k = 0; k < kMaxD; ++k)
      if (k > c && k < D) M[k] -= f * __shfl_sync(0xffffffffu, M[k], piv);
#pragma unroll
    for (int k = 0; k < kMaxD; ++k)
      if (k < D) V[k] -= f * __shfl_sync(0xffffffffu, V[k], piv);
  }
  const float inv = 1.f / diag;
  int from = lane;
  for (int c = 0; c < D; ++c) {
    const int src = __ffs(__ballot_sync(0xffffffffu, var == c)) - 1;
    if (lane == c) from = src;
  }
#pragma unroll
  for (int k = 0; k < kMaxD; ++k)
    if (k < D) V[k] = __shfl_sync(0xffffffffu, V[k] * inv, from);
  return true;
}

// Row `lane` < D of a vertex's Newton system: gradient M; returns the right-hand
// side.  Other lanes get zeros.
__device__ __forceinline__ double newton_row(const NetDesc& net, const State& st, long long v, const int* s_zl,
                                             const double* A, const double* gv, double (&M)[kMaxD]) {
  const int D = net.D, m = net.m, lane = threadIdx.x & 31;
#pragma unroll
  for (int c = 0; c < kMaxD; ++c) M[c] = 0.0;
  if (lane >= D) return 0.0;
  const int j = s_zl[lane];
  if (j < m) {
    const int d = j >> 1;
    const double xd = st.X[(long long)d * st.Vcap + v];
#pragma unroll
    for (int c = 0; c < kMaxD; ++c) M[c] = c == d ? ((j & 1) ? -1.0 : 1.0) : 0.0;
    return -((j & 1) ? (net.hi[d] - xd) : (xd - net.lo[d]));
  }
#pragma unroll
  for (int c = 0; c < kMaxD; ++c)
    if (c < D) M[c] = A[lane * D + c];
  return -gv[lane];
}

// The step by elimination in float64 (Gauss-Jordan, partial pivoting), for the
// systems that float32 solves do not converge on; rare, so its registers and
// the ~2000 clocks of each of its divisions stay out of the common path.
// False when the system is singular or not finite.
static __device__ __noinline__ bool newton_warp64(const NetDesc& net, const State& st, long long v, const int* s_zl,
                                                  const double* A, const double* gv, double& dl) {
  const int D = net.D, lane = threadIdx.x & 31;
  double M[kMaxD];
  double r = newton_row(net, st, v, s_zl, A, gv, M);
  int var = -1;  // the column whose pivot this lane's row is
  double diag = 1.0;
#pragma unroll
  for (int c = 0; c < kMaxD; ++c) {
    if (c >= D) break;
    double top = lane < D && var < 0 ? fabs(M[c]) : 0.0;
    int piv = lane;
    for (int o = 16; o > 0; o >>= 1) {
      const double t = __shfl_xor_sync(0xffffffffu, top, o);
      const int p = __shfl_xor_sync(0xffffffffu, piv, o);
      if (t > top || (t == top && p < piv)) {
        top = t;
        piv = p;
      }
    }
    top = __shfl_sync(0xffffffffu, top, 0);  // one answer for the warp, whatever a NaN compared to
    piv = __shfl_sync(0xffffffffu, piv, 0);
    if (!(top > 0.0)) return false;
    const double pv = __shfl_sync(0xffffffffu, M[c], piv);
    if (lane == piv) {
      var = c;
      diag = pv;
    }
    const double f = lane == piv ? 0.0 : M[c] / pv;
#pragma unroll
    for (int k = 0; k < kMaxD; ++k)
      if (k > c && k < D) M[k] -= f * __shfl_sync(0xffffffffu, M[k], piv);
    r -= f * __shfl_sync(0xffffffffu, r, piv);
  }
  const double mine = r / diag;
  dl = 0.0;
  for (int c = 0; c < D; ++c) {
    const int src = __ffs(__ballot_sync(0xffffffffu, var == c)) - 1;
    const double y = __shfl_sync(0xffffffffu, mine, src);
    if (lane == c) dl = y;
  }
  return true;
}

// The same step by one warp (all lanes call it; the zero set has D entries) to
// the accuracy of an elimination in float64, which took 9,500 clocks at D = 3
// (a float64 division takes ~2000 on this chip): float32 solves, by one inverse,
// of residuals formed in float64 (iterative refinement: a correction is about rho
// times the one before, rho ~ condition number x 2^-24).  Two corrections do for
// condition numbers up to a few hundred: the second is then below 2^-29 of the
// step, and what is left, rho x 2^-29, below what the elimination's own rounding
// leaves (condition number x 2^-53).  More are made until that holds.  A system
// whose corrections do not halve, or would take more than kNewtonSolves solves (rho
// above ~1/6), or that is singular in float32 is eliminated in float64.  dl:
// component of the step in lane d < D.  False when the system is singular.
// An elimination per solve instead of the inverse: neuron loop of a 3-64x4-1 net
// 5.25 ms, so 5.11 (5.18 with two corrections and no look at them).
constexpr int kNewtonSolves = 12;

__device__ inline bool newton_warp(const NetDesc& net, const State& st, long long v, const int* s_zl, const double* A,
                                   const double* gv, double& dl) {
  const int D = net.D;
  double M[kMaxD];
  float F[kMaxD];
  double r = newton_row(net, st, v, s_zl, A, gv, M);
  // rows scaled by an exact power of two, so that float32 holds them
  int top = 0;
#pragma unroll
  for (int c = 0; c < kMaxD; ++c) top = max(top, __double2hiint(fabs(M[c])) >> 20);
  const double scale = top > 0 && top < 2046 ? __hiloint2double((2046 - top) << 20, 0) : 1.0;
#pragma unroll
  for (int c = 0; c < kMaxD; ++c) F[c] = static_cast<float>(M[c] * scale);
  float V[kMaxD];
  if (!invert_warp(D, F, V)) return newton_warp64(net, st, v, s_zl, A, gv, dl);
  dl = 0.0;
  float first = 0.f, before = 0.f;  // the largest components of the first solve and of the last one
  for (int it = 0; it < kNewtonSolves; ++it) {
    const float rf = static_cast<float>(r * scale);
    float x = 0.f;
#pragma unroll
    for (int c = 0; c < kMaxD; ++c)
      if (c < D) x = fmaf(V[c], __shfl_sync(0xffffffffu, rf, c), x);
    if ((threadIdx.x & 31) >= D) x = 0.f;
    dl += static_cast<double>(x);
    const float size = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(fabsf(x))));
    if (it == 0) first = size;
    if (it >= 2 && size <= 0x1p-29f * first) return true;
    if (it > 0 && !(size <= 0.5f * before)) break;  // also a NaN
    before = size;
#pragma unroll
    for (int c = 0; c < kMaxD; ++c)
      if (c < D) r = fma(-M[c], static_cast<double>(__shfl_sync(0xffffffffu, x, c)), r);
  }
  return newton_warp64(net, st, v, s_zl, A, gv, dl);
}

// ---------------------------------------------------------------------------
// Float-float evaluation for the coordinate polish.
//
// A value is the unevaluated sum hi + lo of two floats.  Dot products use
// the compensated scheme of Ogita, Rump and Oishi ("Accurate sum and dot
// product", 2005, Dot2): each product is split exactly with the FMA
// (p = a*b, e = fma(a, b, -p)), each addition of p to the running sum is
// split exactly with Knuth's TwoSum, and the error terms (plus the cross
// terms of the low parts) are summed in a float, which is as accurate as a
// dot product in twice the working precision (about 2^-44 of the sum of
// |terms| here).  Parameters come as (hi = float(w), lo = float(w - hi))
// pairs, inputs as hi = float(x), lo = float(x - hi).  On GB300 the FP32
// pipes run about 64x faster than the FP64 units.
struct ff {
  float hi, lo;
};

__device__ __forceinline__ ff ff_fast_two_sum(float a, float b) {  // Dekker; |a| >= |b|
  const float s = a + b;
  return {s, b - (s - a)};
}

}  // namespace pc
