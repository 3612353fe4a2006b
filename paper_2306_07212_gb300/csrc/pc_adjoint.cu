// Adjoint of the vertex coordinates with respect to the network parameters.
//
// The forward pass (Section 4.2) computes every vertex created at neuron n of
// layer l from its edge's endpoints p (+) and q (-) by
//     t  = a / (a - b),  a = z_i(p), b = z_i(q)
//     x0 = x_p + t (x_q - x_p)
//     z0_j = z_j(p) + t (z_j(q) - z_j(p))  (j != i),  z0_i = 0
// and, at the start of every layer, the values of the vertices present then
//     Z_l = W_l act(Z_{l-1}) + b_l,  act_k = z_k if the vertex's entry is +
// (Z_0 = W_0 x + b_0 at the box corners).  With the interpolation tape
// (p, q, t per created vertex) and the per-layer values kept by the forward
// pass, the adjoint replays these formulas in reverse: neuron steps from the
// last to the first (one warp per created vertex scatters to its two
// parents), and at each layer start the products give dL/dW_l, dL/db_l and
// the previous layer's value adjoint.
//
// A few ill-conditioned crossings (dt/da ~ 1 / (a - b)) carry most of a
// gradient, so float32 roundings along their chain show in it directly (2e-7
// of the gradient, other roundings with every run's order of atomic additions).
// The vertices' adjoints are float64 (the steps are bound by their launches and
// round trips, not by arithmetic), and the layer products, which are bound by
// the rate of multiply-adds, are sums of float pairs (Ogita-Rump-Oishi Dot2,
// ~44 bits; activations, weights and adjoints all as pairs) on the FP32 pipes, 64
// times FP64's rate.  The parameter gradient is
// accumulated in float64.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <string>
#include <vector>

#include "pc.h"
#include "pc_ctx.h"
#include "pc_device.cuh"

namespace pc {

constexpr int kAdjLd = 33;  // row stride of the staged tiles of 32 vertices
constexpr int kAdjSmemMax = sizeof(float2) * 2 * kMaxWidth * kAdjLd;
constexpr int kAdjTile = 16;  // vertices of a k_adj_back tile
constexpr int kAdjBackMax = sizeof(float2) * kAdjTile * kMaxWidth;

__device__ __forceinline__ float2 split_pair(double x) {
  const float h = static_cast<float>(x);
  return make_float2(h, static_cast<float>(x - static_cast<double>(h)));
}

// s + e += a b for float pairs a, b (Dot2: exact product, TwoSum, error terms).
__device__ __forceinline__ void dot2(float2 a, float2 b, float& s, float& e) {
  const float p = __fmul_rn(a.x, b.x);
  float er = fmaf(a.x, b.x, -p);
  er = fmaf(a.x, b.y, er);
  er = fmaf(a.y, b.x, er);
  const float t = __fadd_rn(s, p), bb = __fsub_rn(t, s);
  e = __fadd_rn(e, __fadd_rn(__fadd_rn(__fsub_rn(s, __fsub_rn(t, bb)), __fsub_rn(p, bb)), er));
  s = t;
}

__global__ void k_adj_init(const double* gx, double* xbar, long long nV, int D) {
  const long long n = nV * D;
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
    const long long d = t / nV, v = t - d * nV;
    xbar[v * D + d] = gx[t];
  }
}

// Reverse of one neuron step: one warp per vertex created at that step.
template <typename ZT>
__global__ void k_adj_split(NetDesc net, State st, double* xbar, double* zbar, int l, int i, long long v_begin,
                            long long count) {
  const int lane = threadIdx.x & 31;
  const long long w0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
  const long long Vcap = st.Vcap;
  const int D = net.D, H = net.w[l + 1];
  const ZT* Z = static_cast<const ZT*>(st.Z[l]);
  for (long long w = w0; w < count; w += nw) {
    const long long v0 = v_begin + w;
    const int p = st.tape_pq[v0], q = st.tape_pq[st.tape_cap + v0];
    const double t = st.tape_t[v0];
    const ZT* zp = Z + (long long)p * H;
    const ZT* zq = Z + (long long)q * H;
    const double a = static_cast<double>(zp[i]), b = static_cast<double>(zq[i]);
    const double inv = 1.0 / (a - b);
    double tb = 0.0;
    if (lane < D) {
      const double xb = xbar[v0 * D + lane];
      if (xb != 0.0) {
        atomicAdd(&xbar[(long long)p * D + lane], xb - t * xb);
        atomicAdd(&xbar[(long long)q * D + lane], t * xb);
        tb = xb * (st.X[(long long)lane * Vcap + q] - st.X[(long long)lane * Vcap + p]);
      }
    }
    for (int j = lane; j < H; j += 32) {
      if (j == i) continue;
      const double zb = zbar[v0 * H + j];
      if (zb == 0.0) continue;
      atomicAdd(&zbar[(long long)p * H + j], zb - t * zb);
      atomicAdd(&zbar[(long long)q * H + j], t * zb);
      tb += zb * (static_cast<double>(zq[j]) - static_cast<double>(zp[j]));
    }
    for (int o = 16; o > 0; o >>= 1) tb += __shfl_xor_sync(0xffffffffu, tb, o);
    if (lane < 2 && tb != 0.0)  // dt/da = -b / (a - b)^2, dt/db = a / (a - b)^2
      atomicAdd(&zbar[(long long)(lane ? q : p) * H + i], tb * inv * ((lane ? a : -b) * inv));
  }
}

// Layer start, parameter part: dW_l[j][k] += sum_v zbar_l[j][v] act_k(v) and
// db_l[j] += sum_v zbar_l[j][v] over the vertices present at the layer start.
// Tiles of 32 vertices are staged in shared memory; each thread owns up to 32
// (j, k) entries; blockIdx.y selects a group of 512 x 32 entries.
template <typename ZT>
__global__ void __launch_bounds__(512) k_adj_wgrad(NetDesc net, State st, const double* zbar, double* gW, int l,
                                                   long long nVl) {
  extern __shared__ float2 sh[];
  constexpr int EPT = 32, TV = 32, LD = kAdjLd;  // rows padded: a tile is stored vertex by vertex, read row by row
  const int H = net.w[l + 1], K = net.w[l];
  float2* zt = sh;            // [H][LD]
  float2* at = sh + H * LD;   // [K][LD]
  const long long Vcap = st.Vcap;
  const ZT* Zin = static_cast<const ZT*>(st.Z[l > 0 ? l - 1 : 0]);
  const int e0 = blockIdx.y * blockDim.x * EPT;
  float s[EPT], er[EPT];
#pragma unroll
  for (int q = 0; q < EPT; ++q) s[q] = er[q] = 0.f;
  float bs = 0.f, be = 0.f;
  for (long long base = (long long)blockIdx.x * TV; base < nVl; base += (long long)gridDim.x * TV) {
    for (int t = threadIdx.x; t < H * TV; t += blockDim.x) {
      const int c = t / H, r = t - c * H;
      zt[r * LD + c] = base + c < nVl ? split_pair(zbar[base * H + t]) : make_float2(0.f, 0.f);
    }
    for (int t = threadIdx.x; t < K * TV; t += blockDim.x) {
      const int c = t / K, k = t - c * K;
      double val = 0.0;
      if (base + c < nVl) {
        if (l == 0) {
          val = st.X[(long long)k * Vcap + base + c];
        } else {
          const ZT z = Zin[base * K + t];
          val = z <= ZT(0) ? 0.0 : static_cast<double>(z);  // active iff its sign entry is +
        }
      }
      at[k * LD + c] = split_pair(val);
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < EPT; ++q) {
      const int e = e0 + q * blockDim.x + threadIdx.x;
      if (e < H * K) {
        const int j = e / K, k = e % K;
#pragma unroll 4
        for (int c = 0; c < TV; ++c) dot2(zt[j * LD + c], at[k * LD + c], s[q], er[q]);
      }
    }
    if (blockIdx.y == 0 && threadIdx.x < H)
      for (int c = 0; c < TV; ++c) dot2(zt[threadIdx.x * LD + c], make_float2(1.f, 0.f), bs, be);
    __syncthreads();
  }
#pragma unroll
  for (int q = 0; q < EPT; ++q) {
    const int e = e0 + q * blockDim.x + threadIdx.x;
    const double g = static_cast<double>(s[q]) + static_cast<double>(er[q]);
    if (e < H * K && g != 0.0) atomicAdd(&gW[net.wofs[l] + e], g);
  }
  const double g = static_cast<double>(bs) + static_cast<double>(be);
  if (blockIdx.y == 0 && threadIdx.x < H && g != 0.0) atomicAdd(&gW[net.bofs[l] + threadIdx.x], g);
}

// Layer start, value part: zbar_{l-1}[v][k] = act'_k(v) sum_j W_l[j][k] zbar_l[v][j].
// A tile's rows of zbar_l are split into float pairs once in shared memory;
// consecutive threads take consecutive k, so weights and rows are coalesced and
// zbar_l[v][j] is one broadcast.  A weight is a float pair too; the remainders are
// read only for a network that has any (NetDesc::rem).
template <typename ZT, bool PAIRS>
__device__ __forceinline__ void adj_back(const NetDesc& net, const State& st, const double* zbar, double* zprev, int l,
                                         long long nVl, float2* sh) {
  const int H = net.w[l + 1], K = net.w[l];
  const float* W = net.W32 + net.wofs[l];
  const float* R = net.R32 + net.wofs[l];
  const ZT* Zin = static_cast<const ZT*>(st.Z[l - 1]);
  for (long long base = (long long)blockIdx.x * kAdjTile; base < nVl; base += (long long)gridDim.x * kAdjTile) {
    const int n = nVl - base < kAdjTile ? int(nVl - base) : kAdjTile;
    for (int t = threadIdx.x; t < n * H; t += blockDim.x) sh[t] = split_pair(zbar[base * H + t]);
    __syncthreads();
    for (int t = threadIdx.x; t < n * K; t += blockDim.x) {
      const int c = t / K, k = t - c * K;
      float s = 0.f, e = 0.f;
      if (!(Zin[base * K + t] <= ZT(0)))  // active iff its sign entry is +
        for (int j = 0; j < H; ++j)
          dot2(sh[c * H + j], make_float2(W[(long long)j * K + k], PAIRS ? R[(long long)j * K + k] : 0.f), s, e);
      zprev[base * K + t] = static_cast<double>(s) + static_cast<double>(e);
    }
    __syncthreads();
  }
}

template <typename ZT>
__global__ void __launch_bounds__(256) k_adj_back(NetDesc net, State st, const double* zbar, double* zprev, int l,
                                                  long long nVl) {
  extern __shared__ float2 sh[];  // [kAdjTile][H]
  if (*net.rem) adj_back<ZT, true>(net, st, zbar, zprev, l, nVl, sh);
  else adj_back<ZT, false>(net, st, zbar, zprev, l, nVl, sh);
}

template <typename ZT>
static void run_backward(pc_ctx* c, const State& st, double* xbar, double* zb[2], double* gW) {
  const NetDesc& net = c->net;
  const Counters* hc = static_cast<const Counters*>(c->h_cnt);
  for (int l = net.L - 1; l >= 0; --l) {
    double* zl = zb[l & 1];
    for (int i = net.w[l + 1] - 1; i >= 0; --i) {
      const int n = net.off[l] + i;
      const long long cnt = hc[n + 1].nsplit, vb = hc[n + 1].nV_before;
      if (cnt <= 0) continue;
      const int blocks = int(std::min<long long>((cnt + 7) / 8, 4096));
      k_adj_split<ZT><<<blocks, 256, 0, c->stream>>>(net, st, xbar, zl, l, i, vb, cnt);
      if (cudaPeekAtLastError() != cudaSuccess) return;
    }
    const Counters& s0 = hc[net.off[l]];
    const long long nVl = s0.nV_before + s0.nsplit;
    const int H = net.w[l + 1], K = net.w[l];
    const int gy = (H * K + 512 * 32 - 1) / (512 * 32);
    const size_t smem = sizeof(float2) * (H + K) * kAdjLd;  // <= kAdjSmemMax (widths <= 256)
    const int gx = int(std::max<long long>(1, std::min<long long>((nVl + 31) / 32, 2 * c->num_sms)));
    k_adj_wgrad<ZT><<<dim3(gx, gy), 512, smem, c->stream>>>(net, st, zl, gW, l, nVl);
    if (l > 0) {
      const int gb = int(std::max<long long>(1, std::min<long long>((nVl + kAdjTile - 1) / kAdjTile, 8 * c->num_sms)));
      k_adj_back<ZT><<<gb, 256, sizeof(float2) * kAdjTile * H, c->stream>>>(net, st, zl, zb[(l - 1) & 1], l, nVl);
    }
  }
}


}  // namespace pc

using namespace pc;

void pc_adjoint_set_attributes() {
  cudaFuncSetAttribute(k_adj_wgrad<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, kAdjSmemMax);
  cudaFuncSetAttribute(k_adj_wgrad<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, kAdjSmemMax);
  static_assert(kAdjBackMax <= 48 * 1024, "k_adj_back runs without a shared-memory attribute");
}

extern "C" pc_status pc_backward(pc_ctx* c, const double* grad_x, double* grad_params, void* stream) {
  if (!c || !grad_x || !grad_params) return PC_ERR_INVALID;
  if (!c->have_result) return c->fail(PC_ERR_INVALID, "no extraction result");
  if (!c->opt.keep_tape) return c->fail(PC_ERR_NO_TAPE, "extraction ran without keep_tape");
  cudaSetDevice(c->device);
  c->stream = static_cast<cudaStream_t>(stream);
  const NetDesc& net = c->net;
  const int D = net.D;
  const long long nV = c->nV;
  long long np = 0;
  for (int l = 0; l < net.L; ++l) np += (long long)net.w[l + 1] * (net.w[l] + 1);
  // value adjoints of layer l: of the vertices there at its end, in the buffer
  // of its parity
  const Counters* hc = static_cast<const Counters*>(c->h_cnt);
  size_t zneed[2] = {0, 0};
  for (int l = 0; l < net.L; ++l) {
    const Counters& end = hc[net.off[l + 1]];
    const long long n = l + 1 < net.L ? end.nV_before + end.nsplit : nV;
    zneed[l & 1] = std::max<size_t>(zneed[l & 1], sizeof(double) * net.w[l + 1] * n);
  }
  const size_t need[4] = {sizeof(double) * D * nV, zneed[0], zneed[1], sizeof(double) * (np + D * nV)};
  for (int k = 0; k < 4; ++k) {
    if (c->adj_bytes[k] < need[k]) {
      ctx_free(c, c->adj[k]);
      c->adj[k] = ctx_alloc(c, need[k]);
      c->adj_bytes[k] = c->adj[k] ? need[k] : 0;
      if (!c->adj[k]) return c->fail(PC_ERR_OOM, "adjoint buffer allocation failed");
    }
  }
  double* xbar = static_cast<double*>(c->adj[0]);
  double* zb[2] = {static_cast<double*>(c->adj[1]), static_cast<double*>(c->adj[2])};
  double* gW = static_cast<double*>(c->adj[3]);
  double* gx = gW + np;
  cudaError_t e = cudaSuccess;
  auto ok = [&](cudaError_t r) { if (e == cudaSuccess) e = r; };
  ok(cudaMemsetAsync(gW, 0, sizeof(double) * np, c->stream));
  // the last layer's adjoints start at zero; the others are written whole by
  // k_adj_back before they are added to
  ok(cudaMemsetAsync(zb[(net.L - 1) & 1], 0, sizeof(double) * net.w[net.L] * nV, c->stream));
  ok(cudaMemcpyAsync(gx, grad_x, sizeof(double) * D * nV, cudaMemcpyDefault, c->stream));
  if (e != cudaSuccess) return c->fail(PC_ERR_CUDA, cudaGetErrorString(e));
  k_adj_init<<<std::max<long long>(1, std::min<long long>((D * nV + 255) / 256, 4096)), 256, 0, c->stream>>>(
      gx, xbar, nV, D);
  const State st = pc_make_state(c);
  if (net.precision == PC_PREC_FP64) run_backward<double>(c, st, xbar, zb, gW);
  else run_backward<float>(c, st, xbar, zb, gW);
  ok(cudaGetLastError());
  ok(cudaMemcpyAsync(grad_params, gW, sizeof(double) * np, cudaMemcpyDefault, c->stream));
  ok(cudaStreamSynchronize(c->stream));
  if (e != cudaSuccess) return c->fail(PC_ERR_CUDA, cudaGetErrorString(e));
  return PC_OK;
}
