// The D x D Newton solve of the FP64 sign re-decision (newton_warp) on systems
// of every dimension and of condition numbers from 1 to ~2^45: two rows differ by
// 2^-k.  The reference is an elimination in long double.  The step must be as
// accurate as an elimination in float64 with partial pivoting, whose forward
// error is at most a small multiple of D^2 x condition number x 2^-53 of the
// largest component (growth factors of such matrices are a few units): 32 of
// them.  Prints one line per failure, exits 1 if any.
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>

#include "pc_newton.cuh"

constexpr int MD = pc::kMaxD;

__global__ void k_solve(int D, const double* A, const double* gv, double* dl, int* ok, int n) {
  const int w = blockIdx.x, lane = threadIdx.x;
  if (w >= n) return;
  pc::NetDesc net{};
  net.D = D;
  net.m = 0;  // no facets: every row comes from A and gv
  pc::State st{};
  __shared__ int zl[MD];
  if (lane < MD) zl[lane] = lane;
  __syncwarp();
  double d = 0.0;
  const bool r = pc::newton_warp(net, st, 0, zl, A + (long long)w * D * D, gv + (long long)w * D, d);
  if (lane < D) dl[(long long)w * D + lane] = d;
  if (lane == 0) ok[w] = r;
}

// x = A^-1 b; false if singular.
static bool solve(int D, std::vector<long double> A, std::vector<long double> b, std::vector<long double>& x) {
  for (int c = 0; c < D; ++c) {
    int p = c;
    for (int r = c + 1; r < D; ++r)
      if (fabsl(A[r * D + c]) > fabsl(A[p * D + c])) p = r;
    if (A[p * D + c] == 0) return false;
    for (int k = 0; k < D; ++k) std::swap(A[c * D + k], A[p * D + k]);
    std::swap(b[c], b[p]);
    for (int r = c + 1; r < D; ++r) {
      const long double f = A[r * D + c] / A[c * D + c];
      for (int k = c; k < D; ++k) A[r * D + k] -= f * A[c * D + k];
      b[r] -= f * b[c];
    }
  }
  x.assign(D, 0);
  for (int r = D - 1; r >= 0; --r) {
    long double s = b[r];
    for (int k = r + 1; k < D; ++k) s -= A[r * D + k] * x[k];
    x[r] = s / A[r * D + r];
  }
  return true;
}

int main() {
  int bad = 0;
  std::mt19937_64 rng(5);
  std::normal_distribution<double> normal;
  for (int D = 2; D <= MD; ++D) {
    std::vector<double> A, g, cond;
    std::vector<std::vector<long double>> want;
    for (int k = 0; k <= 40; ++k)
      for (int t = 0; t < 8; ++t) {
        std::vector<double> M(D * D), b(D);
        for (int r = 0; r < D; ++r) {
          double s = 0;
          for (int c = 0; c < D; ++c) s += (M[r * D + c] = normal(rng)) * M[r * D + c];
          for (int c = 0; c < D; ++c) M[r * D + c] /= std::sqrt(s);
          b[r] = 1e-6 * normal(rng);
        }
        for (int c = 0; c < D; ++c) M[D + c] = M[c] + std::ldexp(M[D + c], -k);  // rows 0 and 1 differ by 2^-k
        if (t & 1)  // as a network's gradients are: float32 entries (a system that becomes singular by it is left out)
          for (auto& x : M) x = static_cast<float>(x);
        std::vector<long double> L(M.begin(), M.end()), B(D), x, col;
        for (int r = 0; r < D; ++r) B[r] = -static_cast<long double>(b[r]);
        if (!solve(D, L, B, x)) continue;
        long double nA = 0, nI = 0;
        std::vector<long double> rows(D, 0);
        for (int c = 0; c < D; ++c) {
          std::vector<long double> e(D, 0);
          e[c] = 1;
          solve(D, L, e, col);
          for (int r = 0; r < D; ++r) rows[r] += fabsl(col[r]);
        }
        for (int r = 0; r < D; ++r) {
          long double s = 0;
          for (int c = 0; c < D; ++c) s += fabsl(L[r * D + c]);
          nA = std::fmax(nA, s);
          nI = std::fmax(nI, rows[r]);
        }
        const double cn = static_cast<double>(nA * nI);
        if (cn > std::ldexp(1.0, 45)) continue;
        A.insert(A.end(), M.begin(), M.end());
        g.insert(g.end(), b.begin(), b.end());
        cond.push_back(cn);
        want.push_back(x);
      }
    const int n = static_cast<int>(cond.size());
    double *dA, *dg, *dx;
    int* dok;
    if (cudaMalloc(&dA, 8 * A.size()) || cudaMalloc(&dg, 8 * g.size()) || cudaMalloc(&dx, 8 * g.size()) ||
        cudaMalloc(&dok, 4 * n)) {
      std::printf("allocation failed\n");
      return 1;
    }
    cudaMemcpy(dA, A.data(), 8 * A.size(), cudaMemcpyHostToDevice);
    cudaMemcpy(dg, g.data(), 8 * g.size(), cudaMemcpyHostToDevice);
    k_solve<<<n, 32>>>(D, dA, dg, dx, dok, n);
    std::vector<double> x(g.size());
    std::vector<int> ok(n);
    cudaMemcpy(x.data(), dx, 8 * x.size(), cudaMemcpyDeviceToHost);
    if (cudaMemcpy(ok.data(), dok, 4 * n, cudaMemcpyDeviceToHost) != cudaSuccess) {
      std::printf("%s\n", cudaGetErrorString(cudaGetLastError()));
      return 1;
    }
    double worst = 0;
    for (int i = 0; i < n; ++i) {
      long double err = 0, size = 0;
      for (int c = 0; c < D; ++c) {
        err = std::fmax(err, fabsl(x[i * D + c] - want[i][c]));
        size = std::fmax(size, fabsl(want[i][c]));
      }
      const double rel = static_cast<double>(err / size) / (D * D * cond[i] * 0x1p-53);
      if (ok[i]) worst = std::fmax(worst, rel);
      if (!ok[i] || !(rel <= 32.0)) {
        if (bad < 20) std::printf("D %d condition %.2e: ok %d, error %.2e of D^2 cond 2^-53\n", D, cond[i], ok[i], rel);
        ++bad;
      }
    }
    std::printf("D %d: %d systems, largest error %.3f D^2 cond 2^-53\n", D, n, worst);
    cudaFree(dA);
    cudaFree(dg);
    cudaFree(dx);
    cudaFree(dok);
  }
  std::printf("%d failures\n", bad);
  return bad ? 1 : 0;
}
