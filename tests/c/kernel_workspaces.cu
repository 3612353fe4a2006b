// Host-side check of the polish's launches, of the re-decision's and the other
// kernels' shared memory, for every layer width, input dimension, sign-word count
// and number of parameters the library accepts: whole warps within the CTA,
// workspace and staged weights within the launch attribute, regions aligned, in
// place and without overlap, list entries and weight-row offsets within 16 bits,
// one pass of the inputs wherever the outputs overwrite them.  It includes the
// sources as they are and launches nothing.  Prints one line per failure, exits 1
// if any.
#include <cstdio>
#include <utility>
#include <vector>

#include "pc_polish.cu"
#include "pc_phases.cuh"

int main() {
  int bad = 0;
  auto fail = [&](const char* what, int mw, int D, int S, long long v) {
    if (bad < 20) std::printf("%s: width %d D %d S %d -> %lld\n", what, mw, D, S, v);
    ++bad;
  };
  // (offset, bytes) regions in order: aligned, not overlapping, up to total
  auto regions = [&](const char* what, std::vector<std::pair<size_t, size_t>> r, size_t total, int mw, int D, int S) {
    size_t end = 0;
    for (auto& x : r) {
      if (x.first % 16 || x.first < end) fail(what, mw, D, S, (long long)x.first);
      end = x.first + x.second;
    }
    if (end > total) fail(what, mw, D, S, (long long)end);
  };
  using namespace pc;
  for (int mw = 1; mw <= kMaxWidth; ++mw)
    for (int S = 1; S <= kMaxWords; ++S)
      for (int D = 1; D <= kMaxD && D <= mw; ++D) {
        const int LN = pt_lanes(mw, D);
        if (LN < D) fail("fewer lanes than rows of the system", mw, D, S, LN);
        const size_t fit = kPtSmemAll - pt_layout(pt_tile_vertices(mw, S, D), mw, S, D).total;
        const long long most = 16ll * kMaxWidth * (kMaxWidth + 1), edge = (long long)(fit / 4);
        for (long long n : {1ll, (long long)mw * (D + 1), edge - 1, edge, edge + 1, 2 * edge, 20000ll, 50000ll, most}) {
          if (n < 1) continue;
          const PtShape p = pt_shape(mw, S, D, n);
          const PtLayout L = pt_layout(p.TV, mw, S, D);
          if (p.TV < 4 || p.threads % 32 || p.threads > kPtThreads || p.threads != p.TV * LN)
            fail("polish threads", mw, D, S, p.threads);
          if (p.smem > (size_t)kPtSmemAll || L.total + (p.staged ? 4 * n : 0) > p.smem)
            fail("polish shared memory", mw, D, S, (long long)p.smem);
          const size_t rec = (size_t)p.TV * L.rows * pt_record(D) * 4;
          const bool two = L.rows > kPtRows * LN;  // more outputs than a pass: the next layer's records have their own place
          if (two != (L.alo + rec <= L.J)) fail("polish records", mw, D, S, L.rows);
          regions("polish regions", {{L.A, 4ull * p.TV * D * D}, {L.gv, 8ull * p.TV * D}, {L.ahi, rec}, {L.alo, two ? rec : 0},
                                     {L.J, 4ull * p.TV * L.rows}, {L.zl, 4ull * p.TV * D}, {L.nz, 4ull * pt_record(D)}},
                  L.total, mw, D, S);
        }
        const int P = rd_batch_size(mw, D, S);
        if (P < 1 || P > kWarps / 2) fail("re-decision batch size", mw, D, S, P);
        const RdLayout R = rd_layout(P, mw, D, S);
        if (R.total > (size_t)kRdSmemMax) fail("re-decision shared memory", mw, D, S, (long long)R.total);
        const size_t q = P;
        regions("re-decision regions",
                {{R.a, q * mw * 8}, {R.an, q * mw * 8}, {R.A, q * D * D * 8}, {R.gv, q * D * 8}, {R.dlt, q * D * 8},
                 {R.J, q * mw * D * 4}, {R.Jn, q * mw * D * 4}, {R.sc, q * mw * 4}, {R.zl, q * D * 4}, {R.nz, q * 4},
                 {R.ok, q * 4}, {R.li, q * 32 * S * 2}, {R.cnt, q * kMaxL * 4}},
                R.total, mw, D, S);
      }
  static_assert((kMaxWidth - 1) * kMaxWidth < 1 << 16, "an input's weight row, as a 16-bit offset");
  // a warp's buffers and the queues hold what comes between two looks at them
  static_assert(2 * 2 * (kMaxD - 1) <= kPairCap && 32 <= kLaCap, "a round of a warp");
  static_assert(kPendCap >= 2 * kPendRounds * kSplits, "splits queued between two looks");
  static_assert(kDecideCap % (2 * kBlock) == 0 && kDecideCap % (2 * kSplits) == 0, "vertices queued between two looks");
  static_assert(kMaxD - 1 <= 16 && kMaxWords <= 2 * kGroup, "zeros and words of a half warp");
  std::printf("%d failures\n", bad);
  return bad ? 1 : 0;
}
