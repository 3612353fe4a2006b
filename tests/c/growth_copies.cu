// Host-side check of the copies that grow a context's buffers and hand out its
// results: cudaMemcpy2DAsync takes pitches up to 2^31 - 1 bytes, and no copy
// asks for more, whatever the capacities, also where rows lie further apart; the
// copied ranges stay inside the buffers and cover every live row.  The source is
// included as it is with the copies recorded instead of made (no GPU is needed).
// Prints one line per failure, exits 1 if any.
#include <cuda_runtime.h>

#include <cstdio>
#include <map>
#include <vector>

struct Copied {
  const char *dst, *src;
  size_t bytes;
};
static std::vector<Copied> copies;
static int bad = 0;
static cudaError_t copy_rows(void* dst, size_t dpitch, const void* src, size_t spitch, size_t width, size_t rows,
                             cudaMemcpyKind, cudaStream_t) {
  if (dpitch > 0x7fffffffull || spitch > 0x7fffffffull) {
    std::printf("pitch %zu / %zu\n", dpitch, spitch);
    ++bad;
  }
  for (size_t r = 0; r < rows; ++r)
    copies.push_back({static_cast<char*>(dst) + r * dpitch, static_cast<const char*>(src) + r * spitch, width});
  return cudaSuccess;
}
static cudaError_t copy_one(void* dst, const void* src, size_t n, cudaMemcpyKind, cudaStream_t) {
  copies.push_back({static_cast<char*>(dst), static_cast<const char*>(src), n});
  return cudaSuccess;
}
static cudaError_t no_set(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
static cudaError_t no_sync(cudaStream_t) { return cudaSuccess; }
#define cudaMemcpy2DAsync copy_rows
#define cudaMemcpyAsync copy_one
#define cudaMemsetAsync no_set
#define cudaStreamSynchronize no_sync
#include "pc_core.cu"

static std::map<const char*, size_t> buffers;  // address space that nothing backs
static char* next_address = reinterpret_cast<char*>(1ull << 44);
static void* take(size_t bytes, void*, void*) {
  char* p = next_address;
  next_address += (bytes + 4095) / 4096 * 4096 + 4096;
  buffers[p] = bytes;
  return p;
}
static void give(void*, size_t, void*, void*) {}

static bool inside(const char* p, size_t bytes) {
  auto it = buffers.upper_bound(p);
  if (it == buffers.begin()) return false;
  --it;
  return p + bytes <= it->first + it->second;
}

static void grow(int D, int S, int H, size_t zs, bool tape, long long V, long long E) {
  pc_ctx c;
  c.opt.keep_tape = tape;
  c.alloc_fn = take;
  c.free_fn = give;
  c.shape_D = D;
  c.shape_S = S;
  c.shape_H = H;
  c.shape_zs = zs;
  c.shape_tape = tape;
  c.shape_nz = 3;
  realloc_state(&c, V, E, 1 << 16, false);
  const StateBufs was = c.bufs;
  const long long oV = c.Vcap, oE = c.Ecap;
  copies.clear();
  realloc_state(&c, 2 * V, 2 * E, 1 << 16, true);
  size_t values = 0, rows_x = 0;
  for (const Copied& k : copies) {
    if (!inside(k.dst, k.bytes) || !inside(k.src, k.bytes)) {
      std::printf("copy outside its buffer: V %lld H %d\n", V, H);
      ++bad;
    }
    for (int l = 0; l < was.nz; ++l)
      if (k.src == was.Z[l]) values += k.bytes;
    const char* x = static_cast<const char*>(was.X);
    if (k.src >= x && k.src < x + 8 * D * oV) rows_x += k.bytes;
  }
  if (values != was.nz * zs * H * oV || rows_x != 8ull * D * oV || oE < E) {
    std::printf("rows missing: V %lld H %d: values %zu, coordinates %zu\n", V, H, values, rows_x);
    ++bad;
  }
  // results to the caller
  c.nV = 2 * V - 7;
  c.nE = 2 * E - 7;
  c.net.D = D;
  c.net.S = S;
  c.have_result = true;
  copies.clear();
  char* out = static_cast<char*>(take(8ull * 64 * c.nE, nullptr, nullptr));
  if (pc_vertices(&c, nullptr, nullptr, reinterpret_cast<double*>(out)) != PC_OK ||
      pc_edges(&c, nullptr, nullptr, reinterpret_cast<int32_t*>(out)) != PC_OK ||
      pc_signvectors(&c, nullptr, nullptr, reinterpret_cast<uint64_t*>(out)) != PC_OK) {
    std::printf("results refused: V %lld\n", V);
    ++bad;
  }
  size_t total = 0;
  for (const Copied& k : copies) {
    total += k.bytes;
    if (!inside(k.dst, k.bytes) || !inside(k.src, k.bytes)) ++bad;
  }
  if (total != 8ull * (D + S) * c.nV + 8ull * c.nE) {
    std::printf("result rows missing: V %lld\n", V);
    ++bad;
  }
}

int main() {
  grow(2, 1, 8, 4, false, 1 << 14, 1 << 15);
  grow(4, 17, 128, 4, false, 1 << 21, 1 << 23);   // 1 -> 2 GiB of values
  grow(2, 16, 128, 4, false, 5 << 20, 10 << 20);  // 2.7 -> 5.4
  grow(5, 6, 40, 8, false, 7 << 20, 35 << 20);
  grow(3, 9, 64, 8, true, 9 << 20, 27 << 20);
  grow(2, 1, 4, 4, false, 1ll << 28, 1ll << 29);  // coordinate and sign rows 2 -> 4 GiB apart
  std::printf("%d failures\n", bad);
  return bad ? 1 : 0;
}
