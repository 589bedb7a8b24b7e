// Exclusive prefix sum of int arrays (collider cell offsets, per-body CSR
// offsets).  Two launches: the sum of every tile of 2048 items, then a pass that
// scans each tile through shared memory (coalesced loads, per-thread serial scan of
// 8 items, warp-shuffle scan of the thread totals) on top of the sum of the tiles
// before it, which every block adds up for itself -- a few hundred to a few thousand
// ints that sit in L2, cheaper than the launches of a scan of the tile sums.  One
// tile needs the second launch only.  More than kMaxDirect tiles (16.8M items): the
// tile sums are scanned first, by the same two launches.
// Two arrays of the same length can share the launches (grid y).
// out has n + 1 entries: out[n] is the total.  Deterministic (integers; sums are modulo 2^32,
// and the callers whose totals can exceed that check them).
//
// The five launches this replaced (tile scan, scan of the sums with its total, add,
// total) took 2.0-5.8 us each on a GB300 for 1M items, most of it launch latency.
#include "dem_internal.cuh"

namespace dem {

namespace {
constexpr int kThreads = 256;
constexpr int kItems = 8;
constexpr int kTile = kThreads * kItems;
constexpr long long kMaxDirect = 8192;   // tiles whose sums every block adds up itself

struct ScanArgs {
  const int *in[2];
  int *out[2];
  int *sums[2];        // tile sums, or (scanned) their exclusive prefix sums
};

__device__ inline unsigned block_sum(unsigned v) {
  __shared__ unsigned part[kThreads / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
  __syncthreads();
  unsigned s = 0;
#pragma unroll
  for (int w = 0; w < kThreads / 32; ++w) s += part[w];
  return s;
}

__global__ void __launch_bounds__(kThreads) k_tile_sums(ScanArgs a, long long n) {
  const int *__restrict__ in = a.in[blockIdx.y];
  const long long base = (long long)blockIdx.x * kTile;
  unsigned s = 0;
#pragma unroll
  for (int i = 0; i < kItems; ++i) {
    const long long g = base + i * kThreads + threadIdx.x;
    s += g < n ? in[g] : 0;
  }
  s = block_sum(s);
  if (threadIdx.x == 0) a.sums[blockIdx.y][blockIdx.x] = (int)s;
}

// scanned: a.sums already holds the exclusive prefix of the tile sums
__global__ void __launch_bounds__(kThreads) k_scan_tiles(ScanArgs a, long long n, int scanned) {
  __shared__ unsigned tile[kTile];
  __shared__ unsigned warp_tot[kThreads / 32];
  const int *__restrict__ in = a.in[blockIdx.y];
  int *__restrict__ out = a.out[blockIdx.y];
  const int *__restrict__ sums = a.sums[blockIdx.y];
  const long long base = (long long)blockIdx.x * kTile;
  const int t = threadIdx.x;
#pragma unroll
  for (int i = 0; i < kItems; ++i) {
    const long long g = base + i * kThreads + t;
    tile[i * kThreads + t] = (g < n) ? in[g] : 0;
  }
  unsigned before = 0;   // items of the tiles before this one
  if (scanned) {
    before = sums[blockIdx.x];
  } else if (blockIdx.x > 0) {
    for (unsigned b = t; b < blockIdx.x; b += kThreads) before += sums[b];
    before = block_sum(before);
  }
  __syncthreads();
  unsigned v[kItems];
  unsigned run = 0;
#pragma unroll
  for (int i = 0; i < kItems; ++i) {
    v[i] = run;
    run += tile[t * kItems + i];
  }
  // inclusive warp scan of the per-thread totals
  const int lane = t & 31, wid = t >> 5;
  unsigned x = run;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    unsigned y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) warp_tot[wid] = x;
  __syncthreads();
  unsigned off = before + (x - run);
  for (int w = 0; w < wid; ++w) off += warp_tot[w];
#pragma unroll
  for (int i = 0; i < kItems; ++i) tile[t * kItems + i] = v[i] + off;
  if (t == kThreads - 1 && base + kTile >= n) out[n] = (int)(off + run);
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kItems; ++i) {
    const long long g = base + i * kThreads + t;
    if (g < n) out[g] = (int)tile[i * kThreads + t];
  }
}

long long ntiles(long long n) { return (n + kTile - 1) / kTile; }

// ws: scan_workspace_bytes(n)
void scan(ScanArgs a, int narr, long long n, int *ws, cudaStream_t st) {
  if (n <= 0) {
    for (int k = 0; k < narr; ++k) cudaMemsetAsync(a.out[k], 0, sizeof(int), st);
    return;
  }
  const long long nb = ntiles(n);
  int scanned = 0;
  if (nb > 1) {
    for (int k = 0; k < narr; ++k) a.sums[k] = ws + k * nb;
    k_tile_sums<<<dim3((unsigned)nb, narr), kThreads, 0, st>>>(a, n);
    if (nb > kMaxDirect) {
      ScanArgs b{};
      int *next = ws + narr * nb;
      for (int k = 0; k < narr; ++k) {
        b.in[k] = a.sums[k];
        b.out[k] = a.sums[k] = next + k * (nb + 1);
      }
      scan(b, narr, nb, next + narr * (nb + 1), st);
      scanned = 1;
    }
  }
  k_scan_tiles<<<dim3((unsigned)nb, narr), kThreads, 0, st>>>(a, n, scanned);
}
}  // namespace

size_t scan_workspace_bytes(long long n) {
  size_t bytes = 0;
  while (true) {
    long long nb = ntiles(n);
    bytes += (size_t)(4 * nb + 4) * sizeof(int);   // sums and their scan, two arrays
    if (nb <= 1) break;
    n = nb;
  }
  return bytes + 256;
}

void exclusive_scan(const int *in, int *out, long long n, int *ws, cudaStream_t st) {
  scan(ScanArgs{{in, nullptr}, {out, nullptr}, {nullptr, nullptr}}, 1, n, ws, st);
}

void exclusive_scan2(const int *in0, int *out0, const int *in1, int *out1, long long n, int *ws,
                     cudaStream_t st) {
  scan(ScanArgs{{in0, in1}, {out0, out1}, {nullptr, nullptr}}, 2, n, ws, st);
}

}  // namespace dem
