// Bare collider query: all pairs of spheres closer than r_i + r_j + margin in a
// caller-provided configuration (device arrays in, device arrays out) -- the
// collision detection of section 2.1.1 (both passes: bounding-volume filter,
// then the exact sphere test) without a scene.
//
// Same grid as the scene collider: spheres are binned by Morton cell and sorted by a
// counting sort (by index within a cell); each one scans the forward half of its 27-cell
// neighbourhood (grid.cuh).  The FP32 distance decides every pair that is
// not within its rounding allowance of the threshold; the others pass the exact FP64
// test |x_j + H c - x_i| < (r_i + r_j) + margin, evaluated with round-to-nearest
// operations in the order written (shift, branch vector, squared length left to right),
// in the orientation i < j of the caller's indices, so the result is bit-for-bit the
// set that definition gives.  (Tested in FP64, a candidate cost its warp about 16
// FP64-pipe instructions for one or two active lanes: 1.73 ms of each of the two walks
// of a million spheres, the FP64 pipe busy throughout.)
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <string>
#include <thread>
#include <vector>

#include "dem_internal.cuh"
#include "grid.cuh"
#include "pinned_words.h"
#include "dem.h"

namespace dem {

namespace {
constexpr int kT = 256;

inline unsigned blocks(long long n) { return (unsigned)((n + kT - 1) / kT); }

// Counters of a query, zeroed at its start.
struct PairCtl {
  int bad, blocks;            // extent pass: bad input, blocks done
  // The pairs are summed in 32 bits.  Spheres with more pairs than `many` (2^31 / n) are added
  // up in 64 bits as well; the others have 2^31 pairs together at most, so the sum of
  // all is known: big <= pairs < big + 2^31, `low` the pairs modulo 2^32.
  unsigned long long big;
  unsigned low;
};

// extent of the configuration: min x, max x per axis and max r per block, as ordered keys; the
// last block to finish reduces the partials to ext[0..6] and sets ext[7] to 1 for bad input.
// ctl: zeroed (bad input, blocks done).  In FP64 the comparisons alone kept the
// FP64 pipe busy: 62 us for a million spheres, 18 us for 3001 (now 23 and 8).
__global__ void __launch_bounds__(kT) k_extent(const double *__restrict__ pos,
                                               const double *__restrict__ rad, long long n,
                                               unsigned long long *partials, PairCtl *ctl, double *ext) {
  __shared__ unsigned long long sh[7][kT / 32];
  __shared__ int last;
  unsigned long long v[7] = {~0ull, ~0ull, ~0ull, 0, 0, 0, 0};
  bool bad = false;
  for (long long i = (long long)blockIdx.x * kT + threadIdx.x; i < n; i += (long long)gridDim.x * kT) {
    const double x[3] = {pos[3 * i], pos[3 * i + 1], pos[3 * i + 2]}, r = rad[i];
    const long long rb = __double_as_longlong(r);
    bad |= rb <= 0;   // not positive (NaN, infinity: below)
    unsigned e = (unsigned)(rb >> 52);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      e = max(e, (unsigned)(__double_as_longlong(x[k]) >> 52) & 0x7ff);
      const unsigned long long key = ord_key(x[k]);
      v[k] = min(v[k], key);
      v[3 + k] = max(v[3 + k], key);
    }
    // x + y + z + r must be finite; it is where every magnitude is below 2^1022
    if (e >= 0x7fd) bad |= !isfinite(x[0] + x[1] + x[2] + r);
    v[6] = max(v[6], (unsigned long long)rb);
  }
  if (bad) atomicOr(&ctl->bad, 1);
  auto reduce = [&]() {   // v of thread 0: the block's
#pragma unroll
    for (int q = 0; q < 7; ++q) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long y = __shfl_down_sync(0xffffffffu, v[q], o);
        v[q] = q < 3 ? min(v[q], y) : max(v[q], y);
      }
      if ((threadIdx.x & 31) == 0) sh[q][threadIdx.x >> 5] = v[q];
    }
    __syncthreads();
    if (threadIdx.x == 0)
#pragma unroll
      for (int q = 0; q < 7; ++q)
        for (int w = 1; w < kT / 32; ++w) v[q] = q < 3 ? min(v[q], sh[q][w]) : max(v[q], sh[q][w]);
  };
  reduce();
  if (threadIdx.x == 0) {
    for (int q = 0; q < 7; ++q) partials[7 * blockIdx.x + q] = v[q];
    __threadfence();
    last = atomicAdd(&ctl->blocks, 1) == (int)gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  for (int q = 0; q < 7; ++q) v[q] = q < 3 ? ~0ull : 0ull;
  for (int b = threadIdx.x; b < (int)gridDim.x; b += kT)
    for (int q = 0; q < 7; ++q) {
      const unsigned long long y = __ldcg(&partials[7 * b + q]);
      v[q] = q < 3 ? min(v[q], y) : max(v[q], y);
    }
  reduce();
  if (threadIdx.x == 0) {
    for (int q = 0; q < 6; ++q) ext[q] = key_double(v[q]);
    ext[6] = __longlong_as_double((long long)v[6]);
    ext[7] = *(volatile int *)&ctl->bad;
  }
}

// Cell key, place among the cell's arrivals and walk record of every sphere.  The FP64
// work of the cell (floor, products, conversions) is done here once; k_place permutes it.
__global__ void k_bin_q(const double *__restrict__ pos, const double *__restrict__ rad, long long n,
                        Grid g, uint32_t *key, int *rank, int *count, CellRec raw) {
  long long i = (long long)blockIdx.x * kT + threadIdx.x;
  if (i >= n) return;
  const double x[3] = {pos[3 * i], pos[3 * i + 1], pos[3 * i + 2]};
  int c[3], img[3];
  cell_of(g, x[0], x[1], x[2], c, img);
  const uint32_t m = morton3(c[0], c[1], c[2]);
  key[i] = m;
  rank[i] = atomicAdd(&count[m], 1);
  float f[3];
  for (int k = 0; k < 3; ++k)
    f[k] = g.periodic ? (float)(x[k] - g.L[k] * img[k]) : (float)(x[k] - g.lo[k]);
  raw.wpos[i] = make_float4(f[0], f[1], f[2], (float)rad[i]);
  raw.info[i] = make_int4(c[0] | (c[1] << 10) | (c[2] << 20), img[0], img[1], img[2]);
}

__global__ void k_scatter_q(long long n, const uint32_t *__restrict__ key,
                            const int *__restrict__ rank, const int *__restrict__ start, int *tmp) {
  long long i = (long long)blockIdx.x * kT + threadIdx.x;
  if (i < n) tmp[start[key[i]] + rank[i]] = (int)i;
}

// Each sphere to its slot: cell by cell, by index within a cell (the atomics above left
// that order open).  The records of a cell's members are read by its neighbours in the
// warp as well, so the count of smaller indices costs no memory traffic to speak of.
__global__ void k_place(long long n, const int *__restrict__ tmp, const uint32_t *__restrict__ key,
                        const int *__restrict__ start, CellRec raw, int *order, CellRec cr) {
  long long p = (long long)blockIdx.x * kT + threadIdx.x;
  if (p >= n) return;
  const int i = tmp[p];
  const uint32_t m = key[i];
  const int first = start[m], end = start[m + 1];
  int s = first;
  for (int q = first; q < end; ++q) s += tmp[q] < i;
  order[s] = i;
  cr.wpos[s] = raw.wpos[i];
  cr.info[s] = raw.info[i];
}

// exact test in the caller's orientation (a has the lower index), shift c of b
__device__ inline bool exact_pair(const double4_32a &a, const double4_32a &b, const int c[3],
                                  const Grid &g, double margin) {
  double h0 = 0, h1 = 0, h2 = 0;
  if (g.periodic) {
    h0 = __dmul_rn(g.L[0], (double)c[0]);
    h1 = __dmul_rn(g.L[1], (double)c[1]);
    h2 = __dmul_rn(g.L[2], (double)c[2]);
  }
  const double d0 = __dsub_rn(__dadd_rn(b.x, h0), a.x);
  const double d1 = __dsub_rn(__dadd_rn(b.y, h1), a.y);
  const double d2 = __dsub_rn(__dadd_rn(b.z, h2), a.z);
  const double l2 = __dadd_rn(__dadd_rn(__dmul_rn(d0, d0), __dmul_rn(d1, d1)), __dmul_rn(d2, d2));
  const double R = __dadd_rn(__dadd_rn(a.w, b.w), margin);
  return l2 < __dmul_rn(R, R);
}

// What the walk needs of a configuration.
struct PairView {
  const double *pos, *rad;   // the caller's
  const int *order;          // index of the sphere in each slot
  CellRec cr;
  const int *start;
  double margin;
  long long n;
};

__device__ inline double4_32a sphere(const PairView &v, int i) {
  return make_double4_32a(v.pos[3 * (long long)i], v.pos[3 * (long long)i + 1],
                          v.pos[3 * (long long)i + 2], v.rad[i]);
}

// shift of slot j seen from slot s, over the wrap of j's neighbour cell
__device__ inline void pair_shift(const PairView &v, const Grid &g, int s, int j, const int w[3],
                                  int c[3]) {
  c[0] = c[1] = c[2] = 0;
  if (!g.periodic) return;
  const int4 a = v.cr.info[s], b = v.cr.info[j];
  c[0] = a.y - b.y + w[0]; c[1] = a.z - b.z + w[1]; c[2] = a.w - b.w + w[2];
}

// Is the candidate (s, j) a pair?  d2 and R are FP32 values of the squared distance and
// of the reach plus the grid's slack, which covers their rounding: below (reach - slack)^2
// the exact test holds, so only the band between decides in FP64.
__device__ inline bool is_pair(const PairView &v, const Grid &g, int s, int j, const int w[3],
                               float d2, float R) {
  const float in = R - 2.0f * g.slack, in2 = in * in;
  // (squares outside FP32's normal range say nothing: those sizes go to the exact test)
  if (in > 0.0f && in2 > 1e-30f && in2 < 1e37f && d2 < in2) return true;
  int c[3];
  pair_shift(v, g, s, j, w, c);
  const int is = v.order[s], ij = v.order[j];
  if (is < ij) return exact_pair(sphere(v, is), sphere(v, ij), c, g, v.margin);
  c[0] = -c[0]; c[1] = -c[1]; c[2] = -c[2];
  return exact_pair(sphere(v, ij), sphere(v, is), c, g, v.margin);
}

// Pairs kept per slot in the lists of the count pass (a slot with more walks again when
// its rows are written); slot and wrap in 32 bits, so the lists need n <= 2^26.
constexpr int kPairKeep = 16;
constexpr long long kPairSlots = 1LL << 26;

// Count pass, a thread per slot.  A million spheres at solid fraction 0.62, whole query:
// 4.15 -> 0.53 ms; 3001 spheres: 0.35 -> 0.16 ms.
__global__ void __launch_bounds__(kT) k_pair_count(PairView v, Grid g, unsigned *list, int keep,
                                                   long long many, int *cnt, PairCtl *ctl) {
  const long long sl = (long long)blockIdx.x * kT + threadIdx.x;
  if (sl >= v.n) return;
  const int s = (int)sl;
  int n = 0;
  unsigned *mine = list + sl * kPairKeep;
  walk_cells<true>(g, v.cr.wpos, v.start, v.cr.info[s].x, s, [&](int j, int code, float d2, float R) {
    int w[3];
    code_wrap(code, w);
    if (!is_pair(v, g, s, j, w, d2, R)) return;
    if (n < keep) mine[n] = (unsigned)j | ((unsigned)code << 26);
    ++n;
  });
  cnt[s] = n;
  if (n > many) atomicAdd(&ctl->big, (unsigned long long)n);
}

struct PairOut {
  long long cap;
  int *I, *J, *C;
};

__device__ inline void put_pair(const PairView &v, const Grid &g, const PairOut &o, long long r,
                                int s, int j, const int w[3]) {
  if (r >= o.cap) return;
  int c[3];
  pair_shift(v, g, s, j, w, c);
  const int is = v.order[s], ij = v.order[j];
  const bool fwd = is < ij;
  const int sg = fwd ? 1 : -1;
  o.I[r] = fwd ? is : ij;
  o.J[r] = fwd ? ij : is;
  if (o.C) { o.C[3 * r] = sg * c[0]; o.C[3 * r + 1] = sg * c[1]; o.C[3 * r + 2] = sg * c[2]; }
}

// Rows of the pairs: a warp takes 32 slots, whose rows are consecutive, and writes 32 rows
// at a time from the lists; a slot with more pairs than its list holds walks its cells again.
// Offsets are unsigned (up to 2^32 - 1 pairs), those within a warp's rows relative to its first.
__global__ void __launch_bounds__(kT) k_pair_emit(PairView v, Grid g, const unsigned *__restrict__ list,
                                                  int keep, const unsigned *__restrict__ off,
                                                  PairCtl *ctl, PairOut o) {
  const unsigned all = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const long long base = ((long long)blockIdx.x * kT + threadIdx.x) & ~31LL;
  if (base >= v.n) return;
  const long long me = base + lane < v.n ? base + lane : v.n;
  const unsigned at = off[me], to = off[me < v.n ? me + 1 : v.n];
  const bool listed = to - at <= (unsigned)keep;
  const unsigned begin = __shfl_sync(all, at, 0), lo = at - begin, end = __shfl_sync(all, to, 31) - begin;
  for (unsigned r0 = 0; r0 < end; r0 += 32) {
    const unsigned r = r0 + lane;
    int q = 0;   // the last slot whose rows begin at or before r
#pragma unroll
    for (int step = 16; step > 0; step >>= 1) {
      const unsigned b = __shfl_sync(all, lo, q + step);
      if (b <= r) q += step;
    }
    const unsigned from = __shfl_sync(all, lo, q);
    const bool mine = __shfl_sync(all, (int)listed, q);
    if (r < end && mine) {
      const int s = (int)base + q;
      const unsigned e = list[(long long)s * kPairKeep + (r - from)];
      int w[3];
      code_wrap((int)(e >> 26), w);
      put_pair(v, g, o, (long long)begin + r, s, (int)(e & 0x3ffffffu), w);
    }
  }
  if (!listed) {
    const int s = (int)me;
    long long r = at;
    walk_cells<true>(g, v.cr.wpos, v.start, v.cr.info[s].x, s, [&](int j, int code, float d2, float R) {
      int w[3];
      code_wrap(code, w);
      if (is_pair(v, g, s, j, w, d2, R)) put_pair(v, g, o, r++, s, j, w);
    });
  }
  if (me == v.n - 1) ctl->low = to;
}

double now_s() {
  return std::chrono::duration<double>(std::chrono::steady_clock::now().time_since_epoch()).count();
}

// bounded wait on the caller's stream (DEM_TIMEOUT_S, default 120 s)
cudaError_t bounded_wait(cudaStream_t st, bool *timed_out) {
  *timed_out = false;
  cudaEvent_t ev;
  cudaError_t e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
  if (e != cudaSuccess) return e;
  e = cudaEventRecord(ev, st);
  if (e != cudaSuccess) { cudaEventDestroy(ev); return e; }
  const char *env = std::getenv("DEM_TIMEOUT_S");
  double lim = env ? std::atof(env) : 120.0;
  if (!(lim > 0)) lim = 120.0;
  const double deadline = now_s() + lim;
  while (true) {
    e = cudaEventQuery(ev);
    if (e != cudaErrorNotReady) break;
    if (now_s() > deadline) { *timed_out = true; break; }
    std::this_thread::yield();
  }
  cudaEventDestroy(ev);
  return e == cudaErrorNotReady ? cudaSuccess : e;
}
}  // namespace

// Grid of a pair query: cell edge >= 2 r_max + margin, at most max_side cells per axis.
dem_status pair_grid(int periodic, const double *H, const double lo[3], const double hi[3],
                     double rmax, double margin, Grid &g, std::string &err,
                     int max_side = kMaxGridSide) {
  const double hmin = 2 * rmax + margin;
  g = Grid{};
  g.periodic = periodic;
  g.reach = margin;
  double ext = 0;
  for (int k = 0; k < 3; ++k) {
    if (periodic) {
      const double L = H[4 * k];
      const int n = (int)std::floor(L / hmin);
      if (n < 3) {
        err = "periodic cell edge shorter than 3 * (2 r_max + margin)";
        return DEM_ERR_GEOMETRY;
      }
      g.n[k] = std::min(n, max_side);
      g.L[k] = L;
      g.scale[k] = 1.0 / L;
      ext = std::max(ext, L);
    } else {
      const double e = std::max(hi[k] - lo[k] + 2 * rmax, hmin);
      const int n = std::max(1, std::min((int)std::floor(e / hmin), max_side));
      g.n[k] = n;
      g.lo[k] = lo[k] - rmax;
      g.scale[k] = n / e;
      ext = std::max(ext, e);
    }
    g.Lf[k] = (float)g.L[k];
  }
  g.reachf = (float)margin;
  g.slack = (float)(8.0 * ext * std::ldexp(1.0, -23) + 1e-5 * hmin);
  unsigned B = 1;
  while ((int)B < std::max(g.n[0], std::max(g.n[1], g.n[2]))) B <<= 1;
  g.B = (int)B;
  g.base = 0;
  g.morton = 1;
  return DEM_OK;
}

// Scratch of one query, carved from caller-chosen memory.  The walk's lists take over the
// place of the unsorted records, which are dead once the spheres are in their slots.
struct PairScratch {
  unsigned long long *partials;
  double *ext;
  PairCtl *ctl;
  uint32_t *key;
  int *count, *start, *tmp, *order, *cnt, *off, *ws;
  CellRec raw, cr;
  unsigned *list;
};

constexpr size_t kPairListBytes = kPairKeep * sizeof(unsigned);   // >= one raw record

int extent_blocks(long long n) {
  return (int)std::min<long long>(1024, std::max<long long>(1, (n + kT - 1) / kT));
}

// first part: the extent; second part: the grid of ncell cells
size_t carve_extent(char *base, long long n, PairScratch &s) {
  auto up = [](size_t b) { return (b + 255) / 256 * 256; };
  char *p = base;
  s.ctl = (PairCtl *)p; p += 256;
  s.ext = (double *)p; p += 256;
  s.partials = (unsigned long long *)p; p += up(8 * 7 * extent_blocks(n));
  return (size_t)(p - base);
}
size_t carve_grid(char *base, long long n, long long ncell, PairScratch &s) {
  auto up = [](size_t b) { return (b + 255) / 256 * 256; };
  char *p = base;
  s.count = (int *)p; p += up(sizeof(int) * ncell);
  s.start = (int *)p; p += up(sizeof(int) * (ncell + 1));
  s.list = (unsigned *)p;
  s.raw.wpos = (float4 *)p;
  s.raw.info = (int4 *)(p + up(sizeof(float4) * n));
  p += std::max(up(kPairListBytes * n), up(sizeof(float4) * n) + up(sizeof(int4) * n));
  s.cr.wpos = (float4 *)p; p += up(sizeof(float4) * n);
  s.cr.info = (int4 *)p; p += up(sizeof(int4) * n);
  s.key = (uint32_t *)p; p += up(sizeof(uint32_t) * n);
  s.tmp = (int *)p; p += up(sizeof(int) * n);
  s.order = (int *)p; p += up(sizeof(int) * n);
  s.cnt = (int *)p; p += up(sizeof(int) * n);
  s.off = (int *)p; p += up(sizeof(int) * (n + 1));
  s.ws = (int *)p; p += up(scan_workspace_bytes(std::max<long long>(ncell + 1, n + 1)));
  return (size_t)(p - base);
}

// First phase of a query: the extent of the inputs, into S.ext (device).
void pairs_extent(const double *pos, const double *rad, long long n, const PairScratch &S,
                  cudaStream_t st) {
  cudaMemsetAsync(S.ctl, 0, sizeof(PairCtl), st);
  k_extent<<<extent_blocks(n), kT, 0, st>>>(pos, rad, n, S.partials, S.ctl, S.ext);
}

// Second phase: bin, sort, count, scan, emit; the pair count ends up in S.ctl.
cudaError_t pairs_launch(const double *pos, const double *rad, long long n, const Grid &g,
                         double margin, const PairScratch &S, long long cap, int *I, int *J, int *C,
                         cudaStream_t st) {
  const long long ncell = (long long)g.B * g.B * g.B;
  cudaMemsetAsync(S.count, 0, sizeof(int) * ncell, st);
  k_bin_q<<<blocks(n), kT, 0, st>>>(pos, rad, n, g, S.key, S.cnt, S.count, S.raw);
  exclusive_scan(S.count, S.start, ncell, S.ws, st);
  k_scatter_q<<<blocks(n), kT, 0, st>>>(n, S.key, S.cnt, S.start, S.tmp);
  k_place<<<blocks(n), kT, 0, st>>>(n, S.tmp, S.key, S.start, S.raw, S.order, S.cr);
  const PairView v{pos, rad, S.order, S.cr, S.start, margin, n};
  const int keep = n <= kPairSlots ? kPairKeep : 0;
  k_pair_count<<<blocks(n), kT, 0, st>>>(v, g, S.list, keep, (1LL << 31) / n, S.cnt, S.ctl);
  exclusive_scan(S.cnt, S.off, n, S.ws, st);
  k_pair_emit<<<blocks(n), kT, 0, st>>>(v, g, S.list, keep, (const unsigned *)S.off, S.ctl,
                                        PairOut{cap, I, J, C});
  return cudaGetLastError();
}

// The pair count as the host reads it.
dem_status read_count(const PairCtl &ctl, long long *count, std::string &err) {
  const unsigned long long total = ctl.big + (ctl.low - (unsigned)ctl.big);
  if (total > 0xffffffffULL) {
    err = "more than 2^32-1 pairs";
    return DEM_ERR_CAPACITY;
  }
  *count = (long long)total;
  return DEM_OK;
}

// The extent as the host reads it: errors of the inputs, box and largest radius.
dem_status read_extent(const double ext[8], double lo[3], double hi[3], double *rmax,
                       std::string &err) {
  if (ext[7] != 0) { err = "non-finite position or non-positive radius"; return DEM_ERR_NONFINITE; }
  for (int k = 0; k < 3; ++k) {
    lo[k] = ext[k];
    hi[k] = ext[3 + k];
  }
  *rmax = ext[6];
  return DEM_OK;
}

// Words for the results of the queries under way: a copy into pageable memory stages
// through the driver and returns only when it is done, and a stream synchronization makes
// the default memory pool give its freed memory back, which the next call's scratch pays for.
PinnedWords g_pinned(
    [](size_t bytes) -> void * {
      void *p = nullptr;
      if (cudaHostAlloc(&p, bytes, cudaHostAllocPortable) == cudaSuccess) return p;
      cudaGetLastError();
      return nullptr;
    },
    [](void *p) { cudaFreeHost(p); });

}  // namespace dem

namespace dem {
void set_global_error(const std::string &msg);
}

using namespace dem;

extern "C" dem_status dem_find_pairs(const double *pos_dev, const double *radius_dev, long long n,
                                     int periodic, const double *cell_h, double margin,
                                     long long cap, int *id1_dev, int *id2_dev,
                                     int *cell_dist_dev, long long *count, void *cuda_stream) {
  std::string err;
  auto fail = [&](dem_status c, const std::string &m) { set_global_error(m); return c; };
  if (!count || n < 0 || cap < 0 || !(margin >= 0) || (n > 0 && (!pos_dev || !radius_dev)) ||
      (cap > 0 && (!id1_dev || !id2_dev)))
    return fail(DEM_ERR_INVALID_ARG, "bad pair-query arguments");
  if (periodic && (!cell_h || cell_h[1] != 0 || cell_h[2] != 0 || cell_h[3] != 0 ||
                   cell_h[5] != 0 || cell_h[6] != 0 || cell_h[7] != 0 || !(cell_h[0] > 0) ||
                   !(cell_h[4] > 0) || !(cell_h[8] > 0)))
    return fail(DEM_ERR_INVALID_ARG, "the periodic cell must be diagonal with positive edges");
  if (n > 0x7fffffffLL) return fail(DEM_ERR_CAPACITY, "more than 2^31-1 spheres");
  *count = 0;
  set_global_error("");
  if (n < 2) return DEM_OK;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  PinnedLease pinned(g_pinned);
  char *mem = nullptr, *mem2 = nullptr;
  auto done = [&](dem_status c, const std::string &m) {
    if (mem2) cudaFreeAsync(mem2, st);
    if (mem) cudaFreeAsync(mem, st);
    return c == DEM_OK ? c : fail(c, m);
  };
  // bounded wait for `bytes` copied from the device to the pinned words
  auto fetch = [&](const void *src, size_t bytes) -> dem_status {
    cudaError_t e = cudaGetLastError();
    bool to = false;
    if (e == cudaSuccess &&
        pinned.fetch(
            [&] {
              e = cudaMemcpyAsync(pinned.words(), src, bytes, cudaMemcpyDeviceToHost, st);
              return e == cudaSuccess;
            },
            [&] {
              e = bounded_wait(st, &to);
              return e == cudaSuccess && !to;
            }))
      return DEM_OK;
    if (to) { err = "timed out waiting for the GPU"; return DEM_ERR_TIMEOUT; }
    err = std::string("pair query: ") + cudaGetErrorString(e);
    return DEM_ERR_CUDA;
  };
  if (!pinned.words()) return done(DEM_ERR_OOM, "pinned host allocation failed");
  // phase 1: extent
  PairScratch S{};
  if (cudaMallocAsync((void **)&mem, carve_extent(nullptr, n, S), st) != cudaSuccess) {
    cudaGetLastError();
    mem = nullptr;
    return done(DEM_ERR_OOM, "device allocation failed");
  }
  carve_extent(mem, n, S);
  pairs_extent(pos_dev, radius_dev, n, S, st);
  double lo[3], hi[3], rmax = 0;
  dem_status r = fetch(S.ext, 8 * sizeof(double));
  if (!r) r = read_extent(pinned.words(), lo, hi, &rmax, err);
  Grid g;
  if (!r) r = pair_grid(periodic, cell_h, lo, hi, rmax, margin, g, err);
  if (r) return done(r, err);
  // phase 2: scratch for this grid
  const long long ncell = (long long)g.B * g.B * g.B;
  if (cudaMallocAsync((void **)&mem2, carve_grid(nullptr, n, ncell, S), st) != cudaSuccess) {
    cudaGetLastError();
    mem2 = nullptr;
    return done(DEM_ERR_OOM, "device allocation failed");
  }
  carve_grid(mem2, n, ncell, S);
  const cudaError_t e = pairs_launch(pos_dev, radius_dev, n, g, margin, S, cap, id1_dev, id2_dev,
                                     cell_dist_dev, st);
  if (e != cudaSuccess) return done(DEM_ERR_CUDA, std::string("pair query: ") + cudaGetErrorString(e));
  PairCtl ctl;
  if ((r = fetch(S.ctl, sizeof ctl))) return done(r, err);
  std::memcpy(&ctl, pinned.words(), sizeof ctl);
  r = read_count(ctl, count, err);
  return done(r, err);
}

// ---------------------------------------------------------------------------
// Pair query without allocation.
//
// The scratch of dem_find_pairs_noalloc lives in one file-scope device array
// of fixed size, present on every GPU that loads this library until the process
// exits.  Host code cannot pass the array's name to a kernel (in host code the
// name is only a host-side stand-in); the device address is fetched with
// cudaGetSymbolAddress once per device, with that device current, on the first
// call there.
namespace dem {
namespace {
constexpr long long kNoAllocMaxSpheres = 1LL << 16;   // 65,536 spheres
constexpr int kNoAllocMaxSide = 64;                     // grid cells per axis
constexpr long long kNoAllocMaxCells = (long long)kNoAllocMaxSide * kNoAllocMaxSide * kNoAllocMaxSide;
constexpr size_t up256(size_t b) { return (b + 255) / 256 * 256; }
// the layout of carve_extent() and carve_grid() at the maximum sizes, with room for the
// scan workspace
constexpr size_t kNoAllocBytes =
    2 * 256 + up256(8 * 7 * 256) + up256(4 * kNoAllocMaxCells) + up256(4 * (kNoAllocMaxCells + 1)) +
    up256(kPairListBytes * kNoAllocMaxSpheres) + 2 * up256(16 * kNoAllocMaxSpheres) +
    4 * up256(4 * kNoAllocMaxSpheres) + up256(4 * (kNoAllocMaxSpheres + 1)) + up256(16384);

__device__ __align__(256) unsigned char g_pairs_scratch[kNoAllocBytes];

constexpr int kMaxDevices = 64;
std::mutex g_scratch_mu;
void *g_scratch_dev[kMaxDevices] = {nullptr};

// device address of the scratch array on the current device (set up on first use)
cudaError_t scratch_address(void **out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_scratch_mu);
  if (!g_scratch_dev[dev]) {
    void *p = nullptr;
    e = cudaGetSymbolAddress(&p, g_pairs_scratch);
    if (e != cudaSuccess) return e;
    g_scratch_dev[dev] = p;
  }
  *out = g_scratch_dev[dev];
  return cudaSuccess;
}

// bounded wait that creates nothing: poll the stream until its work is done
cudaError_t bounded_stream_wait(cudaStream_t st, bool *timed_out) {
  *timed_out = false;
  const char *env = std::getenv("DEM_TIMEOUT_S");
  double lim = env ? std::atof(env) : 120.0;
  if (!(lim > 0)) lim = 120.0;
  const double deadline = now_s() + lim;
  while (true) {
    cudaError_t e = cudaStreamQuery(st);
    if (e != cudaErrorNotReady) return e;
    if (now_s() > deadline) { *timed_out = true; return cudaSuccess; }
    std::this_thread::yield();
  }
}
}  // namespace
}  // namespace dem

extern "C" dem_status dem_find_pairs_noalloc(const double *pos_dev, const double *radius_dev,
                                             long long n, int periodic, const double *cell_h,
                                             double margin, long long cap, int *id1_dev,
                                             int *id2_dev, int *cell_dist_dev, long long *count,
                                             void *cuda_stream) {
  std::string err;
  auto fail = [&](dem_status c, const std::string &m) { set_global_error(m); return c; };
  if (!count || n < 0 || cap < 0 || !(margin >= 0) || (n > 0 && (!pos_dev || !radius_dev)) ||
      (cap > 0 && (!id1_dev || !id2_dev)))
    return fail(DEM_ERR_INVALID_ARG, "bad pair-query arguments");
  if (periodic && (!cell_h || cell_h[1] != 0 || cell_h[2] != 0 || cell_h[3] != 0 ||
                   cell_h[5] != 0 || cell_h[6] != 0 || cell_h[7] != 0 || !(cell_h[0] > 0) ||
                   !(cell_h[4] > 0) || !(cell_h[8] > 0)))
    return fail(DEM_ERR_INVALID_ARG, "the periodic cell must be diagonal with positive edges");
  if (n > kNoAllocMaxSpheres)
    return fail(DEM_ERR_CAPACITY, "dem_find_pairs_noalloc takes at most 65536 spheres; use "
                                  "dem_find_pairs for larger configurations");
  *count = 0;
  set_global_error("");
  // set-up first (also for n < 2): the lookup loads this file's device module, and
  // with it the scratch array, on the current device
  void *base = nullptr;
  cudaError_t e = scratch_address(&base);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return fail(DEM_ERR_CUDA, std::string("scratch address: ") + cudaGetErrorString(e));
  }
  if (n < 2) return DEM_OK;
  // one layout for both phases, carved at the largest grid; the previous call's
  // contents are stale: the control words and the cell counters are cleared by the phases
  PairScratch S{};
  const size_t head = carve_extent((char *)base, n, S);
  if (head + carve_grid(nullptr, n, kNoAllocMaxCells, S) > kNoAllocBytes)
    return fail(DEM_ERR_CAPACITY, "internal: pair-query scratch exceeds its static size");
  carve_grid((char *)base + head, n, kNoAllocMaxCells, S);
  cudaStream_t st = (cudaStream_t)cuda_stream;
  pairs_extent(pos_dev, radius_dev, n, S, st);
  // poll (bounded) until the kernels are done, and only then copy to the host: a
  // device-to-pageable copy returns only once it is done, so it must not be the wait
  bool to = false;
  auto fetch = [&](void *dst, const void *src, size_t bytes) -> dem_status {
    cudaError_t q = cudaGetLastError();
    if (q == cudaSuccess) q = bounded_stream_wait(st, &to);
    if (to) { err = "timed out waiting for the GPU"; return DEM_ERR_TIMEOUT; }
    if (q == cudaSuccess) q = cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDeviceToHost, st);
    if (q == cudaSuccess) q = cudaStreamSynchronize(st);
    if (q != cudaSuccess) { err = std::string("pair query: ") + cudaGetErrorString(q); return DEM_ERR_CUDA; }
    return DEM_OK;
  };
  double ext[8], lo[3], hi[3], rmax = 0;
  dem_status r = fetch(ext, S.ext, sizeof ext);
  if (!r) r = read_extent(ext, lo, hi, &rmax, err);
  Grid g;
  if (!r) r = pair_grid(periodic, cell_h, lo, hi, rmax, margin, g, err, kNoAllocMaxSide);
  if (r) return fail(r, err);
  if (pairs_launch(pos_dev, radius_dev, n, g, margin, S, cap, id1_dev, id2_dev, cell_dist_dev,
                   st) != cudaSuccess)
    return fail(DEM_ERR_CUDA, "pair query launch failed");
  PairCtl ctl;
  if ((r = fetch(&ctl, S.ctl, sizeof ctl))) return fail(r, err);
  if ((r = read_count(ctl, count, err))) return fail(r, err);
  return DEM_OK;
}
