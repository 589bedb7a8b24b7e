// Collider: the first, approximate pass of the two-pass detection of the
// Yade text (section 2.1.1, eq. 2.1-2.2), run only when a body has moved more
// than the sweep margin ("Verlet distance", eq. 2.3-2.4).
//
// GB300 design (replaces the single-threaded insertion-sort sweep and prune):
//   1. bin every sphere into a uniform grid of cell edge >= 2 r_max + 2 dL
//      (periodic: in the wrapped reference cell, keeping the integer image);
//   2. counting sort over the Morton codes of the cells (atomics only for the
//      per-cell counts and arrival places), each cell's bodies by id, so the
//      resulting body order ("slots") is deterministic;
//   3. permute the body arrays into that order (spatial locality for every
//      later gather);
//   4. each body scans its whole 27-cell neighbourhood and keeps
//      the partners with |x2 + H c - x1| < r1 + r2 + 2 dL, tested conservatively in FP32
//      on wrapped coordinates; each body's partners are sorted by id on chip.  A
//      row is oriented by id, not by slot: body 1 is the sphere with the smaller id
//      (the canonical id1 < id2 of the interaction container), so a body's partners of
//      larger id are its rows and those of smaller id its "down" list, both in order;
//   5. prefix sums of the two counts, then one pass over the rows writes them and
//      merges the contact history of the previous table by looking each pair up in the
//      old row range of its body 1 (the potential / real interaction lifecycle of
//      section 3.1.7);
//   6. one pass over the down entries finds the row of each.
// Each pair is met from both sides (twice the distance tests of a forward half shell),
// which is what makes every list come out complete and sorted without atomics, scattered
// writes or sorts of the table.
// So a body's rows, down list first, then its own range, run in increasing order
// of partner id; the force gather sums them in that order.  With the orientation
// by id, the FP64 arithmetic of a step depends on the bodies and their contact
// histories only, not on the slot order, the times of the collider runs or the
// other sub-scenes in the arrays: a sub-scene advances bit for bit as it would
//   alone.
#include "dem_internal.cuh"
#include "grid.cuh"

namespace dem {

namespace {
constexpr int kT = 256;

__global__ void k_bbox(const double4_32a *__restrict__ pos, long long N, double *partials) {
  __shared__ double sh[6][kT];
  double lo[3] = {1e300, 1e300, 1e300}, hi[3] = {-1e300, -1e300, -1e300};
  for (long long i = (long long)blockIdx.x * kT + threadIdx.x; i < N; i += (long long)gridDim.x * kT) {
    double4_32a p = pos[i];
    lo[0] = fmin(lo[0], p.x - p.w); hi[0] = fmax(hi[0], p.x + p.w);
    lo[1] = fmin(lo[1], p.y - p.w); hi[1] = fmax(hi[1], p.y + p.w);
    lo[2] = fmin(lo[2], p.z - p.w); hi[2] = fmax(hi[2], p.z + p.w);
  }
  for (int k = 0; k < 3; ++k) { sh[k][threadIdx.x] = lo[k]; sh[3 + k][threadIdx.x] = hi[k]; }
  __syncthreads();
  for (int o = kT / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o)
      for (int k = 0; k < 3; ++k) {
        sh[k][threadIdx.x] = fmin(sh[k][threadIdx.x], sh[k][threadIdx.x + o]);
        sh[3 + k][threadIdx.x] = fmax(sh[3 + k][threadIdx.x], sh[3 + k][threadIdx.x + o]);
      }
    __syncthreads();
  }
  if (threadIdx.x == 0)
    for (int k = 0; k < 6; ++k) partials[6 * blockIdx.x + k] = sh[k][0];
}

// Grid of body i: the one grid, or the grid of its sub-scene.
__device__ __forceinline__ const Grid &grid_of(const Grid *__restrict__ grids,
                                               const int *__restrict__ sid, int multi, long long i) {
  return grids[multi ? sid[i] : 0];
}

// Bounding boxes of the sub-scenes: keys[k * cap + q] (k = 0..2 lower, 3..5 upper
// bounds of x - r / x + r), lower keys preset to all ones and upper to zero.  A
// warp whose bodies share one sub-scene (the usual case: bodies are grouped by
// sub-scene) reduces in registers and issues six atomics.
__global__ void k_bbox_sub(const double4_32a *__restrict__ pos, const int *__restrict__ sid,
                           long long N, int cap, unsigned long long *keys) {
  const int lane = threadIdx.x & 31;
  const long long stride = (long long)gridDim.x * kT;
  for (long long base = (long long)blockIdx.x * kT + (threadIdx.x & ~31); base < N; base += stride) {
    const long long i = base + lane;
    int q = -1;
    unsigned long long k[6] = {~0ull, ~0ull, ~0ull, 0ull, 0ull, 0ull};
    if (i < N) {
      q = sid[i];
      const double4_32a p = pos[i];
      k[0] = ord_key(p.x - p.w); k[1] = ord_key(p.y - p.w); k[2] = ord_key(p.z - p.w);
      k[3] = ord_key(p.x + p.w); k[4] = ord_key(p.y + p.w); k[5] = ord_key(p.z + p.w);
    }
    const int q0 = __shfl_sync(0xffffffffu, q, 0);
    const bool uniform = __all_sync(0xffffffffu, q == q0 || q < 0);
    if (uniform) {
      for (int o = 16; o > 0; o >>= 1)
        for (int c = 0; c < 6; ++c) {
          const unsigned long long v = __shfl_down_sync(0xffffffffu, k[c], o);
          k[c] = c < 3 ? (v < k[c] ? v : k[c]) : (v > k[c] ? v : k[c]);
        }
      if (lane == 0 && q0 >= 0)
        for (int c = 0; c < 6; ++c) {
          if (c < 3) atomicMin(&keys[(long long)c * cap + q0], k[c]);
          else atomicMax(&keys[(long long)c * cap + q0], k[c]);
        }
    } else if (q >= 0) {
      for (int c = 0; c < 6; ++c) {
        if (c < 3) atomicMin(&keys[(long long)c * cap + q], k[c]);
        else atomicMax(&keys[(long long)c * cap + q], k[c]);
      }
    }
  }
}

// Cell key, place among the cell's arrivals and walk record (FP32 position relative to the
// grid, cell, image) of every body; bodies of a removed sub-scene (grid with no cells) get
// the sentinel key `dead`, which sorts them behind every live body.  The FP64 work of the
// cell (floor, products, conversions) is done here once; k_reorder permutes the record.
__global__ void k_bin(const double4_32a *__restrict__ pos, const int *__restrict__ sid, long long N,
                      const Grid *__restrict__ grids, int multi, uint32_t dead, uint32_t *key,
                      int *rank, int *count, CellRec raw) {
  long long i = (long long)blockIdx.x * kT + threadIdx.x;
  if (i >= N) return;
  const Grid &g = grid_of(grids, sid, multi, i);
  uint32_t m = dead;
  if (g.n[0] > 0) {
    const double4_32a p = pos[i];
    int c[3], img[3];
    cell_of(g, p.x, p.y, p.z, c, img);
    m = (uint32_t)cell_index(g, c[0], c[1], c[2]);
    const double x[3] = {p.x, p.y, p.z};
    float f[3];
    for (int k = 0; k < 3; ++k) {
      double shift = g.L[k] * img[k];
      if (g.periodic && g.sheared)   // wrapped position x - H img
        shift = g.H[3 * k] * img[0] + g.H[3 * k + 1] * img[1] + g.H[3 * k + 2] * img[2];
      f[k] = g.periodic ? (float)(x[k] - shift) : (float)(x[k] - g.lo[k]);
    }
    raw.wpos[i] = make_float4(f[0], f[1], f[2], (float)p.w);
    raw.info[i] = make_int4(c[0] | (c[1] << 10) | (c[2] << 20), img[0], img[1], img[2]);
  }
  key[i] = m;
  rank[i] = atomicAdd(&count[m], 1);
}

__global__ void k_scatter(long long N, const uint32_t *__restrict__ key,
                          const int *__restrict__ rank, const int *__restrict__ start, int *tmp) {
  long long i = (long long)blockIdx.x * kT + threadIdx.x;
  if (i < N) tmp[start[key[i]] + rank[i]] = (int)i;
}

// Bodies to their slots: cell by cell, by id within a cell (the order the atomics left
// open).  N: the live bodies (the sentinel cell comes last and is dropped).
__global__ void k_reorder(Bodies src, Bodies dst, long long N, long long cap,
                          const int *__restrict__ tmp, const uint32_t *__restrict__ key,
                          const int *__restrict__ start, CellRec raw,
                          CellRec cr, int *new_to_old, int *slot_of_id, int has_walls, int mixed,
                          const int *__restrict__ id_shift, const CellState *__restrict__ cs,
                          int multi) {
  const long long at = (long long)blockIdx.x * kT + threadIdx.x;
  if (at >= N) return;
  const int o = tmp[at];
  const int oid = src.id[o];
  const uint32_t m = key[o];
  const int first = start[m], end = start[m + 1];
  int p = first;
  for (int q = first; q < end; ++q) p += src.id[tmp[q]] < oid;
  new_to_old[p] = o;
  cr.wpos[p] = raw.wpos[o];
  cr.info[p] = raw.info[o];
  double4_32a x = src.pos[o];
  dst.pos[p] = x;
  const double4_32a v = src.vel[o], w = src.angvel[o];
  dst.vel[p] = v;
  dst.angvel[p] = w;
  if (mixed) {   // the new reference position is x itself: zero offset
    dst.p32[p] = make_float4(0.0f, 0.0f, 0.0f, (float)x.w);
    dst.vw32[2 * p] = make_float4((float)v.x, (float)v.y, (float)v.z, (float)w.x);
    dst.vw32[2 * p + 1] = make_float4((float)w.y, (float)w.z, 0.0f, 0.0f);
    dst.xref32[p] = make_float4((float)x.x, (float)x.y, (float)x.z, 0.0f);
    dst.mprop32[p] = src.mprop32[o];
    dst.ori32[p] = src.ori32[o];   // the mixed path keeps the orientation in FP32
  }
  if (!mixed) dst.ori[p] = src.ori[o];
  dst.mprop[p] = src.mprop[o];
  dst.rdsc[p] = src.rdsc[o];
  dst.xref[p] = make_double4_32a(x.x, x.y, x.z, 0.0);
  const int q = src.sid[o];
  // ids close up over the ranges of removed sub-scenes
  const int id = oid - (id_shift ? id_shift[q] : 0);
  dst.id[p] = id;
  dst.sid[p] = q;
  dst.mat[p] = src.mat[o];
  const uint8_t flags = src.flags[o];
  dst.flags[p] = flags;
  slot_of_id[id] = p;
  dst.live[p] = 0;
  uint8_t near = 0;
  if (has_walls) {
    // a body moves at most the sweep margin from x before the next run, so it can only meet
    // the walls within r + margin now (FP32 distances, with room for their rounding)
    const CellState &c = cs[multi ? q : 0];
    const float reach = (float)(x.w + c.verlet) * 1.0001f;
    const double xs[3] = {x.x, x.y, x.z};
    for (int w = 0; w < 6; ++w) {
      if (c.wall_mask & (1 << w)) {
        const int ax = w >> 1;
        const float d = (float)(xs[ax] - ((w & 1) ? c.box_hi[ax] : c.box_lo[ax]));
        if (!(fabsf(d) * 0.9999f > reach)) near |= (uint8_t)(1 << w);
      }
      // a wall history is read only while its flag is set
      if (flags & (2 << w)) dst.whist[w * cap + p] = src.whist[w * cap + o];
    }
  }
  dst.wnear[p] = near;
}

__global__ void k_slots(const int *__restrict__ id, long long N, int *slot_of_id) {
  const long long s = (long long)blockIdx.x * kT + threadIdx.x;
  if (s < N) slot_of_id[id[s]] = (int)s;
}

// Does the shift of j seen from s leave the range of a packed shift?
__device__ inline bool shift_overflow(const CellRec &cr, int s, int j, int code) {
  int w[3];
  code_wrap(code, w);
  const int4 a = cr.info[s], b = cr.info[j];
  return abs(a.y - b.y + w[0]) > kShiftMax || abs(a.z - b.z + w[1]) > kShiftMax ||
         abs(a.w - b.w + w[2]) > kShiftMax;
}

// Partners of every body, by partner id: the down partners (smaller ids), then the rows'.
//
// Two shapes of the same search.  A thread per body keeps the hits in a shared-memory
// column and places them by rank (the count of smaller ids): 111 us for 300k bodies at
// three rows a body, 605 us for 1M at five (a warp per body 223 us for the 300k; a warp
// per cell 164 and 777 us).  Its 27 cells in turn are a chain of dependent loads, some
// 55 us however few the bodies, so smaller scenes take a warp per body, a lane per
// neighbour cell: 7 us for 1000 bodies, 25 us for 20k, 99 us for 100k (a thread per body 61).
constexpr int kPT = 128;
constexpr long long kWarpBodies = 65536;

__global__ void __launch_bounds__(kPT) k_partners(CellRec cr, const int *__restrict__ sid,
                                                  const int *__restrict__ id, long long N,
                                                  const Grid *__restrict__ grids, int multi,
                                                  const int *__restrict__ start, int *cnt_up,
                                                  int *cnt_down, DevStatus *ds, CandList cl) {
  __shared__ unsigned ent[kCandKeep][kPT];
  __shared__ int ids[kCandKeep][kPT];
  const int tid = threadIdx.x;
  const long long sl = (long long)blockIdx.x * kPT + tid;
  if (sl >= N) return;
  const int s = (int)sl, me = id[s];
  const Grid &g = grid_of(grids, sid, multi, sl);
  int n = 0;
  walk_cells<false>(g, cr.wpos, start, cr.info[s].x, s, [&](int j, int code, float, float) {
    if (n < kCandKeep) ent[n][tid] = (unsigned)j | ((unsigned)code << 26);
    ++n;
  });
  if (n > kCandKeep) {   // for k_partners_warp (no others can exceed cl.many: N < 2^26)
    cl.long_ids[atomicAdd(&ds->n_long, 1)] = s;
    return;
  }
  bool bad = false;
  for (int k = 0; k < n; ++k) {
    const unsigned e = ent[k][tid];
    const int j = (int)(e & 0x3ffffffu);
    ids[k][tid] = __ldg(id + j);
    if (g.periodic) bad |= shift_overflow(cr, s, j, (int)(e >> 26));
  }
  int down = 0;
  unsigned *mine = cl.list + (long long)s * kCandKeep;
  for (int k = 0; k < n; ++k) {
    const int ik = ids[k][tid];
    int rank = 0;
    for (int q = 0; q < n; ++q) rank += ids[q][tid] < ik;
    mine[rank] = ent[k][tid];
    down += ik < me;
  }
  cnt_down[s] = down;
  cnt_up[s] = n - down;
  if (bad) atomicOr(&ds->error, kErrShiftRange);
}

// kLong: the bodies of cl.long_ids; else all N.  A list of more than a warp's lanes is
// ranked in shared memory and written to the spill buffer, so that its body too is walked
// once: with the lists of 32 alone, and such bodies walked four times by single threads,
// a run over 1M dense spheres took 5.0 ms at a sweep margin of r_min (27 partners a body) and
// 14.8 ms at 1.25 r_min (40); now 2.6 and 4.3 ms.
template <bool kLong>
__global__ void __launch_bounds__(kT) k_partners_warp(CellRec cr, const int *__restrict__ sid,
                                                      const int *__restrict__ id, long long N,
                                                      const Grid *__restrict__ grids, int multi,
                                                      const int *__restrict__ start, int *cnt_up,
                                                      int *cnt_down, DevStatus *ds, CandList cl) {
  __shared__ unsigned ent[kT / 32][kLongKeep];
  __shared__ int ids[kT / 32][kLongKeep];
  const unsigned all = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  unsigned *mine = ent[threadIdx.x >> 5];
  int *idm = ids[threadIdx.x >> 5];
  const long long total = kLong ? ds->n_long : N;
  const long long stride = ((long long)gridDim.x * kT) >> 5;
  bool bad = false;
  for (long long at = ((long long)blockIdx.x * kT + threadIdx.x) >> 5; at < total; at += stride) {
    const int s = kLong ? cl.long_ids[at] : (int)at, me = id[s];
    const Grid &g = grid_of(grids, sid, multi, s);
    const float4 a = cr.wpos[s];
    const int packed = cr.info[s].x;
    const int ci[3] = {packed & 1023, (packed >> 10) & 1023, (packed >> 20) & 1023};
    int first = 0, end = 0, code = kNoWrap;
    if (lane < kStencil) stencil_cell(g, start, ci, lane, first, end, code);
    CellShift sh{make_float3(a.x, a.y, a.z), make_float3(0.0f, 0.0f, 0.0f)};
    if (code != kNoWrap && end > first) {
      int w[3];
      code_wrap(code, w);
      sh = cell_shift(g, a, w, lane > kStencil / 2);
    }
    auto near = [&](int j) {
      float d2, R;
      return j < end && cand_f32(g, sh, a.w, __ldg(cr.wpos + j), d2, R) && j != s;
    };
    int n = 0;
    for (int j = first; __any_sync(all, j < end); ++j) {
      const bool keep = near(j);
      const unsigned m = __ballot_sync(all, keep);
      const int k = n + __popc(m & ((1u << lane) - 1u));
      if (keep && k < kLongKeep) mine[k] = (unsigned)j | ((unsigned)code << 26);
      n += __popc(m);
    }
    __syncwarp();
    int down = 0;
    if (n <= cl.keep) {
      const unsigned e = lane < n ? mine[lane] : 0u;
      const int j = (int)(e & 0x3ffffffu), idj = lane < n ? __ldg(id + j) : 0x7fffffff;
      int rank = 0;
      for (int q = 0; q < n; ++q) rank += __shfl_sync(all, idj, q) < idj;
      down = __popc(__ballot_sync(all, lane < n && idj < me));
      if (lane < n) {
        cl.list[(long long)s * kCandKeep + rank] = e;
        if (g.periodic) bad |= shift_overflow(cr, s, j, (int)(e >> 26));
      }
    } else if (cl.keep > 0 && n <= kLongKeep) {
      unsigned place = 0;
      if (lane == 0) place = atomicAdd(&ds->long_total, (unsigned)n);
      place = __shfl_sync(all, place, 0);
      const bool fits = (unsigned)n <= cl.spill_cap && place <= cl.spill_cap - (unsigned)n;
      for (int k = lane; k < n; k += 32) {
        const unsigned e = mine[k];
        const int j = (int)(e & 0x3ffffffu), idj = __ldg(id + j);
        idm[k] = idj;
        down += idj < me;
        if (g.periodic) bad |= shift_overflow(cr, s, j, (int)(e >> 26));
      }
      down = __reduce_add_sync(all, down);
      __syncwarp();
      if (fits)
        for (int k = lane; k < n; k += 32) {
          const int ik = idm[k];
          int rank = 0;
          for (int q = 0; q < n; ++q) rank += idm[q] < ik;
          cl.spill[place + rank] = mine[k];
        }
      if (lane == 0) cl.list[(long long)s * kCandKeep] = fits ? place : kNoList;
    } else {   // no list: the counts alone
      for (int j = first; j < end; ++j) {
        if (!near(j)) continue;
        down += __ldg(id + j) < me;
        if (g.periodic) bad |= shift_overflow(cr, s, j, code);
      }
      down = __reduce_add_sync(all, down);
      if (lane == 0 && cl.keep > 0) cl.list[(long long)s * kCandKeep] = kNoList;
    }
    if (lane == 0) {
      cnt_down[s] = down;
      cnt_up[s] = n - down;
      if (n > cl.many) atomicAdd(&ds->many_total, (unsigned long long)n);
    }
    __syncwarp();
  }
  if (bad) atomicOr(&ds->error, kErrShiftRange);
}

// What the row passes read: the walk's records and lists, the bodies in slot order, the
// new table (its ranges set) and the previous one.
struct RowArgs {
  CellRec cr;
  Bodies b;
  const Grid *grids;
  const int *start, *new_to_old;
  Table t, old;
  long long N, N_old;
  CandList cl;
  int multi, mixed;
};

// Row r = (s, j), w the wrap of j's cell seen from s: the pair and its shift, the contact
// history of the previous table, and in mixed precision the reference branch vector.
__device__ inline void write_row(const RowArgs &a, int r, int s, int j, const int w[3]) {
  const Table &nt = a.t, &ot = a.old;
  const Grid &g = grid_of(a.grids, a.b.sid, a.multi, s);
  int c[3] = {0, 0, 0};
  if (g.periodic) {   // shift of body 2
    const int4 is = a.cr.info[s], ij = a.cr.info[j];
    c[0] = is.y - ij.y + w[0]; c[1] = is.z - ij.z + w[1]; c[2] = is.w - ij.w + w[2];
  }
  const int cp = pack_shift(c[0], c[1], c[2]);
  nt.pair[r] = make_int2(s, j);
  nt.cpack[r] = cp;
  // both tables orient a pair by id (ids survive a collider run, or shift by the same
  // amount within a sub-scene), so the old row is in the old range of body 1
  int hit = -1;
  if (ot.P > 0) {
    const int o1 = a.new_to_old[s], o2 = a.new_to_old[j];
    if (o1 < a.N_old && o2 < a.N_old) {
      // only a row that was real has a history: its bit of the last step (whole words of
      // bits are zero for most bodies of a loose scene)
      const int first = ot.row_start[o1], e = ot.row_start[o1 + 1];
      for (int q0 = first; q0 < e && hit < 0; q0 += 32) {
        unsigned m = __funnelshift_r(ot.bits[q0 >> 5], ot.bits[(q0 >> 5) + 1], q0 & 31);
        if (e - q0 < 32) m &= (1u << (e - q0)) - 1u;
        for (; m; m &= m - 1) {
          const int q = q0 + __ffs(m) - 1;
          if (ot.pair[q].y == o2 && ot.cpack[q] == cp) { hit = q; break; }
        }
      }
    }
  }
  const double4_32a z = make_double4_32a(0, 0, 0, 0);
  double4_32a fs = z;
  if (a.mixed) {
    const float4 zf = make_float4(0, 0, 0, 0);
    float4 hn = zf;
    float kn = 0.0f;
    if (hit >= 0) {
      kn = ot.g32[hit].w;
      if (kn != 0.0f) {
        fs = ot.hfs[hit];
        hn = ot.hn32[hit];
        ot.found[hit] = 1;
      }
    }
    // reference branch vector of this run, x2 + Href c - x1 formed in FP64 and rounded
    // once to FP32; rows inside the cell have c = 0 and H c = 0 exactly, and a warp none of
    // whose rows crosses the cell skips the conversions and products (FP64-pipe work)
    const double4_32a p1 = a.b.pos[s], p2 = a.b.pos[j];
    double h[3] = {0, 0, 0};
    if (__any_sync(__activemask(), cp != 0) && g.periodic) {
      h[0] = g.L[0] * c[0]; h[1] = g.L[1] * c[1]; h[2] = g.L[2] * c[2];
      if (g.sheared)   // Href c of a sheared cell
        for (int q = 0; q < 3; ++q)
          h[q] = g.H[3 * q] * c[0] + g.H[3 * q + 1] * c[1] + g.H[3 * q + 2] * c[2];
    }
    const double gx = (p2.x + h[0]) - p1.x, gy = (p2.y + h[1]) - p1.y, gz = (p2.z + h[2]) - p1.z;
    nt.g32[r] = make_float4((float)gx, (float)gy, (float)gz, kn);
    // the squared gap of the reference configuration, in FP64 before any rounding: the
    // mixed kernel's penetration is this minus the FP32 terms of the offsets, so it keeps
    // FP32's relative precision of the gap rather than of the branch length
    const double R = p1.w + p2.w;
    nt.s0[r] = (float)(R * R - (gx * gx + gy * gy + gz * gz));
    nt.hfs[r] = fs;
    nt.hn32[r] = hn;
    nt.oFM32[2 * (long long)r] = zf;
    nt.oFM32[2 * (long long)r + 1] = zf;
    return;
  }
  double4_32a hn = z;
  double tp = 0;
  if (hit >= 0) {
    const double4_32a ofs = ot.hfs[hit];
    if (ofs.w != 0.0) {
      fs = ofs;
      hn = ot.hn[hit];
      tp = ot.tanphi[hit];
      ot.found[hit] = 1;
    }
  }
  nt.hfs[r] = fs;
  nt.hn[r] = hn;
  nt.tanphi[r] = tp;
  nt.oFM[2 * (long long)r] = z;
  nt.oFM[2 * (long long)r + 1] = z;
}

// The entry of a warp's 32 consecutive ranges that holds item r: lo[lane] is the first item
// of the lane's range (ascending; all 32 lanes call).
__device__ inline int range_of(int lo, int r) {
  int q = 0;   // the last range that begins at or before r
#pragma unroll
  for (int step = 16; step > 0; step >>= 1) {
    const int b = __shfl_sync(0xffffffffu, lo, q + step);
    if (b <= r) q += step;
  }
  return q;
}

// Where the list of body s with n partners is: kListed (its part of cl.list), its place in
// the spill buffer, or kNoList.
__device__ inline unsigned list_place(const CandList &cl, long long s, int n) {
  if (n <= cl.keep) return kListed;
  return cl.keep > 0 ? cl.list[s * kCandKeep] : kNoList;
}
__device__ inline unsigned list_entry(const CandList &cl, int s, unsigned place, int k) {
  return place == kListed ? cl.list[(long long)s * kCandKeep + k] : cl.spill[(size_t)place + k];
}

// Rows, 32 at a time: a warp takes 32 bodies, whose rows are consecutive, so every store
// to the new table is coalesced whatever the bodies' row counts.
__global__ void __launch_bounds__(kT) k_rows(RowArgs a) {
  const unsigned all = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const long long base = ((long long)blockIdx.x * kT + threadIdx.x) & ~31LL;
  if (base >= a.N) return;
  const long long me = base + lane < a.N ? base + lane : a.N;
  const int lo = a.t.row_start[me], hi = me < a.N ? a.t.row_start[me + 1] : lo;
  const int nd = me < a.N ? a.t.down_start[me + 1] - a.t.down_start[me] : 0;
  const unsigned place = list_place(a.cl, me, nd + hi - lo);
  const int end = __shfl_sync(all, hi, 31);
  for (int r0 = __shfl_sync(all, lo, 0); r0 < end; r0 += 32) {
    const int r = r0 + lane;
    const int q = range_of(lo, r);
    const int from = __shfl_sync(all, lo, q), skip = __shfl_sync(all, nd, q);
    const unsigned mine = __shfl_sync(all, place, q);
    if (r < end && mine != kNoList) {
      const int s = (int)base + q;
      const unsigned e = list_entry(a.cl, s, mine, skip + (r - from));
      int w[3];
      code_wrap((int)(e >> 26), w);
      write_row(a, r, s, (int)(e & 0x3ffffffu), w);
    }
  }
  if (place != kNoList) return;
  // no list: walk again, by insertion in order of id (found: the
  // partner's id until the row is complete; cpack: its wrap)
  const int s = (int)me, ids = a.b.id[s];
  const Grid &g = grid_of(a.grids, a.b.sid, a.multi, s);
  int k = lo;
  walk_cells<false>(g, a.cr.wpos, a.start, a.cr.info[s].x, s, [&](int j, int code, float, float) {
    const int idj = a.b.id[j];
    if (idj < ids) return;
    int q = k++;
    for (; q > lo && a.t.found[q - 1] > idj; --q) {
      a.t.found[q] = a.t.found[q - 1];
      a.t.pair[q] = a.t.pair[q - 1];
      a.t.cpack[q] = a.t.cpack[q - 1];
    }
    a.t.found[q] = idj;
    a.t.pair[q] = make_int2(s, j);
    a.t.cpack[q] = code;
  });
  for (int r = lo; r < hi; ++r) {
    int w[3];
    code_wrap(a.t.cpack[r], w);
    write_row(a, r, s, a.t.pair[r].y, w);
  }
}

// the row of the pair (p, s), p the body 1
__device__ inline int row_of(const Table &t, int p, int s) {
  const int first = t.row_start[p], end = t.row_start[p + 1];
  for (int r = first; r < end; ++r)
    if (t.pair[r].y == s) return r;
  return first;   // not reached: the walk keeps a pair from both sides or neither
}

// Down lists: the rows where a body is body 2, by id of body 1, 32 entries at a time.
__global__ void __launch_bounds__(kT) k_downs(RowArgs a) {
  const unsigned all = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const long long base = ((long long)blockIdx.x * kT + threadIdx.x) & ~31LL;
  if (base >= a.N) return;
  const long long me = base + lane < a.N ? base + lane : a.N;
  const int lo = a.t.down_start[me], hi = me < a.N ? a.t.down_start[me + 1] : lo;
  const int nu = me < a.N ? a.t.row_start[me + 1] - a.t.row_start[me] : 0;
  const unsigned place = list_place(a.cl, me, nu + hi - lo);
  const int end = __shfl_sync(all, hi, 31);
  for (int e0 = __shfl_sync(all, lo, 0); e0 < end; e0 += 32) {
    const int e = e0 + lane;
    const int q = range_of(lo, e);
    const int from = __shfl_sync(all, lo, q);
    const unsigned mine = __shfl_sync(all, place, q);
    if (e < end && mine != kNoList) {
      const int s = (int)base + q;
      const int p = (int)(list_entry(a.cl, s, mine, e - from) & 0x3ffffffu);
      a.t.down[e] = row_of(a.t, p, s);
    }
  }
  if (place != kNoList) return;
  const int s = (int)me, ids = a.b.id[s];
  const Grid &g = grid_of(a.grids, a.b.sid, a.multi, s);
  int k = lo;
  walk_cells<false>(g, a.cr.wpos, a.start, a.cr.info[s].x, s, [&](int j, int, float, float) {
    const int idj = a.b.id[j];
    if (idj > ids) return;
    int q = k++;
    for (; q > lo && a.b.id[a.t.pair[a.t.down[q - 1]].x] > idj; --q) a.t.down[q] = a.t.down[q - 1];
    a.t.down[q] = row_of(a.t, j, s);
  });
}

// Integration order of the FP64 path, within runs of kChunk consecutive slots: the bodies
// of a run by decreasing number of real rows, so that the lanes of a warp walk row lists that
// end together (the sum over a body's rows is a loop whose trip count is the warp's longest
// list), the run itself staying where it is, so that the bodies a block touches stay spatial
// neighbours (slot order is Morton order) and their records and rows are fetched into L2 once.
// The rows counted are those that carry a contact into this run; a run of slots without any
// (a first run) goes by candidate rows.  The order inside a group is left to the atomics:
// it changes no result, only which lane integrates which body.  By candidate rows (half of
// which are not in contact) the 1M dense integration took 313 us, by real rows 288.
constexpr int kChunk = 1024;
__global__ void __launch_bounds__(kChunk) k_degree_chunk(Table t, long long N, int count_real) {
  __shared__ int cnt[kDegreeBuckets], base[kDegreeBuckets];
  if (threadIdx.x < kDegreeBuckets) cnt[threadIdx.x] = 0;
  const long long c0 = (long long)blockIdx.x * kChunk, sl = c0 + threadIdx.x;
  int rows = 0, real = 0;
  if (sl < N) {
    const int a = t.row_start[sl], b = t.row_start[sl + 1];
    const int e0 = t.down_start[sl], e1 = t.down_start[sl + 1];
    rows = (b - a) + (e1 - e0);
    if (count_real) {
      for (int k = a; k < b; ++k) real += !is_zero_bits(t.hfs[k].w);
      for (int e = e0; e < e1; ++e) real += !is_zero_bits(t.hfs[t.down[e]].w);
    }
  }
  const int any = __syncthreads_or(real);
  const int d = min(any ? real : rows, kDegreeBuckets - 1);
  int bucket = -1, local = 0;
  if (sl < N) {
    bucket = kDegreeBuckets - 1 - d;
    local = atomicAdd(&cnt[bucket], 1);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int acc = 0;
    for (int i = 0; i < kDegreeBuckets; ++i) {
      base[i] = acc;
      acc += cnt[i];
    }
  }
  __syncthreads();
  if (bucket >= 0) t.ord[c0 + base[bucket] + local] = (int)sl;
}

// A real row of the previous table that no candidate carried over: an error only
// if the pair still overlaps at the positions of this collider run (a pair that
// separated within the step is dropped by the contact law anyway; a body may move
// farther than the sweep margin in the step that triggers the run).  ob: the body
// buffer in the old slot order, still holding the current positions.
__global__ void k_lost(Table ot, Bodies ob, const Grid *__restrict__ grids, int multi, int *err,
                       int mixed) {
  long long r = (long long)blockIdx.x * kT + threadIdx.x;
  if (r >= ot.P) return;
  const bool real = mixed ? (ot.g32[r].w != 0.0f) : (ot.hfs[r].w != 0.0);
  if (!real || ot.found[r]) return;
  const int2 pr = ot.pair[r];
  const double4_32a p1 = ob.pos[pr.x], p2 = ob.pos[pr.y];
  const Grid &g = grid_of(grids, ob.sid, multi, pr.x);
  double h[3] = {0, 0, 0};
  if (g.periodic) {
    int c0, c1, c2;
    unpack_shift(ot.cpack[r], c0, c1, c2);
    for (int k = 0; k < 3; ++k) h[k] = g.H[3 * k] * c0 + g.H[3 * k + 1] * c1 + g.H[3 * k + 2] * c2;
  }
  const double dx = (p2.x + h[0]) - p1.x, dy = (p2.y + h[1]) - p1.y, dz = (p2.z + h[2]) - p1.z;
  const double R = p1.w + p2.w;
  if (dx * dx + dy * dy + dz * dz < R * R) atomicOr(err, kErrHistoryLost);
}

inline unsigned blocks(long long n) { return (unsigned)((n + kT - 1) / kT); }
}  // namespace

int bbox_blocks(long long N) {
  long long b = (N + kT - 1) / kT;
  return (int)(b < 1 ? 1 : (b > 1024 ? 1024 : b));
}

void launch_bbox(const Bodies &b, long long N, double *partials, int nblk, cudaStream_t st) {
  k_bbox<<<nblk, kT, 0, st>>>(b.pos, N, partials);
}

void launch_bbox_sub(const Bodies &b, long long N, int cap, unsigned long long *keys,
                     int nsm, cudaStream_t st) {
  if (N <= 0) return;
  const long long need = (N + kT - 1) / kT;
  const long long lim = (long long)nsm * 4;
  k_bbox_sub<<<(unsigned)(need < lim ? need : lim), kT, 0, st>>>(b.pos, b.sid, N, cap, keys);
}

void launch_bin(const Bodies &b, long long N, const Grid *grids, int multi, uint32_t dead,
                uint32_t *key, int *rank, int *count, CellRec raw, cudaStream_t st) {
  if (N > 0)
    k_bin<<<blocks(N), kT, 0, st>>>(b.pos, b.sid, N, grids, multi, dead, key, rank, count, raw);
}

void launch_scatter(long long N, const uint32_t *key, const int *rank, const int *start, int *tmp,
                    cudaStream_t st) {
  if (N > 0) k_scatter<<<blocks(N), kT, 0, st>>>(N, key, rank, start, tmp);
}

void launch_reorder(const Bodies &src, const Bodies &dst, long long N, long long cap,
                    const int *tmp, const uint32_t *key, const int *start, CellRec raw, CellRec cr,
                    int *new_to_old, int *slot_of_id, int has_walls,
                    int mixed, const int *id_shift, const CellState *cs, int multi, cudaStream_t st) {
  if (N > 0)
    k_reorder<<<blocks(N), kT, 0, st>>>(src, dst, N, cap, tmp, key, start, raw, cr,
                                        new_to_old, slot_of_id, has_walls, mixed, id_shift, cs, multi);
}

void launch_slots(const int *id, long long N, int *slot_of_id, cudaStream_t st) {
  if (N > 0) k_slots<<<blocks(N), kT, 0, st>>>(id, N, slot_of_id);
}

void launch_partners(CellRec cr, const int *sid, const int *id, long long N, const Grid *grids,
                     int multi, const int *start, int *cnt_up, int *cnt_down, DevStatus *ds,
                     CandList cl, bool long_lists, bool again, int nsm, cudaStream_t st) {
  if (N <= 0) return;
  if (N < kWarpBodies || long_lists || cl.keep == 0) {
    k_partners_warp<false><<<blocks(32 * N), kT, 0, st>>>(cr, sid, id, N, grids, multi, start,
                                                          cnt_up, cnt_down, ds, cl);
    return;
  }
  if (!again)
    k_partners<<<(unsigned)((N + kPT - 1) / kPT), kPT, 0, st>>>(cr, sid, id, N, grids, multi, start,
                                                               cnt_up, cnt_down, ds, cl);
  k_partners_warp<true><<<7 * nsm, kT, 0, st>>>(cr, sid, id, N, grids, multi, start, cnt_up,
                                                cnt_down, ds, cl);
}

void launch_rows(CellRec cr, const Bodies &b, const Grid *grids, int multi, const int *start,
                 const Table &nt, const Table &ot, long long N, long long N_old,
                 const int *new_to_old, CandList cl, int mixed, cudaStream_t st) {
  if (N <= 0) return;
  const RowArgs a{cr, b, grids, start, new_to_old, nt, ot, N, N_old, cl, multi, mixed};
  k_rows<<<blocks(N), kT, 0, st>>>(a);
  k_downs<<<blocks(N), kT, 0, st>>>(a);
}

void launch_degree_order(const Table &t, long long N, int count_real, cudaStream_t st) {
  if (N <= 0) return;
  k_degree_chunk<<<(unsigned)((N + kChunk - 1) / kChunk), kChunk, 0, st>>>(t, N, count_real);
}

namespace {
// Cell flip (section 2.1.6, fig. 6): H' = H M keeps every image when each row's
// shift becomes c' = M^-1 c.  Pass 0 records the largest |c'| component of the rows
// of sub-scene `sub` (all rows without sub-scenes); pass 1 rewrites them.
__global__ void k_flip_shift(Table t, const int *__restrict__ sid, int multi, int sub, int3 m0,
                             int3 m1, int3 m2, int *maxabs, int apply) {
  for (long long k = (long long)blockIdx.x * kT + threadIdx.x; k < t.P;
       k += (long long)gridDim.x * kT) {
    if (multi && sid[t.pair[k].x] != sub) continue;
    int c0, c1, c2;
    unpack_shift(t.cpack[k], c0, c1, c2);
    const int n0 = m0.x * c0 + m0.y * c1 + m0.z * c2;
    const int n1 = m1.x * c0 + m1.y * c1 + m1.z * c2;
    const int n2 = m2.x * c0 + m2.y * c1 + m2.z * c2;
    if (apply) {
      t.cpack[k] = pack_shift(n0, n1, n2);
    } else {
      const int m = max(abs(n0), max(abs(n1), abs(n2)));
      if (m > kShiftMax) atomicMax(maxabs, m);
    }
  }
}
}  // namespace

void launch_flip_shift(const Table &t, const int *sid, int multi, int sub, const int Minv[9],
                       int *maxabs, int apply, cudaStream_t st) {
  if (t.P <= 0) return;
  const long long b = std::min<long long>(blocks(t.P), 4096);
  k_flip_shift<<<(unsigned)b, kT, 0, st>>>(t, sid, multi, sub, make_int3(Minv[0], Minv[1], Minv[2]),
                                          make_int3(Minv[3], Minv[4], Minv[5]),
                                          make_int3(Minv[6], Minv[7], Minv[8]), maxabs, apply);
}

void launch_lost(const Table &ot, const Bodies &ob, const Grid *grids, int multi, int *err,
                 int mixed, cudaStream_t st) {
  if (ot.P > 0) k_lost<<<blocks(ot.P), kT, 0, st>>>(ot, ob, grids, multi, err, mixed);
}

}  // namespace dem
