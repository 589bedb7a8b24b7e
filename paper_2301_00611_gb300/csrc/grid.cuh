// Uniform-grid helpers shared by the collider (collider.cu) and the bare pair
// query (pairs.cu): Morton codes of cells, the cell and integer image of a
// position, the conservative FP32 candidate test and the walk of the 27-cell stencil.
#pragma once
#include "dem_internal.cuh"

namespace dem {
namespace {

// Order-preserving map of doubles to unsigned integers (sign bit flipped for
// positives, all bits for negatives), so that integer minima and maxima (atomic or not) are
// those of the doubles, off the FP64 pipe; key_double is its inverse.
__device__ __forceinline__ unsigned long long ord_key(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}
__device__ __forceinline__ double key_double(unsigned long long k) {
  return __longlong_as_double((long long)((k >> 63) ? k & 0x7fffffffffffffffull : ~k));
}

__host__ __device__ inline uint32_t spread3(uint32_t x) {  // 8 bits -> every third bit
  x &= 0xffu;
  x = (x | (x << 8)) & 0x0000f00fu;
  x = (x | (x << 4)) & 0x000c30c3u;
  x = (x | (x << 2)) & 0x00249249u;
  return x;
}
__host__ __device__ inline uint32_t morton3(int i, int j, int k) {
  return spread3((uint32_t)i) | (spread3((uint32_t)j) << 1) | (spread3((uint32_t)k) << 2);
}

// global index of cell (i, j, k) of grid g: Morton code (one scene) or row-major
// (sub-scenes), offset by the grid's first cell
__host__ __device__ inline long long cell_index(const Grid &g, int i, int j, int k) {
  return g.base + (g.morton ? (long long)morton3(i, j, k)
                            : ((long long)k * g.n[1] + j) * g.n[0] + i);
}

// cell coordinates (and, periodic, the integer image) of a position
__device__ inline void cell_of(const Grid &g, double x, double y, double z, int c[3], int img[3]) {
  const double p[3] = {x, y, z};
  double u[3] = {x * g.scale[0], y * g.scale[1], z * g.scale[2]};   // fractional (periodic)
  if (g.periodic && g.sheared)   // sheared cell: s = Hinv x
    for (int k = 0; k < 3; ++k)
      u[k] = g.Hinv[3 * k] * x + g.Hinv[3 * k + 1] * y + g.Hinv[3 * k + 2] * z;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    int ck;
    if (g.periodic) {
      double s = u[k];
      double fi = floor(s);
      double f = s - fi;
      ck = (int)(f * g.n[k]);
      img[k] = (int)fi;
    } else {
      ck = (int)floor((p[k] - g.lo[k]) * g.scale[k]);
      img[k] = 0;
    }
    c[k] = ck < 0 ? 0 : (ck >= g.n[k] ? g.n[k] - 1 : ck);
  }
}

// Image shift of the cells of wrap w, in FP32 (H w of a sheared cell): the shift of -w is
// its exact negative.
__device__ inline void wrap_shift_f32(const Grid &g, const int w[3], float sh[3]) {
  const float f0 = (float)w[0], f1 = (float)w[1], f2 = (float)w[2];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    if (g.sheared)
      sh[k] = __fmaf_rn(g.Hf[3 * k + 2], f2, __fmaf_rn(g.Hf[3 * k + 1], f1, __fmul_rn(g.Hf[3 * k], f0)));
    else
      sh[k] = __fmul_rn(k == 0 ? f0 : (k == 1 ? f1 : f2), g.Lf[k]);
  }
}

// Conservative FP32 candidate test of (s, j): keeps every pair whose FP64 distance is
// below r1 + r2 + reach (the slack covers the FP32 rounding of coordinates bounded by the
// cell size), so the candidate set is a superset of the exact one.  A pair met from both
// sides must be decided alike, so the image shift goes to the same of the two spheres from
// either side: to the one in the forward half of the other's stencil ((dz, dy, dx)
// lexicographically positive), as when every pair is met from that side only.  Every
// operation is written out: no contraction that differs by call site.
struct CellShift {
  float3 me, partner;   // the body's own position; what is added to the partners'
};
__device__ inline CellShift cell_shift(const Grid &g, const float4 &a, const int w[3], bool fwd) {
  float sh[3];
  wrap_shift_f32(g, w, sh);
  if (fwd) return {make_float3(a.x, a.y, a.z), make_float3(sh[0], sh[1], sh[2])};
  return {make_float3(__fsub_rn(a.x, sh[0]), __fsub_rn(a.y, sh[1]), __fsub_rn(a.z, sh[2])),
          make_float3(0.0f, 0.0f, 0.0f)};
}
__device__ inline bool cand_f32(const Grid &g, const CellShift &at, float ra, const float4 &b,
                                float &d2, float &R) {
  const float dx = __fsub_rn(__fadd_rn(b.x, at.partner.x), at.me.x);
  const float dy = __fsub_rn(__fadd_rn(b.y, at.partner.y), at.me.y);
  const float dz = __fsub_rn(__fadd_rn(b.z, at.partner.z), at.me.z);
  R = __fadd_rn(__fadd_rn(__fadd_rn(ra, b.w), g.reachf), g.slack);
  d2 = __fmaf_rn(dz, dz, __fmaf_rn(dx, dx, __fmul_rn(dy, dy)));
  return d2 < __fmul_rn(R, R);
}

constexpr int kStencil = 27;
constexpr int kNoWrap = 13;   // wrap code of no wrap at all: (w0 + 1) + 3 (w1 + 1) + 9 (w2 + 1)

__device__ inline void code_wrap(int code, int w[3]) {
  w[0] = code % 3 - 1;
  w[1] = (code / 3) % 3 - 1;
  w[2] = code / 9 - 1;
}

// One axis of a stencil cell: coordinate c (outside the grid by at most one) wrapped or
// refused, and its part of the cell index.
__device__ inline bool axis_cell(const Grid &g, int k, int &c, int &w) {
  w = 0;
  if (c >= 0 && c < g.n[k]) return true;
  if (!g.periodic) return false;
  w = c < 0 ? -1 : 1;
  c -= w * g.n[k];
  return true;
}
__device__ inline int axis_part(const Grid &g, int k, int c) {
  if (g.morton) return (int)(spread3((uint32_t)c) << k);
  return k == 0 ? c : (k == 1 ? c * g.n[0] : c * g.n[0] * g.n[1]);
}

// Neighbour cell t (0..26, dx fastest) of cell ci: its slots [first, end) and wrap code;
// none beyond the faces of an aperiodic grid.
__device__ inline void stencil_cell(const Grid &g, const int *__restrict__ start, const int ci[3],
                                    int t, int &first, int &end, int &code) {
  int c[3] = {ci[0] + t % 3 - 1, ci[1] + (t / 3) % 3 - 1, ci[2] + t / 9 - 1}, w[3];
  bool ok = true;
  for (int k = 0; k < 3; ++k) ok = axis_cell(g, k, c[k], w[k]) && ok;
  const long long m =
      ok ? g.base + axis_part(g, 0, c[0]) + axis_part(g, 1, c[1]) + axis_part(g, 2, c[2]) : 0;
  first = ok ? start[m] : 0;
  end = ok ? start[m + 1] : 0;
  code = (w[0] + 1) + 3 * (w[1] + 1) + 9 * (w[2] + 1);
}

// Walk of one body's neighbour cells by one thread, in stencil order (dz, dy, dx, slot):
// f(j, code, d2, R) for every candidate j (FP32 squared distance, reach with slack).
//   kHalf: the forward half of the stencil (own cell from slot s + 1 on, then the 13 cells
//   with (dz, dy, dx) lexicographically positive), so every pair is met from one side;
//   else all 27 cells, the body itself left out: every pair is met from both sides.
// A cell costs its index and two loads (the three of a row together), a partner about 17
// instructions and a load; kAhead partners are loaded before the first is tested.  Loading
// one at a time left the walk waiting: all 27 cells of 300k bodies at three rows a body
// 136 -> 111 us, of 1M bodies at five 852 -> 605 us with four ahead (118 and 697 with
// two); the half shell of 1M bodies 236 -> 219 us with two (254 with four).  Where cells run
// along x in memory (row-major grids), the three cells of a row inside the grid are one run.
template <bool kHalf, class F>
__device__ inline void walk_cells(const Grid &g, const float4 *__restrict__ wpos,
                                  const int *__restrict__ start, int packed, int s, F &&f) {
  constexpr int kAhead = kHalf ? 2 : 4;
  const float4 me = wpos[s];
  const int ci[3] = {packed & 1023, (packed >> 10) & 1023, (packed >> 20) & 1023};
  bool okx[3];
  int px[3], wx[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    int c = ci[0] + i - 1;
    okx[i] = axis_cell(g, 0, c, wx[i]);
    px[i] = okx[i] ? axis_part(g, 0, c) : 0;
  }
  const bool run = !kHalf && !g.morton && wx[0] == 0 && wx[2] == 0;
#pragma unroll 1
  for (int dz = kHalf ? 0 : -1; dz <= 1; ++dz) {
    int cz = ci[2] + dz, wz;
    if (!axis_cell(g, 2, cz, wz)) continue;
    const long long pz = g.base + axis_part(g, 2, cz);
#pragma unroll 1
    for (int dy = kHalf && dz == 0 ? 0 : -1; dy <= 1; ++dy) {
      int cy = ci[1] + dy, wy;
      if (!axis_cell(g, 1, cy, wy)) continue;
      const long long row = pz + axis_part(g, 1, cy);
      const bool own_row = dz == 0 && dy == 0;
      int a[3], b[3];
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        a[i] = b[i] = 0;
        if (okx[i] && !(kHalf && own_row && i == 0)) {
          a[i] = start[row + px[i]];
          b[i] = start[row + px[i] + 1];
        }
      }
      if (kHalf && own_row) a[1] = s + 1;
      if (run) {   // one run of slots
        if (okx[0]) a[1] = a[0];
        if (okx[2]) b[1] = b[2];
        a[0] = b[0] = a[2] = b[2] = 0;
      }
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        const int code = (wx[i] + 1) + 3 * (wy + 1) + 9 * (wz + 1);
        CellShift at{make_float3(me.x, me.y, me.z), make_float3(0.0f, 0.0f, 0.0f)};
        if (code != kNoWrap) {
          const int w[3] = {wx[i], wy, wz};
          at = cell_shift(g, me, w, dz > 0 || (dz == 0 && (dy > 0 || (dy == 0 && i == 2))));
        }
        for (int j = a[i]; j < b[i]; j += kAhead) {
          float4 p[kAhead];
#pragma unroll
          for (int q = 0; q < kAhead; ++q) p[q] = __ldg(wpos + min(j + q, b[i] - 1));
#pragma unroll
          for (int q = 0; q < kAhead; ++q) {
            float d2, R;
            const bool near = cand_f32(g, at, me.w, p[q], d2, R);
            if (near && j + q < b[i] && (kHalf || j + q != s)) f(j + q, code, d2, R);
          }
        }
      }
    }
  }
}

}  // namespace
}  // namespace dem
