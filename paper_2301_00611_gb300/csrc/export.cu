// State and contacts in the order callers see them: bodies by id, contacts by (id1, id2),
// packed on the device so that the host receives each array with one copy and touches no
// element of it.
//
// Bodies: one thread an id, reading the 32-byte records of its slot and writing packed
// doubles (consecutive ids are neighbours in the output, so the stores are coalesced and the
// scattered reads are whole sectors): bound by HBM and, over all, by the copy to the host.
//
// Contacts: rows are oriented by id and sorted by id2 within body 1's range already, so the
// canonical order needs no sort: the real rows of body 1 are counted id by id, a prefix sum
// gives each body's first place, and a second pass writes them there.  Wall contacts
// (id1 = -(wall + 1)) come first: six more runs of counts, wall 5 to wall 0.
// The state of 1M spheres on the host: 33 -> 0.7 ms; 315k contacts, counted and exported:
// about 100 -> 0.7 ms (the host copied whole tables, picked and sorted the rows, twice).
#include "dem_internal.cuh"

namespace dem {

namespace {
constexpr int kT = 256;
inline unsigned blocks(long long n) { return (unsigned)((n + kT - 1) / kT); }

__global__ void __launch_bounds__(kT) k_state_pack(const int *__restrict__ slot_of_id, long long n,
                                                   StatePack a) {
  const long long i = (long long)blockIdx.x * kT + threadIdx.x;
  if (i >= n) return;
  const int s = slot_of_id[i];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    if (!a.dst3[k]) continue;
    const double4_32a v = a.src3[k][s];
    double *o = a.dst3[k] + 3 * i;
    o[0] = v.x; o[1] = v.y; o[2] = v.z;
  }
  if (a.ori) {
    if (a.ori32) {
      const float4 q = a.ori32[s];
      a.ori[i] = make_double4_32a(q.x, q.y, q.z, q.w);
    } else {
      a.ori[i] = a.ori64[s];
    }
  }
}

__device__ inline bool real_row(const Table &t, long long k, int mixed) {
  return mixed ? t.g32[k].w != 0.0f : t.hfs[k].w != 0.0;
}

// Counts of the contacts whose first entry is (run, id): runs 0..5 are walls 5..0 (with
// walls), the last run the sphere pairs.
__global__ void __launch_bounds__(kT) k_contact_count(const int *__restrict__ slot_of_id, Bodies b,
                                                      Table t, long long N, int mixed, int walls,
                                                      int *cnt) {
  const long long i = (long long)blockIdx.x * kT + threadIdx.x;
  if (i >= N) return;
  const int s = slot_of_id[i];
  int n = 0;
  for (int k = t.row_start[s]; k < t.row_start[s + 1]; ++k) n += real_row(t, k, mixed);
  if (walls) {
    const uint8_t f = b.flags[s];
    for (int w = 5; w >= 0; --w) cnt[(5 - w) * N + i] = (f >> (1 + w)) & 1;
    cnt += 6 * N;
  }
  cnt[i] = n;
}

__device__ inline void put3(double *a, long long r, double x, double y, double z) {
  if (!a) return;
  a[3 * r] = x; a[3 * r + 1] = y; a[3 * r + 2] = z;
}

__device__ inline void put_sphere(const ContactPack &o, long long r, const Bodies &b, const Table &t,
                                  long long k, int s, int id1, int mixed) {
  const int2 pr = t.pair[k];
  int c0, c1, c2;
  unpack_shift(t.cpack[k], c0, c1, c2);
  double F[3], fs[3], n[3], d1, kn, ks, tp;
  const double4_32a h = t.hfs[k];
  fs[0] = h.x; fs[1] = h.y; fs[2] = h.z;
  if (mixed) {
    const float4 f = t.oFM32[2 * k], m = t.hn32[k];
    F[0] = f.x; F[1] = f.y; F[2] = f.z; d1 = f.w;
    n[0] = m.x; n[1] = m.y; n[2] = m.z; ks = m.w;
    kn = t.g32[k].w;
    tp = h.w;
  } else {
    const double4_32a f = t.oFM[2 * k], m = t.hn[k];
    F[0] = f.x; F[1] = f.y; F[2] = f.z; d1 = f.w;
    n[0] = m.x; n[1] = m.y; n[2] = m.z; ks = m.w;
    kn = h.w;
    tp = t.tanphi[k];
  }
  const double4_32a p = b.pos[s];
  if (o.id1) o.id1[r] = id1;
  if (o.id2) o.id2[r] = b.id[pr.y];
  if (o.c) { o.c[3 * r] = c0; o.c[3 * r + 1] = c1; o.c[3 * r + 2] = c2; }
  put3(o.fn, r, F[0] - fs[0], F[1] - fs[1], F[2] - fs[2]);
  put3(o.fs, r, fs[0], fs[1], fs[2]);
  put3(o.n, r, n[0], n[1], n[2]);
  // contact point x1 + (r1 - pen/2) n from the current position of body 1
  put3(o.cp, r, __dadd_rn(p.x, __dmul_rn(d1, n[0])), __dadd_rn(p.y, __dmul_rn(d1, n[1])),
       __dadd_rn(p.z, __dmul_rn(d1, n[2])));
  put3(o.phys, r, kn, ks, tp);
  if (o.pen) o.pen[r] = 2.0 * (p.w - d1);
}

__device__ inline void put_wall(const ContactPack &o, long long r, const Bodies &b, long long cap,
                                int w, int s, int id, const CellState &c, const Mat *mats) {
  const double4_32a h = b.whist[w * cap + s], p = b.pos[s];
  const int ax = w >> 1;
  const double sn = h.w >= 0 ? 1.0 : -1.0, Fn = fabs(h.w), rr = p.w;
  // stiffnesses of the contact in the order the host writes them (no contraction)
  const Mat mw = mats[c.wall_mat], ms = mats[b.mat[s]];
  double kn, ks;
  const double tp = fmin(mw.tanphi, ms.tanphi);
  if (c.law) {
    mindlin_phys(ms, rr, mw, -1.0, kn, ks);
  } else {
    const double d = 2 * rr, k1 = __dmul_rn(mw.young, d), k2 = __dmul_rn(ms.young, d);
    kn = __dmul_rn(k1, k2) / __dadd_rn(k1, k2);
    const double s1 = __dmul_rn(__dmul_rn(mw.young, mw.poisson), d);
    const double s2 = __dmul_rn(__dmul_rn(ms.young, ms.poisson), d);
    ks = __dmul_rn(s1, s2) / __dadd_rn(s1, s2);
  }
  const double pen = wall_pen(Fn, kn, c.law), arm = __dsub_rn(rr, __dmul_rn(0.5, pen));
  const double n[3] = {ax == 0 ? sn : 0.0, ax == 1 ? sn : 0.0, ax == 2 ? sn : 0.0};
  if (o.id1) o.id1[r] = -(w + 1);
  if (o.id2) o.id2[r] = id;
  if (o.c) { o.c[3 * r] = 0; o.c[3 * r + 1] = 0; o.c[3 * r + 2] = 0; }
  put3(o.fn, r, ax == 0 ? sn * Fn : 0.0, ax == 1 ? sn * Fn : 0.0, ax == 2 ? sn * Fn : 0.0);
  put3(o.fs, r, h.x, h.y, h.z);
  put3(o.n, r, n[0], n[1], n[2]);
  put3(o.cp, r, __dsub_rn(p.x, __dmul_rn(arm, n[0])), __dsub_rn(p.y, __dmul_rn(arm, n[1])),
       __dsub_rn(p.z, __dmul_rn(arm, n[2])));
  put3(o.phys, r, kn, ks, tp);
  if (o.pen) o.pen[r] = pen;
}

// Contacts of places [first, first + count), into records [0, count) of o.
__global__ void __launch_bounds__(kT) k_contact_emit(const int *__restrict__ slot_of_id, Bodies b,
                                                     Table t, long long N, long long cap, int mixed,
                                                     int walls, int multi,
                                                     const CellState *__restrict__ cs,
                                                     const Mat *__restrict__ mats,
                                                     const int *__restrict__ off, long long first,
                                                     long long count, ContactPack o) {
  const long long i = (long long)blockIdx.x * kT + threadIdx.x;
  if (i >= N) return;
  const int s = slot_of_id[i];
  if (walls) {
    const uint8_t f = b.flags[s];
    for (int w = 5; w >= 0; --w) {
      if (!(f & (2 << w))) continue;
      const long long r = off[(5 - w) * N + i] - first;
      if (r >= 0 && r < count) put_wall(o, r, b, cap, w, s, (int)i, cs[multi ? b.sid[s] : 0], mats);
    }
    off += 6 * N;
  }
  long long r = off[i] - first;
  if (r >= count || off[i + 1] - first <= 0) return;
  for (int k = t.row_start[s]; k < t.row_start[s + 1]; ++k) {
    if (!real_row(t, k, mixed)) continue;
    if (r >= 0 && r < count) put_sphere(o, r, b, t, k, s, (int)i, mixed);
    ++r;
  }
}
}  // namespace

void launch_state_pack(const int *slot_of_id, long long n, const StatePack &a, cudaStream_t st) {
  if (n > 0) k_state_pack<<<blocks(n), kT, 0, st>>>(slot_of_id, n, a);
}

void launch_contact_count(const int *slot_of_id, const Bodies &b, const Table &t, long long N,
                          int mixed, int walls, int *cnt, cudaStream_t st) {
  if (N > 0) k_contact_count<<<blocks(N), kT, 0, st>>>(slot_of_id, b, t, N, mixed, walls, cnt);
}

void launch_contact_emit(const int *slot_of_id, const Bodies &b, const Table &t, long long N,
                         long long cap, int mixed, int walls, int multi, const CellState *cs,
                         const Mat *mats, const int *off, long long first, long long count,
                         const ContactPack &o, cudaStream_t st) {
  if (N > 0 && count > 0)
    k_contact_emit<<<blocks(N), kT, 0, st>>>(slot_of_id, b, t, N, cap, mixed, walls, multi, cs, mats,
                                             off, first, count, o);
}

}  // namespace dem
