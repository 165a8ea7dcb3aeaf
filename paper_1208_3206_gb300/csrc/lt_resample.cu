// lt_resample.cu -- resampling of the tetrahedral tessellation onto a
// periodic n x n x n grid (Sec. 4.3, Eq. 10-12) and the stream-count field
// (Sec. 3.2).
//
// Cell (a, b, c) of edge g = box / n receives, from every tetrahedron t,
// q_t times the length of the part of the cell's central line along z
// (x = (a + 1/2) g, y = (b + 1/2) g) that lies inside t and inside the
// cell's slab [c g, (c + 1) g): the slab-wise form of the paper's
// resampling, in which each slab is a projection of the tetrahedra clipped
// to that slab. q_t = rho_t = m / |V_t| (Eq. 3) gives rho dl, the paper's
// estimate of the cell's mass over its face area; q_t = 1 gives the summed
// stream length, which over g is the mean number of streams on the line.
//
// A warp takes 32 tetrahedra of the lattice:
//   * one lane per tetrahedron forms its vertices, volume and face normals in
//     float-float, in units of the cell and relative to a vertex. On the line of
//     column (A0 + da, B0 + db) a face lies at the height C + A da + B db, which
//     the lane leaves in shared memory as three 64-bit integers (42 fraction
//     bits), with the columns the bounding box reaches;
//   * the columns of all of them are flattened, and the warp takes 32 at a time:
//     the largest of the lower faces' heights and the smallest of the upper ones'
//     bound the interval of z inside, in exact integer arithmetic;
//   * the cells of the intervals found are flattened again, 32 at a time: a whole
//     cell adds a number computed once, the two ends of an interval one 64 x
//     64-bit product each (one tetrahedron at a time, every lane with its own
//     column and loop over cells, kept half of the lanes busy: 15.4 ms);
//   * a cell's share is added as a 64-bit fixed-point integer with a global
//     atomic. Integer sums do not depend on the order of the adds, so the grid is
//     bitwise reproducible. Consecutive warps take consecutive cubes, whose cells
//     share the L2.
// A and B are rounded to 2^-43 of a cell, so a height is good to that times the
// columns that the tetrahedron spans: 2^-40 for eight of them, 2^-32 for two
// thousand (a cell holds FP32 numbers). A tetrahedron whose volume cancels beyond
// float-float, with a face so near to vertical (2^12 cells per column) or numbers
// so large that the integers would not hold them, is clipped in FP64. A last
// kernel converts the integer grid to float.
//
// What bounds it: with the planes, the intervals and their pieces in FP64 the
// FP64 pipe took 148 ms for 128^3 particles onto 512^3 cells (1.6e8 intervals,
// 3.0e8 pieces), 19 of them the setup, done once for each tile of columns that a
// tetrahedron touched. Now 8.6 ms for the call, of which the
// grid's clearing and conversion are 0.45; the kernel issues in about 60% of its
// slots, and waits for global memory most in the others.
#include "lt_ff.cuh"
#include "lt_internal.h"

namespace lt {

// Two warps: they are done at different times, and the shared memory of a small
// block goes on to the next one sooner (blocks of four warps 9.45 ms, of one 8.65).
constexpr int kResampleThreads = 64;
constexpr int kZBits = 42;  // fraction bits of a height in cells
constexpr long long kZOne = 1LL << kZBits;
constexpr float kTieAxis = 0.3719f;  // see the vertical faces of resample_fixed

struct ResampleArgs {
  Lattice L;
  int snapshot, n, weight;
  bool use_ff;
  ff h, inv_g, cells;  // box / N; cells per length; cells per lattice spacing
  ff q_num;            // accumulator units of a whole cell: over 6 |V| (density) or as it is (streams)
  double gs;           // cell edge box / n
  double m_tet;        // mass of one tetrahedron
  double inv_unit;     // accumulator units per (q x length)
  unsigned long long* acc;  // [n][n][n] fixed-point cells
  DevCounters* ctr;
};

// One tetrahedron of the current batch, as the warp's lanes read it.
struct ResampleTet {
  union {
    struct {
      long long C[4], A[4], B[4];  // heights C + A da + B db (vertical faces: a signed distance, inside >= 0)
      unsigned long long whole;    // units of a whole cell
      unsigned long long Q;        // the same as Q 2^(e - 62), 62 <= log2 Q < 63
      int shift;                   // 61 - e
      int upper, vertical;         // bits: faces that bound from above, vertical faces
    } f;
    struct {
      double nx[4], ny[4], d[4], inz[4];  // face planes: inside when nx x + ny y + nz z <= d; inz = 1 / nz (0: vertical face)
      double q, qx, qy, qz;               // rho (density weighting) or 1; the cube's Lagrangian corner
    } d;
  };
  int A0, B0, wa, wb;  // columns (A0, B0 in [0, n) for the integer form), their numbers
  float inv_wa;
  int K0;              // cell that heights count from, in [0, n)
  int form;            // 1: integers, 2: FP64
};

__device__ __forceinline__ void cell_add(const ResampleArgs& a, unsigned long long* cell, unsigned long long n) {
  if (n == 0ull) return;
  const unsigned long long old = atomicAdd(cell, n);
  if (old > ~0ull - n) {
    atomicOr(&a.ctr->errors, kErrRange);
    atomicAdd(&a.ctr->range_overflow, 1ull);
  }
}

// A float-float number below 2^20 in 2^-42, rounded: 22 + 10, 16 and 16 bits in turn.
__device__ __forceinline__ long long to_fixed(ff a) {
  const float s = a.h * 1024.0f;  // exact
  const int i1 = __float2int_rd(s);
  const ff r = ff_two_sum(__fsub_rn(s, (float)i1), a.l * 1024.0f);
  const float s2 = r.h * 65536.0f;
  const int i2 = __float2int_rd(s2);
  const int i3 = __float2int_rn(__fmaf_rn(r.l, 65536.0f, __fsub_rn(s2, (float)i2)) * 65536.0f);
  return ((long long)i1 << 32) + ((long long)i2 << 16) + (long long)i3;
}

// FP64 setup (the planes relative to the cube's Lagrangian corner).
__device__ __noinline__ bool resample_f64(const ResampleArgs& a, int i, int j, int k, int s, ResampleTet& r) {
  bool ok = true;
  TetF64 t;
  tet_f64(a.L, (long long)a.snapshot * a.L.n_particles, i, j, k, s, ok, t);
  if (!ok) atomicOr(&a.ctr->errors, kErrNonFinite);
  if (!ok || t.V == 0.0) return false;
  const double h = (double)a.L.box / a.L.N, inv_gs = 1.0 / a.gs;
  bool above = false, below = false;
  for (int f = 0; f < 4; ++f) {
    r.d.nx[f] = t.n[f][0];
    r.d.ny[f] = t.n[f][1];
    r.d.d[f] = t.d[f];
    const double big = fmax(fabs(t.n[f][0]), fabs(t.n[f][1]));
    r.d.inz[f] = fabs(t.n[f][2]) > 1e-12 * big ? 1.0 / t.n[f][2] : 0.0;
    above = above || r.d.inz[f] > 0.0;
    below = below || r.d.inz[f] < 0.0;
  }
  // flat in a vertical plane (particles that coincide, but for the rounding of
  // their place): no face bounds a column in z, and it has no volume but rounding
  if (!above || !below) return false;
  r.d.q = a.weight == 0 ? a.m_tet / fabs(t.V) : 1.0;
  r.d.qx = i * h;
  r.d.qy = j * h;
  r.d.qz = k * h;
  double xmn = t.v[0][0], xmx = xmn, ymn = t.v[0][1], ymx = ymn;
  for (int c = 1; c < 4; ++c) {
    xmn = fmin(xmn, t.v[c][0]); xmx = fmax(xmx, t.v[c][0]);
    ymn = fmin(ymn, t.v[c][1]); ymx = fmax(ymx, t.v[c][1]);
  }
  // at most 8 periods of columns per axis
  const double A0 = ceil((r.d.qx + xmn) * inv_gs - 0.5), A1 = fmin(floor((r.d.qx + xmx) * inv_gs - 0.5), A0 + 8.0 * a.n - 1.0);
  const double B0 = ceil((r.d.qy + ymn) * inv_gs - 0.5), B1 = fmin(floor((r.d.qy + ymx) * inv_gs - 0.5), B0 + 8.0 * a.n - 1.0);
  if (!(A0 <= A1 && B0 <= B1) || !(fabs(A0) < 1e9 && fabs(B0) < 1e9)) return false;
  r.A0 = (int)A0;
  r.B0 = (int)B0;
  r.wa = (int)(A1 - A0) + 1;
  r.wb = (int)(B1 - B0) + 1;
  // columns on a vertical face: on one side of it, as in the integer form
  const double tie = (8.0 * ((double)r.wa + (double)r.wb + 8.0)) / (double)kZOne * a.gs;
  for (int f = 0; f < 4; ++f)
    if (r.d.inz[f] == 0.0) {
      const double nx = r.d.nx[f], ny = r.d.ny[f];
      r.d.d[f] += (nx + (double)kTieAxis * ny < 0.0 ? tie : -tie) * fmax(fabs(nx), fabs(ny));
    }
  r.form = 2;
  return true;
}

// Integer setup; 0: nothing to add, 1: done, 2: FP64 has to take it.
__device__ __forceinline__ int resample_fixed(const ResampleArgs& a, int i, int j, int k, int s, ResampleTet& r) {
  bool ok = true;
  ff v[4][3], det;
  tet_ff(a.L, a.h, (long long)a.snapshot * a.L.n_particles, i, j, k, s, ok, v);
  if (!ok) {
    atomicOr(&a.ctr->errors, kErrNonFinite);
    return 0;
  }
  if (!volume6_ff(v, det)) return 2;
  // vertex 0 in cells, as a whole number and a fraction
  const int idx[3] = {i, j, k};
  int base[3];
  ff frac[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const float f = (float)idx[q];
    const ff p = ff_two_prod(f, a.cells.h);
    const ff x = ff_fast_sum(p.h, __fmaf_rn(f, a.cells.l, p.l)) + v[0][q] * a.inv_g;
    const float b = floorf(x.h);
    if (!(fabsf(b) < 1.0e9f)) return 2;
    base[q] = (int)b;
    frac[q] = ff_two_sum(__fsub_rn(x.h, b), x.l);
  }
  ff e[3][3];
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int q = 0; q < 3; ++q) e[c][q] = v[c + 1][q] - v[0][q];
  // columns whose line can meet the tetrahedron (widened for FP32's rounding)
  const float g = a.inv_g.h;
  int lo[2], w[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const float mn = fminf(fminf(0.f, e[0][q].h), fminf(e[1][q].h, e[2][q].h)) * g;
    const float mx = fmaxf(fmaxf(0.f, e[0][q].h), fmaxf(e[1][q].h, e[2][q].h)) * g;
    if (!(mx - mn < 4096.0f)) return 2;
    lo[q] = __float2int_ru(frac[q].h + mn - 0.5f - 1e-3f);
    w[q] = __float2int_rd(frac[q].h + mx - 0.5f + 1e-3f) - lo[q] + 1;
    if (w[q] < 1) return 0;
    if (w[q] > 8 * a.n) return 2;
  }
  // the first column's place relative to vertex 0
  const ff dx = -frac[0] + ((float)lo[0] + 0.5f), dy = -frac[1] + ((float)lo[1] + 0.5f);
  ff m[4][3];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const int u = (q + 1) % 3, t = (q + 2) % 3;
    m[1][q] = e[1][u] * e[2][t] - e[1][t] * e[2][u];
    m[2][q] = e[2][u] * e[0][t] - e[2][t] * e[0][u];
    m[3][q] = e[0][u] * e[1][t] - e[0][t] * e[1][u];
    m[0][q] = -((m[1][q] + m[2][q]) + m[3][q]);
  }
  // (face 0 is vertical where its sum is the rounding of its terms)
  if (fabsf(m[0][2].h) <= 0x1p-38f * (fabsf(m[1][2].h) + fabsf(m[2][2].h) + fabsf(m[3][2].h))) m[0][2] = {0.f, 0.f};
  // face f holds vertex 0 (f = 1..3) or vertex 1 (f = 0); inside m . (p - v) / det >= 0
  int upper = 0, vertical = 0;
#pragma unroll
  for (int f = 0; f < 4; ++f) {
    ff px = dx, py = dy, z = frac[2];
    if (f == 0) {
      px = px - e[0][0] * a.inv_g;
      py = py - e[0][1] * a.inv_g;
      z = z + e[0][2] * a.inv_g;
    }
    ff A, B;
    if (m[f][2].h == 0.0f) {
      const float big = fmaxf(fabsf(m[f][0].h), fabsf(m[f][1].h));
      if (!(big > 0.0f)) return 2;
      const ff sc = ff{det.h > 0.f ? 1.0f : -1.0f, 0.f} / ff{big, 0.f};
      A = m[f][0] * sc;
      B = m[f][1] * sc;
      z = {0.f, 0.f};
      vertical |= 1 << f;
    } else {
      const ff iz = ff{-1.f, 0.f} / m[f][2];
      A = m[f][0] * iz;
      B = m[f][1] * iz;
      if ((m[f][2].h > 0.f) != (det.h > 0.f)) upper |= 1 << f;
    }
    const ff C = (z + A * px) + B * py;
    const float slope = fabsf(A.h) + fabsf(B.h);
    if (!(slope < 4096.0f) || !(fabsf(C.h) + fabsf(A.h) * (float)w[0] + fabsf(B.h) * (float)w[1] < 1.0e6f)) return 2;
    r.f.A[f] = to_fixed(A);
    r.f.B[f] = to_fixed(B);
    r.f.C[f] = to_fixed(C);
    if ((vertical >> f) & 1) {
      // a column on the face, within rounding, belongs to the tetrahedron on the
      // one side and not to that on the other (a lattice at rest has whole planes
      // of columns on faces: counted on both sides they held up to four times
      // their mass). The side: by the direction's sign along an axis that no
      // lattice face is parallel to, so that a component's rounding does not matter
      const long long tie = 8LL * (w[0] + w[1] + 8);
      r.f.C[f] += A.h + kTieAxis * B.h > 0.f ? tie : -tie - 1;
    }
  }
  r.f.upper = upper;
  r.f.vertical = vertical;
  // units of a whole cell as Q 2^(ex - 62)
  const ff q = a.weight == 0 ? a.q_num / (det.h < 0.f ? -det : det) : a.q_num;
  const int ex = ((__float_as_int(q.h) >> 23) & 255) - 127;
  if (!(ex <= 60)) return 2;
  if (ex < -1) return 0;  // no part of a cell rounds to a unit
  const float up = __int_as_float((23 - ex + 127) << 23);  // 2^(23 - ex)
  r.f.Q = ((unsigned long long)__float2uint_rn(q.h * up) << 39) + (unsigned long long)((long long)__float2int_rn(q.l * up * 524288.0f) << 20);
  r.f.shift = 61 - ex;
  r.f.whole = (r.f.Q + (1ull << (61 - ex))) >> (62 - ex);
  auto wrap = [&](int x) { x %= a.n; return x < 0 ? x + a.n : x; };
  r.A0 = wrap(base[0] + lo[0]);
  r.B0 = wrap(base[1] + lo[1]);
  r.K0 = wrap(base[2]);
  r.wa = w[0];
  r.wb = w[1];
  r.inv_wa = 1.0f / (float)w[0];
  r.form = 1;
  return 1;
}

// Units of a part L 2^-42 of a cell, 0 < L < 2^42, rounded.
__device__ __forceinline__ unsigned long long part_units(long long L, unsigned long long Q, int shift) {
  const unsigned long long p = __umul64hi((unsigned long long)L << (63 - kZBits), Q);
  return (p + (1ull << (shift - 1))) >> shift;
}

// One interval of a column: its first and last parts, the column, its first
// cell and the tetrahedron, its cells and where they start among the step's.
struct Interval {
  long long first, last;
  unsigned column;
  unsigned cell_tet;  // cell | tetrahedron << 16
  int start, cells;
};

struct ResampleWarp {
  ResampleTet tets[32];
  int2 runs[32];       // tetrahedra with columns: their slot, where their columns start
  Interval found[32];  // the intervals of a step
};

// One column (da, db) of a tetrahedron in the FP64 form.
__device__ __noinline__ void column_f64(const ResampleArgs& a, const ResampleTet& r, int da, int db, unsigned& n_int,
                                        unsigned& n_piece) {
  const int n = a.n;
  const double gs = a.gs, inv_gs = 1.0 / gs;
  const long long aa = (long long)r.A0 + da, bb = (long long)r.B0 + db;
  // the column's line (x, y, z), relative to the cube's corner
  const double x = ((double)aa + 0.5) * gs - r.d.qx;
  const double y = ((double)bb + 0.5) * gs - r.d.qy;
  double z_in = -1e300, z_out = 1e300;
  bool empty = false;
  for (int f = 0; f < 4; ++f) {
    const double rr = fma(-r.d.ny[f], y, fma(-r.d.nx[f], x, r.d.d[f]));
    const double iz = r.d.inz[f];
    if (iz > 0.0) z_out = fmin(z_out, rr * iz);
    else if (iz < 0.0) z_in = fmax(z_in, rr * iz);
    else if (rr < 0.0) empty = true;
  }
  if (empty || !(z_out > z_in)) return;
  ++n_int;
  const long long aw = ((aa % n) + n) % n, bw = ((bb % n) + n) % n;
  const double zl = r.d.qz + z_in, zh = r.d.qz + z_out;
  long long c = (long long)floor(zl * inv_gs);
  for (int guard = 0; guard < 1 << 20 && (double)c * gs < zh; ++guard, ++c) {
    const double lo = fmax(zl, (double)c * gs), hi = fmin(zh, (double)(c + 1) * gs);
    if (!(hi > lo)) continue;
    ++n_piece;
    const double u = r.d.q * (hi - lo) * a.inv_unit;
    const long long cw = ((c % n) + n) % n;
    if (u < 9.2e18) {
      cell_add(a, a.acc + ((cw * n + bw) * n + aw), __double2ull_rn(u));
    } else {
      atomicOr(&a.ctr->errors, kErrRange);
      atomicAdd(&a.ctr->range_overflow, 1ull);
    }
  }
}

__global__ void __launch_bounds__(kResampleThreads) k_resample(ResampleArgs a) {
  __shared__ ResampleWarp ws[kResampleThreads / 32];
  const long long ntet = 6LL * a.L.n_particles;
  const int lane = threadIdx.x & 31, n = a.n;
  const unsigned FULL = 0xffffffffu, lt_mask = (1u << lane) - 1u, le_mask = (2u << lane) - 1u;
  ResampleWarp& S = ws[threadIdx.x >> 5];
  // ---- one tetrahedron per lane
  const long long tau = (long long)blockIdx.x * kResampleThreads + threadIdx.x;
  int have = 0;
  if (tau < ntet) {
    const long long cube = tau / 6;
    const int s = (int)(tau - 6 * cube);
    const unsigned mask = cube_mask(a.L, a.snapshot, cube);
    if (mask & kNonFiniteCube) {
      atomicOr(&a.ctr->errors, kErrNonFinite);
    } else if (!((mask >> s) & 1u)) {  // zero volume: contributes nothing
      int i, j, k;
      cube_ijk(a.L, cube, i, j, k);
      have = a.use_ff ? resample_fixed(a, i, j, k, s, S.tets[lane]) : 2;
      if (have == 2 && !resample_f64(a, i, j, k, s, S.tets[lane])) have = 0;
    }
  }
  unsigned n_int = 0, n_piece = 0;
  // ---- the columns of the integer-form tetrahedra, 32 at a time
  auto excl_scan = [&](int v, int& total) {
    int incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(FULL, incl, o);
      if (lane >= o) incl += y;
    }
    total = __shfl_sync(FULL, incl, 31);
    return incl - v;
  };
  const int cols = have == 1 ? S.tets[lane].wa * S.tets[lane].wb : 0;  // below 2^25
  int n_cols;
  const int col0 = excl_scan(cols, n_cols);
  const unsigned with_cols = __ballot_sync(FULL, cols > 0);
  if (cols > 0) S.runs[__popc(with_cols & lt_mask)] = make_int2(lane, col0);
  __syncwarp();
  const long long plane = (long long)n * n;
  // the sum before the last add and the add, looked at when the next one is made
  unsigned long long old = 0ull, added = 0ull;
  bool wrapped = false;
  int runs_before = 0;
  for (int cb = 0; cb < n_cols; cb += 32) {
    // the run (tetrahedron) of a position: those started before the step plus
    // those started in it up to the position, minus one
    const int rel = col0 - cb;
    const unsigned starts = __reduce_or_sync(FULL, (cols > 0 && rel >= 0 && rel < 32) ? 1u << rel : 0u);
    const int run = runs_before + __popc(starts & le_mask) - 1;
    runs_before += __popc(starts);
    long long zi = -(1LL << 62), zo = 1LL << 62;
    int da = 0, db = 0;
    const int2 rs = S.runs[min(max(run, 0), 31)];
    const ResampleTet& r = S.tets[rs.x & 31];
    bool live = cb + lane < n_cols;
    if (live) {
      const int p = cb + lane - rs.y, wa = r.wa;
      db = (int)(((float)p + 0.5f) * r.inv_wa);
      da = p - db * wa;
      if (da < 0) { --db; da += wa; }  // (from 2^20 columns on FP32 can be one off)
      if (da >= wa) { ++db; da -= wa; }
      const int upper = r.f.upper, vertical = r.f.vertical;
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        const long long z = r.f.C[f] + r.f.A[f] * da + r.f.B[f] * db;
        if ((vertical >> f) & 1) live = live && z >= 0;
        else if ((upper >> f) & 1) zo = min(zo, z);
        else zi = max(zi, z);
      }
      live = live && zo > zi;
    }
    const int c0 = (int)(zi >> kZBits), c1 = (int)((zo - 1) >> kZBits);
    const int cells = live ? c1 - c0 + 1 : 0;
    n_int += live ? 1u : 0u;
    n_piece += (unsigned)cells;
    int n_cells;
    const int cell0 = excl_scan(cells, n_cells);
    const unsigned found = __ballot_sync(FULL, live);
    if (live) {
      int aa = r.A0 + da, bb = r.B0 + db, cw = r.K0 + c0;
      while (aa >= n) aa -= n;
      while (bb >= n) bb -= n;
      while (cw >= n) cw -= n;
      while (cw < 0) cw += n;
      Interval v;
      v.first = c0 == c1 ? zo - zi : ((long long)(c0 + 1) << kZBits) - zi;
      v.last = zo - ((long long)c1 << kZBits);
      v.column = (unsigned)bb * (unsigned)n + (unsigned)aa;
      v.cell_tet = (unsigned)cw | (unsigned)rs.x << 16;
      v.start = cell0;
      v.cells = cells;
      S.found[__popc(found & lt_mask)] = v;
    }
    __syncwarp();
    // ---- their cells, 32 at a time
    int before = 0;
    for (int pb = 0; pb < n_cells; pb += 32) {
      const int prel = cell0 - pb;
      const unsigned pstarts = __reduce_or_sync(FULL, (cells > 0 && prel >= 0 && prel < 32) ? 1u << prel : 0u);
      const int o = before + __popc(pstarts & le_mask) - 1;
      before += __popc(pstarts);
      if (pb + lane < n_cells) {
        const Interval v = S.found[o & 31];
        const ResampleTet& t = S.tets[v.cell_tet >> 16];
        const int k = pb + lane - v.start;
        int cw = (int)(v.cell_tet & 0xffffu) + k;
        if (cw >= n) cw = cw < 2 * n ? cw - n : cw % n;
        const long long len = k == 0 ? v.first : k == v.cells - 1 ? v.last : kZOne;
        const unsigned long long u = len == kZOne ? t.f.whole : part_units(len, t.f.Q, t.f.shift);
        if (u) {
          wrapped = wrapped || old > ~added;
          added = u;
          old = atomicAdd(a.acc + (cw * plane + v.column), u);
        }
      }
    }
    __syncwarp();
  }
  wrapped = wrapped || old > ~added;
  if (wrapped) {
    atomicOr(&a.ctr->errors, kErrRange);
    atomicAdd(&a.ctr->range_overflow, 1ull);
  }
  // ---- the others in turn, in FP64: the warp's lanes take the columns of one
  unsigned todo = __ballot_sync(FULL, have == 2);
  while (todo) {
    const int src = __ffs(todo) - 1;
    todo &= todo - 1u;
    const ResampleTet& r = S.tets[src];
    const int wa = r.wa;
    for (int db = 0; db < r.wb; ++db)
      for (int da = lane; da < wa; da += 32) column_f64(a, r, da, db, n_int, n_piece);
  }
  const unsigned wi = __reduce_add_sync(FULL, n_int), wp = __reduce_add_sync(FULL, n_piece);
  if (lane == 0) {
    if (wi) atomicAdd(&a.ctr->resample_intervals, (unsigned long long)wi);
    if (wp) atomicAdd(&a.ctr->resample_pieces, (unsigned long long)wp);
  }
}

cudaError_t launch_resample(const Lattice& L, int snapshot, int n, int weight, double m_tet, double unit,
                            unsigned long long* d_acc, float* d_out, DevCounters* ctr, cudaStream_t s) {
  const long long cells = (long long)n * n * n;
  cudaError_t e = cudaMemsetAsync(d_acc, 0, sizeof(unsigned long long) * cells, s);
  if (e != cudaSuccess) return e;
  ResampleArgs a;
  a.L = L;
  a.snapshot = snapshot;
  a.n = n;
  a.weight = weight;
  a.gs = (double)L.box / n;
  a.m_tet = m_tet;
  a.inv_unit = 1.0 / unit;
  auto split = [](double v) { ff f; f.h = (float)v; f.l = (float)(v - (double)f.h); return f; };
  const double h = (double)L.box / L.N;
  a.h = split(h);
  a.inv_g = split(n / (double)L.box);
  a.cells = split((double)n / L.N);
  const double whole = (weight == 0 ? 6.0 * m_tet : 1.0) * a.gs * a.inv_unit;
  a.q_num = split(whole);
  // lengths, and products down to h^3 2^-60 and units over h^3, inside FP32's range
  auto within = [](double v, double lo, double hi) { return v > lo && v < hi; };
  a.use_ff = within(h, 1e-6, 1e4) && within(n / (double)L.box, 1e-6, 1e9) && within(whole, 1e-20, 1e18) &&
             (weight != 0 || within(whole / (h * h * h), 1e-6, 1e18));
  a.acc = d_acc;
  a.ctr = ctr;
  const long long blocks = (6LL * L.n_particles + kResampleThreads - 1) / kResampleThreads;
  k_resample<<<(unsigned)blocks, kResampleThreads, 0, s>>>(a);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return launch_fixed_finalize(d_acc, cells, unit, false, nullptr, d_out, s);
}

}  // namespace lt
