// lt_slice.cu -- the total density of overlapping streams (Eq. 4) and the
// number of streams (Sec. 3.2) on a plane z = z0 of the periodic box, at the
// centres of an n x n grid over the box: the paper's 2D density slices
// through the tessellation.
//
// A point's total density is the sum of rho_t = m / |V_t| (Eq. 3) over the
// tetrahedra t that contain it (any periodic copy); its stream count is the
// number of them. A block takes four groups
// of 128 consecutive cubes, a quarter of the lattice apart (the cubes at the
// plane are neighbours: no block holds many of them):
//   * one thread per cube finds the cube's z-range in FP32, widened by the
//     rounding it can carry, and for the cubes that reach the plane (or a
//     periodic copy of it) the same for the six tetrahedra; those that reach
//     it go to a list in shared memory;
//   * the listed tetrahedra are set up 32 at a time, one per lane,
//     in FP64 relative to the cube's Lagrangian corner: the bounding box of
//     the cross-section, bounded by the crossings of the six edges, and the
//     four face planes;
//   * each of them is walked by its warp, 32 candidate points at a time. A
//     point is inside when it lies on the inner side of all four face planes
//     (a point on a face counts, like for the closed tetrahedron). The side is
//     taken in FP32 where its value exceeds the rounding it can carry, else in
//     FP64, so the decision is the FP64 one;
//   * q_t is added to the point's 64-bit fixed-point sum with a global
//     integer atomic, so the slice does not depend on the order of the adds.
// A second kernel converts the sums to float.
//
// What bounds it: with the corners of every cube in FP64 and one thread per
// cube walking its points, the FP64 pipe took 29.4 ms for 256^3 particles and
// 2048^2 points; now 1.1 ms, of which the FP32 scan of all cubes is about 0.4
// (its 16-byte particles alone 0.04), the FP64 setup at the plane 0.5, the points
// 0.15. Six resident blocks, what shared memory holds, hide the scan's loads (72
// registers, cut for seven; 80, cut for six, are 3% slower): five (96 registers)
// took 1.19 ms, three (148) 1.35, blocks of 64 threads 1.22.
#include <math.h>

#include "lt_internal.h"

namespace lt {

constexpr int kSliceThreads = 128;
constexpr int kSliceCubes = 512;  // per block: four independent sets of loads per thread in the scan

struct SliceArgs {
  Lattice L;
  int snapshot, n, weight;
  double z0, gs, m_tet, inv_unit;
  float z0_in_box, z_margin;  // z0 reduced to [0, box); rounding of the FP32 z-range
  unsigned long long* acc;  // [n][n] fixed-point sums
  DevCounters* ctr;
};

// One tetrahedron (and periodic copy of the plane) as the warp's lanes read it.
struct SliceTet {
  double nx[4], ny[4], nz[4], off[4];  // inside face f: nx x + ny y + nz z <= off
  float fa[4], fb[4], fc[4];   // fc - fa da - fb db: the same side in FP32, (da, db) from the first point
  float err;                   // rounding bound of that value
  double qx, qy, z;            // the cube's Lagrangian corner; the plane relative to it
  long long A0, B0;
  unsigned long long add;      // q_t in fixed point (0: out of range)
  int wa, wb;
};

// Bit s: the z-range of tetrahedron s of the cube may reach the plane (or a
// periodic copy of it).
__device__ __forceinline__ unsigned slice_reaches(const SliceArgs& a, long long soff, int i, int j, int k) {
  const Lattice& L = a.L;
  const int N = L.N;
  const int ip = i + 1 == N ? 0 : i + 1, jp = j + 1 == N ? 0 : j + 1, kp = k + 1 == N ? 0 : k + 1;
  float z[8];
  float zmn = 3.0e38f, zmx = -3.0e38f;
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const int im = c & 1 ? ip : i, jm = c & 2 ? jp : j, km = c & 4 ? kp : k;
    const long long id = soff + particle_id(im, jm, km, N);
    float d;
    if (L.fmt == 0) d = min_image(__ldg(reinterpret_cast<const float*>(L.pos) + 4 * id + 2), (float)km * L.h, L.box, L.half_box);
    else d = __half2float(__ldg(reinterpret_cast<const __half*>(L.pos) + 4 * id + 2)) * L.h;
    z[c] = (c & 4 ? L.h : 0.f) + d;
    zmn = fminf(zmn, z[c]);
    zmx = fmaxf(zmx, z[c]);
  }
  const float q = (float)k * L.h - a.z0_in_box, ib = 1.0f / L.box;
  auto reach = [&](float lo, float hi) { return ceilf((q + lo - a.z_margin) * ib) <= floorf((q + hi + a.z_margin) * ib); };
  if (!reach(zmn, zmx)) return 0u;
  unsigned m = 0u;
#pragma unroll
  for (int s = 0; s < 6; ++s) {
    const float z0 = z[tet_corner(s, 0)], z1 = z[tet_corner(s, 1)], z2 = z[tet_corner(s, 2)], z3 = z[tet_corner(s, 3)];
    if (reach(fminf(fminf(z0, z1), fminf(z2, z3)), fmaxf(fmaxf(z0, z1), fmaxf(z2, z3)))) m |= 1u << s;
  }
  return m;
}

// Periodic copies p0 .. p1 of the plane that cross the cube, in FP64; false
// when a corner is not finite (the cube contributes nothing).
__device__ __forceinline__ bool slice_copies(const SliceArgs& a, long long soff, int i, int j, int k, long long& p0,
                                             long long& p1) {
  const Lattice& L = a.L;
  const int N = L.N;
  const double h = (double)L.box / N, box = (double)L.box;
  double zmn = 1e300, zmx = -1e300;
  bool ok = true;
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const float3 df = load_disp(L, soff, i, j, k, c, ok);
    double d = df.z;
    if (L.fmt == 0) {
      const int im = i + (c & 1) == N ? 0 : i + (c & 1), jm = j + ((c >> 1) & 1) == N ? 0 : j + ((c >> 1) & 1);
      const int km = k + (c >> 2) == N ? 0 : k + (c >> 2);
      d = (double)__ldg(reinterpret_cast<const float*>(L.pos) + 4 * (soff + particle_id(im, jm, km, N)) + 2) - km * h;
      if (d > 0.5 * box) d -= box;
      else if (d < -0.5 * box) d += box;
    }
    const double z = (c >> 2) * h + d;
    zmn = fmin(zmn, z);
    zmx = fmax(zmx, z);
  }
  const double qz = k * h;
  p0 = (long long)ceil((qz + zmn - a.z0) / box);
  p1 = min((long long)floor((qz + zmx - a.z0) / box), p0 + 3);
  return ok;
}

__device__ __forceinline__ void slice_add(const SliceArgs& a, long long bw, long long aw, unsigned long long add) {
  if (add) {
    const unsigned long long old = atomicAdd(a.acc + (bw * a.n + aw), add);
    if (old <= ~0ull - add) return;
  }
  atomicOr(&a.ctr->errors, kErrRange);
  atomicAdd(&a.ctr->range_overflow, 1ull);
}

__global__ void __launch_bounds__(kSliceThreads, 7) k_slice(SliceArgs a) {
  __shared__ SliceTet tets[kSliceThreads];
  __shared__ unsigned short list[6 * kSliceCubes];  // 6 x cube of the block + s
  __shared__ int n_list;
  const int N = a.L.N, n = a.n;
  const double h = (double)a.L.box / N, box = (double)a.L.box, gs = a.gs;
  const long long soff = (long long)a.snapshot * a.L.n_particles;
  // cube c of the block: c % 128 of group blockIdx.x + (c / 128) gridDim.x
  auto cube_at = [&](int c) {
    return ((long long)(c / kSliceThreads) * gridDim.x + blockIdx.x) * kSliceThreads + c % kSliceThreads;
  };
  const int lane = threadIdx.x & 31;
  const unsigned FULL = 0xffffffffu;
  if (threadIdx.x == 0) n_list = 0;
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kSliceCubes / kSliceThreads; ++r) {
    const int c = r * kSliceThreads + threadIdx.x;
    const long long cube = cube_at(c);
    if (cube < a.L.n_particles) {
      int i, j, k;
      cube_ijk(a.L, cube, i, j, k);
      unsigned m = slice_reaches(a, soff, i, j, k);
      if (m) {
        int at = atomicAdd(&n_list, __popc(m));
        for (; m; m &= m - 1u) list[at++] = (unsigned short)(6 * c + __ffs(m) - 1);
      }
    }
  }
  __syncthreads();
  const int ntet = n_list;
  SliceTet* wt = tets + (threadIdx.x & ~31);
  for (int tb = threadIdx.x & ~31; tb < ntet; tb += kSliceThreads) {
    // ---- one tetrahedron per lane
    const int tau = tb + lane;
    bool live = false;
    double v[4][3], nrm[4][3], off[4], q = 0.0;
    double qx = 0.0, qy = 0.0, qz = 0.0;
    long long p0 = 0, p1 = -1;
    if (tau < ntet) {
      const int s = list[tau] % 6;
      const long long cube = cube_at(list[tau] / 6);
      if (!tet_degenerate(a.L, a.snapshot, cube, s)) {  // zero volume: contributes nothing
        int i, j, k;
        cube_ijk(a.L, cube, i, j, k);
        if (slice_copies(a, soff, i, j, k, p0, p1) && p0 <= p1) {
          bool ok = true;
          TetF64 t;
          tet_f64(a.L, soff, i, j, k, s, ok, t);
          qx = i * h;
          qy = j * h;
          qz = k * h;
          live = t.V != 0.0;
          q = a.weight == 0 ? a.m_tet / fabs(t.V) : 1.0;
#pragma unroll
          for (int f = 0; f < 4; ++f) {
#pragma unroll
            for (int c = 0; c < 3; ++c) { v[f][c] = t.v[f][c]; nrm[f][c] = t.n[f][c]; }
            off[f] = t.d[f];
          }
        }
      }
    }
    const int copies = live ? (int)(p1 - p0 + 1) : 0;
    const int rounds = __reduce_max_sync(FULL, copies);
    for (int pc = 0; pc < rounds; ++pc) {
      bool have = false;
      if (pc < copies) {
        const double zr = a.z0 + (double)(p0 + pc) * box - qz;  // the plane, relative to the cube
        // bounding box of the cross-section: vertices on the plane and the
        // crossings of the edges that span it. In FP32 from the FP64 heights
        // (the two of a crossing differ in sign, so its parameter is off by a
        // few ulp), widened by far more than that: the points' own test decides
        float xmn = 3.0e38f, xmx = -3.0e38f, ymn = 3.0e38f, ymx = -3.0e38f, xr = 0.f;
        float zf[4], xf[4], yf[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          zf[c] = (float)(v[c][2] - zr);
          xf[c] = (float)v[c][0];
          yf[c] = (float)v[c][1];
          xr = fmaxf(xr, fmaxf(fabsf(xf[c]), fabsf(yf[c])));
        }
#pragma unroll
        for (int c1 = 0; c1 < 4; ++c1) {
          if (zf[c1] == 0.f) {
            xmn = fminf(xmn, xf[c1]); xmx = fmaxf(xmx, xf[c1]);
            ymn = fminf(ymn, yf[c1]); ymx = fmaxf(ymx, yf[c1]);
          }
#pragma unroll
          for (int c2 = c1 + 1; c2 < 4; ++c2) {
            const float za = zf[c1], zb = zf[c2];
            if ((za < 0.f && zb > 0.f) || (za > 0.f && zb < 0.f)) {
              const float t = za / (za - zb);
              const float x = fmaf(t, xf[c2] - xf[c1], xf[c1]), y = fmaf(t, yf[c2] - yf[c1], yf[c1]);
              xmn = fminf(xmn, x); xmx = fmaxf(xmx, x);
              ymn = fminf(ymn, y); ymx = fmaxf(ymx, y);
            }
          }
        }
        if (xmn <= xmx) {
          // slice points (unwrapped indices) whose centre can lie in the cross-section
          const double inv = 1.0 / gs, eps = (double)(4.0e-6f * xr) * inv + 1e-9;
          const long long A0 = (long long)ceil((qx + (double)xmn) * inv - 0.5 - eps);
          const long long A1 = (long long)floor((qx + (double)xmx) * inv - 0.5 + eps);
          const long long B0 = (long long)ceil((qy + (double)ymn) * inv - 0.5 - eps);
          const long long B1 = (long long)floor((qy + (double)ymx) * inv - 0.5 + eps);
          if (A0 <= A1 && B0 <= B1) {
            have = true;
            SliceTet& r = wt[lane];
            const long long wa = min(A1 - A0, 4LL * n) + 1, wb = min(B1 - B0, 4LL * n) + 1;
            r.A0 = A0;
            r.B0 = B0;
            r.wa = (int)wa;
            r.wb = (int)wb;
            r.qx = qx;
            r.qy = qy;
            r.z = zr;
            const double x0 = ((double)A0 + 0.5) * gs - qx, y0 = ((double)B0 + 0.5) * gs - qy;
            float err = 0.f;
#pragma unroll
            for (int f = 0; f < 4; ++f) {
              r.nx[f] = nrm[f][0];
              r.ny[f] = nrm[f][1];
              r.nz[f] = nrm[f][2];
              r.off[f] = off[f];
              // the plane's value over its gradient per point step, so that the
              // four sides share one scale and one rounding bound
              const double ga = nrm[f][0] * gs, gb = nrm[f][1] * gs;
              const double tx = nrm[f][0] * x0, ty = nrm[f][1] * y0, tz = nrm[f][2] * zr;
              // (a face nearly in the plane has no gradient: there the scale is
              // that of the FP64 form's own rounding)
              const double sc = fmax(fabs(ga) + fabs(gb), 1e-9 * (fabs(off[f]) + fabs(tx) + fabs(ty) + fabs(tz)));
              const double is = sc > 0.0 ? 1.0 / sc : 1.0;
              const double c = (off[f] - (tx + ty + tz)) * is;
              r.fa[f] = (float)(ga * is);
              r.fb[f] = (float)(gb * is);
              r.fc[f] = (float)c;
              // |fc| and, over the points, |fa| da + |fb| db <= wa + wb
              err = fmaxf(err, fabsf(r.fc[f]));
            }
            // three roundings of 2^-24 each, and the FP64 form's own
            r.err = (err + (float)wa + (float)wb) * 4.0e-7f;
            const double u = q * a.inv_unit;
            r.add = u < 9.2e18 ? (unsigned long long)__double2ull_rn(u) : 0ull;
            // (a value that rounds to nothing adds nothing; 0 marks one out of range)
            if (r.add == 0ull && u < 9.2e18) have = false;
          }
        }
      }
      unsigned todo = __ballot_sync(FULL, have);
      __syncwarp();
      // ---- every tetrahedron in turn: the warp's lanes take its points
      while (todo) {
        const int src = __ffs(todo) - 1;
        todo &= todo - 1u;
        const SliceTet& r = wt[src];
        const int wa = r.wa, wb = r.wb;
        const int step = 0x3fffffff / wa;  // rows per 32-bit index (one pass but for sections of 2^30 points)
        for (int row = 0; row < wb; row += step) {
          const int np = min(step, wb - row) * wa;
          for (int p = lane; p < np; p += 32) {
            const int pr = p / wa, da = p - pr * wa, db = row + pr;
            bool inside = true, close = false;
#pragma unroll
            for (int f = 0; f < 4; ++f) {
              const float sd = fmaf(-r.fb[f], (float)db, fmaf(-r.fa[f], (float)da, r.fc[f]));
              inside = inside && sd > 0.f;
              close = close || !(fabsf(sd) > r.err);
            }
            const long long aa = r.A0 + da, bb = r.B0 + db;
            if (close) {
              const double x = ((double)aa + 0.5) * gs - r.qx, y = ((double)bb + 0.5) * gs - r.qy;
              inside = true;
#pragma unroll
              for (int f = 0; f < 4; ++f) inside = inside && (r.nx[f] * x + r.ny[f] * y + r.nz[f] * r.z <= r.off[f]);
            }
            if (!inside) continue;
            long long aw = aa, bw = bb;
            if (aw < 0 || aw >= n) aw = ((aa % n) + n) % n;
            if (bw < 0 || bw >= n) bw = ((bb % n) + n) % n;
            slice_add(a, bw, aw, r.add);
          }
        }
      }
      __syncwarp();
    }
  }
}

cudaError_t launch_slice(const Lattice& L, int snapshot, int n, int weight, double z0, double m_tet, double unit,
                         unsigned long long* d_acc, float* d_out, DevCounters* ctr, cudaStream_t s) {
  const long long np = (long long)n * n;
  cudaError_t e = cudaMemsetAsync(d_acc, 0, sizeof(unsigned long long) * np, s);
  if (e != cudaSuccess) return e;
  SliceArgs a;
  a.L = L;
  a.snapshot = snapshot;
  a.n = n;
  a.weight = weight;
  a.z0 = z0;
  a.gs = (double)L.box / n;
  a.m_tet = m_tet;
  a.inv_unit = 1.0 / unit;
  a.acc = d_acc;
  a.ctr = ctr;
  // the FP32 z-range: a few roundings of numbers up to a box (and the FP16
  // offsets' range of 65504 cells), and z0 reduced to the box in FP64
  a.z0_in_box = a.z_margin = 0.f;
  const double zred = z0 - floor(z0 / (double)L.box) * (double)L.box;
  a.z0_in_box = (float)zred;
  a.z_margin = L.box * (L.fmt == 0 ? 1.0f : fmaxf(1.0f, 65536.0f / (float)L.N)) * 2.0e-6f;
  if (!(fabs(z0) < 1e9 * (double)L.box)) a.z_margin = INFINITY;  // too far to reduce: every cube goes to FP64
  const long long blocks = (L.n_particles + kSliceCubes - 1) / kSliceCubes;
  k_slice<<<(unsigned)(blocks < 1 ? 1 : blocks), kSliceThreads, 0, s>>>(a);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return launch_fixed_finalize(d_acc, np, unit, false, nullptr, d_out, s);
}

}  // namespace lt
