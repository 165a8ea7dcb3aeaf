// lt_build.cu -- per-tetrahedron signed volume (Eq. 9) and density (Eq. 3)
// for every cube of every snapshot, tetrahedra generated on the fly from the
// lattice index (Sec. 3.1, Sec. 4.1). FP32 determinant on local edge vectors;
// where |V| falls below 0.1 of a lattice cell (sheet-like tetrahedra at
// caustics), recomputed from exact edge vectors in float-float arithmetic, or
// in FP64 for the few whose determinant cancels by more than 2^18.
//
// What bounds it: about half of a deformed lattice's tetrahedra take the
// recomputation. In FP64, with an FP64 division for every density, the FP64
// pipe was 85% busy: 27.2 ms for 256^3 particles with densities, 1.91 ms now
// (671 MB moved, 5% of the copy bandwidth: the FP32 arithmetic, selects of
// the minimum image among it, is what is left).
#include "lt_ff.cuh"
#include "lt_internal.h"

namespace lt {

__device__ __forceinline__ void warp_add_u64(unsigned long long* dst, unsigned v) {
  const unsigned tot = __reduce_add_sync(0xffffffffu, v);
  if ((threadIdx.x & 31) == 0 && tot) atomicAdd(dst, (unsigned long long)tot);
}

// Signed volume of tetrahedron s of cube (i, j, k) in FP64 from the exact
// displacements (the FP32 ones round when they exceed the position's own
// precision range). Out of line: it runs for one tetrahedron in thousands.
__device__ __noinline__ double volume_f64(const Lattice& L, long long soff, int i, int j, int k, int s) {
  const int N = L.N;
  const double hd = (double)L.h, bx = (double)L.box;
  double v[4][3];
#pragma unroll 1
  for (int c = 0; c < 4; ++c) {
    const int n = tet_corner_dyn(s, c);
    const int o[3] = {n & 1, (n >> 1) & 1, (n >> 2) & 1};
    const int im[3] = {i + o[0] == N ? 0 : i + o[0], j + o[1] == N ? 0 : j + o[1], k + o[2] == N ? 0 : k + o[2]};
    double d[3];
    if (L.fmt != 0) {
      bool ok = true;
      const float3 df = load_disp(L, soff, i, j, k, n, ok);  // exact
      d[0] = df.x; d[1] = df.y; d[2] = df.z;
    } else {
      const float4 p = __ldg(reinterpret_cast<const float4*>(L.pos) + soff + particle_id(im[0], im[1], im[2], N));
      const float pv[3] = {p.x, p.y, p.z};
      for (int q = 0; q < 3; ++q) {
        double dd = (double)pv[q] - (double)im[q] * hd;
        if (dd > 0.5 * bx) dd -= bx;
        else if (dd < -0.5 * bx) dd += bx;
        d[q] = dd;
      }
    }
    for (int q = 0; q < 3; ++q) v[c][q] = d[q];
  }
  double e[3][3];
  const int n0 = tet_corner_dyn(s, 0);
  for (int r = 0; r < 3; ++r) {
    const int n = tet_corner_dyn(s, r + 1);
    for (int q = 0; q < 3; ++q) e[r][q] = (v[r + 1][q] - v[0][q]) + (((n >> q) & 1) - ((n0 >> q) & 1)) * hd;
  }
  return (e[0][0] * (e[1][1] * e[2][2] - e[1][2] * e[2][1]) + e[0][1] * (e[1][2] * e[2][0] - e[1][0] * e[2][2]) +
          e[0][2] * (e[1][0] * e[2][1] - e[1][1] * e[2][0])) / 6.0;
}

struct BuildArgs {
  Lattice L;
  double m;
  ff m_ff, box_ff, period_ff, inv6;  // mass of a tetrahedron, box, N h, 1 / 6
  int use_ff;       // the pairs (and their products down to h^3 2^-60) are inside FP32's range
  int rho_vec;      // rho_out is 16-byte aligned
  float* rho_out;
  unsigned char* degen;
  DevCounters* ctr;
};

constexpr int kBuildThreads = 256;

// Volume of tetrahedron s of a cube recomputed: signed volume in float-float
// from exact edge vectors, or (in_f64) in FP64 from volume_f64. An edge vector
// is the exact difference of two stored coordinates (positions, or FP16
// displacements plus lattice offsets), plus, in the cubes that have any, what
// unwraps them: whole boxes for particles that crossed the boundary and
// lattice periods N h for corners past the last lattice plane (not quite the
// same number when h = box / N rounds).
template <bool F16>
__device__ __forceinline__ ff volume_again(const BuildArgs& a, long long soff, long long cube, int s, bool& in_f64,
                                           double& Vd) {
  const Lattice& L = a.L;
  const float h = L.h;
  int i, j, k;
  cube_ijk(L, cube, i, j, k);
  float p[4][3], w[4][3];
  float r[4][3];
  bool wrapped = false;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const int n = tet_corner_dyn(s, c);
    const int ii = i + (n & 1), jj = j + ((n >> 1) & 1), kk = k + (n >> 2);
    if (F16) {
      bool ok = true;
      const float3 d = load_disp(L, soff, i, j, k, n, ok);
      p[c][0] = d.x; p[c][1] = d.y; p[c][2] = d.z;
      w[c][0] = (float)(n & 1) * h; w[c][1] = (float)((n >> 1) & 1) * h; w[c][2] = (float)(n >> 2) * h;
    } else {
      const bool rx = ii == L.N, ry = jj == L.N, rz = kk == L.N;
      const int im = rx ? 0 : ii, jm = ry ? 0 : jj, km = rz ? 0 : kk;
      const float4 v = __ldg(reinterpret_cast<const float4*>(L.pos) + soff + particle_id(im, jm, km, L.N));
      p[c][0] = v.x; p[c][1] = v.y; p[c][2] = v.z;
      auto boxes = [&](float x, float q) { return x - q > L.half_box ? -1.f : x - q < -L.half_box ? 1.f : 0.f; };
      w[c][0] = boxes(v.x, (float)im * h); w[c][1] = boxes(v.y, (float)jm * h); w[c][2] = boxes(v.z, (float)km * h);
      r[c][0] = rx ? 1.f : 0.f; r[c][1] = ry ? 1.f : 0.f; r[c][2] = rz ? 1.f : 0.f;
      wrapped = wrapped || rx || ry || rz || w[c][0] != 0.f || w[c][1] != 0.f || w[c][2] != 0.f;
    }
  }
  in_f64 = !a.use_ff;
  ff V = {0.f, 0.f};
  if (!in_f64) {
    ff e[3][3];
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        e[c][q] = ff_two_diff(p[c + 1][q], p[0][q]);
        if (F16) e[c][q] = e[c][q] + (w[c + 1][q] - w[0][q]);
        else if (wrapped) e[c][q] = (e[c][q] + a.box_ff * (w[c + 1][q] - w[0][q])) + a.period_ff * (r[c + 1][q] - r[0][q]);
      }
    const ff det = e[0][0] * (e[1][1] * e[2][2] - e[1][2] * e[2][1]) + e[0][1] * (e[1][2] * e[2][0] - e[1][0] * e[2][2]) +
                   e[0][2] * (e[1][0] * e[2][1] - e[1][1] * e[2][0]);
    // every operation is off by about 2^-45 of the terms it adds: down to
    // 2^-18 of their sum the determinant keeps 2^-26, below FP32's rounding
    // of the density
    const float mag = fabsf(e[0][0].h) * (fabsf(e[1][1].h * e[2][2].h) + fabsf(e[1][2].h * e[2][1].h)) +
                      fabsf(e[0][1].h) * (fabsf(e[1][2].h * e[2][0].h) + fabsf(e[1][0].h * e[2][2].h)) +
                      fabsf(e[0][2].h) * (fabsf(e[1][0].h * e[2][1].h) + fabsf(e[1][1].h * e[2][0].h));
    V = det * a.inv6;
    // (also taken when the comparison is with a NaN)
    in_f64 = !(fabsf(det.h) >= mag * (1.0f / 262144.0f)) || !(fabsf(det.h) > 1e-30f);
  }
  if (in_f64) Vd = volume_f64(L, soff, i, j, k, s);
  return V;
}

// One thread per cube takes the FP32 determinants of its six tetrahedra; the
// small ones (half of them on a deformed lattice) become jobs, packed in
// shared memory and recomputed 32 at a time by the warp, so that all its
// lanes work and the recomputation appears once in the code (unrolled six
// times it overflowed the instruction cache: 3.05 ms for 256^3 particles
// against 1.91). Densities and flags come together in shared memory; the
// densities leave as 16-byte stores.
template <bool F16>
__global__ void __launch_bounds__(kBuildThreads) k_build_tets(BuildArgs a) {
  __shared__ __align__(16) float rho_s[kBuildThreads * 6];
  __shared__ unsigned char job_s[kBuildThreads * 6];  // lane * 8 + s
  __shared__ unsigned zero_s[kBuildThreads];
  const Lattice& L = a.L;
  const long long ncube = L.n_particles;
  const int snap = blockIdx.y;
  const long long soff = (long long)snap * ncube;
  // FP32 determinant error is about 3 * 2^-24 * |e|^3 / |V| relative; below
  // 0.1 h^3 (0.6 of an undeformed tetrahedron) that could exceed 1e-5
  const float h = L.h, thr = 0.1f * h * h * h;
  const int lane = threadIdx.x & 31, wbase = threadIdx.x & ~31;
  float* wrho = rho_s + wbase * 6;
  unsigned char* wjob = job_s + wbase * 6;
  unsigned* wzero = zero_s + wbase;
  const unsigned FULL = 0xffffffffu;
  for (long long base = (long long)blockIdx.x * blockDim.x; base < ncube; base += (long long)gridDim.x * blockDim.x) {
    const long long cube = base + threadIdx.x;
    unsigned n_nonfinite = 0, n_degen = 0, n_fb = 0, n_inv = 0, small = 0u, zero = 0u;
    bool finite = true;
    if (cube < ncube) {
      int i, j, k;
      cube_ijk(L, cube, i, j, k);
      float3 d[8];
      bool ok0 = true;
      d[0] = load_disp(L, soff, i, j, k, 0, ok0);
      finite = ok0;
#pragma unroll
      for (int n = 1; n < 8; ++n) d[n] = load_disp(L, soff, i, j, k, n, finite);
      n_nonfinite = ok0 ? 0u : 1u;  // each particle is corner 0 of exactly one cube
#pragma unroll
      for (int s = 0; s < 6; ++s) {
        const int n0 = tet_corner(s, 0), n1 = tet_corner(s, 1), n2 = tet_corner(s, 2), n3 = tet_corner(s, 3);
        // edge vectors: displacement differences plus exact lattice offsets
        const float ax = (d[n1].x - d[n0].x) + (float)((n1 & 1) - (n0 & 1)) * h;
        const float ay = (d[n1].y - d[n0].y) + (float)(((n1 >> 1) & 1) - ((n0 >> 1) & 1)) * h;
        const float az = (d[n1].z - d[n0].z) + (float)(((n1 >> 2) & 1) - ((n0 >> 2) & 1)) * h;
        const float bx = (d[n2].x - d[n0].x) + (float)((n2 & 1) - (n0 & 1)) * h;
        const float by = (d[n2].y - d[n0].y) + (float)(((n2 >> 1) & 1) - ((n0 >> 1) & 1)) * h;
        const float bz = (d[n2].z - d[n0].z) + (float)(((n2 >> 2) & 1) - ((n0 >> 2) & 1)) * h;
        const float cx = (d[n3].x - d[n0].x) + (float)((n3 & 1) - (n0 & 1)) * h;
        const float cy = (d[n3].y - d[n0].y) + (float)(((n3 >> 1) & 1) - ((n0 >> 1) & 1)) * h;
        const float cz = (d[n3].z - d[n0].z) + (float)(((n3 >> 2) & 1) - ((n0 >> 2) & 1)) * h;
        const float V = (ax * (by * cz - bz * cy) + ay * (bz * cx - bx * cz) + az * (bx * cy - by * cx)) * (1.0f / 6.0f);
        if (fabsf(V) < thr) {
          small |= 1u << s;
        } else if (V == 0.0f) {  // a lattice so small that the threshold underflows
          ++n_degen;
          zero |= 1u << s;
        } else if (V > 0.0f) {
          ++n_inv;
        }
        if (a.rho_out) {
          float rho = 0.0f;
          if (finite && V != 0.0f) {
            const float v = fabsf(V);
            if (a.use_ff) {
              // m / |V| to about 2^-44 before its one rounding (the residual of a volume
              // past FP32's range, of particles far outside the box, is taken at the
              // range's end: 0 times infinity is no number)
              const float rv = __frcp_rn(v), q = __fmul_rn(a.m_ff.h, rv);
              rho = __fadd_rn(q, __fmul_rn(__fadd_rn(__fmaf_rn(-q, fminf(v, 3.4028235e38f), a.m_ff.h), a.m_ff.l), rv));
            } else {
              rho = (float)(a.m / (double)v);
            }
          }
          wrho[lane * 6 + s] = rho;
        }
      }
      n_fb = __popc(small);
    }
    // ---- the small ones, packed
    wzero[lane] = zero;
    int off = n_fb;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(FULL, off, o);
      if (lane >= o) off += y;
    }
    const int total = __shfl_sync(FULL, off, 31);
    off -= n_fb;
    for (unsigned m = small; m; m &= m - 1u) wjob[off++] = (unsigned char)(lane * 8 + __ffs(m) - 1);
    const unsigned fin = __ballot_sync(FULL, finite);
    __syncwarp();
    for (int t = lane; t < total; t += 32) {
      const int src = wjob[t] >> 3, s = wjob[t] & 7;
      bool in_f64;
      double Vd = 0.0;
      const ff V = volume_again<F16>(a, soff, base + wbase + src, s, in_f64, Vd);
      const bool none = in_f64 && Vd == 0.0;
      if (none) {
        ++n_degen;
        atomicOr(&wzero[src], 1u << s);
      }
      if (in_f64 ? Vd > 0.0 : V.h > 0.0f) ++n_inv;
      if (a.rho_out) {
        float rho = 0.0f;
        if (!none && ((fin >> src) & 1u)) {
          if (in_f64) {
            rho = (float)(a.m / fabs(Vd));
          } else {
            const ff q = a.m_ff / (V.h < 0.0f ? -V : V);
            rho = __fadd_rn(q.h, q.l);
          }
        }
        wrho[src * 6 + s] = rho;
      }
    }
    __syncwarp();
    if (cube < ncube) a.degen[soff + cube] = (unsigned char)(wzero[lane] | (finite ? 0u : kNonFiniteCube));
    if (a.rho_out) {
      const long long w0 = base + wbase;  // the warp's first cube
      float* out = a.rho_out + (soff + w0) * 6;
      const int n = (int)max(0LL, min(32LL, ncube - w0)) * 6;  // values of the warp
      if (a.rho_vec && n == 192) {
        reinterpret_cast<float4*>(out)[lane] = reinterpret_cast<const float4*>(wrho)[lane];
        if (lane < 16) reinterpret_cast<float4*>(out)[32 + lane] = reinterpret_cast<const float4*>(wrho)[32 + lane];
      } else {
        for (int q = lane; q < n; q += 32) out[q] = wrho[q];
      }
    }
    __syncwarp();
    warp_add_u64(&a.ctr->nonfinite, n_nonfinite);
    warp_add_u64(&a.ctr->degenerate, n_degen);
    warp_add_u64(&a.ctr->fp64_fallbacks, n_fb);
    warp_add_u64(&a.ctr->inverted, n_inv);
    if (n_nonfinite) atomicOr(&a.ctr->errors, kErrNonFinite);
  }
}

cudaError_t launch_build_tets(const Lattice& L, int n_snap, double m, float* rho_out, unsigned char* degen,
                              DevCounters* ctr, cudaStream_t s) {
  BuildArgs a;
  a.L = L;
  a.m = m;
  auto split = [](double v) { ff f; f.h = (float)v; f.l = (float)(v - (double)f.h); return f; };
  a.m_ff = split(m);
  a.box_ff = split((double)L.box);
  a.period_ff = split((double)L.N * (double)L.h);
  a.inv6 = split(1.0 / 6.0);
  // h^3 down to 2^-60 of itself, and m / V for V down to 1e-30, in FP32's normal range
  a.use_ff = L.h > 1e-6f && L.h < 1e4f && m > 1e-18 && m < 1e6;
  // (an odd number of particles puts odd snapshots on 8-byte boundaries)
  a.rho_vec = ((uintptr_t)rho_out & 15) == 0 && (n_snap == 1 || (L.n_particles & 1) == 0);
  a.rho_out = rho_out;
  a.degen = degen;
  a.ctr = ctr;
  long long blocks = (L.n_particles + kBuildThreads - 1) / kBuildThreads;
  if (blocks > 152LL * 64) blocks = 152LL * 64;
  if (blocks < 1) blocks = 1;
  // snapshots along the grid's second axis, 65535 at a time
  for (int s0 = 0; s0 < n_snap; s0 += 65535) {
    BuildArgs b = a;
    const int ns = n_snap - s0 < 65535 ? n_snap - s0 : 65535;
    const long long off = (long long)s0 * L.n_particles;
    b.L.pos = (const char*)L.pos + off * (L.fmt == 0 ? 16 : 8);
    if (rho_out) b.rho_out = rho_out + 6 * off;
    b.degen = degen + off;
    if (s0 && b.rho_vec) b.rho_vec = ((uintptr_t)b.rho_out & 15) == 0;
    const dim3 grid((unsigned)blocks, (unsigned)ns);
    if (L.fmt != 0) k_build_tets<true><<<grid, kBuildThreads, 0, s>>>(b);
    else k_build_tets<false><<<grid, kBuildThreads, 0, s>>>(b);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaGetLastError();
}

}  // namespace lt
