// lt_backward.cu -- adjoint of the orthographic projection: dL/d(position)
// from dL/dI, differentiating the per-tetrahedron pyramid form of
// rho_t * dl_t (Eq. 6, 3, 9) with respect to the projected vertices.
//
// Inside the region where hull edge e = (j, k) is the lowest of the pyramid
// faces, the value is f_e(x) = Kn * sigma * N(x) / (o1 o2) with
// N(x) = orient(v_j, v_k, x) and o1, o2 = orient(v_j, v_k, v_l1 / v_l2).
// Its derivative with respect to any vertex is affine in x, so the sums over
// a tetrahedron's fragments only need the moments sum g, sum g X, sum g Y
// of dL/dI per active edge. One thread per tetrahedron walks its fragments as a
// gather from dL/dI (no atomics); a block's six warps take the same 32 cubes, a
// row of the connectivity table each, so that a warp's tetrahedra are neighbours
// of one shape. The block then adds them up per cube corner in the table's order
// and keeps the corner gradients in registers over all frames, and a second
// kernel gathers them per particle in a fixed order.
//
// What bounds it: instruction issue and divergence in the walk. One thread per
// cube, with six tetrahedra and eight corner gradients in 254 registers, ran at
// 10% occupancy with 12 of 32 threads an instruction: 1.57 ms for 64^3 particles
// at 512^2. Now 0.75 ms (four blocks per SM; 14 threads an instruction). A
// tetrahedron's moments keep their order, pixel by pixel: sums in another order
// round by as much as their terms cancel, a thousand times the last bit.
#include "lt_internal.h"

namespace lt {

struct Moments {
  float g0[4], gx[4], gy[4];
};

// Gradient of the projected canonical vertices (pixel units) from the moments.
__device__ __forceinline__ void edge_grad(const TetCanon& K, int e, float Kn, float tiny, const Moments& m,
                                          float* gxv, float* gyv) {
  const EdgeRef r = edge_ref(K, e);
  const float prod = r.o1 * r.o2;
  if (!(fabsf(prod) > tiny) || m.g0[e] == 0.0f) return;
  if (!K.caseB && e == 3) return;
  const float sg = (r.o1 + r.o2) < 0.0f ? -1.0f : 1.0f;
  const float A = Kn * sg / prod;
  const float xj = sel4(K.x, r.j), yj = sel4(K.y, r.j);
  const float xl1 = sel4(K.x, r.l1), yl1 = sel4(K.y, r.l1);
  const float xl2 = sel4(K.x, r.l2), yl2 = sel4(K.y, r.l2);
  const float SGy = m.gy[e] - yj * m.g0[e];  // sum g (Y - y_j)
  const float SGx = m.gx[e] - xj * m.g0[e];  // sum g (X - x_j)
  const float SN = r.ex * SGy - r.ey * SGx;  // sum g N
  const float R1 = SN / r.o1, R2 = SN / r.o2;
  const float s1x = xl1 - xj, s1y = yl1 - yj, s2x = xl2 - xj, s2y = yl2 - yj;
  // vertex k
  const float gkx = A * (SGy - R1 * s1y - R2 * s2y);
  const float gky = A * (-SGx + R1 * s1x + R2 * s2x);
  // vertex j
  const float gjx = A * ((-SGy + r.ey * m.g0[e]) - R1 * (-s1y + r.ey) - R2 * (-s2y + r.ey));
  const float gjy = A * ((SGx - r.ex * m.g0[e]) - R1 * (s1x - r.ex) - R2 * (s2x - r.ex));
  // the two others
  const float gl1x = A * R1 * r.ey, gl1y = -A * R1 * r.ex;
  const float gl2x = A * R2 * r.ey, gl2y = -A * R2 * r.ex;
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    gxv[v] += (v == r.k ? gkx : 0.f) + (v == r.j ? gjx : 0.f) + (v == r.l1 ? gl1x : 0.f) + (v == r.l2 ? gl2x : 0.f);
    gyv[v] += (v == r.k ? gky : 0.f) + (v == r.j ? gjy : 0.f) + (v == r.l1 ? gl1y : 0.f) + (v == r.l2 ? gl2y : 0.f);
  }
}

constexpr int kBackCubes = 32;                // cubes of a block
constexpr int kBackThreads = 6 * kBackCubes;  // their tetrahedra
constexpr int kBackItems = 8 * kBackCubes;    // their corners

// Gradient of one tetrahedron's projected vertices (pixel units, in the table's
// order) in one frame, added to gx, gy.
__device__ __forceinline__ void backward_tet(const Lattice& L, const FrameDev& F, long long cube, int s,
                                             const float* __restrict__ gimg, float (&gx)[4], float (&gy)[4]) {
  TetProj P;
  if (!project_tet<false>(L, F, cube, s, P)) return;
  const float Kn = 6.0f * F.K;
  TetRaster t;
  if (!tet_setup<false, true>(P.x[0], P.y[0], P.x[1], P.y[1], P.x[2], P.y[2], P.x[3], P.y[3], 0.f, 0.f, 0.f, 0.f, Kn, 0.f,
                              0.f, t))
    return;
  float ia[4];  // (the spans have room for its rounding)
#pragma unroll
  for (int e = 0; e < 4; ++e) ia[e] = inv_or_zero(t.a[e]);
  int sx0, sx1, sy0, sy1;
  const float axa = P.axh + P.axl, aya = P.ayh + P.ayl;
  shift_range(axa + t.xmin, axa + t.xmax, -0.5f, (float)F.W - 0.5f, (float)F.W, F.wrap != 0, sx0, sx1);
  shift_range(aya + t.ymin, aya + t.ymax, -0.5f, (float)F.H - 0.5f, (float)F.H, F.wrap != 0, sy0, sy1);
  sx1 = min(sx1, sx0 + 63);
  sy1 = min(sy1, sy0 + 63);
  for (int sy = sy0; sy <= sy1; ++sy)
    for (int sx = sx0; sx <= sx1; ++sx) {
      const int shx = sx * F.W, shy = sy * F.H;
      const float ax = axa + (float)shx, ay = aya + (float)shy;
      const int qx0 = max(0, (int)ceilf(ax + t.xmin - 1e-3f)), qx1 = min(F.W - 1, (int)floorf(ax + t.xmax + 1e-3f));
      const int qy0 = max(0, (int)ceilf(ay + t.ymin - 1e-3f)), qy1 = min(F.H - 1, (int)floorf(ay + t.ymax + 1e-3f));
      if (qx0 > qx1 || qy0 > qy1) continue;
      Moments m;
#pragma unroll
      for (int e = 0; e < 4; ++e) m.g0[e] = m.gx[e] = m.gy[e] = 0.f;
      for (int py = qy0; py <= qy1; ++py) {
        const float Y = rel_coord(py, shy, P.ayh, P.ayl);
        float erow[4];
        float lo = -3.0e38f, hi = 3.0e38f;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          // pixels where every edge function is >= 0, with a small margin
          erow[e] = fmaf(t.b[e], Y, t.c[e]);
          const float xb = -erow[e] * ia[e];
          if (t.a[e] > 0.0f) lo = fmaxf(lo, xb);
          else if (t.a[e] < 0.0f) hi = fminf(hi, xb);
          else if (erow[e] < 0.0f) hi = -3.0e38f;
        }
        const int xa = max(qx0, (int)ceilf(fmaxf(lo - 1e-3f + ax, -1.0e9f)));
        const int xb = min(qx1, (int)floorf(fminf(hi + 1e-3f + ax, 1.0e9f)));
        const float* grow = gimg + (long long)py * F.W;
        for (int px = xa; px <= xb; ++px) {
          const float X = rel_coord(px, shx, P.axh, P.axl);
          float v[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) v[e] = fmaf(t.a[e], X, erow[e]);
          int am = 0;
          float mn = v[0];
#pragma unroll
          for (int e = 1; e < 4; ++e)
            if (v[e] < mn) { mn = v[e]; am = e; }
          if (!(mn > 0.0f)) continue;
          const float g = __ldg(grow + px);
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float w = (am == e) ? g : 0.f;
            m.g0[e] += w;
            m.gx[e] = fmaf(w, X, m.gx[e]);
            m.gy[e] = fmaf(w, Y, m.gy[e]);
          }
        }
      }
      TetCanon K;
      if (!tet_canon<true>(P.x[0], P.y[0], P.x[1], P.y[1], P.x[2], P.y[2], P.x[3], P.y[3], 0.f, 0.f, 0.f, 0.f, K)) continue;
      const float tiny = K.S * K.S * 1e-12f;
      float cx[4] = {0.f, 0.f, 0.f, 0.f}, cy[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int e = 0; e < 4; ++e) edge_grad(K, e, Kn, tiny, m, cx, cy);
      // canonical position -> the table's place
#pragma unroll
      for (int v = 0; v < 4; ++v)
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (K.perm[v] == q) { gx[q] += cx[v]; gy[q] += cy[v]; }
    }
}

__global__ void __launch_bounds__(kBackThreads, 4) k_backward(Lattice L, const FrameDev* __restrict__ frames, int n_frames,
                                                           long long stride, const float* __restrict__ dLdI,
                                                           float* __restrict__ corner_grad) {
  __shared__ float2 part[6][4][kBackCubes];  // per tetrahedron and vertex
  const long long ncube = L.n_particles;
  const int snap = blockIdx.y;
  const int s = threadIdx.x / kBackCubes, c = threadIdx.x % kBackCubes;
  for (long long base = (long long)blockIdx.x * kBackCubes; base < ncube; base += (long long)gridDim.x * kBackCubes) {
    const long long cube = base + c;
    // zero volume, or a cube with a corner that is not finite: contributes nothing
    const bool drawn = cube < ncube && !(cube_mask(L, snap, cube) & (1u << s | kNonFiniteCube));
    float G[2][3];  // corner items threadIdx.x and, for the first threads, kBackThreads further
#pragma unroll
    for (int h = 0; h < 2; ++h) G[h][0] = G[h][1] = G[h][2] = 0.f;
    for (int f = 0; f < n_frames; ++f) {
      const FrameDev& F = frames[f];
      if (F.snapshot != snap || F.persp) continue;
      float gx[4] = {0.f, 0.f, 0.f, 0.f}, gy[4] = {0.f, 0.f, 0.f, 0.f};
      if (drawn) backward_tet(L, F, cube, s, dLdI + (long long)f * stride, gx, gy);
#pragma unroll
      for (int q = 0; q < 4; ++q) part[s][q][c] = make_float2(gx[q], gy[q]);
      __syncthreads();
      // pixel -> world: x_pix = (r . P) sx + const, y_pix = (u . P) sy + const; the
      // edge functions are in fixed-point accumulator units, converted by F.unit
      const float unit = (float)F.unit;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int item = threadIdx.x + h * kBackThreads;
        if (item >= kBackItems) break;
        const int n = item / kBackCubes, ci = item % kBackCubes;
        float px = 0.f, py = 0.f;
#pragma unroll
        for (int r = 0; r < 6; ++r)
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (tet_corner(r, q) == n) {
              const float2 v = part[r][q][ci];
              px += v.x;
              py += v.y;
            }
#pragma unroll
        for (int q = 0; q < 3; ++q) G[h][q] += (px * F.sx * F.r[q] + py * F.sy * F.u[q]) * unit;
      }
      __syncthreads();
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int item = threadIdx.x + h * kBackThreads;
      const long long ic = base + item % kBackCubes;
      if (item >= kBackItems || ic >= ncube) continue;
      float* out = corner_grad + ((long long)snap * ncube + ic) * 24 + 3 * (item / kBackCubes);
      out[0] = G[h][0];
      out[1] = G[h][1];
      out[2] = G[h][2];
    }
  }
}

// dL/d(particle) = sum over the 8 cubes sharing the particle as corner n.
__global__ void k_gather(Lattice L, const float* __restrict__ corner_grad, float* __restrict__ dLdpos) {
  const long long np = L.n_particles;
  const int snap = blockIdx.y;
  const int N = L.N;
  for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < np; p += (long long)gridDim.x * blockDim.x) {
    int i, j, k;
    cube_ijk(L, p, i, j, k);
    float gx = 0.f, gy = 0.f, gz = 0.f;
#pragma unroll
    for (int n = 0; n < 8; ++n) {
      const int a = n & 1, b = (n >> 1) & 1, c = (n >> 2) & 1;
      const int ci = i - a < 0 ? i - a + N : i - a, cj = j - b < 0 ? j - b + N : j - b, ck = k - c < 0 ? k - c + N : k - c;
      const long long cube = particle_id(ci, cj, ck, N);
      const float* g = corner_grad + ((long long)snap * np + cube) * 24 + n * 3;
      gx += g[0];
      gy += g[1];
      gz += g[2];
    }
    float* o = dLdpos + ((long long)snap * np + p) * 3;
    o[0] = gx;
    o[1] = gy;
    o[2] = gz;
  }
}

cudaError_t launch_backward(const Lattice& L, const FrameDev* d_frames, long long stride, int n_frames, int n_snap,
                            const float* dLdI, float* corner_grad, cudaStream_t s) {
  long long b = (L.n_particles + kBackCubes - 1) / kBackCubes;
  if (b > 65536) b = 65536;
  dim3 grid((unsigned)(b < 1 ? 1 : b), n_snap);
  k_backward<<<grid, kBackThreads, 0, s>>>(L, d_frames, n_frames, stride, dLdI, corner_grad);
  return cudaGetLastError();
}

cudaError_t launch_gather_grad(const Lattice& L, int n_snap, const float* corner_grad, float* dLdpos,
                               cudaStream_t s) {
  long long b = (L.n_particles + 255) / 256;
  if (b > 8192) b = 8192;
  dim3 grid((unsigned)(b < 1 ? 1 : b), n_snap);
  k_gather<<<grid, 256, 0, s>>>(L, corner_grad, dLdpos);
  return cudaGetLastError();
}

}  // namespace lt
