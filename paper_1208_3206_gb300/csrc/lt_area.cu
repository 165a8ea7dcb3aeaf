// lt_area.cu -- area-averaged pixels of an orthographic view: each pixel holds
// the mean of the column density of Eq. 6 over its square, instead of the
// value at its centre.
//
// In an orthographic view the chord of one tetrahedron is a continuous,
// piecewise-linear function of the image point: zero on the boundary of the
// projected hull and linear on each triangle that joins the apex to a hull
// edge. The apex is the projected vertex lying inside the triangle of the
// other three, or for a four-vertex hull the crossing of its diagonals. The
// pyramid the chord forms over the hull holds the tetrahedron's volume, so
// rho times the chord at the apex is 3 m / A, with A the hull's area. On the
// triangle of hull edge e the column density is k_e d_e(p), where d_e is that
// edge's line function. Its integral over a pixel is then
// k_e (a_e Mx + b_e My + c_e |P|), where |P|, Mx and My are the area and
// first moments of the triangle clipped to the pixel's square.
//
// Each warp takes 32 tetrahedra (one per lane). A lane projects the vertices to
// pixel units, finds the apex and the hull, and forms the lines of the hull
// edges and of the rays from the apex through the hull vertices, in
// float-float, or in FP64 for projections too near to degenerate (GB300's FP64
// pipe is narrow: the whole setup in FP64 was 27 ms of a frame). The lines are
// relative to the apex's pixel, normalised to |a| + |b| of about 1, and kept as
// float-float pairs in shared memory. Then three stages, each of which packs its
// work to 32 lanes whatever tetrahedra it comes from:
//   1. the pixels of the bounding rectangles, flattened: FP32 hull lines reject
//      those clearly outside (more than half);
//   2. the others, 32 at a time: the lines at the pixel's corner in float-float
//      arithmetic (error-free products and sums), so a line's offset there
//      carries only its own rounding, however far the pixel lies from the apex.
//      A square within one sector, or within the hull over one ray, is the
//      integral of a linear function's positive part (half_square);
//   3. the (pixel, sector) pairs of the other squares, 32 at a time
//      (sector_part).
// Hulls thinner than kThinHull pixels and apexes within kThinSector pixels of a
// hull edge are clipped in FP64 in stage 2: there FP32 rounding of the clip
// would show next to the pixel's own small value. A pixel's sectors are summed
// in 64ths of the accumulator's unit, and the sums added as 64-bit
// fixed-point integers by global atomics, so the image is bitwise reproducible.
// A last kernel converts them to float.
//
// What bounds it: one tetrahedron at a time with a lane per pixel through all
// of it, lanes took different paths: 8.3 of 32 threads an instruction, 273 ms
// for 128^3 particles at 1024^2 (1.58e9 pixels of rectangles). Now
// 58 ms: 3 the setup, 11 stage 1, 30 stage 2 (the eight lines and the tests on
// them, about 800 instructions for 32 pixels), 14 stage 3, at 23 threads an
// instruction.
#include "lt_ff.cuh"
#include "lt_internal.h"

namespace lt {

namespace {

constexpr double kThinHull = 0.05;     // pixels: hull width below which the clip runs in FP64
constexpr double kThinSector = 1e-3;  // pixels: apex distance to a hull edge below which it does too
constexpr int kAreaThreads = 128;

struct AreaArgs {
  Lattice L;
  const FrameDev* frame;
  double m_tet, inv_unit;
  bool use_ff;        // lattice and view inside FP32's range with room
  ff h, axis[2][3];   // box / N; pixels per length along the image's axes
  ff apex;            // 6 m in accumulator units over a pixel's area: column density at the apex times twice the hull
  unsigned long long* acc;  // [H][W]
  DevCounters* ctr;
};

// One tetrahedron's pyramid, lines a x + b y + c relative to the anchor pixel
// (ax, ay), high and low parts of four in turn. Hull edge e (from vertex e to
// e + 1): >= 0 inside; ray from the apex through hull vertex e: >= 0 on the side
// of edge e. (92 words: the strides of neighbours fall on different banks.)
struct __align__(16) AreaTet {
  float hull_h[3][4], hull_l[3][4];
  float ray_h[3][4], ray_l[3][4];
  float k[4];         // column density per unit of hull line e, in accumulator units
  float kr[4];        // what sector e - 1's column density exceeds sector e's by, per unit of ray e
  float vx_h[4], vx_l[4], vy_h[4], vy_l[4];  // hull vertices
  float qx, qy;       // the apex (in the anchor pixel)
  int n, ax, ay, thin;
  int x0, y0, wx;
  float inv_wx;
  float margin;       // FP32 rounding of a hull line anywhere in the rectangle
  int np, flat, pad[3];   // flat: some sector has no area
};

__device__ __forceinline__ double orient(double ax, double ay, double bx, double by, double cx, double cy) {
  return (bx - ax) * (cy - ay) - (by - ay) * (cx - ax);
}

__device__ __forceinline__ float2 split_ff(double x) {
  const float hi = (float)x;
  return make_float2(hi, (float)(x - (double)hi));
}

// Line through (px, py) with direction (dx, dy), positive on its left.
__device__ __forceinline__ void make_line(double px, double py, double dx, double dy, float (*h)[4], float (*l)[4], int e) {
  const double a = -dy, b = dx, s = fabs(a) + fabs(b);
  const double inv = s > 0.0 ? 1.0 / s : 0.0;
  const double v[3] = {a * inv, b * inv, (dy * px - dx * py) * inv};
  for (int q = 0; q < 3; ++q) {
    const float2 p = split_ff(v[q]);
    h[q][e] = p.x;
    l[q][e] = p.y;
  }
}

__device__ __forceinline__ void make_line(ff px, ff py, ff dx, ff dy, float (*h)[4], float (*l)[4], int e) {
  const float s = fabsf(dx.h) + fabsf(dy.h), inv = s > 0.f ? fast_rcp(s) : 0.f;
  const ff a = -dy * inv, b = dx * inv, c = (dy * px - dx * py) * inv;
  h[0][e] = a.h; l[0][e] = a.l;
  h[1][e] = b.h; l[1][e] = b.l;
  h[2][e] = c.h; l[2][e] = c.l;
}

// a ox + b oy + c for float-float a, b, c and integer ox, oy (exact in FP32):
// error-free products and two-sums, then the small terms (Dekker, Knuth).
__device__ __forceinline__ float line_ff(const float (*h)[4], const float (*l)[4], int e, float ox, float oy) {
  const float ah = h[0][e], bh = h[1][e], ch = h[2][e];
  const float p1 = __fmul_rn(ah, ox), e1 = __fmaf_rn(l[0][e], ox, __fmaf_rn(ah, ox, -p1));
  const float p2 = __fmul_rn(bh, oy), e2 = __fmaf_rn(l[1][e], oy, __fmaf_rn(bh, oy, -p2));
  const ff s = ff_two_sum(p1, p2), t = ff_two_sum(ch, s.h);
  return __fadd_rn(t.h, __fadd_rn(__fadd_rn(__fadd_rn(t.l, s.l), __fadd_rn(e1, e2)), l[2][e]));
}

__device__ __forceinline__ double line_f64(const float (*h)[4], const float (*l)[4], int e, double ox, double oy) {
  const double a = (double)h[0][e] + (double)l[0][e], b = (double)h[1][e] + (double)l[1][e];
  return fma(b, oy, fma(a, ox, (double)h[2][e] + (double)l[2][e]));
}

// Clip the convex polygon (xi, yi)[n] to a x + b y + c >= 0 (Sutherland-Hodgman).
template <typename T, typename Buf>
__device__ __forceinline__ int clip_poly(Buf xi, Buf yi, int n, T a, T b, T c, Buf xo, Buf yo) {
  int m = 0;
  T dp = c + a * xi[n - 1] + b * yi[n - 1];
  int j = n - 1;
  for (int i = 0; i < n; ++i) {
    const T d = c + a * xi[i] + b * yi[i];
    if ((d >= T(0)) != (dp >= T(0))) {
      const T t = dp / (dp - d);
      xo[m] = xi[j] + t * (xi[i] - xi[j]);
      yo[m] = yi[j] + t * (yi[i] - yi[j]);
      ++m;
    }
    if (d >= T(0)) {
      xo[m] = xi[i];
      yo[m] = yi[i];
      ++m;
    }
    dp = d;
    j = i;
  }
  return m;
}

// Integral over the unit square, in FP64, of the hull line function l0 = (a0, b0, c0),
// restricted to l0 >= 0, l1 >= 0 and l2 >= 0; xa, ya, xb, yb hold 8 vertices each.
template <typename T, typename Buf>
__device__ T sector_integral(T a0, T b0, T c0, T a1, T b1, T c1, T a2, T b2, T c2, Buf xa, Buf ya, Buf xb, Buf yb) {
  const T la[3] = {a0, a1, a2}, lb[3] = {b0, b1, b2}, lc[3] = {c0, c1, c2};
  bool inside[3];
#pragma unroll
  for (int l = 0; l < 3; ++l) {
    // largest and smallest value over the square's corners
    const T hi = lc[l] + (la[l] > T(0) ? la[l] : T(0)) + (lb[l] > T(0) ? lb[l] : T(0));
    const T lo = lc[l] + (la[l] < T(0) ? la[l] : T(0)) + (lb[l] < T(0) ? lb[l] : T(0));
    if (hi <= T(0)) return T(0);
    inside[l] = lo >= T(0);
  }
  if (inside[0] && inside[1] && inside[2]) return T(0.5) * (a0 + b0) + c0;
  xa[0] = T(0); xa[1] = T(1); xa[2] = T(1); xa[3] = T(0);
  ya[0] = T(0); ya[1] = T(0); ya[2] = T(1); ya[3] = T(1);
  int n = 4;
  bool in_a = true;
#pragma unroll
  for (int l = 0; l < 3; ++l) {
    if (inside[l]) continue;
    if (in_a) n = clip_poly(xa, ya, n, la[l], lb[l], lc[l], xb, yb);
    else n = clip_poly(xb, yb, n, la[l], lb[l], lc[l], xa, ya);
    in_a = !in_a;
    if (n < 3) return T(0);
  }
  const Buf x = in_a ? xa : xb;
  const Buf y = in_a ? ya : yb;
  // twice the area and six times the first moments, relative to vertex 0 (a
  // fan of triangles), so that a thin piece keeps its relative accuracy (the
  // square is counter-clockwise; clipping keeps it)
  T A = T(0), Mx = T(0), My = T(0);
  for (int i = 1; i + 1 < n; ++i) {
    const T ux = x[i] - x[0], uy = y[i] - y[0], vx = x[i + 1] - x[0], vy = y[i + 1] - y[0];
    const T cr = ux * vy - vx * uy;
    A += cr;
    Mx += (ux + vx) * cr;
    My += (uy + vy) * cr;
  }
  // the line's integral: its value at vertex 0 times the area plus the moments
  const T d0 = c0 + a0 * x[0] + b0 * y[0];
  const T v = d0 * (A / T(2)) + a0 * (Mx / T(6)) + b0 * (My / T(6));
  return v > T(0) ? v : T(0);
}

// Narrow [lo, hi] to the u where p + q u >= 0 (iq = 1 / q).
__device__ __forceinline__ void keep_from(float p, float q, float iq, float& lo, float& hi) {
  const float root = -p * iq;
  if (q > 0.f) lo = fmaxf(lo, root);
  if (q < 0.f) hi = fminf(hi, root);
  if (q == 0.f && p < 0.f) hi = -1.f;
}

// Where the line a x + b y + c = 0 crosses the unit square's boundary: its signs
// at the corners, of which rounding cannot make more than two neighbours differ,
// and its root on each side. The sides' parts and the line's own part within the
// square both come from these, so that they close whatever the rounding (a line
// within it of a side, and parallel, crosses either two sides or none).
struct Crossing {
  bool s00, s10, s01, s11;   // >= 0 at (0, 0), (1, 0), (0, 1), (1, 1)
  float ub, ut, ul, ur;      // roots on the bottom and top (x), left and right (y)
};

__device__ __forceinline__ Crossing cross_square(float a, float b, float c) {
  const float ia = __fdividef(1.0f, a), ib = __fdividef(1.0f, b), v10 = c + a, v01 = c + b;
  return {c >= 0.f, v10 >= 0.f, v01 >= 0.f, v10 + b >= 0.f,
          __saturatef(-c * ia), __saturatef(-v01 * ia), __saturatef(-c * ib), __saturatef(-v10 * ib)};
}

// The part of [0, 1] on a side where the line is >= 0, from its signs at the ends
// and its root.
__device__ __forceinline__ void keep_side(bool s0, bool s1, float u, float& lo, float& hi) {
  lo = s0 ? lo : fmaxf(lo, u);
  hi = s1 ? hi : fminf(hi, u);
}

// A sector's integral over its part of the unit square is a sixth of the sum,
// over the stretches of the part's boundary, of w (h0 + h1 + hq): h0 and h1 the
// hull line's function h at the stretch's ends, hq its value at a point Q, and w
// the stretch's length times its line's distance from Q, positive where Q lies
// inside (the divergence theorem for h (p - Q)). This is that term of a ray from
// the apex (Ax, Ay) to the hull vertex (Vx, Vy), in direction sgn (b, -a).
__device__ __forceinline__ float ray_term(float a, float b, float c, float sgn, const Crossing& k, float Ax, float Ay,
                                          float Vx, float Vy, float Qx, float Qy, float ha, float hb, float hc, float hq) {
  const bool cb = k.s00 != k.s10, ct = k.s01 != k.s11, cl = k.s00 != k.s01, cr = k.s10 != k.s11;
  // (two crossings or none)
  const float x1 = cb ? k.ub : ct ? k.ut : 0.f, y1 = cb ? 0.f : ct ? 1.f : k.ul;
  const float x2 = cr ? 1.f : cl ? 0.f : k.ut, y2 = cr ? k.ur : cl ? k.ul : 1.f;
  const float dx = sgn * b, dy = -sgn * a, in = __fdividef(1.0f, fmaf(a, a, b * b));
  const float l = fmaf(x2 - x1, dx, (y2 - y1) * dy) * in;
  const float x0 = l < 0.f ? x2 : x1, y0 = l < 0.f ? y2 : y1;
  const float t0 = fmaxf(fmaf(Ax - x0, dx, (Ay - y0) * dy) * in, 0.f);
  const float t1 = fminf(fmaf(Vx - x0, dx, (Vy - y0) * dy) * in, fabsf(l));
  const float h = fmaf(ha, x0, fmaf(hb, y0, hc)), hs = fmaf(ha, dx, hb * dy);
  const float w = fmaf(a, Qx, fmaf(b, Qy, c)) * (t1 - t0);
  return (cb || ct || cl || cr) && t1 > t0 ? w * (fmaf(t0 + t1, hs, 2.0f * h) + hq) : 0.f;
}

// Integral of the hull line's function h over the part of the unit square in
// its sector: h, z, o >= 0, as coefficient triples, o the line of the ray from
// the apex (Ax, Ay) through the vertex (Ox, Oy), z minus that of the ray through
// (Zx, Zy); all relative to the square.
//
// Taken around the part (see ray_term): with Q on the hull line where that cuts
// the square, its stretch adds nothing; left are the rays' stretches and the
// square's sides. A term's rounding is that of a vertex's place times h, as for a
// polygon's, and all lanes take one path (clipping the square line by line into
// vertex lists took about 800 instructions at 15 of 32 lanes: 123 ms of a frame
// against 14). An integral in the coordinates (z, h), which needs no second ray,
// divides by the sine of their angle: 3e-6 of a pixel next to long flat sectors.
__device__ __forceinline__ float sector_part(float ha, float hb, float hc, float za, float zb, float zc, float oa, float ob,
                                             float oc, float Ax, float Ay, float Zx, float Zy, float Ox, float Oy) {
  const Crossing kz = cross_square(za, zb, zc), ko = cross_square(oa, ob, oc);
  // Q: the foot of the square's centre on the hull line, or the corner nearest to it
  const float least = hc + fminf(ha, 0.f) + fminf(hb, 0.f), hq = fmaxf(least, 0.f);
  const float back = __fdividef(fmaf(0.5f, ha + hb, hc), fmaf(ha, ha, hb * hb));
  const float Qx = least < 0.f ? fmaf(-ha, back, 0.5f) : ha < 0.f ? 1.f : 0.f;
  const float Qy = least < 0.f ? fmaf(-hb, back, 0.5f) : hb < 0.f ? 1.f : 0.f;
  float sum = ray_term(oa, ob, oc, 1.0f, ko, Ax, Ay, Ox, Oy, Qx, Qy, ha, hb, hc, hq) +
              ray_term(za, zb, zc, -1.0f, kz, Ax, Ay, Zx, Zy, Qx, Qy, ha, hb, hc, hq);
  const float iha = __fdividef(1.0f, ha), ihb = __fdividef(1.0f, hb);
  // the square's sides
  auto side = [&](float p, float q, float iq, bool o0, bool o1, float uo, bool z0, bool z1, float uz, float dist) {
    float lo = 0.f, hi = 1.f;
    keep_side(o0, o1, uo, lo, hi);
    keep_side(z0, z1, uz, lo, hi);
    keep_from(p, q, iq, lo, hi);
    if (hi > lo) sum = fmaf(dist * (hi - lo), fmaf(lo + hi, q, 2.0f * p) + hq, sum);
  };
  side(hc, ha, iha, ko.s00, ko.s10, ko.ub, kz.s00, kz.s10, kz.ub, Qy);
  side(hc + hb, ha, iha, ko.s01, ko.s11, ko.ut, kz.s01, kz.s11, kz.ut, 1.0f - Qy);
  side(hc, hb, ihb, ko.s00, ko.s01, ko.ul, kz.s00, kz.s01, kz.ul, Qx);
  side(hc + ha, hb, ihb, ko.s10, ko.s11, ko.ur, kz.s10, kz.s11, kz.ur, 1.0f - Qx);
  // (1 / 6 in two parts: in FP32 alone it is 3e-8 too large, which shows in the
  // frame's mass)
  return fmaf(sum, 0.16666667f, sum * -4.967054e-9f);
}

// Mean column density over pixel (ox, oy) (offsets from the anchor) of one
// tetrahedron, in accumulator units, clipped in FP64: for thin hulls and
// sectors, out of line (rare: it keeps the hot loop small).
__device__ __noinline__ float pixel_mean_f64(const AreaTet& t, int ox, int oy) {
  double xa[8], ya[8], xb[8], yb[8], r[4][3];
  double v = 0.0;
  for (int e = 0; e < t.n; ++e)
    for (int q = 0; q < 3; ++q)
      r[e][q] = q < 2 ? (double)t.ray_h[q][e] + (double)t.ray_l[q][e] : line_f64(t.ray_h, t.ray_l, e, (double)ox, (double)oy);
  for (int e = 0; e < t.n; ++e) {
    const int f = e + 1 == t.n ? 0 : e + 1;
    const double ha = (double)t.hull_h[0][e] + (double)t.hull_l[0][e], hb = (double)t.hull_h[1][e] + (double)t.hull_l[1][e];
    const double hc = line_f64(t.hull_h, t.hull_l, e, (double)ox, (double)oy);
    if (hc + fmax(ha, 0.0) + fmax(hb, 0.0) <= 0.0) return 0.f;
    v += (double)t.k[e] * sector_integral<double, double*>(ha, hb, hc, r[e][0], r[e][1], r[e][2], -r[f][0], -r[f][1], -r[f][2],
                                                           xa, ya, xb, yb);
  }
  return (float)v;
}

// Add units, or a value of any size, to pixel (px, py) (unwrapped) of the image.
__device__ __forceinline__ unsigned long long* area_cell(const AreaArgs& a, const FrameDev& F, int px, int py) {
  const int W = F.W, H = F.H;
  if (F.wrap) {
    if (px < 0 || px >= W) px = ((px % W) + W) % W;
    if (py < 0 || py >= H) py = ((py % H) + H) % H;
  }
  if (!LT_IN_BOUNDS(px >= 0 && px < W && py >= 0 && py < H, &a.ctr->errors)) return a.acc;
  return a.acc + ((long long)py * W + px);
}

__device__ __forceinline__ void area_add_units(const AreaArgs& a, const FrameDev& F, int px, int py, unsigned long long u) {
  if (!u) return;
  const unsigned long long old = atomicAdd(area_cell(a, F, px, py), u);
  if (old > ~0ull - u) {
    atomicOr(&a.ctr->errors, kErrRange);
    atomicAdd(&a.ctr->range_overflow, 1ull);
  }
}

__device__ __noinline__ void area_add(const AreaArgs& a, const FrameDev& F, int px, int py, float v) {
  accum_fixed(area_cell(a, F, px, py), v, a.ctr);
}

__device__ __forceinline__ void clear_edges(AreaTet& t, int n) {
  for (int e = n; e < 4; ++e) {
    for (int q = 0; q < 3; ++q) t.hull_h[q][e] = t.hull_l[q][e] = t.ray_h[q][e] = t.ray_l[q][e] = 0.f;
    t.k[e] = t.kr[e] = 0.f;
  }
}

// The rays' kr from the sectors' slopes: along ray e the functions of sectors
// e - 1 and e agree, so their difference is a multiple of the ray's line, taken
// from the larger component of its gradient.
__device__ __forceinline__ void ray_slopes(AreaTet& t) {
  t.flat = 0;
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    if (e >= t.n) break;
    if (!(t.k[e] > 0.f)) t.flat = 1;
    const int b = e == 0 ? t.n - 1 : e - 1;
    const int q = fabsf(t.ray_h[0][e]) >= fabsf(t.ray_h[1][e]) ? 0 : 1;
    const float d = fmaf(t.k[b], t.hull_h[q][b], -t.k[e] * t.hull_h[q][e]);
    t.kr[e] = __fdividef(d, t.ray_h[q][e]);
  }
}

// Integral over the unit square of max(0, a x + b y + c). By reflection a >= b
// >= 0: with m the value at the far corner the positive part is a triangle (m <=
// b), a quadrilateral (m <= a), or all but a triangle; no form subtracts nearly
// equal numbers.
__device__ __forceinline__ float half_square(float a, float b, float c) {
  const float lo = c + fminf(a, 0.f) + fminf(b, 0.f), ua = fabsf(a), ub = fabsf(b);
  const float p = fmaxf(ua, ub), q = fminf(ua, ub);
  const float m = lo + p + q;  // far corner's value; lo is the near corner's
  const float i6p = __fdividef(1.0f, 6.0f * p);
  const float r = fminf(m, -lo);  // the triangle's height: of the positive part, or of what is cut off
  const float tri = r > 0.f ? r * (r * i6p) * __fdividef(r, q) : 0.f;
  const float quad = fmaf(3.0f * m, m - q, q * q) * i6p;
  const float all = fmaf(0.5f, a + b, c);
  return m <= 0.f ? 0.f : m <= q ? tri : m <= p ? quad : all + (lo < 0.f ? tri : 0.f);
}

// The rectangle of pixels from the hull's bounds (offsets from the anchor, in
// pixels); false when it is empty.
__device__ __forceinline__ bool set_rectangle(const AreaArgs& a, const FrameDev& F, double xmn, double xmx, double ymn,
                                              double ymx, AreaTet& t) {
  int x0 = (int)fmax(xmn, -2.0e9), x1 = (int)fmin(xmx, 2.0e9);
  int y0 = (int)fmax(ymn, -2.0e9), y1 = (int)fmin(ymx, 2.0e9);
  if (!F.wrap) {
    x0 = max(x0, 0); x1 = min(x1, F.W - 1);
    y0 = max(y0, 0); y1 = min(y1, F.H - 1);
  } else {
    // at most a few periods per axis (a tetrahedron spans less than one)
    x1 = min(x1, x0 + 4 * F.W);
    y1 = min(y1, y0 + 4 * F.H);
  }
  if (x0 > x1 || y0 > y1) return false;
  if ((long long)(x1 - x0 + 1) * (y1 - y0 + 1) > 0x7fffffffLL) {
    // more than 2^31 pixels (a window zoomed far into one tetrahedron): the
    // walk's 32-bit pixel index cannot hold it
    atomicOr(&a.ctr->errors, kErrRange);
    return false;
  }
  t.x0 = x0;
  t.y0 = y0;
  t.wx = x1 - x0 + 1;
  t.inv_wx = 1.0f / (float)t.wx;
  t.np = t.wx * (y1 - y0 + 1);
  const float far = fmaxf(fmaxf(fabsf((float)(x0 - t.ax)), fabsf((float)(x1 - t.ax))),
                          fmaxf(fabsf((float)(y0 - t.ay)), fabsf((float)(y1 - t.ay))));
  float c = 0.f;
  for (int e = 0; e < 4; ++e) c = fmaxf(c, fabsf(t.hull_h[2][e]));
  t.margin = (far + c + 2.0f) * 1.0e-6f;  // eight roundings of 2^-24 and room
  return true;
}

// The whole setup of a lane's tetrahedron in FP64; false when it covers no area.
__device__ __noinline__ bool setup_f64(const AreaArgs& a, const FrameDev& F, int i, int j, int k, int s, AreaTet& t) {
  bool ok = true;
  TetF64 tf;
  tet_f64(a.L, (long long)F.snapshot * a.L.n_particles, i, j, k, s, ok, tf);
  if (!ok || tf.V == 0.0) return false;
  const double hl = (double)a.L.box / a.L.N;
  const double base[3] = {i * hl, j * hl, k * hl};
  double P[4][2], eps[2] = {0.0, 0.0};
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    double w[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) w[q] = base[q] + tf.v[c][q];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const double* axis = q == 0 ? F.rd : F.ud;
      P[c][q] = (axis[0] * w[0] + axis[1] * w[1] + axis[2] * w[2] - F.lod[q]) / F.pxd[q];
      // its rounding: a few 2^-53 of the terms
      const double size = fabs(axis[0] * w[0]) + fabs(axis[1] * w[1]) + fabs(axis[2] * w[2]) + fabs(F.lod[q]);
      eps[q] = fmax(eps[q], 0x1p-50 * size / F.pxd[q]);
    }
  }
  // the apex and the hull, counter-clockwise, by the signed areas c_i = (-1)^i
  // orient(the others), which sum to zero: a lone sign marks the vertex inside the
  // triangle of the others, two of each the diagonals. An area of rounding's size
  // counts as none: the vertex of the lone sign then lies on a hull edge, or, with
  // two such areas, on a hull vertex (lattices seen along an axis at which they
  // are at rest), and the triangles beside it have no area.
  double D[3][2], dmax[2] = {0.0, 0.0};
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      D[c][q] = P[c + 1][q] - P[0][q];
      dmax[q] = fmax(dmax[q], fabs(D[c][q]));
    }
  const double o12 = D[0][0] * D[1][1] - D[0][1] * D[1][0], o13 = D[0][0] * D[2][1] - D[0][1] * D[2][0];
  const double o23 = D[1][0] * D[2][1] - D[1][1] * D[2][0];
  const double cc[4] = {(o12 + o23) - o13, -o23, o13, -o12};
  double none = 8.0 * (eps[0] * dmax[1] + eps[1] * dmax[0]);
  int pos = 0, neg = 0;
  for (int c = 0; c < 4; ++c) {
    if (cc[c] > none) pos |= 1 << c;
    if (cc[c] < -none) neg |= 1 << c;
  }
  if (pos == 0 || neg == 0) {  // a whole hull of that size: by the signs as they are
    none = 0.0;
    pos = neg = 0;
    for (int c = 0; c < 4; ++c) {
      if (cc[c] > 0.0) pos |= 1 << c;
      if (cc[c] < 0.0) neg |= 1 << c;
    }
    if (pos == 0 || neg == 0) return false;
  }
  double Ax, Ay, Hx[4], Hy[4];
  int n, ord[4];
  if (__popc(pos) == 2 && __popc(neg) == 2) {
    // the diagonals are (0, d) and (u, w), vertex 0 and d as far from the other as
    // their triangles' areas
    const int same = pos & 1 ? pos : neg;
    const int d = (same >> 1) & 1 ? 1 : (same >> 2) & 1 ? 2 : 3;
    int u = d == 1 ? 2 : 1, w = 6 - d - u;
    if (orient(P[u][0], P[u][1], P[w][0], P[w][1], P[0][0], P[0][1]) < 0.0) { const int x = u; u = w; w = x; }
    const double tt = cc[d] / (cc[d] + cc[0]);
    Ax = P[0][0] + tt * (P[d][0] - P[0][0]);
    Ay = P[0][1] + tt * (P[d][1] - P[0][1]);
    ord[0] = 0; ord[1] = u; ord[2] = d; ord[3] = w;
    n = 4;
  } else {
    const int c = 31 - __clz(__popc(pos) == 1 ? pos : neg);
    const int p = (c + 1) & 3, q = (c + 2) & 3, r = (c + 3) & 3;
    const bool ccw = orient(P[p][0], P[p][1], P[q][0], P[q][1], P[r][0], P[r][1]) > 0.0;
    Ax = P[c][0];
    Ay = P[c][1];
    ord[0] = p; ord[1] = ccw ? q : r; ord[2] = ccw ? r : q; ord[3] = p;
    n = 3;
  }
  for (int e = 0; e < 4; ++e) {
    Hx[e] = P[ord[e]][0];
    Hy[e] = P[ord[e]][1];
  }
  // twice the hull's area: the two triangles beside a diagonal, or the one around
  // the apex
  const double area2 = 0.5 * (fabs(cc[0]) + fabs(cc[1]) + fabs(cc[2]) + fabs(cc[3]));
  double emax = 0.0;
  for (int e = 0; e < n; ++e) {
    const int f = e + 1 == n ? 0 : e + 1;
    emax = fmax(emax, hypot(Hx[f] - Hx[e], Hy[f] - Hy[e]));
  }
  // column density at the apex: 3 m / (hull area in world units)
  const double h = 3.0 * a.m_tet / (0.5 * area2 * F.pxd[0] * F.pxd[1]);
  t.ax = (int)fmin(fmax(floor(Ax), -1.0e9), 1.0e9);
  t.ay = (int)fmin(fmax(floor(Ay), -1.0e9), 1.0e9);
  const double qx = Ax - t.ax, qy = Ay - t.ay;
  t.qx = (float)qx;
  t.qy = (float)qy;
  double xmn = Hx[0], xmx = Hx[0], ymn = Hy[0], ymx = Hy[0];
  bool thin_sector = false;
  for (int e = 0; e < n; ++e) {
    const int f = e + 1 == n ? 0 : e + 1;
    make_line(Hx[e] - t.ax, Hy[e] - t.ay, Hx[f] - Hx[e], Hy[f] - Hy[e], t.hull_h, t.hull_l, e);
    make_line(qx, qy, Hx[e] - Ax, Hy[e] - Ay, t.ray_h, t.ray_l, e);
    const float2 vx = split_ff(Hx[e] - t.ax), vy = split_ff(Hy[e] - t.ay);
    t.vx_h[e] = vx.x; t.vx_l[e] = vx.y;
    t.vy_h[e] = vy.x; t.vy_l[e] = vy.y;
    const double len = fabs(Hx[f] - Hx[e]) + fabs(Hy[f] - Hy[e]);
    double dA = line_f64(t.hull_h, t.hull_l, e, qx, qy);
    if (dA * len <= none) dA = 0.0;  // twice the area of the apex's triangle
    t.k[e] = dA > 0.0 ? (float)(h / dA * a.inv_unit) : 0.0f;
    // an apex next to a hull edge: a long thin face whose FP32 clip would lose
    // its relative accuracy while k_e grows as 1 / dA
    thin_sector = thin_sector || (dA > 0.0 && dA < kThinSector);
    xmn = fmin(xmn, Hx[e]); xmx = fmax(xmx, Hx[e]);
    ymn = fmin(ymn, Hy[e]); ymx = fmax(ymx, Hy[e]);
  }
  clear_edges(t, n);
  t.n = n;
  ray_slopes(t);
  t.thin = 0.5 * area2 < kThinHull * emax || thin_sector;
  return set_rectangle(a, F, floor(xmn), floor(xmx), floor(ymn), floor(ymx), t);
}

// The setup in float-float, with all coordinates relative to a pixel near the
// tetrahedron: 1 done, 0 nothing to draw, 2 when FP64 has to take it.
__device__ __forceinline__ int setup_ff(const AreaArgs& a, const FrameDev& F, int i, int j, int k, int s, AreaTet& t) {
  bool ok = true;
  ff v[4][3];
  tet_ff(a.L, a.h, (long long)F.snapshot * a.L.n_particles, i, j, k, s, ok, v);
  if (!ok) return 0;
  // pixel coordinates (a pixel p covers [p, p + 1]) less the anchor's whole part
  float base[2];
  ff P[4][2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    float hi, lo;
    anchor_affine(F, q, i, j, k, hi, lo);
    base[q] = floorf(hi);
    const ff anchor = ff_two_sum(__fsub_rn(hi, base[q]), lo) + 0.5f;  // (the frame's own have centres at whole numbers)
#pragma unroll
    for (int c = 0; c < 4; ++c) P[c][q] = ((a.axis[q][0] * v[c][0] + a.axis[q][1] * v[c][1]) + a.axis[q][2] * v[c][2]) + anchor;
  }
  if (!(fabsf(base[0]) < 1.0e9f && fabsf(base[1]) < 1.0e9f)) return 2;
  // signed areas: c_i = (-1)^i orient(the others) sum to zero; a lone sign marks
  // the vertex inside the triangle of the others, two of each the diagonals
  ff d[3][2];
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int q = 0; q < 2; ++q) d[c][q] = P[c + 1][q] - P[0][q];
  auto cross = [](const ff (&u)[2], const ff (&w)[2]) { return u[0] * w[1] - u[1] * w[0]; };
  const ff o12 = cross(d[0], d[1]), o13 = cross(d[0], d[2]), o23 = cross(d[1], d[2]);
  const ff o123 = (o12 + o23) - o13;  // orient(1, 2, 3)
  // orient of the triangle opposite vertex 0, 1, 2, 3, with the sign of its place
  const ff cc[4] = {o123, -o23, o13, -o12};
  float S = 0.f, least = 3.0e38f;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    S += fabsf(cc[c].h);
    least = fminf(least, fabsf(cc[c].h));
  }
  // too near to degenerate for the 2^-40 or so that the areas are good to
  if (!(least > S * 1.0e-6f) || !(S > 1e-20f)) return 2;
  int pos = 0, mask = 0;
#pragma unroll
  for (int c = 0; c < 4; ++c)
    if (cc[c].h > 0.f) { ++pos; mask |= 1 << c; }
  int order[4], n;
  int inner = -1;
  ff Ax, Ay;
  auto pick = [&](int c, int q) {
    return c == 0 ? P[0][q] : c == 1 ? P[1][q] : c == 2 ? P[2][q] : P[3][q];
  };
  if (pos == 2) {
    // the diagonals are (0, p) and (u, w); counter-clockwise 0, u, p, w
    const int same = (mask & 1) ? mask : mask ^ 15;  // the signs of vertex 0's kind
    const int p = (same >> 1) & 1 ? 1 : (same >> 2) & 1 ? 2 : 3;
    int u = p == 1 ? 2 : 1, w = 6 - p - u;
    const ff ux = pick(u, 0), uy = pick(u, 1), wx = pick(w, 0), wy = pick(w, 1);
    const ff px = pick(p, 0), py = pick(p, 1);
    // the crossing: vertex 0 and p on either side of the line u w
    const ff ex = wx - ux, ey = wy - uy;
    const ff s0 = ex * (P[0][1] - uy) - ey * (P[0][0] - ux), sp = ex * (py - uy) - ey * (px - ux);
    const ff den = s0 - sp;
    if (!(fabsf(den.h) > 0.f)) return 2;
    const ff tt = s0 / den;
    Ax = P[0][0] + tt * (px - P[0][0]);
    Ay = P[0][1] + tt * (py - P[0][1]);
    // u on the right of 0 -> p, which is where 0 -> u -> w turns left
    if (s0.h < 0.f) { const int x = u; u = w; w = x; }
    order[0] = 0; order[1] = u; order[2] = p; order[3] = w;
    n = 4;
  } else {
    const int lone = pos == 1 ? mask : mask ^ 15;
    inner = 31 - __clz(lone);
    order[0] = inner == 0 ? 1 : 0;
    order[1] = inner <= 1 ? 2 : 1;
    order[2] = inner <= 2 ? 3 : 2;
    order[3] = order[0];
    // orient(order) = (-1)^inner c_inner
    const ff ci = inner == 0 ? cc[0] : inner == 1 ? cc[1] : inner == 2 ? cc[2] : cc[3];
    if ((ci.h > 0.f) == ((inner & 1) != 0)) { const int x = order[1]; order[1] = order[2]; order[2] = x; }
    Ax = pick(inner, 0);
    Ay = pick(inner, 1);
    n = 3;
  }
  ff Hx[4], Hy[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    Hx[e] = pick(order[e], 0);
    Hy[e] = pick(order[e], 1);
  }
  // twice the hull's area from vertex 0 of the hull
  ff area2 = (Hx[1] - Hx[0]) * (Hy[2] - Hy[0]) - (Hy[1] - Hy[0]) * (Hx[2] - Hx[0]);
  if (n == 4) area2 = area2 + ((Hx[2] - Hx[0]) * (Hy[3] - Hy[0]) - (Hy[2] - Hy[0]) * (Hx[3] - Hx[0]));
  if (!(area2.h > 0.f)) return 2;
  // column density at the apex: 3 m / (hull area), in accumulator units
  const ff h = a.apex / area2;
  const float bx = floorf(Ax.h), by = floorf(Ay.h);
  t.ax = (int)base[0] + (int)bx;
  t.ay = (int)base[1] + (int)by;
  const ff qx = Ax + (-bx), qy = Ay + (-by);
  t.qx = qx.h;
  t.qy = qy.h;
  float emax = 0.f, xmn = 3.0e38f, xmx = -3.0e38f, ymn = 3.0e38f, ymx = -3.0e38f;
  bool thin_sector = false;
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    if (e >= n) break;
    const int f = e + 1 == n ? 0 : (e + 1) & 3;
    const ff fx = f == 0 ? Hx[0] : Hx[(e + 1) & 3], fy = f == 0 ? Hy[0] : Hy[(e + 1) & 3];
    const ff ex = fx - Hx[e], ey = fy - Hy[e];
    const ff vx = Hx[e] + (-bx), vy = Hy[e] + (-by);
    t.vx_h[e] = vx.h; t.vx_l[e] = vx.l;
    t.vy_h[e] = vy.h; t.vy_l[e] = vy.l;
    make_line(vx, vy, ex, ey, t.hull_h, t.hull_l, e);
    make_line(qx, qy, Hx[e] - Ax, Hy[e] - Ay, t.ray_h, t.ray_l, e);
    const ff dA = (ff{t.hull_h[0][e], t.hull_l[0][e]} * qx + ff{t.hull_h[1][e], t.hull_l[1][e]} * qy) +
                  ff{t.hull_h[2][e], t.hull_l[2][e]};
    const ff ke = h / dA;
    t.k[e] = dA.h > 0.f ? __fadd_rn(ke.h, ke.l) : 0.f;
    // an apex next to a hull edge: a long thin face whose FP32 clip would lose
    // its relative accuracy while k_e grows as 1 / dA
    thin_sector = thin_sector || (dA.h > 0.f && dA.h < (float)kThinSector);
    emax = fmaxf(emax, sqrtf(fmaf(ex.h, ex.h, ey.h * ey.h)));
    // (an ulp outwards where the low part points there)
    xmn = fminf(xmn, floorf(Hx[e].h + fminf(Hx[e].l, 0.f) * 2.f));
    xmx = fmaxf(xmx, floorf(Hx[e].h + fmaxf(Hx[e].l, 0.f) * 2.f));
    ymn = fminf(ymn, floorf(Hy[e].h + fminf(Hy[e].l, 0.f) * 2.f));
    ymx = fmaxf(ymx, floorf(Hy[e].h + fmaxf(Hy[e].l, 0.f) * 2.f));
  }
  clear_edges(t, n);
  t.n = n;
  ray_slopes(t);
  t.thin = 0.5f * area2.h < (float)kThinHull * emax || thin_sector;
  // (whole numbers, each within FP32's exact range of the anchor's pixel)
  if (!(fabsf(xmn) < 8.0e6f && fabsf(xmx) < 8.0e6f && fabsf(ymn) < 8.0e6f && fabsf(ymx) < 8.0e6f)) return 2;
  return set_rectangle(a, F, (double)((int)base[0] + (int)xmn), (double)((int)base[0] + (int)xmx),
                       (double)((int)base[1] + (int)ymn), (double)((int)base[1] + (int)ymx), t) ? 1 : 0;
}

// A warp's share of shared memory.
struct AreaWarp {
  AreaTet tets[32];
  int2 runs[32];             // tetrahedra with pixels: their slot, where their pixels start
  int2 near[64];             // pixels that stage 1 kept: slot, index in the rectangle
  float line[8][32];         // stage 2's lines at the pixel's corner: four of the hull, four rays
  int slot[32];              // stage 2's tetrahedra
  unsigned sum[2][32];       // stage 2's pixels: sectors clipped in stage 3, in 64ths of a unit
  unsigned char job[128];    // pixels of stage 2 << 2 | sector
};

// Sums past this many units go to the image by themselves.
constexpr float kDirect = 1.0e12f;
// A pixel's sectors are summed in 64ths of a unit: rounded to a unit only once
// (16ths: 0.8% more rounding where a thousand tetrahedra meet in a pixel).
constexpr int kPartBits = 6;
constexpr float kParts = 64.0f;

__global__ void __launch_bounds__(kAreaThreads, 4) k_area(AreaArgs a) {
  extern __shared__ __align__(16) float area_smem[];
  AreaWarp& S = reinterpret_cast<AreaWarp*>(area_smem)[threadIdx.x >> 5];
  const FrameDev& F = *a.frame;
  const long long ntet = 6LL * a.L.n_particles;
  const int lane = threadIdx.x & 31;
  const unsigned FULL = 0xffffffffu, lt_mask = (1u << lane) - 1u, le_mask = (2u << lane) - 1u;
  const long long warps = (long long)gridDim.x * (kAreaThreads / 32);
  const long long wid = (long long)blockIdx.x * (kAreaThreads / 32) + (threadIdx.x >> 5);

  // ---- stages 2 and 3 for the last n (at most 32) of the pixels kept
  auto batch = [&](int first, int n) {
    float whole = 0.f;
    int px = 0, py = 0, njobs = 0;
    unsigned clip = 0u;
    S.sum[0][lane] = S.sum[1][lane] = 0u;
    if (lane < n) {
      const int2 q = S.near[first + lane];
      const AreaTet& t = S.tets[q.x];
      int ry = (int)(((float)q.y + 0.5f) * t.inv_wx);
      if (t.np > 1 << 20) ry = q.y / t.wx;
      px = t.x0 + (q.y - ry * t.wx);
      py = t.y0 + ry;
      const int ox = px - t.ax, oy = py - t.ay;
      S.slot[lane] = q.x;
      if (t.thin) {
        whole = pixel_mean_f64(t, ox, oy);
      } else {
        float hc[4];
        bool outside = false;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          hc[e] = line_ff(t.hull_h, t.hull_l, e, (float)ox, (float)oy);
          const float hi = hc[e] + fmaxf(t.hull_h[0][e], 0.f) + fmaxf(t.hull_h[1][e], 0.f);
          outside = outside || (e < t.n && hi <= 0.f);
        }
        if (!outside) {
          float rlo[4], rhi[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float rc = line_ff(t.ray_h, t.ray_l, e, (float)ox, (float)oy);
            const float ra = t.ray_h[0][e], rb = t.ray_h[1][e];
            // smallest and largest value over the square's corners
            rlo[e] = rc + fminf(ra, 0.f) + fminf(rb, 0.f);
            rhi[e] = rc + fmaxf(ra, 0.f) + fmaxf(rb, 0.f);
            S.line[e][lane] = hc[e];
            S.line[4 + e][lane] = rc;
          }
          // sectors (between ray e and the next, within hull line e) that reach
          // the square, and those whose hull line cuts it
          unsigned reach = 0u, cut = 0u;
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const bool wraps = e + 1 == t.n;
            const float nlo = wraps ? rlo[0] : rlo[(e + 1) & 3];
            if (t.k[e] > 0.f && rhi[e] > 0.f && nlo < 0.f) reach |= 1u << e;
            if (hc[e] + fminf(t.hull_h[0][e], 0.f) + fminf(t.hull_h[1][e], 0.f) < 0.f) cut |= 1u << e;
          }
          cut &= reach;
          // sector index and the one before it, of the reached ones
          // (where a sector has no area, at an apex on the hull, a neighbour's
          // ray is the hull's edge: every sector is clipped)
          const int count = t.flat ? 5 : __popc(reach), first_e = __ffs(reach) - 1;
          if (reach == 0u) {
          } else if (count == 1) {
            // the square is inside one sector
            const int e = first_e;
            whole = t.k[e] * half_square(t.hull_h[0][e], t.hull_h[1][e], S.line[e][lane]);
          } else if (count == 2 && cut == 0u) {
            // inside the hull, over one ray: the smaller of the two sectors'
            // functions is that of the larger side less kr times the other side's
            // part of the ray's line
            const int last_e = 31 - __clz(reach);
            const int f = last_e == first_e + 1 ? last_e : first_e;   // the ray between the sectors
            const int b = f == last_e ? first_e : last_e;             // sector b before it, f after it
            const float rc = S.line[4 + f][lane], ra = t.ray_h[0][f], rb = t.ray_h[1][f];
            const bool after = fmaf(0.5f, ra + rb, rc) > 0.f;  // the centre lies in sector f
            const int e = after ? f : b;
            const float all = t.k[e] * (fmaf(0.5f, t.hull_h[0][e] + t.hull_h[1][e], S.line[e][lane]));
            const float part = t.kr[f] * (after ? half_square(-ra, -rb, -rc) : half_square(ra, rb, rc));
            whole = all - part;
            // (a part as large as the result would carry its rounding over)
            if (!(part <= 0.5f * all)) {
              whole = 0.f;
              clip = reach;
            }
          } else {
            clip = reach;
          }
        }
      }
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const unsigned m = __ballot_sync(FULL, (clip >> e) & 1u);
      if ((clip >> e) & 1u) S.job[njobs + __popc(m & lt_mask)] = (unsigned char)(lane << 2 | e);
      njobs += __popc(m);
    }
    __syncwarp();
    for (int jb = 0; jb < njobs; jb += 32) {
      if (jb + lane < njobs) {
        const int o = S.job[jb + lane] >> 2, e = S.job[jb + lane] & 3;
        const AreaTet& t = S.tets[S.slot[o]];
        const int f = e + 1 == t.n ? 0 : e + 1;
        const int2 q = S.near[first + o];
        int ry = (int)(((float)q.y + 0.5f) * t.inv_wx);
        if (t.np > 1 << 20) ry = q.y / t.wx;
        const float ox = (float)(t.x0 + (q.y - ry * t.wx) - t.ax), oy = (float)(t.y0 + ry - t.ay);
        const float ha = t.hull_h[0][e], hb = t.hull_h[1][e];
        const float ra = t.ray_h[0][e], rb = t.ray_h[1][e], rc = S.line[4 + e][o];
        const float ga = -t.ray_h[0][f], gb = -t.ray_h[1][f], gc = -S.line[4 + f][o];
        const float in = sector_part(ha, hb, S.line[e][o], ga, gb, gc, ra, rb, rc, t.qx - ox, t.qy - oy,
                                     (t.vx_h[f] - ox) + t.vx_l[f], (t.vy_h[f] - oy) + t.vy_l[f],
                                     (t.vx_h[e] - ox) + t.vx_l[e], (t.vy_h[e] - oy) + t.vy_l[e]);
        const float v = t.k[e] * in;
        if (v < 3.3e7f) {
          // (rounding can leave a part next to nothing on either side of zero:
          // signed, so that the parts' errors do not add up)
          const int i = __float2int_rn(kParts * fmaxf(v, -3.3e7f));
          const unsigned u = (unsigned)i;
          const unsigned hi = (i < 0 ? ~0u : 0u) + (atomicAdd(&S.sum[0][o], u) > ~u ? 1u : 0u);
          if (hi) atomicAdd(&S.sum[1][o], hi);
        } else if (v < kDirect) {
          const unsigned long long u = __float2ull_rn(kParts * v);
          const unsigned lo = (unsigned)u;
          const unsigned hi = (unsigned)(u >> 32) + (atomicAdd(&S.sum[0][o], lo) > ~lo ? 1u : 0u);
          if (hi) atomicAdd(&S.sum[1][o], hi);
        } else {
          area_add(a, F, t.x0 + (q.y - ry * t.wx), t.y0 + ry, v);
        }
      }
      __syncwarp();
    }
    if (lane < n) {
      if (whole < kDirect) {
        unsigned long long u = (unsigned long long)max((long long)((unsigned long long)S.sum[1][lane] << 32 | S.sum[0][lane]), 0LL);
        u += whole < 6.6e7f ? (unsigned long long)__float2uint_rn(kParts * whole) : __float2ull_rn(kParts * whole);
        area_add_units(a, F, px, py, (u + 31ull + ((u >> kPartBits) & 1ull)) >> kPartBits);  // (to the nearest, halves to even)
      } else {
        area_add_units(a, F, px, py, (unsigned long long)max((long long)((unsigned long long)S.sum[1][lane] << 32 | S.sum[0][lane]), 0LL) >> kPartBits);
        area_add(a, F, px, py, whole);
      }
    }
    __syncwarp();
  };

  for (long long base = wid * 32; base < ntet; base += warps * 32) {
    // ---- one tetrahedron per lane
    const long long tau = base + lane;
    AreaTet& mine = S.tets[lane];
    bool live = false;
    if (tau < ntet) {
      const long long cube = tau / 6;
      const int s = (int)(tau - 6 * cube);
      if (!tet_degenerate(a.L, F.snapshot, cube, s)) {
        int i, j, k;
        cube_ijk(a.L, cube, i, j, k);
        const int how = a.use_ff ? setup_ff(a, F, i, j, k, s, mine) : 2;
        live = how == 1 || (how == 2 && setup_f64(a, F, i, j, k, s, mine));
      }
    }
    const int np = live ? mine.np : 0;
    const int thin = live && mine.thin ? np : 0;
    // (counted in two halves of 16 bits)
    const unsigned p_lo = __reduce_add_sync(FULL, (unsigned)np & 0xffffu), p_hi = __reduce_add_sync(FULL, (unsigned)np >> 16);
    const unsigned t_lo = __reduce_add_sync(FULL, (unsigned)thin & 0xffffu), t_hi = __reduce_add_sync(FULL, (unsigned)thin >> 16);
    if (lane == 0) {
      const unsigned long long pn = ((unsigned long long)p_hi << 16) + p_lo, tn = ((unsigned long long)t_hi << 16) + t_lo;
      if (pn) atomicAdd(&a.ctr->area_pairs, pn);
      if (tn) atomicAdd(&a.ctr->area_fp64_pairs, tn);
    }
    // ---- stage 1: the rectangles' pixels, at most 2^22 of a tetrahedron at a time
    for (int done = 0; __any_sync(FULL, np > done); done += 1 << 22) {
      const int mine_n = np > done ? min(np - done, 1 << 22) : 0;
      int incl = mine_n;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += y;
      }
      const int total = __shfl_sync(FULL, incl, 31), off = incl - mine_n;
      const unsigned with = __ballot_sync(FULL, mine_n > 0);
      __syncwarp();
      if (mine_n > 0) S.runs[__popc(with & lt_mask)] = make_int2(lane, off);
      __syncwarp();
      int runs_before = 0, kept = 0;
      for (int pb = 0; pb < total; pb += 32) {
        const int rel = off - pb;
        const unsigned starts = __reduce_or_sync(FULL, (mine_n > 0 && rel >= 0 && rel < 32) ? 1u << rel : 0u);
        const int run = runs_before + __popc(starts & le_mask) - 1;
        runs_before += __popc(starts);
        const int2 rs = S.runs[min(max(run, 0), 31)];
        const AreaTet& t = S.tets[rs.x & 31];
        const int p = pb + lane - rs.y + done;
        int ry = (int)(((float)p + 0.5f) * t.inv_wx);
        if (t.np > 1 << 20) ry = p / t.wx;
        const float ox = (float)(t.x0 + (p - ry * t.wx) - t.ax), oy = (float)(t.y0 + ry - t.ay);
        bool keep = pb + lane < total;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float la = t.hull_h[0][e], lb = t.hull_h[1][e];
          const float hi = fmaf(la, ox, fmaf(lb, oy, t.hull_h[2][e])) + fmaxf(la, 0.f) + fmaxf(lb, 0.f);
          keep = keep && (e >= t.n || hi > -t.margin);
        }
        const unsigned km = __ballot_sync(FULL, keep);
        if (keep) S.near[kept + __popc(km & lt_mask)] = make_int2(rs.x, p);
        kept += __popc(km);
        const bool last = pb + 32 >= total;
        while (kept >= 32 || (last && kept > 0)) {
          __syncwarp();
          const int n = min(kept, 32);
          kept -= n;
          batch(kept, n);
        }
      }
      __syncwarp();
    }
    __syncwarp();
  }
}

}  // namespace

cudaError_t launch_area(const Lattice& L, const FrameDev& F, const FrameDev* d_frame, unsigned long long* d_acc, float* d_out,
                        DevCounters* ctr, cudaStream_t s) {
  const long long np = (long long)F.W * F.H;
  cudaError_t e = cudaMemsetAsync(d_acc, 0, sizeof(unsigned long long) * np, s);
  if (e != cudaSuccess) return e;
  AreaArgs a;
  a.L = L;
  a.frame = d_frame;
  a.m_tet = F.m_tet;
  a.inv_unit = 1.0 / F.unit;
  auto split = [](double v) { ff f; f.h = (float)v; f.l = (float)(v - (double)f.h); return f; };
  const double h = (double)L.box / L.N;
  a.h = split(h);
  for (int q = 0; q < 3; ++q) {
    a.axis[0][q] = split(F.rd[q] / F.pxd[0]);
    a.axis[1][q] = split(F.ud[q] / F.pxd[1]);
  }
  const double apex = 6.0 * F.m_tet / (F.pxd[0] * F.pxd[1]) * a.inv_unit;
  a.apex = split(apex);
  // cells, pixels and units whose products and quotients stay in FP32's range
  auto within = [](double v, double lo, double hi) { return v > lo && v < hi; };
  a.use_ff = within(h, 1e-6, 1e4) && within(h / F.pxd[0], 1e-4, 1e6) && within(h / F.pxd[1], 1e-4, 1e6) &&
             within(apex, 1e-6, 1e24);
  a.acc = d_acc;
  a.ctr = ctr;
  const size_t smem = sizeof(AreaWarp) * (kAreaThreads / 32);
  if ((e = cudaFuncSetAttribute(k_area, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess) return e;
  long long blocks = (6LL * L.n_particles + kAreaThreads - 1) / kAreaThreads;
  if (blocks > 152LL * 64) blocks = 152LL * 64;
  k_area<<<(unsigned)(blocks < 1 ? 1 : blocks), kAreaThreads, smem, s>>>(a);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return launch_fixed_finalize(d_acc, np, F.unit, false, nullptr, d_out, s);
}

}  // namespace lt
