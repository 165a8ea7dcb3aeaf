// lt_tile.cu -- the persistent tile raster of Eq. 6 (and the fragment
// counter built on the same walk).
//
// One CTA takes work items from an atomic counter: a (frame, tile) and up to
// work_chunk() cubes of its list. For its item, each warp repeatedly takes a
// batch of kCB cubes:
//   0. two lanes per cube project its anchor and its eight corners (four
//      each) into the warp's corner table in shared memory, so every corner
//      is projected once per tile whatever the number of tetrahedra sharing
//      it; then, 32 tetrahedra (one per lane) at a time:
//   1. every lane reads its tetrahedron's four corners from the table and
//      builds its raster form (the per-tetrahedron setup of lt_common.cuh)
//      in tile pixel coordinates; the records of the drawable ones are
//      compacted into a per-warp table in shared memory;
//   2. a warp scan flattens the (tetrahedron, row) jobs of their bounding
//      boxes; 32 jobs at a time, each lane finds the pixel span of its row
//      where every edge function is >= 0 (the owner of a job is found from the
//      popcount of the step's start mask, without shared memory);
//   3. each lane walks its own span with the row's terms in registers, kPix
//      pixels at a time for the latency of the shared atomics, evaluates
//      rho * dl and adds it to the pixel's 64-bit fixed-point accumulator in
//      shared memory;
//   4. a fragment whose FP32 error, bounded once for the tetrahedron, may
//      pass the tolerance is put aside; 32 of them at a time are bounded edge
//      by edge, and those that still may are queued and evaluated exactly in
//      FP64 after the walk.
// Integer accumulation makes the result independent of the order of the adds.
// After the walk every pixel of the tile is converted and stored once. A tile
// whose list is longer than a chunk has several items: each adds its sums to
// the tile's 64-bit slot in global memory, and the item that finishes last (a
// counter tells; nothing waits) stores the pixels from the slot. So a halo's
// tile, with a list a hundred times the mean, does not hold up the frame, and
// a small frame's few tiles still fill the chip.
//
// What bounds it: instruction issue, 73% of the slots in use at 24 warps per SM
// (128^3 particles at 1024^2; 42% of the time in step 3, a quarter in step 2,
// 17% in step 1, 13% in step 4). A span averages 2.5 to 4 pixels and the longest of
// 32 about 7, so the lanes of step 3 are busy 45% of the time, but a pixel is
// about 25 instructions there; flattening the spans as well (32 pixels at a
// time, the job and the record read again for each) kept them 90% busy at about
// 110. With that, the item split, the exact evaluation's shorter form and three
// CTAs per SM the kernel went from 6.8 to 3.9 ms there, and a frame of 256^3
// particles at 2048^2 in perspective from 16.9 to 12.9 (tile 64).
#include "lt_ff.cuh"
#include "lt_internal.h"

namespace lt {

constexpr int kRec = 40;  // words per tetrahedron record
constexpr int kCB = 16;          // cubes per warp batch (two lanes each in step 0)
constexpr int kTB = 6 * kCB;     // their tetrahedra: kTB / 32 rounds of steps 1-3
constexpr int kPix = 2;          // pixels of a span in flight at a time (1: 6.2 ms, 2: 5.5, 3: 5.4, 4: 5.3 at 128^3
                                 // / 1024^2 when the walk was alone; 2 is the best in perspective and over all)
constexpr int kCheck = 32 * kPix + 32;  // one step's worth on top of less than a batch
constexpr int kCorStride = 9;    // float4 per cube in the corner table (eight corners and a pad)

// Per-warp shared memory.
struct WarpSmem {
  float4 cor[kCB * kCorStride];  // corner (x, y, 1/Z - 1/Z_anchor, Z) relative to the cube's anchor
  float4 anc[kCB];               // anchor pixel coordinate as hi + lo: axh, axl, ayh, ayl
  float3 cinfo[kCB];             // 1/Z_anchor, perspective uncertainty factor, flags
  float recs[32 * kRec];         // records of the drawable tetrahedra of the current 32
  unsigned check[kCheck];        // pixels whose FP32 error has to be bounded edge by edge: record << 12 | y << 6 | x
};
constexpr unsigned kCubeValid = 0x100u;  // cinfo flags: bits 0..5 zero-volume mask, this bit: drawable
// Ill-conditioned fragments are queued per CTA in global memory (a.xq_cap
// entries per CTA) and evaluated exactly after the tile's walk.

// Record layout, in float4 groups so the walk reads it with a few 128-bit
// loads: [0] qx0 | qy0 << 8 | qx1 << 16 (bounding box in tile pixels) | flags,
// first row job, error bound over the tolerance (absolute part, relative
// part); [1] a[4]; [2] b[4]; [3] c[4] (edge functions); [4] 1/a[4] (row
// spans); [5] pa0, pb0, pc0, pa1; [6] pb1, pc1, g (perspective depth planes);
// [7] edge steepness st[4]; [8] periodic copy (sx + 64 | (sy + 64) << 8),
// tetrahedron index within the item's list (6 x list position + s), vertex
// uncertainty ([7] and [8] only where a fragment may need the exact path);
// [9] kRecWide: what the row terms gain to widen the spans.
constexpr int kRecWide = 1 << 24, kRecWhole = 1 << 25;  // flags: widened spans, whole rows of the box

__device__ __forceinline__ unsigned long long pack_frag(unsigned tau, int sx, int sy, int X, int Y) {
  return (unsigned long long)tau | ((unsigned long long)(unsigned)(sx + 64) << 32) |
         ((unsigned long long)(unsigned)(sy + 64) << 39) | ((unsigned long long)(unsigned)X << 46) |
         ((unsigned long long)(unsigned)Y << 52);
}

// Narrow [lo, hi] to the X where a X + rr >= 0 (rr the row term b Y + c). An
// edge constant along the row (a == 0) does not constrain it: where its rr is
// negative the walk's values are too, and add nothing.
__device__ __forceinline__ void span_edge(float a, float rr, float ia, float& lo, float& hi) {
  const float xe = -rr * ia;
  if (a > 0.0f) lo = fmaxf(lo, xe);
  if (a < 0.0f) hi = fminf(hi, xe);
}

// Periodic copies s0 .. s1 whose span [a + s P, b + s P] can overlap [lo, hi]
// (inv_p = 1 / P; a copy that only comes near is found to cover no pixel).
__device__ __forceinline__ void copies(float a, float b, float lo, float hi, float inv_p, int& s0, int& s1) {
  s0 = __float2int_ru(fmaf(lo - b, inv_p, -1e-5f));
  s1 = __float2int_rd(fmaf(hi - a, inv_p, 1e-5f));
}

// The four corners of tetrahedron s (a row of the connectivity table), three bits each.
__device__ __forceinline__ unsigned tet_code(int s) {
  constexpr unsigned c0 = tet_corner(0, 0) | tet_corner(0, 1) << 3 | tet_corner(0, 2) << 6 | tet_corner(0, 3) << 9;
  constexpr unsigned c1 = tet_corner(1, 0) | tet_corner(1, 1) << 3 | tet_corner(1, 2) << 6 | tet_corner(1, 3) << 9;
  constexpr unsigned c2 = tet_corner(2, 0) | tet_corner(2, 1) << 3 | tet_corner(2, 2) << 6 | tet_corner(2, 3) << 9;
  constexpr unsigned c3 = tet_corner(3, 0) | tet_corner(3, 1) << 3 | tet_corner(3, 2) << 6 | tet_corner(3, 3) << 9;
  constexpr unsigned c4 = tet_corner(4, 0) | tet_corner(4, 1) << 3 | tet_corner(4, 2) << 6 | tet_corner(4, 3) << 9;
  constexpr unsigned c5 = tet_corner(5, 0) | tet_corner(5, 1) << 3 | tet_corner(5, 2) << 6 | tet_corner(5, 3) << 9;
  const unsigned pair = s < 2 ? (c0 | c1 << 16) : s < 4 ? (c2 | c3 << 16) : (c4 | c5 << 16);
  return pair >> (16 * (s & 1));
}

// Exclusive warp scan of n; total receives the warp's sum.
__device__ __forceinline__ int warp_excl_scan(int n, int& total) {
  const int lane = threadIdx.x & 31;
  int incl = n;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  total = __shfl_sync(0xffffffffu, incl, 31);
  return incl - n;
}

// Pixel sums: 64-bit fixed-point integers as two planes of 32-bit words in
// shared memory (a 32-bit shared atomic is one instruction). Carries into the high word are rare: the low word
// holds 2^32 units, 16 times the mean column density at the default 28
// fraction bits.
//
// The rest of an add whose low word wrapped, or whose value passes 32 bits (u
// is then the saturated 2^32 - 1): brings the sum to what adding the whole
// value gives. A value that cannot be converted (2^63 units or more; it adds
// nothing) and an add that carries the sum past 2^64 are counted in *wraps:
// the high word's atomic returns the word before the add, so a wrap is seen by
// the add that causes it. (Inline and without global pointers: a call in the
// walk cost it its registers.)
__device__ __forceinline__ void accum_rest(unsigned lo, unsigned plane, float v, unsigned u, unsigned old, unsigned* wraps) {
  unsigned hi = old > ~u ? 1u : 0u;
  bool wrapped = false;
  if (v >= 4294967040.0f) {
    wrapped = !(v < 9223372036854775808.0f);
    const unsigned long long rest = (wrapped ? 0ull : __float2ull_rn(v)) - u;
    const unsigned rl = (unsigned)rest;
    hi += (unsigned)(rest >> 32);
    if (rl && smem_add(lo, rl) > ~rl) ++hi;
  }
  if (hi) {
    const unsigned before = smem_add(lo + plane, hi);
    wrapped = wrapped || before > ~hi;
  }
  if (wrapped) atomicAdd(wraps, 1u);
}

// Add max(v, 0), rounded to an integer, to the pixel whose low word is at lo
// and whose high word `plane` bytes further.
__device__ __forceinline__ void accum_tile(unsigned lo, unsigned plane, float v, unsigned* wraps) {
  const unsigned u = __float2uint_rn(v);  // saturates: 0 below zero (and for NaN), 2^32 - 1 above
  const unsigned old = smem_add(lo, u);
  if (old >= ~u) accum_rest(lo, plane, v, u, old, wraps);
}

// MIN_CTAS: resident 256-thread CTAs per SM that the register budget is cut for
// (see tile_min_ctas).
template <bool ANY_PERSP, bool COUNT, int MIN_CTAS>
__global__ void __launch_bounds__(256, MIN_CTAS) k_tile(RasterArgs a, unsigned long long* __restrict__ counts) {
  extern __shared__ __align__(16) float4 smem4[];
  const int T = a.tile;
  const int AS = T + 1;  // accumulator row stride: consecutive rows start on different banks
  const int nw = blockDim.x >> 5;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  WarpSmem& S = reinterpret_cast<WarpSmem*>(smem4)[warp];
  unsigned* acc = reinterpret_cast<unsigned*>(reinterpret_cast<WarpSmem*>(smem4) + nw);
  const unsigned acc_s = (unsigned)__cvta_generic_to_shared(acc), plane = 4u * T * AS;
  float* recs = S.recs;
  __shared__ unsigned long long item_s;
  __shared__ double mass_w[32];
  __shared__ unsigned qn, last_s, next_s, wraps_s;
  unsigned long long* xq = a.xq + (size_t)blockIdx.x * a.xq_cap;
  const unsigned FULL = 0xffffffffu;
  unsigned long long nfrag = 0;

  for (;;) {
    if (threadIdx.x == 0) {
      item_s = atomicAdd(&a.ctr->work_next, 1ull);
      qn = 0u;
      next_s = 0u;
      wraps_s = 0u;
    }
    if (!COUNT)
      for (int q = threadIdx.x; q < 2 * T * AS; q += blockDim.x) acc[q] = 0u;
    __syncthreads();
    const unsigned long long item = item_s;
    if (item >= (unsigned long long)*a.n_items) break;
    const unsigned long long wi = a.work[item];
    const long long tg = (long long)(wi >> kWorkChunkBits);
    const unsigned chunk = (unsigned)(wi & ((1u << kWorkChunkBits) - 1u));
    const long long tpf = (long long)a.frames[0].tiles_x * a.frames[0].tiles_y;
    const int f = (int)(tg / tpf);
    const FrameDev& F = a.frames[f];
    const bool persp = ANY_PERSP && F.persp;
    const long long tl = tg - (long long)f * tpf;
    const int tyi = (int)(tl / F.tiles_x), txi = (int)(tl - (long long)tyi * F.tiles_x);
    const int tx0 = txi * T, ty0 = tyi * T;
    const int tw = min(T, F.W - tx0), th = min(T, F.H - ty0);
    unsigned long long e0 = a.off[tg], e1 = a.off[tg + 1];
    const unsigned long long per = work_chunk(a.off[a.n_tiles], a.work_target);
    const unsigned n_chunks = work_chunks(e1 - e0, per);
    e0 += per * chunk;
    e1 = min(e1, e0 + per);
    // a graph replayed after the positions changed can need more list entries
    // than it was sized for: the scatter dropped the excess (and latched the
    // error), and the walk reads only what the lists hold
    if (e1 > a.list_cap) {
      if (threadIdx.x == 0) atomicOr(&a.ctr->errors, kErrCapacity);
      e0 = min(e0, a.list_cap);
      e1 = a.list_cap;
    }
    const unsigned ncl = (unsigned)(e1 - e0);  // (a chunk: below 2^32)
    const bool wrap = (!persp) && F.wrap;
    const float Kn0 = 6.0f * F.K;
    const float sig = F.sigma_units, inv_w = 1.0f / (float)F.W, inv_h = 1.0f / (float)F.H;
    const long long snap_off = (long long)F.snapshot * a.L.n_particles;

    for (;;) {
      // the warps take batches as they get to them (given out in turn instead,
      // they waited for one another at the item's end a fifth of the time)
      unsigned cb = 0;
      if (lane == 0) cb = atomicAdd(&next_s, (unsigned)kCB);
      cb = __shfl_sync(FULL, cb, 0);
      if (cb >= ncl) break;
      // ---- 0. lanes c and c + 16 project cube c: its anchor and corners 0-3 / 4-7
      {
        const int c = lane & (kCB - 1), hh = lane >> 4;
        const unsigned cidx = cb + c;
        bool ok = true, front = true;
        unsigned zmask = 0;
        float axh = 0.f, axl = 0.f, ayh = 0.f, ayl = 0.f, w0 = 0.f;
        if (cidx < ncl) {
          const unsigned long long li = e0 + (unsigned long long)cidx;
          const long long cube = LT_IN_BOUNDS(li < e1, &a.ctr->errors) ? (long long)a.list[li] : 0;
          zmask = a.L.degen ? (unsigned)__ldg(a.L.degen + snap_off + cube) & 63u : 0u;
          if (cube_far(a.L, F, cube)) ok = false;  // hybrid rendering: drawn as splats
          int i, j, k;
          cube_ijk(a.L, cube, i, j, k);
          float X0 = 0.f, Y0 = 0.f, Z0 = 1.f;
          if (!persp) {
            anchor_affine(F, 0, i, j, k, axh, axl);
            anchor_affine(F, 1, i, j, k, ayh, ayl);
          } else {
            float Xh, Xl, Yh, Yl, Zh, Zl;
            anchor_affine(F, 0, i, j, k, Xh, Xl);
            anchor_affine(F, 1, i, j, k, Yh, Yl);
            anchor_affine(F, 2, i, j, k, Zh, Zl);
            X0 = Xh + Xl; Y0 = Yh + Yl; Z0 = Zh + Zl;
            front = Z0 > F.near_z;
            const float rz = fast_rcp(Zh);
            ff_project(Xh, Xl, Zh, Zl, rz, F.kxh, F.kxl, F.cx, axh, axl);
            ff_project(Yh, Yl, Zh, Zl, rz, F.kyh, F.kyl, F.cy, ayh, ayl);
            w0 = fast_rcp(Z0);
          }
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int n = 4 * hh + q;
            const float3 l = load_corner(a.L, snap_off, i, j, k, n, ok);
            float4 cv;
            if (!persp) {
              cv.x = (F.r[0] * l.x + F.r[1] * l.y + F.r[2] * l.z) * F.sx;
              cv.y = (F.u[0] * l.x + F.u[1] * l.y + F.u[2] * l.z) * F.sy;
              cv.z = 0.f;
              cv.w = 1.f;
            } else {
              const float dX = F.r[0] * l.x + F.r[1] * l.y + F.r[2] * l.z;
              const float dY = F.u[0] * l.x + F.u[1] * l.y + F.u[2] * l.z;
              const float dZ = F.f[0] * l.x + F.f[1] * l.y + F.f[2] * l.z;
              const float Zn = Z0 + dZ;
              front = front && (Zn > F.near_z);
              const float inv = fast_rcp(Zn * Z0);
              // X_n/Z_n - X0/Z0 = (dX Z0 - X0 dZ) / (Z_n Z0), free of cancellation
              cv.x = (dX * Z0 - X0 * dZ) * inv * F.kx;
              cv.y = (dY * Z0 - Y0 * dZ) * inv * F.ky;
              cv.z = -dZ * inv;
              cv.w = Zn;
            }
            S.cor[c * kCorStride + n] = cv;
          }
        }
        // both halves of a cube must be finite and in front of the eye
        const bool good = __shfl_xor_sync(FULL, (int)(ok && front), 16) && ok && front;
        if (hh == 0) {
          // perspective: the anchor's offset from the view axis times the
          // depth offsets enters the vertex uncertainty (per corner |dw| / w0)
          const float offw = persp ? __fdividef(fmaxf(fabsf(axh - F.cx), fabsf(ayh - F.cy)), w0) : 0.f;
          const unsigned flags = zmask | ((cidx < ncl && good) ? kCubeValid : 0u);
          S.anc[c] = make_float4(axh, axl, ayh, ayl);
          S.cinfo[c] = make_float3(w0, offw, __int_as_float((int)flags));
        }
      }
      __syncwarp();
#pragma unroll 1
      for (int qr = 0; qr < kTB / 32; ++qr) {
        // one pass per periodic copy that reaches the tile (nearly always one);
        // a pass reads its tetrahedra from the corner table again, so that
        // nothing of the setup stays in registers through steps 2-4
        int rounds = 1;
#pragma unroll 1
        for (int r = 0; r < rounds; ++r) {
          // ---- 1. one tetrahedron per lane
          const int ts = qr * 32 + lane;  // tetrahedron slot of the batch
          const int c = ts / 6, s = ts - 6 * c;
          const unsigned tau = (cb + c) * 6u + s;  // index within the item's tetrahedra
          const float3 ci = S.cinfo[c];
          const unsigned cfl = (unsigned)__float_as_int(ci.z);
          const bool ok = (cfl & kCubeValid) && !((cfl >> s) & 1u);  // zero volume: contributes nothing
          int nrows = 0, qx0 = 0, qx1 = 0, qy0 = 0, sx = 0, sy = 0, ncp = 0;
          float delta = 0.f;
          TetRaster t;
          if (ok) {
            const float4 an = S.anc[c];
            float px[4], py[4], pdw[4], pz[4];
            const unsigned code = tet_code(s);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const float4 v = S.cor[c * kCorStride + ((code >> (3 * k)) & 7u)];
              px[k] = v.x; py[k] = v.y; pdw[k] = v.z; pz[k] = v.w;
            }
            const float bx0 = fminf(fminf(px[0], px[1]), fminf(px[2], px[3]));
            const float bx1 = fmaxf(fmaxf(px[0], px[1]), fmaxf(px[2], px[3]));
            const float by0 = fminf(fminf(py[0], py[1]), fminf(py[2], py[3]));
            const float by1 = fmaxf(fmaxf(py[0], py[1]), fmaxf(py[2], py[3]));
            int ncx = 1, sx0 = 0, sy0 = 0;
            ncp = 1;
            if (wrap) {
              int sx1, sy1;
              const float axa = an.x + an.y, aya = an.z + an.w;
              copies(axa + bx0, axa + bx1, (float)tx0 - 0.5f, (float)(tx0 + tw) - 0.5f, inv_w, sx0, sx1);
              copies(aya + by0, aya + by1, (float)ty0 - 0.5f, (float)(ty0 + th) - 0.5f, inv_h, sy0, sy1);
              ncx = max(0, min(sx1 - sx0, 63) + 1);
              ncp = ncx * max(0, min(sy1 - sy0, 63) + 1);
            }
            float Rv = fmaxf(fmaxf(fabsf(bx0), fabsf(bx1)), fmaxf(fabsf(by0), fabsf(by1)));
            if (persp) Rv += ci.y * fmaxf(fmaxf(fabsf(pdw[0]), fabsf(pdw[1])), fmaxf(fabsf(pdw[2]), fabsf(pdw[3])));
            delta = vertex_uncertainty(Rv, persp);
            const float margin = 1e-3f + delta;
            if (r < ncp) {
              if (wrap) {
                sx = sx0 + r % ncx;
                sy = sy0 + r / ncx;
              }
              // vertex coordinates relative to the tile origin: anchor + shift - tile corner
              const float ox = ((float)(tx0 - sx * F.W) - an.x) - an.y;
              const float oy = ((float)(ty0 - sy * F.H) - an.z) - an.w;
              qx0 = max(0, (int)ceilf(bx0 - ox - margin));
              qx1 = min(tw - 1, (int)floorf(bx1 - ox + margin));
              qy0 = max(0, (int)ceilf(by0 - oy - margin));
              const int qy1 = min(th - 1, (int)floorf(by1 - oy + margin));
              if (qx0 <= qx1 && qy0 <= qy1) {
                // the raster form relative to the bounding box's first pixel:
                // small coordinates keep the round-off of evaluating a x + b y + c
                // (and with it the exact path's share) small. In two steps, over
                // the tile's origin: the difference taken at once from the anchor
                // rounds a little less, but it changes which fragments of ultra-flat
                // tetrahedra are evaluated exactly, and with them pixels by up to
                // 1e-3 of their value
                const float lx = (float)qx0, ly = (float)qy0;
                const float x0 = (px[0] - ox) - lx, x1 = (px[1] - ox) - lx, x2 = (px[2] - ox) - lx, x3 = (px[3] - ox) - lx;
                const float y0 = (py[0] - oy) - ly, y1 = (py[1] - oy) - ly, y2 = (py[2] - oy) - ly, y3 = (py[3] - oy) - ly;
                float Kn = Kn0;
                if (persp) Kn = __fdividef(Kn0, pz[0] * pz[1] * pz[2] * pz[3]);
                const bool set =
                    persp ? tet_setup<true, true>(x0, y0, x1, y1, x2, y2, x3, y3, pdw[0], pdw[1], pdw[2], pdw[3], Kn, ci.x,
                                            fast_rcp(Kn), t)
                          : tet_setup<false, true>(x0, y0, x1, y1, x2, y2, x3, y3, 0.f, 0.f, 0.f, 0.f, Kn, 0.f, 0.f, t);
                if (set) nrows = qy1 - qy0 + 1;
              }
            }
          }
          if (wrap && r == 0) rounds = __reduce_max_sync(FULL, ncp);
          // ---- 2. records of the drawable tetrahedra, compacted, and the
          // flattened (tetrahedron, row) jobs
          const unsigned lt_mask = (1u << lane) - 1u, le_mask = (2u << lane) - 1u;
          const int slot = __popc(__ballot_sync(FULL, nrows > 0) & lt_mask);
          int rtotal;
          const int roff = warp_excl_scan(nrows, rtotal);
          if (nrows > 0 && LT_IN_BOUNDS(slot < 32, &a.ctr->errors)) {
            float4* R = reinterpret_cast<float4*>(recs + slot * kRec);
            // bounds of a fragment's error, in units of the tolerance, over its
            // edges and the box: err_a + err_b |f| (zero: never beyond it)
            float err_a = 0.f, err_b = 0.f;
            int flags = 0;
            if (COUNT) {
              flags = may_miss_fragments(t, sig, delta) ? kRecWhole : 0;
            } else if (may_need_exact(t, sig, delta)) {
              const float scale = t.vscale * (1.0f / kFragTol);
              const float slope = kFragErr * fmaxf(fmaxf(t.st[0], t.st[1]), fmaxf(t.st[2], t.st[3]));
              err_a = fmaf(max_edge_slope(t), delta, max_eval_error(t, (float)T)) * scale;
              err_b = slope * scale;
              R[7] = make_float4(t.st[0], t.st[1], t.st[2], t.st[3]);
              R[8] = make_float4(__int_as_float((sx + 64) | (sy + 64) << 8), __int_as_float((int)tau), delta, 0.f);
              if (may_miss_fragments(t, sig, delta)) {
                // a steep sliver: pixels that the bounds could move inside are
                // checked too, so the spans go to where f_e + e_e <= 0, which for
                // a relative part below 1/2 is f_e below minus twice the absolute
                // one (else over whole rows of the box)
                flags = slope < 0.5f ? kRecWide : kRecWhole;
                const float pos = delta + kEvalErr * (float)T;
                float w[4];
#pragma unroll
                for (int e = 0; e < 4; ++e)
                  w[e] = 2.0f * fmaf(fabsf(t.a[e]) + fabsf(t.b[e]), pos, kEvalErr * fabsf(t.c[e]));
                R[9] = make_float4(w[0], w[1], w[2], w[3]);
              }
            }
            R[0] = make_float4(__int_as_float(qx0 | qy0 << 8 | qx1 << 16 | flags), __int_as_float(roff), err_a, err_b);
            R[1] = make_float4(t.a[0], t.a[1], t.a[2], t.a[3]);
            R[2] = make_float4(t.b[0], t.b[1], t.b[2], t.b[3]);
            R[3] = make_float4(t.c[0], t.c[1], t.c[2], t.c[3]);
            R[4] = make_float4(inv_or_zero(t.a[0]), inv_or_zero(t.a[1]), inv_or_zero(t.a[2]), inv_or_zero(t.a[3]));
            if (persp) {
              R[5] = make_float4(t.pa[0], t.pb[0], t.pc[0], t.pa[1]);
              R[6] = make_float4(t.pb[1], t.pc[1], t.g, 0.f);
            }
          }
          __syncwarp();
          // The owner of a position in a 32-wide step is the last run starting
          // at or before it: with runs compacted, its index is the number of
          // runs started before the step plus those started in the step up to
          // the position, minus one.
          int rprev = 0, nchk = 0;
          for (int rb = 0; rb < rtotal; rb += 32) {
            const int rrel = roff - rb;
            const unsigned rmask = __reduce_or_sync(FULL, (nrows > 0 && rrel >= 0 && rrel < 32) ? (1u << rrel) : 0u);
            const int o = rprev + __popc(rmask & le_mask) - 1;
            rprev += __popc(rmask);
            // ---- 3. pixel span of the job's row: every edge function >= 0
            // (coordinates relative to the record's bounding-box corner)
            // (lanes past the last job go through the motions on some record, with
            // no pixels)
            const float4* R = reinterpret_cast<const float4*>(recs + min(max(o, 0), 31) * kRec);
            const float4 r0 = R[0], ra = R[1], rbv = R[2], rc = R[3], ri = R[4];
            const int yl = rb + lane - __float_as_int(r0.y);
            const float fy = (float)yl;
            const float4 rr = make_float4(fmaf(rbv.x, fy, rc.x), fmaf(rbv.y, fy, rc.y), fmaf(rbv.z, fy, rc.z),
                                          fmaf(rbv.w, fy, rc.w));
            const int box = __float_as_int(r0.x);
            const int bqx0 = box & 0xff, bqy0 = (box >> 8) & 0xff;
            const float wf = (float)(((box >> 16) & 0xff) - bqx0);  // last pixel of the box, local
            float4 sp = rr;
            if (box & kRecWide) {
              const float4 w = R[9];
              sp.x += w.x; sp.y += w.y; sp.z += w.z; sp.w += w.w;
            }
            float lo = __int_as_float(0xff800000), hi = __int_as_float(0x7f800000);
            span_edge(ra.x, sp.x, ri.x, lo, hi);
            span_edge(ra.y, sp.y, ri.y, lo, hi);
            span_edge(ra.z, sp.z, ri.z, lo, hi);
            span_edge(ra.w, sp.w, ri.w, lo, hi);
            lo = box & kRecWhole ? 0.0f : fmaxf(lo - 1e-3f, 0.0f);
            hi = box & kRecWhole ? wf : fminf(hi + 1e-3f, wf);
            const int xl = __float2int_ru(lo);
            int len = __float2int_rd(hi) - xl + 1;
            if (!(lo <= hi) || rb + lane >= rtotal) len = 0;
            const float err_a = r0.z, err_b = r0.w;
            float4 r5 = make_float4(0.f, 0.f, 0.f, 0.f);
            float m0 = 0.f, m1 = 0.f, g = 0.f;
            if (persp) {
              r5 = R[5];
              const float4 r6 = R[6];
              m0 = fmaf(r5.y, fy, r5.z);
              m1 = fmaf(r6.x, fy, r6.y);
              g = r6.z;
            }
            unsigned pix = acc_s + 4u * ((bqy0 + yl) * AS + bqx0 + xl);  // the span's first pixel
            if (!LT_IN_BOUNDS(len <= 0 || (o >= 0 && o < 32 && bqx0 + xl >= 0 && bqx0 + xl + len <= tw && bqy0 + yl < th),
                              &a.ctr->errors))
              len = 0;
            // ---- 4. the spans' pixels, kPix at a time
            const int longest = __reduce_max_sync(FULL, len);
            const unsigned long long a01 = pack2(ra.x, ra.y), a23 = pack2(ra.z, ra.w);
            const unsigned long long c01 = pack2(rr.x, rr.y), c23 = pack2(rr.z, rr.w);
            const unsigned long long pm = pack2(r5.x, r5.w), cm = pack2(m0, m1);
            float fx = (float)xl;
            for (int k0 = 0;;) {
              unsigned u[kPix], old[kPix];
              float v[kPix];
              bool chk[kPix], any_chk = false;
#pragma unroll
              for (int k = 0; k < kPix; ++k) {
                const float x = fx + (float)k;
                const unsigned long long xx = pack2(x, x);
                const float2 f01 = unpack2(fma2(a01, xx, c01)), f23 = unpack2(fma2(a23, xx, c23));
                const float fm = fminf(fminf(f01.x, f01.y), fminf(f23.x, f23.y));
                v[k] = fm;
                if (persp) {
                  const float2 M2 = unpack2(fma2(pm, xx, cm));
                  const float Tv = fmaxf(fm, 0.0f), M = fmaxf(M2.x, M2.y);
                  v[k] = __fdividef(Tv, M * fmaf(g, Tv, M));
                }
                u[k] = __float2uint_rn(v[k]);  // saturates: 0 below zero (and for NaN), 2^32 - 1 above
                old[k] = 0u;
                const bool in = k0 + k < len;
                if (COUNT) nfrag += in && v[k] > 0.0f ? 1u : 0u;
                // (a non-finite bound fails the test too)
                chk[k] = !COUNT && in && !(fmaf(err_b, fabsf(fm), err_a) <= fmaxf(v[k], sig));
                any_chk = any_chk || chk[k];
              }
              if (!COUNT) {
#pragma unroll
                for (int k = 0; k < kPix; ++k)
                  if (k0 + k < len && !chk[k]) old[k] = smem_add(pix + 4u * k, u[k]);
                bool rest = false;
#pragma unroll
                for (int k = 0; k < kPix; ++k) rest = rest || (k0 + k < len && !chk[k] && old[k] >= ~u[k]);
                if (rest) {
#pragma unroll
                  for (int k = 0; k < kPix; ++k)
                    if (k0 + k < len && !chk[k] && old[k] >= ~u[k])
                      accum_rest(pix + 4u * k, plane, v[k], u[k], old[k], &wraps_s);
                }
                if (__any_sync(FULL, any_chk)) {
#pragma unroll
                  for (int k = 0; k < kPix; ++k) {
                    const unsigned m = __ballot_sync(FULL, chk[k]);
                    if (chk[k] && LT_IN_BOUNDS(nchk + __popc(m & lt_mask) < kCheck, &a.ctr->errors))
                      S.check[nchk + __popc(m & lt_mask)] = (unsigned)(o << 12 | yl << 6 | (xl + k0 + k));
                    nchk += __popc(m);
                  }
                }
              }
              k0 += kPix;
              fx += (float)kPix;
              pix += 4u * kPix;
              if (!COUNT) {
                // pixels to check, a warp's worth at a time (the rest of them after
                // the last step): fragments whose error bound is too large, and
                // pixels the vertex uncertainty could move inside, go to the exact
                // evaluation
                const bool last = k0 >= longest && rb + 32 >= rtotal;
                while (nchk >= 32 || (last && nchk > 0)) {
                  __syncwarp();
                  const int n = min(nchk, 32);
                  nchk -= n;
                  if (lane < n) {
                    const unsigned q = S.check[nchk + lane];
                    const float4* R = reinterpret_cast<const float4*>(recs + (q >> 12) * kRec);
                    const int x = (int)(q & 63u), y = (int)((q >> 6) & 63u);
                    const float fxc = (float)x, fyc = (float)y;
                    const float4 ca = R[1], cb = R[2], cc = R[3], r0 = R[0], r8 = R[8];
                    const float f0 = fmaf(ca.x, fxc, fmaf(cb.x, fyc, cc.x)), f1 = fmaf(ca.y, fxc, fmaf(cb.y, fyc, cc.y));
                    const float f2 = fmaf(ca.z, fxc, fmaf(cb.z, fyc, cc.z)), f3 = fmaf(ca.w, fxc, fmaf(cb.w, fyc, cc.w));
                    const float Tv = fmaxf(fminf(fminf(f0, f1), fminf(f2, f3)), 0.0f);
                    float vc = Tv, dq = 1.0f;
                    if (persp) {
                      const float4 p5 = R[5], p6 = R[6];
                      const float M = fmaxf(fmaf(p5.x, fxc, fmaf(p5.y, fyc, p5.z)), fmaf(p5.w, fxc, fmaf(p6.x, fyc, p6.y)));
                      const float den = M * fmaf(p6.z, Tv, M);
                      vc = __fdividef(Tv, den);
                      dq = __fdividef(M, den);  // d value / d T = (M / den)^2
                    }
                    const int X = (__float_as_int(r0.x) & 0xff) + x, Y = ((__float_as_int(r0.x) >> 8) & 0xff) + y;
                    bool done = false;
                    if (fragment_needs_exact(f0, f1, f2, f3, ca, cb, cc, R[7], fxc, fyc, r8.z, dq * dq, vc, sig)) {
                      const unsigned at = atomicAdd(&qn, 1u);
                      done = at < a.xq_cap;  // queue full: keep the FP32 value (counted in the statistics)
                      const int sxy = __float_as_int(r8.x);
                      if (done)
                        xq[at] = pack_frag((unsigned)__float_as_int(r8.y), (sxy & 255) - 64, (sxy >> 8) - 64, X, Y);
                    }
                    if (!done && vc > 0.0f) accum_tile(acc_s + 4u * (Y * AS + X), plane, vc, &wraps_s);
                  }
                }
              }
              if (k0 >= longest) break;
            }
          }
          __syncwarp();  // the records are read until here
        }
      }
      __syncwarp();
    }
    if (COUNT) {
      unsigned long long c = nfrag;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) c += __shfl_down_sync(FULL, c, o);
      if (lane == 0 && c) atomicAdd(&counts[f], c);
      nfrag = 0;
      __syncthreads();
      continue;
    }
    __syncthreads();
    // ---- ill-conditioned fragments: exact FP64 evaluation, all lanes busy
    const unsigned nq = min(qn, a.xq_cap);
    if (threadIdx.x == 0 && qn) {
      atomicAdd(&a.ctr->exact_fragments, (unsigned long long)nq);
      atomicMax(&a.ctr->exact_tile_max, (unsigned long long)qn);
      if (qn > a.xq_cap) atomicAdd(&a.ctr->queue_overflow, (unsigned long long)(qn - a.xq_cap));
    }
    for (unsigned qi = threadIdx.x; qi < nq; qi += blockDim.x) {
      const unsigned long long q = xq[qi];
      const unsigned tau_o = (unsigned)(q & 0xffffffffull);
      const int sxo = (int)((q >> 32) & 127u) - 64, syo = (int)((q >> 39) & 127u) - 64;
      const int X = (int)((q >> 46) & 63u), Y = (int)((q >> 52) & 63u);
      const unsigned long long li = e0 + (unsigned long long)(tau_o / 6);
      if (!LT_IN_BOUNDS(li < e1 && X < tw && Y < th, &a.ctr->errors)) continue;
      const long long cube = (long long)a.list[li];
      const float val = exact_fragment(a.L, F, cube, (int)(tau_o % 6), sxo, syo, tx0 + X, ty0 + Y);
      if (val > 0.0f) accum_tile(acc_s + 4u * (Y * AS + X), plane, val, &wraps_s);
    }
    __syncthreads();
    if (threadIdx.x == 0 && wraps_s) {
      atomicOr(&a.ctr->errors, kErrRange);
      atomicAdd(&a.ctr->range_overflow, (unsigned long long)wraps_s);
    }
    // ---- one store per pixel, and the tile's share of the frame mass
    unsigned long long* slot = nullptr;
    if (n_chunks > 1) {
      // part of a tile: into its slot, and on to the next item unless this is
      // the last of them (the fences order the sums before the count)
      const unsigned si = a.slot[tg];
      slot = a.slot_acc + (size_t)si * T * T;
      for (int li = threadIdx.x; li < tw * th; li += blockDim.x) {
        const int ly = li / tw, lx = li - ly * tw;
        const unsigned* px = acc + ly * AS + lx;
        const unsigned long long v = (unsigned long long)px[T * AS] << 32 | px[0];
        if (v && atomicAdd(slot + ly * T + lx, v) > ~v) {
          atomicOr(&a.ctr->errors, kErrRange);
          atomicAdd(&a.ctr->range_overflow, 1ull);
        }
      }
      __threadfence();
      __syncthreads();
      if (threadIdx.x == 0) {
        const bool last = atomicAdd(&a.slot_done[si], 1u) == n_chunks - 1u;
        if (last) a.slot_done[si] = 0u;
        last_s = last ? 1u : 0u;
      }
      __syncthreads();
      if (!last_s) continue;
      __threadfence();
    }
    double msum = 0.0;
    float* img = a.image + (long long)f * a.image_stride;
    for (int li = threadIdx.x; li < tw * th; li += blockDim.x) {
      const int ly = li / tw, lx = li - ly * tw;
      const unsigned* px = acc + ly * AS + lx;
      float scale = 1.0f;
      if (persp) {
        const float xt = F.tan_x * (2.0f * ((float)(tx0 + lx) + 0.5f) / (float)F.W - 1.0f);
        const float yt = F.tan_y * (2.0f * ((float)(ty0 + ly) + 0.5f) / (float)F.H - 1.0f);
        scale = sqrtf(1.0f + xt * xt + yt * yt);
      }
      unsigned long long v = (unsigned long long)px[T * AS] << 32 | px[0];
      if (slot) {
        unsigned long long* sp = slot + ly * T + lx;
        v = __ldcg(sp);
        *sp = 0ull;  // slots are zero between renders
      }
      const float vf = fixed_to_float(v, F.scale, scale);
      img[(long long)(ty0 + ly) * F.W + (tx0 + lx)] = vf;
      msum += (double)vf;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) msum += __shfl_down_sync(FULL, msum, o);
    if (lane == 0) mass_w[warp] = msum;
    __syncthreads();
    if (threadIdx.x < 32) {
      double w = threadIdx.x < (unsigned)nw ? mass_w[threadIdx.x] : 0.0;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) w += __shfl_down_sync(FULL, w, o);
      if (threadIdx.x == 0) a.mass_tile[tg] = w * F.pix_area;
    }
    __syncthreads();
  }
}

static size_t tile_smem(int threads, int tile) {
  const int nw = threads / 32;
  return sizeof(WarpSmem) * nw + 2 * sizeof(unsigned) * tile * (tile + 1);
}

// Three CTAs of 80 registers (24 warps) are 6% to 8% faster than two of 128 at
// 128^3 / 1024^2 and in perspective (3.65 against 3.89 ms, 2.40 against 2.51),
// spills around the exact evaluation's call included; four of 64 are slower
// (3.85, 2.67). Tiles of 64 pixels leave shared memory for two.
static int tile_min_ctas(int tile) { return tile > 32 ? 2 : 3; }

typedef void (*TileKernel)(RasterArgs, unsigned long long*);
static TileKernel tile_kernel(int tile, bool any_persp) {
  if (tile_min_ctas(tile) == 2) return any_persp ? k_tile<true, false, 2> : k_tile<false, false, 2>;
  return any_persp ? k_tile<true, false, 3> : k_tile<false, false, 3>;
}

int raster_max_ctas_per_sm(int threads, int tile, int any_persp) {
  if (threads > 256 || threads % 32) return 0;  // the kernel is compiled for at most 256 threads
  int n = 0;
  const size_t smem = tile_smem(threads, tile);
  TileKernel k = tile_kernel(tile, any_persp);
  cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, threads, smem) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

cudaError_t launch_count_fragments(const RasterArgs& a, unsigned long long* d_counts, int n_frames, int ctas,
                                   int threads, cudaStream_t s) {
  (void)n_frames;
  const size_t smem = tile_smem(threads, a.tile);
  cudaFuncSetAttribute(k_tile<true, true, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  k_tile<true, true, 2><<<ctas, threads, smem, s>>>(a, d_counts);
  return cudaGetLastError();
}

cudaError_t launch_raster(const RasterArgs& a, int ctas, int threads, int any_persp, cudaStream_t s) {
  const size_t smem = tile_smem(threads, a.tile);
  TileKernel k = tile_kernel(a.tile, any_persp);
  cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  k<<<ctas, threads, smem, s>>>(a, nullptr);
  return cudaGetLastError();
}

}  // namespace lt
