// Inverse polygon mapping on the device (Sec. 3.2, Fig. 3): a mapped
// triangle's unit of flux is split among the pixels it covers in proportion
// to area(T n pixel) / |area(T)|.  Each share is rounded to a multiple of
// 2^-32 triangle and summed as an integer in a uint64 map, so sums are exact
// and independent of the order of the atomics.
//
// Vertices arrive in a canonical pixel form (integer pixel + fraction in
// [0, 1)) that does not depend on which warp computed them, so the two
// triangles sharing an edge see bit-identical edge geometry.  A triangle is
// processed in the frame of its first vertex's pixel, where FP32 coordinates
// of small triangles are exact to ~1e-7 pixel.
//
// Area of T inside a box.  Projecting the plane onto a closed box B by
// clamping, (x, y) -> (clamp(x, B), clamp(y, B)), maps T's boundary to a
// closed curve in B that winds around every interior point of B exactly as
// often as T's boundary does (a horizontal ray from such a point meets both
// curves in the same signed crossings) and around no point outside B, so the
// shoelace sum of the projected boundary is area(T n B).  Each edge is cut
// where it crosses the box's lines, so every projected piece is straight.
// With the box translated to [0, 1]^2 every term is O(1): no cancellation,
// no polygon arrays, everything in registers.  The same identity with a
// quadrant (x < X, y < Y) gives the three areas that split a triangle
// covering a 2 x 2 pixel box; for a pixel of a larger triangle the shoelace
// sum is taken edge by edge as the integral of the clamped x over the
// clamped y.  These are exactly the areas that the column-then-row
// Sutherland-Hodgman clipping of Fig. 3 produces.
//
// Paths:
//   * the triangle lies inside one pixel (the common case at ~100 rays per
//     pixel): that pixel gains exactly 2^32;
//   * it spans two pixels split by one grid line: the vertex alone on its
//     side cuts off a similar triangle whose area fraction is a product of
//     two edge parameters;
//   * it spans 2 x 2 pixels: three quadrant areas by inclusion-exclusion;
//   * larger (cells next to a star map to triangles up to hundreds of
//     pixels wide; cells along a caustic to long slivers): the pixel rows of
//     32 such triangles are dealt out to the lanes, each row adds the
//     constant 1/|area| to its run of fully covered pixels through a per-row
//     difference array, and the partially covered pixels of those rows are
//     then dealt out one per lane and measured from the row's edge pieces
//     (row_pieces, piece_mean).  Work is proportional to the perimeter, not
//     the area, and no lane loops on its own.
// All but the first are queued per warp in shared memory and finished 32 of
// a kind at a time.
#pragma once
#include <climits>

#include "mm_common.cuh"

namespace mm {

#define MM_VTX_INVALID INT_MIN
#define MM_FIX_ONE 4294967296ull  // one whole triangle in fixed-point units
#define MM_U24_ONE 16777216u      // and in 2^-24 triangles

__device__ __forceinline__ float rcp_approx_f(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Share of a triangle in fixed-point units (2^32 = the whole triangle).  An
// FP32 fraction carries 24 significant bits, so it is rounded at 2^-24 and
// shifted: 32-bit conversions only (64-bit ones would run on the FP64 pipe).
__device__ __forceinline__ unsigned frac_to_u24(float f) {  // in 2^-24 triangles
  f = __saturatef(f);  // clamp to [0, 1] (NaN -> 0)
  return __float2uint_rn(f * 16777216.0f);
}
__device__ __forceinline__ unsigned long long frac_to_fixed(float f) {
  return (unsigned long long)frac_to_u24(f) << 8;
}

// The map edges a vertex lies beyond, one bit each (0 when non-finite): a
// triangle lies wholly beyond one edge when its vertices share a bit.
__device__ __forceinline__ unsigned outcode(const MapCore &M, const Vtx &v) {
  const unsigned c = (v.px < 0 ? 1u : 0u) | (v.px >= M.npix ? 2u : 0u) | (v.py < 0 ? 4u : 0u) |
                     (v.py >= M.npix_y ? 8u : 0u);
  return v.px == MM_VTX_INVALID ? 0u : c;
}

// ---------------------------------------------------------------------------
// accumulation
// ---------------------------------------------------------------------------

// MM_DEBUG builds check every accumulator and row-difference index against
// its array before the atomic and, out of range, skip the access and set
// ERR_BOUNDS in the error word (read back through mm_get_stats).  Other
// builds compile the check to nothing.
#ifdef MM_DEBUG
__device__ __forceinline__ bool mm_index_ok(unsigned *err, long long idx, long long n) {
  if (idx >= 0 && idx < n) return true;
  atomicOr(err, ERR_BOUNDS);
  return false;
}
#define MM_INDEX_OK(err, idx, n) mm_index_ok((err), (long long)(idx), (long long)(n))
#else
#define MM_INDEX_OK(err, idx, n) true
#endif

// Add u (in 2^-24 triangles) to map pixel idx if `in` the map.
__device__ __forceinline__ void deposit(const MapCore &M, bool in, long long idx, unsigned u) {
  if (in && u && MM_INDEX_OK(M.err, idx, (long long)M.npix * M.npix_y))
    atomicAdd(&M.acc[idx], (unsigned long long)u << 8);
}

// The map's accumulators alone, passed as scalars to the out-of-line row
// and pixel dealing (so the kernel's MapDev, a launch parameter, is never
// copied to local memory to be addressed).
struct MapAcc {
  unsigned long long *acc, *span;
  int npix, npix_y;
  unsigned *err;
};

// Lane-private run accumulator: consecutive one-pixel triangles (or rays) of
// a lane's column usually hit the same pixel; they are counted in a
// register.  UNIT is one triangle's (or ray's) fixed-point units.
struct RunAcc {
  int px, py;  // the pixel being counted, px < 0 for none
  unsigned n;
};
#define MM_RUN_NONE RunAcc{-1, 0, 0u}

template <unsigned long long UNIT>
__device__ __forceinline__ void run_flush(const MapCore &M, RunAcc &a) {
  const long long idx = (long long)a.py * M.npix + a.px;
  if (a.px >= 0 && MM_INDEX_OK(M.err, idx, (long long)M.npix * M.npix_y))
    atomicAdd(&M.acc[idx], a.n * UNIT);
  a = MM_RUN_NONE;
}

// Count one in in-map pixel (px, py).
template <unsigned long long UNIT>
__device__ __forceinline__ void run_add(const MapCore &M, RunAcc &a, int px, int py) {
  if (px == a.px && py == a.py) {
    a.n++;
    return;
  }
  run_flush<UNIT>(M, a);
  a = RunAcc{px, py, 1u};
}

// ---------------------------------------------------------------------------
// areas
// ---------------------------------------------------------------------------

// Split of T by one grid line u = L (u = x or y, coordinates u0, u1, u2):
// the vertex alone on its side cuts off a triangle similar to T, whose
// share of the area is d^2 / ((u_a - u_l)(u_b - u_l)), d = L - u_l (the
// two edge parameters at the line, multiplied).  Returns that share and
// whether the lone vertex lies on the low side u < L.
__device__ __forceinline__ float lone_vertex_share(float u0, float u1, float u2, float L,
                                                   bool &lone_low) {
  const bool b0 = u0 < L, b1 = u1 < L, b2 = u2 < L;
  lone_low = (b0 + b1 + b2) == 1;
  float ul = u2, ua = u0, ub = u1;
  if (b0 == lone_low) {
    ul = u0;
    ua = u1;
    ub = u2;
  } else if (b1 == lone_low) {
    ul = u1;
    ua = u0;
    ub = u2;
  }
  const float d = L - ul;
  return d * d * rcp_approx_f((ua - ul) * (ub - ul));
}

// Share of T (in 2^-24 triangles) on the low side u < L of one grid line it
// crosses.  The line is chosen from the vertices' integer pixels, and a
// vertex's FP32 coordinate in a neighbouring pixel's frame can round onto the
// line (k + f with f within 2^-24 of 1), leaving no vertex strictly below it:
// then nothing of T lies below the line (and all of it when none lies above).
__device__ __forceinline__ unsigned low_side_u24(float u0, float u1, float u2, float L) {
  const int nlow = (u0 < L) + (u1 < L) + (u2 < L);
  bool lone_low;
  const float v = lone_vertex_share(u0, u1, u2, L, lone_low);
  const float low = nlow == 0 ? 0.f : (nlow == 3 ? 1.f : (lone_low ? v : 1.f - v));
  return frac_to_u24(low);
}

// Contribution of edge P -> Q to the signed area of T n {x < X, y < Y}
// (Green's theorem on the boundary clamped to the quadrant): the edge's
// piece below Y, times the mean of min(x - X, 0) over it.  The terms in X
// itself sum to zero around T and are left out.
__device__ __forceinline__ float quadrant_edge(float px, float py, float qx, float qy, float X,
                                               float Y) {
  const float ys = fminf(py, Y), ye = fminf(qy, Y);
  const float xY = fmaf(Y - py, (qx - px) * rcp_approx_f(qy - py), px);  // x on the edge at Y
  const float xs = py <= Y ? px : xY, xe = qy <= Y ? qx : xY;
  const float a = fminf(xs, xe) - X, b = fmaxf(xs, xe) - X;
  const float m = b <= 0.f ? 0.5f * (a + b) : (a >= 0.f ? 0.f : -0.5f * a * a * rcp_approx_f(b - a));
  return ye != ys ? (ye - ys) * m : 0.f;
}

// ---------------------------------------------------------------------------
// queued triangles
// ---------------------------------------------------------------------------

// A triangle waiting in a warp's queue, 32 bytes.
//   * Within 2 x 2 pixels (the line and quad queues): (x, y) is the low
//     corner of its pixel box, f[2 k], f[2 k + 1] vertex k's position inside
//     its own pixel, whose offset from the corner (0 or 1 per axis) is the
//     sign bit.
//   * Larger (the big queue and the map's device queue): (x, y) is the first
//     vertex's pixel and f the three vertices in its frame; the sign bit of
//     f[0] (a fraction, >= 0) marks a box of at most MM_MED_PIXELS map pixels
//     while the triangle is in the warp's queue.
// The scan that finds a triangle only stores it: areas, slopes and shares
// are formed when 32 of a kind are taken off a queue, every lane busy,
// instead of in branches that a few lanes take on nearly every row (the
// larger triangles' three slopes and inverse area are IEEE divisions).
struct __align__(16) RawTri {
  int x, y;
  float f[6];
};
static_assert(sizeof(RawTri) == MM_TRIJOB_BYTES, "RawTri layout");

__device__ __forceinline__ void raw_store(RawTri *e, int x, int y, float f0, float f1, float f2,
                                          float f3, float f4, float f5) {
  float4 *w = reinterpret_cast<float4 *>(e);
  w[0] = make_float4(__int_as_float(x), __int_as_float(y), f0, f1);
  w[1] = make_float4(f2, f3, f4, f5);
}
__device__ __forceinline__ RawTri raw_load(const RawTri *e) {
  const float4 *w = reinterpret_cast<const float4 *>(e);
  const float4 u = w[0], v = w[1];
  RawTri t;
  t.x = __float_as_int(u.x);
  t.y = __float_as_int(u.y);
  t.f[0] = u.z;
  t.f[1] = u.w;
  t.f[2] = v.x;
  t.f[3] = v.y;
  t.f[4] = v.z;
  t.f[5] = v.w;
  return t;
}

// Twice the signed area of a triangle in its frame.
// (one rounding order for every caller, so that counts against the
// near-critical threshold do not depend on where the area is formed)
__device__ __forceinline__ float tri_area2(const float (&t)[6]) {
  return fmaf(t[2] - t[0], t[5] - t[1], -__fmul_rn(t[4] - t[0], t[3] - t[1]));
}

// Vertex k's fraction with its pixel's offset from the box corner (0 or 1)
// in the sign bit.
__device__ __forceinline__ float with_offset(float f, int px, int lo) {
  return __int_as_float(__float_as_int(f) | ((px - lo) << 31));
}

// A triangle within 2 x 2 pixels in the frame of its first vertex's pixel
// (t), and that pixel's offset (ax, ay) from the box corner.
__device__ __forceinline__ void small_frame(const RawTri &e, float (&t)[6], int &ax, int &ay) {
  const int b0 = __float_as_int(e.f[0]), b1 = __float_as_int(e.f[1]);
  ax = b0 < 0;
  ay = b1 < 0;
  const float fx = (float)ax, fy = (float)ay;
  t[0] = fabsf(e.f[0]);
  t[1] = fabsf(e.f[1]);
#pragma unroll
  for (int k = 1; k < 3; k++) {
    // the vertex's pixel relative to the first vertex's (-1, 0 or 1), then its fraction
    t[2 * k] = ((__float_as_int(e.f[2 * k]) < 0 ? 1.f : 0.f) - fx) + fabsf(e.f[2 * k]);
    t[2 * k + 1] = ((__float_as_int(e.f[2 * k + 1]) < 0 ? 1.f : 0.f) - fy) + fabsf(e.f[2 * k + 1]);
  }
}

// Counters of a lane: triangles dropped (non-finite, or without area) and
// triangles whose local |mu| exceeds the near-critical threshold.
struct LaneCount {
  unsigned dropped, critical;
};

// Area test of a triangle that meets the map: false (and counted) when it
// has none; near-critical ones are counted.
__device__ __forceinline__ bool area_ok(const MapCore &M, float area2, LaneCount &lc) {
  if (!(area2 != 0.f) || !isfinite(area2)) {
    lc.dropped++;
    return false;
  }
  lc.critical += fabsf(area2) < M.crit_area2;
  return true;
}

// A triangle across one grid line u = L (u = x or y) of two pixels.  The
// vertex alone on its side cuts off a triangle similar to the whole, of area
// fraction d^2 / ((u_a - u_l)(u_b - u_l)) with d = L - u_l (the two edge
// parameters at the line, multiplied).  The two shares are complements in
// fixed point, so the pair sums to exactly one triangle.
__device__ __forceinline__ bool line_tri_apportion(const MapCore &M, const RawTri &e,
                                                   LaneCount &lc) {
  float t[6];
  int ax, ay;
  small_frame(e, t, ax, ay);
  if (!area_ok(M, tri_area2(t), lc)) return false;
  // the axis whose offsets differ: 0 a vertical line, 1 a horizontal one
  const int x0 = __float_as_int(e.f[0]), x1 = __float_as_int(e.f[2]), x2 = __float_as_int(e.f[4]);
  const int o = ((x0 ^ x1) | (x0 ^ x2)) >= 0;
  const float L = 1.f - (float)(o ? ay : ax);
  const float u0 = o ? t[1] : t[0], u1 = o ? t[3] : t[2], u2 = o ? t[5] : t[4];
  const unsigned low = low_side_u24(u0, u1, u2, L);
  // (pixel indices stay within +-2^29)
  const int hx = e.x + 1 - o, hy = e.y + o;
  const long long idx = (long long)e.y * M.npix + e.x;
  deposit(M, (unsigned)e.x < (unsigned)M.npix && (unsigned)e.y < (unsigned)M.npix_y, idx, low);
  deposit(M, (unsigned)hx < (unsigned)M.npix && (unsigned)hy < (unsigned)M.npix_y,
          idx + (o ? M.npix : 1), MM_U24_ONE - low);
  return true;
}

// A triangle across both grid lines of a 2 x 2 pixel block: the shares left
// of X and below Y from the lone vertex on each line, the lower-left share
// from the quadrant integral; the four pixel shares are differences of
// those in fixed point and add up to exactly one triangle.
__device__ __forceinline__ bool quad_tri_apportion(const MapCore &M, const RawTri &e,
                                                   LaneCount &lc) {
  float t[6];
  int ax, ay;
  small_frame(e, t, ax, ay);
  if (!area_ok(M, tri_area2(t), lc)) return false;
  const float x0 = t[0], y0 = t[1];
  const float d1x = t[2] - t[0], d1y = t[3] - t[1], d2x = t[4] - t[0], d2y = t[5] - t[1];
  const int c0 = (int)floorf(x0 + fminf(0.f, fminf(d1x, d2x)));
  const int r0 = (int)floorf(y0 + fminf(0.f, fminf(d1y, d2y)));
  // the grid lines, relative to the first vertex
  const float X = (float)(c0 + 1) - x0, Y = (float)(r0 + 1) - y0;
  const int vL = (int)low_side_u24(0.f, d1x, d2x, X);
  const int vB = (int)low_side_u24(0.f, d1y, d2y, Y);
  const float lb = quadrant_edge(0.f, 0.f, d1x, d1y, X, Y) +
                   quadrant_edge(d1x, d1y, d2x, d2y, X, Y) +
                   quadrant_edge(d2x, d2y, 0.f, 0.f, X, Y);
  const float A2 = d1x * d2y - d2x * d1y;  // twice the signed area
  const int vLB = (int)frac_to_u24(2.f * lb * rcp_approx_f(A2));
  const int gx = e.x + ax + c0, gy = e.y + ay + r0;
  const bool x0in = (unsigned)gx < (unsigned)M.npix, x1in = (unsigned)(gx + 1) < (unsigned)M.npix;
  const bool y0in = (unsigned)gy < (unsigned)M.npix_y, y1in = (unsigned)(gy + 1) < (unsigned)M.npix_y;
  const long long idx = (long long)gy * M.npix + gx;
  deposit(M, x0in && y0in, idx, (unsigned)vLB);
  deposit(M, x0in && y1in, idx + M.npix, (unsigned)max(vL - vLB, 0));
  deposit(M, x1in && y0in, idx + 1, (unsigned)max(vB - vLB, 0));
  deposit(M, x1in && y1in, idx + M.npix + 1, (unsigned)max((int)MM_U24_ONE - vL - vB + vLB, 0));
  return true;
}

// A larger triangle ready to be dealt out: frame pixel, frame coordinates,
// 2 / signed area and the inverse slope dx/dy of each edge k -> k + 1
// (infinite or NaN for a horizontal edge, which is never used).
struct __align__(16) TriJob {
  int ox, oy;
  float t[6];
  float inv2;
  float k[3];
};

static_assert(sizeof(TriJob) == 48, "TriJob layout");
__device__ __forceinline__ TriJob job_load(const TriJob *p) {
  TriJob J;
  const float4 *w = reinterpret_cast<const float4 *>(p);
  float4 *d = reinterpret_cast<float4 *>(&J);
#pragma unroll
  for (int k = 0; k < 3; k++) d[k] = w[k];
  return J;
}

__device__ __forceinline__ TriJob make_job(const RawTri &e) {
  TriJob J;
  J.ox = e.x;
  J.oy = e.y;
#pragma unroll
  for (int k = 0; k < 6; k++) J.t[k] = e.f[k];
  const float(&t)[6] = e.f;
  // 2 / area from the difference of products rounded once (Kahan's FMA
  // method): the area of a long thin triangle cancels heavily in FP32
  const float pa = t[2] - t[0], pd = t[5] - t[1], pb = t[4] - t[0], pc = t[3] - t[1];
  const float wbc = pb * pc;
  const float a2 = fmaf(pa, pd, -wbc) + fmaf(-pb, pc, wbc);
  J.inv2 = 2.0f / ((a2 != 0.f && isfinite(a2)) ? a2 : tri_area2(t));
#pragma unroll
  for (int k = 0; k < 3; k++)
    J.k[k] = (t[(2 * k + 2) % 6] - t[2 * k]) / (t[(2 * k + 3) % 6] - t[2 * k + 1]);
  return J;
}

// ---------------------------------------------------------------------------
// larger triangles: the whole warp, lanes over pixel rows, then over the
// partially covered pixels of those rows
// ---------------------------------------------------------------------------

// Pixel areas of a larger triangle (Green's theorem on the clamped
// boundary, as above): area(T n [0, 1]^2) is the sum over T's edges of the
// integral over y in [0, 1] of clamp(x(y), 0, 1) along the edge, signed by
// the direction of y.  The clamped y-range of an edge and its x there depend
// only on the pixel row, so they are found once per row (row_pieces) and
// each pixel of the row only shifts them by its column (piece_integral).

// x on edge P -> Q (inverse slope k) at height y, extrapolated from the
// nearer endpoint, which halves the error the rounding of k makes on long
// edges.
__device__ __forceinline__ float edge_x_at(float y, float px, float py, float qx, float qy,
                                          float k) {
  const float d1 = y - py, d2 = y - qy;
  return fabsf(d1) <= fabsf(d2) ? fmaf(d1, k, px) : fmaf(d2, k, qx);
}

// Mean of clamp(x, 0, 1) over x in [a, b] (a piece shifted to its pixel),
// formed from sub-interval lengths so that a nearly vertical piece loses no
// precision; h times it is the piece's integral.
__device__ __forceinline__ float piece_mean(float a, float b) {
  const float w = __saturatef(a), v = __saturatef(b);  // clamp to [0, 1]
  const float in = fmaf(0.5f * (v - w), v + w, fmaxf(b - fmaxf(a, 1.f), 0.f));
  const float len = b - a;
  return len > 0.f ? in * rcp_approx_f(len) : w;
}

// piece_mean of two pieces in packed pairs, each half rounded the same.
__device__ __forceinline__ F2 piece_mean2(F2 a, F2 b) {
  const F2 minus = {-1.f, -1.f};
  const F2 w = {__saturatef(a.x), __saturatef(a.y)}, v = {__saturatef(b.x), __saturatef(b.y)};
  const F2 over = f2_fma(F2{fmaxf(a.x, 1.f), fmaxf(a.y, 1.f)}, minus, b);
  const F2 in = f2_fma(f2_mul(f2_fma(w, minus, v), F2{0.5f, 0.5f}), f2_add(v, w),
                       F2{fmaxf(over.x, 0.f), fmaxf(over.y, 0.f)});
  const F2 len = f2_fma(a, minus, b);
  const F2 m = f2_mul(in, F2{rcp_approx_f(len.x), rcp_approx_f(len.y)});
  return F2{len.x > 0.f ? m.x : w.x, len.y > 0.f ? m.y : w.y};
}

// Frame row r of J: each edge's piece inside the band r <= y <= r + 1
// (x-range [a, b] and signed height h, all zero when it misses the band),
// the columns [c0, c1] the band meets (widened by a small margin; extra
// columns get zero area) and the fully covered run [fa, fb) (empty when
// fa >= fb).  A pixel of the row is fully covered when the band lies within
// T's height and the pixel between T's two sides; the sides are the pieces
// that fall and those that rise when T is traversed anticlockwise, and each
// (T convex) comes closest to the other side at an end of a piece.
__device__ __forceinline__ void row_pieces(const TriJob &J, int r, float (&a)[3], float (&b)[3],
                                           float (&h)[3], int &c0, int &c1, int &fa, int &fb) {
  const float y0 = (float)r, y1 = (float)(r + 1);
  float lo = 3.0e38f, hi = -3.0e38f;      // the band's extent
  float left = -3.0e38f, right = 3.0e38f;  // furthest points of the two sides
#pragma unroll
  for (int e = 0; e < 3; e++) {
    const float px = J.t[2 * e], py = J.t[2 * e + 1];
    const float qx = J.t[(2 * e + 2) % 6], qy = J.t[(2 * e + 3) % 6];
    const float ys = fminf(fmaxf(py, y0), y1), ye = fminf(fmaxf(qy, y0), y1);
    const float xs = edge_x_at(ys, px, py, qx, qy, J.k[e]);
    const float xe = edge_x_at(ye, px, py, qx, qy, J.k[e]);
    const bool cross = ye != ys;
    a[e] = cross ? fminf(xs, xe) : 0.f;
    b[e] = cross ? fmaxf(xs, xe) : 0.f;
    h[e] = cross ? ye - ys : 0.f;
    if (cross) {
      lo = fminf(lo, a[e]);
      hi = fmaxf(hi, b[e]);
      if ((h[e] > 0.f) == (J.inv2 > 0.f))
        right = fminf(right, a[e]);
      else
        left = fmaxf(left, b[e]);
    }
  }
  const float ymin = fminf(J.t[1], fminf(J.t[3], J.t[5]));
  const float ymax = fmaxf(J.t[1], fmaxf(J.t[3], J.t[5]));
  // (conversions saturate: the caller clamps to the map before any arithmetic)
  const float eps = 1e-3f;
  c0 = __float2int_rd(lo - eps);
  c1 = __float2int_rd(hi + eps);
  const bool full = ymin <= y0 && ymax >= y1;
  fa = full ? __float2int_ru(left + eps) : 1;
  fb = full ? __float2int_rd(right - eps) : 1;
}

// Dealing tasks from a warp's lanes: lane j owns n_j tasks, numbered
// [ex_j, ex_j + n_j) in lane order (ex the exclusive scan), and the lanes
// with n_j > 0 are ranked by slot = their rank among them.  For the 32 tasks
// [base, base + 32), the owner of task base + l has slot
//   |{starts ex_j <= base + l}| - 1,
// the rounds' counts added up as they go: one OR-reduction of start bits and
// two popcounts, no chain of shuffles
// (`first`: slots of the rounds before, advanced for the next one).
__device__ __forceinline__ int deal_owner_slot(int n, int ex, int base, int lane, int &first) {
  const unsigned d = (unsigned)(ex - base);
  const unsigned bit = (n > 0 && d < 32u) ? (1u << d) : 0u;
  const unsigned starts = __reduce_or_sync(0xffffffffu, bit);
  const int slot = first - 1 + __popc(starts & ((2u << lane) - 1u));
  first += __popc(starts);
  return slot;
}

__device__ __forceinline__ int warp_incl_scan(int v, int lane) {
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, v, d);
    if (lane >= d) v += u;
  }
  return v;
}

// The pixel rows of one round of a larger-triangle batch, by slot (rank
// among the rows with partially covered pixels), shared by the lanes that
// measure their partially covered pixels.  Per edge: its piece [a, b] in the
// row band, x relative to column c0, with height times 2/area (h), so that
// the weighted sum of piece means is the pixel's share.  Then the
// first column of the fully covered run relative to c0 (INT_MAX: none) and
// its length, the address of the map's pixel (c0, row), and the row's first
// pixel task.  One array per 16-byte word: consecutive slots fall on distinct
// banks without padding.
struct RowRecs {
  float4 piece[32];   // a0, a1, b0, b1
  float4 height[32];  // h0, h1, a2, b2
  int4 pixel[32];     // h2, run, address
  int2 task[32];      // run length, first task
  int2 tri[32];       // triangles with rows: lane, first row less first row task
};

// Add v to the 64-bit word at global address `at` (an address kept as an
// integer would otherwise make this a generic atomic that returns a value:
// the second pass was 20 % slower with it).
__device__ __forceinline__ void red_add(unsigned long long at, unsigned long long v) {
  asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(at), "l"(v) : "memory");
}

// Partially covered pixel number `task` of a round's rows, owned by the row
// in slot o.  The first two pieces are measured in packed pairs.
__device__ __forceinline__ void pixel_task(const MapAcc &M, const RowRecs *rr, int o, int task,
                                           int ptotal) {
  if (task < ptotal) {
    const float4 p0 = rr->piece[o], p1 = rr->height[o];
    const int4 p2 = rr->pixel[o];
    const int2 p3 = rr->task[o];
    int c = task - p3.y;
    if (c >= p2.y) c += p3.x;
    const float nc = -(float)c;
    const F2 nc2 = {nc, nc};
    const F2 m01 =
        piece_mean2(f2_add(F2{p0.x, p0.y}, nc2), f2_add(F2{p0.z, p0.w}, nc2));
    float sh = p1.x * m01.x;
    sh = fmaf(p1.y, m01.y, sh);
    sh = fmaf(__int_as_float(p2.x), piece_mean(p1.z + nc, p1.w + nc), sh);
    // the row and its columns lie in the map (clamped when the row was set up)
    const unsigned long long at =
        ((unsigned long long)(unsigned)p2.z | ((unsigned long long)(unsigned)p2.w << 32)) +
        (long long)c * 8;
    const unsigned u = frac_to_u24(sh);
    if (u && MM_INDEX_OK(M.err, (long long)(at - __cvta_generic_to_global(M.acc)) / 8,
                         (long long)M.npix * M.npix_y))
      red_add(at, (unsigned long long)u << 8);
  }
}

// Instruction-bound: per 32 pixels 88 instructions (deal, four loads of the
// row's record, three piece means, one reduction), per 32 rows 228, and 169 to
// set up 32 triangles.  The first two pieces' means in packed pairs, the pixel's
// address and the run's gap prepared once a row, the row's run from its two
// sides, and owners found from one reduction took the second pass of the 2000^2
// map from 12.25 to 10.44 ms, bit for bit the same.  Its L2 reductions run at
// 1.3e11/s (that map at one ray a pixel), 60 % of the measured scattered rate.
//
// The nb (<= 32) triangles q[0..nb) (warp shared memory) spanning more than
// 2 x 2 pixels.  Their pixel rows within the map are dealt out to the lanes,
// 32 at a time; a row adds 1/|area| to its fully covered run through the
// row difference array and records its edge pieces in rr[lane]; the
// partially covered pixels of those 32 rows are then dealt out one per lane.
// Work is proportional to the perimeter, and the lanes stay busy however
// the rows differ.  Call with all 32 lanes.
__device__ __forceinline__ void warp_tri_jobs(unsigned long long *acc,
                                                  unsigned long long *span, int npix,
                                                  int npix_y, unsigned *err,
                                                  const TriJob *q, int nb, RowRecs *rr,
                                                  int lane, int row_lo, int row_hi) {
  const MapAcc M = {acc, span, npix, npix_y, err};
  int rl = 0, nrows = 0;
  if (lane < nb) {
    const TriJob &J = q[lane];
    const float ymin = fminf(J.t[1], fminf(J.t[3], J.t[5]));
    const float ymax = fmaxf(J.t[1], fmaxf(J.t[3], J.t[5]));
    const int r0 = max((int)floorf(fmaxf(ymin, -1.0e9f)), row_lo - J.oy);
    const int r1 = min((int)floorf(fminf(ymax, 1.0e9f)), row_hi - 1 - J.oy);
    rl = r0;
    nrows = r1 >= r0 ? r1 - r0 + 1 : 0;
  }
  const int incl = warp_incl_scan(nrows, lane);
  const int excl = incl - nrows;
  const int total = __shfl_sync(0xffffffffu, incl, 31);
  const unsigned with_rows = __ballot_sync(0xffffffffu, nrows > 0);
  if (nrows > 0) rr->tri[__popc(with_rows & ((1u << lane) - 1u))] = make_int2(lane, rl - excl);
  __syncwarp();
  int row_first = 0;
#pragma unroll 1
  for (int base = 0; base < total; base += 32) {
    const int task = base + lane;
    const int o = deal_owner_slot(nrows, excl, base, lane, row_first);
    int np = 0, c0 = 0, gx = 0, gy = 0, run = INT_MAX, run_len = 0;
    float pa[3], pb[3], ph[3], inv2 = 0.f;
    if (task < total) {
      const int2 t = rr->tri[o];
      const TriJob J = job_load(q + t.x);
      int c1, fa, fb;
      row_pieces(J, t.y + task, pa, pb, ph, c0, c1, fa, fb);
      inv2 = J.inv2;
      gy = J.oy + t.y + task;
      c0 = max(c0, -J.ox);
      c1 = min(c1, M.npix - 1 - J.ox);
      fa = max(fa, c0);
      fb = min(fb, c1 + 1);
      gx = J.ox + c0;
      if (c0 <= c1) {
        np = c1 - c0 + 1;
        if (fa < fb) {
          run = fa - c0;
          run_len = fb - fa;
          np -= run_len;
          // a fully covered pixel holds 1/|area| of the triangle (< 1 when any does)
          const unsigned long long full = frac_to_fixed(fabsf(inv2));
          const long long at = (long long)gy * (M.npix + 1) + (gx + run);
          const long long sn = (long long)M.npix_y * (M.npix + 1);
          if (MM_INDEX_OK(M.err, at, sn) && MM_INDEX_OK(M.err, at + run_len, sn)) {
            atomicAdd(&M.span[at], full);
            atomicAdd(&M.span[at + run_len], 0ull - full);
          }
        }
      }
    }
    // the partially covered pixels of these 32 rows: records by slot
    const int pincl = warp_incl_scan(np, lane);
    const int pexcl = pincl - np;
    const int ptotal = __shfl_sync(0xffffffffu, pincl, 31);
    const int slot = __popc(__ballot_sync(0xffffffffu, np > 0) & ((1u << lane) - 1u));
    __syncwarp();  // the previous round's readers are done with the records
    if (np > 0) {
      const float fc0 = (float)c0;
#pragma unroll
      for (int e = 0; e < 3; e++) {
        // x relative to column c0 (zero-height pieces stay zero)
        pa[e] = ph[e] != 0.f ? pa[e] - fc0 : 0.f;
        pb[e] = ph[e] != 0.f ? pb[e] - fc0 : 0.f;
        ph[e] *= inv2;
      }
      const unsigned long long at =
          __cvta_generic_to_global(M.acc + ((long long)gy * M.npix + gx));
      rr->piece[slot] = make_float4(pa[0], pa[1], pb[0], pb[1]);
      rr->height[slot] = make_float4(ph[0], ph[1], pa[2], pb[2]);
      rr->pixel[slot] = make_int4(__float_as_int(ph[2]), run, (int)(unsigned)at,
                                  (int)(unsigned)(at >> 32));
      rr->task[slot] = make_int2(run_len, pexcl);
    }
    __syncwarp();
    int px_first = 0;
#pragma unroll 1
    for (int pbase = 0; pbase < ptotal; pbase += 32)
      pixel_task(M, rr, deal_owner_slot(np, pexcl, pbase, lane, px_first), pbase + lane, ptotal);
  }
  __syncwarp();
}

// ---------------------------------------------------------------------------
// a warp's queues
// ---------------------------------------------------------------------------

// Map statistics (MapDev::stat): [0] dropped, [1] multi-pixel (clipped) in
// the map, [2] within a 2 x 2 box crossing both grid lines, [3] box of at
// most MM_MED_PIXELS map pixels, [4] larger, [5] two pixels split by one
// grid line, [6] vertex rows not computed because culling proved them beyond
// the map, [7] near-critical.
#define MM_N_COUNTERS 8
enum { ST_DROPPED, ST_CLIPPED, ST_QUAD, ST_BOX, ST_ROWS, ST_LINE, ST_CULLED, ST_CRITICAL };

// A row of cells adds at most 62 triangles (two per cell of a warp's 31) to
// the queues, which are emptied to fewer than 32 of a kind after each row:
// the line and quad queues share one array from its two ends.
#define MM_SMALL_QUEUE (31 + 31 + 62)
#define MM_BIG_QUEUE (31 + 62)

// Shared memory of one warp.  A batch of larger triangles dealt out here has
// its row records and jobs over the line and quad queues (emptied first).
// 8000 bytes: three blocks of the shooting kernel then leave the L1 60 KB in
// place of 28 (shared memory is taken in steps, 196 and 228 KB the last), and
// 85 % of the records' sectors hit it in place of 60 %: first pass of the
// 2000^2 map 11.97 -> 11.48 ms, 12 maps in a batch 35.1 -> 32.3 ms.
struct __align__(16) WarpSmem {
  union {
    RawTri small[MM_SMALL_QUEUE];
    struct {
      RowRecs rows;
      TriJob job[32];
    };
  };
  RawTri big[MM_BIG_QUEUE];
  Vtx row[32];                    // the last vertex row, one vertex per lane
  Vtx next[32];                   // the next one, where it was shot with it
  unsigned count[MM_N_COUNTERS];  // (dropped and critical are per lane, LaneCount)
};
#define MM_SHOOT_SMEM_BYTES (8 * sizeof(WarpSmem))  // 8 warps per block

struct WarpQueues {
  WarpSmem *s;
  int line, quad, big;  // triangles waiting (warp-uniform)
};

// Apportion or queue one triangle (a, b, c) of each lane (`on`: the lane
// has one, not wholly beyond one edge of the map).  A triangle inside one
// pixel is finished here.
__device__ __forceinline__ void tri_scan(const MapCore &M, WarpQueues &q, const Vtx &a,
                                         const Vtx &b, const Vtx &c, bool on, RunAcc &ra,
                                         LaneCount &lc, int lane) {
  // the pixel box from the vertices' pixels (a vertex's pixel is the floor
  // of its coordinate, MM_VTX_INVALID = INT_MIN below any valid one)
  const int xlo = min(a.px, min(b.px, c.px)), xhi = max(a.px, max(b.px, c.px));
  const int ylo = min(a.py, min(b.py, c.py)), yhi = max(a.py, max(b.py, c.py));
  if (on && xlo == MM_VTX_INVALID) {
    lc.dropped++;
    on = false;
  }
  const int sx = xhi - xlo, sy = yhi - ylo;
  const unsigned span = (unsigned)(sx | sy);
  const bool one = on && span == 0u;
  const bool line = on && span == 1u && !(sx & sy);
  const bool quad = on && span == 1u && (sx & sy);
  const bool big = on && span > 1u;
  const unsigned ml = __ballot_sync(0xffffffffu, line), mq = __ballot_sync(0xffffffffu, quad),
                 mb = __ballot_sync(0xffffffffu, big);
  const unsigned below = (1u << lane) - 1u;
  if (one) {
    // all three vertices in one (closed) map pixel: all of the area is there
    const float t[6] = {a.fx, a.fy, b.fx, b.fy, c.fx, c.fy};
    if (area_ok(M, tri_area2(t), lc))
      run_add<MM_FIX_ONE>(M, ra, a.px, a.py);
  } else if (line || quad) {
    const int k = line ? q.line + __popc(ml & below)
                       : MM_SMALL_QUEUE - 1 - q.quad - __popc(mq & below);
    raw_store(q.s->small + k, xlo, ylo, with_offset(a.fx, a.px, xlo), with_offset(a.fy, a.py, ylo),
              with_offset(b.fx, b.px, xlo), with_offset(b.fy, b.py, ylo),
              with_offset(c.fx, c.px, xlo), with_offset(c.fy, c.py, ylo));
  } else if (big) {
    // the box within the map (indices within +-2^29)
    const int w = min(xhi, M.npix - 1) - max(xlo, 0) + 1;
    const int h = min(yhi, M.npix_y - 1) - max(ylo, 0) + 1;
    const bool med = (long long)w * h <= MM_MED_PIXELS;
    // pixel indices stay within +-2^29, so differences fit in 32 bits
    raw_store(q.s->big + q.big + __popc(mb & below), a.px, a.py, med ? -a.fx : a.fx, a.fy,
              (float)(b.px - a.px) + b.fx, (float)(b.py - a.py) + b.fy,
              (float)(c.px - a.px) + c.fx, (float)(c.py - a.py) + c.fy);
  }
  q.line += __popc(ml);
  q.quad += __popc(mq);
  q.big += __popc(mb);
  __syncwarp();
}

// Empty the queues down to fewer than 32 triangles of a kind (`flush`:
// entirely).  Batches of larger triangles go to the map's device queue for
// the larger-triangle kernel (k_big_ipm), which deals them out at a higher
// occupancy than this kernel's; a batch that does not fit is dealt out here,
// its reserved queue slots filled with triangles without pixel rows.
__device__ __forceinline__ void share_out(const MapCore &M, WarpQueues &q, bool flush,
                                          LaneCount &lc, int lane) {
  if (!flush && ((q.line | q.quad | q.big) & ~31) == 0) return;
  int deal = 0;  // jobs set up to be dealt out here
#pragma unroll 1
  while (true) {
    const bool rest = flush || deal > 0;
#pragma unroll 1
    while (q.line >= 32 || (rest && q.line > 0)) {
      const int nb = min(q.line, 32);
      q.line -= nb;
      const bool done =
          lane < nb && line_tri_apportion(M, raw_load(q.s->small + q.line + lane), lc);
      const unsigned n = __popc(__ballot_sync(0xffffffffu, done));
      if (lane == 0) q.s->count[ST_LINE] += n;
    }
#pragma unroll 1
    while (q.quad >= 32 || (rest && q.quad > 0)) {
      const int nb = min(q.quad, 32);
      q.quad -= nb;
      const bool done =
          lane < nb &&
          quad_tri_apportion(M, raw_load(q.s->small + MM_SMALL_QUEUE - 1 - q.quad - lane), lc);
      const unsigned n = __popc(__ballot_sync(0xffffffffu, done));
      if (lane == 0) q.s->count[ST_QUAD] += n;
    }
    __syncwarp();
    if (deal > 0) {
      if (lane < deal) q.s->job[lane] = make_job(raw_load(q.s->big + q.big + lane));
      __syncwarp();
      warp_tri_jobs(M.acc, M.span, M.npix, M.npix_y, M.err, q.s->job, deal, &q.s->rows, lane, 0,
                    M.npix_y);
      deal = 0;
    }
    if (!(q.big >= 32 || (flush && q.big > 0))) break;
    const int nb = min(q.big, 32);
    q.big -= nb;
    RawTri e;
    e.x = e.y = -(1 << 30);  // no pixel rows: a frame far below any map
#pragma unroll
    for (int k = 0; k < 6; k++) e.f[k] = 0.f;
    bool ok = false, med = false;
    if (lane < nb) {
      RawTri t = raw_load(q.s->big + q.big + lane);
      med = __float_as_int(t.f[0]) < 0;
      t.f[0] = fabsf(t.f[0]);
      ok = area_ok(M, tri_area2(t.f), lc);
      if (ok) e = t;
    }
    const unsigned m_ok = __ballot_sync(0xffffffffu, ok);
    const unsigned m_med = __ballot_sync(0xffffffffu, ok && med);
    if (lane == 0) {
      q.s->count[ST_BOX] += __popc(m_med);
      q.s->count[ST_ROWS] += __popc(m_ok & ~m_med);
    }
    unsigned long long base = 0;
    bool fits = false;
    if (M.bigq_cap > 0) {
      if (lane == 0) base = atomicAdd(M.bigq_n, (unsigned long long)nb);
      base = __shfl_sync(0xffffffffu, base, 0);
      fits = base + nb <= (unsigned long long)M.bigq_cap;
      if (!fits && lane < nb && base + lane < (unsigned long long)M.bigq_cap)
        raw_store(M.bigq + base + lane, -(1 << 30), -(1 << 30), 0.f, 0.f, 0.f, 0.f, 0.f, 0.f);
    }
    if (fits) {
      if (lane < nb)
        raw_store(M.bigq + base + lane, e.x, e.y, e.f[0], e.f[1], e.f[2], e.f[3], e.f[4], e.f[5]);
      __syncwarp();
    } else {
      // (back to its place above the queue's end until the others are empty)
      if (lane < nb)
        raw_store(q.s->big + q.big + lane, e.x, e.y, e.f[0], e.f[1], e.f[2], e.f[3], e.f[4],
                  e.f[5]);
      deal = nb;
    }
  }
}

__device__ __forceinline__ void counts_clear(WarpSmem *s, int lane) {
  if (lane < MM_N_COUNTERS) s->count[lane] = 0u;
  __syncwarp();
}

// Add the warp's counters to the map's statistics and clear them.
__device__ __forceinline__ void counts_flush(const MapCore &M, WarpSmem *s, LaneCount &lc,
                                             int lane) {
  const unsigned d = __reduce_add_sync(0xffffffffu, lc.dropped);
  const unsigned c = __reduce_add_sync(0xffffffffu, lc.critical);
  lc = LaneCount{0u, 0u};
  __syncwarp();
  if (lane < MM_N_COUNTERS) {
    unsigned v = s->count[lane];
    if (lane == ST_DROPPED) v = d;
    if (lane == ST_CRITICAL) v = c;
    // every multi-pixel triangle is of one of the four kinds
    if (lane == ST_CLIPPED)
      v = s->count[ST_QUAD] + s->count[ST_BOX] + s->count[ST_ROWS] + s->count[ST_LINE];
    if (v) atomicAdd(&M.stat[lane], (unsigned long long)v);
  }
  __syncwarp();
  if (lane < MM_N_COUNTERS) s->count[lane] = 0u;
  __syncwarp();
}

}  // namespace mm
