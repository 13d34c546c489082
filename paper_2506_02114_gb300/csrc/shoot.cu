// Fused ray deflection + inverse polygon mapping (the hot kernel), the
// normalisation kernel and the deflection probe.
//
// Per ray vertex (Sec. 3.3, App. C): the vertex's leaf supplies
//   - the near-field stars (the leaf and its neighbours, at most leaf_size):
//     direct sum of m / conj(z - z_i);
//   - the local (Taylor) expansion of the far field about the leaf centre:
//     alpha_far = conj(dpsi/dz), dpsi/dz = (1/L) sum_l l c_l zeta^(l-1);
//   - the FP64 image of the leaf centre W_c (macro model + sheet + far field
//     at the centre), so that only small, centre-relative quantities are
//     evaluated in FP32 per ray.
// The lens equation (Sec. 2.2, circular sheet of Sec. 3.1) then gives
//   w - W_c = (1-kappa+kappa_*) d + gamma conj(d) - alpha_near
//             - conj(sum_{l>=2} l c_l zeta^(l-1) / L),   d = z - z_c.
#include <algorithm>

#include "ipm.cuh"
#include "mm_kernels.h"

namespace mm {

__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Record of the sub-cell of the active leaf containing finest-level cell
// (cx, cy); -1 if none.
__device__ __forceinline__ int lookup_leaf(const MapCore &M, int cx, int cy) {
  int gx = (cx >> M.gshift) - M.gx0, gy = (cy >> M.gshift) - M.gy0;
  if (gx < 0 || gy < 0 || gx >= M.gw || gy >= M.gh) return -1;
  int e = __ldg(&M.grid[(int64_t)gy * M.gw + gx]);
  if (e >= 0) return e;
  int node = -e - 1;
#pragma unroll 1
  for (int lvl = M.glevel + 1; lvl <= MM_DMAX; lvl++) {
    int fc = __ldg(&M.first_child[node]);
    if (fc < 0) break;
    int sh = MM_DMAX - lvl;
    node = fc + (((cx >> sh) & 1) | (((cy >> sh) & 1) << 1));
  }
  const int a = __ldg(&M.node_active[node]);
  if (a < 0) return -1;
  // the host keeps every leaf level + sub <= MM_DMAX
  const int sh = MM_DMAX - __ldg(&M.node_level[node]) - M.sub, mask = (1 << M.sub) - 1;
  return (a << (2 * M.sub)) + (((cy >> sh) & mask) << M.sub) + ((cx >> sh) & mask);
}

// The records of vertex row j in every lane's column (lookup_leaf), whether
// the lane's record can prove a vertex beyond the map at all, and the first
// row after j that may lie in other records: a grid entry that names a record
// holds for every row of its grid row (the lanes' columns are fixed), so the
// rows up to `j_same` need no lookup.  Rows up to je.
__device__ __forceinline__ int lookup_rows(const MapCore &M, int cx, int j, int je, int lane,
                                           bool vvalid, int &j_same, bool &c_cull) {
  const int cy = __ldg(&M.row_cell[j]);
  const int gy = (cy >> M.gshift) - M.gy0, gx = (cx >> M.gshift) - M.gx0;
  const int ahead = __ldg(&M.row_cell[min(j + 1 + lane, je)]);
  int e = -1;
  if (gx >= 0 && gy >= 0 && gx < M.gw && gy < M.gh) e = __ldg(&M.grid[(int64_t)gy * M.gw + gx]);
  const bool direct = e >= 0;
  if (!direct) e = lookup_leaf(M, cx, cy);
  c_cull = e >= 0 && __ldg(&M.leaf[e].cull_side) != MM_CULL_NONE;
  j_same = j + 1;
  if (__all_sync(0xffffffffu, direct || !vvalid)) {
    const unsigned other = __ballot_sync(0xffffffffu, (ahead >> M.gshift) - M.gy0 != gy);
    j_same += other ? __ffs(other) - 1 : 32;
  }
  return e;
}

// Far field f = sum_{k>=0} e_k zeta^(k+1), e_k = (k+2) c_(k+2) / (L delta), as
// zeta E(w) + w O(w), w = zeta^2, E and O the even and odd k: two independent
// Horner chains as one chain of packed pairs, one (e_2j, e_2j+1) pair per
// 16-byte load.  State of the chains at one point.
struct FarField {
  float zx, zy, wx, wy;
  F2 re, im;  // (E, O)
};
__device__ __forceinline__ void far_start(FarField &f, float zx, float zy, float4 c) {
  f.zx = zx;
  f.zy = zy;
  f.wx = fmaf(zx, zx, -zy * zy);
  f.wy = 2.f * zx * zy;
  f.re = F2{c.x, c.y};
  f.im = F2{c.z, c.w};
}
// (E, O) <- (E, O) w + c in complex arithmetic.
__device__ __forceinline__ void far_step(FarField &f, float4 c) {
  const F2 wx = {f.wx, f.wx}, wy = {f.wy, f.wy}, nwy = {-f.wy, -f.wy};
  const F2 re = f2_fma(f.re, wx, f2_fma(f.im, nwy, F2{c.x, c.y}));
  f.im = f2_fma(f.re, wy, f2_fma(f.im, wx, F2{c.z, c.w}));
  f.re = re;
}
__device__ __forceinline__ void far_end(const FarField &f, float &fr, float &fi) {
  const float Er = f.re.x, Or = f.re.y, Ei = f.im.x, Oi = f.im.y;
  fr = fmaf(f.zx, Er, fmaf(-f.zy, Ei, fmaf(f.wx, Or, -f.wy * Oi)));
  fi = fmaf(f.zx, Ei, fmaf(f.zy, Er, fmaf(f.wx, Oi, f.wy * Or)));
}

// The coefficient pairs after the last, highest first, each applied to N
// points; loaded G at a time, so that their latencies overlap (the usual 15
// terms have six after the first pair).  G = 3 in the polygon-mapping kernel,
// which has no registers for more and whose loop has to fit the instruction
// cache; 6 in k_shoot_irs (2.64 ms against 2.72 with 3, 1537^2 map).
template <int G, int N>
__device__ __forceinline__ void far_chain(FarField (&f)[N], const float4 *e, int npair) {
  int j = npair - 2;
#pragma unroll 1
  for (; j >= G - 1; j -= G) {
    float4 cc[G];
#pragma unroll
    for (int q = 0; q < G; q++) cc[q] = __ldg(e + j - q);
#pragma unroll
    for (int q = 0; q < G; q++)
#pragma unroll
      for (int k = 0; k < N; k++) far_step(f[k], cc[q]);
  }
#pragma unroll 1
  for (; j >= 0; j--) {
    const float4 c = __ldg(e + j);
#pragma unroll
    for (int k = 0; k < N; k++) far_step(f[k], c);
  }
}

// A source position (u, v) in pixels relative to pixel (Ui, Vi) in canonical
// form.
__device__ __forceinline__ Vtx pixel_form(bool ok, float u, float v, int Ui, int Vi) {
  Vtx out;
  if (!ok || !isfinite(u) || !isfinite(v)) {
    out.px = MM_VTX_INVALID;
    out.py = MM_VTX_INVALID;
    out.fx = 0.f;
    out.fy = 0.f;
    return out;
  }
  const float lim = 268435456.0f;  // 2^28 pixels: far outside any map
  u = fminf(fmaxf(u, -lim), lim);
  v = fminf(fmaxf(v, -lim), lim);
  float flu = floorf(u), flv = floorf(v);
  out.px = Ui + (int)flu;
  out.py = Vi + (int)flv;
  out.fx = u - flu;
  out.fy = v - flv;
  return out;
}

// Source-plane position of grid point (i + ti, j + tj) in pixel units:
// returns the integer pixel and the fraction.  ti = tj = 0 for ray vertices.
template <bool SQUARE, bool FRAC, int G = 3>
__device__ __forceinline__ Vtx shoot_point(const MapCore &M, int leaf, int i, int j,
                                           float ti, float tj, bool valid) {
  const int4 *rp = reinterpret_cast<const int4 *>(M.leaf + (leaf < 0 ? 0 : leaf));
  int4 q0 = __ldg(rp), q1 = __ldg(rp + 1), q2 = __ldg(rp + 2), q3 = __ldg(rp + 3);
  const int i_ref = q0.x, j_ref = q0.y;
  const float fcx = __int_as_float(q0.z), fcy = __int_as_float(q0.w);
  const int Ui = q1.x, Vi = q1.y;
  const float Uf = __int_as_float(q1.z), Vf = __int_as_float(q1.w);
  const float zsx = __int_as_float(q2.x), zsy = __int_as_float(q2.y);
  const int near_off = q2.z, near_cnt = (leaf < 0) ? 0 : q2.w;
  const int coef_off = q3.x;

  // vertex position relative to the reference vertex, in grid units (exact
  // integers), and relative to the leaf centre
  const float fi = (float)(i - i_ref), fj = (float)(j - j_ref);
  float gx = fi - fcx, gy = fj - fcy;
  if (FRAC) {
    gx += ti;
    gy += tj;
  }

  // near field: S = sum m g / |g|^2 in grid units (|g|^2 = gx^2 + rho gy^2)
  // two stars per iteration into two accumulator pairs (independent chains)
  float Sx = 0.f, Sy = 0.f, Sx2 = 0.f, Sy2 = 0.f;
  const int maxcnt = __reduce_max_sync(0xffffffffu, near_cnt);
  const float4 *np_ = reinterpret_cast<const float4 *>(M.near_pos) + near_off;
  const float *nm_ = M.near_m + near_off;
  // a lane with fewer stars than the warp's most runs stand-ins whose
  // contribution is selected away after the reciprocal (a stand-in on a
  // vertex would otherwise give 0 x 1/0 = NaN there)
  int k = 0;
#pragma unroll 1
  for (; k + 1 < maxcnt; k += 2) {
    const bool a0 = k < near_cnt, a1 = k + 1 < near_cnt;
    const float4 s0 = a0 ? __ldg(np_ + k) : make_float4(0.f, 1.f, 0.f, 0.f);
    const float4 s1 = a1 ? __ldg(np_ + k + 1) : make_float4(0.f, 1.f, 0.f, 0.f);
    const float m0 = a0 ? __ldg(nm_ + k) : 0.f, m1 = a1 ? __ldg(nm_ + k + 1) : 0.f;
    float dx0 = (fi - s0.x) - s0.y, dy0 = (fj - s0.z) - s0.w;
    float dx1 = (fi - s1.x) - s1.y, dy1 = (fj - s1.z) - s1.w;
    if (FRAC) {
      dx0 += ti;
      dy0 += tj;
      dx1 += ti;
      dy1 += tj;
    }
    const float r0 = SQUARE ? fmaf(dx0, dx0, dy0 * dy0) : fmaf(dx0, dx0, M.rho * dy0 * dy0);
    const float r1 = SQUARE ? fmaf(dx1, dx1, dy1 * dy1) : fmaf(dx1, dx1, M.rho * dy1 * dy1);
    const float q0 = a0 ? m0 * rcp_approx(r0) : 0.f, q1 = a1 ? m1 * rcp_approx(r1) : 0.f;
    Sx = fmaf(q0, dx0, Sx);
    Sy = fmaf(q0, dy0, Sy);
    Sx2 = fmaf(q1, dx1, Sx2);
    Sy2 = fmaf(q1, dy1, Sy2);
  }
  if (k < maxcnt && k < near_cnt) {
    const float4 s0 = __ldg(np_ + k);
    const float m0 = __ldg(nm_ + k);
    float dx0 = (fi - s0.x) - s0.y, dy0 = (fj - s0.z) - s0.w;
    if (FRAC) {
      dx0 += ti;
      dy0 += tj;
    }
    const float r0 = SQUARE ? fmaf(dx0, dx0, dy0 * dy0) : fmaf(dx0, dx0, M.rho * dy0 * dy0);
    const float q0 = m0 * rcp_approx(r0);
    Sx = fmaf(q0, dx0, Sx);
    Sy = fmaf(q0, dy0, Sy);
  }
  Sx += Sx2;
  Sy += Sy2;

  float fr = 0.f, fim = 0.f;
  const int npair = M.p >> 1;
  if (npair >= 1 && leaf >= 0) {
    const float4 *e = reinterpret_cast<const float4 *>(M.coef + coef_off);
    FarField f[1];
    far_start(f[0], gx * zsx, gy * zsy, __ldg(e + (npair - 1)));
    far_chain<G>(f, e, npair);
    far_end(f[0], fr, fim);
  }

  const float u = Uf + (fmaf(M.A1, gx, -Sx * M.sx) - fr);
  const float v = Vf + (fmaf(M.A2, gy, -Sy * M.sy) + fim);
  return pixel_form(valid && leaf >= 0, u, v, Ui, Vi);
}

// Rows j and j + 1 of column i, both in record `leaf`: the same steps as
// shoot_point with the two rows as packed pairs, bit for bit the same
// vertices.  The record, its stars and coefficients are loaded once, a star's
// x distance is formed once, and most of the rest issues one instruction for
// both rows (k_shoot_irs on the 1537^2 map 3.28 -> 2.64 ms).
template <bool SQUARE, int G>
__device__ __forceinline__ void shoot_rows2(const MapCore &M, int leaf, int i, int j, bool valid,
                                            Vtx &out0, Vtx &out1) {
  const int4 *rp = reinterpret_cast<const int4 *>(M.leaf + (leaf < 0 ? 0 : leaf));
  const int4 q0 = __ldg(rp), q1 = __ldg(rp + 1), q2 = __ldg(rp + 2), q3 = __ldg(rp + 3);
  const int near_cnt = (leaf < 0) ? 0 : q2.w;
  const float fi = (float)(i - q0.x);
  const F2 fj = {(float)(j - q0.y), (float)(j + 1 - q0.y)};
  const float gx = fi - __int_as_float(q0.z);
  const float nfcy = -__int_as_float(q0.w);
  const F2 gy = f2_add(fj, F2{nfcy, nfcy});

  // near field, two stars per iteration into two accumulator pairs
  F2 Sx = {0.f, 0.f}, Sy = {0.f, 0.f}, Sx2 = {0.f, 0.f}, Sy2 = {0.f, 0.f};
  const int maxcnt = __reduce_max_sync(0xffffffffu, near_cnt);
  const float4 *np_ = reinterpret_cast<const float4 *>(M.near_pos) + q2.z;
  const float *nm_ = M.near_m + q2.z;
  auto star = [&](bool on, int k, F2 &ax, F2 &ay) {
    const float4 s = on ? __ldg(np_ + k) : make_float4(0.f, 1.f, 0.f, 0.f);
    const float m = on ? __ldg(nm_ + k) : 0.f;
    const float dx = (fi - s.x) - s.y;
    const F2 dx2 = {dx, dx};
    const F2 dy = f2_add(f2_add(fj, F2{-s.z, -s.z}), F2{-s.w, -s.w});
    const F2 yy = SQUARE ? f2_mul(dy, dy) : f2_mul(f2_mul(F2{M.rho, M.rho}, dy), dy);
    const F2 r = f2_fma(dx2, dx2, yy);
    F2 q = f2_mul(F2{m, m}, F2{rcp_approx(r.x), rcp_approx(r.y)});
    q = F2{on ? q.x : 0.f, on ? q.y : 0.f};
    ax = f2_fma(q, dx2, ax);
    ay = f2_fma(q, dy, ay);
  };
  int k = 0;
#pragma unroll 1
  for (; k < maxcnt; k += 2) {
    star(k < near_cnt, k, Sx, Sy);
    star(k + 1 < near_cnt, k + 1, Sx2, Sy2);
  }
  Sx = f2_add(Sx, Sx2);
  Sy = f2_add(Sy, Sy2);

  float fr[2] = {0.f, 0.f}, fm[2] = {0.f, 0.f};
  const int npair = M.p >> 1;
  if (npair >= 1 && leaf >= 0) {
    const float4 *e = reinterpret_cast<const float4 *>(M.coef + q3.x);
    const float4 c = __ldg(e + (npair - 1));
    const float zx = gx * __int_as_float(q2.x), zsy = __int_as_float(q2.y);
    FarField f[2];
    far_start(f[0], zx, gy.x * zsy, c);
    far_start(f[1], zx, gy.y * zsy, c);
    far_chain<G>(f, e, npair);
    far_end(f[0], fr[0], fm[0]);
    far_end(f[1], fr[1], fm[1]);
  }
  const float Uf = __int_as_float(q1.z), Vf = __int_as_float(q1.w);
  const bool ok = valid && leaf >= 0;
  out0 = pixel_form(ok, Uf + (fmaf(M.A1, gx, -Sx.x * M.sx) - fr[0]),
                    Vf + (fmaf(M.A2, gy.x, -Sy.x * M.sy) + fm[0]), q1.x, q1.y);
  out1 = pixel_form(ok, Uf + (fmaf(M.A1, gx, -Sx.y * M.sx) - fr[1]),
                    Vf + (fmaf(M.A2, gy.y, -Sy.y * M.sy) + fm[1]), q1.x, q1.y);
}

// Map edge that vertex (i, j) of record `leaf` is proven to land beyond
// (MM_CULL_*), from the record's culling bound and the vertex's distances to
// the record's direct stars, measured as the near field measures them;
// MM_CULL_NONE when not proven.  `run` receives how many rows from j on
// (this one included) the proof holds for: the column's vertices stay in
// the sub-cell (below its upper edge, with a row to spare) and outside the
// culling radius of every direct star (a star above is approached by one
// row per row; one below or level only recedes).
template <bool SQUARE>
__device__ __forceinline__ int vertex_cull_side(const MapCore &M, int leaf, int i, int j,
                                                int &run) {
  run = 0;
  if (leaf < 0) return MM_CULL_NONE;
  const int4 *rp = reinterpret_cast<const int4 *>(M.leaf + leaf);
  const int4 q3 = __ldg(rp + 3);
  if (q3.z == MM_CULL_NONE) return MM_CULL_NONE;
  const int4 q0 = __ldg(rp), q2 = __ldg(rp + 2);
  const float r2 = __int_as_float(q3.w);
  const float fi = (float)(i - q0.x), fj = (float)(j - q0.y);
  // rows to the sub-cell's upper edge (centre + half-length, grid units)
  const float top = __int_as_float(q0.w) + 1.0f / __int_as_float(q2.y);
  int n = (int)floorf(fminf(top - fj, 1.0e6f)) - 1;
  const float rho = SQUARE ? 1.f : M.rho;
  const float4 *np_ = reinterpret_cast<const float4 *>(M.near_pos) + q2.z;
#pragma unroll 1
  for (int k = 0; k < q2.w; k++) {
    const float4 s = __ldg(np_ + k);
    const float dx = (fi - s.x) - s.y, dy = (fj - s.z) - s.w;
    const float dx2 = dx * dx;
    if (!(fmaf(rho * dy, dy, dx2) > r2)) return MM_CULL_NONE;
    if (dx2 > r2 || dy >= 0.f) continue;
    // rows until |dy| falls to sqrt((r2 - dx^2) / rho), less one to spare
    const float kin = -dy - sqrtf((r2 - dx2) / rho);
    n = min(n, (int)floorf(kin) - 1);
  }
  run = max(n, 1);
  return q3.z;
}

// The map edge a whole row of the warp's vertices is proven to lie beyond
// (lanes without a vertex agree with anything), and the rows from j on the
// proof holds for in every lane; MM_CULL_NONE otherwise.
template <bool SQUARE>
__device__ __forceinline__ int row_cull_side(const MapCore &M, int leaf, int i, int j,
                                             bool vvalid, int &run) {
  int r = 1 << 30;
  const int s = vvalid ? vertex_cull_side<SQUARE>(M, leaf, i, j, r) : -1;
  const int S = __reduce_max_sync(0xffffffffu, s);
  run = (int)__reduce_min_sync(0xffffffffu, (unsigned)r);
  return (S > 0 && __all_sync(0xffffffffu, s == S || s < 0)) ? S : MM_CULL_NONE;
}

// Persistent warps; each work item is a strip of 31 cell columns by
// rows_per_item cell rows of one map.  Lane l computes vertex column
// 31*s + l for every vertex row of the item; the row below and the right
// neighbour's vertices wait in shared memory; lanes 0..30 then map cells (i, j-1) as the triangles {v00, v10, v11} and
// {v00, v11, v01} (diagonal from lower-left to upper-right).
// Issue- and latency-bound (no pipe saturated): the kernel is shaped to run 3
// blocks of 8 warps per SM, 80 registers a thread without spills -- the row
// below waits in shared memory, every apportioning waits in queues emptied
// once a row, when no vertex is live, and the counters are kept per warp.  Its
// loop has to stay in the instruction cache: with the loops below unrolled as
// the compiler likes (77 KB of code in place of 51) a third of the issue slots
// went to fetching and it took 17.3 ms.
// 2000^2 map, 9 rays per pixel: 16.9 ms at 2 blocks with the apportioning in
// divergent branches, 15.3 ms with the queues at 2 blocks, 13.0 ms at 3 (4
// spill and are slower), 11.9 ms with rows shot in pairs, one lookup for up
// to 33 rows and outcodes in place of box tests, 11.5 with a larger L1
// (WarpSmem).
#ifndef MM_SHOOT_MINB
#define MM_SHOOT_MINB 3  // resident 256-thread blocks per SM the register budget targets
#endif

// A single map (BATCH = false) arrives by value as a launch parameter, so
// its fields are read from the constant bank instead of held in registers;
// a batch reads its maps from the device array `maps`.
template <bool SQUARE, bool BATCH>
__global__ void __launch_bounds__(256, MM_SHOOT_MINB)
    k_shoot_ipm(const MapDev *__restrict__ maps, const MapDev M1, int n_maps, int64_t total_work,
                unsigned long long *work_counter, unsigned *err) {
  const int lane = threadIdx.x & 31;
  extern __shared__ __align__(16) unsigned char s_dyn[];
  WarpSmem *ws = reinterpret_cast<WarpSmem *>(s_dyn) + (threadIdx.x >> 5);
  WarpQueues q = {ws, 0, 0, 0};
  LaneCount lc = {0u, 0u};
  counts_clear(ws, lane);
  int last_map = -1;
  // A batch's current map, copied per warp into shared memory when the warp
  // moves to another map: its fields are then read there like a launch
  // parameter's, which leaves the registers to the per-ray work (reading
  // them from the descriptor array in global memory costs registers, and
  // spills, that the single-map kernel never pays).
  static_assert(MM_SHOOT_MINB != 3 ||
                    3 * (MM_SHOOT_SMEM_BYTES + 8 * sizeof(MapCore) + 64 + 1024) <= 196 * 1024,
                "a step of shared memory taken from the L1");
  __shared__ MapCore s_md[BATCH ? 8 : 1];
  MapCore &SM = s_md[BATCH ? threadIdx.x >> 5 : 0];
  while (true) {
    // (a single map whose larger triangles may exceed its queue stops at the
    // limit; its next launch goes on where this one stopped)
    unsigned long long w = (unsigned long long)total_work;
    if (lane == 0 && (BATCH || M1.bigq_limit == INT64_MAX ||
                      (int64_t)__ldcg(M1.bigq_n) < M1.bigq_limit))
      w = atomicAdd(work_counter, 1ull);
    w = __shfl_sync(0xffffffffu, w, 0);
    if ((int64_t)w >= total_work) break;
    int mi = 0;
    if (BATCH && n_maps > 1) {
      int lo = 0, hi = n_maps - 1;
#pragma unroll 1
      while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (maps[mid].work_begin <= (int64_t)w)
          lo = mid;
        else
          hi = mid - 1;
      }
      mi = lo;
    }
    if (BATCH && mi != last_map) {  // warp-uniform
      if (last_map >= 0) counts_flush(SM, ws, lc, lane);
      __syncwarp();
      const unsigned long long *src = reinterpret_cast<const unsigned long long *>(
          static_cast<const MapCore *>(maps + mi));
      unsigned long long *dst = reinterpret_cast<unsigned long long *>(&SM);
      if (lane < (int)(sizeof(MapCore) / 8)) dst[lane] = src[lane];
      __syncwarp();
      last_map = mi;
    }
    if (!BATCH) last_map = 0;
    const MapCore &M = BATCH ? SM : static_cast<const MapCore &>(M1);
    const MapItems &I = BATCH ? maps[mi] : M1;
    const int64_t local = (int64_t)w - I.work_begin;
    const int64_t s = local % I.strips, b = (local / I.strips) * I.item_stride;
    // grid indices fit 32 bits (at most 2^31 - 1 rays per axis)
    const int i = (int)(I.col_begin + s * MM_STRIP) + lane;
    const int jb = (int)(I.row_begin + b * I.rows_per_item);
    const int je = (int)min((int64_t)jb + I.rows_per_item, I.row_end);
    const int col_end = (int)I.col_end;
    const bool vvalid = i <= col_end;  // vertex columns [col_begin, col_end]
    const int cx = __ldg(&M.col_cell[vvalid ? i : col_end]);
    const bool cell_col = (lane < MM_STRIP) && (i < col_end);
    RunAcc ra = MM_RUN_NONE;
    // culling state of the previous row (warp-uniform): the map edge it is
    // proven to lie beyond, and whether its vertices were computed (they are
    // in ws->row); `side` is row j's
    int prev_side = MM_CULL_NONE, side = MM_CULL_NONE;
    bool prev_exact = false;
    int c_leaf = -1, j_same = INT_MIN;  // this lane's record, up to row j_same
    bool c_cull = false;                // it has a culling bound
    int cull_wait = 0, cull_pause = 0;  // rows left before the next culling test
    // One pass shoots one vertex row and maps the cells between it and the
    // row below: row jb (nothing to map), then rows j = jb + 1 .. je; a row
    // below that culling left out is shot first (`back`).  A row whose
    // successor needs no culling test and lies in the same records is shot
    // with it, and the successor's pass finds its vertices in ws->next
    // (`ahead`).  One pass more shares out what is left in the queues.
    bool back = false, ahead = false;
    unsigned below_out = 0;  // outcodes of the row below: this lane's and (<< 4) its neighbour's
    for (int j = jb;;) {
      const bool fin = j > je;  // warp-uniform
      if (!fin) {
        int js = j;
        Vtx v01;
        if (ahead) {
          side = MM_CULL_NONE;
          if (cull_wait > 0) cull_wait--;
          v01 = ws->next[lane];
          ahead = false;
        } else {
          if (j >= j_same) {
            c_leaf = lookup_rows(M, cx, j, je, lane, vvalid, j_same, c_cull);
            if (c_leaf < 0 && vvalid) atomicOr(err, ERR_LOOKUP);
          }
          int leaf = c_leaf;
          // a row is provably beyond the map only if every lane's record has a
          // culling bound; otherwise the per-vertex test cannot succeed
          if (M.cull && !back) {
            int run = 0;
            side = MM_CULL_NONE;
            if (cull_wait > 0) {
              cull_wait--;
            } else if (!__any_sync(0xffffffffu, vvalid && !c_cull)) {
              side = row_cull_side<SQUARE>(M, leaf, i, j, vvalid, run);
              // a failed test pauses the tests of the next rows (1, 3, ... up to 8)
              if (j > jb) {
                cull_pause = side == MM_CULL_NONE ? min(2 * cull_pause + 1, 8) : 0;
                cull_wait = cull_pause;
              }
            }
            if (j > jb && side != MM_CULL_NONE && side == prev_side) {
              // rows j .. j + run - 1 and the one below lie beyond the same map
              // edge: the cells between them map nothing, and none of those
              // rows is computed
              const int skip = min(run, je - j + 1);
              prev_exact = false;
              if (lane == 0) ws->count[ST_CULLED] += (unsigned)skip;
              j += skip;
              continue;
            }
          }
          if (j > jb && !prev_exact) {
            // the row below was not computed; its cells with this row are needed
            js = j - 1;
            leaf = lookup_leaf(M, cx, __ldg(&M.row_cell[js]));
          }
          // (the next row is not tested while the tests pause, and cannot pass
          // where a lane's record has no bound)
          ahead = js == j && j < je && j + 1 < j_same &&
                  (!M.cull || cull_wait > 0 || __any_sync(0xffffffffu, vvalid && !c_cull));
          if (ahead) {
            Vtx nx;
            shoot_rows2<SQUARE, 3>(M, leaf, i, j, vvalid, v01, nx);
            ws->next[lane] = nx;  // (read back by this lane)
          } else {
            v01 = shoot_point<SQUARE, false>(M, leaf, i, js, 0.f, 0.f, vvalid);
          }
        }
        // the row below waits in shared memory (not in eight registers held
        // across the deflection), where a lane also finds its right neighbour
        const Vtx v00 = ws->row[lane], v10 = ws->row[min(lane + 1, 31)];
        __syncwarp();
        ws->row[lane] = v01;
        __syncwarp();
        const unsigned o01 = outcode(M, v01);
        const unsigned o11 = __shfl_down_sync(0xffffffffu, o01, 1);
        const unsigned o00 = below_out & 15u, o10 = below_out >> 4;
        below_out = o01 | (o11 << 4);
        if (j == jb || js < j) {
          back = js < j;
          prev_exact = true;
          if (j == jb) {
            prev_side = side;
            j++;
          }
          continue;
        }
        back = false;
        prev_side = side;
        // most triangles of a shooting region lie wholly beyond one edge of
        // the map: integer tests before any arithmetic (a non-finite vertex
        // lies beyond none, and is counted)
        const bool on0 = cell_col && !(o00 & o10 & o11), on1 = cell_col && !(o00 & o11 & o01);
        if (!__any_sync(0xffffffffu, on0 || on1)) {
          j++;
          continue;
        }
        // (diagonal v00 - v11)
        const Vtx v11 = ws->row[min(lane + 1, 31)];
        tri_scan(M, q, v00, v10, v11, on0, ra, lc, lane);
        tri_scan(M, q, v00, v11, v01, on1, ra, lc, lane);
      }
      share_out(M, q, fin, lc, lane);
      if (fin) break;
      j++;
    }
    run_flush<MM_FIX_ONE>(M, ra);
  }
  if (last_map >= 0) counts_flush(BATCH ? SM : static_cast<const MapCore &>(M1), ws, lc, lane);
}

// Inverse ray shooting (Sec. 3.2; the IRS column of Table 1): every grid
// vertex is one ray, and the pixel it lands in gains one count.  The work
// items, deflection and culling are k_shoot_ipm's; lane l < 31 owns vertex
// column 31 s + l (lane 31 only the grid's last column) and a work item owns
// its vertex rows [jb, je) (the map's last item also je), so every ray is
// counted once.  Rows proven to land beyond a map edge are skipped: none of
// their rays can count, and a culled vertex is never non-finite (a ray on a
// star lies inside that star's culling radius).
// 4 blocks of 8 warps per SM (64 registers, no spills): the deflection
// alone gains from the occupancy that k_shoot_ipm's mapping code cannot
// afford (on the 2000^2 grid 3 blocks were 17 % faster than 2, and 4 are
// 8 % faster than 3; 5 spill and are slower).
#define MM_IRS_MINB 4
template <bool SQUARE>
__global__ void __launch_bounds__(256, MM_IRS_MINB)
    k_shoot_irs(const MapDev M, int64_t total_work, unsigned long long *work_counter,
                unsigned *err) {
  const int lane = threadIdx.x & 31;
  unsigned dropped = 0, culled = 0;
  while (true) {
    unsigned long long w = 0;
    if (lane == 0) w = atomicAdd(work_counter, 1ull);
    w = __shfl_sync(0xffffffffu, w, 0);
    if ((int64_t)w >= total_work) break;
    const int64_t local = (int64_t)w - M.work_begin;
    const int64_t s = local % M.strips, b = (local / M.strips) * M.item_stride;
    const int i = (int)(M.col_begin + s * MM_STRIP) + lane;
    const int jb = (int)(M.row_begin + b * M.rows_per_item);
    const int je = (int)min((int64_t)jb + M.rows_per_item, M.row_end);
    const int jl = je == (int)M.row_end ? je : je - 1;  // last vertex row owned
    const int col_end = (int)M.col_end;
    const bool vvalid = i <= col_end;
    const bool owner = vvalid && (lane < MM_STRIP || i == col_end);
    const int cx = __ldg(&M.col_cell[vvalid ? i : col_end]);
    RunAcc ra = MM_RUN_NONE;
    int c_leaf = -1, j_same = INT_MIN;  // this lane's record, up to row j_same
    bool c_cull = false;                // it has a culling bound
    int cull_wait = 0, cull_pause = 0;  // rows left before the next culling test
    auto count = [&](const Vtx &v) {
      if (!owner) return;
      if (v.px == MM_VTX_INVALID)
        dropped++;
      else if (v.px >= 0 && v.px < M.npix && v.py >= 0 && v.py < M.npix_y)
        run_add<1ull>(M, ra, v.px, v.py);
    };
    for (int j = jb; j <= jl; j++) {
      if (j >= j_same) {
        c_leaf = lookup_rows(M, cx, j, jl, lane, vvalid, j_same, c_cull);
        if (c_leaf < 0 && vvalid) atomicOr(err, ERR_LOOKUP);
      }
      const int leaf = c_leaf;
      const bool bound = M.cull && !__any_sync(0xffffffffu, vvalid && !c_cull);
      if (M.cull && cull_wait > 0) {
        cull_wait--;
      } else if (bound) {
        int run;
        if (row_cull_side<SQUARE>(M, leaf, i, j, vvalid, run) != MM_CULL_NONE) {
          const int skip = min(run, jl - j + 1);
          if (lane == 0) culled += (unsigned)skip;
          j += skip - 1;
          cull_pause = 0;
          continue;
        }
        // a failed test pauses the tests of the next rows (1, 3, ... up to 8)
        cull_pause = min(2 * cull_pause + 1, 8);
        cull_wait = cull_pause;
      }
      // a row whose successor is not tested and lies in the same records is
      // shot with it
      if (j < jl && j + 1 < j_same && (!bound || cull_wait > 0)) {
        Vtx v0, v1;
        shoot_rows2<SQUARE, 6>(M, leaf, i, j, vvalid, v0, v1);
        count(v0);
        count(v1);
        if (cull_wait > 0) cull_wait--;
        j++;
      } else {
        count(shoot_point<SQUARE, false, 6>(M, leaf, i, j, 0.f, 0.f, vvalid));
      }
    }
    run_flush<1ull>(M, ra);
  }
  dropped = __reduce_add_sync(0xffffffffu, dropped);
  if (lane == 0 && dropped) atomicAdd(&M.stat[ST_DROPPED], (unsigned long long)dropped);
  if (lane == 0 && culled) atomicAdd(&M.stat[ST_CULLED], (unsigned long long)culled);
}

// Second pass over the larger triangles k_shoot_ipm (or k_ipm_vertices)
// queued for the map: each warp takes batches of 32 from the device queue
// and deals out their pixel rows and partially covered pixels
// (warp_tri_jobs), at 5 blocks per SM where the first kernel runs 3 (48
// registers allow 5 without spills: 3 % faster than 4; 6 forces spills)
//
// BANDED: a map too large for the L2 is taken band by band (the entries in the
// order k_band_scatter puts them), so that the lines of the rows being worked
// on stay in the L2.  A triangle reaching into several bands has an entry in
// each and is dealt there within that band's rows: triangles near a star are
// large (a height above L for 1/L of them), and whole they would touch lines
// far from the band.  3001^2 map near the critical line, 4.3e8 triangles: 173 ms
// in queue order, 73 ms by bands; 5000^2 map, 2.6e8 triangles: 51 ms by bands
// with whole triangles (10 GB written in 1.3e8), 39 ms cut (the map once).
#define MM_BIG_MINB 5

// Queued triangles that found a slot.
__device__ __forceinline__ long long queued(const MapCore &M) {
  const unsigned long long cap = (unsigned long long)M.bigq_cap, qn = *M.bigq_n;
  return (long long)(qn < cap ? qn : cap);
}
// The bands of a triangle's rows within the map; x > y: none.
__device__ __forceinline__ int2 band_range(const MapDev &M, const RawTri &t) {
  const float ymin = fminf(t.f[1], fminf(t.f[3], t.f[5]));
  const float ymax = fmaxf(t.f[1], fmaxf(t.f[3], t.f[5]));
  const int r0 = max(t.y + __float2int_rd(fminf(fmaxf(ymin, -1.0e9f), 1.0e9f)), 0);
  const int r1 = min(t.y + __float2int_rd(fminf(fmaxf(ymax, -1.0e9f), 1.0e9f)), M.npix_y - 1);
  if (r0 > r1) return make_int2(1, 0);
  return make_int2(r0 >> M.band_shift, r1 >> M.band_shift);
}
// s_end[k]: entries of bands 0 .. k.  False: more than there is room for (then
// the queue is taken in its own order).  Call with all threads of the block.
__device__ __forceinline__ bool band_ends(const MapCore &M, unsigned long long *s_end) {
  if (threadIdx.x < MM_BANDS) {
    unsigned long long n = 0;
    for (int k = 0; k <= threadIdx.x; k++) n += M.bigq_n[2 + k];
    s_end[threadIdx.x] = n;
  }
  __syncthreads();
  return s_end[MM_BANDS - 1] <= MM_BAND_ENTRIES * (unsigned long long)M.bigq_cap;
}

// SMALL: a queue that gives its warps less than two batches of 32 is dealt in
// batches of 16 .. 4: a batch's rows are a chain of rounds (48^2 map, 13 000
// triangles: 23 -> 12 us).
template <bool BANDED, bool SMALL>
__global__ void __launch_bounds__(256, MM_BIG_MINB) k_big_ipm(const MapDev M) {
  __shared__ TriJob q[8][32];
  __shared__ RowRecs rr[8];
  __shared__ unsigned long long s_end[BANDED ? MM_BANDS : 1];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const bool sorted = BANDED && band_ends(M, s_end);
  const long long n = sorted ? (long long)s_end[BANDED ? MM_BANDS - 1 : 0] : queued(M);
  int log_size = 5;
  if (SMALL)
    while (log_size > 2 && (n >> (log_size + 1)) < gridDim.x * 8) log_size--;
  while (true) {
    unsigned long long b = 0;
    if (lane == 0) b = atomicAdd(M.bigq_n + 1, 1ull);
    b = __shfl_sync(0xffffffffu, b, 0);
    const long long base = (long long)b << log_size;
    if (base >= n) break;
    const int nb = (int)min(1ll << log_size, n - base);
    int row_lo = 0, row_hi = M.npix_y;
    if (lane < nb) {
      const long long slot = sorted ? (long long)M.bigq_order[base + lane] : base + lane;
      const RawTri t = raw_load(M.bigq + slot);
      q[w][lane] = make_job(t);
      if (sorted) {
        int band = 0;  // the first band that ends beyond this entry
#pragma unroll
        for (int step = MM_BANDS / 2; step > 0; step >>= 1)
          if (s_end[band + step - 1] <= (unsigned long long)(base + lane)) band += step;
        const int2 r = band_range(M, t);
        // (the outer bands take what rounding puts beyond them)
        if (band > r.x) row_lo = band << M.band_shift;
        if (band < r.y) row_hi = (band + 1) << M.band_shift;
      }
    }
    __syncwarp();
    warp_tri_jobs(M.acc, M.span, M.npix, M.npix_y, M.err, q[w], nb, &rr[w], lane, row_lo, row_hi);
  }
}

// The bands of each queued triangle, and the entries per band (bigq_n[2 +
// band]; a warp's lanes of one first band count together).  Here and not where
// the triangle is queued: one more pass over the queue (0.2 ms a 1.3e8 slots)
// against spills in the first pass's batch kernel (5 % slower).
#define MM_BAND_CHUNK 4096  // slots per block of the two kernels below
__device__ __forceinline__ void band_tally(unsigned *s_n, int2 r, int lane) {
  const int first = r.x <= r.y ? r.x : -1;
  const unsigned m = __match_any_sync(0xffffffffu, first);
  if (first >= 0 && lane == __ffs(m) - 1) atomicAdd(&s_n[first], (unsigned)__popc(m));
  for (int k = r.x + 1; k <= r.y; k++) atomicAdd(&s_n[k], 1u);
}
__global__ void __launch_bounds__(256) k_band_count(const MapDev M) {
  __shared__ unsigned s_n[MM_BANDS];
  if (threadIdx.x < MM_BANDS) s_n[threadIdx.x] = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const long long n = queued(M);
  for (long long c = (long long)blockIdx.x * MM_BAND_CHUNK; c < n;
       c += (long long)gridDim.x * MM_BAND_CHUNK) {
    const long long e = min(n, c + MM_BAND_CHUNK);
    for (long long k = c + threadIdx.x; k - lane < e; k += 256) {
      int2 r = make_int2(1, 0);
      if (k < e) {
        r = band_range(M, raw_load(M.bigq + k));
        M.bigq_band[k] = make_uchar2((unsigned char)r.x, (unsigned char)r.y);
      }
      band_tally(s_n, r, lane);
    }
  }
  __syncthreads();
  if (threadIdx.x < MM_BANDS && s_n[threadIdx.x])
    atomicAdd(M.bigq_n + 2 + threadIdx.x, (unsigned long long)s_n[threadIdx.x]);
}

// The slots in the order of their bands (any order within one): each chunk
// counts its entries per band, reserves their places, and writes them.
__global__ void __launch_bounds__(256) k_band_scatter(const MapDev M) {
  __shared__ unsigned s_n[MM_BANDS];
  __shared__ unsigned long long s_end[MM_BANDS], s_at[MM_BANDS];
  if (!band_ends(M, s_end)) return;
  const int lane = threadIdx.x & 31;
  const long long n = queued(M);
  for (long long c = (long long)blockIdx.x * MM_BAND_CHUNK; c < n;
       c += (long long)gridDim.x * MM_BAND_CHUNK) {
    const long long e = min(n, c + MM_BAND_CHUNK);
    __syncthreads();
    if (threadIdx.x < MM_BANDS) s_n[threadIdx.x] = 0;
    __syncthreads();
    for (long long k = c + threadIdx.x; k - lane < e; k += 256) {
      const uchar2 r = k < e ? M.bigq_band[k] : make_uchar2(1, 0);
      band_tally(s_n, make_int2(r.x, r.y), lane);
    }
    __syncthreads();
    if (threadIdx.x < MM_BANDS) {
      const unsigned cnt = s_n[threadIdx.x];
      if (cnt)
        s_at[threadIdx.x] =
            (threadIdx.x ? s_end[threadIdx.x - 1] : 0ull) +
            atomicAdd(M.bigq_n + 2 + MM_BANDS + threadIdx.x, (unsigned long long)cnt);
      s_n[threadIdx.x] = 0;
    }
    __syncthreads();
    for (long long k = c + threadIdx.x; k - lane < e; k += 256) {
      const uchar2 r = k < e ? M.bigq_band[k] : make_uchar2(1, 0);
      const int band = r.x <= r.y ? r.x : -1;
      const unsigned m = __match_any_sync(0xffffffffu, band);
      const int first = __ffs(m) - 1;
      unsigned at = 0;
      if (band >= 0 && lane == first) at = atomicAdd(&s_n[band], (unsigned)__popc(m));
      at = __shfl_sync(0xffffffffu, at, first);
      if (band >= 0)
        M.bigq_order[s_at[band] + at + __popc(m & ((1u << lane) - 1u))] = (uint32_t)k;
      for (int o = r.x + 1; o <= r.y; o++)
        M.bigq_order[s_at[o] + atomicAdd(&s_n[o], 1u)] = (uint32_t)k;
    }
  }
}

// mu = (acc + row-prefix(span)) * 2^-32 * (h_x h_y / 2) / delta^2; one block
// per map row.
__global__ void __launch_bounds__(256) k_normalize(const unsigned long long *__restrict__ acc,
                                                   const unsigned long long *__restrict__ span,
                                                   int npix, double scale, float *out) {
  __shared__ unsigned long long part[256];
  const int row = blockIdx.x;
  const int t = threadIdx.x;
  const int chunk = (npix + 255) / 256;
  const int c0 = t * chunk, c1 = min(npix, c0 + chunk);
  const unsigned long long *sp = span + (int64_t)row * (npix + 1);
  unsigned long long s = 0;
  for (int c = c0; c < c1; c++) s += sp[c];
  part[t] = s;
  __syncthreads();
  // inclusive scan of the 256 partial sums (Hillis-Steele)
  for (int d = 1; d < 256; d <<= 1) {
    unsigned long long v = (t >= d) ? part[t - d] : 0ull;
    __syncthreads();
    part[t] += v;
    __syncthreads();
  }
  unsigned long long run = (t > 0) ? part[t - 1] : 0ull;
  const unsigned long long *ar = acc + (int64_t)row * npix;
  float *o = out + (int64_t)row * npix;
  for (int c = c0; c < c1; c++) {
    run += sp[c];
    unsigned long long tot = ar[c] + run;
    o[c] = (float)((double)tot * scale);
  }
}

// mu = acc * scale for an accumulator already folded with its difference
// array (the same arithmetic as k_normalize, so a folded map normalises to
// the same floats)
__global__ void __launch_bounds__(256) k_scale_fixed(const unsigned long long *__restrict__ acc,
                                                     int64_t n, double scale, float *out) {
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n;
       k += (int64_t)gridDim.x * blockDim.x)
    out[k] = (float)((double)acc[k] * scale);
}

// acc += row-prefix(span): folds the difference array into the accumulator so
// the raw fixed-point map can be read back.
__global__ void k_fold_span(unsigned long long *acc, const unsigned long long *span, int npix,
                            int npix_y, unsigned long long *out) {
  const int row = blockIdx.x * blockDim.x + threadIdx.x;
  if (row >= npix_y) return;
  const unsigned long long *sp = span + (int64_t)row * (npix + 1);
  unsigned long long run = 0;
  for (int c = 0; c < npix; c++) {
    run += sp[c];
    out[(int64_t)row * npix + c] = acc[(int64_t)row * npix + c] + run;
  }
}

// Deflection probe: w (FP64) at arbitrary image-plane points, through the
// same per-vertex code as the map kernel.
template <bool SQUARE>
__global__ void k_probe(const MapDev *maps, int64_t n, const double *z, double *w, double x0,
                        double y0, double hx, double hy, double R0, double lox, double loy,
                        double delta, unsigned *err) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool ok = t < n;
  const MapDev &M = maps[0];
  double zx = ok ? z[2 * t] : x0, zy = ok ? z[2 * t + 1] : y0;
  double gi = (zx - x0) / hx, gj = (zy - y0) / hy;
  double fi = floor(gi), fj = floor(gj);
  int64_t i = (int64_t)fi, j = (int64_t)fj;
  float ti = (float)(gi - fi), tj = (float)(gj - fj);
  const double scale = (double)(1 << MM_DMAX) / (2.0 * R0);
  double cxd = floor((zx + R0) * scale), cyd = floor((zy + R0) * scale);
  int cx = (int)fmin(fmax(cxd, 0.0), (double)((1 << MM_DMAX) - 1));
  int cy = (int)fmin(fmax(cyd, 0.0), (double)((1 << MM_DMAX) - 1));
  int leaf = ok ? lookup_leaf(M, cx, cy) : -1;
  Vtx v = shoot_point<SQUARE, true>(M, leaf, (int)i, (int)j, ti, tj, ok && leaf >= 0);
  if (!ok) return;
  if (v.px == MM_VTX_INVALID) {
    w[2 * t] = nan("");
    w[2 * t + 1] = nan("");
    return;
  }
  w[2 * t] = lox + ((double)v.px + (double)v.fx) * delta;
  w[2 * t + 1] = loy + ((double)v.py + (double)v.fy) * delta;
}

// ---------------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------------

template <bool SQUARE, bool BATCH>
static cudaError_t launch_shoot_t(const MapDev *d_maps, const MapDev &m1, int n_maps,
                                  int64_t total_work, unsigned long long *counter, unsigned *err,
                                  int grid, cudaStream_t st) {
  const int smem = (int)MM_SHOOT_SMEM_BYTES;
  cudaError_t e = cudaFuncSetAttribute(k_shoot_ipm<SQUARE, BATCH>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  k_shoot_ipm<SQUARE, BATCH><<<grid, 256, smem, st>>>(d_maps, m1, n_maps, total_work, counter,
                                                      err);
  return cudaGetLastError();
}

cudaError_t launch_shoot_ipm(const MapDev *d_maps, const MapDev *h_single, int n_maps,
                             int64_t total_work, bool square, unsigned long long *counter,
                             unsigned *err, int grid, cudaStream_t st) {
  if (total_work <= 0) return cudaSuccess;
  if (n_maps == 1 && h_single)
    return square ? launch_shoot_t<true, false>(nullptr, *h_single, 1, total_work, counter, err,
                                                grid, st)
                  : launch_shoot_t<false, false>(nullptr, *h_single, 1, total_work, counter, err,
                                                 grid, st);
  const MapDev none{};
  return square ? launch_shoot_t<true, true>(d_maps, none, n_maps, total_work, counter, err, grid,
                                             st)
                : launch_shoot_t<false, true>(d_maps, none, n_maps, total_work, counter, err,
                                              grid, st);
}

// Device-side assembly of a batch's descriptor array from the handles' own
// device copies (no host staging, so a batch can be captured in a CUDA
// graph): block i copies map i's descriptor and sets its first work item.
#define MM_GATHER_MAX 64
struct BatchGather {
  const MapDev *src[MM_GATHER_MAX];
  int64_t work_begin[MM_GATHER_MAX];
  int n;
};
static_assert(sizeof(MapDev) % 8 == 0 && sizeof(MapCore) % 8 == 0 && sizeof(MapCore) <= 256,
              "copied in 8-byte words, the core's one a lane");

__global__ void k_batch_gather(const BatchGather g, MapDev *dst) {
  const int i = blockIdx.x;
  if (i >= g.n) return;
  const unsigned long long *s = reinterpret_cast<const unsigned long long *>(g.src[i]);
  unsigned long long *d = reinterpret_cast<unsigned long long *>(dst + i);
  for (int k = threadIdx.x; k < (int)(sizeof(MapDev) / 8); k += blockDim.x) d[k] = s[k];
  __syncthreads();
  if (threadIdx.x == 0) dst[i].work_begin = g.work_begin[i];
}

cudaError_t launch_batch_gather(const MapDev *const *src, const int64_t *work_begin, int n,
                                MapDev *dst, int &launches, cudaStream_t st) {
  for (int b = 0; b < n; b += MM_GATHER_MAX) {
    BatchGather g;
    g.n = min(MM_GATHER_MAX, n - b);
    for (int k = 0; k < g.n; k++) {
      g.src[k] = src[b + k];
      g.work_begin[k] = work_begin[b + k];
    }
    k_batch_gather<<<g.n, 64, 0, st>>>(g, dst + b);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    launches++;
  }
  return cudaSuccess;
}

cudaError_t launch_shoot_irs(const MapDev &m, int64_t total_work, bool square,
                             unsigned long long *counter, unsigned *err, cudaStream_t st) {
  if (total_work <= 0) return cudaSuccess;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int grid = sms * MM_IRS_MINB;
  if (square)
    k_shoot_irs<true><<<grid, 256, 0, st>>>(m, total_work, counter, err);
  else
    k_shoot_irs<false><<<grid, 256, 0, st>>>(m, total_work, counter, err);
  return cudaGetLastError();
}

cudaError_t launch_big_ipm(const MapDev &m, int &launches, cudaStream_t st) {
  if (m.bigq_cap <= 0) return cudaSuccess;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int grid = sms * MM_BIG_MINB;
  if (m.band_shift >= 0) {
    k_band_count<<<sms * 8, 256, 0, st>>>(m);
    k_band_scatter<<<sms * 8, 256, 0, st>>>(m);
    k_big_ipm<true, false><<<grid, 256, 0, st>>>(m);
    launches += 3;
  } else if (m.bigq_cap < 64 * 8 * (int64_t)grid) {
    k_big_ipm<false, true><<<grid, 256, 0, st>>>(m);
    launches++;
  } else {
    k_big_ipm<false, false><<<grid, 256, 0, st>>>(m);
    launches++;
  }
  return cudaGetLastError();
}

cudaError_t launch_normalize(const unsigned long long *acc, const unsigned long long *span,
                             int npix, int npix_y, double scale, float *out, cudaStream_t st) {
  k_normalize<<<npix_y, 256, 0, st>>>(acc, span, npix, scale, out);
  return cudaGetLastError();
}

cudaError_t launch_scale_fixed(const unsigned long long *acc, int64_t n, double scale,
                               float *out, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int64_t blocks = std::min<int64_t>((n + 255) / 256, (int64_t)std::max(sms, 1) * 8);
  k_scale_fixed<<<(unsigned)blocks, 256, 0, st>>>(acc, n, scale, out);
  return cudaGetLastError();
}

cudaError_t launch_fold_span(unsigned long long *acc, const unsigned long long *span, int npix,
                             int npix_y, unsigned long long *out, cudaStream_t st) {
  k_fold_span<<<(npix_y + 127) / 128, 128, 0, st>>>(acc, span, npix, npix_y, out);
  return cudaGetLastError();
}

cudaError_t launch_probe(const MapDev *d_maps, bool square, int64_t n, const double *z,
                         double *w, double x0, double y0, double hx, double hy, double R0,
                         double lox, double loy, double delta, unsigned *err,
                         cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  int64_t blocks = (n + 255) / 256;
  if (square)
    k_probe<true><<<(unsigned)blocks, 256, 0, st>>>(d_maps, n, z, w, x0, y0, hx, hy, R0, lox,
                                                    loy, delta, err);
  else
    k_probe<false><<<(unsigned)blocks, 256, 0, st>>>(d_maps, n, z, w, x0, y0, hx, hy, R0, lox,
                                                     loy, delta, err);
  return cudaGetLastError();
}

}  // namespace mm
