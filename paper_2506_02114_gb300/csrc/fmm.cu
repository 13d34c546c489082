// Multipole and local expansions of the quadtree FMM (App. C.2), FP64.
//
// Coefficients are complex and normalised to the node half-length L about
// the node centre, as in App. C.2:
//   multipole  psi(z) = a_0 log(zeta) + sum_{k=1..p} a_k zeta^-k
//   local      psi(z) = sum_{l=0..p} c_l zeta^l,      zeta = (z - z_node)/L.
// The three shift operators depend only on the relative position of the two
// nodes in units of L, so they are fixed (p+1)x(p+1) complex matrices built
// once on the host: 4 for M2M (child quadrant), 49 slots (40 used) for M2L
// (same-level offsets in [-3, 3]^2 with Chebyshev distance >= 2) and 4 for
// L2L.  Each is stored as [op][k][l] so that threads indexed by the output
// coefficient l read consecutive entries.
//
// The l = 0 (logarithmic) terms of the locals are not formed: the deflection
// needs only dpsi/dz (Sec. 3.3), so c_0 never reaches a ray.
#include <algorithm>
#include <cmath>
#include <vector>

#include "mm_kernels.h"

namespace mm {

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ double2 cfma(double2 a, double2 b, double2 c) {
  return make_double2(fma(a.x, b.x, fma(-a.y, b.y, c.x)), fma(a.x, b.y, fma(a.y, b.x, c.y)));
}

// 2^e as a double, -1022 <= e <= 1023.
__device__ __forceinline__ double pow2(int e) { return __hiloint2double((1023 + e) << 20, 0); }

// Level, cell, centre and half-length of a node (R0 is a power of two, so
// every step but the centre's sum is exact; no FP64 division, which takes
// some twenty instructions of a pipe with 2 lanes per SM).
__device__ __forceinline__ void node_geom(const TreeDev &T, int64_t node, int &level, int &cx,
                                          int &cy, double &zx, double &zy, double &L) {
  level = T.lvl[node];
  uint32_t x, y;
  morton_decode(T.code[node], x, y);
  cx = (int)x;
  cy = (int)y;
  const double side = 2.0 * T.R0 * pow2(-level);
  zx = -T.R0 + ((double)cx + 0.5) * side;
  zy = -T.R0 + ((double)cy + 0.5) * side;
  L = 0.5 * side;
}

// 1/L of a power of two L = 2^e, exactly.
__device__ __forceinline__ double inv_pow2(double L) {
  return pow2(1023 - (__double2hiint(L) >> 20));
}

// x with its sign flipped if `neg`, by an integer operation.
__device__ __forceinline__ double flip(double x, bool neg) {
  return __hiloint2double(__double2hiint(x) ^ (neg ? 0x80000000 : 0), __double2loint(x));
}

// Real part (im = false) or imaginary part of a b + c, c that part of the
// addend: the two halves of cfma, in two FP64 instructions either way.
__device__ __forceinline__ double cfma_part(double2 a, double2 b, double c, bool im) {
  return fma(a.x, im ? b.y : b.x, fma(flip(a.y, !im), im ? b.x : b.y, c));
}

// 0, 1, ..., MM_PMAX (a conversion is an FP64 instruction too).
__constant__ double c_int[MM_PMAX + 1] = {
    0,  1,  2,  3,  4,  5,  6,  7,  8,  9,  10, 11, 12, 13, 14, 15, 16, 17, 18, 19, 20, 21,
    22, 23, 24, 25, 26, 27, 28, 29, 30, 31, 32, 33, 34, 35, 36, 37, 38, 39, 40, 41, 42, 43,
    44, 45, 46, 47, 48, 49, 50, 51, 52, 53, 54, 55, 56, 57, 58, 59, 60, 61, 62, 63, 64};

// x / k, correctly rounded, from the rounded reciprocal of the small integer
// k (Markstein's correction of the quotient by its exact remainder).
__device__ __forceinline__ double div_by(double x, double k, double inv_k) {
  const double q = x * inv_k;
  return fma(fma(-k, q, x), inv_k, q);
}

// Squares z^2, z^4, ... for power_of.
#define MM_POW_BITS 7  // exponents up to MM_PMAX
__device__ __forceinline__ void powers_of_two(double2 z, int kmax, double2 *sq) {
  sq[0] = z;
  for (int b = 1; b < MM_POW_BITS && (1 << b) <= kmax; b++) {
    z = cmul(z, z);
    sq[b] = z;
  }
}
// z^k (k >= 1) from the squares, multiplied in the order of the binary digits
// from the lowest.
__device__ __forceinline__ double2 power_of(const double2 *sq, int k) {
  int b = __ffs(k) - 1;
  double2 r = sq[b];
  for (k >>= b + 1, b++; k; k >>= 1, b++)
    if (k & 1) r = cmul(r, sq[b]);
  return r;
}

// ---------------------------------------------------------------------------
// P2M: a_0 = sum m_i, a_k = -(1/k) sum m_i zeta_i^k  (leaves only)
// FP64-bound, a thread per (node, coefficient) and four lanes per star for its
// powers: z^k is z^(k - 2^b) times the square z^(2^b), b the top digit of k,
// one product a power and formed once for the node.  Stars staged side by side,
// so that the four lanes of few stars fill warps, and nodes without stars take
// no threads.  50 000 stars, p = 25: 0.25 ms with a block per node, 0.11 ms
// with the powers formed by each (node, coefficient) from the squares, 0.06 ms
// like this (64 us in blocks of 256 threads, 73 of 128, 61 of 512; two lanes a
// star: 58, but 84 in place of 76 where most leaves hold none or one).
// ---------------------------------------------------------------------------
#define MM_P2M_THREADS 256
#define MM_P2M_STARS 4  // stars of a node staged at a time
#define MM_P2M_LANES 4  // lanes that share a star's powers
__global__ void __launch_bounds__(MM_P2M_THREADS)
    k_p2m(TreeDev T, int64_t n_nodes, int p, int per_block, const double *__restrict__ inv,
          double2 *mp) {
  grid_begin();
  extern __shared__ __align__(16) double2 s_p2m[];
  const int P1 = p + 1;
  // per staged star: z^0 (unused) .. z^p, then the masses
  double2 *zs = s_p2m;
  double *sm = reinterpret_cast<double *>(zs + per_block * MM_P2M_STARS * P1);
  __shared__ int s_node[32], s_beg[32], s_cnt[32], s_off[33];  // the block's nodes with stars
  const int64_t first = (int64_t)blockIdx.x * per_block;
  if (threadIdx.x < 32) {
    const int64_t nd = first + threadIdx.x;
    const bool leaf = threadIdx.x < per_block && nd < n_nodes && T.first_child[nd] < 0;
    const int beg = leaf ? T.sbeg[nd] : 0, cnt = leaf ? T.send[nd] - beg : 0;
    const unsigned with = __ballot_sync(0xffffffffu, cnt > 0);
    s_cnt[threadIdx.x] = 0;
    __syncwarp();
    if (cnt > 0) {
      const int o = __popc(with & ((1u << threadIdx.x) - 1u));
      s_node[o] = threadIdx.x;
      s_beg[o] = beg;
      s_cnt[o] = cnt;
    }
  }
  __syncthreads();
  const int local = threadIdx.x / P1, k = threadIdx.x - local * P1;
  const bool mine = local < per_block && s_cnt[local] > 0;
  const int64_t node = first + (mine ? s_node[local] : 0);
  double2 s = make_double2(0.0, 0.0);
  for (int c = 0;; c += MM_P2M_STARS) {
    // the next stars of each node, the nodes' one after another
    if (threadIdx.x < 32) {
      int n = min(max(s_cnt[threadIdx.x] - c, 0), MM_P2M_STARS);
      for (int d = 1; d < 32; d <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, n, d);
        if (threadIdx.x >= d) n += u;
      }
      if (threadIdx.x == 0) s_off[0] = 0;
      s_off[threadIdx.x + 1] = n;
    }
    __syncthreads();
    const int staged = s_off[32];
    if (staged == 0) break;
    const int r = threadIdx.x % MM_P2M_LANES;
    for (int base = 0; base < staged; base += MM_P2M_THREADS / MM_P2M_LANES) {
      const int t = base + threadIdx.x / MM_P2M_LANES;
      if (base + (int)(threadIdx.x & ~31u) / MM_P2M_LANES >= staged) break;  // (warp-uniform)
      double2 sq = make_double2(0.0, 0.0);
      if (t < staged) {
        int q = 0;
        for (int step = 16; step > 0; step >>= 1)
          if (s_off[q + step] <= t) q += step;
        const int i = s_beg[q] + c + t - s_off[q];
        int level, cx, cy;
        double zx, zy, L;
        node_geom(T, first + s_node[q], level, cx, cy, zx, zy, L);
        const double invL = inv_pow2(L);
        sq = make_double2((T.sx[i] - zx) * invL, (T.sy[i] - zy) * invL);
        if (r == 0) {
          if (p > 0) zs[t * P1 + 1] = sq;
          sm[t] = T.sm[i];
        }
      }
      for (int top = 2; top <= p; top *= 2) {
        __syncwarp();
        sq = cmul(sq, sq);
        if (t < staged) {
          if (r == 0) zs[t * P1 + top] = sq;
          for (int j = 1 + r; j < top && top + j <= p; j += MM_P2M_LANES)
            zs[t * P1 + top + j] = cmul(zs[t * P1 + j], sq);
        }
      }
    }
    __syncthreads();
    const int cnt = mine ? min(MM_P2M_STARS, s_cnt[local] - c) : 0;
    const int at = mine ? s_off[local] : 0;
    for (int i = at; i < at + cnt; i++) {
      const double m = sm[i];
      if (k == 0) {
        s.x += m;
      } else {
        const double2 zk = zs[i * P1 + k];
        s.x = fma(m, zk.x, s.x);
        s.y = fma(m, zk.y, s.y);
      }
    }
    __syncthreads();  // (the next stars take these places)
  }
  if (!mine) return;  // (a node without stars is nobody's source)
  if (k > 0) {
    const double dk = c_int[k], ik = inv[k];
    s = make_double2(div_by(-s.x, dk, ik), div_by(-s.y, dk, ik));
  }
  mp[node * P1 + k] = s;
}

// ---------------------------------------------------------------------------
// M2M: parent b = sum over the four children of MM[q] a_child (App. C.2)
// FP64-bound at the fine levels and a chain of latencies at the coarse ones:
// a thread takes rows l and p + 1 - l of one child (p + 1 terms whatever l,
// so that the triangle of binomials keeps every lane busy), and the four
// children's sums are added up afterwards in their order.  Children without
// stars (a quarter of the finest) add exact zeros and are left out.  Finest
// level of 50 000 stars, p = 25: 148 us with a thread per row and the
// children one after another, 70 us like this.
// ---------------------------------------------------------------------------
__global__ void k_m2m(TreeDev T, int level, int64_t n, int p, int per_block,
                      const double2 *__restrict__ MMop, double2 *mp) {
  grid_begin();
  extern __shared__ __align__(16) double2 s_m2m[];
  const int P1 = p + 1, half = (p + 1) / 2;
  double2 *a = s_m2m, *t = s_m2m + per_block * 4 * P1;  // [node][child][k]
  const int64_t first = T.level_off[level] + (int64_t)blockIdx.x * per_block;
  const int cnt = (int)min((int64_t)per_block, n - (int64_t)blockIdx.x * per_block);
  // factored M2M: b_k = z0^-k a_k per child, then
  // c_l = sum_q (z0/2)^l (-a_0 / l + sum_{k<=l} C(l-1, k-1) b_k), c_0 = sum_q a_0
  for (int idx = threadIdx.x; idx < cnt * 4 * P1; idx += blockDim.x) {
    const int nq = idx / P1, k = idx - nq * P1, q = nq & 3;
    const int fc = T.first_child[first + (nq >> 2)];
    if (fc < 0 || T.sbeg[fc + q] == T.send[fc + q]) continue;
    const double2 v = mp[(int64_t)(fc + q) * P1 + k];
    a[idx] = k ? cfma(MMop[(int64_t)P1 * P1 + q * 2 * P1 + k], v, make_double2(0.0, 0.0)) : v;
  }
  __syncthreads();
  const double *bt = reinterpret_cast<const double *>(MMop);  // binomials [k][l], 1/l at k = 0
  for (int idx = threadIdx.x; idx < cnt * 4 * half; idx += blockDim.x) {
    const int nq = idx / half, r = idx - nq * half;
    const int fc = T.first_child[first + (nq >> 2)];
    if (fc < 0 || T.sbeg[fc + (nq & 3)] == T.send[fc + (nq & 3)]) continue;
    const double2 *src = a + nq * P1;
    // rows r + 1 and p - r one after the other (the middle row of an odd p
    // once), each from its k = 0 term on
    int l = r + 1, k = 0;
    const int steps = 2 * l == p + 1 ? l + 1 : p + 3;
    double tx = 0.0, ty = 0.0;
#pragma unroll 4
    for (int i = 0; i < steps; i++) {
      const double b = bt[k * P1 + l];
      const double2 u = src[k];
      // (-a_0 / l first: a product rounded once, as the first of its sum)
      tx = fma(b, flip(u.x, k == 0), k ? tx : 0.0);
      ty = fma(b, flip(u.y, k == 0), k ? ty : 0.0);
      if (++k > l) {
        t[nq * P1 + l] = make_double2(tx, ty);
        l = p - r;
        k = 0;
      }
    }
  }
  __syncthreads();
  for (int idx = threadIdx.x; idx < cnt * P1; idx += blockDim.x) {
    const int nd = idx / P1, l = idx - nd * P1;
    const int fc = T.first_child[first + nd];
    if (fc < 0) continue;
    double2 s = make_double2(0.0, 0.0);
    for (int q = 0; q < 4; q++) {
      if (T.sbeg[fc + q] == T.send[fc + q]) continue;
      if (l == 0) {
        const double2 a0 = a[(nd * 4 + q) * P1];
        s = make_double2(s.x + a0.x, s.y + a0.y);
      } else {
        s = cfma(MMop[(int64_t)P1 * P1 + q * 2 * P1 + P1 + l], t[(nd * 4 + q) * P1 + l], s);
      }
    }
    mp[(first + nd) * P1 + l] = s;
  }
}

// ---------------------------------------------------------------------------
// Locals of an active node at level >= 2 (App. C.2):
//   L2L from the parent, M2L from the parent's neighbours' children that are
//   not adjacent (<= 27), P2L from the parent's unsplit neighbours that are
//   not adjacent (<= 5).
// One block per node and part of its rows l (one part where a level has
// nodes enough; a node's work is 11 us of one SM's FP64 pipe, so small levels
// share it out over SMs).  The sums over k of all its sources are independent:
// thread (group g, row l) takes sources g, g + G, ... two at a time, which
// fills the lanes for any p and gives each binomial it loads two uses; the
// sources' results are then added up row by row in the order of the list.
// FP64-bound at the fine levels (about 60 p instructions a source), latency
// at the coarse ones, where the sources one after another took 100 us a level
// whatever its size.  Sources without stars (a quarter of the finest level's)
// add exact zeros and are left out.  50 000 stars, p = 25: 1.21 ms over all
// levels with a warp per node, 0.56 ms like this; the finest level 477 and
// 283 us, with the FP64 pipe 93 % busy both times.
// ---------------------------------------------------------------------------
#define MM_LOCAL_THREADS 128
#define MM_LOCAL_STARS 8  // P2L stars staged at a time
struct LocalSources {
  int n;
  int src[32];   // first child or leaf of the source
  int slot[32];  // M2L: offset slot; -1: P2L from the leaf's stars
};

// Shared memory: the scaled multipoles b [source][k] (then the factors of the
// sums) and the sums t [source][l] of up to 27 sources, the L2L sum [l], the
// parent's local and the staged stars.
static __host__ __device__ __forceinline__ size_t local_smem(int p) {
  const size_t P1 = (size_t)p + 1;
  return sizeof(double2) * (2 * 27 * P1 + 2 * P1 + MM_LOCAL_STARS * (P1 + MM_POW_BITS)) +
         sizeof(double) * MM_LOCAL_STARS * (1 + P1);
}

__global__ void __launch_bounds__(MM_LOCAL_THREADS, 8)
    k_local(TreeDev T, int level, int64_t n, int p, const int32_t *node_act,
            const double2 *__restrict__ MLop, const double2 *__restrict__ LLop,
            const double2 *mp, double2 *loc, unsigned *err) {
  grid_begin();
  extern __shared__ __align__(16) double2 s_loc[];
  __shared__ LocalSources S;
  const int64_t node = T.level_off[level] + blockIdx.x;
  if (!node_act[node]) return;
  const int P1 = p + 1, tid = threadIdx.x;
  // this block's rows: r0 + 1 .. r0 + nr
  const int per = (p + (int)gridDim.y - 1) / (int)gridDim.y, r0 = (int)blockIdx.y * per;
  const int nr = min(per, p - r0);
  if (nr <= 0) return;
  double2 *bs = s_loc, *ts = bs + 27 * P1, *l2l = ts + 27 * P1, *pl = l2l + P1;
  double2 *zs = pl + P1;                   // [star][l]
  double2 *sq = zs + MM_LOCAL_STARS * P1;  // [star][MM_POW_BITS]
  double *sm = reinterpret_cast<double *>(sq + MM_LOCAL_STARS * MM_POW_BITS);  // [star]
  double *fs = sm + MM_LOCAL_STARS;        // [star][l]
  int lv, nx, ny;
  double zx, zy, L;
  node_geom(T, node, lv, nx, ny, zx, zy, L);
  const int64_t parent = T.parent[node];

  // the sources in the order of the parent's neighbours (row-major) and their
  // children: slot t = 4 neighbour + child
  if (tid < 32) {
    const int k = tid >> 2, c = tid & 3, j = k < 4 ? k : k + 1;
    const int qx = (nx >> 1) + j % 3 - 1, qy = (ny >> 1) + j / 3 - 1, side = 1 << (level - 1);
    bool on = false;
    int src = 0, slot = -1;
    if (qx >= 0 && qy >= 0 && qx < side && qy < side) {
      const int qid = T.nb[9 * parent + j];
      if (qid < 0) {
        if (c == 0) atomicOr(err, ERR_TREE_INVARIANT);
      } else {
        const int fc = T.first_child[qid];
        if (fc >= 0) {
          const int ox = 2 * qx + (c & 1) - nx, oy = 2 * qy + (c >> 1) - ny;
          src = fc + c;
          on = abs(ox) > 1 || abs(oy) > 1;  // else a neighbour: near field
          slot = (oy + 3) * 7 + (ox + 3);
        } else {
          // unsplit parent-neighbour: adjacent to the node unless its 2x2
          // level cells all lie at Chebyshev distance >= 2
          const int x0 = 2 * qx, y0 = 2 * qy;
          const bool adj =
              (x0 + 1 >= nx - 1 && x0 <= nx + 1) && (y0 + 1 >= ny - 1 && y0 <= ny + 1);
          on = c == 0 && !adj;
          src = qid;
        }
      }
    }
    on = on && T.sbeg[src] < T.send[src];
    const unsigned m = __ballot_sync(0xffffffffu, on);
    if (on) {
      const int r = __popc(m & ((1u << tid) - 1u));
      S.src[r] = src;
      S.slot[r] = slot;
    }
    if (tid == 0) S.n = __popc(m);
  }
  __syncthreads();
  const int ns = S.n;

  // factored M2L: b_k = (-1/z0)^k a_k, then
  // c_l += (1/z0)^l (-a_0 / l + sum_k C(l+k-1, k-1) b_k)
  const double2 *pw = MLop + (int64_t)P1 * P1;  // per slot: powers of -1/z0, of 1/z0
  for (int idx = tid; idx < ns * P1; idx += MM_LOCAL_THREADS) {
    const int s = idx / P1, k = idx - s * P1, slot = S.slot[s];
    if (slot < 0) continue;
    const double2 a = mp[(int64_t)S.src[s] * P1 + k];
    bs[idx] = k ? cfma(pw[(int64_t)slot * 2 * P1 + k], a, make_double2(0.0, 0.0)) : a;
  }
  for (int k = tid; k < P1; k += MM_LOCAL_THREADS) pl[k] = loc[parent * P1 + k];
  __syncthreads();
  // L2L from the parent: real parts by the last two warps' threads, imaginary
  // parts by the first two's (an FP64 instruction takes 64 cycles of a warp's
  // quarter of the SM, so the two halves of a complex sum go to two quarters)
  const int half = MM_LOCAL_THREADS / 2, hr = tid & (half - 1), im = tid < half;
  if (hr >= half - nr) {
    const int l = r0 + half - hr;
    const int q = (nx & 1) | ((ny & 1) << 1);
    const double2 *op = LLop + (int64_t)q * P1 * P1;
    double acc = 0.0;
#pragma unroll 4
    for (int k = l; k <= p; k++) acc = cfma_part(op[k * P1 + l], pl[k], acc, im);
    (im ? &l2l[l].y : &l2l[l].x)[0] = acc;
  }
  const double *bt = reinterpret_cast<const double *>(MLop);  // binomials [k][l], 1/l at k = 0
  const int G = MM_LOCAL_THREADS / nr;  // (nr <= MM_PMAX < MM_LOCAL_THREADS)
  const int g = tid / nr, l = r0 + tid - g * nr + 1;
  const double il = bt[l];
  for (int s0 = g < G ? g : ns; __any_sync(0xffffffffu, s0 < ns); s0 += 2 * G) {
    // (a P2L source's entry is not formed: its sum is not used)
    const int s1 = s0 + G;
    const bool on0 = s0 < ns, on1 = s1 < ns;
    const double2 *b0 = bs + (on0 ? s0 : 0) * P1, *b1 = bs + (on1 ? s1 : 0) * P1;
    double x0 = -b0[0].x * il, y0 = -b0[0].y * il;
    if (__any_sync(0xffffffffu, on1)) {
      double x1 = -b1[0].x * il, y1 = -b1[0].y * il;
#pragma unroll 4
      for (int k = 1; k <= p; k++) {
        const double b = bt[k * P1 + l];
        const double2 u = b0[k], v = b1[k];
        x0 = fma(b, u.x, x0);
        y0 = fma(b, u.y, y0);
        x1 = fma(b, v.x, x1);
        y1 = fma(b, v.y, y1);
      }
      if (on1) ts[s1 * P1 + l] = make_double2(x1, y1);
    } else {
#pragma unroll 4
      for (int k = 1; k <= p; k++) {
        const double b = bt[k * P1 + l];
        const double2 u = b0[k];
        x0 = fma(b, u.x, x0);
        y0 = fma(b, u.y, y0);
      }
    }
    if (on0) ts[s0 * P1 + l] = make_double2(x0, y0);
  }
  __syncthreads();
  // the factors (1/z0)^l of the M2L sources, in place of their multipoles
  for (int idx = tid; idx < ns * nr; idx += MM_LOCAL_THREADS) {
    const int s = idx / nr, k = r0 + idx - s * nr + 1, slot = S.slot[s];
    if (slot >= 0) bs[s * P1 + k] = pw[(int64_t)slot * 2 * P1 + P1 + k];
  }
  __syncthreads();

  // add up row `row` in the order of the list, real and imaginary parts apart
  const bool on = hr < nr;
  const int row = r0 + hr + 1;
  double acc = on ? (im ? l2l[row].y : l2l[row].x) : 0.0;
  const double invL = inv_pow2(L);
  for (int s = 0; s < ns; s++) {
    const int slot = S.slot[s];
    if (slot >= 0) {
      if (on) acc = cfma_part(bs[s * P1 + row], ts[s * P1 + row], acc, im);
      continue;
    }
    // P2L: the leaf's stars, staged; block-uniform.  Powers and weights of
    // every (star, row) side by side, then added up star by star.
    const int b = T.sbeg[S.src[s]], e = T.send[S.src[s]];
    for (int c = b; c < e; c += MM_LOCAL_STARS) {
      const int cnt = min(MM_LOCAL_STARS, e - c);
      __syncthreads();
      if (tid < cnt) {
        const double2 zeta =
            make_double2((T.sx[c + tid] - zx) * invL, (T.sy[c + tid] - zy) * invL);
        const double d = zeta.x * zeta.x + zeta.y * zeta.y;
        powers_of_two(make_double2(zeta.x / d, -zeta.y / d), p, sq + tid * MM_POW_BITS);
        sm[tid] = T.sm[c + tid];
      }
      __syncthreads();
      if (g < G)
        for (int i = g; i < cnt; i += G) {
          zs[i * P1 + l] = power_of(sq + i * MM_POW_BITS, l);
          fs[i * P1 + l] = div_by(-sm[i], (double)l, il);
        }
      __syncthreads();
      if (on)
        for (int i = 0; i < cnt; i++) {
          const double2 zl = zs[i * P1 + row];
          acc = fma(fs[i * P1 + row], im ? zl.y : zl.x, acc);
        }
    }
  }
  if (on) (im ? &loc[node * P1 + row].y : &loc[node * P1 + row].x)[0] = acc;  // (c_0 has no reader)
}

// ---------------------------------------------------------------------------
// Leaf records.  A block of 128 threads forms 16 consecutive sub-cell records
// (one leaf's with the default 4 x 4 sub-cells), eight lanes a record.
// ---------------------------------------------------------------------------
#define MM_REC 16  // records per block
#define MM_REC_THREADS (8 * MM_REC)

// The near field of the block's leaves: the leaf, its same-level neighbour
// cells that are nodes (with all their descendants), and the unsplit nodes one
// level up covering the missing neighbour cells, in row-major order and each
// once.  Star i of leaf q is off[q][k] + i for the first k with i < end[q][k].
struct NearRanges {
  int off[MM_REC][9], end[MM_REC][9];
};

__device__ __forceinline__ void near_ranges(const TreeDev &T, const int32_t *active_list,
                                            int64_t first_leaf, int n_leaf, NearRanges &N,
                                            unsigned *err) {
  const int lane = threadIdx.x & 31, k = threadIdx.x & 15;
  for (int q0 = 0; q0 < n_leaf; q0 += MM_REC_THREADS / 16) {
    const int q = q0 + (threadIdx.x >> 4);
    int src = -1, key = -2 - lane;
    bool up = false;
    if (q < n_leaf && k < 9) {
      const int64_t node = active_list[first_leaf + q];
      const int level = T.lvl[node], side = 1 << level;
      uint32_t nx, ny;
      morton_decode(T.code[node], nx, ny);
      const int x = (int)nx + k % 3 - 1, y = (int)ny + k / 3 - 1;
      if (x >= 0 && y >= 0 && x < side && y < side) {
        src = T.nb[9 * node + k];
        if (src < 0) {
          up = true;
          src = T.nb[9 * (int64_t)T.parent[node] + ((y >> 1) - (int)(ny >> 1) + 1) * 3 +
                     ((x >> 1) - (int)(nx >> 1) + 1)];
          if (src < 0) atomicOr(err, ERR_TREE_INVARIANT);
          if (src >= 0) key = src;
        }
      }
    }
    // a coarser node covers several cells: taken at the first
    const unsigned same = __match_any_sync(0xffffffffu, key) & (0xffffu << (lane & 16));
    if (up && (same & ((1u << lane) - 1u))) src = -1;
    const int b = src >= 0 ? T.sbeg[src] : 0, cnt = src >= 0 ? T.send[src] - b : 0;
    int incl = cnt;
#pragma unroll
    for (int d = 1; d < 16; d <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, incl, d, 16);
      if (k >= d) incl += u;
    }
    if (q < n_leaf && k < 9) {
      N.off[q][k] = b - (incl - cnt);
      N.end[q][k] = incl;
    }
  }
}

__device__ __forceinline__ int near_star(const NearRanges &N, int q, int i) {
  int k = 0;
  while (k < 8 && i >= N.end[q][k]) k++;
  return N.off[q][k] + i;
}

// Sub-cell record g (records are numbered 4^s t + q for active leaf t, q
// row-major with y major): its leaf's node and, along axis ax, the leaf's and
// the sub-cell's centre.
__device__ __forceinline__ void sub_cell_axis(const TreeDev &T, const FmmConst &C, int64_t node,
                                              int64_t g, int ax, double &z, double &L, double &c,
                                              double &Lq) {
  const int ns = 1 << C.sub, q = (int)(g & (ns * ns - 1));
  const int qa = ax ? q >> C.sub : q & (ns - 1);
  int level, nx, ny;
  double zx, zy;
  node_geom(T, node, level, nx, ny, zx, zy, L);
  z = ax ? zy : zx;
  Lq = L * pow2(-C.sub);
  c = z + (double)(2 * qa + 1 - ns) * Lq;
}

// Whether a star of the leaf's near field stays in the sub-cell's direct
// sum: without sub-cells every one does; with them, those within the
// (2 MM_NEAR_K + 1)^2 block of sub-cells around it (L-inf distance below
// (2 MM_NEAR_K + 1) L_q from its centre).  The others join its local
// expansion (P2L), which they leave converging at least as fast as the
// ratio sqrt(2) / (2 MM_NEAR_K + 1).
__device__ __forceinline__ bool stays_direct(const FmmConst &C, double dx, double dy,
                                             double Lq) {
  if (C.sub == 0) return true;
  const double hw = (2 * MM_NEAR_K + 1) * Lq;
  return fabs(dx) < hw && fabs(dy) < hw;
}

// Direct-sum stars of the block's record `rec` (all eight lanes).
__device__ __forceinline__ int count_direct(const TreeDev &T, const FmmConst &C,
                                            const NearRanges &N, int q, int total, int longest,
                                            double cx, double cy, double Lq, unsigned &mine) {
  const int j = threadIdx.x & 7, sh = threadIdx.x & 24;
  mine = ~0u;
  if (C.sub == 0) return total;
  mine = 0u;
  int cnt = 0;
  for (int c = 0; c < longest; c += 8) {
    bool d = false;
    if (c + j < total) {
      const int i = near_star(N, q, c + j);
      d = stays_direct(C, T.sx[i] - cx, T.sy[i] - cy, Lq);
      if (d && c < 256) mine |= 1u << (c >> 3);
    }
    cnt += __popc((__ballot_sync(0xffffffffu, d) >> sh) & 0xffu);
  }
  return cnt;
}

// Direct-sum stars of all records, added to *total (the plan sizes their
// arrays with it).
__global__ void __launch_bounds__(MM_REC_THREADS)
    k_near_count(TreeDev T, FmmConst C, int64_t n_rec, const int32_t *active_list,
                 unsigned *total, unsigned *err) {
  grid_begin();
  __shared__ NearRanges N;
  const int n_leaf_max = MM_REC >> (2 * C.sub);
  const int64_t g0 = (int64_t)blockIdx.x * MM_REC, first_leaf = g0 >> (2 * C.sub);
  const int n_leaf = (int)min((int64_t)n_leaf_max, (n_rec >> (2 * C.sub)) - first_leaf);
  near_ranges(T, active_list, first_leaf, n_leaf, N, err);
  __syncthreads();
  const int rec = threadIdx.x >> 3, q = rec >> (2 * C.sub);
  const bool valid = g0 + rec < n_rec;
  double cx = 0.0, cy = 0.0, z, L, Lq = 0.0;
  if (valid) {
    const int64_t node = active_list[first_leaf + q];
    sub_cell_axis(T, C, node, g0 + rec, 0, z, L, cx, Lq);
    sub_cell_axis(T, C, node, g0 + rec, 1, z, L, cy, Lq);
  }
  const int mine = valid ? N.end[q][8] : 0;
  const int longest = __reduce_max_sync(0xffffffffu, mine);
  unsigned direct;
  const int cnt = count_direct(T, C, N, valid ? q : 0, mine, longest, cx, cy, Lq, direct);
  if ((threadIdx.x & 7) == 0 && cnt) atomicAdd(total, (unsigned)cnt);
}

// Complex product a b in FP32 with a fixed order of rounding (a sum of two
// products could be contracted either way).
__device__ __forceinline__ float2 cmul32(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -__fmul_rn(a.y, b.y)), fmaf(a.x, b.y, __fmul_rn(a.y, b.x)));
}

// Powers u^k of the sub-cells' positions u = (z_q - z_c)/L in their leaf, in
// FP64 and FP32, [k][q], and the binomials C(n + m, n) in FP32, [n][m]: what
// every re-centring of a plan shares.
__global__ void k_sub_tables(int sub, int p, double2 *up, float2 *fp, float *bin) {
  grid_begin();
  const int ns = 1 << sub, NS = ns * ns, t = threadIdx.x;
  if (t < NS) {
    const double ux = (double)(2 * (t & (ns - 1)) + 1 - ns) / ns;
    const double uy = (double)(2 * (t >> sub) + 1 - ns) / ns;
    const double2 u = make_double2(ux, uy);
    const float2 fu = make_float2((float)ux, (float)uy);
    double2 w = make_double2(1.0, 0.0);
    float2 fw = make_float2(1.f, 0.f);
    for (int k = 0; k <= p; k++) {
      up[k * NS + t] = w;
      fp[k * NS + t] = fw;
      w = cmul(w, u);
      fw = cmul32(fw, fu);
    }
  }
  for (int n = t; n <= p; n += blockDim.x) {
    float binom = 1.f;
    for (int l = n; l <= p; l++) {
      bin[n * (p + 1) + l - n] = binom;
      binom = binom * (float)(l + 1) / (float)(l + 1 - n);
    }
  }
}

// 1/x: hardware approximation refined by two Newton-Raphson steps.
__device__ __forceinline__ double rcp_near(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  double e = fma(-x, y, 1.0);
  y = fma(y, e, y);
  e = fma(-x, y, 1.0);
  return fma(y, e, y);
}
// a / x from y ~ 1/x: the quotient corrected by its exact remainder.
__device__ __forceinline__ double div_near(double a, double x, double y) {
  const double q = a * y;
  return fma(fma(-x, q, a), y, q);
}

// x / n for a small integer n, correctly rounded (Markstein's correction).
__device__ __forceinline__ float div_by_f(float x, float n, float inv_n) {
  const float q = x * inv_n;
  return fmaf(fmaf(-n, q, x), inv_n, q);
}

// Place of coefficient k's real part in its record's floats (the imaginary
// part two further): pairs are stored real parts first.
__device__ __forceinline__ int coef_slot(int k) { return 4 * (k >> 1) + (k & 1); }


// Shared memory of k_leaf_finalize<NB>.
template <int NB>
struct RecSmem {
  NearRanges N;
  double c[2][MM_REC], r[2][MM_REC], Lq[MM_REC], d1[2][MM_REC];
  float fs[MM_REC];                         // 1 / (L_q delta)
  double star[MM_REC][8][3];                // far stars of a round: mass, 1/w; at the end
                                            // [2]: a lane's share of the direct mass
  float2 v[MM_REC][8 * (NB - 1) + 2];       // their terms m w^-n / n
  float F[MM_REC];
  int cnt[MM_REC];
  unsigned off[MM_REC], base;
  double2 lg[MM_REC][4];                    // corner logarithms (rectangular region)
};

// The leaf's local expansion psi = sum_l c_l zeta^l, zeta = (z - z_c)/L, is
// re-centred exactly on each sub-cell's centre z_q (an L2L translation to a
// descendant of the leaf, which receives no further M2L terms: its far field
// is the leaf's):
//   d_n = (L_q/L)^n sum_{l>=n} C(l, n) c_l u^(l-n),  u = (z_q - z_c)/L;
// the leaf's near-field stars that leave the direct sum (stays_direct) add
// their own expansion about z_q (P2L): m log(z - z_i) contributes
//   d_n += -m / (n w^n),  w = (z_i - z_q)/L_q,  n >= 1,
// and the result is kept to n <= p_eval.  A record's coefficients
// e_n = n d_n / (L_q delta), n = 2..p_eval, take coef_stride(p_eval) slots
// (an even count, zero-padded) so the kernel loads them in pairs; its direct
// stars are stored in its own grid frame.  d_1 sets the FP64 image of the
// centre and is formed in FP64; d_2..d_pe are stored as FP32 coefficients,
// scaled to the sub-cell (terms decay like the convergence ratio), and are
// formed in FP32 from FP32 copies of the leaf's coefficients (GB300's FP64
// rate is 1/64 of its FP32 rate).
//
// Bound by the FP64 pipe where there are many records (two lanes an SM: the
// stars' positions and 1/w, the centre's image) and by the length of a
// record's chain of steps where there are few.  Eight lanes a record: a lane
// sums every eighth n of d_n, the stars' FP64 work and powers go one to a
// lane, eight at a time, and their terms are then added up n by n in the
// stars' order; the direct stars of a record are only noted in that pass and
// put into its frame together; powers and binomials come from the plan's
// tables; 32 threads form the 16 records' centres, d_1 and images, one axis
// each.  Records reserve their direct stars' slots themselves.  67 000 records
// of 50 000 stars: 307 us with a thread a record (after a count and a scan of
// 32 us), 162 us like this (171 with IEEE divisions by the grid steps and the
// pixel, and the near stars tested twice), 167 with the direct masses' FP64 sum; a 48^2 map's 848 records 160 and 24 us.
// NB >= p_eval.
template <int NB>
__global__ void __launch_bounds__(MM_REC_THREADS) k_leaf_finalize(
    TreeDev T, FmmConst C, int64_t n_rec, const int32_t *active_list, SubTables tb,
    const double2 *loc, LeafRec *leaf, NearPos *near_pos, float *near_m,
    float2 *coef, unsigned *near_total, unsigned near_cap, unsigned *err) {
  grid_begin();
  extern __shared__ __align__(16) unsigned char s_rec[];
  RecSmem<NB> &S = *reinterpret_cast<RecSmem<NB> *>(s_rec);
  const int p = C.p, P1 = p + 1, pe = min(C.p_eval, NB), cs = coef_stride(pe);
  const int sub2 = 2 * C.sub, NS = 1 << sub2, bs = P1 | 1;
  float2 *cf = reinterpret_cast<float2 *>(&S + 1);  // [leaf][l]
  float2 *fp = cf + (MM_REC >> sub2) * P1;          // [k][q]
  float *bin = reinterpret_cast<float *>(fp + P1 * NS);  // [n][m], stride bs
  const int tid = threadIdx.x, rec = tid >> 3, j = tid & 7, sh = tid & 24;
  const int64_t g0 = (int64_t)blockIdx.x * MM_REC, g = g0 + rec;
  const int64_t first_leaf = g0 >> sub2;
  const int n_leaf = (int)min((int64_t)(MM_REC >> sub2), (n_rec >> sub2) - first_leaf);
  const int n_here = n_leaf << sub2;  // records of this block
  const bool valid = rec < n_here;
  const int q = valid ? rec >> sub2 : 0, sq = rec & (NS - 1);

  near_ranges(T, active_list, first_leaf, n_leaf, S.N, err);
  for (int i = tid; i < n_leaf * P1; i += MM_REC_THREADS) {
    const int lf = i / P1;
    const double2 c = loc[(int64_t)active_list[first_leaf + lf] * P1 + (i - lf * P1)];
    cf[i] = make_float2((float)c.x, (float)c.y);
  }
  for (int i = tid; i < P1 * NS; i += MM_REC_THREADS) fp[i] = tb.fp[i];
  for (int i = tid; i < (pe + 1) * P1; i += MM_REC_THREADS)
    bin[(i / P1) * bs + i % P1] = tb.bin[i];

  // threads 0..31: record tid / 2, axis tid % 2
  const int rec2 = tid >> 1, ax = tid & 1;
  int ref = 0;
  float fc = 0.f;
  double ctr = 0.0, Lq2 = 1.0;
  int node2 = 0;
  if (tid < 32 && rec2 < n_here) {
    node2 = active_list[first_leaf + (rec2 >> sub2)];
    double z, L;
    sub_cell_axis(T, C, node2, g0 + rec2, ax, z, L, ctr, Lq2);
    // the grid vertex nearest the sub-cell centre
    const double h = ax ? C.hy : C.hx, ih = ax ? C.inv_hy : C.inv_hx, x0 = ax ? C.y0 : C.x0;
    const double gi = rint(div_near(ctr - x0, h, ih)), xr = x0 + gi * h;
    ref = (int)gi;
    fc = (float)div_near(ctr - xr, h, ih);
    S.c[ax][rec2] = ctr;
    S.r[ax][rec2] = xr;
    if (!ax) {
      S.Lq[rec2] = Lq2;
      S.fs[rec2] = (float)(C.inv_delta * inv_pow2(Lq2));
    }
    // d_1 of the leaf's expansion (pe >= 1: p >= 1)
    const double2 *c = loc + (int64_t)node2 * P1;
    double sum = 0.0;
#pragma unroll 4
    for (int l = 1; l <= p; l++) {
      const double2 cl = c[l], u = tb.up[(l - 1) * NS + (rec2 & (NS - 1))];
      sum = fma(c_int[l], fma(cl.x, ax ? u.y : u.x, cl.y * flip(ax ? u.x : u.y, !ax)), sum);
    }
    S.d1[ax][rec2] = sum * pow2(-C.sub);
  }
  __syncthreads();

  // re-centred coefficients: lane j holds n = 2 + j, 10 + j, ...
  constexpr int NPL = (NB - 1 + 7) / 8;
  float2 d[NPL];
  {
    const float2 *c = cf + q * P1;
#pragma unroll
    for (int i = 0; i < NPL; i++) {
      const int n = 2 + j + 8 * i;
      float sx = 0.f, sy = 0.f;
      if (n <= pe) {
        for (int m = 0; n + m <= p; m++) {
          const float2 t = cmul32(c[n + m], fp[m * NS + sq]);
          const float b = bin[n * bs + m];
          sx = fmaf(b, t.x, sx);
          sy = fmaf(b, t.y, sy);
        }
      }
      const float rn = __int_as_float((127 - C.sub * n) << 23);  // (L_q/L)^n = 2^(-s n)
      d[i] = make_float2(sx * rn, sy * rn);
    }
  }

  // slots of the direct stars
  const double cx = S.c[0][valid ? rec : 0], cy = S.c[1][valid ? rec : 0];
  const double Lq = S.Lq[valid ? rec : 0];
  const int total = valid ? S.N.end[q][8] : 0;
  const int longest = __reduce_max_sync(0xffffffffu, total);
  unsigned direct;  // the lane's direct stars among the first 256
  const int n_dir = count_direct(T, C, S.N, q, total, longest, cx, cy, Lq, direct);
  if (j == 0) S.cnt[rec] = n_dir;
  __syncthreads();
  if (tid == 0) {
    int sum = 0;
    for (int r = 0; r < MM_REC; r++) {
      const int c = S.cnt[r];
      S.cnt[r] = sum;
      sum += c;
    }
    S.base = atomicAdd(near_total, (unsigned)sum);
  }
  __syncthreads();
  const unsigned off = S.base + (unsigned)S.cnt[rec];
  // (the plan counted the same stars: a record without room is an error)
  const bool room = off + (unsigned)n_dir <= near_cap;
  if (!room && j == 0) atomicOr(err, ERR_NEAR_SLOTS);

  // near-field stars, eight at a time: into the expansion, or noted as direct
  double d1 = j < 2 ? S.d1[j][rec] : 0.0;
  int k = 0;
  for (int c = 0; c < longest; c += 8) {
    const bool on = c + j < total;
    bool dir = false;
    int i = 0;
    if (on) {
      i = near_star(S.N, q, c + j);
      dir = c < 256 ? direct >> (c >> 3) & 1u
                    : stays_direct(C, T.sx[i] - cx, T.sy[i] - cy, Lq);
      if (!dir) {
        const double dx = T.sx[i] - cx, dy = T.sy[i] - cy;
        // 1/w = L_q / (z_i - z_q); d_1 in FP64, the rest in FP32
        const double den = fma(dx, dx, dy * dy), rc = rcp_near(den);
        const double ix = div_near(Lq * dx, den, rc), iy = div_near(-Lq * dy, den, rc);
        const double m = T.sm[i];
        S.star[rec][j][0] = m;
        S.star[rec][j][1] = ix;
        S.star[rec][j][2] = iy;
        const float2 iw = make_float2((float)ix, (float)iy);
        const float fm = (float)m;
        float2 t = make_float2(fmaf(iw.x, iw.x, -__fmul_rn(iw.y, iw.y)), 2.f * iw.x * iw.y);  // w^-2
        float2 *v = &S.v[rec][j * (NB - 1)];
#pragma unroll
        for (int n = 2; n <= NB; n++) {
          v[n - 2] = make_float2(div_by_f(fm * t.x, (float)n, 1.f / n),
                                 div_by_f(fm * t.y, (float)n, 1.f / n));
          t = cmul32(t, iw);
        }
      }
    }
    const unsigned md = (__ballot_sync(0xffffffffu, on && dir) >> sh) & 0xffu;
    unsigned mf = (__ballot_sync(0xffffffffu, on && !dir) >> sh) & 0xffu;
    if (on && dir && room) near_m[off + k + __popc(md & ((1u << j) - 1u))] = __int_as_float(i);
    k += __popc(md);
    __syncwarp();
    for (; mf; mf &= mf - 1) {
      const int t = __ffs(mf) - 1;
      if (j < 2) d1 -= S.star[rec][t][0] * S.star[rec][t][1 + j];
#pragma unroll
      for (int e = 0; e < NPL; e++) {
        const int n = 2 + j + 8 * e;
        if (n <= pe) {
          const float2 v = S.v[rec][t * (NB - 1) + n - 2];
          d[e].x -= v.x;
          d[e].y -= v.y;
        }
      }
    }
    __syncwarp();
  }
  // the direct stars in the record's grid frame, and their mass (for the
  // culling bound alone, in FP64: a bound has to hold for any number of stars)
  double md = 0.0;
  if (room) {
    const double xr = S.r[0][rec], yr = S.r[1][rec];
    for (int t = j; t < n_dir; t += 8) {
      const int i = __float_as_int(near_m[off + t]);
      const double sxg = div_near(T.sx[i] - xr, C.hx, C.inv_hx);
      const double syg = div_near(T.sy[i] - yr, C.hy, C.inv_hy);
      const double Kx = rint(sxg), Ky = rint(syg);
      NearPos np;
      np.Kx = (float)Kx;
      np.fx = (float)(sxg - Kx);
      np.Ky = (float)Ky;
      np.fy = (float)(syg - Ky);
      near_pos[off + t] = np;
      const double m = T.sm[i];
      near_m[off + t] = (float)m;
      md = t < 8 ? m : md + m;
    }
  }
  S.star[rec][j][2] = md;

  // Rectangular star region: the sheet's part beyond -kappa_star z is the
  // conjugate of At, analytic inside the rectangle, so its potential joins
  // the expansion like a far source: d_n += At^(n-1)(z_q) L_q^n / n!, with
  //   At'    = (kappa_star i / pi) sum_a s_a (-log(a - z)) - kappa_star,
  //   At^(k) = (kappa_star i / pi) sum_a s_a (k - 2)! / (a - z)^(k - 1), k >= 2,
  // i.e. d_n += (kappa_star i / pi) L_q^2 sum_a s_a r_a^(n-2) / (n (n-1) (n-2))
  // for n >= 3, r_a = L_q / (a - z_q).  No per-ray cost.
  if (C.rect_c1 > 0.0) {
    __syncthreads();
    if (tid < 4 * MM_REC && (tid >> 2) < n_here) {
      double ax_, ay_, sg;
      rect_corner(C.rect_c1, C.rect_c2, tid & 3, ax_, ay_, sg);
      S.lg[tid >> 2][tid & 3] = clog64(ax_ - S.c[0][tid >> 2], ay_ - S.c[1][tid >> 2]);
    }
    __syncthreads();
    if (tid < n_here) {
      const double zx = S.c[0][tid], zy = S.c[1][tid], lq = S.Lq[tid];
      const double f = C.kappa_star / 3.14159265358979323846;
      double gx = 0.0, gy = 0.0, lx = 0.0, ly = 0.0, rx[4], ry[4], px[4], py[4], sg[4];
      double dmin2 = 1e300;
#pragma unroll
      for (int a = 0; a < 4; a++) {
        double ax_, ay_;
        rect_corner(C.rect_c1, C.rect_c2, a, ax_, ay_, sg[a]);
        const double dx = ax_ - zx, dy = ay_ - zy, w = lq / (dx * dx + dy * dy);
        dmin2 = fmin(dmin2, dx * dx + dy * dy);
        const double2 l = S.lg[tid][a];
        gx += sg[a] * (dx * l.x - dy * l.y);
        gy += sg[a] * fma(dy, l.x, dx * l.y);
        lx -= sg[a] * l.x;
        ly -= sg[a] * l.y;
        rx[a] = dx * w;   // L_q / (a - z_q)
        ry[a] = -dy * w;
        px[a] = 1.0;      // r_a^(n-2)
        py[a] = 0.0;
      }
      // At(z_q) (see rect_sheet_At)
      S.star[tid][0][0] = -f * gy - C.kappa_star * (2.0 * C.rect_c1 + zx);
      S.star[tid][0][1] = f * gx - C.kappa_star * zy;
      // the series converges like sqrt(2) L_q / (distance to the nearest
      // corner) over the record; beyond 1/2 its truncation is not negligible
      // (only sub-cells meeting the ray grid are ever evaluated)
      const bool on_grid = zx + lq >= C.x0 && zx - lq <= C.x1 && zy + lq >= C.y0 &&
                           zy - lq <= C.y1;
      if (on_grid && 2.0 * lq * lq > 0.25 * dmin2) atomicOr(err, ERR_RECT_CORNER);
      const double l2 = lq * lq;
      float2 *v = S.v[tid];
      v[0] = make_float2((float)((-f * ly - C.kappa_star) * l2 * 0.5), (float)(f * lx * l2 * 0.5));
      for (int n = 3; n <= pe; n++) {
        double sx = 0.0, sy = 0.0;
#pragma unroll
        for (int a = 0; a < 4; a++) {
          const double t = px[a] * rx[a] - py[a] * ry[a];
          py[a] = px[a] * ry[a] + py[a] * rx[a];
          px[a] = t;
          sx += sg[a] * px[a];
          sy += sg[a] * py[a];
        }
        const double w = f * l2 / ((double)n * (n - 1) * (n - 2));  // times i
        v[n - 2] = make_float2((float)(-w * sy), (float)(w * sx));
      }
    }
    __syncthreads();
    if (valid) {
      if (j < 2) d1 = fma(S.star[rec][0][j], Lq, d1);
#pragma unroll
      for (int e = 0; e < NPL; e++) {
        const int n = 2 + j + 8 * e;
        if (n <= pe) {
          d[e].x += S.v[rec][n - 2].x;
          d[e].y += S.v[rec][n - 2].y;
        }
      }
    }
  }

  // coefficients, and the bound of the evaluated series over the sub-cell:
  // sum_n |e_n| zeta_max^(n-1)
  const float fs = S.fs[valid ? rec : 0];
  const float hmax = (float)fmax(C.hx, C.hy), fLq = (float)Lq;
  const float zmax = 1.4142137f * (fLq + hmax) / fLq;
  float F = 0.f;
#pragma unroll
  for (int e = 0; e < NPL; e++) {
    const int n = 2 + j + 8 * e;
    if (n <= pe) {
      const float2 v = make_float2(n * d[e].x * fs, n * d[e].y * fs);
      if (valid) {
        float *out = reinterpret_cast<float *>(coef + g * cs) + coef_slot(n - 2);
        out[0] = v.x;
        out[2] = v.y;
      }
      F = fmaf(sqrtf(fmaf(v.x, v.x, v.y * v.y)), powf(zmax, (float)(n - 1)), F);
    }
  }
  for (int b = 1; b < 8; b <<= 1) F += __shfl_xor_sync(0xffffffffu, F, b);
  if (valid && j == 0) {
    for (int kk = pe - 1; kk < cs; kk++) {
      float *out = reinterpret_cast<float *>(coef + g * cs) + coef_slot(kk);
      out[0] = out[2] = 0.f;
    }
    S.F[rec] = F;
    S.cnt[rec] = room ? n_dir : 0;
    S.off[rec] = off;
  }
  if (valid && j < 2) S.d1[j][rec] = d1;
  __syncthreads();
  if (tid >= 32) return;

  // FP64 image of the sub-cell centre: macro model + sheet - far field there
  const bool here = rec2 < n_here;
  const int r2 = here ? rec2 : 0;
  const double ak = 1.0 - C.kappa + C.kappa_star, a = ax ? ak - C.gamma : ak + C.gamma;
  const double iLq = inv_pow2(Lq2), dq = S.d1[ax][r2] * iLq;
  // - conj(d1/L_q)
  const double W = ax ? fma(a, ctr, dq) : __dsub_rn(__dmul_rn(a, ctr), dq);
  double U = div_near(W - (ax ? C.loy : C.lox), C.delta, C.inv_delta);
  // |Ui| < 2^28 keeps vertex pixel indices within +-2^29
  U = fmin(fmax(U, -2.0e8), 2.0e8);
  const double Ui = floor(U);
  const int iU = (int)Ui;
  const float fU = (float)(U - Ui), zs = (float)((ax ? C.hy : C.hx) * iLq);

  // Culling bounds.  A vertex of this sub-cell (grid offset within
  // L_s + h of its centre) lands at the centre's image plus the macro term,
  // the evaluated far-field series and the direct stars' deflection, all in
  // pixels.  The first two stay within a box of half-widths B about (U, V):
  // |macro| <= |1 - kappa + kappa_* +- gamma| (L_s + h)/delta and
  // |series| <= F.  If that box lies D pixels beyond a map edge, a vertex
  // whose direct stars are all farther than M_direct / (delta (D - margin))
  // is deflected by them less than D - margin, so it lands beyond that edge
  // too.  (F is a sum of at most 63 FP32 terms: 1 % covers its rounding.)
  const double margin = 2.0;
  const double B = div_near(fabs(a) * (Lq2 + fmax(C.hx, C.hy)), C.delta, C.inv_delta) +
                   1.01 * (double)S.F[r2];
  const double Dlo = -(U + B), Dhi = (U - B) - (double)(ax ? C.npix_y : C.npix);
  double D = Dlo;
  int side = ax ? MM_CULL_BOTTOM : MM_CULL_LEFT;
  if (Dhi > D) D = Dhi, side = ax ? MM_CULL_TOP : MM_CULL_RIGHT;
  const bool in = U > -1.9e8 && U < 1.9e8;
  // the direct stars' mass: half of the lanes' shares by each axis' thread
  const double *m8 = &S.star[r2][4 * ax][2];
  double md2 = ((m8[0] + m8[3]) + m8[6]) + m8[9];
  md2 += __shfl_xor_sync(0xffffffffu, md2, 1);
  // axis 1's numbers to axis 0's thread, which writes the record
  const double D1 = __shfl_down_sync(0xffffffffu, D, 1);
  const int side1 = __shfl_down_sync(0xffffffffu, side, 1);
  const int in1 = __shfl_down_sync(0xffffffffu, (int)in, 1);
  const int ref1 = __shfl_down_sync(0xffffffffu, ref, 1);
  const int iU1 = __shfl_down_sync(0xffffffffu, iU, 1);
  const float fc1 = __shfl_down_sync(0xffffffffu, fc, 1);
  const float fU1 = __shfl_down_sync(0xffffffffu, fU, 1);
  const float zs1 = __shfl_down_sync(0xffffffffu, zs, 1);
  if (ax || !here) return;
  if (D1 > D) D = D1, side = side1;
  LeafRec R;
  R.i_ref = ref;
  R.j_ref = ref1;
  R.fcx = fc;
  R.fcy = fc1;
  R.Ui = iU;
  R.Vi = iU1;
  R.Uf = fU;
  R.Vf = fU1;
  R.zsx = zs;
  R.zsy = zs1;
  R.near_off = (int32_t)S.off[rec2];
  R.near_cnt = S.cnt[rec2];
  R.coef_off = (int32_t)((g0 + rec2) * cs);
  R.node = node2;
  R.cull_side = MM_CULL_NONE;
  R.cull_r2 = -1.f;
  if (C.cull && D > 2.0 * margin && in && in1) {
    const double rc = md2 / (C.delta * (D - margin) * C.hx);  // of h_x
    R.cull_side = side;
    R.cull_r2 = (float)(rc * rc * 1.01);
  }
  leaf[g0 + rec2] = R;
}

// ---------------------------------------------------------------------------
// host: operator tables and launchers
// ---------------------------------------------------------------------------

struct cplx {
  double x, y;
};
static inline cplx cm(cplx a, cplx b) { return {a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x}; }
static inline cplx cpw(cplx z, int k) {
  cplx r{1.0, 0.0};
  for (int i = 0; i < k; i++) r = cm(r, z);
  return r;
}
static inline cplx cinv(cplx z) {
  double d = z.x * z.x + z.y * z.y;
  return {z.x / d, -z.y / d};
}

// binomial coefficients C(n, k) for n <= 2 p (Pascal's triangle, FP64)
static std::vector<std::vector<double>> binomials(int nmax) {
  std::vector<std::vector<double>> C(nmax + 1, std::vector<double>(nmax + 1, 0.0));
  for (int n = 0; n <= nmax; n++) {
    C[n][0] = 1.0;
    for (int k = 1; k <= n; k++) C[n][k] = C[n - 1][k - 1] + (k <= n - 1 ? C[n - 1][k] : 0.0);
  }
  return C;
}

void build_operator_tables(int p, std::vector<double2> &MM, std::vector<double2> &ML,
                           std::vector<double2> &LL) {
  const int P1 = p + 1;
  auto C = binomials(2 * p + 1);
  // M2M factored like M2L below: op[k][l] = (z0/2)^l C(l-1, k-1) z0^-k for
  // 1 <= k <= l and op[0][l] = -(z0/2)^l / l: the real binomials (P1 x P1
  // doubles [k][l], 1/l at k = 0, at the head of P1 x P1 entries), then per
  // child quadrant the powers z0^-k and (z0/2)^l
  MM.assign((size_t)P1 * P1 + (size_t)4 * 2 * P1, make_double2(0.0, 0.0));
  double *mb = &MM[0].x;
  for (int l = 1; l <= p; l++) {
    mb[l] = 1.0 / l;
    for (int k = 1; k <= l; k++) mb[(size_t)k * P1 + l] = C[l - 1][k - 1];
  }
  LL.assign((size_t)4 * P1 * P1, make_double2(0.0, 0.0));
  ML.assign((size_t)49 * P1 * P1, make_double2(0.0, 0.0));
  for (int q = 0; q < 4; q++) {
    // M2M: child centre relative to the parent, in child half-lengths
    cplx z0{(q & 1) ? 1.0 : -1.0, (q >> 1) ? 1.0 : -1.0};
    double2 *pw = &MM[(size_t)P1 * P1 + (size_t)q * 2 * P1];
    const cplx iz = cinv(z0), hz{0.5 * z0.x, 0.5 * z0.y};
    for (int k = 0; k <= p; k++) {
      const cplx a = cpw(iz, k), b = cpw(hz, k);
      pw[k] = make_double2(a.x, a.y);
      pw[P1 + k] = make_double2(b.x, b.y);
    }
    // L2L: child centre relative to the parent, in parent half-lengths
    cplx w0{(q & 1) ? 0.5 : -0.5, (q >> 1) ? 0.5 : -0.5};
    double2 *ol = &LL[(size_t)q * P1 * P1];
    for (int l = 0; l <= p; l++) {
      const double s = std::ldexp(1.0, -l);
      for (int k = l; k <= p; k++) {
        cplx zz = cpw(w0, k - l);
        double b = C[k][l] * s;
        ol[k * P1 + l] = make_double2(zz.x * b, zz.y * b);
      }
    }
  }
  // M2L: source centre relative to the target, z0 = 2 (dx + i dy).  The
  // operator factors as op[k][l] = (1/z0)^l C(l+k-1, k-1) (-1/z0)^k for
  // k >= 1 and op[0][l] = -(1/z0)^l / l, so the table holds the real
  // binomials once (P1 x P1 doubles [k][l], with 1/l in the unused k = 0 row,
  // at the head of P1 x P1 entries) and, per
  // offset, the powers of -1/z0 (scaling the multipoles) and of 1/z0
  // (scaling the sums): P1^2 + 49 x 2 P1 entries.
  ML.assign((size_t)P1 * P1 + (size_t)49 * 2 * P1, make_double2(0.0, 0.0));
  double *lb = &ML[0].x;
  for (int l = 1; l <= p; l++) {
    lb[l] = 1.0 / l;
    for (int k = 1; k <= p; k++) lb[(size_t)k * P1 + l] = C[l + k - 1][k - 1];
  }
  for (int dy = -3; dy <= 3; dy++)
    for (int dx = -3; dx <= 3; dx++) {
      if (std::abs(dx) <= 1 && std::abs(dy) <= 1) continue;
      cplx z0{2.0 * dx, 2.0 * dy};
      cplx iz = cinv(z0);
      cplx imz = cinv(cplx{-z0.x, -z0.y});
      double2 *pw = &ML[(size_t)P1 * P1 + (size_t)((dy + 3) * 7 + (dx + 3)) * 2 * P1];
      for (int k = 0; k <= p; k++) {
        const cplx a = cpw(imz, k), b = cpw(iz, k);
        pw[k] = make_double2(a.x, a.y);
        pw[P1 + k] = make_double2(b.x, b.y);
      }
    }
}

static inline unsigned blocks_for(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }

cudaError_t launch_p2m(const TreeDev &T, int64_t n_nodes, int p, const double2 *MLop, double2 *mp,
                       cudaStream_t st) {
  if (n_nodes <= 0) return cudaSuccess;
  const int per_block = std::min(32, MM_P2M_THREADS / (p + 1));
  const size_t smem = (size_t)per_block * MM_P2M_STARS *
                      ((p + 1) * sizeof(double2) + sizeof(double));
  // (the head of MLop holds 1/k)
  launch_next(k_p2m, blocks_for(n_nodes, per_block), MM_P2M_THREADS, smem, st,
      T, n_nodes, p, per_block, reinterpret_cast<const double *>(MLop), mp);
  return cudaGetLastError();
}

cudaError_t launch_m2m(const TreeDev &T, int level, int64_t n, int p, const double2 *MMop,
                       double2 *mp, int sms, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  // 8 nodes a block fill its warps (4 children x p/2 rows each); fewer where
  // their coefficients would not fit 48 KB, and where a level's nodes would
  // leave less than two blocks an SM (a node's work is 2 us of one SM's FP64
  // pipe)
  int per_block = p <= 32 ? 8 : 4;
  while (per_block > 1 && n < 2 * (int64_t)sms * per_block) per_block >>= 1;
  const int threads = 32 * ((per_block * 4 * ((p + 1) / 2) + 31) / 32);
  const size_t smem = sizeof(double2) * 2 * per_block * 4 * (size_t)(p + 1);
  launch_next(k_m2m, blocks_for(n, per_block), threads, smem, st, T, level, n, p, per_block, MMop, mp);
  return cudaGetLastError();
}

cudaError_t launch_local(const TreeDev &T, int level, int64_t n, int p, const int32_t *node_act,
                         const double2 *MLop, const double2 *LLop, const double2 *mp,
                         double2 *loc, unsigned *err, int sms, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const size_t smem = local_smem(p);
  if (smem + sizeof(LocalSources) > 48 * 1024) {  // (the sources lie in the block's own)
    cudaError_t e = cudaFuncSetAttribute(k_local, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
  }
  // parts per node where a level's nodes (most of them inactive when the grid
  // is a small part of the star region) leave SMs idle: the levels of 16 and 64
  // nodes took 24 and 36 us in one part, 14 and 22 in four; above 20 nodes an SM
  // the pipe is busy anyway and a part costs 6 % more of it
  const unsigned parts = n <= 2 * (int64_t)sms ? 4 : n <= 20 * (int64_t)sms ? 2 : 1;
  launch_next(k_local, dim3((unsigned)n, parts), MM_LOCAL_THREADS, smem, st, T, level, n, p, node_act, MLop, LLop, mp,
                                                       loc, err);
  return cudaGetLastError();
}

cudaError_t launch_near_count(const TreeDev &T, const FmmConst &C, int64_t n_active,
                              const int32_t *active_list, unsigned *total, unsigned *err,
                              cudaStream_t st) {
  if (n_active <= 0) return cudaSuccess;
  const int64_t n = n_active << (2 * C.sub);
  launch_next(k_near_count, blocks_for(n, MM_REC), MM_REC_THREADS, 0, st, T, C, n, active_list, total, err);
  return cudaGetLastError();
}

cudaError_t launch_sub_tables(int sub, int p, double2 *up, float2 *fp, float *bin,
                              cudaStream_t st) {
  launch_next(k_sub_tables, 1, 128, 0, st, sub, p, up, fp, bin);
  return cudaGetLastError();
}

template <int NB>
static cudaError_t launch_finalize_t(const TreeDev &T, const FmmConst &C, int64_t n,
                                     const int32_t *active_list, const SubTables &tb,
                                     const double2 *loc, LeafRec *leaf, NearPos *near_pos,
                                     float *near_m, float2 *coef, unsigned *near_total,
                                     unsigned near_cap, unsigned *err, cudaStream_t st) {
  const size_t P1 = (size_t)C.p + 1;
  const size_t smem = sizeof(RecSmem<NB>) +
                      sizeof(float2) * ((MM_REC >> (2 * C.sub)) * P1 + (P1 << (2 * C.sub))) +
                      sizeof(float) * (std::min(C.p_eval, NB) + 1) * (P1 | 1);
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(k_leaf_finalize<NB>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  launch_next(k_leaf_finalize<NB>, blocks_for(n, MM_REC), MM_REC_THREADS, smem, st,
      T, C, n, active_list, tb, loc, leaf, near_pos, near_m, coef, near_total, near_cap, err);
  return cudaGetLastError();
}

cudaError_t launch_leaf_finalize(const TreeDev &T, const FmmConst &C, int64_t n_active,
                                 const int32_t *active_list, const SubTables &tb,
                                 const double2 *loc, LeafRec *leaf, NearPos *near_pos,
                                 float *near_m, float2 *coef, unsigned *near_total,
                                 unsigned near_cap, unsigned *err, cudaStream_t st) {
  if (n_active <= 0) return cudaSuccess;
  const int64_t n = n_active << (2 * C.sub);
  if (C.p_eval <= 16)
    return launch_finalize_t<16>(T, C, n, active_list, tb, loc, leaf, near_pos, near_m, coef,
                                 near_total, near_cap, err, st);
  if (C.p_eval <= 32)
    return launch_finalize_t<32>(T, C, n, active_list, tb, loc, leaf, near_pos, near_m, coef,
                                 near_total, near_cap, err, st);
  return launch_finalize_t<MM_PMAX>(T, C, n, active_list, tb, loc, leaf, near_pos, near_m, coef,
                                    near_total, near_cap, err, st);
}

}  // namespace mm
