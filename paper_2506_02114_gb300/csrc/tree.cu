// Adaptive quadtree on the device (Sec. 3.3 and App. C.1).
//
// The root is the square [-R0, R0)^2 centred on the origin.  A node splits
// into four children when the stars in the node and its same-level
// neighbour cells (those sharing a side or a corner) exceed leaf_size.  With
// this rule a split node's eight same-level neighbours always exist, every
// leaf's near field (itself, its same-level neighbours and the adjacent
// leaves one level up) holds at most leaf_size stars, and the interaction
// lists of App. C.2 are exact: at most 27 same-level nodes and at most 5
// leaves one level up.
//
// Build: Morton keys of the stars (21 bits per axis), a radix sort, then one
// level at a time: each node's eight neighbours from its parent's (a child of
// a neighbour of the parent, if that one is split), split flags from the nine
// star counts, ranks of the split nodes, and the children written in Morton
// order so that each level's node array stays sorted by code.  The levels of
// at most MM_TOP_NODES nodes are built by one block in one launch, larger
// ones by two launches each.  Every step is a short chain of dependent loads
// (a binary search runs only inside an unsplit neighbour of the parent, at
// most leaf_size stars, and over a node's own stars), so the time is latency:
// 50 000 stars take 0.20 ms (0.09 of it the sort); 0.54 ms with counts by
// binary search over all stars, one thread per node, and five launches a
// level.  The one block is the faster way up to 256 nodes a level (with 1024,
// the level of 864 took 21 us in it, 14 in two launches).
#include "mm_kernels.h"

namespace mm {

__device__ __forceinline__ int cell_of(double x, double R0) {
  const double scale = (double)(1 << MM_DMAX) / (2.0 * R0);
  double c = floor(__dmul_rn(__dadd_rn(x, R0), scale));
  c = fmin(fmax(c, 0.0), (double)((1 << MM_DMAX) - 1));
  return (int)c;
}

__global__ void k_star_keys(const double *__restrict__ pos, int64_t n, double R0,
                            uint64_t *keys, int32_t *idx) {
  grid_begin();
  int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  int cx = cell_of(pos[2 * t], R0), cy = cell_of(pos[2 * t + 1], R0);
  keys[t] = morton2((uint32_t)cx, (uint32_t)cy);
  idx[t] = (int32_t)t;
}

__global__ void k_gather_stars(const double *__restrict__ pos, const double *__restrict__ m,
                               const int32_t *idx, int64_t n, double *sx,
                               double *sy, double *sm) {
  grid_begin();
  int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  int32_t k = idx[t];
  sx[t] = pos[2 * k];
  sy[t] = pos[2 * k + 1];
  sm[t] = m[k];
}

// Neighbour s (0..7, row-major around the node without the middle) of a
// node: the node of that cell, or -1 (no node, or outside the root), and the
// cell's stars.
__device__ __forceinline__ int neighbour(const TreeDev &T, int level, int64_t node, int s,
                                         int &count) {
  count = 0;
  if (level == 0) return -1;
  const int k = s < 4 ? s : s + 1;
  const uint64_t c = T.code[node];
  uint32_t cx, cy;
  morton_decode(c, cx, cy);
  const int x = (int)cx + k % 3 - 1, y = (int)cy + k / 3 - 1, side = 1 << level;
  if (x < 0 || y < 0 || x >= side || y >= side) return -1;
  // (the parent is split, so all its neighbours inside the root are nodes)
  const int j = ((y >> 1) - (int)(cy >> 1) + 1) * 3 + ((x >> 1) - (int)(cx >> 1) + 1);
  const int q = T.nb[9 * (int64_t)T.parent[node] + j];
  if (q < 0) return -1;
  const int fc = T.first_child[q];
  if (fc >= 0) {
    const int id = fc + ((x & 1) | ((y & 1) << 1));
    count = T.send[id] - T.sbeg[id];
    return id;
  }
  const int sh = 2 * (MM_DMAX - level);
  const uint64_t key = morton2((uint32_t)x, (uint32_t)y);
  const int64_t e = T.send[q];
  const int64_t a = lower_bound_u64(T.keys, T.sbeg[q], e, key << sh);
  count = (int)(lower_bound_u64(T.keys, a, e, (key + 1) << sh) - a);
  return -1;
}

// Eight lanes per node (s = lane & 7): writes the node's neighbours and
// returns whether it splits (in all eight lanes).  Call with whole warps.
__device__ __forceinline__ bool node_split(const TreeDev &T, const TreeOut &O, int level,
                                           int64_t node, bool valid, int s, int limit) {
  int count = 0, own = 0;
  if (valid) {
    const int id = neighbour(T, level, node, s, count);
    O.nb[9 * node + (s < 4 ? s : s + 1)] = id;
    if (s == 0) O.nb[9 * node + 4] = (int32_t)node;
    own = T.send[node] - T.sbeg[node];
  }
#pragma unroll
  for (int d = 1; d < 8; d <<= 1) count += __shfl_xor_sync(0xffffffffu, count, d);
  return valid && level < MM_DMAX && count + own > limit;
}

__device__ __forceinline__ void write_child(const TreeDev &T, const TreeOut &O, int level,
                                            int64_t node, int q, int64_t id, int b, int e) {
  O.code[id] = (T.code[node] << 2) | (uint64_t)q;
  O.lvl[id] = level + 1;
  O.sbeg[id] = b;
  O.send[id] = e;
  O.parent[id] = (int32_t)node;
}

__global__ void __launch_bounds__(256) k_level_split(TreeDev T, TreeOut O, int level, int64_t n,
                                                     int limit, int32_t *split, int32_t *group,
                                                     int32_t *total) {
  grid_begin();
  __shared__ int s_n[8];
  const int64_t t = (int64_t)blockIdx.x * MM_SPLIT_GROUP + (threadIdx.x >> 3);
  const int s = threadIdx.x & 7;
  const bool f = node_split(T, O, level, T.level_off[level] + t, t < n, s, limit);
  if (s == 0 && t < n) split[t] = f;
  const unsigned m = __ballot_sync(0xffffffffu, f && s == 0);
  if ((threadIdx.x & 31) == 0) s_n[threadIdx.x >> 5] = __popc(m);
  __syncthreads();
  if (threadIdx.x == 0) {
    int c = 0;
    for (int k = 0; k < 8; k++) c += s_n[k];
    group[blockIdx.x] = c;
    if (total && c) atomicAdd(total, c);
  }
}

// Split nodes (active leaves) before group g, from the groups' counts or, where
// those are many, from their running sum (k_group_scan).  Adding up the counts
// in every block is quadratic in a level's nodes, but spares a launch (see
// MM_SUM_GROUPS).  Call with all threads of a block of 256; the sum is in *s_base
// after the block's next __syncthreads.
__device__ __forceinline__ void before_group(const int32_t *group, int64_t g, bool scanned,
                                             int *s_base) {
  int before = 0;
  if (scanned) {
    if (threadIdx.x == 0) *s_base = group[g];
    return;
  }
  for (int64_t k = threadIdx.x; k < g; k += 256) before += group[k];
  before = __reduce_add_sync(0xffffffffu, before);
  if (threadIdx.x == 0) *s_base = 0;
  __syncthreads();
  if ((threadIdx.x & 31) == 0 && before) atomicAdd(s_base, before);
}

// group[k] <- group[0] + .. + group[k - 1], one block.  16 counts a thread and
// round; the array is 16-byte aligned.
#define MM_SCAN_EACH 16
__global__ void __launch_bounds__(1024) k_group_scan(int32_t *group, int64_t n) {
  grid_begin();
  __shared__ int s_w[32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int carry = 0;
  for (int64_t base = 0; base < n; base += 1024 * MM_SCAN_EACH) {
    const int64_t k0 = base + (int64_t)threadIdx.x * MM_SCAN_EACH;
    const bool whole = k0 + MM_SCAN_EACH <= n;
    int v[MM_SCAN_EACH], sum = 0;
#pragma unroll
    for (int k = 0; k < MM_SCAN_EACH; k += 4) {
      int4 a = make_int4(0, 0, 0, 0);
      if (whole) {
        a = *reinterpret_cast<const int4 *>(group + k0 + k);
      } else {
        if (k0 + k < n) a.x = group[k0 + k];
        if (k0 + k + 1 < n) a.y = group[k0 + k + 1];
        if (k0 + k + 2 < n) a.z = group[k0 + k + 2];
        if (k0 + k + 3 < n) a.w = group[k0 + k + 3];
      }
      v[k] = a.x;
      v[k + 1] = a.y;
      v[k + 2] = a.z;
      v[k + 3] = a.w;
      sum += a.x + a.y + a.z + a.w;
    }
    int incl = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += u;
    }
    if (lane == 31) s_w[w] = incl;
    __syncthreads();
    int before = carry + incl - sum;
    for (int k = 0; k < 32; k++) {
      if (k < w) before += s_w[k];
      carry += s_w[k];
    }
#pragma unroll
    for (int k = 0; k < MM_SCAN_EACH; k += 4) {
      const int4 a = make_int4(before, before + v[k], before + v[k] + v[k + 1],
                               before + v[k] + v[k + 1] + v[k + 2]);
      before = a.w + v[k + 3];
      if (whole) {
        *reinterpret_cast<int4 *>(group + k0 + k) = a;
      } else {
        if (k0 + k < n) group[k0 + k] = a.x;
        if (k0 + k + 1 < n) group[k0 + k + 1] = a.y;
        if (k0 + k + 2 < n) group[k0 + k + 2] = a.z;
        if (k0 + k + 3 < n) group[k0 + k + 3] = a.w;
      }
    }
    __syncthreads();  // (s_w is written anew)
  }
}

// Four lanes per node, 64 nodes (two groups) per block.
__global__ void __launch_bounds__(256) k_level_children(TreeDev T, TreeOut O, int level, int64_t n,
                                                        const int32_t *split, const int32_t *group,
                                                        bool scanned) {
  grid_begin();
  __shared__ int s_w[8], s_base;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, q = threadIdx.x & 3;
  before_group(group, 2 * (int64_t)blockIdx.x, scanned, &s_base);
  const int64_t t = (int64_t)blockIdx.x * 64 + (threadIdx.x >> 2);
  const int64_t node = T.level_off[level] + t;
  const bool f = t < n && split[t];
  const unsigned m = __ballot_sync(0xffffffffu, f && q == 0);
  if (lane == 0) s_w[w] = __popc(m);
  int b = 0, e = 0, end = 0;
  if (f) {
    b = T.sbeg[node];
    e = T.send[node];
    const int sh = 2 * (MM_DMAX - level - 1);
    end = q == 3 ? e
                 : (int)lower_bound_u64(T.keys, b, e, ((T.code[node] << 2) + (uint64_t)q + 1) << sh);
  }
  const int up = __shfl_up_sync(0xffffffffu, end, 1);
  __syncthreads();
  if (!f) {
    if (q == 0 && t < n) O.first_child[node] = -1;
    return;
  }
  int rank = s_base + __popc(m & ((1u << (lane & ~3)) - 1u));
  for (int k = 0; k < w; k++) rank += s_w[k];
  const int64_t base = T.level_off[level + 1] + 4 * (int64_t)rank;
  if (q == 0) O.first_child[node] = (int32_t)base;
  write_child(T, O, level, node, q, base + q, q ? up : b, end);
}

// First index in [lo, hi) with a[idx] >= key, by a whole warp: 32 probes a
// step.
__device__ __forceinline__ int64_t warp_lower_bound(const uint64_t *a, int64_t lo, int64_t hi,
                                                    uint64_t key, int lane) {
  while (hi - lo > 32) {
    const int64_t step = (hi - lo + 32) / 33;
    const int64_t p = lo + (lane + 1) * step;
    const int c = __popc(__ballot_sync(0xffffffffu, p < hi && a[p] < key));
    // a[lo + c step] < key <= a[lo + (c + 1) step]
    const int64_t end = lo + (c + 1) * step;
    if (c) lo += c * step + 1;
    if (end < hi) hi = end;
  }
  return lo + __popc(__ballot_sync(0xffffffffu, lo + lane < hi && a[lo + lane] < key));
}

// The levels of at most MM_TOP_NODES nodes, one block.
__global__ void __launch_bounds__(1024) k_tree_top(TreeDev T, TreeOut O, int limit,
                                                   int32_t *info) {
  grid_begin();
  static_assert(MM_TOP_NODES <= 1024, "one thread per node");
  __shared__ int s_flag[MM_TOP_NODES], s_w[32], s_end[3 * MM_TOP_NODES];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  if (tid == 0) {
    O.code[0] = 0;
    O.lvl[0] = 0;
    O.sbeg[0] = 0;
    O.send[0] = (int32_t)T.n_stars;
    O.parent[0] = -1;
    O.level_off[0] = 0;
    O.level_off[1] = 1;
  }
  if (tid < MM_TOP_INFO) info[tid] = 0;
  __syncthreads();
  int n = 1, level = 0, done = 0;
  int64_t off = 0;
  while (n <= MM_TOP_NODES) {
    if (tid == 0) info[2 + level] = n;
    for (int b = 0; b < 8 * n; b += 1024) {
      const int t = (b + tid) >> 3;
      const bool f = node_split(T, O, level, off + t, t < n, tid & 7, limit);
      if ((tid & 7) == 0 && t < n) s_flag[t] = f;
    }
    __syncthreads();
    // rank of each split node, and the split nodes in all
    const int f = tid < n && s_flag[tid];
    const unsigned m = __ballot_sync(0xffffffffu, f);
    if (lane == 0) s_w[w] = __popc(m);
    // the ends of the first three children of the split nodes: a warp per
    // search while there are few and long ones, else a thread per search
    const int sh = 2 * (MM_DMAX - level - 1);
    const bool by_warp = n <= 32;
    for (int k = by_warp ? w : tid; k < 3 * n; k += by_warp ? 32 : 1024) {
      const int t = k / 3;
      if (!s_flag[t]) continue;
      const int64_t b = T.sbeg[off + t], e = T.send[off + t];
      const uint64_t key = ((T.code[off + t] << 2) + (uint64_t)(k - 3 * t) + 1) << sh;
      const int64_t r = by_warp ? warp_lower_bound(T.keys, b, e, key, lane)
                                : lower_bound_u64(T.keys, b, e, key);
      if (!by_warp || lane == 0) s_end[k] = (int)r;
    }
    __syncthreads();
    int before = 0, total = 0;
    for (int k = 0; k < 32; k++) {
      if (k < w) before += s_w[k];
      total += s_w[k];
    }
    if (tid < n) {
      const int64_t node = off + tid;
      const int64_t base = off + n + 4 * (int64_t)(before + __popc(m & ((1u << lane) - 1u)));
      O.first_child[node] = f ? (int32_t)base : -1;
      if (f) {
        int b = T.sbeg[node];
        for (int q = 0; q < 4; q++) {
          const int e = q == 3 ? T.send[node] : s_end[3 * tid + q];
          write_child(T, O, level, node, q, base + q, b, e);
          b = e;
        }
      }
    }
    off += n;
    if (tid == 0 && level + 2 <= MM_DMAX + 1) O.level_off[level + 2] = off + 4 * (int64_t)total;
    n = 4 * total;
    level++;
    done = total == 0;
    __syncthreads();
    if (done) break;
  }
  if (tid == 0) {
    info[0] = level;
    info[1] = done;
    if (level <= MM_DMAX + 1) info[2 + level] = n;
  }
}

// Finest-level cells of the vertex columns (first n0 threads) and rows.
__global__ void k_axis_cells(double x0, double y0, double hx, double hy, int64_t n0, int64_t n1,
                             double R0, int32_t *col, int32_t *row) {
  grid_begin();
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n0)
    col[t] = cell_of(__dadd_rn(x0, __dmul_rn((double)t, hx)), R0);
  else if (t < n0 + n1)
    row[t - n0] = cell_of(__dadd_rn(y0, __dmul_rn((double)(t - n0), hy)), R0);
}

__global__ void k_active_flags(TreeDev T, int64_t n_nodes, const int32_t *col_cell,
                               int64_t col_lo, int64_t col_hi, const int32_t *row_cell,
                               int64_t row_lo, int64_t row_hi, int32_t *node_act,
                               int32_t *leaf_flag, int32_t *group) {
  grid_begin();
  int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool valid = t < n_nodes;
  if (!valid) t = n_nodes - 1;
  const int CX0 = col_cell[col_lo], CX1 = col_cell[col_hi];
  const int CY0 = row_cell[row_lo], CY1 = row_cell[row_hi];
  uint32_t cx, cy;
  morton_decode(T.code[t], cx, cy);
  const int sh = MM_DMAX - T.lvl[t];
  const int64_t x0 = (int64_t)cx << sh, x1 = (((int64_t)cx + 1) << sh) - 1;
  const int64_t y0 = (int64_t)cy << sh, y1 = (((int64_t)cy + 1) << sh) - 1;
  const int act = (x1 >= CX0 && x0 <= CX1 && y1 >= CY0 && y0 <= CY1) ? 1 : 0;
  const int leaf = valid && act && T.first_child[t] < 0;
  if (valid) {
    node_act[t] = act;
    leaf_flag[t] = leaf;
  }
  const int n = __syncthreads_count(leaf);
  if (threadIdx.x == 0) group[blockIdx.x] = n;
}

// Numbers the active leaves in the order of their nodes, block by block of
// k_active_flags; the last block stores how many there are.
__global__ void __launch_bounds__(256) k_compact_leaves(int64_t n_nodes, const int32_t *leaf_flag,
                                                        const int32_t *group, bool scanned,
                                                        int32_t *node_active,
                                                        int32_t *active_list, int32_t *total) {
  grid_begin();
  __shared__ int s_w[8], s_base;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  before_group(group, blockIdx.x, scanned, &s_base);
  const int64_t t = (int64_t)blockIdx.x * 256 + threadIdx.x;
  const bool f = t < n_nodes && leaf_flag[t];
  const unsigned m = __ballot_sync(0xffffffffu, f);
  if (lane == 0) s_w[w] = __popc(m);
  __syncthreads();
  int rank = s_base + __popc(m & ((1u << lane) - 1u)), all = s_base;
  for (int k = 0; k < 8; k++) {
    if (k < w) rank += s_w[k];
    all += s_w[k];
  }
  if (t < n_nodes) node_active[t] = f ? rank : -1;
  if (f) active_list[rank] = (int32_t)t;
  if (threadIdx.x == 0 && blockIdx.x == gridDim.x - 1) *total = all;
}

// Lookup grid over the active region at level glevel: the active leaf
// covering each cell, or -(node + 1) for a split node at glevel.
// Grid cell (gx, gy) of level glevel: the sub-cell record of the active leaf
// containing it when the leaf is at least `sub` levels coarser (the cell then
// lies in one sub-cell), else -(node + 1) for the node where the device walk
// continues.
__global__ void k_lookup_grid(TreeDev T, const int32_t *node_active, int glevel, int sub,
                              int gx0, int gy0, int gw, int gh, int32_t *grid) {
  grid_begin();
  int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (int64_t)gw * gh) return;
  const int gx = gx0 + (int)(t % gw), gy = gy0 + (int)(t / gw);
  int node = 0, l = 0;
  for (; l < glevel; l++) {
    int fc = T.first_child[node];
    if (fc < 0) break;
    int sh = glevel - l - 1;
    node = fc + (((gx >> sh) & 1) | (((gy >> sh) & 1) << 1));
  }
  const int a = (T.first_child[node] < 0) ? node_active[node] : -1;
  if (a >= 0 && l + sub <= glevel) {
    const int sh = glevel - l - sub, mask = (1 << sub) - 1;
    grid[t] = (a << (2 * sub)) + (((gy >> sh) & mask) << sub) + ((gx >> sh) & mask);
  } else {
    grid[t] = -(node + 1);
  }
}

static inline unsigned blocks_for(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }

cudaError_t launch_star_keys(const double *pos, int64_t n, double R0, uint64_t *keys,
                             int32_t *idx, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  launch_next(k_star_keys, blocks_for(n, 256), 256, 0, st, pos, n, R0, keys, idx);
  return cudaGetLastError();
}

cudaError_t launch_gather_stars(const double *pos, const double *m, const int32_t *idx,
                                int64_t n, double *sx, double *sy, double *sm,
                                cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  launch_next(k_gather_stars, blocks_for(n, 256), 256, 0, st, pos, m, idx, n, sx, sy, sm);
  return cudaGetLastError();
}

cudaError_t launch_tree_top(const TreeDev &T, const TreeOut &O, int limit, int32_t *info,
                            cudaStream_t st) {
  launch_next(k_tree_top, 1, 1024, 0, st, T, O, limit, info);
  return cudaGetLastError();
}

cudaError_t launch_level_split(const TreeDev &T, const TreeOut &O, int level, int64_t n, int limit,
                               int32_t *split, int32_t *group, int32_t *total, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  launch_next(k_level_split, blocks_for(n, MM_SPLIT_GROUP), 256, 0, st, T, O, level, n, limit, split, group,
                                                               total);
  return cudaGetLastError();
}

cudaError_t launch_group_scan(int32_t *group, int64_t n, cudaStream_t st) {
  launch_next(k_group_scan, 1, 1024, 0, st, group, n);
  return cudaGetLastError();
}

cudaError_t launch_level_children(const TreeDev &T, const TreeOut &O, int level, int64_t n,
                                  const int32_t *split, const int32_t *group, bool scanned,
                                  cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  launch_next(k_level_children, blocks_for(n, 64), 256, 0, st, T, O, level, n, split, group, scanned);
  return cudaGetLastError();
}

cudaError_t launch_axis_cells(double x0, double y0, double hx, double hy, int64_t n0, int64_t n1,
                              double R0, int32_t *col, int32_t *row, cudaStream_t st) {
  if (n0 + n1 <= 0) return cudaSuccess;
  launch_next(k_axis_cells, blocks_for(n0 + n1, 256), 256, 0, st, x0, y0, hx, hy, n0, n1, R0, col, row);
  return cudaGetLastError();
}

cudaError_t launch_active_flags(const TreeDev &T, int64_t n_nodes, const int32_t *col_cell,
                                int64_t col_lo, int64_t col_hi, const int32_t *row_cell,
                                int64_t row_lo, int64_t row_hi, int32_t *node_act,
                                int32_t *leaf_flag, int32_t *group, cudaStream_t st) {
  if (n_nodes <= 0) return cudaSuccess;
  launch_next(k_active_flags, blocks_for(n_nodes, MM_ACTIVE_GROUP), MM_ACTIVE_GROUP, 0, st,
      T, n_nodes, col_cell, col_lo, col_hi, row_cell, row_lo, row_hi, node_act, leaf_flag, group);
  return cudaGetLastError();
}

cudaError_t launch_compact_leaves(int64_t n_nodes, const int32_t *leaf_flag, const int32_t *group,
                                  bool scanned, int32_t *node_active, int32_t *active_list,
                                  int32_t *total, cudaStream_t st) {
  static_assert(MM_ACTIVE_GROUP == 256, "one thread per node of a group");
  if (n_nodes <= 0) return cudaSuccess;
  launch_next(k_compact_leaves, blocks_for(n_nodes, 256), 256, 0, st, n_nodes, leaf_flag, group, scanned,
              node_active, active_list, total);
  return cudaGetLastError();
}

cudaError_t launch_lookup_grid(const TreeDev &T, const int32_t *node_active, int glevel,
                               int sub, int gx0, int gy0, int gw, int gh, int32_t *grid,
                               cudaStream_t st) {
  int64_t n = (int64_t)gw * gh;
  if (n <= 0) return cudaSuccess;
  launch_next(k_lookup_grid, blocks_for(n, 256), 256, 0, st, T, node_active, glevel, sub, gx0, gy0, gw,
                                                    gh, grid);
  return cudaGetLastError();
}

}  // namespace mm
