// Host-side launchers of the libmm kernels (one declaration per kernel
// family; definitions live next to the kernels).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include <vector>

#include "mm_common.cuh"

namespace mm {

// Message returned by mm_last_error on this thread (api.cu).
void set_last_error(const char *msg);

// While one lives, launch_next on its thread launches like any other launch.
// For a batch: its streams fill the GPU between them, and blocks that wait
// there take places from those that could run (12 maps: 33.1 ms, 32.2 with
// this).  For a handle's creation: its short chains end in host reads, and
// the attribute costs more than it hides (0.05 ms).
struct LaunchApart {
  static thread_local int depth;
  LaunchApart() { depth++; }
  ~LaunchApart() { depth--; }
};

// Launch a kernel that calls grid_begin: its blocks are set up while the
// kernel before it in the stream still runs, which takes the launch latency
// off the chains of small kernels of a run's tree and expansions (48^2 map
// 0.260 -> 0.235 ms, 601 x 1003 map 4.04 -> 4.01 ms).  The mapping kernels are
// long and launched like any other: with it a batch's took 0.4 % more.
template <class... P, class... A>
inline cudaError_t launch_next(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem,
                               cudaStream_t st, const A &...args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = LaunchApart::depth > 0 ? 0 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// ---- tree (tree.cu) --------------------------------------------------------
struct TreeDev {
  // sorted stars (Morton order), SoA, FP64
  const uint64_t *keys;
  const double *sx, *sy, *sm;
  int64_t n_stars;
  double R0;                  // root half-length (power of two)
  // nodes (flattened over levels)
  const uint64_t *code;
  const int32_t *lvl, *sbeg, *send, *first_child;
  const int32_t *parent;      // -1 for the root
  const int32_t *nb;          // per node: the nine same-level cells around it (row-major,
                              // itself in the middle), -1 where the cell is no node
  const int64_t *level_off;   // [MM_DMAX + 2]
};

cudaError_t launch_star_keys(const double *pos, int64_t n, double R0, uint64_t *keys,
                             int32_t *idx, cudaStream_t st);
cudaError_t launch_gather_stars(const double *pos, const double *m, const int32_t *idx,
                                int64_t n, double *sx, double *sy, double *sm,
                                cudaStream_t st);
// The node arrays a level's kernels write (sizes: see TreeDev).
struct TreeOut {
  uint64_t *code;
  int32_t *lvl, *sbeg, *send, *first_child, *parent, *nb;
  int64_t *level_off;
};
// Levels from the root down to the first with more than MM_TOP_NODES nodes,
// in one launch.  info[0]: the level it stopped at (not yet split); info[1]:
// 1 when the tree is complete; info[2 + l]: nodes of level l.
#define MM_TOP_NODES 256
#define MM_TOP_CAPACITY ((MM_DMAX + 1) * MM_TOP_NODES + 4 * MM_TOP_NODES)
#define MM_TOP_INFO (2 + MM_DMAX + 2)
cudaError_t launch_tree_top(const TreeDev &T, const TreeOut &O, int limit, int32_t *info,
                            cudaStream_t st);
// One larger level: neighbours and split flags of its n nodes, the number of
// split nodes per group of MM_SPLIT_GROUP, and (total not NULL) in all.
#define MM_SPLIT_GROUP 32
cudaError_t launch_level_split(const TreeDev &T, const TreeOut &O, int level, int64_t n, int limit,
                               int32_t *split, int32_t *group, int32_t *total, cudaStream_t st);
// Counts per group become running sums, in place.  Above MM_SUM_GROUPS groups:
// up to there a level's blocks add the counts up themselves, which spares a
// launch (a level of 160 000 nodes 3 us) but is quadratic (tree of 3e6 stars
// 0.98 ms, 0.87 with the sums; of 1e8 298 and 25; 2048, 8192 and no limit the
// same at 1e6).
#define MM_SUM_GROUPS 8192
cudaError_t launch_group_scan(int32_t *group, int64_t n, cudaStream_t st);
// Its children, in Morton order.  scanned: group holds the running sums.
cudaError_t launch_level_children(const TreeDev &T, const TreeOut &O, int level, int64_t n,
                                  const int32_t *split, const int32_t *group, bool scanned,
                                  cudaStream_t st);
cudaError_t launch_axis_cells(double x0, double y0, double hx, double hy, int64_t n0, int64_t n1,
                              double R0, int32_t *col, int32_t *row, cudaStream_t st);
// flags[node] = 1 for active leaves (leaf containing ray vertices) and their
// number per group of MM_ACTIVE_GROUP nodes; also node_act[node] = 1 for every
// active node
#define MM_ACTIVE_GROUP 256
cudaError_t launch_active_flags(const TreeDev &T, int64_t n_nodes, const int32_t *col_cell,
                                int64_t col_lo, int64_t col_hi, const int32_t *row_cell,
                                int64_t row_lo, int64_t row_hi, int32_t *node_act,
                                int32_t *leaf_flag, int32_t *group, cudaStream_t st);
cudaError_t launch_compact_leaves(int64_t n_nodes, const int32_t *leaf_flag, const int32_t *group,
                                  bool scanned, int32_t *node_active, int32_t *active_list,
                                  int32_t *total, cudaStream_t st);
cudaError_t launch_lookup_grid(const TreeDev &T, const int32_t *node_active, int glevel,
                               int sub, int gx0, int gy0, int gw, int gh, int32_t *grid,
                               cudaStream_t st);

// ---- expansions (fmm.cu) ---------------------------------------------------
struct FmmConst {
  int p;                      // expansion order of the FMM
  int p_eval;                 // terms kept of each sub-cell's re-centred expansion
  int sub;                    // sub-cell levels s: 4^s sub-cells per leaf
  int npix, npix_y;           // map pixels along x and y (culling bounds)
  int cull;                   // 1: compute the culling bounds
  double kappa, gamma, kappa_star;
  double x0, y0, hx, hy;      // ray grid
  double inv_hx, inv_hy, inv_delta;  // 1 / hx, 1 / hy, 1 / delta
  double x1, y1;              // the grid's last vertex
  double lox, loy, delta;     // map lower-left corner and pixel side
  double rect_c1, rect_c2;    // > 0: rectangular star region |x| <= c1, |y| <= c2 (App. B)
};

cudaError_t launch_p2m(const TreeDev &T, int64_t n_nodes, int p, const double2 *MLop, double2 *mp,
                       cudaStream_t st);
cudaError_t launch_m2m(const TreeDev &T, int level, int64_t n, int p, const double2 *MMop,
                       double2 *mp, int sms, cudaStream_t st);
cudaError_t launch_local(const TreeDev &T, int level, int64_t n, int p, const int32_t *node_act,
                         const double2 *MLop, const double2 *LLop, const double2 *mp,
                         double2 *loc, unsigned *err, int sms, cudaStream_t st);
// *total += direct-sum stars of all records (the plan sizes their arrays)
cudaError_t launch_near_count(const TreeDev &T, const FmmConst &C, int64_t n_active,
                              const int32_t *active_list, unsigned *total, unsigned *err,
                              cudaStream_t st);
// What every re-centring of a plan shares (k_sub_tables): powers of the
// sub-cells' positions [k][q], k = 0 .. p, and binomials [n][m], n, m <= p.
struct SubTables {
  const double2 *up;
  const float2 *fp;
  const float *bin;
};
cudaError_t launch_sub_tables(int sub, int p, double2 *up, float2 *fp, float *bin,
                              cudaStream_t st);
// near_total: slots reserved so far (0 before the call), of near_cap
cudaError_t launch_leaf_finalize(const TreeDev &T, const FmmConst &C, int64_t n_active,
                                 const int32_t *active_list, const SubTables &tb,
                                 const double2 *loc, LeafRec *leaf, NearPos *near_pos,
                                 float *near_m, float2 *coef, unsigned *near_total,
                                 unsigned near_cap, unsigned *err, cudaStream_t st);
void build_operator_tables(int p, std::vector<double2> &MM, std::vector<double2> &ML,
                           std::vector<double2> &LL);

// ---- shooting + mapping (shoot.cu) -----------------------------------------
// dst[i] = *src[i] with work_begin[i], on the device (n descriptors)
cudaError_t launch_batch_gather(const MapDev *const *src, const int64_t *work_begin, int n,
                                MapDev *dst, int &launches, cudaStream_t st);
// inverse ray shooting of one map's work items (no second pass)
cudaError_t launch_shoot_irs(const MapDev &m, int64_t total_work, bool square,
                             unsigned long long *counter, unsigned *err, cudaStream_t st);
// the second pass over the map's queued larger triangles (no-op without a
// queue); launches += its kernels
cudaError_t launch_big_ipm(const MapDev &m, int &launches, cudaStream_t st);
// h_single: the map by value when n_maps == 1 (else NULL: maps from d_maps)
cudaError_t launch_shoot_ipm(const MapDev *d_maps, const MapDev *h_single, int n_maps,
                             int64_t total_work, bool square,
                             unsigned long long *counter, unsigned *err, int grid,
                             cudaStream_t st);
cudaError_t launch_normalize(const unsigned long long *acc, const unsigned long long *span,
                             int npix, int npix_y, double scale, float *out, cudaStream_t st);
// out[k] = acc[k] * scale for n fixed-point values (the normalisation of an
// accumulator already folded with its row-difference array)
cudaError_t launch_scale_fixed(const unsigned long long *acc, int64_t n, double scale,
                               float *out, cudaStream_t st);
cudaError_t launch_fold_span(unsigned long long *acc, const unsigned long long *span, int npix,
                             int npix_y,
                             unsigned long long *out, cudaStream_t st);
cudaError_t launch_probe(const MapDev *d_maps, bool square, int64_t n, const double *z,
                         double *w, double x0, double y0, double hx, double hy, double R0,
                         double lox, double loy, double delta, unsigned *err, cudaStream_t st);

// ---- plain FP64 path (direct64.cu) -----------------------------------------
struct DirectConst {
  double kappa, gamma, kappa_star;
  double x0, y0, hx, hy;
  double lox, loy, delta;
  double rect_c1, rect_c2;    // > 0: rectangular star region (App. B); 0: disk
};
// vertices of columns [col0, col0 + width) and rows [row_lo, row_hi], row-major
cudaError_t launch_direct64_vertices(const double *sx, const double *sy, const double *sm,
                                     int64_t n_stars, const DirectConst &C, int64_t col0,
                                     int64_t width, int64_t row_lo, int64_t row_hi, Vtx *out,
                                     cudaStream_t st);
cudaError_t launch_direct64_points(const double *sx, const double *sy, const double *sm,
                                   int64_t n_stars, const DirectConst &C, int64_t n,
                                   const double *z, double *w, cudaStream_t st);
cudaError_t launch_ipm_vertices(const MapDev *d_map, const Vtx *verts, int64_t width,
                                int64_t row_lo, int64_t row_hi, unsigned long long *counter,
                                unsigned *err, int grid, cudaStream_t st);

}  // namespace mm
