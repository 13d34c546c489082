// Leaf records (k_near_count, k_leaf_finalize) of one leaf, for
// test_gpu_leaf_records.py: a root without children, the n given stars its
// near field, far field zero, the map far to one side.
#include <cstring>
#include <vector>

#include "mm_kernels.h"

using namespace mm;

thread_local int LaunchApart::depth = 0;

namespace {
template <class T>
T *dev(std::vector<void *> &all, size_t n, const T *src = nullptr) {
  void *p = nullptr;
  if (cudaMalloc(&p, n * sizeof(T)) != cudaSuccess) return nullptr;
  all.push_back(p);
  if (src)
    cudaMemcpy(p, src, n * sizeof(T), cudaMemcpyHostToDevice);
  else
    cudaMemset(p, 0, n * sizeof(T));
  return static_cast<T *>(p);
}
}  // namespace

// Room for `cap` direct stars (< 0: as many as k_near_count finds, less -1 - cap),
// of `slots` allocated and filled with 0xff.  Returns a CUDA error.  recs: 4^sub records.
extern "C" int leaf_records(const double *x, const double *y, const double *m, int64_t n, int sub,
                            int64_t cap, double lox, LeafRec *recs, unsigned *total,
                            unsigned *written, unsigned *err_word) {
  std::vector<void *> all;
  const int64_t off[2] = {0, 1};
  const int32_t zero = 0, none = -1, n32 = (int32_t)n, nb[9] = {-1, -1, -1, -1, 0, -1, -1, -1, -1};
  const uint64_t code = 0;
  TreeDev T;
  memset(&T, 0, sizeof T);
  T.n_stars = n;
  T.R0 = 8.0;
  T.sx = dev(all, n, x);
  T.sy = dev(all, n, y);
  T.sm = dev(all, n, m);
  T.code = dev(all, 1, &code);
  T.lvl = dev(all, 1, &zero);
  T.sbeg = dev(all, 1, &zero);
  T.send = dev(all, 1, &n32);
  T.first_child = dev(all, 1, &none);
  T.parent = dev(all, 1, &none);
  T.nb = dev(all, 9, nb);
  T.level_off = dev(all, 2, off);
  FmmConst C;
  memset(&C, 0, sizeof C);
  C.p = C.p_eval = 4;
  C.sub = sub;
  C.npix = C.npix_y = 16;
  C.cull = 1;
  C.kappa = 0.4;
  C.gamma = 0.3;
  C.kappa_star = 0.4;
  C.x0 = C.y0 = -8.0;
  C.hx = C.hy = 0.5;
  C.inv_hx = C.inv_hy = 2.0;
  C.x1 = C.y1 = 8.0;
  C.lox = lox;
  C.loy = -8.0;
  C.delta = C.inv_delta = 1.0;
  const int NS = 1 << (2 * sub), P1 = C.p + 1;
  const int32_t *active = dev(all, 1, &zero);
  unsigned *err = dev<unsigned>(all, 2);
  cudaError_t e = launch_near_count(T, C, 1, active, err + 1, err, 0);
  if (e == cudaSuccess) e = cudaMemcpy(total, err + 1, sizeof *total, cudaMemcpyDeviceToHost);
  cudaMemset(err, 0, 2 * sizeof(unsigned));
  const size_t slots = (size_t)*total + 1;
  const unsigned room = cap < 0 ? *total + 1 + (int)cap : (unsigned)cap;
  SubTables tb;
  double2 *up = dev<double2>(all, (size_t)P1 * NS);
  float2 *fp = dev<float2>(all, (size_t)P1 * NS);
  float *bin = dev<float>(all, (size_t)P1 * P1);
  tb.up = up;
  tb.fp = fp;
  tb.bin = bin;
  const double2 *loc = dev<double2>(all, P1);
  LeafRec *leaf = dev<LeafRec>(all, NS);
  NearPos *np = dev<NearPos>(all, slots);
  float *nm = dev<float>(all, slots);
  float2 *coef = dev<float2>(all, (size_t)NS * coef_stride(C.p_eval));
  if (!np || !nm || !coef || !leaf) e = cudaErrorMemoryAllocation;
  if (e == cudaSuccess) {
    cudaMemset(nm, 0xff, slots * sizeof(float));
    e = launch_sub_tables(sub, C.p, up, fp, bin, 0);
    if (e == cudaSuccess)
      e = launch_leaf_finalize(T, C, 1, active, tb, loc, leaf, np, nm, coef, err + 1, room, err, 0);
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    cudaMemcpy(recs, leaf, NS * sizeof(LeafRec), cudaMemcpyDeviceToHost);
    cudaMemcpy(err_word, err, sizeof *err_word, cudaMemcpyDeviceToHost);
    // slots with a mass in them, and whether one lies beyond the room
    std::vector<float> h(slots);
    cudaMemcpy(h.data(), nm, slots * sizeof(float), cudaMemcpyDeviceToHost);
    written[0] = written[1] = 0;
    for (size_t k = 0; k < slots; k++)
      if (h[k] == h[k]) written[k < room ? 0 : 1]++;
  }
  for (void *p : all) cudaFree(p);
  return (int)e;
}
