// Column-strip solve: the layout of an instance and the dispatch over element
// type and dimensions (the kernels are compiled in kpm_cols_*.cu).
#include "kpm_cols.h"

#include <algorithm>

namespace kpm {

cudaError_t launch_cols_f32_2d(bool, const ColsTask*, int, int*, int, int, size_t, cudaStream_t);
cudaError_t launch_cols_f32_3d(bool, const ColsTask*, int, int*, int, int, size_t, cudaStream_t);
cudaError_t launch_cols_f64_2d(bool, const ColsTask*, int, int*, int, int, size_t, cudaStream_t);
cudaError_t launch_cols_f64_3d(bool, const ColsTask*, int, int*, int, int, size_t, cudaStream_t);
int cols_clusters_f32_2d(bool, int, size_t);
int cols_clusters_f32_3d(bool, int, size_t);
int cols_clusters_f64_2d(bool, int, size_t);
int cols_clusters_f64_3d(bool, int, size_t);

// FP32 (run_slots): three vector buffers of thread slots, the dots of two
// batches of kb products and the dot sweep's table; FP64 (run_rows): two
// buffers, the diagonal and the dots.
static size_t cols_bytes(const ColsShape& s, bool fp32, int ncol, int kb) {
  if (fp32)
    return (size_t)3 * ((s.height * (COLS_THREADS + 1) + 3) / 4 * 4) * 4 +
           (size_t)2 * kb * ncol * s.ranks * 16 * 8 + s.table;
  return ((2 * (size_t)ncol + 1) * s.rows * s.plane * 8 + 15) / 16 * 16 +
         (size_t)2 * kb * (COLS_THREADS / 32) * 2 * 16;  // 16 bytes: fixed point's two words
}

// Products per batch of the dot sums: up to 16, within COLS_RING_BYTES and
// the CTA's shared memory.
static int cols_batch(const ColsShape& s, bool fp32, int ncol) {
  const size_t one = fp32 ? (size_t)ncol * s.ranks * 16 * 8 : (size_t)COLS_THREADS / 32 * 32;
  int kb = 16;
  while (kb > 1 && (2 * kb * one > COLS_RING_BYTES || cols_bytes(s, fp32, ncol, kb) > COLS_MAX_SMEM))
    kb /= 2;
  return kb;
}

size_t cols_smem(const ColsShape& s, bool fp32, int ncol) {
  return cols_bytes(s, fp32, ncol, cols_batch(s, fp32, ncol));
}

void cols_set_layout(ColsTask& t, const ColsShape& s, bool fp32, int col0, int ncol) {
  t.col0 = col0;
  t.ncol = ncol;
  t.strips = s.strips;
  t.height = s.height;
  t.tpc = s.tpc;
  t.rows = s.rows;
  t.pitch = s.pitch;
  t.spi = s.spi;
  t.lines = s.lines;
  t.batch = cols_batch(s, fp32, ncol);
}

// Estimated clocks of one warp per product: FP32 about 10 (2D) or 14 (3D)
// issue slots per site for the recursion and 13 for the dots, and 100 for
// their reduction; FP64 64 clocks of a scheduler's share of the FP64 pipe per
// instruction, 2 dots, the recursion's FMA and one per bond, and 5 adds of the
// reduction.
static bool shape_at(const StencilGeom& g, int64_t n, int R, bool fp32, int C, bool pad,
                     ColsShape* out) {
  if (g.dims != 2 && g.dims != 3) return false;
  const int L = g.L[g.dims - 1];
  if (L < C || n < 1 || n > (1 << 20) || (fp32 && C > 1)) return false;
  ColsShape proto;
  proto.C = C;
  proto.rows = (L + C - 1) / C;
  proto.pitch = g.L[0];
  if (fp32) {
    // the global-memory form's rows per pass (threads over chunks per row)
    // and traversal (as plan_instance)
    int Rp, G;
    padded_width(R, true, false, &Rp, &G);
    if (G > 32) return false;
    proto.spi = 256 / G;
    const int64_t lines = n / g.L[0], padded = (lines + proto.spi - 1) / proto.spi * proto.spi;
    int64_t passes = (n + proto.spi - 1) / proto.spi;
    if (g.L[0] >= 4 && lines >= proto.spi && 8 * (padded - lines) <= lines) {
      proto.lines = (int)lines;
      passes = padded / proto.spi * g.L[0];
      // adjacent lines on different banks, where the padding leaves the fit
      if (g.dims == 3 && pad) proto.pitch = g.L[0] | 1;
    }
    proto.ranks = (int)std::min<int64_t>(4, (passes + 3) / 4);
    proto.table = proto.lines ? (size_t)proto.lines * 2
                              : (size_t)((passes + 15) / 16) * proto.ranks * proto.spi * 8;
  }
  proto.plane = g.dims == 2 ? proto.pitch : proto.pitch * g.L[1];
  const int U = proto.plane;
  if (U > COLS_THREADS) return false;
  ColsShape best{};
  double best_cost = 1e300;
  const int rows = proto.rows, hmax = fp32 ? COLS_MAX_H_F32 : COLS_MAX_H_F64;
  for (int S = (rows + hmax - 1) / hmax; S <= rows && U * S <= COLS_THREADS; ++S) {
    ColsShape s = proto;
    s.strips = S;
    s.height = (rows + S - 1) / S;
    s.tpc = (U * S + 31) / 32 * 32;
    s.max_cols = COLS_THREADS / s.tpc;
    while (s.max_cols > 0 && cols_smem(s, fp32, s.max_cols) > COLS_MAX_SMEM) --s.max_cols;
    if (s.max_cols < 1) continue;
    const double warp = fp32 ? (g.dims == 2 ? 23.0 : 27.0) * s.height + 100.0
                             : 64.0 * ((2 * g.dims + 3) * s.height + 5);
    s.us_fixed = C > 1 ? 0.6 : 0.2;
    s.us_col = s.tpc / 32 * 0.25 * warp / 1900.0;
    const double cost = s.us_fixed / s.max_cols + s.us_col;
    if (cost < best_cost) {
      best_cost = cost;
      best = s;
    }
  }
  if (best.strips == 0) return false;
  *out = best;
  return true;
}

bool cols_shape(const StencilGeom& g, int64_t n, int R, bool fp32, int C, ColsShape* out) {
  *out = ColsShape{};
  return shape_at(g, n, R, fp32, C, true, out) || shape_at(g, n, R, fp32, C, false, out);
}

int cols_max_clusters(bool fp32, int dims, bool ds, int C, size_t smem) {
  if (smem > COLS_MAX_SMEM) return 0;
  if (fp32) return dims == 2 ? cols_clusters_f32_2d(ds, C, smem) : cols_clusters_f32_3d(ds, C, smem);
  return dims == 2 ? cols_clusters_f64_2d(ds, C, smem) : cols_clusters_f64_3d(ds, C, smem);
}

cudaError_t launch_cols(bool fp32, int dims, bool ds, const ColsTask* tasks, int ntasks, int* queue,
                        int clusters, int C, size_t smem, cudaStream_t st) {
  if (smem > COLS_MAX_SMEM || clusters < 1) return cudaErrorInvalidConfiguration;
  if (fp32)
    return dims == 2 ? launch_cols_f32_2d(ds, tasks, ntasks, queue, clusters, C, smem, st)
                     : launch_cols_f32_3d(ds, tasks, ntasks, queue, clusters, C, smem, st);
  return dims == 2 ? launch_cols_f64_2d(ds, tasks, ntasks, queue, clusters, C, smem, st)
                   : launch_cols_f64_3d(ds, tasks, ntasks, queue, clusters, C, smem, st);
}

}  // namespace kpm
