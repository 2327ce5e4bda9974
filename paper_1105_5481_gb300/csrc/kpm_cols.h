// Column-strip solve (kpm_cols.cu): the vector columns of one or many stencil
// instances as independent tasks of one persistent launch, each column's
// recursion run from its first to its last product by one CTA (or one
// cluster), v_n in shared memory and v_{n-1} in registers.
#pragma once

#include "kpm_internal.h"

namespace kpm {

// Threads of a CTA, the largest strip heights with a compiled body, and the
// shared memory for the dots of two batches of products.
constexpr int COLS_THREADS = 512;
constexpr int COLS_MAX_H_F32 = 32, COLS_MAX_H_F64 = 16;
constexpr size_t COLS_RING_BYTES = 16 * 1024;
constexpr size_t COLS_MAX_SMEM = 231168;  // of 232,448, less the kernel's static variables

// How one CTA (of a cluster of C) lays out a column of an instance: its band
// of at most `rows` rows of the last dimension, each row a plane of `plane`
// sites, is cut into `strips` strips of at most `height` rows; a thread owns
// one plane position of one strip.
struct ColsShape {
  int C = 0;
  int plane = 0, rows = 0;
  int strips = 0, height = 0;
  int pitch = 0;      // thread positions of a lattice line
  int spi = 0, lines = 0;  // FP32 dots: rows per pass and (line traversal) lines of the
                           // global-memory batch form, its CTAs that have rows,
                           // bytes of the sweep's table
  int ranks = 0;
  size_t table = 0;
  int tpc = 0;        // threads per column (a multiple of 32)
  int max_cols = 0;   // columns a CTA can hold
  double us_fixed = 0.0, us_col = 0.0;  // estimated microseconds per product
};

struct ColsTask {
  StencilGeom geom;
  int64_t n;
  const ScalarBlock* sc;
  const void* ds;             // scaled diagonal [N], or NULL (uniform)
  double* sums;               // [steps][2][Rp] per-step sums over rows of this realisation
  double* part;               // C > 1: [C][M / 2][2 ncol] scratch
  const RunParams* prm;       // not NULL: seed and first realisation are read from here
  unsigned long long seed;
  long long s;                // realisation (added to prm->s0 when prm is given)
  int Rp, R, M;
  int col0, ncol;
  int strips, height, tpc, rows, pitch, spi, lines;  // ColsShape
  int batch;                  // products per batch of the dot sums
  int fixq;                   // FP64, > 0: 64-bit fixed point of unit 2^-fixq (kpm_fixed.cuh;
                              // ds in its format)
  // finalisation in the kernel (batches): the instance's per-vector moments
  // and mean, written by the last of its `ntiles` tasks; per_vec NULL: none
  double* per_vec;
  double* mu;
  int* flags;                 // bit 0: a moment left [-1, 1]
  int* tiles_done;
  int ntiles;
};

// The layout of an instance with R columns at cluster size C (false: it does
// not fit; FP32 takes C = 1).  Depends on the instance, the element type and C
// alone.
bool cols_shape(const StencilGeom& g, int64_t n, int R, bool fp32, int C, ColsShape* out);
// The layout of a task of ncol columns (the other members are left alone).
void cols_set_layout(ColsTask& t, const ColsShape& s, bool fp32, int col0, int ncol);
size_t cols_smem(const ColsShape& s, bool fp32, int ncol);
// Clusters of C CTAs that are resident at once (0: cannot be launched).
int cols_max_clusters(bool fp32, int dims, bool ds, int C, size_t smem);
cudaError_t launch_cols(bool fp32, int dims, bool ds, const ColsTask* tasks, int ntasks, int* queue,
                        int clusters, int C, size_t smem, cudaStream_t st);

}  // namespace kpm
