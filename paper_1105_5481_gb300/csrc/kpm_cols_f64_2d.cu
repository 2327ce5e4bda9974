// Column-strip solve: FP64 vectors, 2D stencils.
#include "kpm_cols.cuh"

namespace kpm {

cudaError_t launch_cols_f64_2d(bool ds, const ColsTask* tasks, int ntasks, int* queue, int clusters,
                                int C, size_t smem, cudaStream_t st) {
  return ds ? cols::launch<double, 2, true>(tasks, ntasks, queue, clusters, C, smem, st)
            : cols::launch<double, 2, false>(tasks, ntasks, queue, clusters, C, smem, st);
}

int cols_clusters_f64_2d(bool ds, int C, size_t smem) {
  return ds ? cols::max_clusters<double, 2, true>(C, smem)
            : cols::max_clusters<double, 2, false>(C, smem);
}

}  // namespace kpm
