// Fixed-point instantiations of the fused Chebyshev step (FP64
// vectors) and the conversions to its formats.
#include "kpm_fixed.cuh"
#include "kpm_step_dispatch.cuh"

namespace kpm {

namespace {

// FP64 values in [-2^(61-q), 2^(61-q)] to (x1, x0) of unit 2^-q, in place.
__global__ void to_fixed_kernel(int64_t count, double scale, double* v) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < count;
       e += (int64_t)gridDim.x * blockDim.x) {
    const long long L = __double2ll_rn(v[e] * scale);
    const int lo = (int)L;
    reinterpret_cast<int2*>(v)[e] = make_int2((int)((L - lo) >> 32), lo);
  }
}

__global__ void to_fix_coef_kernel(int64_t count, const double* __restrict__ src, Fix* dst) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < count;
       e += (int64_t)gridDim.x * blockDim.x)
    dst[e] = Fix::of(src[e]);
}

unsigned blocks(int64_t n) { return (unsigned)std::min<int64_t>((n + 255) / 256, 152 * 16); }

}  // namespace

cudaError_t launch_step_i64(bool stencil, bool cplx, StepMode mode, const StepArgs& a, const LaunchCfg& cfg,
                            cudaStream_t st) {
  if (mode == MODE_FIRST)
    return cplx ? run_mode<ChunkI64<true>, MODE_FIRST>(stencil, a, cfg, st)
                : run_mode<ChunkI64<false>, MODE_FIRST>(stencil, a, cfg, st);
  if (mode == MODE_STEP)
    return cplx ? run_mode<ChunkI64<true>, MODE_STEP>(stencil, a, cfg, st)
                : run_mode<ChunkI64<false>, MODE_STEP>(stencil, a, cfg, st);
  return cudaErrorInvalidValue;
}

int occ_step_i64(bool stencil, bool cplx, const StepArgs& a, int block) {
  return cplx ? occ_mode<ChunkI64<true>, MODE_STEP>(stencil, a, block)
              : occ_mode<ChunkI64<false>, MODE_STEP>(stencil, a, block);
}

cudaError_t launch_to_fixed(int64_t count, int q, void* v, cudaStream_t st) {
  to_fixed_kernel<<<blocks(count), 256, 0, st>>>(count, ldexp(1.0, q), (double*)v);
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return cudaGetLastError();
}

cudaError_t launch_to_fix_coef(int64_t count, const void* src, void* dst, cudaStream_t st) {
  to_fix_coef_kernel<<<blocks(count), 256, 0, st>>>(count, (const double*)src, (Fix*)dst);
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return cudaGetLastError();
}

}  // namespace kpm
