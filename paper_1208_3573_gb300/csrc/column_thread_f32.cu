// Four lanes per column: the mixed-precision DIAF-S kernel for small real tiles.
#include "column_thread.cuh"
#include "launch.cuh"

namespace {

// f(kernel, index) with the instance for tiles of at most K columns
template <class F>
cudaError_t with_instance(int K, F f) {
  switch (thread_instance(K)) {
    case 8: return f(column_thread_kernel<8>, 0);
    case 13: return f(column_thread_kernel<13>, 1);
    default: return f(column_thread_kernel<16>, 2);
  }
}

size_t g_thread_smem_configured[3] = {0, 0, 0};

}  // namespace

cudaError_t thread_columns_shape(int M, int K, int count_hint, ThreadShape* out) {
  *out = ThreadShape{};
  if (count_hint <= 0) return cudaSuccess;
  if (M < 1 || K < 1 || M > kThreadMMax || K > kThreadKMax) return cudaErrorInvalidValue;
  const size_t smem = thread_warp_smem(M, K, thread_instance(K)) * kQuadWarps;
  int dev = 0, sms = 0, per_sm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  e = with_instance(K, [&](auto kern, int i) {
    if (g_thread_smem_configured[i] < smem) {
      const cudaError_t r = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (r != cudaSuccess) return r;
      g_thread_smem_configured[i] = smem;
    }
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32 * kQuadWarps, smem);
  });
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidValue;
  int grid = sms * per_sm;
  const int need = ceil_div(count_hint, kQuadCols * kQuadWarps);
  if (grid > need) grid = need;
  out->grid = grid;
  out->block = 32 * kQuadWarps;
  out->smem = smem;
  out->nquads = grid * kQuadWarps * kQuadCols;
  return cudaSuccess;
}

cudaError_t launch_columns_thread_f32(const ColArgs& a, const ThreadArgs& ta, const ThreadShape& sh, cudaStream_t s) {
  if (sh.grid <= 0) return cudaSuccess;
  return with_instance(ta.K, [&](auto kern, int) {
    kern<<<sh.grid, sh.block, sh.smem, s>>>(a, ta);
    DIAF_COUNT_LAUNCH();
    return cudaGetLastError();
  });
}
