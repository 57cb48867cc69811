// One forward-kernel variant per object file.  The build compiles this file once per
// variant with -DQP_T=<float|double> -DQP_KIND=<0 fixed-size, 1 global-memory (fixed-size and
// packed) below the wide line, 2 packed shared-memory, 3 global-memory of wide sizes> (kinds 1 and 3
// share routines, and in one file the wide kernels' needs cost the others 1 to 2%) and, for kinds 0 and 2, -DQP_SW/-DQP_CH (the register-tile
// slots of the sweep and of the Cholesky).
#include "qp_launch.cuh"

#if !defined(QP_T) || !defined(QP_KIND)
#error "qp_fwd_variant.cu needs -DQP_T and -DQP_KIND"
#endif

namespace qpk {

#if QP_KIND == 0
template <typename T, int SW, int CH>
cudaError_t launch_fwd_v(const FwdParams<T>& P, size_t smem, cudaStream_t st) {
  auto k = qp_fwd_kernel<T, SW, CH>;
  cudaError_t e = prepare_smem(k, smem);
  if (e != cudaSuccess) return e;
  k<<<P.B, NTHREADS, smem, st>>>(P);
  return cudaGetLastError();
}
template cudaError_t launch_fwd_v<QP_T, QP_SW, QP_CH>(const FwdParams<QP_T>&, size_t, cudaStream_t);
#elif QP_KIND == 1
template <typename T>
cudaError_t launch_fwd_large_v(const FwdParams<T>& P, size_t smem, cudaStream_t st) {
  if (P.blocks > 0) return launch_fwd_wide_v<T>(P, smem, st);
  auto k = qp_fwd_large_kernel<T, 0>;
  cudaError_t e = prepare_smem(k, smem);
  if (e != cudaSuccess) return e;
  k<<<P.B, NTHREADS, smem, st>>>(P);
  return cudaGetLastError();
}
template cudaError_t launch_fwd_large_v<QP_T>(const FwdParams<QP_T>&, size_t, cudaStream_t);
template <typename T>
cudaError_t launch_fwd_packed_large_v(const PackedFwdParams<T>& P, size_t smem, cudaStream_t st) {
  if (P.blocks > 0) return launch_fwd_packed_wide_v<T>(P, smem, st);
  auto k = qp_fwd_packed_large_kernel<T, 0>;
  cudaError_t e = prepare_smem(k, smem);
  if (e != cudaSuccess) return e;
  k<<<P.B, NTHREADS, smem, st>>>(P);
  return cudaGetLastError();
}
template cudaError_t launch_fwd_packed_large_v<QP_T>(const PackedFwdParams<QP_T>&, size_t, cudaStream_t);
#elif QP_KIND == 3
// A launch of clusters of `blocks` blocks, `count` of them.
template <typename K, typename P>
static cudaError_t launch_clusters(K kernel, const P& params, int count, int blocks, size_t smem,
                                   cudaStream_t st) {
#if defined(QP_HOST_EMULATION)
  emu_launch_clusters(kernel, count, blocks, smem, params);
  return cudaSuccess;
#else
  cudaLaunchConfig_t c = {};
  c.gridDim = dim3((unsigned)(count * blocks));
  c.blockDim = dim3(NTHREADS);
  c.dynamicSmemBytes = smem;
  c.stream = st;
  cudaLaunchAttribute a;
  a.id = cudaLaunchAttributeClusterDimension;
  a.val.clusterDim.x = (unsigned)blocks;
  a.val.clusterDim.y = a.val.clusterDim.z = 1;
  c.attrs = &a;
  c.numAttrs = 1;
  return cudaLaunchKernelEx(&c, kernel, params);
#endif
}
template <typename T>
cudaError_t launch_fwd_wide_v(const FwdParams<T>& P, size_t smem, cudaStream_t st) {
  auto k = P.blocks == 1 ? qp_fwd_large_kernel<T, 1> : qp_fwd_large_kernel<T, 2>;
  cudaError_t e = prepare_smem(k, smem);
  if (e != cudaSuccess) return e;
  if (P.blocks > 1) return launch_clusters(k, P, P.B, P.blocks, smem, st);
  k<<<P.B, NTHREADS, smem, st>>>(P);
  return cudaGetLastError();
}
template cudaError_t launch_fwd_wide_v<QP_T>(const FwdParams<QP_T>&, size_t, cudaStream_t);
template <typename T>
cudaError_t launch_fwd_packed_wide_v(const PackedFwdParams<T>& P, size_t smem, cudaStream_t st) {
  auto k = P.blocks == 1 ? qp_fwd_packed_large_kernel<T, 1> : qp_fwd_packed_large_kernel<T, 2>;
  cudaError_t e = prepare_smem(k, smem);
  if (e != cudaSuccess) return e;
  if (P.blocks > 1) return launch_clusters(k, P, P.B, P.blocks, smem, st);
  k<<<P.B, NTHREADS, smem, st>>>(P);
  return cudaGetLastError();
}
template cudaError_t launch_fwd_packed_wide_v<QP_T>(const PackedFwdParams<QP_T>&, size_t, cudaStream_t);
#elif QP_KIND == 2
template <typename T, int SW, int CH>
cudaError_t launch_fwd_packed_v(const PackedFwdParams<T>& P, size_t smem, int grid, cudaStream_t st) {
  auto k = qp_fwd_packed_kernel<T, SW, CH>;
  cudaError_t e = prepare_smem(k, smem);
  if (e != cudaSuccess) return e;
  k<<<grid, NTHREADS, smem, st>>>(P);
  return cudaGetLastError();
}
template cudaError_t launch_fwd_packed_v<QP_T, QP_SW, QP_CH>(const PackedFwdParams<QP_T>&, size_t, int,
                                                             cudaStream_t);
#else
#error "unknown QP_KIND"
#endif

}  // namespace qpk
