// lbm_batch_cascaded.cu -- batch kernels (one step, and several steps per launch) for the cascaded collision.
#include "lbm_batch_fused.cuh"
#include "lbm_batch_impl.cuh"

namespace lbm {
cudaError_t launch_batch_cascaded(int grid, const BatchDomain* doms, const int* tiles, int ntiles, int lbx, int rows, int flip,
                            int policy, int* counter, const unsigned* rtab, int rstride, int kstep,
                            cudaStream_t s) {
    batch_kernel<LBM_CASCADED><<<grid, kBatchThreads, 0, s>>>(doms, tiles, ntiles, lbx, rows, flip, policy, counter, rtab, rstride, kstep);
    return cudaGetLastError();
}
int batch_blocks_per_sm_cascaded() {
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, batch_kernel<LBM_CASCADED>, kBatchThreads, 0) != cudaSuccess) return 1;
    return n > 0 ? n : 1;
}
cudaError_t launch_batch_fused_cascaded(int cls, int ntiles, const BatchDomain* doms, const BatchPair* pairs,
                                  const int* tiles, int k, const unsigned* rtab, int rstride, int kstep, int* err,
                                  cudaStream_t s) {
    return launch_batch_fused_model<LBM_CASCADED>(cls, ntiles, doms, pairs, tiles, k, rtab, rstride, kstep, err, s);
}
cudaError_t launch_batch_multi_cascaded(int store, int ntiles, const BatchDomain* doms, const BatchPair* pairs,
                                        const int* tiles, int k, int steps, int* err, cudaStream_t s) {
    switch (store) {
        case LBM_F32: return launch_batch_multi<LBM_F32>(ntiles, doms, pairs, tiles, k, steps, err, s);
        case LBM_F16DEV: return launch_batch_multi<LBM_F16DEV>(ntiles, doms, pairs, tiles, k, steps, err, s);
        default: return launch_batch_multi<LBM_BF16DEV>(ntiles, doms, pairs, tiles, k, steps, err, s);
    }
}
}  // namespace lbm
