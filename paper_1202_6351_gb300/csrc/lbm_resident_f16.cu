// lbm_resident_f16.cu -- the on-chip kernel of small lattices for LBM_F16DEV storage.
#include "lbm_resident.cuh"

namespace lbm {
cudaError_t launch_resident_f16(const Args& a, int model, int force, unsigned long long t0, int n, cudaStream_t s) {
    return launch_resident_store<LBM_F16DEV>(a, model, force, t0, n, s);
}
}  // namespace lbm
