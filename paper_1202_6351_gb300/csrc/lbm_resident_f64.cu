// lbm_resident_f64.cu -- the on-chip kernel of small lattices for LBM_F64 storage.
#include "lbm_resident.cuh"

namespace lbm {
cudaError_t launch_resident_f64(const Args& a, int model, int force, unsigned long long t0, int n, cudaStream_t s) {
    return launch_resident_store<LBM_F64>(a, model, force, t0, n, s);
}
}  // namespace lbm
