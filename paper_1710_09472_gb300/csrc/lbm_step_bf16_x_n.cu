// Step kernels instantiated for StoreBF16 storage, D3V27 and D1V3, nearest rounding (see lbm_step.cuh).
#include "lbm_step.cuh"

namespace lbm {
int launch_step_bf16_x_n(int vel, int force, bool efield, const void* fin, void* fout, const uint32_t* nbr, const float* Ef,
    const KParams& p, cudaStream_t s) {
    return stepk::launch_storage<StoreBF16, false, 1>(vel, force, efield, fin, fout, nbr, Ef, p, s);
}
}  // namespace lbm
