// Many steps of a small box in one launch, StoreF32 storage (see lbm_multi.cuh).
#include "lbm_multi.cuh"

namespace lbm {
int launch_multi_f32(int vel, int force, bool sr, void* fin, void* fout, const uint32_t* nbr, const float* Ef, int n,
                     unsigned* count, bool* in_fin, const KParams& p, cudaStream_t s) {
    return multik::launch_storage<StoreF32, false>(vel, force, sr, fin, fout, nbr, Ef, n, count, in_fin, p, s);
}
}  // namespace lbm
