// Many steps of a small box in one launch, StoreF16 storage (see lbm_multi.cuh).
#include "lbm_multi.cuh"

namespace lbm {
int launch_multi_f16(int vel, int force, bool sr, void* fin, void* fout, const uint32_t* nbr, const float* Ef, int n,
                     unsigned* count, bool* in_fin, const KParams& p, cudaStream_t s) {
    return multik::launch_storage<StoreF16, true>(vel, force, sr, fin, fout, nbr, Ef, n, count, in_fin, p, s);
}
}  // namespace lbm
