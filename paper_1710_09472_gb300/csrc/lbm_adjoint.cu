// Reverse-step dispatch: per-storage launchers (lbm_adjoint_{f32,f16,bf16}.cu)
// and the gradient slot count.
#include "lbm_adjoint.cuh"

namespace lbm {

int launch_adjoint_seed_f32(int, const void*, const uint32_t*, const float*, const float*, float*, double*, bool,
                            const KParams&, cudaStream_t);
int launch_adjoint_seed_f16(int, const void*, const uint32_t*, const float*, const float*, float*, double*, bool,
                            const KParams&, cudaStream_t);
int launch_adjoint_seed_bf16(int, const void*, const uint32_t*, const float*, const float*, float*, double*, bool,
                             const KParams&, cudaStream_t);
int launch_adjoint_step_f32(int, int, bool, bool, const void*, const float*, float*, const uint32_t*, const float*,
                            const float*, const float*, float*, double*, const KParams&, cudaStream_t);
int launch_adjoint_step_f16(int, int, bool, bool, const void*, const float*, float*, const uint32_t*, const float*,
                            const float*, const float*, float*, double*, const KParams&, cudaStream_t);
int launch_adjoint_step_bf16(int, int, bool, bool, const void*, const float*, float*, const uint32_t*, const float*,
                             const float*, const float*, float*, double*, const KParams&, cudaStream_t);

// the same for D3V27 and D1V3 (lbm_adjoint_*_x.cu)
int launch_adjoint_seed_f32_x(int, const void*, const uint32_t*, const float*, const float*, float*, double*, bool,
                              const KParams&, cudaStream_t);
int launch_adjoint_step_f32_x(int, int, bool, bool, const void*, const float*, float*, const uint32_t*, const float*,
                              const float*, const float*, float*, double*, const KParams&, cudaStream_t);
int launch_adjoint_seed_f16_x(int, const void*, const uint32_t*, const float*, const float*, float*, double*, bool,
                              const KParams&, cudaStream_t);
int launch_adjoint_step_f16_x(int, int, bool, bool, const void*, const float*, float*, const uint32_t*, const float*,
                              const float*, const float*, float*, double*, const KParams&, cudaStream_t);
int launch_adjoint_seed_bf16_x(int, const void*, const uint32_t*, const float*, const float*, float*, double*, bool,
                               const KParams&, cudaStream_t);
int launch_adjoint_step_bf16_x(int, int, bool, bool, const void*, const float*, float*, const uint32_t*, const float*,
                               const float*, const float*, float*, double*, const KParams&, cudaStream_t);

// the local chemical-potential model, D2V9 and D3V19 (lbm_adjoint_*_lmu.cu)
int launch_adjoint_step_f32_lmu(int, int, bool, bool, const void*, const float*, float*, const uint32_t*,
                                const float*, const float*, const float*, float*, double*, const KParams&,
                                cudaStream_t);
int launch_adjoint_step_f16_lmu(int, int, bool, bool, const void*, const float*, float*, const uint32_t*,
                                const float*, const float*, const float*, float*, double*, const KParams&,
                                cudaStream_t);
int launch_adjoint_step_bf16_lmu(int, int, bool, bool, const void*, const float*, float*, const uint32_t*,
                                 const float*, const float*, const float*, float*, double*, const KParams&,
                                 cudaStream_t);

namespace {
// Blocks stride over chunks of blockDim.x cells of the padded rows.
__global__ void k_fold_partials(float* __restrict__ part, double* __restrict__ acc, int64_t rows, int nx, int nxp) {
    const int chunks = (nx + blockDim.x - 1) / blockDim.x;
    for (int64_t t = blockIdx.x; t < rows * chunks; t += gridDim.x) {
        const int64_t r = t / chunks;
        const int x = (int)(t % chunks) * blockDim.x + threadIdx.x;
        if (x < nx) {
            acc[r * nx + x] += (double)part[r * nxp + x];
            part[r * nxp + x] = 0.f;
        }
    }
}
}  // namespace

int launch_fold_partials(float* part, double* acc, int D, const KParams& p, cudaStream_t s) {
    const int64_t rows = (int64_t)D * p.ny * p.nz;
    const int threads = p.nx >= 256 ? 256 : ((p.nx + 31) / 32) * 32;
    const int64_t want = rows * ((p.nx + threads - 1) / threads), cap = (int64_t)sm_count() * 8;
    k_fold_partials<<<(unsigned)(want < cap ? want : cap), threads, 0, s>>>(part, acc, rows, p.nx, p.nxp);
    return 1;
}

int64_t adjoint_slot_count(const KParams& p) {
    return adjk::slot_blocks(p) * adjk::kSlots;
}

int launch_adjoint_seed(int vel, int storage, const void* P, const uint32_t* nbr, const float* w_rho,
                        const float* w_j, float* lam, double* slots, bool in_window, const KParams& p,
                        cudaStream_t s) {
    if (vel == LBM_D3V27 || vel == LBM_D1V3) {
        if (storage == LBM_F16_DEV)
            return launch_adjoint_seed_f16_x(vel, P, nbr, w_rho, w_j, lam, slots, in_window, p, s);
        if (storage == LBM_BF16_DEV)
            return launch_adjoint_seed_bf16_x(vel, P, nbr, w_rho, w_j, lam, slots, in_window, p, s);
        return launch_adjoint_seed_f32_x(vel, P, nbr, w_rho, w_j, lam, slots, in_window, p, s);
    }
    if (storage == LBM_F16_DEV) return launch_adjoint_seed_f16(vel, P, nbr, w_rho, w_j, lam, slots, in_window, p, s);
    if (storage == LBM_BF16_DEV)
        return launch_adjoint_seed_bf16(vel, P, nbr, w_rho, w_j, lam, slots, in_window, p, s);
    return launch_adjoint_seed_f32(vel, P, nbr, w_rho, w_j, lam, slots, in_window, p, s);
}

int launch_adjoint_step(int vel, int storage, int force, bool efield, bool in_window, const void* P,
                        const float* lam_in, float* lam_out, const uint32_t* nbr, const float* Ef,
                        const float* w_rho, const float* w_j, float* gE, double* slots, const KParams& p,
                        cudaStream_t s) {
    if (p.lmu_tab && (vel == LBM_D2V9 || vel == LBM_D3V19)) {
        if (storage == LBM_F16_DEV)
            return launch_adjoint_step_f16_lmu(vel, force, efield, in_window, P, lam_in, lam_out, nbr, Ef, w_rho,
                                               w_j, gE, slots, p, s);
        if (storage == LBM_BF16_DEV)
            return launch_adjoint_step_bf16_lmu(vel, force, efield, in_window, P, lam_in, lam_out, nbr, Ef, w_rho,
                                                w_j, gE, slots, p, s);
        return launch_adjoint_step_f32_lmu(vel, force, efield, in_window, P, lam_in, lam_out, nbr, Ef, w_rho, w_j,
                                           gE, slots, p, s);
    }
    if (vel == LBM_D3V27 || vel == LBM_D1V3) {
        if (storage == LBM_F16_DEV)
            return launch_adjoint_step_f16_x(vel, force, efield, in_window, P, lam_in, lam_out, nbr, Ef, w_rho, w_j,
                                             gE, slots, p, s);
        if (storage == LBM_BF16_DEV)
            return launch_adjoint_step_bf16_x(vel, force, efield, in_window, P, lam_in, lam_out, nbr, Ef, w_rho, w_j,
                                              gE, slots, p, s);
        return launch_adjoint_step_f32_x(vel, force, efield, in_window, P, lam_in, lam_out, nbr, Ef, w_rho, w_j, gE,
                                         slots, p, s);
    }
    if (storage == LBM_F16_DEV)
        return launch_adjoint_step_f16(vel, force, efield, in_window, P, lam_in, lam_out, nbr, Ef, w_rho, w_j, gE,
                                       slots, p, s);
    if (storage == LBM_BF16_DEV)
        return launch_adjoint_step_bf16(vel, force, efield, in_window, P, lam_in, lam_out, nbr, Ef, w_rho, w_j, gE,
                                        slots, p, s);
    return launch_adjoint_step_f32(vel, force, efield, in_window, P, lam_in, lam_out, nbr, Ef, w_rho, w_j, gE, slots,
                                   p, s);
}

}  // namespace lbm
