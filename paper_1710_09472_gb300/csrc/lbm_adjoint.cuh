// Adjoint (reverse-mode) kernels of the fused semiclassical-LBM step
// (templates; included by one translation unit per storage type).
//
// Forward map per step: f_{t+1} = Stream(Collide(f_t)) (Sec. 9.1), with the
// collision of Sec. 9.1 and the forcing of Sec. 7.  For a loss
//   L = sum_{t in window} sum_x [w_rho(x) rho_t(x) + w_j(x) . j_t(x)]
// one reverse step maps lam_{t+1} = dL/df_{t+1} to lam_t = dL/df_t:
//   lamt_a(y) = lam_{t+1,a}(y + e_a)        (y + e_a fluid)
//             = lam_{t+1,abar}(y)           (y + e_a solid: transpose of bounce-back)
//   lam_t = (dCollide/df_t)^T lamt + [t in window] (w_rho + w_j . xi_a),
// and accumulates dL/dE(x), dL/dB, dL/dtau from lamt and f_t.  The collision
// Jacobian is applied through the chain rule over rho = sum f,
// j = sum f xi, u = j / rho; the formulas are the derivatives of the forward
// kernel's own expressions (direct N = 2 EDF of Sec. 5.1, forcing term of
// Sec. 7), so the reverse step is consistent with the FP32 forward.
//
// An adjoint field is lam[a * N + cell] (f-space, population layout) followed,
// at byte offset p.lgofs, by a link buffer: for every link of a fluid cell y
// into a solid cell (outgoing direction b) the slot of (y, b) in the forward's
// link numbering holds lam_bbar(y).  The bounced gather lamt_b(y) =
// lam_{t+1,bbar}(y) is then one contiguous range per row, as in the forward's
// pull.
//
// f_t is rebuilt by pulling the stored state of the forward replay.
// Parameter gradients: dL/dE(x) is accumulated per cell in FP32 partials
// that the driver folds into FP64 every few reverse steps; dL/dB,
// dL/dtau and the loss are block-reduced into per-block FP64 slots that each
// block owns (deterministic for a fixed launch shape).
#pragma once

#include <algorithm>

#include "lbm_device.cuh"

namespace lbm {
namespace adjk {

using dev::Cell;
using dev::cross3;
using dev::edot;
using dev::kBlock;
using dev::warp_sum;
constexpr int kSlots = 5;         // gB[3], gtau, loss

// Adds the block's sums of acc[FIRST .. kSlots) into slots[block * kSlots + k].
template <int FIRST = 0>
__device__ __forceinline__ void block_accumulate(double* acc, double* __restrict__ slots, int64_t block) {
    __shared__ double sh[32][kSlots];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int k = FIRST; k < kSlots; ++k) acc[k] = warp_sum(acc[k]);
    if (lane == 0) {
#pragma unroll
        for (int k = FIRST; k < kSlots; ++k) sh[wid][k] = acc[k];
    }
    __syncthreads();
    if (wid == 0) {
        const int nw = (blockDim.x + 31) / 32;
#pragma unroll
        for (int k = FIRST; k < kSlots; ++k) {
            double v = lane < nw ? sh[lane][k] : 0.0;
            v = warp_sum(v);
            if (lane == 0) slots[block * kSlots + k] += v;
        }
    }
}

// Local chemical-potential model (KParams::lmu_*): dth = thetabar - thetabar_w
// and d dth / d rho at the unscaled density deviation drho, from the same
// cubic Hermite table as the forward step (node and fraction taken relative
// to the node r = 1; outside the table the end value, slope 0).
__device__ __forceinline__ void lmu_table(const KParams& p, float drho, float& dth, float& ddth) {
    const float a = p.lmu_a * p.scale;  // table units per unit of unscaled deviation
    float x = drho * a;
    const float lo = -p.lmu_b, hi = (float)(p.lmu_n - 1) - p.lmu_b;
    const bool inside = x > lo && x < hi;
    x = fminf(fmaxf(x, lo), hi);  // also maps NaN to node 0
    const float fl = floorf(x);
    int i = (int)fl + (int)p.lmu_b;
    float t = x - fl;
    if (i > p.lmu_n - 2) {
        i = p.lmu_n - 2;
        t = 1.f;
    }
    const float t2 = t * t, t3 = t2 * t;
    const float2 A = __ldg(p.lmu_tab + i), B = __ldg(p.lmu_tab + i + 1);
    dth = (2.f * t3 - 3.f * t2 + 1.f) * A.x + (t3 - 2.f * t2 + t) * A.y + (3.f * t2 - 2.f * t3) * B.x +
          (t3 - t2) * B.y;
    const float dx = (6.f * t2 - 6.f * t) * A.x + (3.f * t2 - 4.f * t + 1.f) * A.y + (6.f * t - 6.f * t2) * B.x +
                     (3.f * t2 - 2.f * t) * B.y;
    ddth = inside ? dx * a : 0.f;
}

template <class L, bool EF>
__device__ __forceinline__ void load_E(const float* __restrict__ Ef, const KParams& p, int64_t pcell, float* E) {
    if (EF) {  // the padded field, at row * nxp + x
        E[0] = __ldg(Ef + pcell);
        E[1] = (L::D >= 2) ? __ldg(Ef + p.NP + pcell) : 0.f;
        E[2] = (L::D == 3) ? __ldg(Ef + 2 * p.NP + pcell) : 0.f;
    } else {
        E[0] = p.E[0];
        E[1] = p.E[1];
        E[2] = p.E[2];
    }
}

template <class L, bool WIN>
__device__ __forceinline__ void load_weights(const float* __restrict__ w_rho, const float* __restrict__ w_j,
                                             const KParams& p, uint32_t cell, float& wr, float* wj) {
    wr = 0.f;
    wj[0] = wj[1] = wj[2] = 0.f;
    if (WIN) {
        wr = w_rho ? __ldg(w_rho + cell) : 0.f;
#pragma unroll
        for (int d = 0; d < L::D; ++d) wj[d] = w_j ? __ldg(w_j + (int64_t)d * p.N + cell) : 0.f;
    }
}


// The reverse step at one fluid cell.  h: unscaled deviations of f_t at the
// cell; lt: lamt; E: the field there; wr, wj: its loss weights (used when WIN).
// Writes lam = lam_t at the cell and gEc = its dL/dE term; adds
// {dL/dB, dL/dtau, loss} into acc[0..4].
//
// Every sum over directions that the chain rule needs is a moment of
// mu_a = lt_a w_a: with the forcing-free part F_a = rho w_a [A + Bp (e.v) +
// Cp (e.v)^2 + k2_a v^2] and the term S_a = rho w_a [Bp (e.E) + 2 Cp (e.u)(e.E)
// + 2 k2_a (u.E + u.(e x B)/c_s)] of the forward step,
//   sum lt F   = rho [A M0 + Bp M1.v + Cp v.M2.v + v^2 K0],
//   d/dv       = rho [Bp M1 + 2 Cp M2 v + 2 K0 v],
//   sum lt S   = rho [Bp M1.E + 2 Cp u.M2.E + 2 K0 u.E + 2 u.(K1 x B)/c_s],
// with M0 = sum mu, M1 = sum mu e, M2 = sum mu e e^T, K0 = sum mu k2,
// K1 = sum mu k2 e.  Since w_a and k2_a are constant on each shell (|e|^2 =
// 1, 2, 3: axes, face diagonals, corners), the per-direction work is only
// the unweighted shell moments of lt.
template <class L, int FORCE, bool WIN, bool LMU = false>
__device__ __forceinline__ void adjoint_cell(const float* h, const float* lt, const float* E, const KParams& p,
                                             float wr, const float* wj, float* lam, float* gEc, double* acc) {
    constexpr int kR1 = shell_first<L>(1), kR2 = shell_first<L>(2), kR3 = shell_first<L>(3);
    // forward moments of f_t
    float drho = 0.f, j[3] = {0.f, 0.f, 0.f}, lth = 0.f;
    float rho, inv_rho, u[3], M0, K0, M1[3], K1[3], Mxx, Myy, Mzz, Mxy, Mxz, Myz;
    if constexpr (kR1 > 0 && kR2 > 0 && kR3 < 0) {
        // two moving shells (D2V9, D3V19): axis and diagonal
        constexpr int kAx = kR1, kDg = kR2;
        // shell moments of lt: axis (1) and diagonal (2); the rest shell adds to M0 only
        float L0a = 0.f, L0d = 0.f, L1a[3] = {0.f, 0.f, 0.f}, L1d[3] = {0.f, 0.f, 0.f};
        float L2a[3] = {0.f, 0.f, 0.f};                     // axis shell: diagonal of sum lt e e^T
        float L2d[3] = {0.f, 0.f, 0.f}, L2o[3] = {0.f, 0.f, 0.f};  // diagonal shell: diagonal; (xy, xz, yz)
#pragma unroll
        for (int a = 0; a < L::Q; ++a) {
            const int ex = L::c(a, 0), ey = L::c(a, 1), ez = L::c(a, 2);
            drho += h[a];
            j[0] += ex * h[a];
            j[1] += ey * h[a];
            j[2] += ez * h[a];
            lth = fmaf(lt[a], h[a], lth);
            const int sh = esq_of<L>(a);
            if (sh == 1) {
                L0a += lt[a];
                if (ex) { L1a[0] += ex * lt[a]; L2a[0] += lt[a]; }
                if (ey) { L1a[1] += ey * lt[a]; L2a[1] += lt[a]; }
                if (ez) { L1a[2] += ez * lt[a]; L2a[2] += lt[a]; }
            } else if (sh == 2) {
                L0d += lt[a];
                if (ex) { L1d[0] += ex * lt[a]; L2d[0] += lt[a]; }
                if (ey) { L1d[1] += ey * lt[a]; L2d[1] += lt[a]; }
                if (ez) { L1d[2] += ez * lt[a]; L2d[2] += lt[a]; }
                if (ex * ey) L2o[0] += ex * ey * lt[a];
                if (ex * ez) L2o[1] += ex * ez * lt[a];
                if (ey * ez) L2o[2] += ey * ez * lt[a];
            }
        }
        j[0] *= p.cs_inv;
        j[1] *= p.cs_inv;
        j[2] = (L::D == 3) ? j[2] * p.cs_inv : 0.f;
        rho = p.rho0 + drho;
        inv_rho = 1.0f / rho;
        u[0] = j[0] * inv_rho;
        u[1] = j[1] * inv_rho;
        u[2] = j[2] * inv_rho;
        // weighted moments
        const float w0 = p.w[0], w1 = p.w[kAx], w2 = p.w[kDg];
        const float k1 = p.k2[kAx], k2d = p.k2[kDg];
        M0 = w0 * lt[0] + w1 * L0a + w2 * L0d;
        K0 = w0 * p.k2[0] * lt[0] + w1 * k1 * L0a + w2 * k2d * L0d;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            M1[d] = w1 * L1a[d] + w2 * L1d[d];
            K1[d] = w1 * k1 * L1a[d] + w2 * k2d * L1d[d];
        }
        // M2 = w1 diag(L2a) + w2 [L2d on the diagonal, L2o off it]
        Mxx = w1 * L2a[0] + w2 * L2d[0];
        Myy = w1 * L2a[1] + w2 * L2d[1];
        Mzz = w1 * L2a[2] + w2 * L2d[2];
        Mxy = w2 * L2o[0];
        Mxz = w2 * L2o[1];
        Myz = w2 * L2o[2];
    } else {
        // unweighted moments of lt per shell s = |e|^2: sum lt, sum lt e, the
        // diagonal of sum lt e e^T, and its (xy, xz, yz) entries; the rest
        // direction adds to M0 and K0 only
        float L0[4] = {0.f, 0.f, 0.f, 0.f}, L1[4][3] = {}, L2[4][3] = {}, L2o[4][3] = {};
#pragma unroll
        for (int a = 0; a < L::Q; ++a) {
            const int ex = L::c(a, 0), ey = L::c(a, 1), ez = L::c(a, 2);
            drho += h[a];
            j[0] += ex * h[a];
            j[1] += ey * h[a];
            j[2] += ez * h[a];
            lth = fmaf(lt[a], h[a], lth);
            const int sh = esq_of<L>(a);
            if (sh == 0) continue;
            L0[sh] += lt[a];
            if (ex) { L1[sh][0] += ex * lt[a]; L2[sh][0] += lt[a]; }
            if (ey) { L1[sh][1] += ey * lt[a]; L2[sh][1] += lt[a]; }
            if (ez) { L1[sh][2] += ez * lt[a]; L2[sh][2] += lt[a]; }
            if (ex * ey) L2o[sh][0] += ex * ey * lt[a];
            if (ex * ez) L2o[sh][1] += ex * ez * lt[a];
            if (ey * ez) L2o[sh][2] += ey * ez * lt[a];
        }
        j[0] *= p.cs_inv;
        j[1] *= p.cs_inv;
        j[2] = (L::D == 3) ? j[2] * p.cs_inv : 0.f;
        rho = p.rho0 + drho;
        inv_rho = 1.0f / rho;
        u[0] = j[0] * inv_rho;
        u[1] = j[1] * inv_rho;
        u[2] = j[2] * inv_rho;
        // weighted moments: shell s contributes with w_s and w_s k2_s
        M0 = p.w[0] * lt[0];
        K0 = p.w[0] * p.k2[0] * lt[0];
        M1[0] = M1[1] = M1[2] = 0.f;
        K1[0] = K1[1] = K1[2] = 0.f;
        Mxx = Myy = Mzz = Mxy = Mxz = Myz = 0.f;
#pragma unroll
        for (int sh = 1; sh <= 3; ++sh) {
            const int r = sh == 1 ? kR1 : (sh == 2 ? kR2 : kR3);
            if (r < 0) continue;
            const float ws = p.w[r], wk = p.w[r] * p.k2[r];
            M0 += ws * L0[sh];
            K0 += wk * L0[sh];
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                M1[d] += ws * L1[sh][d];
                K1[d] += wk * L1[sh][d];
            }
            Mxx += ws * L2[sh][0];
            Myy += ws * L2[sh][1];
            Mzz += ws * L2[sh][2];
            Mxy += ws * L2o[sh][0];
            Mxz += ws * L2o[sh][1];
            Myz += ws * L2o[sh][2];
        }
    }
    auto m2v = [&](const float* v, float* out) {
        out[0] = Mxx * v[0] + Mxy * v[1] + Mxz * v[2];
        out[1] = Mxy * v[0] + Myy * v[1] + Myz * v[2];
        out[2] = Mxz * v[0] + Myz * v[1] + Mzz * v[2];
    };
    float acc_f[3], ue[3];
    if (FORCE == 0) {
        float uxb[3];
        cross3(u, p.B, uxb);
        acc_f[0] = E[0] + uxb[0];
        acc_f[1] = E[1] + uxb[1];
        acc_f[2] = (L::D == 3) ? E[2] + uxb[2] : 0.f;
        ue[0] = u[0] + p.tau * acc_f[0];
        ue[1] = u[1] + p.tau * acc_f[1];
        ue[2] = u[2] + p.tau * acc_f[2];
    } else {
        ue[0] = u[0];
        ue[1] = u[1];
        ue[2] = u[2];
    }
    const float u2 = ue[0] * ue[0] + ue[1] * ue[1] + ue[2] * ue[2];
    float M2v[3];
    m2v(ue, M2v);
    const float M1v = M1[0] * ue[0] + M1[1] * ue[1] + M1[2] * ue[2];
    const float vM2v = M2v[0] * ue[0] + M2v[1] * ue[1] + M2v[2] * ue[2];
    const float inv_tau = p.omega;
    // sum_a lt_a F_a / rho and sum_a lt_a heq_a
    const float ltF = p.A * M0 + p.Bp * M1v + p.Cp * vM2v + u2 * K0;
    const float ltHeq = p.A * drho * M0 + rho * (p.Bp * M1v + p.Cp * vM2v + u2 * K0);
    float gtau = (lth - ltHeq) * inv_tau * inv_tau;
    // dF/dv summed against mu: rho [Bp M1 + 2 Cp M2 v + 2 K0 v]
    float dF[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) dF[d] = rho * (p.Bp * M1[d] + 2.f * p.Cp * M2v[d] + 2.f * K0 * ue[d]);
    float rho_bar, u_bar[3], gBc[3];
    if (FORCE == 0) {
        rho_bar = ltF * inv_tau;
        const float ue_bar[3] = {dF[0] * inv_tau, dF[1] * inv_tau, dF[2] * inv_tau};
        gtau += ue_bar[0] * acc_f[0] + ue_bar[1] * acc_f[1] + ue_bar[2] * acc_f[2];
        float t1[3], t2[3];
        cross3(ue_bar, u, t1);    // d(u x B)/dB transposed
        cross3(p.B, ue_bar, t2);  // d(u x B)/du transposed
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            gEc[d] = p.tau * ue_bar[d];
            gBc[d] = p.tau * t1[d];
            u_bar[d] = ue_bar[d] + p.tau * t2[d];
        }
    } else {
        float M2E[3], K1xB[3];
        m2v(E, M2E);
        cross3(K1, p.B, K1xB);
        const float uE = u[0] * E[0] + u[1] * E[1] + u[2] * E[2];
        const float ltS = p.Bp * (M1[0] * E[0] + M1[1] * E[1] + M1[2] * E[2]) +
                          2.f * p.Cp * (u[0] * M2E[0] + u[1] * M2E[1] + u[2] * M2E[2]) +
                          2.f * (K0 * uE + (u[0] * K1xB[0] + u[1] * K1xB[1] + u[2] * K1xB[2]) * p.cs_inv);
        rho_bar = ltF * inv_tau + ltS;
        // d(sum lt S)/du = rho [2 Cp M2 E + 2 K0 E + 2 (K1 x B)/c_s]; d/dE = dF; d/dB = (2 rho / c_s) u x K1
        float uxK[3];
        cross3(u, K1, uxK);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            u_bar[d] = dF[d] * inv_tau + rho * (2.f * p.Cp * M2E[d] + 2.f * (K0 * E[d] + K1xB[d] * p.cs_inv));
            gEc[d] = dF[d];
            gBc[d] = 2.f * rho * p.cs_inv * uxK[d];
        }
    }
    if constexpr (LMU && kR1 > 0 && kR2 > 0 && kR3 < 0) {
        // local-mu model (D2V9, D3V19): the collision adds w rho w_a K_a dth(rho),
        // whose rho-derivative feeds rho_bar and whose w-derivative dL/dtau.
        // K_a = K_0 + (K_1 - K_0) |e_a|^2 is affine in |e_a|^2, so
        // sum_a lt_a w_a K_a = K_0 M0 + (K_1 - K_0) trace(M2).
        {
            const float KM = p.lmu_K[0] * M0 + (p.lmu_K[1] - p.lmu_K[0]) * (Mxx + Myy + Mzz);
            float dth, ddth;
            lmu_table(p, drho, dth, ddth);
            rho_bar += inv_tau * (dth + rho * ddth) * KM;
            gtau -= inv_tau * inv_tau * rho * dth * KM;
        }
    }
    rho_bar -= (u_bar[0] * u[0] + u_bar[1] * u[1] + u_bar[2] * u[2]) * inv_rho;
    const float ub[3] = {u_bar[0] * inv_rho * p.cs_inv, u_bar[1] * inv_rho * p.cs_inv,
                         u_bar[2] * inv_rho * p.cs_inv};
    float wjs[3] = {0.f, 0.f, 0.f};
    if (WIN) {
#pragma unroll
        for (int d = 0; d < L::D; ++d) wjs[d] = wj[d] * p.cs_inv;
        acc[4] += (double)wr * (double)rho + (double)wj[0] * (double)j[0] + (double)wj[1] * (double)j[1] +
                  (double)wj[2] * (double)j[2];
    }
    const float omm = 1.0f - p.omega;
#pragma unroll
    for (int b = 0; b < L::Q; ++b) {
        float v = omm * lt[b] + rho_bar + edot<L>(b, ub);
        if (WIN) v += wr + edot<L>(b, wjs);
        lam[b] = v;
    }
    acc[0] += gBc[0];
    acc[1] += gBc[1];
    acc[2] += gBc[2];
    acc[3] += gtau;
}

// The link-buffer copies of a fluid cell's lam_t: slot (y, b) = lam_bbar(y)
// for every outgoing direction b into a solid cell.
template <class L>
__device__ __forceinline__ void store_lam_links(float* __restrict__ lamG, uint32_t o, uint32_t lb, const float* lam) {
#pragma unroll
    for (int b = 1; b < L::Q; ++b)
        if ((o >> b) & 1u) lamG[link_slot(lb, o, b)] = lam[opposite(b)];
}

__device__ __forceinline__ float* link_part(float* lam, const KParams& p) {
    return reinterpret_cast<float*>(reinterpret_cast<char*>(lam) + p.lgofs);
}
__device__ __forceinline__ const float* link_part(const float* lam, const KParams& p) {
    return reinterpret_cast<const float*>(reinterpret_cast<const char*>(lam) + p.lgofs);
}

// ---------------------------------------------------------------------------
// lam_T = dl_T/df_T (zero outside the window) and the loss term of step T.
// ---------------------------------------------------------------------------
template <class L, class S>
__global__ void __launch_bounds__(kBlock) k_adjoint_seed(const typename S::T* __restrict__ P,
                                                         const uint32_t* __restrict__ nbr,
                                                         const float* __restrict__ w_rho,
                                                         const float* __restrict__ w_j, float* __restrict__ lam,
                                                         double* __restrict__ slots, int in_window, int chunks, KParams p) {
    double acc[kSlots] = {0.0, 0.0, 0.0, 0.0, 0.0};
    const int64_t tiles = (int64_t)p.ny * p.nz * chunks;
    for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
        Cell c;
        if (!dev::cell_at(p, (int)(t / chunks), (int)(t % chunks) * blockDim.x + threadIdx.x, c)) continue;
        const uint32_t m = nbr[c.cell];
        if (m & kSolidBit) {
#pragma unroll
            for (int a = 0; a < L::Q; ++a) lam[dev::pop_at<L>(p, c, a, 0)] = 0.f;
        } else {
            float wr = 0.f, wj[3] = {0.f, 0.f, 0.f};
            if (in_window) {
                wr = w_rho ? w_rho[c.cell] : 0.f;
#pragma unroll
                for (int d = 0; d < L::D; ++d) wj[d] = w_j ? w_j[(int64_t)d * p.N + c.cell] * p.cs_inv : 0.f;
                // loss of step T: w_rho rho + w_j . j
                float h[L::Q];
                dev::pull<L, S>(P, p, m, c, h);
                float drho = 0.f, jx = 0.f, jy = 0.f, jz = 0.f;
#pragma unroll
                for (int a = 0; a < L::Q; ++a) {
                    const float ha = h[a] * p.inv_scale;
                    drho += ha;
                    jx += L::c(a, 0) * ha;
                    jy += L::c(a, 1) * ha;
                    jz += L::c(a, 2) * ha;
                }
                acc[4] += (double)wr * (double)(p.rho0 + drho) + (double)wj[0] * jx + (double)wj[1] * jy +
                         (double)wj[2] * jz;
            }
            float lm[L::Q];
#pragma unroll
            for (int a = 0; a < L::Q; ++a) {
                lm[a] = wr + edot<L>(a, wj);
                lam[dev::pop_at<L>(p, c, a, 0)] = lm[a];
            }
            const uint32_t o = outgoing<L::Q>(m);
            if (o) store_lam_links<L>(link_part(lam, p), o, __ldg(p.lbase + c.cell), lm);
        }
    }
    if (in_window) block_accumulate<4>(acc, slots, blockIdx.x);  // the loss only
}

// ---------------------------------------------------------------------------
// One reverse step, general kernel: one thread per cell, direct global loads.
// The blocks stride over the tiles (kAdjPerSm of them per SM) and reduce their
// FP64 sums once at the end.  A reduction per 128 cells took the FP64 pipe
// (two adds per cycle and SM) longer than the step itself: 0.095 ms on 1024^2
// cells of D2V9 FP32, 0.112 ms inside the loss window.
// ---------------------------------------------------------------------------
template <class L, class S, int FORCE, bool EF, bool WIN>
__global__ void __launch_bounds__(kBlock) k_adjoint_step(
    const typename S::T* __restrict__ P,  // stored state of the forward replay at step t
    const float* __restrict__ lam_in,     // lam_{t+1}
    float* __restrict__ lam_out,          // lam_t
    const uint32_t* __restrict__ nbr, const float* __restrict__ Ef, const float* __restrict__ w_rho,
    const float* __restrict__ w_j, float* __restrict__ gE, double* __restrict__ slots, int chunks, KParams p) {
    double acc[kSlots] = {0.0, 0.0, 0.0, 0.0, 0.0};
    const int64_t tiles = (int64_t)p.ny * p.nz * chunks;
    for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
        Cell c;
        if (!dev::cell_at(p, (int)(t / chunks), (int)(t % chunks) * blockDim.x + threadIdx.x, c)) continue;
        const uint32_t m = __ldg(nbr + c.cell);
        if (m & kSolidBit) {
#pragma unroll
            for (int a = 0; a < L::Q; ++a) lam_out[dev::pop_at<L>(p, c, a, 0)] = 0.f;
        } else {
            // f_t(y): pull of the stored state; lamt(y): gather from downstream
            float h[L::Q], lt[L::Q];
            dev::pull<L, S>(P, p, m, c, h);
            const uint32_t o = outgoing<L::Q>(m);
            const uint32_t lb = m ? __ldg(p.lbase + c.cell) : 0u;
            const float* lg = link_part(lam_in, p) + lb;
#pragma unroll
            for (int a = 0; a < L::Q; ++a) {
                h[a] *= p.inv_scale;
                // x + e_a solid: the next link slot (address selected, as in pull)
                const bool bounced = a != 0 && ((o >> a) & 1u);
                const float* q = lam_in + dev::pop_at<L>(p, c, a, +1);
                if (bounced) q = lg;
                lg += bounced;
                lt[a] = __ldg(q);
            }
            float E[3], wr, wj[3], lam[L::Q], gEc[3];
            load_E<L, EF>(Ef, p, c.pcell, E);
            load_weights<L, WIN>(w_rho, w_j, p, c.cell, wr, wj);
            // the local-mu model is built for D2V9 and D3V19 (the host refuses others)
            constexpr bool kLmu = L::Q == 9 || L::Q == 19;
            if (kLmu && p.lmu_tab)
                adjoint_cell<L, FORCE, WIN, kLmu>(h, lt, E, p, wr, wj, lam, gEc, acc);
            else
                adjoint_cell<L, FORCE, WIN>(h, lt, E, p, wr, wj, lam, gEc, acc);
#pragma unroll
            for (int b = 0; b < L::Q; ++b) lam_out[dev::pop_at<L>(p, c, b, 0)] = lam[b];
            if (o) store_lam_links<L>(link_part(lam_out, p), o, lb, lam);
            if (gE) {
#pragma unroll
                for (int d = 0; d < L::D; ++d) gE[(int64_t)d * p.NP + c.pcell] += gEc[d];
            }
        }
    }
    block_accumulate(acc, slots, blockIdx.x);
}

// ---------------------------------------------------------------------------
// Row-staged reverse step (persistent; block b takes units b, b + G, ...: rows,
// or segments of long rows).  One stage holds, for the unit at row (y, z):
//   - with dL/dE, the unit's D rows of its FP32 partials (accumulated in place
//     and stored back after the unit); with a per-cell field, its D rows of E;
//   - the Q pull rows of the forward state P_t in slot order: direction a
//     from row (y - e_ay, z - e_az), read at x - e_ax (dev::stage_rows; the
//     columns beside a segment as in the forward kernel);
//   - the unit's cell order (fluid cells first, ascending x);
//   - its window of P_t's link buffer (bounced pulls);
//   - the Q gather rows of lam_{t+1} in slot order: direction a from row
//     (y + e_ay, z + e_az), read at x + e_ax;
//   - its windows of lam_{t+1}'s link buffer (bounced gathers) and of the
//     link descriptors;
// all by bulk asynchronous copies, completing on the stage's mbarrier, issued by
// lane 0 of the last two warps (waits are bounded, as in the forward's
// row-staged kernel).  One pass over the
// unit's links patches both bounced reads into the staged rows (the solid
// neighbour's slot, read by that cell alone), so cells read their rows
// without link logic.  Thread i takes the i-th cell of the row's order, so
// each thread's FP64 sums see the same cells in the same order on every run.
// lam_t goes through shared-memory output rows (zeros for solid cells) that
// leave by one bulk store (lam has the populations' slot layout), and one pass
// over the links copies lam_bbar(x) into the unit's range of the new link
// buffer.  dL/dB, dL/dtau and the loss stay
// in registers until the block's single reduction at the end.
// ---------------------------------------------------------------------------
template <class L, class S>
struct AdjLayout {
    int rs, lorder, gcapP, gcapL;  // shared-memory row stride (elements), order entries; gcapL also bounds the
                                   // descriptor window (4-byte elements)
    int gerow, efrow;              // bytes of the staged dL/dE rows and E rows (FP32), 0 when absent
    int hP, hL;                    // bytes of the halo arrays of P_t and lam (segments)
    __device__ __host__ int prow() const { return L::Q * rs * S::kBytes; }
    __device__ __host__ int lrow() const { return L::Q * rs * 4; }
    __device__ __host__ int bytes() const {
        return gerow + prow() + 2 * lorder + gcapP + lrow() + 2 * gcapL + efrow + hP + hL;
    }
    __device__ unsigned char* gerows(unsigned char* st) const { return st; }
    __device__ unsigned char* prows(unsigned char* st) const { return st + gerow; }
    __device__ unsigned char* order(unsigned char* st) const { return st + gerow + prow(); }
    __device__ unsigned char* plinks(unsigned char* st) const { return order(st) + 2 * lorder; }
    __device__ unsigned char* lrows(unsigned char* st) const { return plinks(st) + gcapP; }
    __device__ unsigned char* llinks(unsigned char* st) const { return lrows(st) + lrow(); }
    __device__ unsigned char* descs(unsigned char* st) const { return llinks(st) + gcapL; }
    __device__ unsigned char* efrows(unsigned char* st) const { return descs(st) + gcapL; }
    __device__ unsigned char* phalo(unsigned char* st) const { return efrows(st) + efrow; }
    __device__ unsigned char* lhalo(unsigned char* st) const { return phalo(st) + hP; }
};

// Two threads fill a stage with unit `unit` (links [g0, g1)), all copies
// completing on bar.  The first (adj_stage_state) arms the mbarrier with the
// byte count of all, records where the windows start (ws[0]: P_t's link window;
// ws[1]: lam's link window and the descriptor window, which start at the same
// element) and copies P_t's rows, the cell order, P_t's links and the
// descriptors; the other (adj_stage_lam) lam's rows and links and, where they
// exist, the unit's dL/dE partials (accumulated in place, stored back after the
// unit) and its E.  A copy holds its issuing thread for a hundred cycles or
// more and there are up to 28; the phase cannot complete before the first
// thread has armed it, so the order of the two does not matter.
template <class L, class S, int RS, int MODE>
__device__ __forceinline__ void adj_stage_state(unsigned char* st, const AdjLayout<L, S>& lay, uint64_t* bar,
                                                const typename S::T* P, int unit, uint32_t g0, uint32_t g1,
                                                uint32_t* ws, const KParams& p) {
    uint64_t pb0, pb1, lb0, lb1;
    dev::window_bytes(g0, g1, S::kBytes, pb0, pb1);
    dev::window_bytes(g0, g1, 4, lb0, lb1);
    ws[0] = (uint32_t)(pb0 / S::kBytes);
    ws[1] = (uint32_t)(lb0 / 4);
    dev::mbar_expect_tx(bar, (uint32_t)(lay.prow() + lay.lrow() + lay.gerow + lay.efrow) +
                                 2u * (uint32_t)lay.lorder + (uint32_t)(pb1 - pb0) + 2u * (uint32_t)(lb1 - lb0));
    dev::stage_rows<L, RS, MODE, true>(reinterpret_cast<typename S::T*>(lay.prows(st)), P,
                                      dev::unit_at<RS, MODE>(p, unit), bar, p);
    dev::bulk_load(lay.order(st), p.rorder + (int64_t)unit * lay.lorder, 2u * (uint32_t)lay.lorder, bar);
    if (pb1 > pb0)
        dev::bulk_load(lay.plinks(st), reinterpret_cast<const unsigned char*>(P) + p.gofs + pb0, (uint32_t)(pb1 - pb0),
                       bar);
    if (lb1 > lb0)
        dev::bulk_load(lay.descs(st), reinterpret_cast<const unsigned char*>(p.ldesc) + lb0, (uint32_t)(lb1 - lb0),
                       bar);
}
template <class L, class S, int RS, int MODE>
__device__ __forceinline__ void adj_stage_lam(unsigned char* st, const AdjLayout<L, S>& lay, uint64_t* bar,
                                              const float* lam, const float* gE, const float* Ef, int unit,
                                              uint32_t g0, uint32_t g1, const KParams& p) {
    uint64_t lb0, lb1;
    dev::window_bytes(g0, g1, 4, lb0, lb1);
    dev::stage_rows<L, RS, MODE, false>(reinterpret_cast<float*>(lay.lrows(st)), lam,
                                       dev::unit_at<RS, MODE>(p, unit), bar, p);
    if (lb1 > lb0)
        dev::bulk_load(lay.llinks(st), reinterpret_cast<const unsigned char*>(lam) + p.lgofs + lb0,
                       (uint32_t)(lb1 - lb0), bar);
    const uint32_t fb = (uint32_t)lay.rs * 4u;  // bytes of a field row
    const int64_t f0 = (int64_t)unit * lay.rs;
    if (lay.gerow) {
#pragma unroll
        for (int d = 0; d < L::D; ++d)
            dev::bulk_load(lay.gerows(st) + d * lay.rs * 4, gE + (int64_t)d * p.NP + f0, fb, bar);
    }
    if (lay.efrow) {
#pragma unroll
        for (int d = 0; d < L::D; ++d)
            dev::bulk_load(lay.efrows(st) + d * lay.rs * 4, Ef + (int64_t)d * p.NP + f0, fb, bar);
    }
}

template <class L, class S, int FORCE, bool EF, bool WIN, int STAGES, int RS, int MODE, bool LMU = false>
__global__ void __launch_bounds__(256, 2) k_adjoint_rows(const typename S::T* __restrict__ P,
                                                         const float* __restrict__ lam_in,
                                                         float* __restrict__ lam_out,
                                                         const float* __restrict__ Ef,
                                                         const float* __restrict__ w_rho,
                                                         const float* __restrict__ w_j, float* __restrict__ gE,
                                                         double* __restrict__ slots, int gcapP, int gcapL, KParams p) {
    using T = typename S::T;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    // RS: units of that many columns (a compile-time stride; 0: a run-time one).
    // MODE: rows of exactly RS cells (kExactRow), rows (kWholeRow) or segments
    constexpr bool kOne = MODE != kSegment, kExact = RS && MODE == kExactRow;
    const int rs = RS ? RS : p.seglen;
    const bool halo = !kOne;
    const AdjLayout<L, S> lay{rs, p.lorder, gcapP, gcapL, gE ? L::D * rs * 4 : 0, EF ? L::D * rs * 4 : 0,
                              kOne ? 0 : dev::halo_bytes(L::Q, p.nseg, S::kBytes),
                              kOne ? 0 : dev::halo_bytes(L::Q, p.nseg, 4)};
    const int sbytes = lay.bytes();
    float* outrow = reinterpret_cast<float*>(smem_raw + STAGES * sbytes);
    __shared__ __align__(8) uint64_t bar[STAGES];
    __shared__ uint32_t wstart[STAGES][2];
    float* lamG_out = link_part(lam_out, p);
    const int U = p.ny * p.nz * (kOne ? 1 : p.nseg);
    const int G = gridDim.x;
    const bool leader = threadIdx.x == 0;
    const int warp = (int)(threadIdx.x >> 5), nw = (int)(blockDim.x >> 5), lane = (int)(threadIdx.x & 31);
    // lane 0 of the last warp and of the one before it (the same in a block of one warp)
    const bool issuer = (int)threadIdx.x == (int)blockDim.x - 32;
    const bool lam_issuer = nw > 1 ? (int)threadIdx.x == (int)blockDim.x - 64 : issuer;
    auto range = [&](int unit, uint32_t& g0, uint32_t& g1) {
        g0 = g1 = 0u;
        if (unit < U) {
            g0 = __ldg(p.rowG + unit);
            g1 = __ldg(p.rowG + unit + 1);
        }
    };
    if (leader) {
#pragma unroll
        for (int k = 0; k < STAGES; ++k) dev::mbar_init(&bar[k], 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    static_assert(STAGES == 2, "the halo values are fetched one unit ahead");
    if (halo && dev::halo_thread<L>()) {
        const dev::UnitAt at = dev::unit_at<RS, MODE>(p, blockIdx.x);
        dev::halo_put<L, true>(reinterpret_cast<T*>(lay.phalo(smem_raw)), dev::halo_fetch<L, true>(P, at, p));
        dev::halo_put<L, false>(reinterpret_cast<float*>(lay.lhalo(smem_raw)), dev::halo_fetch<L, false>(lam_in, at, p));
    }
    __syncthreads();
    if (issuer || lam_issuer) {
#pragma unroll
        for (int k = 0; k < STAGES - 1; ++k) {
            const int uk = blockIdx.x + k * G;
            if (uk < p.staged) {
                uint32_t g0, g1;
                range(uk, g0, g1);
                unsigned char* st = smem_raw + k * sbytes;
                if (issuer) adj_stage_state<L, S, RS, MODE>(st, lay, &bar[k], P, uk, g0, g1, wstart[k], p);
                if (lam_issuer) adj_stage_lam<L, S, RS, MODE>(st, lay, &bar[k], lam_in, gE, Ef, uk, g0, g1, p);
            }
        }
    }
    double acc[kSlots] = {0.0, 0.0, 0.0, 0.0, 0.0};
    int it = 0;
    bool ok = true;  // false once a wait has run out (the same in every thread after the first barrier)
    for (int u = blockIdx.x; u < U; u += G, ++it) {
        const int cs = it % STAGES;
        const int un = u + (STAGES - 1) * G;       // the unit fetched during this one ...
        const int sn = (it + STAGES - 1) % STAGES;  // ... into the stage of the previous unit
        uint32_t g0, g1;
        range(u, g0, g1);
        unsigned char* st = smem_raw + cs * sbytes;
        uint16_t* ord = reinterpret_cast<uint16_t*>(lay.order(st));
        ok = dev::stage_wait(&bar[cs], (uint32_t)(it / STAGES) & 1u, ok, 2, g0, g1, ord, p);
        T* prow = reinterpret_cast<T*>(lay.prows(st));
        float* ge_s = reinterpret_cast<float*>(lay.gerows(st));
        const float* ef_s = reinterpret_cast<const float*>(lay.efrows(st));
        float* lrow = reinterpret_cast<float*>(lay.lrows(st));
        const uint32_t* desc = reinterpret_cast<const uint32_t*>(lay.descs(st));
        const uint32_t d0 = wstart[cs][1];
        T* phal = reinterpret_cast<T*>(lay.phalo(st));
        float* lhal = reinterpret_cast<float*>(lay.lhalo(st));
        dev::patch_links<true, !kOne>(prow, rs, phal, L::Q, reinterpret_cast<const T*>(lay.plinks(st)),
                                        wstart[cs][0], g0, g1, desc, d0);
        dev::patch_links<false, !kOne>(lrow, rs, lhal, L::Q, reinterpret_cast<const float*>(lay.llinks(st)), d0, g0,
                                         g1, desc, d0);
        dev::bulk_wait_read();  // this thread's bulk stores of the previous unit have read their sources
        // bounced values in place, output rows free; a timeout anywhere in
        // the block stops the copies
        ok = __syncthreads_and(ok) != 0;
        if ((issuer || lam_issuer) && ok && un < U) {
            // refill the stage of the previous unit (every thread is past its
            // reads of it and its wait on that stage's barrier)
            uint32_t n0, n1;
            range(un, n0, n1);
            unsigned char* sst = smem_raw + sn * sbytes;
            if (issuer) adj_stage_state<L, S, RS, MODE>(sst, lay, &bar[sn], P, un, n0, n1, wstart[sn], p);
            if (lam_issuer) adj_stage_lam<L, S, RS, MODE>(sst, lay, &bar[sn], lam_in, gE, Ef, un, n0, n1, p);
        }
        const bool fetch = halo && un < U && dev::halo_thread<L>();
        T hvP{};
        float hvL = 0.f;
        if (fetch) {
            const dev::UnitAt next = dev::unit_at<RS, MODE>(p, un);
            hvP = dev::halo_fetch<L, true>(P, next, p);
            hvL = dev::halo_fetch<L, false>(lam_in, next, p);
        }
        const int nf = ord[0];
        const dev::UnitAt at = dev::unit_at<RS, MODE>(p, u);
        const int nx = at.len;  // cells of the unit
        const uint32_t rowbase = (uint32_t)at.row * (uint32_t)(kExact ? RS : p.nx) + (uint32_t)at.x0;  // first cell
        for (int i = threadIdx.x; i < nx; i += blockDim.x) {
            const int x = (int)ord[8 + i];
            if (i < nf) {
                const uint32_t cell = rowbase + (uint32_t)x;
                // columns x - 1 and x + 1, as in the forward kernel
                const int xm = x == 0 ? nx - 1 : x - 1, xp = x == nx - 1 ? 0 : x + 1;
                const T *pm = prow + xm, *pp = prow + xp;
                const float *lm = lrow + xm, *lp = lrow + xp;
                int rm = rs, rp = rs;
                if (halo && x == 0) {
                    pm = phal;
                    lm = lhal;
                    rm = 1;
                }
                if (halo && x == nx - 1) {
                    pp = phal + L::Q;
                    lp = lhal + L::Q;
                    rp = 1;
                }
                float h[L::Q], lt[L::Q];
#pragma unroll
                for (int a = 0; a < L::Q; ++a) {
                    const int ex = L::c(a, 0), s = pop_slot<L>(a);
                    const int sm = s * (kOne ? rs : rm), sp = s * (kOne ? rs : rp);
                    h[a] = S::cvt(ex > 0 ? pm[sm] : (ex < 0 ? pp[sp] : prow[s * rs + x])) * p.inv_scale;
                    lt[a] = ex > 0 ? lp[sp] : (ex < 0 ? lm[sm] : lrow[s * rs + x]);
                }
                float E[3], wr, wj[3], lam[L::Q], gEc[3];
                if (EF) {
                    E[0] = ef_s[x];
                    E[1] = (L::D >= 2) ? ef_s[rs + x] : 0.f;
                    E[2] = (L::D == 3) ? ef_s[2 * rs + x] : 0.f;
                } else {
                    load_E<L, false>(Ef, p, 0, E);
                }
                load_weights<L, WIN>(w_rho, w_j, p, cell, wr, wj);
                adjoint_cell<L, FORCE, WIN, LMU>(h, lt, E, p, wr, wj, lam, gEc, acc);
#pragma unroll
                for (int b = 0; b < L::Q; ++b) outrow[pop_slot<L>(b) * rs + x] = lam[b];
                if (gE) {
#pragma unroll
                    for (int d = 0; d < L::D; ++d) ge_s[d * rs + x] += gEc[d];
                }
            } else {
#pragma unroll
                for (int b = 0; b < L::Q; ++b) outrow[b * rs + x] = 0.f;
            }
        }
        if (fetch) {
            dev::halo_put<L, true>(reinterpret_cast<T*>(lay.phalo(smem_raw + sn * sbytes)), hvP);
            dev::halo_put<L, false>(reinterpret_cast<float*>(lay.lhalo(smem_raw + sn * sbytes)), hvL);
        }
        dev::fence_proxy_async();
        __syncthreads();  // output rows complete
        {
            // lane l of warp w takes piece w + l nw: the unit's Q output slots
            // (one block), then its D updated dL/dE rows back from the stage
            // (which is refilled only after the issuing threads' reads are done)
            const int k = warp + lane * nw;
            if (k == 0) {
                dev::bulk_store(lam_out + (int64_t)u * (L::Q * rs), outrow, (uint32_t)lay.lrow());
                dev::bulk_commit();
            } else if (gE && k <= L::D) {
                const int d = k - 1;
                dev::bulk_store(gE + (int64_t)d * p.NP + (int64_t)u * rs, ge_s + d * rs, (uint32_t)rs * 4u);
                dev::bulk_commit();
            }
        }
        // link copies of lam_t: slot k of (x, b) takes lam_bbar(x)
        for (uint32_t k = g0 + threadIdx.x; k < g1; k += blockDim.x) {
            const uint32_t d = desc[k - d0];
            lamG_out[k] = outrow[desc_slot_bar(d) * rs + desc_x(d)];
        }
    }
    dev::bulk_wait_all();
    block_accumulate(acc, slots, blockIdx.x);
}

inline Launch grid_of(const KParams& p) {
    Launch l;
    const int bx = p.nx >= kBlock ? kBlock : ((p.nx + 31) / 32) * 32;
    l.block = dim3(bx);
    l.grid = dim3((unsigned)(p.ny * p.nz), (unsigned)((p.nx + bx - 1) / bx));
    return l;
}

// Blocks of the general reverse kernels.
constexpr int kAdjPerSm = 8;
inline int64_t strided_blocks(const KParams& p) {
    const Launch l = grid_of(p);
    const int64_t tiles = (int64_t)l.grid.x * l.grid.y, cap = (int64_t)sm_count() * kAdjPerSm;
    return tiles < cap ? tiles : cap;
}
// Gradient slots, and with them the most blocks of a reverse kernel.  Narrow rows
// have 12 to 21 staged blocks resident per SM.  Boxes of many units take up to 16
// (us per forward and reverse step: D2V9 FP32 64 x 16384 77.5, with eight 82.3, on
// the general kernel 97.5; D3V19 FP16 32 x 128 x 128 74.4, 88.9, 110.7); boxes whose
// blocks come round once or twice take eight (64 x 2048 27.7, with 16 30.2; at 64 x
// 4096 both 36 to 37).  The line lies between the measured 4096 and 16384 units.
inline int64_t slot_blocks(const KParams& p) {
    const Launch l = grid_of(p);
    const int64_t units = (int64_t)p.ny * p.nz * p.nseg;
    const int64_t most = std::max<int64_t>((int64_t)l.grid.x * l.grid.y, units);
    return std::min<int64_t>(most, (int64_t)sm_count() * (units > 8192 ? 2 * kAdjPerSm : kAdjPerSm));
}

// GROUP 0: D2V9 and D3V19; GROUP 1: D3V27 and D1V3 (separate translation units)
template <int GROUP, class F>
int dispatch_lattice(int vel, F&& f) {
    if constexpr (GROUP == 0 || GROUP == 2) {
        if (vel == LBM_D2V9) return f(LatD2V9{});
        return f(LatD3V19{});
    } else {
        if (vel == LBM_D1V3) return f(LatD1V3{});
        return f(LatD3V27{});
    }
}


// ---------------------------------------------------------------------------
// Launch policy of the reverse step: the row-staged kernel when the context has
// units and their stages fit the shared-memory budget; otherwise the general
// kernel.
// ---------------------------------------------------------------------------
constexpr int kAdjStages = 2;
constexpr int kAdjThreads = 256;
constexpr size_t kAdjSmemBudget = 200 * 1024;

template <class L, class S, int FORCE, bool EF, bool WIN, int RS, int MODE, bool LMU = false>
int launch_rows_rs(const void* P, const float* lam_in, float* lam_out, const uint32_t* nbr, const float* Ef,
                 const float* w_rho, const float* w_j, float* gE, double* slots, const KParams& p, cudaStream_t s) {
    if (!p.rorder || (RS && RS != p.seglen) || (MODE == kExactRow && RS != p.nx) || (MODE == kSegment) != (p.nseg > 1))
        return 0;
    const int gcapP = dev::window_cap(p.max_row_links, S::kBytes);
    const int gcapL = dev::window_cap(p.max_row_links, 4);
    const int rs = p.seglen, hP = dev::halo_bytes(L::Q, p.nseg, S::kBytes), hL = dev::halo_bytes(L::Q, p.nseg, 4);
    const int gerow = L::D * rs * 4, efrow = EF ? L::D * rs * 4 : 0;
    auto smem_for = [&](int ge) {
        return kAdjStages * (size_t)AdjLayout<L, S>{rs, p.lorder, gcapP, gcapL, ge, efrow, hP, hL}.bytes() +
               (size_t)L::Q * rs * 4;
    };
    const size_t smem = smem_for(gE ? gerow : 0);
    // the kernel choice and the persistent grid are taken for the layout with
    // dL/dE rows, whether or not this call has them, so that the blocks (and
    // with them the order of the FP64 gradient sums) are the same either way
    const size_t smem_ref = smem_for(gerow);
    if (smem_ref > kAdjSmemBudget) return 0;
    const int threads = p.seglen >= kAdjThreads ? kAdjThreads : ((p.seglen + 31) / 32) * 32;
    auto kern = k_adjoint_rows<L, S, FORCE, EF, WIN, kAdjStages, RS, MODE, LMU>;
    // persistent grid: co-resident blocks per SM x SMs
    int blocks = staged_shape((const void*)kern, p.seglen, smem_ref, kAdjSmemBudget, threads).blocks;
    const int units = p.ny * p.nz * p.nseg;
    blocks = (int)std::min<int64_t>(blocks, std::min<int64_t>(units, slot_blocks(p)));
    if (blocks <= 0) return 0;
    kern<<<blocks, threads, smem, s>>>((const typename S::T*)P, lam_in, lam_out, Ef, w_rho, w_j, gE, slots,
                                       gcapP, gcapL, p);
    return route(kStaged, MODE, RS);
}

// Rows or segments at a run-time stride.
template <class L, class S, int FORCE, bool EF, bool WIN, bool LMU = false>
int launch_rows_any(const void* P, const float* lam_in, float* lam_out, const uint32_t* nbr, const float* Ef,
                     const float* w_rho, const float* w_j, float* gE, double* slots, const KParams& p,
                     cudaStream_t s) {
    return p.nseg > 1 ? launch_rows_rs<L, S, FORCE, EF, WIN, 0, kSegment, LMU>(P, lam_in, lam_out, nbr, Ef, w_rho, w_j,
                                                                               gE, slots, p, s)
                      : launch_rows_rs<L, S, FORCE, EF, WIN, 0, kWholeRow, LMU>(P, lam_in, lam_out, nbr, Ef, w_rho,
                                                                                w_j, gE, slots, p, s);
}

// The shared-memory row stride is a compile-time constant for the usual units,
// as in the step kernel.
template <class L, class S, int FORCE, bool EF, bool WIN>
int launch_rows(const void* P, const float* lam_in, float* lam_out, const uint32_t* nbr, const float* Ef,
                 const float* w_rho, const float* w_j, float* gE, double* slots, const KParams& p,
                 cudaStream_t s) {
    // the compile-time strides only for the benchmarked lattices (D2V9, D3V19)
    constexpr bool kFixed = L::Q == 9 || L::Q == 19;
    if constexpr (kFixed) {
        constexpr int kSeg = segment_columns<L>();
        if (p.nseg > 1 && p.seglen == kSeg)
            return launch_rows_rs<L, S, FORCE, EF, WIN, kSeg, kSegment>(P, lam_in, lam_out, nbr, Ef, w_rho, w_j, gE,
                                                                        slots, p, s);
        if (p.nseg == 1 && p.nx == 256)
            return launch_rows_rs<L, S, FORCE, EF, WIN, 256, kExactRow>(P, lam_in, lam_out, nbr, Ef, w_rho, w_j, gE,
                                                                        slots, p, s);
        if constexpr (whole_row<L, S>(512)) {
            if (p.nseg == 1 && p.nx == 512)
                return launch_rows_rs<L, S, FORCE, EF, WIN, 512, kExactRow>(P, lam_in, lam_out, nbr, Ef, w_rho, w_j,
                                                                            gE, slots, p, s);
        }
    }
    return launch_rows_any<L, S, FORCE, EF, WIN>(P, lam_in, lam_out, nbr, Ef, w_rho, w_j, gE, slots, p, s);
}

// Launchers for one storage type (instantiated in one translation unit per
// storage).
template <class S, int GROUP>
int seed_storage(int vel, const void* P, const uint32_t* nbr, const float* w_rho, const float* w_j, float* lam,
                 double* slots, bool in_window, const KParams& p, cudaStream_t s) {
    Launch l = grid_of(p);
    return dispatch_lattice<GROUP>(vel, [&](auto lat) {
        using L = decltype(lat);
        k_adjoint_seed<L, S><<<(unsigned)strided_blocks(p), l.block, 0, s>>>(
            (const typename S::T*)P, nbr, w_rho, w_j, lam, slots, in_window ? 1 : 0, (int)l.grid.y, p);
        return 1;
    });
}

template <class S, int GROUP>
int step_storage(int vel, int force, bool efield, bool in_window, const void* P, const float* lam_in,
                 float* lam_out, const uint32_t* nbr, const float* Ef, const float* w_rho, const float* w_j,
                 float* gE, double* slots, const KParams& p, cudaStream_t s) {
    Launch l = grid_of(p);
    const unsigned blocks = (unsigned)strided_blocks(p);
    return dispatch_lattice<GROUP>(vel, [&](auto lat) {
        using L = decltype(lat);
        const auto* Pt = (const typename S::T*)P;
        int done = route(kGeneral);
// GROUP 2: the local-mu model (D2V9, D3V19), whose staged reverse kernel is
// an instantiation of its own with the run-time row stride
#define LBM_ADJ(F, EFV, W)                                                                                    \
    do {                                                                                                      \
        int staged;                                                                                           \
        if constexpr (GROUP == 2)                                                                             \
            staged = launch_rows_any<L, S, F, EFV, W, true>(P, lam_in, lam_out, nbr, Ef, w_rho, w_j, gE,      \
                                                            slots, p, s);                                     \
        else                                                                                                  \
            staged = launch_rows<L, S, F, EFV, W>(P, lam_in, lam_out, nbr, Ef, w_rho, w_j, gE, slots, p, s);  \
        if (staged)                                                                                           \
            done = staged;                                                                                    \
        else                                                                                                  \
            k_adjoint_step<L, S, F, EFV, W>                                                                   \
                <<<blocks, l.block, 0, s>>>(Pt, lam_in, lam_out, nbr, Ef, w_rho, w_j, gE, slots,              \
                                            (int)l.grid.y, p);                                                \
    } while (0)
        if (force == LBM_FORCE_SHIFT) {
            if (efield) {
                if (in_window) LBM_ADJ(0, true, true); else LBM_ADJ(0, true, false);
            } else {
                if (in_window) LBM_ADJ(0, false, true); else LBM_ADJ(0, false, false);
            }
        } else {
            if (efield) {
                if (in_window) LBM_ADJ(1, true, true); else LBM_ADJ(1, true, false);
            } else {
                if (in_window) LBM_ADJ(1, false, true); else LBM_ADJ(1, false, false);
            }
        }
#undef LBM_ADJ
        return done;
    });
}

}  // namespace adjk
}  // namespace lbm
