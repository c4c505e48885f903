// Many steps of a small box in one launch (templates; included by one
// translation unit per storage type).
//
// A step of a small box is over before the host has launched the next one: 100
// steps of 32 x 64 cells of D2V9 FP32 took 4.14 us each, 100 of 4096 x 8 in
// BF16 the same, whatever the kernel (the host was the limit).  Here one cluster of up to 16 blocks
// keeps the whole box in its shared memory and steps through all n steps by
// itself: every thread collides its cells and writes each post-collision value
// straight into the slot that the destination cell pulls next (distributed
// shared memory; into its own slot of the opposite direction where a solid cell
// is behind the link), then the cluster barrier ends the step.  The state
// comes from global memory before the first step and goes back, in the layout
// of the other kernels, with the last one.
//
// What bounds it: the serial chain of a collision (about 0.6 us) plus the
// barrier while a block has a warp or two per scheduler, the issue slots of 16
// SMs beyond that: 0.9 us a step at 32 x 64 (D2V9 FP32); 4.0 us at 4096 x 8 (D2V9
// BF16), measured without the limit that follows, which sends that box elsewhere.
//
// Beyond kClusterWork populations (where 16 SMs take as long as the other
// kernel's barrier costs) a cooperative grid with a thread for every cell does
// the same through global memory (k_step_grid): the two state buffers hold the
// values as they are pulled, [a N + cell], until the last step, and a barrier
// over the grid ends a step.  Boxes of more cells than threads that are
// resident at once are stepped one launch at a time: their steps outlast a
// launch.
// The arithmetic, its order and the rounding stream are those of k_step, so the
// results have the same bits.
#pragma once

#include "lbm_step.cuh"

namespace lbm {
namespace multik {

using dev::Cell;

constexpr int kClusterMax = 16;  // the non-portable limit
constexpr size_t kSmemMax = 128 * 1024;  // of a block of the cluster (see kClusterWork)
constexpr uint32_t kNoCell = 0xFFFFFFFFu;

// Populations up to which the cluster is the faster of the two.  Its step grows
// with the box (0.87 us at 2048 cells of D2V9; 3.97 us at 32768, without this
// limit), the grid's hardly does (2.36 us at 32768): they meet near 16384 cells.
// 16 blocks then need 120 KB of shared memory each at most.
constexpr int64_t kClusterWork = 16384 * 9;
// Threads per block: the FP32 collision of the larger lattices needs more than
// 64 registers.  The grid has one block per SM.
template <class L>
constexpr int kThreads = L::Q <= 9 ? 1024 : 512;
template <class L>
constexpr int kGridThreads = L::Q <= 9 ? 1024 : 640;

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(r));
    return r;
}
// address of this block's shared address `a` in the block of rank r
__device__ __forceinline__ uint32_t map_rank(uint32_t a, uint32_t r) {
    uint32_t d;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(d) : "r"(a), "r"(r));
    return d;
}
__device__ __forceinline__ void cluster_store(uint32_t a, float v) {
    asm volatile("st.shared::cluster.f32 [%0], %1;\n" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void cluster_store(uint32_t a, __half v) {
    asm volatile("st.shared::cluster.u16 [%0], %1;\n" ::"r"(a), "h"(__half_as_ushort(v)) : "memory");
}
__device__ __forceinline__ void cluster_store(uint32_t a, __nv_bfloat16 v) {
    asm volatile("st.shared::cluster.u16 [%0], %1;\n" ::"r"(a), "h"(__bfloat16_as_ushort(v)) : "memory");
}
// all blocks' shared-memory writes before it are visible to all after it
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;\n" ::: "memory");
}

// Block r of the cluster owns the cells r cpc .. r cpc + cpc - 1.  Shared
// memory: two states h~_a at [a * cpc + i], and the destination of each value
// as a cluster address into the second state (direction 0: the cell's place in
// the padded field, or kNoCell for a solid cell).  Ef: the per-cell field, or null.
// Pin and Pout may be the same buffer: every block has pulled its cells from it
// before the first barrier, and none writes to it before the last step (n > 1).
template <class L, class S, int FORCE, bool SR>
__global__ void __launch_bounds__(kThreads<L>) k_step_multi(const typename S::T* Pin, typename S::T* Pout,
                                                            const uint32_t* __restrict__ nbr,
                                                            const float* __restrict__ Ef, int n, int cpc, KParams p) {
    using T = typename S::T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    uint32_t* dst = reinterpret_cast<uint32_t*>(smem_raw);
    T* state = reinterpret_cast<T*>(smem_raw + (size_t)L::Q * cpc * 4);
    const int half = L::Q * cpc;  // elements of one state
    const uint32_t rank = cluster_rank();
    const int64_t first = (int64_t)rank * cpc;
    const int mine = (int)(p.N - first < cpc ? (p.N > first ? p.N - first : 0) : cpc);
    for (int i = threadIdx.x; i < mine; i += blockDim.x) {
        const uint32_t cell = (uint32_t)first + (uint32_t)i;
        const int row = (int)(cell / (uint32_t)p.nx);
        Cell c;
        dev::cell_at(p, row, (int)(cell - (uint32_t)row * (uint32_t)p.nx), c);
        const uint32_t m = __ldg(nbr + cell);
        dst[i] = (m & kSolidBit) ? kNoCell : (uint32_t)c.pcell;
        if (m & kSolidBit) continue;
        float h[L::Q];
        dev::pull<L, S>(Pin, p, m, c, h);
#pragma unroll
        for (int a = 0; a < L::Q; ++a) {
            S::put(state + a * cpc + i, h[a]);  // the stored value itself: it came from this format
            if (a == 0) continue;
            const bool wall = (m >> opposite(a)) & 1u;  // x + e_a is solid
            const uint32_t to = wall ? cell : dev::shifted<L>(p, c, a, +1);
            const uint32_t r = to / (uint32_t)cpc;
            const T* at = state + half + (wall ? opposite(a) : a) * cpc + (int)(to - r * (uint32_t)cpc);
            dst[a * cpc + i] = map_rank(dev::smem_u32(at), r);
        }
    }
    cluster_barrier();
    const uint32_t back = (uint32_t)(half * (int)sizeof(T));
    for (int t = 0; t < n; ++t) {
        const bool last = t == n - 1;
        const T* in = state + (t & 1) * half;
        T* own = state + ((t & 1) ^ 1) * half;
        const uint32_t to = (t & 1) ? back : 0u;  // odd steps write the first state
        const uint32_t key = step_key(p.step + (uint32_t)t, p.seed);
        for (int i = threadIdx.x; i < mine; i += blockDim.x) {
            const uint32_t place = dst[i];
            const uint32_t cell = (uint32_t)first + (uint32_t)i;
            T v[L::Q];
            if (place != kNoCell) {
                float h[L::Q], E[3], out[L::Q];
#pragma unroll
                for (int a = 0; a < L::Q; ++a) h[a] = S::cvt(in[a * cpc + i]);
                stepk::load_E<L>(Ef, Ef != nullptr, p, place, E);
                constexpr bool kLmu = L::Q == 9 || L::Q == 19;
                if (kLmu && p.lmu_tab)
                    stepk::collide_any<L, S, FORCE, kLmu>(h, E, p, out);
                else
                    stepk::collide_any<L, S, FORCE>(h, E, p, out);
                stepk::round_all<L, S, SR>(out, cell, key, v);
                if (!last) {
                    own[i] = v[0];
#pragma unroll
                    for (int a = 1; a < L::Q; ++a) cluster_store(dst[a * cpc + i] - to, v[a]);
                }
            }
            if (last) {
                const int row = (int)(cell / (uint32_t)p.nx);
                Cell c;
                dev::cell_at(p, row, (int)(cell - (uint32_t)row * (uint32_t)p.nx), c);
                if (place == kNoCell) {
#pragma unroll
                    for (int a = 0; a < L::Q; ++a) S::put(Pout + dev::pop_at<L>(p, c, a, 0), 0.f);
                } else {
                    stepk::store_cell<L, S>(Pout, p, __ldg(nbr + cell), c, v);
                }
            }
        }
        if (!last) cluster_barrier();
    }
}

// Barrier over a cooperative grid: `count` grows by one per block and step.  A
// wait that runs out writes code 4 into the status word; the block then waits no
// more, and the kernel ends with invalid results (the places of its values come
// from the geometry, not from other blocks' data, and stay inside its buffers).
__device__ __forceinline__ bool grid_barrier(unsigned* count, unsigned target, bool ok, uint32_t limit, int* status) {
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;\n" ::"l"(count) : "memory");
        if (ok) {
            // counted against a constant from an earlier start: with the limit itself in
            // the comparison a step of 28 x 40 x 21 D3V19 BF16 took 2.80 us, 2.64 so
            const long long t0 = clock64() - (kWaitClocks - (long long)limit);
            for (;;) {
                unsigned v;
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(v) : "l"(count) : "memory");
                if (v >= target) break;
                if (clock64() - t0 > kWaitClocks) {
                    ok = false;
                    if (status) atomicExch(status, 4);
                    break;
                }
            }
        }
    }
    return __syncthreads_and(threadIdx.x != 0 || ok) != 0;
}

__device__ __forceinline__ float load_l2(const float* q) { return __ldcg(q); }
__device__ __forceinline__ __half load_l2(const __half* q) {
    return __ushort_as_half(__ldcg(reinterpret_cast<const unsigned short*>(q)));
}
__device__ __forceinline__ __nv_bfloat16 load_l2(const __nv_bfloat16* q) {
    return __ushort_as_bfloat16(__ldcg(reinterpret_cast<const unsigned short*>(q)));
}

// n steps with one thread per cell, all blocks resident (cooperative launch).
// Step t reads buf[t & 1] and writes the other; dst (shared memory, [a][thread])
// holds the element that each value goes to.  The loads bypass L1, which other
// blocks' stores do not reach.
template <class L, class S, int FORCE, bool SR>
__global__ void __launch_bounds__(kGridThreads<L>) k_step_grid(typename S::T* A, typename S::T* B,
                                                               const uint32_t* __restrict__ nbr,
                                                               const float* __restrict__ Ef, int n, unsigned* count,
                                                               KParams p) {
    using T = typename S::T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    uint32_t* dst = reinterpret_cast<uint32_t*>(smem_raw) + threadIdx.x;
    const int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool in_box = id < p.N;
    const uint32_t cell = in_box ? (uint32_t)id : 0u, N = (uint32_t)p.N;
    const int row = (int)(cell / (uint32_t)p.nx);
    Cell c;
    dev::cell_at(p, row, (int)(cell - (uint32_t)row * (uint32_t)p.nx), c);
    const uint32_t m = __ldg(nbr + cell);
    const bool fluid = in_box && !(m & kSolidBit);
#pragma unroll
    for (int a = 1; a < L::Q; ++a) {
        const bool wall = (m >> opposite(a)) & 1u;  // x + e_a is solid
        dst[(a - 1) * (int)blockDim.x] = wall ? (uint32_t)opposite(a) * N + cell
                                              : (uint32_t)a * N + dev::shifted<L>(p, c, a, +1);
    }
    float h[L::Q];
    if (fluid) dev::pull<L, S>(A, p, m, c, h);  // no block writes A before the first barrier
    bool ok = true;
    const unsigned missing = p.staged < p.ny * p.nz * p.nseg;  // lbm_selftest_withhold: a block that never arrives
    for (int t = 0; t < n; ++t) {
        const T* from = (t & 1) ? B : A;
        T* to = (t & 1) ? A : B;
        if (t > 0) {
            ok = grid_barrier(count, (unsigned)t * gridDim.x + missing, ok, p.wait_clocks, p.status);
            if (fluid) {
#pragma unroll
                for (int a = 0; a < L::Q; ++a) h[a] = S::cvt(load_l2(from + ((uint32_t)a * N + cell)));
            }
        }
        const bool last = t == n - 1;
        if (fluid) {
            float E[3], out[L::Q];
            T v[L::Q];
            stepk::load_E<L>(Ef, Ef != nullptr, p, c.pcell, E);
            constexpr bool kLmu = L::Q == 9 || L::Q == 19;
            if (kLmu && p.lmu_tab)
                stepk::collide_any<L, S, FORCE, kLmu>(h, E, p, out);
            else
                stepk::collide_any<L, S, FORCE>(h, E, p, out);
            stepk::round_all<L, S, SR>(out, cell, step_key(p.step + (uint32_t)t, p.seed), v);
            if (last) {
                stepk::store_cell<L, S>(to, p, m, c, v);
            } else {
                to[cell] = v[0];
#pragma unroll
                for (int a = 1; a < L::Q; ++a) to[dst[(a - 1) * (int)blockDim.x]] = v[a];
            }
        } else if (last && in_box) {
#pragma unroll
            for (int a = 0; a < L::Q; ++a) S::put(to + dev::pop_at<L>(p, c, a, 0), 0.f);
        }
    }
}

// Blocks of the cluster and shared memory of a box, or 0 blocks where it does
// not fit: the smallest power of two of blocks that leaves at most 128 cells
// each (one warp per scheduler), up to 16.
struct Plan {
    int blocks, cpc;
    size_t smem;
};
template <class L, class S>
Plan plan_of(const KParams& p) {
    int blocks = 1;
    while (blocks < kClusterMax && p.N > (int64_t)blocks * 128) blocks *= 2;
    const int64_t cpc = ((p.N + blocks - 1) / blocks + 31) / 32 * 32;
    const size_t smem = (size_t)L::Q * (size_t)cpc * (2 * S::kBytes + 4);
    if (p.N * L::Q > kClusterWork) return {0, 0, 0};
    return {blocks, (int)cpc, smem};
}

// 1 for a launch that went out; the error of one that did not is cleared, since
// the steps are then launched one by one.
inline int launched(cudaError_t e) {
    if (e == cudaSuccess) return 1;
    cudaGetLastError();
    return 0;
}

// Launches n steps, or returns 0: a box that does not fit, or a device on which
// the cluster cannot be placed.  The result is in fin when n is even.
template <class L, class S, int FORCE, bool SR>
int launch_cluster(void* fin, void* fout, const uint32_t* nbr, const float* Ef, int n, const KParams& p,
               cudaStream_t s) {
    using T = typename S::T;
    const Plan plan = plan_of<L, S>(p);
    if (plan.blocks == 0) return 0;
    auto kern = k_step_multi<L, S, FORCE, SR>;
    int threads = plan.cpc < kThreads<L> ? plan.cpc : kThreads<L>;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim = {(unsigned)plan.blocks, 1, 1};
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)plan.blocks);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = plan.smem;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    // whether the device can place this cluster
    const int n_shape = plan.blocks * 4096 + threads;
    Shape sh;
    if (!known_shape((const void*)kern, n_shape, plan.smem, &sh)) {
        int clusters = 0;
        if (!allow_smem((const void*)kern, kSmemMax) ||
            cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
            cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg) != cudaSuccess)
            cudaGetLastError();
        sh = Shape{threads, clusters * plan.blocks, 0};
        keep_shape((const void*)kern, n_shape, plan.smem, sh);
    }
    if (sh.blocks <= 0) return 0;
    return launched(cudaLaunchKernelEx(&cfg, kern, (const T*)fin, (T*)(n % 2 ? fout : fin), nbr, Ef, n, plan.cpc, p))
               ? route(kCluster)
               : 0;
}

// The same for the cooperative grid.
template <class L, class S, int FORCE, bool SR>
int launch_grid(void* fin, void* fout, const uint32_t* nbr, const float* Ef, int n, unsigned* count, const KParams& p,
                cudaStream_t s) {
    using T = typename S::T;
    auto kern = k_step_grid<L, S, FORCE, SR>;
    const int sms = sm_count();
    const int64_t per = ((p.N + sms - 1) / sms + 31) / 32 * 32;
    if (per > kGridThreads<L>) return 0;
    const int threads = (int)per;
    const size_t smem = (size_t)(L::Q - 1) * threads * 4;
    Shape sh;
    if (!known_shape((const void*)kern, threads, smem, &sh)) {
        int dev = 0, coop = 0, per_sm = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
        if (!coop || !allow_smem((const void*)kern, (size_t)(L::Q - 1) * kGridThreads<L> * 4) ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem) != cudaSuccess)
            cudaGetLastError();
        sh = Shape{threads, per_sm * sms, sms};
        keep_shape((const void*)kern, threads, smem, sh);
    }
    const unsigned blocks = (unsigned)((p.N + threads - 1) / threads);
    if ((int64_t)blocks > sh.blocks) return 0;
    if (!launched(cudaMemsetAsync(count, 0, sizeof(unsigned), s))) return 0;
    T *A = (T*)fin, *B = (T*)fout;
    KParams q = p;
    void* args[] = {&A, &B, &nbr, &Ef, &n, &count, &q};
    return launched(cudaLaunchCooperativeKernel(kern, dim3(blocks), dim3((unsigned)threads), args, smem, s))
               ? route(kGrid)
               : 0;
}

template <class L, class S, int FORCE, bool SR>
int launch_one(void* fin, void* fout, const uint32_t* nbr, const float* Ef, int n, unsigned* count, bool* in_fin,
               const KParams& p, cudaStream_t s) {
    // as after n single steps, which a captured call is replayed as
    *in_fin = n % 2 == 0;
    if (int k = launch_cluster<L, S, FORCE, SR>(fin, fout, nbr, Ef, n, p, s)) return k;
    if (p.N * L::Q <= kClusterWork) return 0;
    return launch_grid<L, S, FORCE, SR>(fin, fout, nbr, Ef, n, count, p, s);
}

template <class S, bool HAS_SR>
int launch_storage(int vel, int force, bool sr, void* fin, void* fout, const uint32_t* nbr, const float* Ef, int n,
                   unsigned* count, bool* in_fin, const KParams& p, cudaStream_t s) {
    auto with = [&](auto lat) {
        using L = decltype(lat);
        auto go = [&](auto srt) {
            constexpr bool SR = decltype(srt)::value;
            return force == LBM_FORCE_SHIFT ? launch_one<L, S, 0, SR>(fin, fout, nbr, Ef, n, count, in_fin, p, s)
                                            : launch_one<L, S, 1, SR>(fin, fout, nbr, Ef, n, count, in_fin, p, s);
        };
        if constexpr (HAS_SR) {
            if (sr) return go(std::true_type{});
        }
        return go(std::false_type{});
    };
    if (vel == LBM_D2V9) return with(LatD2V9{});
    if (vel == LBM_D3V27) return with(LatD3V27{});
    if (vel == LBM_D1V3) return with(LatD1V3{});
    return with(LatD3V19{});
}

}  // namespace multik
}  // namespace lbm
