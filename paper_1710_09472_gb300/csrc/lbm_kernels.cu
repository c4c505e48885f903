// Device kernels of the semiclassical LBM step (Sec. 9.1 of arXiv 1710.09472):
// link mask, equilibrium start state, the fused pull-stream + BGK collision +
// Lorentz forcing step, moments with FP64 reductions, and the population
// read-back.
//
// Layout: a row (or segment of a long row) keeps its directions one after
// another (see pop_slot).  P holds post-collision values ("pull"
// scheme): the state f(x, t) of the method is f_a(x, t) = P_a(x - e_a) when
// x - e_a is fluid.
// Halfway bounce-back (Sec. 9.3, 9.4) uses a link buffer G stored after P in
// the same state buffer: every link from a fluid cell x into a solid cell
// (x + e_b solid) owns one slot, numbered in cell order (lbase[x] + rank of b
// among x's outgoing links), so the links of one row form a contiguous range
// rowG[u] .. rowG[u+1] (u a row, or a segment of a long row).  The collision stores f*_b(x) there, and the next
// step reads it back as f_bbar(x).
#include <algorithm>
#include <atomic>
#include <cstdio>
#include <map>
#include <mutex>
#include <new>
#include <tuple>

#include <cub/device/device_scan.cuh>

#include "lbm_step.cuh"

namespace lbm {
namespace {

using dev::Cell;
using dev::kBlock;

// ---------------------------------------------------------------------------
// Link mask: bit a set when x - e_a is solid (the link streaming into x along
// e_a bounces back); kSolidBit when x is solid.
// ---------------------------------------------------------------------------
template <class L>
__global__ void __launch_bounds__(kBlock) k_neighbors(const uint8_t* __restrict__ mask, uint32_t* __restrict__ nbr,
                                                      unsigned long long* __restrict__ fluid_count, KParams p) {
    Cell c;
    unsigned fluid = 0;
    if (dev::cell_of_thread(p, c)) {
        uint32_t m = 0;
        if (mask[c.cell]) {
            m = kSolidBit;
        } else {
            fluid = 1;
#pragma unroll
            for (int a = 1; a < L::Q; ++a)
                if (mask[dev::shifted<L>(p, c, a, -1)]) m |= (1u << a);
        }
        nbr[c.cell] = m;
    }
    const unsigned cnt = __popc(__ballot_sync(0xffffffffu, fluid));
    if ((threadIdx.x & 31) == 0 && cnt) atomicAdd(fluid_count, (unsigned long long)cnt);
}

// ---------------------------------------------------------------------------
// Start state f(x, 0) = f^eq(rho(x), u(x)) for the pull with read-side
// bounce-back: slot P_b(y) of a fluid cell y is pulled by y + e_b when that
// cell is fluid (value f^eq_b(y + e_b)), and by y itself as its bounced
// population bbar when y + e_b is solid (value f^eq_bbar(y)); solid cells'
// slots are never read and hold 0.
// ---------------------------------------------------------------------------
template <class L>
__device__ __forceinline__ float heq_unscaled(const KParams& p, int a, float rho, const float* u) {
    const float eu = dev::edot<L>(a, u);
    const float u2 = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
    return p.w[a] * (p.A * (rho - p.rho0) + rho * (p.Bp * eu + p.Cp * eu * eu + p.k2[a] * u2));
}

template <class L, class S>
__global__ void __launch_bounds__(kBlock) k_init(typename S::T* __restrict__ P, const uint32_t* __restrict__ nbr,
                                                 const float* __restrict__ rho, const float* __restrict__ u,
                                                 KParams p) {
    Cell c;
    if (!dev::cell_of_thread(p, c)) return;
    const uint32_t m = nbr[c.cell];
    typename S::T* G = reinterpret_cast<typename S::T*>(reinterpret_cast<char*>(P) + p.gofs);
    auto fields = [&](uint32_t cell, float& r, float* uu) {
        r = rho ? rho[cell] : p.rho0;
        uu[0] = u ? u[cell] : 0.f;
        uu[1] = (u && L::D >= 2) ? u[p.N + cell] : 0.f;
        uu[2] = (u && L::D == 3) ? u[2 * p.N + cell] : 0.f;
    };
    float r0, u0[3];
    fields(c.cell, r0, u0);
    const bool fluid = !(m & kSolidBit);
    const uint32_t o = fluid ? outgoing<L::Q>(m) : 0u;
    const uint32_t base = (fluid && o) ? p.lbase[c.cell] : 0u;
#pragma unroll
    for (int b = 0; b < L::Q; ++b) {
        float v = 0.f;
        if (fluid) {
            if (b != 0 && ((o >> b) & 1u)) {
                // link into a solid cell: next pull of bbar at this cell reads f^eq_bbar here
                S::put(G + link_slot(base, o, b), heq_unscaled<L>(p, opposite(b), r0, u0) * p.scale);
            } else {
                float r1 = r0, u1[3] = {u0[0], u0[1], u0[2]};
                if (b != 0) fields(dev::shifted<L>(p, c, b, +1), r1, u1);
                v = heq_unscaled<L>(p, b, r1, u1);
            }
        }
        S::put(P + dev::pop_at<L>(p, c, b, 0), v * p.scale);
    }
}

// Link layout: count outgoing links per fluid cell, exclusive scan, row starts.
template <class L>
__global__ void __launch_bounds__(kBlock) k_link_counts(const uint32_t* __restrict__ nbr, uint32_t* __restrict__ cnt,
                                                        KParams p) {
    Cell c;
    if (!dev::cell_of_thread(p, c)) return;
    const uint32_t m = nbr[c.cell];
    cnt[c.cell] = (m & kSolidBit) ? 0u : (uint32_t)__popc(outgoing<L::Q>(m));
}

// Descriptor of every link slot (link_desc): the slots of its outgoing
// direction b and of bbar, the unit column of its fluid cell and the staged
// position of the solid cell behind the link.
template <class L>
__global__ void __launch_bounds__(kBlock) k_link_desc(const uint32_t* __restrict__ nbr,
                                                      const uint32_t* __restrict__ lbase,
                                                      uint32_t* __restrict__ ldesc, KParams p) {
    Cell c;
    if (!dev::cell_of_thread(p, c)) return;
    const uint32_t m = nbr[c.cell];
    if ((m & kSolidBit) || m == 0u) return;
    const uint32_t o = outgoing<L::Q>(m);
    const uint32_t base = lbase[c.cell];
    const int xl = c.x % p.seglen, last = min(p.seglen, p.nx - (c.x - xl)) - 1;
    const int left = xl > 0 ? xl - 1 : (p.nseg == 1 ? p.nx - 1 : kPosLeft);
    const int right = xl < last ? xl + 1 : (p.nseg == 1 ? 0 : kPosRight);
#pragma unroll
    for (int b = 1; b < L::Q; ++b)
        if ((o >> b) & 1u) {
            const int ex = L::c(b, 0);
            ldesc[link_slot(base, o, b)] =
                link_desc(pop_slot<L>(b), pop_slot<L>(opposite(b)), xl, ex < 0 ? left : (ex > 0 ? right : xl));
        }
}

// Cell order of each unit for the row-staged kernels: entry 0 the number of
// fluid cells nf, entries 1..7 zero, entries 8 .. 8 + nf - 1 the fluid x
// ascending, then the solid x ascending, then zeros up to lorder; x counts
// from the unit's first cell.  One warp per unit.
__global__ void __launch_bounds__(kBlock) k_row_order(const uint32_t* __restrict__ nbr, uint16_t* __restrict__ ord,
                                                      KParams p) {
    const int64_t U = (int64_t)p.ny * p.nz * p.nseg;
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < U; r += nwarps) {
        const int first = (int)(r % p.nseg) * p.seglen;
        const int len = min(p.seglen, p.nx - first);
        const uint32_t* m = nbr + (r / p.nseg) * p.nx + first;
        uint16_t* o = ord + r * p.lorder;
        int nf = 0;
        for (int x0 = 0; x0 < len; x0 += 32) {
            const int x = x0 + lane;
            nf += __popc(__ballot_sync(0xffffffffu, x < len && !(m[x] & kSolidBit)));
        }
        int nfl = 0, nso = nf;  // entries written so far: fluid, and nf + solid
        for (int x0 = 0; x0 < len; x0 += 32) {
            const int x = x0 + lane;
            const bool in = x < len;
            const bool fluid = in && !(m[x] & kSolidBit);
            const unsigned bf = __ballot_sync(0xffffffffu, fluid), bs = __ballot_sync(0xffffffffu, in && !fluid);
            if (fluid) o[8 + nfl + __popc(bf & below)] = (uint16_t)x;
            if (in && !fluid) o[8 + nso + __popc(bs & below)] = (uint16_t)x;
            nfl += __popc(bf);
            nso += __popc(bs);
        }
        if (lane < 8) o[lane] = lane == 0 ? (uint16_t)nf : (uint16_t)0;
        for (int k = 8 + len + lane; k < p.lorder; k += 32) o[k] = 0;
    }
}

template <class L>
__global__ void k_row_starts(const uint32_t* __restrict__ nbr, const uint32_t* __restrict__ lbase,
                             uint32_t* __restrict__ rowG, KParams p) {
    const int64_t U = (int64_t)p.ny * p.nz * p.nseg;
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r <= U; r += (int64_t)gridDim.x * blockDim.x) {
        if (r < U) {
            rowG[r] = lbase[(r / p.nseg) * p.nx + (r % p.nseg) * p.seglen];
        } else {
            const uint32_t m = nbr[p.N - 1];
            rowG[U] = lbase[p.N - 1] + ((m & kSolidBit) ? 0u : (uint32_t)__popc(outgoing<L::Q>(m)));
        }
    }
}

// ---------------------------------------------------------------------------
// Moments of f(x, t) and FP64 block partials of the fluid totals
// partials[block] = {sum rho, sum j_x, sum j_y, sum j_z}.
// ---------------------------------------------------------------------------
template <class L>
__device__ __forceinline__ void cell_moments(const float* h, const KParams& p, float& rho, float* j) {
    float drho = 0.f, jj[3] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int a = 0; a < L::Q; ++a) {
        drho += h[a];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            if (L::c(a, d) > 0) jj[d] += h[a];
            if (L::c(a, d) < 0) jj[d] -= h[a];
        }
    }
    rho = p.rho0 + drho * p.inv_scale;
    const float k = p.inv_scale * p.cs_inv;
    j[0] = jj[0] * k;
    j[1] = jj[1] * k;
    j[2] = (L::D == 3) ? jj[2] * k : 0.f;
}

template <class L, class S, bool TOTALS>
__global__ void __launch_bounds__(kBlock) k_moments(const typename S::T* __restrict__ P, const uint32_t* __restrict__ nbr,
                                                    float* __restrict__ rho_out, float* __restrict__ j_out,
                                                    double* __restrict__ partials, int chunks, KParams p) {
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    // tile t: chunk t % chunks of row t / chunks; the grid has a block for
    // every tile (fields only) or strides over them (totals)
    const int64_t tiles = (int64_t)p.ny * p.nz * chunks;
    for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
        Cell c;
        if (dev::cell_at(p, (int)(t / chunks), (int)(t % chunks) * blockDim.x + threadIdx.x, c)) {
            const uint32_t m = __ldg(nbr + c.cell);
            float r = 0.f, j[3] = {0.f, 0.f, 0.f};
            if (!(m & kSolidBit)) {
                float h[L::Q];
                dev::pull<L, S>(P, p, m, c, h);
                cell_moments<L>(h, p, r, j);
                if (TOTALS) {
                    acc[0] += (double)r;
                    acc[1] += (double)j[0];
                    if (L::D >= 2) acc[2] += (double)j[1];
                    if (L::D == 3) acc[3] += (double)j[2];
                }
            }
            if (rho_out) rho_out[c.cell] = r;
            if (j_out) {
#pragma unroll
                for (int d = 0; d < L::D; ++d) j_out[(int64_t)d * p.N + c.cell] = j[d];
            }
        }
        if (!TOTALS) return;
    }
    if (TOTALS) {
        __shared__ double sh[kBlock / 32][4];
        const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[k] = dev::warp_sum(acc[k]);
        if (lane == 0) {
#pragma unroll
            for (int k = 0; k < 4; ++k) sh[wid][k] = acc[k];
        }
        __syncthreads();
        if (wid == 0) {
            const int nw = (blockDim.x + 31) / 32;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                double v = lane < nw ? sh[lane][k] : 0.0;
                v = dev::warp_sum(v);
                if (lane == 0) partials[(int64_t)blockIdx.x * 4 + k] = v;
            }
        }
    }
}

// The same over units staged in shared memory (the step kernel's stages, links
// and cell order; no outputs to stage, so one barrier per unit and twice the
// blocks per SM).  The general kernel spends 370 instructions a cell on
// addresses and links: 0.24 ms on 256^3 porous D3V19 FP16 (0.135 the floor),
// against 0.15 staged.
template <class L, class S, bool TOTALS, int MODE>
__global__ void __launch_bounds__(256) k_moments_rows(const typename S::T* __restrict__ P, float* __restrict__ rho_out,
                                                      float* __restrict__ j_out, double* __restrict__ partials,
                                                      int gcap, int dcap, KParams p) {
    using T = typename S::T;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int rs = p.seglen, U = p.ny * p.nz * p.nseg, G = gridDim.x;
    constexpr bool halo = MODE == kSegment;
    const stepk::StageLayout<L, S> lay{rs, p.lorder, gcap, dcap, dev::halo_bytes(L::Q, p.nseg, S::kBytes)};
    const int sbytes = lay.bytes();
    __shared__ __align__(8) uint64_t bar[2];
    __shared__ uint32_t gstart[2], dstart[2];
    const bool issuer = (int)threadIdx.x == (int)blockDim.x - 32;
    auto stage = [&](int k, int unit) {
        stepk::stage_unit<L, S, 0, MODE>(smem_raw + k * sbytes, lay, &bar[k], P, unit, __ldg(p.rowG + unit),
                                   __ldg(p.rowG + unit + 1), &gstart[k], &dstart[k], p);
    };
    if (threadIdx.x == 0) {
        dev::mbar_init(&bar[0], 1);
        dev::mbar_init(&bar[1], 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (halo && dev::halo_thread<L>())
        dev::halo_put<L, true>(lay.halo(smem_raw), dev::halo_fetch<L, true>(P, dev::unit_at<0, MODE>(p, blockIdx.x), p));
    __syncthreads();
    if (issuer && (int)blockIdx.x < p.staged) stage(0, blockIdx.x);
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    bool ok = true;
    int it = 0;
    for (int u = blockIdx.x; u < U; u += G, ++it) {
        const int cs = it & 1, un = u + G;
        unsigned char* st = smem_raw + cs * sbytes;
        const uint32_t g0 = __ldg(p.rowG + u);
        uint32_t g1 = __ldg(p.rowG + u + 1);
        ok = dev::stage_wait(&bar[cs], (uint32_t)(it >> 1) & 1u, ok, 5, g0, g1, lay.order(st), p);
        T* buf = lay.rows(st);
        dev::patch_links<true, halo>(buf, rs, lay.halo(st), L::Q, lay.links(st), gstart[cs], g0, g1, lay.descs(st),
                                     dstart[cs]);
        dev::fence_proxy_async();  // this stage is overwritten by copies after the next barrier
        // bounced values in place; every thread is past its reads of the other stage
        ok = __syncthreads_and(ok) != 0;
        if (issuer && ok && un < U) stage(cs ^ 1, un);
        const bool fetch = halo && un < U && dev::halo_thread<L>();
        T hv{};
        if (fetch) hv = dev::halo_fetch<L, true>(P, dev::unit_at<0, MODE>(p, un), p);
        const uint16_t* ord = lay.order(st);
        const int nf = ord[0];
        const dev::UnitAt at = dev::unit_at<0, MODE>(p, u);
        const int64_t first = (int64_t)at.row * p.nx + at.x0;
        for (int i = threadIdx.x; i < at.len; i += blockDim.x) {
            const int x = (int)ord[8 + i];
            float r = 0.f, j[3] = {0.f, 0.f, 0.f};
            if (i < nf) {
                // columns x - 1 and x + 1, as in the step kernel
                const T* bm = buf + (x == 0 ? at.len - 1 : x - 1);
                const T* bp = buf + (x == at.len - 1 ? 0 : x + 1);
                int rm = rs, rp = rs;
                if (halo && x == 0) {
                    bm = lay.halo(st);
                    rm = 1;
                }
                if (halo && x == at.len - 1) {
                    bp = lay.halo(st) + L::Q;
                    rp = 1;
                }
                float h[L::Q];
#pragma unroll
                for (int a = 0; a < L::Q; ++a) {
                    const int ex = L::c(a, 0), s = pop_slot<L>(a);
                    h[a] = S::cvt(ex > 0 ? bm[s * (halo ? rm : rs)] : (ex < 0 ? bp[s * (halo ? rp : rs)] : buf[s * rs + x]));
                }
                cell_moments<L>(h, p, r, j);
                if (TOTALS) {
                    acc[0] += (double)r;
                    acc[1] += (double)j[0];
                    if (L::D >= 2) acc[2] += (double)j[1];
                    if (L::D == 3) acc[3] += (double)j[2];
                }
            }
            if (rho_out) rho_out[first + x] = r;
            if (j_out) {
#pragma unroll
                for (int d = 0; d < L::D; ++d) j_out[(int64_t)d * p.N + first + x] = j[d];
            }
        }
        if (halo) {  // the halo values of the next unit, before its link pass
            if (fetch) dev::halo_put<L, true>(lay.halo(smem_raw + (cs ^ 1) * sbytes), hv);
            __syncthreads();
        }
    }
    if (TOTALS) {
        __shared__ double sh[256 / 32][4];
        const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) / 32;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            acc[k] = dev::warp_sum(acc[k]);
            if (lane == 0) sh[wid][k] = acc[k];
        }
        __syncthreads();
        if (threadIdx.x < 4) {
            double v = 0.0;
            for (int w = 0; w < nw; ++w) v += sh[w][threadIdx.x];
            partials[(int64_t)blockIdx.x * 4 + threadIdx.x] = v;
        }
    }
}

// Launches it where the context has units, two stages fit the step kernel's
// budget and there are units for every SM (staged / general, us: D2V9 BF16 4096 x
// 8, 64 units, 2.69 / 2.02; D3V19 FP16 256 x 10 x 15, 150 units, 2.49 / 2.41);
// returns the blocks, 0 where it does not run.
template <class L, class S, bool TOTALS>
int64_t launch_moments_rows(const void* pop, float* rho, float* j, double* partials, int64_t most, const KParams& p,
                            cudaStream_t s) {
    if (!p.rorder) return 0;
    const int gcap = dev::window_cap(p.max_row_links, S::kBytes), dcap = dev::window_cap(p.max_row_links, 4);
    const size_t smem = 2 * ((size_t)L::Q * p.seglen * S::kBytes + 2 * (size_t)p.lorder + gcap + dcap +
                             dev::halo_bytes(L::Q, p.nseg, S::kBytes));
    if (smem > stepk::kSmemBudget) return 0;
    auto kern = p.nseg > 1 ? k_moments_rows<L, S, TOTALS, kSegment> : k_moments_rows<L, S, TOTALS, kWholeRow>;
    const Shape sh = staged_shape((const void*)kern, p.seglen, smem, stepk::kSmemBudget);
    const int units = p.ny * p.nz * p.nseg;
    if (sh.blocks <= 0 || units < sh.sms) return 0;
    const int64_t blocks = std::min<int64_t>(std::min(sh.blocks, units), most);
    kern<<<(unsigned)blocks, sh.threads, smem, s>>>((const typename S::T*)pop, rho, j, partials, gcap, dcap, p);
    return blocks;
}

// One block sums interleaved per-block slots in a fixed order (deterministic);
// with add != 0 the result is added to out (window sums stay on the device).
constexpr int kReduceThreads = 512;
constexpr int kMaxSlots = 8;
__global__ void __launch_bounds__(kReduceThreads) k_reduce_slots(const double* __restrict__ slots, int64_t nb,
                                                                 int ns, double* __restrict__ out, int add) {
    __shared__ double sh[kReduceThreads / 32][kMaxSlots];
    double acc[kMaxSlots];
#pragma unroll
    for (int k = 0; k < kMaxSlots; ++k) acc[k] = 0.0;
    for (int64_t i = threadIdx.x; i < nb; i += blockDim.x) {
#pragma unroll
        for (int k = 0; k < kMaxSlots; ++k)
            if (k < ns) acc[k] += slots[i * ns + k];
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < kMaxSlots; ++k) acc[k] = dev::warp_sum(acc[k]);
    if (lane == 0) {
#pragma unroll
        for (int k = 0; k < kMaxSlots; ++k) sh[wid][k] = acc[k];
    }
    __syncthreads();
    if (wid == 0) {
#pragma unroll
        for (int k = 0; k < kMaxSlots; ++k) {
            double v = lane < (int)(blockDim.x / 32) ? sh[lane][k] : 0.0;
            v = dev::warp_sum(v);
            if (lane == 0 && k < ns) out[k] = add ? out[k] + v : v;
        }
    }
}

// FP32 populations f_a(x, t) = f0_a + h_a (or the deviations h_a).
template <class L, class S>
__global__ void __launch_bounds__(kBlock) k_populations(const typename S::T* __restrict__ P,
                                                        const uint32_t* __restrict__ nbr, float* __restrict__ f,
                                                        bool deviation, KParams p) {
    Cell c;
    if (!dev::cell_of_thread(p, c)) return;
    const uint32_t m = nbr[c.cell];
    if (m & kSolidBit) {
#pragma unroll
        for (int a = 0; a < L::Q; ++a) f[(int64_t)a * p.N + c.cell] = 0.f;
        return;
    }
    float h[L::Q];
    dev::pull<L, S>(P, p, m, c, h);
#pragma unroll
    for (int a = 0; a < L::Q; ++a) {
        const float d = h[a] * p.inv_scale;
        f[(int64_t)a * p.N + c.cell] = deviation ? d : p.f0[a] + d;
    }
}

// Copies an FP32 field in the slot layout of the populations (see pop_slot)
// into direction-major order out[a * N + cell].
template <class L>
__global__ void __launch_bounds__(kBlock) k_unslot(const float* __restrict__ in, float* __restrict__ out, KParams p) {
    Cell c;
    if (!dev::cell_of_thread(p, c)) return;
#pragma unroll
    for (int a = 0; a < L::Q; ++a) out[(int64_t)a * p.N + c.cell] = in[dev::pop_at<L>(p, c, a, 0)];
}

// Units to whole rows (PACK) or back: row r, slot s, column x is element
// (r Q + s) nx + x of the rows.  blockIdx.y is the chunk of columns, blocks stride
// over the rows' slots in x (with the chunk worked out per element, the divisions
// bound it: 173 us for the field of 250 x 256 x 256 cells).
template <class T, bool PACK>
__global__ void __launch_bounds__(256) k_pack_rows(T* __restrict__ units, T* __restrict__ rows, uint32_t Q,
                                                   KParams p) {
    const int x = blockIdx.y * blockDim.x + threadIdx.x;
    if (x >= p.nx) return;
    const int k = p.nseg == 1 ? 0 : x / p.seglen;
    units += (int64_t)k * Q * p.seglen + (x - k * p.seglen);
    rows += x;
    const uint32_t n = (uint32_t)p.ny * (uint32_t)p.nz * Q;  // at most Q N / nx slots
    for (uint32_t t = blockIdx.x; t < n; t += gridDim.x) {
        const uint32_t r = Q == 1 ? t : t / Q, s = t - r * Q;
        T* u = units + ((int64_t)r * p.nseg * Q + s) * p.seglen;
        T* w = rows + (int64_t)t * p.nx;
        if (PACK)
            *w = *u;
        else
            *u = *w;
    }
}

Launch grid_of(const KParams& p) {
    Launch l;
    const int bx = p.nx >= kBlock ? kBlock : ((p.nx + 31) / 32) * 32;
    l.block = dim3(bx);
    l.grid = dim3((unsigned)(p.ny * p.nz), (unsigned)((p.nx + bx - 1) / bx));
    return l;
}

template <class F>
int dispatch_lattice(int vel, F&& f) {
    if (vel == LBM_D2V9) return f(LatD2V9{});
    if (vel == LBM_D3V27) return f(LatD3V27{});
    if (vel == LBM_D1V3) return f(LatD1V3{});
    return f(LatD3V19{});
}

template <class F>
int dispatch_storage(int storage, F&& f) {
    if (storage == LBM_F16_DEV) return f(StoreF16{});
    if (storage == LBM_BF16_DEV) return f(StoreBF16{});
    return f(StoreF32{});
}

}  // namespace

int sm_count() {
    constexpr int kDevices = 64;
    static std::atomic<int> known[kDevices];
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < kDevices) sms = known[dev].load();
    if (sms > 0) return sms;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) return 1;
    if (dev >= 0 && dev < kDevices) known[dev].store(sms);
    return sms;
}

namespace {
using ShapeKey = std::tuple<const void*, int, int, size_t>;
std::mutex g_shapes_mutex;
std::map<ShapeKey, Shape> g_shapes;
ShapeKey shape_key(const void* kernel, int n, size_t smem) {
    int dev = 0;
    cudaGetDevice(&dev);
    return ShapeKey(kernel, dev, n, smem);
}
}  // namespace

bool known_shape(const void* kernel, int n, size_t smem, Shape* s) {
    const ShapeKey key = shape_key(kernel, n, smem);
    std::lock_guard<std::mutex> lock(g_shapes_mutex);
    const auto it = g_shapes.find(key);
    if (it == g_shapes.end()) return false;
    *s = it->second;
    return true;
}

void keep_shape(const void* kernel, int n, size_t smem, const Shape& s) {
    const ShapeKey key = shape_key(kernel, n, smem);
    std::lock_guard<std::mutex> lock(g_shapes_mutex);
    if (g_shapes.size() >= kLaunchShapes) g_shapes.clear();
    try {
        g_shapes[key] = s;
    } catch (const std::bad_alloc&) {  // then it is asked again
    }
}

bool allow_smem(const void* kernel, size_t budget) {
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)budget) == cudaSuccess)
        return true;
    cudaGetLastError();
    return false;
}

Shape staged_shape(const void* kernel, int columns, size_t smem, size_t budget, int fixed_threads) {
    Shape best;
    if (known_shape(kernel, columns, smem, &best)) return best;
    const int tmax = fixed_threads ? fixed_threads
                                   : (columns >= kRowThreads ? kRowThreads : ((columns + 31) / 32) * 32);
    const int tmin = fixed_threads ? fixed_threads : tmax / 2;
    best = Shape{tmax, 0, sm_count()};
    if (allow_smem(kernel, budget)) {
        for (int t = tmax; t >= 32 && t >= tmin; t -= 32) {
            int per_sm = 0;
            if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, t, smem) != cudaSuccess)
                cudaGetLastError();
            if (per_sm * best.sms > best.blocks) {
                best.blocks = per_sm * best.sms;
                best.threads = t;
            }
        }
    }
    keep_shape(kernel, columns, smem, best);
    return best;
}

int64_t moments_partial_count(const KParams& p) {
    Launch l = grid_of(p);
    return (int64_t)l.grid.x * l.grid.y;
}

int launch_build_neighbors(int vel, const uint8_t* mask, uint32_t* nbr, unsigned long long* fluid_count,
                           const KParams& p, cudaStream_t s) {
    Launch l = grid_of(p);
    return dispatch_lattice(vel, [&](auto lat) {
        using L = decltype(lat);
        k_neighbors<L><<<l.grid, l.block, 0, s>>>(mask, nbr, fluid_count, p);
        return 1;
    });
}

int launch_build_links(int vel, const uint32_t* nbr, uint32_t* lbase, uint32_t* rowG, void* temp,
                       size_t* temp_bytes, const KParams& p, cudaStream_t s) {
    const int n = (int)p.N;
    if (!temp) {
        // query the scan's temporary size
        return cub::DeviceScan::ExclusiveSum(nullptr, *temp_bytes, lbase, lbase, n, s) == cudaSuccess ? 0 : -1;
    }
    Launch l = grid_of(p);
    dispatch_lattice(vel, [&](auto lat) {
        using L = decltype(lat);
        k_link_counts<L><<<l.grid, l.block, 0, s>>>(nbr, lbase, p);
        return 1;
    });
    cub::DeviceScan::ExclusiveSum(temp, *temp_bytes, lbase, lbase, n, s);
    const int64_t U = (int64_t)p.ny * p.nz * p.nseg;
    const int blocks = (int)((U + 1 + 255) / 256 < 4096 ? (U + 1 + 255) / 256 : 4096);
    dispatch_lattice(vel, [&](auto lat) {
        using L = decltype(lat);
        k_row_starts<L><<<blocks, 256, 0, s>>>(nbr, lbase, rowG, p);
        return 1;
    });
    return 3;
}

// Failure-path probe: one block waits, with the staged kernels' bounded
// wait, on an mbarrier that nothing completes; the wait runs out after
// `limit` clocks and the block writes code 3 into the status word.
__global__ void k_wait_probe(int* status, uint32_t limit) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        dev::mbar_init(&bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    __syncthreads();
    const bool done = dev::mbar_wait(&bar, 0u, limit);
    if (!done && threadIdx.x == 0 && status) atomicExch(status, 3);
}

int launch_wait_probe(int* status, uint32_t limit, cudaStream_t s) {
    k_wait_probe<<<1, 32, 0, s>>>(status, limit);
    return 1;
}

int launch_unslot(int vel, const float* in, float* out, const KParams& p, cudaStream_t s) {
    Launch l = grid_of(p);
    return dispatch_lattice(vel, [&](auto lat) {
        using L = decltype(lat);
        k_unslot<L><<<l.grid, l.block, 0, s>>>(in, out, p);
        return 1;
    });
}

int launch_pack_rows(int storage, int Q, void* units, void* rows, bool pack, const KParams& p, cudaStream_t s) {
    const int threads = p.nx >= 256 ? 256 : ((p.nx + 31) / 32) * 32;
    const int64_t slots = (int64_t)p.ny * p.nz * Q, chunks = (p.nx + threads - 1) / threads;
    const int64_t most = std::max<int64_t>((int64_t)sm_count() * 32 / chunks, 1);
    const dim3 blocks((unsigned)std::min<int64_t>(slots, most), (unsigned)chunks);
    return dispatch_storage(storage, [&](auto st) {
        using T = typename decltype(st)::T;
        if (pack)
            k_pack_rows<T, true><<<blocks, threads, 0, s>>>((T*)units, (T*)rows, (uint32_t)Q, p);
        else
            k_pack_rows<T, false><<<blocks, threads, 0, s>>>((T*)units, (T*)rows, (uint32_t)Q, p);
        return 1;
    });
}

int launch_build_row_order(const uint32_t* nbr, uint16_t* rorder, const KParams& p, cudaStream_t s) {
    const int64_t U = (int64_t)p.ny * p.nz * p.nseg;
    const int64_t blocks = std::min<int64_t>((U * 32 + kBlock - 1) / kBlock, 65535);
    k_row_order<<<(unsigned)blocks, kBlock, 0, s>>>(nbr, rorder, p);
    return 1;
}

int launch_build_link_desc(int vel, const uint32_t* nbr, const uint32_t* lbase, uint32_t* ldesc, const KParams& p,
                           cudaStream_t s) {
    Launch l = grid_of(p);
    return dispatch_lattice(vel, [&](auto lat) {
        using L = decltype(lat);
        k_link_desc<L><<<l.grid, l.block, 0, s>>>(nbr, lbase, ldesc, p);
        return 1;
    });
}

int launch_init(int vel, int storage, void* pop, const uint32_t* nbr, const float* rho, const float* u,
                const KParams& p, cudaStream_t s) {
    Launch l = grid_of(p);
    return dispatch_lattice(vel, [&](auto lat) {
        using L = decltype(lat);
        return dispatch_storage(storage, [&](auto st) {
            using S = decltype(st);
            k_init<L, S><<<l.grid, l.block, 0, s>>>((typename S::T*)pop, nbr, rho, u, p);
            return 1;
        });
    });
}

int launch_step(int vel, int storage, int force, bool efield, bool sr, const void* fin, void* fout,
                const uint32_t* nbr, const float* Ef, const KParams& p, cudaStream_t s) {
    const bool x = vel == LBM_D3V27 || vel == LBM_D1V3;
    StepLauncher* f;
    if (storage == LBM_F16_DEV)
        f = sr ? (x ? launch_step_f16_x : launch_step_f16) : (x ? launch_step_f16_x_n : launch_step_f16_n);
    else if (storage == LBM_BF16_DEV)
        f = sr ? (x ? launch_step_bf16_x : launch_step_bf16) : (x ? launch_step_bf16_x_n : launch_step_bf16_n);
    else
        f = x ? launch_step_f32_x : launch_step_f32;
    return f(vel, force, efield, fin, fout, nbr, Ef, p, s);
}

// With totals the blocks stride over the tiles, kTotalsPerSm of them per SM,
// and keep their FP64 sums in registers to the end: the chip adds two FP64
// values per cycle and SM, so a block reduction per 128 cells (160 shuffled
// FP64 adds) cost several times the reads (52 us on 1024^2 cells of D2V9 FP32),
// and its 8192 partials another 41 us in the one block that sums them.
constexpr int kTotalsPerSm = 8;

int launch_multi_f32(int, int, bool, void*, void*, const uint32_t*, const float*, int, unsigned*, bool*,
                     const KParams&, cudaStream_t);
int launch_multi_f16(int, int, bool, void*, void*, const uint32_t*, const float*, int, unsigned*, bool*,
                     const KParams&, cudaStream_t);
int launch_multi_bf16(int, int, bool, void*, void*, const uint32_t*, const float*, int, unsigned*, bool*,
                      const KParams&, cudaStream_t);

int launch_multi(int vel, int storage, int force, bool sr, void* fin, void* fout, const uint32_t* nbr, const float* Ef,
                 int n, unsigned* count, bool* in_fin, const KParams& p, cudaStream_t s) {
    if (storage == LBM_F16_DEV)
        return launch_multi_f16(vel, force, sr, fin, fout, nbr, Ef, n, count, in_fin, p, s);
    if (storage == LBM_BF16_DEV)
        return launch_multi_bf16(vel, force, sr, fin, fout, nbr, Ef, n, count, in_fin, p, s);
    return launch_multi_f32(vel, force, false, fin, fout, nbr, Ef, n, count, in_fin, p, s);
}

int launch_moments(int vel, int storage, const void* pop, const uint32_t* nbr, float* rho, float* j,
                   double* partials, int64_t* n_partials, const KParams& p, cudaStream_t s) {
    Launch l = grid_of(p);
    const int chunks = (int)l.grid.y;
    const int64_t tiles = (int64_t)l.grid.x * chunks;
    int64_t blocks = tiles;
    if (partials) blocks = std::min<int64_t>(tiles, (int64_t)sm_count() * kTotalsPerSm);
    return dispatch_lattice(vel, [&](auto lat) {
        using L = decltype(lat);
        return dispatch_storage(storage, [&](auto st) {
            using S = decltype(st);
            using T = typename S::T;
            // the partials of one launch: as many as the general kernel has tiles at most
            const int64_t staged = partials ? launch_moments_rows<L, S, true>(pop, rho, j, partials, tiles, p, s)
                                            : launch_moments_rows<L, S, false>(pop, rho, j, nullptr, tiles, p, s);
            if (n_partials) *n_partials = staged ? staged : blocks;
            if (staged) return route(kStaged, p.nseg > 1 ? kSegment : kWholeRow);
            if (partials)
                k_moments<L, S, true><<<(unsigned)blocks, l.block, 0, s>>>((const T*)pop, nbr, rho, j, partials, chunks, p);
            else
                k_moments<L, S, false><<<(unsigned)blocks, l.block, 0, s>>>((const T*)pop, nbr, rho, j, nullptr, chunks, p);
            return route(kGeneral);
        });
    });
}

int launch_reduce_partials(const double* partials, int64_t n_partials, double* out4, cudaStream_t s) {
    k_reduce_slots<<<1, kReduceThreads, 0, s>>>(partials, n_partials, 4, out4, 0);
    return 1;
}

int launch_reduce_slots(const double* slots, int64_t n_blocks, int n_slots, double* out, cudaStream_t s) {
    if (n_slots > kMaxSlots) return 0;
    k_reduce_slots<<<1, kReduceThreads, 0, s>>>(slots, n_blocks, n_slots, out, 0);
    return 1;
}

int launch_accumulate_totals(const double* partials, int64_t n_partials, double* acc4, cudaStream_t s) {
    k_reduce_slots<<<1, kReduceThreads, 0, s>>>(partials, n_partials, 4, acc4, 1);
    return 1;
}

int launch_populations(int vel, int storage, const void* pop, const uint32_t* nbr, float* f, bool deviation,
                       const KParams& p, cudaStream_t s) {
    Launch l = grid_of(p);
    return dispatch_lattice(vel, [&](auto lat) {
        using L = decltype(lat);
        return dispatch_storage(storage, [&](auto st) {
            using S = decltype(st);
            k_populations<L, S><<<l.grid, l.block, 0, s>>>((const typename S::T*)pop, nbr, f, deviation, p);
            return 1;
        });
    });
}

}  // namespace lbm
