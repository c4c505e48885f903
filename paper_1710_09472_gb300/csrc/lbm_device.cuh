// Device-side helpers shared by the step and adjoint kernels: thread-to-cell
// mapping, periodic neighbour indices, and lattice-vector dot products that
// unroll to adds and subtracts.
#pragma once

#include "lbm_internal.h"

namespace lbm {
namespace dev {

constexpr int kBlock = 128;

// One thread per cell: blockIdx.x is the row (y, z), blockIdx.y the chunk of
// x, threads run along x.  All cell indices fit in 32 bits (N < 2^31).
struct Cell {
    int x, y, z;
    uint32_t cell;
    int xm, xp;       // x - 1, x + 1 with periodic wrap
    int xo[3];        // offsets of the columns xm, x, xp in a row of units, slot 0
    uint32_t r[3][3]; // row (z + dz) * ny + (y + dy) for dy, dz in {-1, 0, 1}
    int64_t pcell;    // row * nxp + x: index into the padded fields (E, dL/dE partials)
};

__device__ __forceinline__ bool cell_at(const KParams& p, int row, int x, Cell& c) {
    c.x = x;
    c.y = row % p.ny;
    c.z = row / p.ny;
    c.cell = (uint32_t)row * (uint32_t)p.nx + (uint32_t)c.x;
    c.xm = c.x == 0 ? p.nx - 1 : c.x - 1;
    c.xp = c.x == p.nx - 1 ? 0 : c.x + 1;
    const int ys[3] = {c.y == 0 ? p.ny - 1 : c.y - 1, c.y, c.y == p.ny - 1 ? 0 : c.y + 1};
    const int zs[3] = {c.z == 0 ? p.nz - 1 : c.z - 1, c.z, c.z == p.nz - 1 ? 0 : c.z + 1};
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int k = 0; k < 3; ++k) c.r[i][k] = (uint32_t)zs[k] * (uint32_t)p.ny + (uint32_t)ys[i];
    c.pcell = (int64_t)row * p.nxp + x;
    const int xs[3] = {c.xm, c.x, c.xp};
#pragma unroll
    for (int i = 0; i < 3; ++i)  // whole rows need no division
        c.xo[i] = p.nseg == 1 ? xs[i] : xs[i] + xs[i] / p.seglen * (p.qm1 * p.seglen);
    return c.x < p.nx;
}
__device__ __forceinline__ bool cell_of_thread(const KParams& p, Cell& c) {
    return cell_at(p, blockIdx.x, blockIdx.y * blockDim.x + threadIdx.x, c);
}

// Index of x + s e_a (s = +1 or -1) with periodic wrap.
template <class L>
__device__ __forceinline__ uint32_t shifted(const KParams& p, const Cell& c, int a, int s) {
    const int ex = s * L::c(a, 0), ey = s * L::c(a, 1), ez = s * L::c(a, 2);
    const int xs = ex > 0 ? c.xp : (ex < 0 ? c.xm : c.x);
    return c.r[ey + 1][ez + 1] * (uint32_t)p.nx + (uint32_t)xs;
}

// Storage index of direction a at the cell x + s e_a (s = -1, 0 or +1): slot
// pop_slot(a) of that cell's row (see pop_slot).
template <class L>
__device__ __forceinline__ int64_t pop_at(const KParams& p, const Cell& c, int a, int s) {
    const int ex = s * L::c(a, 0), ey = s * L::c(a, 1), ez = s * L::c(a, 2);
    return (int64_t)c.r[ey + 1][ez + 1] * (uint32_t)(L::Q * p.nxp) + (pop_slot<L>(a) * p.seglen + c.xo[ex + 1]);
}

template <class L>
__device__ __forceinline__ float edot(int a, const float* v) {
    float r = 0.f;
    if (L::c(a, 0) > 0) r += v[0];
    if (L::c(a, 0) < 0) r -= v[0];
    if (L::c(a, 1) > 0) r += v[1];
    if (L::c(a, 1) < 0) r -= v[1];
    if (L::D == 3) {
        if (L::c(a, 2) > 0) r += v[2];
        if (L::c(a, 2) < 0) r -= v[2];
    }
    return r;
}

__device__ __forceinline__ void cross3(const float* a, const float* b, float* c) {
    c[0] = a[1] * b[2] - a[2] * b[1];
    c[1] = a[2] * b[0] - a[0] * b[2];
    c[2] = a[0] * b[1] - a[1] * b[0];
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// Pull the stored (scaled) deviations of f(x, t) from a state (populations P,
// in the slot layout of pop_slot, followed by the link buffer G):
// f_a(x) = P_a(x - e_a) when x - e_a is fluid;
// when it is solid (bit a of the link mask) the halfway bounce-back value
// f_a(x) = f*_abar(x), which the collision at x stored in the link slot of its
// outgoing direction abar.
// The two cases differ in the address only, which is selected: one load per
// direction, all of them in flight together.  With a branch around each load
// they were issued one after another, and the kernels that pull this way
// waited on them (long scoreboard 17 of 21 stalled cycles per issue): 20 general
// steps and the fields of 250 x 128 x 128 porous D3V19 FP16 took 4.21 ms
// against 3.44 with the selection.  A cell's link slots follow its outgoing directions in
// ascending order, so a running count replaces a popcount per direction.
template <class L, class S>
__device__ __forceinline__ void pull(const typename S::T* __restrict__ P, const KParams& p, uint32_t m, const Cell& c,
                                     float* h) {
    const typename S::T* __restrict__ G =
        reinterpret_cast<const typename S::T*>(reinterpret_cast<const char*>(P) + p.gofs);
    const typename S::T* g = G + (m ? __ldg(p.lbase + c.cell) : 0u);
    h[0] = S::raw(P + pop_at<L>(p, c, 0, -1));
#pragma unroll
    for (int a = 1; a < L::Q; a += 2) {
        // outgoing direction a comes back as a + 1, outgoing a + 1 as a
        const bool s1 = (m >> (a + 1)) & 1u, s0 = (m >> a) & 1u;
        const typename S::T* q1 = P + pop_at<L>(p, c, a + 1, -1);
        const typename S::T* q0 = P + pop_at<L>(p, c, a, -1);
        if (s1) q1 = g;
        g += s1;
        if (s0) q0 = g;
        g += s0;
        h[a] = S::raw(q0);
        h[a + 1] = S::raw(q1);
    }
}

// Bounce-back patch of a staged row set.  Link k of the unit is a fluid cell x
// with an outgoing direction b into a solid cell (descriptor link_desc).  The
// solid neighbour x + e_b is read by exactly one cell for each direction: by x
// itself, in the pull of direction bbar (which reads x - e_bbar = x + e_b) and
// in the adjoint gather of direction b (which reads x + e_b).  So the halfway
// bounce-back value win[k - w0] is written into that staged slot, of direction
// bbar (PULL) or b (gather), and the cells then read their rows without any
// link logic.  The descriptors come from the staged window desc (first element
// d0); they hold the slots and columns worked out once per geometry, which
// leaves half the instructions of a pass that decodes (x, b) and wraps x.
// HALO: a neighbour may lie in a halo array (hal: Q left values, Q right ones).
template <bool PULL, bool HALO, class T>
__device__ __forceinline__ void patch_links(T* rows, int rs, T* hal, int Q, const T* win, uint32_t w0, uint32_t g0,
                                            uint32_t g1, const uint32_t* desc, uint32_t d0) {
    for (uint32_t k = g0 + threadIdx.x; k < g1; k += blockDim.x) {
        const uint32_t d = desc[k - d0];
        const int slot = PULL ? desc_slot_bar(d) : desc_slot(d), pos = desc_pos(d);
        T* q = rows + slot * rs + pos;
        if (HALO && pos >= kPosLeft) q = hal + (pos == kPosLeft ? 0 : Q) + slot;
        *q = win[k - w0];
    }
}

// Bytes reserved for a staged window of up to n elements of esize bytes.
__host__ __device__ __forceinline__ int window_cap(int n, int esize) {
    return (int)((((size_t)n * esize + 15) & ~(size_t)15) + 32);
}

// ---------------------------------------------------------------------------
// Bulk asynchronous copies (the non-tensor form of the Blackwell TMA engine)
// and mbarriers.  A stage is filled by one thread: mbarrier.arrive.expect_tx
// with the stage's byte count, then one cp.async.bulk per contiguous piece,
// each completing its bytes on the stage's mbarrier.  Output rows leave
// shared memory with cp.async.bulk stores (bulk groups).  Addresses and
// sizes are multiples of 16 bytes.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
// One potentially blocking test: the thread may be suspended in hardware
// until the phase completes or a system-dependent time limit passes.
__device__ __forceinline__ bool mbar_try(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// Waits for the phase of the given parity to complete; gives up and returns
// false after `limit` SM clock cycles (32 bits of the clock: a 64-bit count took
// the FP32 step on D3V19 segments from 64 to 74 registers).
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, uint32_t limit) {
    if (mbar_try(bar, parity)) return true;
    const uint32_t t0 = (uint32_t)clock();
    while (!mbar_try(bar, parity))
        if ((uint32_t)clock() - t0 > limit) return false;
    return true;
}
// Sleeps about n SM clock cycles.  After a wait has run out, a block pauses
// so that bulk copies it issued earlier land before it moves on or exits.
__device__ __forceinline__ void pause_cycles(long long n) {
    const long long t0 = clock64();
    while (clock64() - t0 < n) __nanosleep(1000);
}
// Waits for a unit's stage; true when it has arrived.  When the wait runs out
// (or ran out in an earlier unit: ok is false), code goes to the status word and
// nothing of the stage may be taken for an address, so this thread empties its
// link range (its passes over the descriptors do nothing) and its part of the
// unit's cell order (no fluid cells, every column the unit's first).  All threads
// do that, or the stage had arrived after all, before the next block barrier, so
// the unit's passes stay inside their buffers; what they write is invalid.
// The passes themselves have no test for it: one around the link pass took the
// FP16 step of 256^3 D3V19 from 240.8 to 242.9 us, leaving the loop after the
// barrier to 250.5.
__device__ __forceinline__ bool stage_wait(uint64_t* bar, uint32_t parity, bool ok, int code, uint32_t g0,
                                           uint32_t& g1, uint16_t* order, const KParams& p) {
    if (ok && mbar_wait(bar, parity, p.wait_clocks)) return true;
    if (ok) {
        if (p.status) atomicExch(p.status, code);
        pause_cycles(1ll << 22);  // let this block's copies in flight land
    }
    g1 = g0;
    for (int k = threadIdx.x; k < p.lorder; k += blockDim.x) order[k] = 0;
    return false;
}

// global -> shared, completing `bytes` on the mbarrier
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}
// shared -> global, in the current bulk group
__device__ __forceinline__ void bulk_store(void* dst, const void* src, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;\n" ::"l"(dst), "r"(smem_u32(src)),
                 "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;\n" ::: "memory"); }
// the sources of all committed bulk stores have been read
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory"); }
// all committed bulk stores are complete
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;\n" ::: "memory"); }
// orders this thread's generic-proxy shared-memory accesses before later
// async-proxy (bulk copy) accesses
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }

// A unit of the row-staged kernels: its row, segment, first column x0 and cells.
struct UnitAt {
    int row, seg, x0, len;
};
template <int RS, int MODE>
__device__ __forceinline__ UnitAt unit_at(const KParams& p, int unit) {
    UnitAt u{unit, 0, 0, RS && MODE == kExactRow ? RS : p.nx};
    if (MODE == kSegment) {
        u.row = unit / p.nseg;
        u.seg = unit - u.row * p.nseg;
        u.x0 = u.seg * p.seglen;
        u.len = min(p.seglen, p.nx - u.x0);
    }
    return u;
}

// One thread: copies the Q source rows of a unit from the field F (unit
// layout) into rows (slot order, RS or seglen columns each), completing on bar.
// PULL: the rows (y - e_ay, z - e_az), read at x - e_ax; else the gather rows
// (y + e_ay, z + e_az), read at x + e_ax.  The slots of the directions with one
// (e_y, e_z) are consecutive: one copy per neighbouring row.
template <class L, int RS, int MODE, bool PULL, class T>
__device__ __forceinline__ void stage_rows(T* rows, const T* __restrict__ F, const UnitAt& u, uint64_t* bar,
                                           const KParams& p) {
    const int y = u.row % p.ny, z = u.row / p.ny;
    const int yp = y == p.ny - 1 ? 0 : y + 1, ym = y == 0 ? p.ny - 1 : y - 1;
    const int zp = z == p.nz - 1 ? 0 : z + 1, zm = z == 0 ? p.nz - 1 : z - 1;
    const int rs = RS ? RS : p.seglen;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        if (key_count<L>(k) == 0) continue;
        // slots key_first(k) .. of the source row, periodic
        const int ey = PULL ? k / 3 - 1 : 1 - k / 3, ez = PULL ? k % 3 - 1 : 1 - k % 3, s0 = key_first<L>(k);
        const int ys = ey > 0 ? ym : (ey < 0 ? yp : y);
        const int zs = ez > 0 ? zm : (ez < 0 ? zp : z);
        const int su = MODE != kSegment ? zs * p.ny + ys : (zs * p.ny + ys) * p.nseg + u.seg;
        bulk_load(rows + s0 * rs, F + ((int64_t)su * L::Q + s0) * rs,
                  (uint32_t)(key_count<L>(k) * rs) * (uint32_t)sizeof(T), bar);
    }
}

// The directions that read column x - 1 (NEG: x + 1) in a pull, by slot, 5 bits
// each (9 of D3V27 at most), their number, and the velocity components by slot
// (e + 1, 2 bits each); worked out once per lattice.
template <class L>
struct SlotDirs {
    unsigned long long y, z, pos, neg;
    int moving_x;
    constexpr SlotDirs() : y(0), z(0), pos(0), neg(0), moving_x(0) {
        int np = 0, nn = 0;
        for (int a = 0; a < L::Q; ++a) {
            const int s = pop_slot_calc<L>(a);
            y |= (unsigned long long)(L::c(a, 1) + 1) << (2 * s);
            z |= (unsigned long long)(L::c(a, 2) + 1) << (2 * s);
            if (L::c(a, 0) > 0) pos |= (unsigned long long)s << (5 * np++);
            if (L::c(a, 0) < 0) neg |= (unsigned long long)s << (5 * nn++);
        }
        moving_x = np;
    }
};

// Halo values of a segment (nseg > 1): thread i < 2 moving_x fetches one value
// of the field F that a cell at an end of the segment reads beyond it, and
// halo_put writes it to its place in the halo arrays (left, then right, by
// slot).  The fetch goes out when the unit's bulk copies do; the put follows a
// unit later, so the load's latency is covered.
template <class L, bool PULL, class T>
__device__ __forceinline__ T halo_fetch(const T* __restrict__ F, const UnitAt& u, const KParams& p) {
    constexpr SlotDirs<L> dirs{};
    const int i = threadIdx.x;
    const bool right = i >= dirs.moving_x;
    const int k = right ? i - dirs.moving_x : i;
    // a pull reads the left column along e_x > 0, a gather along e_x < 0
    const int s = (int)(((right == PULL ? dirs.neg : dirs.pos) >> (5 * k)) & 31ull);
    const int sy = (int)((dirs.y >> (2 * s)) & 3ull) - 1, sz = (int)((dirs.z >> (2 * s)) & 3ull) - 1;
    const int y = u.row % p.ny, z = u.row / p.ny;
    int ys = PULL ? y - sy : y + sy, zs = PULL ? z - sz : z + sz;
    ys = ys < 0 ? ys + p.ny : (ys >= p.ny ? ys - p.ny : ys);
    zs = zs < 0 ? zs + p.nz : (zs >= p.nz ? zs - p.nz : zs);
    int x = right ? u.x0 + u.len : u.x0 - 1;
    x = x < 0 ? p.nx - 1 : (x >= p.nx ? 0 : x);
    const int seg = x / p.seglen;
    return __ldg(F + (((int64_t)(zs * p.ny + ys) * p.nseg + seg) * L::Q + s) * p.seglen + (x - seg * p.seglen));
}
template <class L, bool PULL, class T>
__device__ __forceinline__ void halo_put(T* hal, T v) {
    constexpr SlotDirs<L> dirs{};
    const int i = threadIdx.x;
    const bool right = i >= dirs.moving_x;
    const int k = right ? i - dirs.moving_x : i;
    const int s = (int)(((right == PULL ? dirs.neg : dirs.pos) >> (5 * k)) & 31ull);
    hal[(right ? L::Q : 0) + s] = v;
}
template <class L>
__device__ __forceinline__ bool halo_thread() {
    constexpr SlotDirs<L> dirs{};
    return (int)threadIdx.x < 2 * dirs.moving_x;
}
// Bytes of the halo arrays of a stage (0 for whole rows).
__host__ __device__ __forceinline__ int halo_bytes(int Q, int nseg, int esize) {
    return nseg == 1 ? 0 : (2 * Q * esize + 15) / 16 * 16;
}

// Bytes [b0, b1) of the 16-byte aligned window covering elements [g0, g1).
__device__ __forceinline__ void window_bytes(uint32_t g0, uint32_t g1, int esize, uint64_t& b0, uint64_t& b1) {
    b0 = ((uint64_t)g0 * esize) & ~15ull;
    b1 = ((uint64_t)g1 * esize + 15ull) & ~15ull;
}

}  // namespace dev
}  // namespace lbm
