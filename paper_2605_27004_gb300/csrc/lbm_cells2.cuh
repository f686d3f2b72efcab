// Two cells per thread for FP16 r-shifted storage where the x-adjacent pairs of lbm_pairs.cuh do not
// apply: rows of odd length, and the even AA step with walls.
//
// The one-cell FP16 kernels are bound by issued instructions (653 a cell for D3Q27, 70 % of the issue
// slots busy at half the DRAM bandwidth). In rows of odd length no word of two cells is aligned, so a
// thread takes two cells half a row apart, each with its own steps to its wrapped neighbours, and
// reads and writes their elements one by one (lanes are consecutive cells, so accesses stay
// coalesced); only the collision is shared, as packed FP32 pairs. Rows are numbered through, so no
// lanes idle at their ends. Measured against one cell a thread: D3Q27 257^3 pull 469 -> 373 us a step,
// 149 x 131 x 113 pull 61.5 -> 55.4, AA 55.1 -> 50.5; D3Q19 151^3 AA 63.0 -> 57.7; D2Q9 1001 x 1003
// 10.1 -> 8.5. The same over the fluid-cell list of a porous box gained nothing for the odd step and lost
// for pull (22 % of the warps resident instead of 43 %, and three dependent loads a cell).
#pragma once
#include "lbm_pairs.cuh"

namespace lbm {
inline namespace LBM_VARIANT {

__device__ __forceinline__ bool bad_pair(const Macro2& m, bool a, bool b) {
    return (a && bad1(m.rho.v.x, m.ux.v.x, m.uy.v.x, m.uz.v.x)) ||
           (b && bad1(m.rho.v.y, m.ux.v.y, m.uy.v.y, m.uz.v.y));
}

// A cell and the steps to its wrapped neighbours (index differences, modulo 2^32).
struct SCell {
    uint32_t n, xp, xm, yp, ym, zp, zm;
};
__device__ __forceinline__ SCell make_scell(const Geom& g, uint32_t x, uint32_t y, uint32_t z) {
    const uint32_t nx = (uint32_t)g.nx, ny = (uint32_t)g.ny, nz = (uint32_t)g.nz, P = nx * ny;
    SCell c;
    c.n = x + nx * (y + ny * z);
    c.xp = x + 1 == nx ? 1u - nx : 1u;
    c.xm = x == 0 ? nx - 1u : ~0u;
    c.yp = y + 1 == ny ? nx - P : nx;
    c.ym = y == 0 ? P - nx : 0u - nx;
    c.zp = z + 1 == nz ? P - g.N : P;
    c.zm = z == 0 ? g.N - P : 0u - P;
    return c;
}
// Makes the compiler form the offsets anew from here on, instead of keeping those of the gather.
__device__ __forceinline__ void forget(SCell& c) {
    asm volatile("" : "+r"(c.n), "+r"(c.xp), "+r"(c.xm), "+r"(c.yp), "+r"(c.ym), "+r"(c.zp), "+r"(c.zm));
}
// index of the cell one step along s
__device__ __forceinline__ uint32_t scell_at(const SCell& c, Vec3 s) {
    uint32_t n = c.n;
    if (s.x) n += s.x > 0 ? c.xp : c.xm;
    if (s.y) n += s.y > 0 ? c.yp : c.ym;
    if (s.z) n += s.z > 0 ? c.zp : c.zm;
    return n;
}

// The neighbour whose slot i (PULL) or opp i (AAODD) holds f_i of the cell: x - c_i.
template <int Q>
__device__ __forceinline__ uint32_t scell_from(const SCell& c, int i) {
    const Vec3 v = vel<Q>(i);
    return scell_at(c, Vec3{-v.x, -v.y, -v.z});
}

template <int Q, int LAYOUT>
__device__ __forceinline__ void gather_cells2(const SCell& a, const SCell& b, const Planes<const __half>& src,
                                              F2 (&d)[Q]) {
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const __half* p = src.p[LAYOUT == LAYOUT_PULL ? i : opp(i)];
        d[i] = LAYOUT == LAYOUT_LOCAL ? f2(ld_rw(src.p[i] + a.n), ld_rw(src.p[i] + b.n))
                                      : f2(ld_rw(p + scell_from<Q>(a, i)), ld_rw(p + scell_from<Q>(b, i)));
    }
}

// Rows of odd length: thread t owns the cells x and x + H of a row, H = (nx + 1) / 2.
__device__ __forceinline__ bool make_row_cells2(const Geom& g, SCell& a, SCell& b, bool& vb) {
    const uint32_t H = ((uint32_t)g.nx + 1u) / 2u;
    const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    const uint32_t row = t / H, x = t - row * H;
    const uint32_t z = row / (uint32_t)g.ny, y = row - z * (uint32_t)g.ny;
    if (z >= (uint32_t)(g.nz - 2 * LBM_SLAB)) return false;
    vb = x + H < (uint32_t)g.nx;
    a = make_scell(g, x, y, z + LBM_SLAB);
    b = make_scell(g, vb ? x + H : x, y, z + LBM_SLAB);
    return true;
}

// Blocks of 128 threads, four (D3Q27, 124 registers) or five per SM; at 257^3 D3Q27 three, four and five
// of them take 433, 373 and 374 us a step (one cell a thread: 469).
constexpr int CELLS2_THREADS = 128;
template <int Q>
__host__ __device__ constexpr int cells2_blocks() {
    return Q == 27 ? 4 : 5;
}

// Rows of odd length, no walls.
template <int Q, bool EARLY>
__global__ void __launch_bounds__(CELLS2_THREADS, cells2_blocks<Q>())
    k_step_pull_rows2(Geom g, Coef<float> cf, const Planes<const __half> src, const Planes<__half> dst,
                      int* __restrict__ flag) {
    SCell a, b;
    bool vb;
    if (!make_row_cells2(g, a, b, vb)) return;
    wait_previous<EARLY>();
    F2 d[Q];
    gather_cells2<Q, LAYOUT_PULL>(a, b, src, d);
    const Macro2 m = bgk<Q, 3>(cf, d);
    if (bad_pair(m, true, true)) *flag = 1;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const __half2 h = __float22half2_rn(d[i].v);
        dst.p[i][a.n] = __low2half(h);
        if (vb) dst.p[i][b.n] = __high2half(h);
    }
}

// ---------------------------------------------------------------------------------------------
// AA steps in place (k_step_aa) in rows of odd length. The slot that takes f*_i in the odd step is the
// one that held f_opp(i) of the same cell, so its index is that of the opposite direction's gather.
// ---------------------------------------------------------------------------------------------
template <int Q, int ODD, bool EARLY>
__global__ void __launch_bounds__(CELLS2_THREADS, cells2_blocks<Q>())
    k_step_aa_rows2(Geom g, Coef<float> cf, const Planes<const __half> src, const Planes<__half> dst,
                    int* __restrict__ flag) {
    SCell a, b;
    bool vb;
    if (!make_row_cells2(g, a, b, vb)) return;
    wait_previous<EARLY>();
    F2 d[Q];
    gather_cells2<Q, ODD ? LAYOUT_AAODD : LAYOUT_LOCAL>(a, b, src, d);
    const Macro2 m = bgk<Q, 3>(cf, d);
    if (bad_pair(m, true, true)) *flag = 1;
    if (ODD) {
        forget(a);
        forget(b);
    }
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const __half2 h = __float22half2_rn(d[i].v);
        __half* p = dst.p[ODD ? i : opp(i)];
        p[ODD ? scell_from<Q>(a, opp(i)) : a.n] = __low2half(h);
        if (vb) p[ODD ? scell_from<Q>(b, opp(i)) : b.n] = __high2half(h);
    }
}

// ---------------------------------------------------------------------------------------------
// Even AA step with walls: purely local, so neither neighbours nor link words are needed, only which
// cells are fluid. Over the list of 16-cell sectors that hold fluid, eight lanes a sector, a lane its
// cells 2 l and 2 l + 1 as one aligned word per plane (the number of cells is even). Slots of solid
// cells are written with the zeros they hold, so that sectors are written whole. Against one cell of
// the fluid-cell list per thread, porous D3Q27 160^3: 90.6 -> 75.3 us.
// ---------------------------------------------------------------------------------------------
template <int Q>
__global__ void __launch_bounds__(CELLS2_THREADS, Q == 27 ? 5 : 6)
    k_step_aa_even_sectors2(Geom g, Coef<float> cf, SectorList L, const Planes<const __half> src,
                            const Planes<__half> dst, int* __restrict__ flag) {
    const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t / 8u >= L.count) return;
    const uint2 s = __ldg(L.sector + t / 8u);
    const uint32_t n = s.x * 16u + 2u * (t % 8u);
    const bool fa = (s.y >> (2u * (t % 8u))) & 1u, fb = (s.y >> (2u * (t % 8u) + 1u)) & 1u;
    if (n >= g.N) return;  // the last sector may reach past the box
    F2 d[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) d[i] = ld2_rw(src.p[i] + n);
    const Macro2 m = bgk<Q, 3>(cf, d);
    if (bad_pair(m, fa, fb)) *flag = 1;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        if (!fa) d[i].v.x = 0.f;
        if (!fb) d[i].v.y = 0.f;
        st2(dst.p[opp(i)] + n, d[i]);
    }
}

}  // namespace LBM_VARIANT
}  // namespace lbm
