// Host-side launchers of one (lattice, storage) pair: kernel choice (one or two cells per
// thread), launch shapes and the dispatch over walls and layouts.
#pragma once
#include <algorithm>
#include "lbm_ade.cuh"
#include "lbm_kernels.cuh"
#include "lbm_adjoint2.cuh"
#include "lbm_lanes.cuh"
#include "lbm_pairs.cuh"
#include "lbm_plane.cuh"
#include "lbm_quads.cuh"
#include "lbm_twice.cuh"

namespace lbm {
inline namespace LBM_VARIANT {

// ---------------------------------------------------------------------------------------------
template <int Q, int S>
struct Launch {
    using ST = typename Store<S>::type;
    using T = typename Store<S>::T;
    using CF = Coef<T>;
    static Planes<const ST> cpl(const void* p, const Geom& g) { return planes_of(static_cast<const ST*>(p), Q, g.N); }
    static Planes<ST> mpl(void* p, const Geom& g) { return planes_of(static_cast<ST*>(p), Q, g.N); }
    static Planes<const T> cfl(const void* p, const Geom& g) { return planes_of(static_cast<const T*>(p), Q, g.N); }
    static Planes<T> mfl(void* p, const Geom& g) { return planes_of(static_cast<T*>(p), Q, g.N); }

    // Launches that take the EARLY instances (wait_previous): the launch gap counts there. Blocks set up
    // while the previous kernel still runs are not spread evenly, so not where an SM gets one to three
    // of them (D3Q19 FP16 64 x 40 x 50, 250 blocks: 3.3 -> 3.6 us a step; D2Q9 301 x 250, 295 blocks: 2.2 ->
    // 2.5; up to four of the D3Q27 FP16 pair blocks: 64 x 40 x 50 4.0 -> 4.2), nor for FP64, bound by the
    // FP64 pipes of the SMs (D2Q9 128 x 300 9.8 -> 16.1, D3Q27 26 x 23 x 31 18.2 -> 35.3). Larger boxes
    // gain nothing: beyond 2M cells, FP16 beyond 90 MB of two arrays (D3Q19 130 x 100 x 100 24.3 -> 24.9),
    // D3Q27 beyond 60 (FP32 96 x 70 x 60 11.9 -> 12.1).
    static bool early(const Geom& g, dim3 grid) {
        const unsigned long long bytes = 2ull * Q * sizeof(ST) * g.N;
        if (g.N > (1u << 21) || bytes > (Q == 27 ? 60000000ull : S == 3 ? 90000000ull : ~0ull)) return false;
        const unsigned long long blocks = (unsigned long long)grid.x * grid.y * grid.z, sms = (unsigned)sm_count();
        return blocks <= sms || blocks >= (Q == 27 && S == 3 ? 4 : 3) * sms;
    }
#define LBM_UNWRAP(...) __VA_ARGS__
#define LBM_EARLY(K, PARAMS, GRID, BLOCK, ...)                                                     \
    do {                                                                                           \
        if constexpr (S != 1) {                                                                    \
            if (early(g, GRID))                                                                    \
                return launch_after(K<LBM_UNWRAP PARAMS, true>, GRID, BLOCK, st, __VA_ARGS__);     \
        }                                                                                          \
        K<LBM_UNWRAP PARAMS, false><<<GRID, BLOCK, 0, st>>>(__VA_ARGS__);                          \
    } while (0)

    static cudaError_t init(const Geom& g, const void* coef, int layout, const void* rho, const void* u, void* dst,
                            cudaStream_t st) {
        const Shape sh = shape_for(g, g.nz - 2 * LBM_SLAB);
        const CF& cf = *static_cast<const CF*>(coef);
        auto r = static_cast<const T*>(rho);
        auto uu = static_cast<const T*>(u);
        const auto o = mpl(dst, g);
        const bool m = g.link != nullptr;
        if (layout == LAYOUT_PULL) {
            if (m)
                k_init<Q, S, true, LAYOUT_PULL><<<sh.grid, sh.block, 0, st>>>(g, cf, r, uu, o);
            else
                k_init<Q, S, false, LAYOUT_PULL><<<sh.grid, sh.block, 0, st>>>(g, cf, r, uu, o);
        } else {
            if (m)
                k_init<Q, S, true, LAYOUT_LOCAL><<<sh.grid, sh.block, 0, st>>>(g, cf, r, uu, o);
            else
                k_init<Q, S, false, LAYOUT_LOCAL><<<sh.grid, sh.block, 0, st>>>(g, cf, r, uu, o);
        }
        return cudaGetLastError();
    }

    // Two cells per thread pay off where the one-cell kernel is instruction-bound: FP16 storage
    // without walls (measured at 256^3: D3Q19 0.61 -> 0.82, D3Q27 0.70 -> 0.83 of the copy peak,
    // the D3Q27 kernels in 128-thread blocks, see pair_threads).
    // FP32 storage is at the bandwidth bound with one cell per thread already, and the wall
    // variants lose occupancy.
    static bool pairs(const Geom& g) { return S == 3 && !g.link && (g.nx % 2) == 0; }
    // Four cells per thread (lbm_quads.cuh) for FP16 D2Q9 / D3Q19 without walls when every warp of
    // a row is full (nx a multiple of 128): measured at 256^3 / 512^3 pull 0.84 -> 0.93 / 0.86 ->
    // 0.96 of the copy peak, AA 0.79 -> 0.84 / 0.81 -> 0.86; at 64^3 (16 threads per row, half of
    // every warp idle) the two-cell kernels stay faster. D3Q27 would need 108 live FP32
    // populations per thread and stays at two cells.
    static bool quads(const Geom& g) { return S == 3 && Q != 27 && !g.link && (g.nx % 128) == 0; }

    // Rows of odd length, FP16 storage without walls: two cells of a row per thread (lbm_cells2.cuh).
    // In small 2D boxes half the threads leave SMs without work (301 x 250 2.2 -> 2.4 us a step). For the
    // scalar there is no such kernel: its rows of odd length run one cell per thread.
    static bool odd_rows(const Geom& g) {
        return S == 3 && !g.link && (g.nx % 2) == 1 && g.nx >= 3 && (Q != 9 || g.N >= 150000u);
    }
    static unsigned blocks_rows2(const Geom& g) {
        const unsigned long long t = (unsigned long long)((g.nx + 1) / 2) * g.ny * (g.nz - 2 * LBM_SLAB);
        return (unsigned)((t + CELLS2_THREADS - 1) / CELLS2_THREADS);
    }

    // Block of the list kernels, as in shape_step: porous D3Q27 256^3 FP32 509 -> 499 us a step, FP16 AA 351 ->
    // 346, 160^3 FP16 pull 103 -> 99; only the D3Q27 FP16 pull step of large boxes is faster with 256 (256^3
    // 432 against 451).
    static constexpr unsigned LIST_THREADS = 128;
    static unsigned pull_list_threads(unsigned long long cells) {
        return Q == 27 && sizeof(ST) == 2 && cells > 8000000ull ? 256u : LIST_THREADS;
    }
    // Block of a one-cell step. 128 threads even out the blocks of an SM sooner than 256: us a step, D3Q19
    // FP32 AA 64^3 6.3 -> 6.1, 96 x 88 x 80 13.5 -> 12.9, 384^3 1368 -> 1350; D3Q27 FP32 75^3 15.4 -> 14.4,
    // porous AA 160^3 148 -> 142, scalar 64 x 70 x 60 7.5 -> 7.1. D3Q27 boxes without walls beyond 2M cells are
    // as fast or 1 % faster with 256 outside the flow's AA steps (pull 256^3 522 against 527).
    // FP64 steps are bound by the FP64 pipes, one per scheduler of an SM, so they run single warps as
    // blocks, which spread evenly: us a step with 32, 64, 128 and 256 threads, D2Q9 64^2 5.3, 5.2, 5.5, 9.5;
    // 96 x 198 5.8, 5.7, 5.7, 9.5; D3Q19 33 x 29 x 41 34.3, 34.3, 42.2, 43.3; D3Q27 42 x 35 x 22 33.9, 36.0,
    // 36.2, 47.7; from 64^3 up they are alike.
    // A box too tall for such blocks (grid.y) keeps 256.
    static Shape shape_step(const Geom& g, bool flow_aa = false) {
        const int nzp = g.nz - 2 * LBM_SLAB;
        const bool wide = Q == 27 && !g.link && g.N > (1u << 21) && !flow_aa;
        const Shape sh = shape_for(g, nzp, S == 1 ? 32 : wide ? 256 : 128);
        return sh.grid.y <= 65535u ? sh : shape_for(g, nzp);
    }

    // D2Q9 FP64: four lanes per cell (lbm_lanes.cuh) while every scheduler (four per SM) gets one warp
    // at most; with two, 80^2 takes the 5.3 us of one lane per cell, and 96 x 80 5.9 instead of 5.3.
    static constexpr bool LANES = S == 1 && Q == 9;
    static bool lanes(const Geom& g) { return !g.link && (g.N + 7) / 8 <= 4u * (uint32_t)sm_count(); }

    static cudaError_t step_pull(const Geom& g, const void* coef, const void* src, void* dst, int* flag,
                                 cudaStream_t st) {
        const Shape sh = shape_step(g);
        const CF& cf = *static_cast<const CF*>(coef);
        const auto a = cpl(src, g);
        const auto b = mpl(dst, g);
        if constexpr (S == 3) {  // pairs(g) holds for FP16 r-shifted storage only
            if constexpr (Q != 27) {
                if (quads(g)) {
                    const Shape sq = shape_quads(g);
                    k_step_pull4<Q><<<sq.grid, sq.block, 0, st>>>(g, cf, VelField<float>{}, a, b, flag);
                    return cudaGetLastError();
                }
            }
            if (pairs(g)) {
                const Shape sp = shape_pairs(g, pair_threads<Q>());
                LBM_EARLY(k_step_pull2, (Q, S, false, false), sp.grid, sp.block, g, cf, VelField<float>{}, a, b, flag);
                return cudaGetLastError();
            }
            if (odd_rows(g)) {
                LBM_EARLY(k_step_pull_rows2, (Q), blocks_rows2(g), CELLS2_THREADS, g, cf, a, b, flag);
                return cudaGetLastError();
            }
        }
        if constexpr (LANES) {
            if (lanes(g)) {
                k_step_lanes<LAYOUT_PULL><<<(g.N + 7) / 8, 32, 0, st>>>(g, cf, static_cast<const double*>(src),
                                                                       static_cast<double*>(dst), flag);
                return cudaGetLastError();
            }
        }
        if (g.link)
            LBM_EARLY(k_step_pull, (Q, S, true), sh.grid, sh.block, g, cf, a, b, flag);
        else
            LBM_EARLY(k_step_pull, (Q, S, false), sh.grid, sh.block, g, cf, a, b, flag);
        return cudaGetLastError();
    }

    static cudaError_t step_aa(const Geom& g, const void* coef, int odd, const void* src, void* dst, int* flag,
                               cudaStream_t st) {
        const Shape sh = shape_step(g, true);
        const CF& cf = *static_cast<const CF*>(coef);
        const auto a = cpl(src, g);
        const auto b = mpl(dst, g);
        if constexpr (S == 3) {  // pairs(g) holds for FP16 r-shifted storage only
            // no walls (see pairs())
            if constexpr (Q != 27) {
                if (quads(g)) {
                    const Shape sq = shape_quads(g);
                    if (odd)
                        k_step_aa_odd4<Q><<<sq.grid, sq.block, 0, st>>>(g, cf, VelField<float>{}, a, b, flag);
                    else
                        k_step_aa_even4<Q><<<sq.grid, sq.block, 0, st>>>(g, cf, VelField<float>{}, a, b, flag);
                    return cudaGetLastError();
                }
            }
            if (pairs(g)) {
                const Shape sp = shape_pairs(g, pair_threads<Q>());
                if (odd)
                    LBM_EARLY(k_step_aa_odd2, (Q, S, false), sp.grid, sp.block, g, cf, VelField<float>{}, a, b, flag);
                else
                    LBM_EARLY(k_step_aa_even2, (Q, S, false, false), sp.grid, sp.block, g, cf, VelField<float>{}, a,
                              b, flag);
                return cudaGetLastError();
            }
            if (odd_rows(g)) {
                if (odd)
                    LBM_EARLY(k_step_aa_rows2, (Q, 1), blocks_rows2(g), CELLS2_THREADS, g, cf, a, b, flag);
                else
                    LBM_EARLY(k_step_aa_rows2, (Q, 0), blocks_rows2(g), CELLS2_THREADS, g, cf, a, b, flag);
                return cudaGetLastError();
            }
        }
        if constexpr (LANES) {
            if (lanes(g)) {
                const auto from = static_cast<const double*>(src);
                const auto to = static_cast<double*>(dst);
                if (odd)
                    k_step_lanes<LAYOUT_AAODD><<<(g.N + 7) / 8, 32, 0, st>>>(g, cf, from, to, flag);
                else
                    k_step_lanes<LAYOUT_LOCAL><<<(g.N + 7) / 8, 32, 0, st>>>(g, cf, from, to, flag);
                return cudaGetLastError();
            }
        }
        if (g.link) {
            if (odd)
                LBM_EARLY(k_step_aa, (Q, S, true, 1), sh.grid, sh.block, g, cf, a, b, flag);
            else
                LBM_EARLY(k_step_aa, (Q, S, true, 0), sh.grid, sh.block, g, cf, a, b, flag);
        } else {
            if (odd)
                LBM_EARLY(k_step_aa, (Q, S, false, 1), sh.grid, sh.block, g, cf, a, b, flag);
            else
                LBM_EARLY(k_step_aa, (Q, S, false, 0), sh.grid, sh.block, g, cf, a, b, flag);
        }
        return cudaGetLastError();
    }

    // the storages and lattices whose contexts with walls have a sector list (lbm_create_ex)
    static constexpr bool SECTORS = sizeof(ST) == 2 || (Q == 27 && sizeof(ST) == 4);
    static cudaError_t step_pull_sectors(const Geom& g, const void* coef, const CellList& L, const void* src,
                                         void* dst, int* flag, cudaStream_t st) {
        if constexpr (SECTORS) {
            if (L.count == 0) return cudaSuccess;
            const CF& cf = *static_cast<const CF*>(coef);
            const unsigned long long threads = (unsigned long long)L.count * (32ull / sizeof(ST));  // a sector each
            const unsigned bt = pull_list_threads(threads);
            k_step_pull_sectors<Q, S><<<(unsigned)((threads + bt - 1) / bt), bt, 0, st>>>(g, cf, L, cpl(src, g),
                                                                                          mpl(dst, g), flag);
            return cudaGetLastError();
        }
        return cudaErrorNotSupported;
    }

    static cudaError_t step_aa_list(const Geom& g, const void* coef, const CellList& L, int odd, const void* src,
                                    void* dst, int* flag, cudaStream_t st) {
        if constexpr (sizeof(ST) == 2) {
            if (L.count == 0) return cudaSuccess;
            const CF& cf = *static_cast<const CF*>(coef);
            const unsigned nb = (L.count + LIST_THREADS - 1) / LIST_THREADS;
            if (odd)
                k_step_aa_list<Q, S, 1><<<nb, LIST_THREADS, 0, st>>>(g, cf, L, cpl(src, g), mpl(dst, g), flag);
            else
                k_step_aa_list<Q, S, 0><<<nb, LIST_THREADS, 0, st>>>(g, cf, L, cpl(src, g), mpl(dst, g), flag);
            return cudaGetLastError();
        }
        return cudaErrorNotSupported;
    }

// Expands to the three layouts times mask / no mask for a kernel template K<Q, S, MASK, LAYOUT>.
#define LBM_BY_LAYOUT(K, ...)                                                                      \
    do {                                                                                           \
        const bool m_ = g.link != nullptr;                                                         \
        if (layout == LAYOUT_PULL) {                                                               \
            if (m_) K<Q, S, true, LAYOUT_PULL><<<sh.grid, sh.block, 0, st>>>(__VA_ARGS__);         \
            else K<Q, S, false, LAYOUT_PULL><<<sh.grid, sh.block, 0, st>>>(__VA_ARGS__);           \
        } else if (layout == LAYOUT_AAODD) {                                                       \
            if (m_) K<Q, S, true, LAYOUT_AAODD><<<sh.grid, sh.block, 0, st>>>(__VA_ARGS__);        \
            else K<Q, S, false, LAYOUT_AAODD><<<sh.grid, sh.block, 0, st>>>(__VA_ARGS__);          \
        } else {                                                                                   \
            if (m_) K<Q, S, true, LAYOUT_LOCAL><<<sh.grid, sh.block, 0, st>>>(__VA_ARGS__);        \
            else K<Q, S, false, LAYOUT_LOCAL><<<sh.grid, sh.block, 0, st>>>(__VA_ARGS__);          \
        }                                                                                          \
    } while (0)
#define LBM_BY_LAYOUT_EARLY(K, ...)                                                                \
    do {                                                                                           \
        const bool m_ = g.link != nullptr;                                                         \
        if (layout == LAYOUT_PULL) {                                                               \
            if (m_) LBM_EARLY(K, (Q, S, true, LAYOUT_PULL), sh.grid, sh.block, __VA_ARGS__);       \
            else LBM_EARLY(K, (Q, S, false, LAYOUT_PULL), sh.grid, sh.block, __VA_ARGS__);         \
        } else if (layout == LAYOUT_AAODD) {                                                       \
            if (m_) LBM_EARLY(K, (Q, S, true, LAYOUT_AAODD), sh.grid, sh.block, __VA_ARGS__);      \
            else LBM_EARLY(K, (Q, S, false, LAYOUT_AAODD), sh.grid, sh.block, __VA_ARGS__);        \
        } else {                                                                                   \
            if (m_) LBM_EARLY(K, (Q, S, true, LAYOUT_LOCAL), sh.grid, sh.block, __VA_ARGS__);      \
            else LBM_EARLY(K, (Q, S, false, LAYOUT_LOCAL), sh.grid, sh.block, __VA_ARGS__);        \
        }                                                                                          \
    } while (0)

    static cudaError_t moments(const Geom& g, const void* coef, int layout, const void* src, void* rho, void* u,
                               void* Pi, void* f, cudaStream_t st) {
        const Shape sh = shape_for(g, g.nz - 2 * LBM_SLAB);
        const CF& cf = *static_cast<const CF*>(coef);
        LBM_BY_LAYOUT_EARLY(k_moments, g, cf, cpl(src, g), static_cast<T*>(rho), static_cast<T*>(u),
                      static_cast<T*>(Pi), static_cast<T*>(f));
        return cudaGetLastError();
    }

    static cudaError_t totals(const Geom& g, const void* coef, int layout, const void* src, double* part, int* flag,
                              cudaStream_t st) {
        const Shape sh = shape_for(g, g.nz - 2 * LBM_SLAB);
        const CF& cf = *static_cast<const CF*>(coef);
        LBM_BY_LAYOUT(k_totals, g, cf, cpl(src, g), part, flag);
        return cudaGetLastError();
    }

    static cudaError_t adj_seed(const Geom& g, const void* coef, int layout, const void* src, const void* grad,
                                void* lam, cudaStream_t st) {
        const Shape sh = shape_for(g, g.nz - 2 * LBM_SLAB);
        const CF& cf = *static_cast<const CF*>(coef);
        LBM_BY_LAYOUT(k_adj_seed, g, cf, cpl(src, g), static_cast<const T*>(grad), mfl(lam, g));
        return cudaGetLastError();
    }

    static cudaError_t adj_step(const Geom& g, const void* coef, int layout, const void* src, const void* lam_next,
                                void* lam, double* gpart, cudaStream_t st) {
        const Shape sh = shape_for(g, g.nz - 2 * LBM_SLAB);
        const CF& cf = *static_cast<const CF*>(coef);
        if constexpr (S == 3 && Q != 27) {  // FP16 storage without walls: two cells per thread (lbm_adjoint2.cuh;
            // D3Q27 stays one cell per thread: at 128 registers the pair kernel would spill)
            const Shape sp = shape_pairs(g, 128);  // the block shape k_adj_step2 is built for
            if (!g.link && (g.nx % 2) == 0 && sp.nblocks <= sh.nblocks) {  // records fit the per-cell grid's
                const auto a = cpl(src, g);
                const auto ln = cfl(lam_next, g);
                const auto l = mfl(lam, g);
                if (layout == LAYOUT_PULL)
                    k_adj_step2<Q, S, LAYOUT_PULL><<<sp.grid, sp.block, 0, st>>>(g, cf, a, ln, l, gpart);
                else if (layout == LAYOUT_AAODD)
                    k_adj_step2<Q, S, LAYOUT_AAODD><<<sp.grid, sp.block, 0, st>>>(g, cf, a, ln, l, gpart);
                else
                    k_adj_step2<Q, S, LAYOUT_LOCAL><<<sp.grid, sp.block, 0, st>>>(g, cf, a, ln, l, gpart);
                return cudaGetLastError();
            }
        }
        LBM_BY_LAYOUT_EARLY(k_adj_step, g, cf, cpl(src, g), cfl(lam_next, g), mfl(lam, g), gpart);
        return cudaGetLastError();
    }
#undef LBM_BY_LAYOUT
#undef LBM_BY_LAYOUT_EARLY

    static cudaError_t adj_init(const Geom& g, const void* coef, const void* rho0, const void* u0, const void* lam0,
                                void* du0, double* gpart, cudaStream_t st) {
        const Shape sh = shape_for(g, g.nz - 2 * LBM_SLAB);
        const CF& cf = *static_cast<const CF*>(coef);
        k_adj_init<Q, T><<<sh.grid, sh.block, 0, st>>>(g, cf, static_cast<const T*>(rho0), static_cast<const T*>(u0),
                                                       cfl(lam0, g), static_cast<T*>(du0), gpart);
        return cudaGetLastError();
    }

    static cudaError_t link_mask(const Geom& g, const uint8_t* solid, uint32_t* link, cudaStream_t st) {
        const Shape sh = shape_for(g, g.nz - 2 * LBM_SLAB);
        k_link_mask<Q><<<sh.grid, sh.block, 0, st>>>(g, solid, link);
        return cudaGetLastError();
    }

    static VelField<T> vel_field(const void* u, const Geom& g) {
        VelField<T> v{};
        auto p = static_cast<const T*>(u);
        for (int a = 0; a < Lat<Q>::D; ++a) v.p[a] = p ? p + (size_t)a * g.N : nullptr;
        return v;
    }

    static cudaError_t ade_pull(const Geom& g, const void* coef, const void* u, const void* src, void* dst, int* flag,
                                cudaStream_t st) {
        const Shape sh = shape_step(g);
        const CF& cf = *static_cast<const CF*>(coef);
        if constexpr (S == 3) {  // pairs(g) holds for FP16 r-shifted storage only
            if constexpr (Q != 27) {
                if (quads(g)) {
                    const Shape sq = shape_quads(g);
                    k_step_pull4<Q, true><<<sq.grid, sq.block, 0, st>>>(g, cf, vel_field(u, g), cpl(src, g),
                                                                       mpl(dst, g), flag);
                    return cudaGetLastError();
                }
            }
            if (pairs(g)) {
                const Shape sp = shape_pairs(g, pair_threads<Q>());
                LBM_EARLY(k_step_pull2, (Q, S, false, true), sp.grid, sp.block, g, cf, vel_field(u, g), cpl(src, g),
                          mpl(dst, g), flag);
                return cudaGetLastError();
            }
        }
        if (g.link)
            LBM_EARLY(k_ade_pull, (Q, S, true), sh.grid, sh.block, g, cf, vel_field(u, g), cpl(src, g), mpl(dst, g),
                      flag);
        else
            LBM_EARLY(k_ade_pull, (Q, S, false), sh.grid, sh.block, g, cf, vel_field(u, g), cpl(src, g), mpl(dst, g),
                      flag);
        return cudaGetLastError();
    }

    static cudaError_t ade_aa(const Geom& g, const void* coef, const void* u, int odd, const void* src, void* dst,
                              int* flag, cudaStream_t st) {
        const Shape sh = shape_step(g);
        const CF& cf = *static_cast<const CF*>(coef);
        const auto v = vel_field(u, g);
        const auto a = cpl(src, g);
        const auto b = mpl(dst, g);
        if constexpr (S == 3) {  // pairs(g) holds for FP16 r-shifted storage only
            if constexpr (Q != 27) {
                if (quads(g)) {
                    const Shape sq = shape_quads(g);
                    if (odd)
                        k_step_aa_odd4<Q, true><<<sq.grid, sq.block, 0, st>>>(g, cf, v, a, b, flag);
                    else
                        k_step_aa_even4<Q, true><<<sq.grid, sq.block, 0, st>>>(g, cf, v, a, b, flag);
                    return cudaGetLastError();
                }
            }
            if (pairs(g)) {
                const Shape sp = shape_pairs(g, pair_threads<Q>());
                if (odd)
                    LBM_EARLY(k_step_aa_odd2, (Q, S, true), sp.grid, sp.block, g, cf, v, a, b, flag);
                else
                    LBM_EARLY(k_step_aa_even2, (Q, S, false, true), sp.grid, sp.block, g, cf, v, a, b, flag);
                return cudaGetLastError();
            }
        }
        if (g.link) {
            if (odd)
                LBM_EARLY(k_ade_aa, (Q, S, true, 1), sh.grid, sh.block, g, cf, v, a, b, flag);
            else
                LBM_EARLY(k_ade_aa, (Q, S, true, 0), sh.grid, sh.block, g, cf, v, a, b, flag);
        } else {
            if (odd)
                LBM_EARLY(k_ade_aa, (Q, S, false, 1), sh.grid, sh.block, g, cf, v, a, b, flag);
            else
                LBM_EARLY(k_ade_aa, (Q, S, false, 0), sh.grid, sh.block, g, cf, v, a, b, flag);
        }
        return cudaGetLastError();
    }

    static cudaError_t ade_pull_sectors(const Geom& g, const void* coef, const CellList& L, const void* u,
                                        const void* src, void* dst, int* flag, cudaStream_t st) {
        if constexpr (SECTORS) {
            if (L.count == 0) return cudaSuccess;
            const CF& cf = *static_cast<const CF*>(coef);
            const unsigned long long threads = (unsigned long long)L.count * (32ull / sizeof(ST));  // a sector each
            const unsigned nb = (unsigned)((threads + LIST_THREADS - 1) / LIST_THREADS);
            k_ade_pull_sectors<Q, S><<<nb, LIST_THREADS, 0, st>>>(g, cf, L, vel_field(u, g), cpl(src, g), mpl(dst, g),
                                                                  flag);
            return cudaGetLastError();
        }
        return cudaErrorNotSupported;
    }

    // FP32 storage on D3Q19 in whole boxes (lbm_twice.cuh)
    static constexpr bool TWICE = (S == 0 || S == 2) && Q == 19 && !LBM_SLAB;
    static int sm_count() {
        int dev = 0, sms = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
            (void)cudaGetLastError();
            return 0;
        }
        return sms;
    }
    // D2Q9 FP32 storage in whole boxes (lbm_plane.cuh)
    static constexpr bool PLANE = (S == 0 || S == 2) && Q == 9;
    static Several plan_several(const Geom& g) {
        Several s{};
        s.sms = sm_count();
        if constexpr (TWICE) s.twice = !g.link && twice_pays(g, s.sms, s.tiles);
        return s;
    }
    static int steps_at_once(const Geom& g, const Several& s, long long left) {
        if (g.link || left < 2) return 1;
        if constexpr (TWICE) return s.twice ? 2 : 1;
        if constexpr (PLANE) return plane_steps(g, s.sms, left);
        return 1;
    }

    static cudaError_t step_several(const Geom& g, const void* coef, const Several& s, int steps, const void* src,
                                    void* dst, int* flag, cudaStream_t st) {
        const CF& cf = *static_cast<const CF*>(coef);
        if constexpr (TWICE) {
            const Tiles& t = s.tiles;
            const cudaError_t e = cudaFuncSetAttribute(k_step_twice<Q, S>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                       twice_smem<Q>());
            if (e != cudaSuccess) return e;
            const long long n = t.chunks ? (long long)t.tiles * t.chunks : ((long long)t.tiles * g.nz + t.run - 1) / t.run;
            k_step_twice<Q, S><<<(unsigned)n, TWICE_THREADS, twice_smem<Q>(), st>>>(g, cf, t, cpl(src, g), mpl(dst, g),
                                                                                    flag);
            return cudaGetLastError();
        }
        if constexpr (PLANE) {
            return launch_planes<S>(g, cf, s.sms, steps, cpl(src, g), mpl(dst, g), flag, st);
        }
        return cudaErrorNotSupported;
    }

    static cudaError_t step_aa_even_sectors(const Geom& g, const void* coef, const SectorList& L, const void* src,
                                            void* dst, int* flag, cudaStream_t st) {
        if constexpr (S == 3) {
            if (L.count == 0) return cudaSuccess;
            const unsigned nb = (unsigned)((L.count * 8ull + CELLS2_THREADS - 1) / CELLS2_THREADS);
            k_step_aa_even_sectors2<Q><<<nb, CELLS2_THREADS, 0, st>>>(g, *static_cast<const CF*>(coef), L, cpl(src, g),
                                                                     mpl(dst, g), flag);
            return cudaGetLastError();
        }
        return cudaErrorNotSupported;
    }

    static const Ops& ops() {
        static const Ops o = {&init,     &step_pull, &step_aa,   &step_pull_sectors, &step_aa_list, &moments,
                              &totals,   &adj_seed,  &adj_step,  &adj_init,          &link_mask,    &ade_pull,
                              &ade_aa,   &ade_pull_sectors, &step_aa_even_sectors, &plan_several, &steps_at_once,
                              &step_several};
        return o;
    }
};

}  // namespace LBM_VARIANT
}  // namespace lbm
