// Several time steps per launch for FP32 storage in 2D without walls (D2Q9, pull scheme).
//
// A step of a small 2D box is a launch: D2Q9 96 x 80 takes 1.6 us whatever it computes. Here a block
// owns a tile of W x H cells and carries it through T steps in shared memory: the first step
// gathers from global memory on the tile and T - 1 rings of neighbours around it, every further
// step works from shared memory on one ring less, and the last one stores the tile. Rings are
// computed by several blocks, from the same values in the same order, so the bits are those of T
// launches (the packed collision of lbm_cells2.cuh: a thread takes the cells k and k + half of the
// region). What bounds a step now is one warp's way through the collision, about 320 instructions at
// 4 to 5 clocks each; in large boxes, where DRAM is 16 % busy, the same with the barriers between
// the steps. One rolled loop over the steps is slower (96 x 80 0.79 -> 0.91 us a step).
#pragma once
#include <algorithm>

#include "lbm_cells2.cuh"

namespace lbm {
inline namespace LBM_VARIANT {

template <int W, int H, int T>
constexpr int plane_smem() {
    return 2 * 9 * (W + 2 * (T - 1)) * (H + 2 * (T - 1)) * (int)sizeof(float);
}

// Offsets of the nine pull sources of the cell at (x, y), wrapped into the box.
struct PlaneCell {
    uint32_t X[3], R[3];
    __device__ __forceinline__ PlaneCell(const Geom& g, int x, int y) {
        x %= g.nx;  // a box may be smaller than the rings
        y %= g.ny;
        if (x < 0) x += g.nx;
        if (y < 0) y += g.ny;
        const uint32_t nx = (uint32_t)g.nx;
        X[0] = x + 1 == g.nx ? 0u : (uint32_t)(x + 1);
        X[1] = (uint32_t)x;
        X[2] = x == 0 ? nx - 1u : (uint32_t)(x - 1);
        R[0] = nx * (uint32_t)(y + 1 == g.ny ? 0 : y + 1);
        R[1] = nx * (uint32_t)y;
        R[2] = nx * (uint32_t)(y == 0 ? g.ny - 1 : y - 1);
    }
    __device__ __forceinline__ uint32_t from(Vec3 v) const { return X[v.x + 1] + R[v.y + 1]; }
};

template <int S, int W, int H, int T, int THREADS>
__global__ void __launch_bounds__(THREADS)
    k_steps_plane(Geom g, Coef<float> cf, const Planes<const float> src, const Planes<float> dst, int* __restrict__ flag) {
    constexpr int EW = W + 2 * (T - 1), EH = H + 2 * (T - 1), E = EW * EH;
    extern __shared__ float sh[];
    const int x0 = blockIdx.x * W - (T - 1), y0 = blockIdx.y * H - (T - 1);  // cell of the extended tile's corner
    bool bad = false;
    wait_previous<true>();
    for (int k = threadIdx.x; k < (E + 1) / 2; k += THREADS) {
        const int kb = min(k + (E + 1) / 2, E - 1);
        const PlaneCell a(g, x0 + k % EW, y0 + k / EW), b(g, x0 + kb % EW, y0 + kb / EW);
        F2 d[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const Vec3 v = vel<9>(i);
            d[i] = to_shifted2<S>(f2(src.p[i][a.from(v)], src.p[i][b.from(v)]), cf.so[i]);
        }
        const Macro2 m = bgk<9, S>(cf, d);
        bad |= bad_pair(m, true, true);
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const F2 o = from_shifted2<S>(d[i], cf.so[i]);
            sh[i * E + k] = o.v.x;
            sh[i * E + kb] = o.v.y;
        }
    }
#pragma unroll
    for (int t = 2; t <= T; ++t) {
        __syncthreads();
        const int m0 = t - 1, w = EW - 2 * m0, n = w * (EH - 2 * m0), half = (n + 1) / 2;  // margin, the region's cells
        const float* from = sh + (t & 1) * (9 * E);
        float* to = sh + ((t & 1) ^ 1) * (9 * E);
        for (int k = threadIdx.x; k < half; k += THREADS) {
            const int kb = min(k + half, n - 1);
            const int xa = m0 + k % w, ya = m0 + k / w, xb = m0 + kb % w, yb = m0 + kb / w;
            const int na = ya * EW + xa, nb = yb * EW + xb;
            F2 d[9];
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                const Vec3 v = vel<9>(i);
                const float* q = from + i * E - v.y * EW - v.x;
                d[i] = to_shifted2<S>(f2(q[na], q[nb]), cf.so[i]);
            }
            const Macro2 m = bgk<9, S>(cf, d);
            bad |= bad_pair(m, true, true);
            if (t < T) {
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    const F2 o = from_shifted2<S>(d[i], cf.so[i]);
                    to[i * E + na] = o.v.x;
                    to[i * E + nb] = o.v.y;
                }
            } else {
                const bool wa = x0 + xa < g.nx && y0 + ya < g.ny, wb = x0 + xb < g.nx && y0 + yb < g.ny;
                const uint32_t ga = (uint32_t)(x0 + xa) + (uint32_t)g.nx * (uint32_t)(y0 + ya);
                const uint32_t gb = (uint32_t)(x0 + xb) + (uint32_t)g.nx * (uint32_t)(y0 + yb);
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    const F2 o = from_shifted2<S>(d[i], cf.so[i]);
                    if (wa) dst.p[i][ga] = o.v.x;
                    if (wb) dst.p[i][gb] = o.v.y;
                }
            }
        }
    }
    if (bad) *flag = 1;
}

template <int S, int W, int H, int T, int THREADS>
cudaError_t launch_plane(const Geom& g, const Coef<float>& cf, const Planes<const float>& src, const Planes<float>& dst,
                         int* flag, cudaStream_t st) {
    const auto k = k_steps_plane<S, W, H, T, THREADS>;
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, plane_smem<W, H, T>());
    if (e != cudaSuccess) return e;
    const dim3 grid((g.nx + W - 1) / W, (g.ny + H - 1) / H);
    return launch_after_shared(k, grid, THREADS, st, plane_smem<W, H, T>(), g, cf, src, dst, flag);
}

// Tile and steps of one launch, W x H x T. A small box takes the smallest tile that gives every SM one
// block at most (8 x 8, 16 x 8, 16 x 16 cells; more blocks than SMs run one after the other), eight
// steps at a time; a larger one 16 x 16 cells and four steps, whose rings cost 1.6 times the cells
// instead of 2.9 and whose blocks of 256 threads fit three to an SM (32 x 32 cells in blocks of 512:
// 4096^2 162 us a step, 64 x 16: 154). Measured, us a step, one step a launch -> this: 64^2 1.68 ->
// 0.78, 96 x 80 1.82 -> 0.78, 128^2 1.68 -> 0.91, 200 x 150 1.82 -> 1.04, 256^2 2.07 -> 1.44, 512^2
// 3.88 -> 3.06, 700^2 5.68 -> 5.02, 1024^2 10.7 -> 9.9, 2048^2 51.4 -> 37.3, 4096^2 194 -> 147.
inline int plane_tile(const Geom& g, int sms) {
    const long long per_sm = ((long long)g.N + std::max(1, sms) - 1) / std::max(1, sms);
    return per_sm <= 64 ? 0 : per_sm <= 128 ? 1 : per_sm <= 256 ? 2 : 3;
}
inline int plane_steps(const Geom& g, int sms, long long left) {
    if (left >= 8 && plane_tile(g, sms) < 3) return 8;
    return left >= 4 ? 4 : 1;
}
template <int S>
cudaError_t launch_planes(const Geom& g, const Coef<float>& cf, int sms, int steps, const Planes<const float>& src,
                          const Planes<float>& dst, int* flag, cudaStream_t st) {
    const int tile = plane_tile(g, sms);
    if (steps == 8)
        return tile == 0   ? launch_plane<S, 8, 8, 8, 256>(g, cf, src, dst, flag, st)
               : tile == 1 ? launch_plane<S, 16, 8, 8, 352>(g, cf, src, dst, flag, st)
                           : launch_plane<S, 16, 16, 8, 480>(g, cf, src, dst, flag, st);
    return launch_plane<S, 16, 16, 4, 256>(g, cf, src, dst, flag, st);
}

}  // namespace LBM_VARIANT
}  // namespace lbm
