// D2Q9 FP64 steps of the smallest boxes without walls: four lanes per cell.
//
// A warp's FP64 instruction takes 64 clocks of its scheduler's pipe whatever its lanes hold, so a box
// with fewer warps than the GPU has schedulers takes one warp's 110 of them, 3.5 us, however small it
// is. Here each lane owns one direction pair of a cell: the moments come from two exchanges within
// the four lanes, and a lane evaluates the equilibrium of its pair only, about 55 instructions in
// four times as many warps: 64^2 5.3 -> 4.2 us a step, 33 x 60 5.3 -> 3.9.
#pragma once
#include "lbm_kernels.cuh"

namespace lbm {
inline namespace LBM_VARIANT {

__device__ __forceinline__ double sum_of_four(double v) {
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    return v + __shfl_xor_sync(0xffffffffu, v, 2);
}

// bgk64<9> with the pair (+v, -v) of lane j in f and g (see there).
__device__ __forceinline__ void bgk_lane(const Coef<double>& cf, int j, double& rest, double& f, double& g, double& rho,
                                         double& usum) {
    const double r0 = cf.so[0], r = j == 0 ? cf.so[1] : j == 1 ? cf.so[3] : j == 2 ? cf.so[5] : cf.so[7];
    const double d0 = rest - r0, o = f - g, p = fma(2.0, g - r, o);
    const double drho = d0 + sum_of_four(p), s = cf.rho0 + drho;
    const double jx = sum_of_four(j == 1 ? 0.0 : o), jy = sum_of_four(j == 0 ? 0.0 : j == 3 ? -o : o);
    const double inv = 1.0 / s, ux = jx * inv, uy = jy * inv;
    const double om1 = 1.0 - cf.omega, half = 0.5 * om1, omrho = cf.omega * s, omdrho = cf.omega * drho;
    const double usq = fma(ux, ux, uy * uy);
    const double kx = fma(cf.K[0], ux, cf.K[3] * uy), ky = fma(cf.K[3], ux, cf.K[1] * uy);
    const double r45 = 4.5 * omrho, r15 = r45 * usq * (1.0 / 3.0);
    const double w = j < 2 ? weight<9>(1) : weight<9>(5);
    const double A = j == 0 ? cf.A[1] : j == 1 ? cf.A[3] : j == 2 ? cf.A[5] : cf.A[7];
    const double B = j == 0 ? cf.B[1] : j == 1 ? cf.B[3] : j == 2 ? cf.B[5] : cf.B[7];
    // c.u and c.K~u of v = (1, 0), (0, 1), (1, 1), (1, -1)
    const double uc = (j == 1 ? 0.0 : ux) + (j == 0 ? 0.0 : j == 3 ? -uy : uy);
    const double ck = (j == 1 ? 0.0 : kx) + (j == 0 ? 0.0 : j == 3 ? -ky : ky);
    const double b = w * (cf.c3 * omrho), uc2 = uc * uc;
    const double E = fma(half, p, fma(w * r45, uc2, fma(omdrho, A, -(w * r15))));
    const double O = fma(half, o, fma(uc, fma(b, uc2 - usq, omrho * B), -((b + b) * ck)));
    rest = fma(om1, d0, fma(omdrho, cf.A[0], -(weight<9>(0) * r15))) + r0;
    f = (E + O) + r;
    g = (E - O) + r;
    rho = s;
    usum = ux + uy;
}

// LAYOUT of the state that is read: PULL (two arrays), LOCAL (even AA step), AAODD (odd AA step).
template <int LAYOUT>
__global__ void __launch_bounds__(32)
    k_step_lanes(Geom g, Coef<double> cf, const double* src, double* dst, int* __restrict__ flag) {
    const uint32_t t = blockIdx.x * 32u + threadIdx.x;
    const bool in = t / 4u < g.N;
    const uint32_t n = in ? t / 4u : g.N - 1u;  // the spare lanes of the last warp go along and write nothing
    const int j = (int)(t & 3u);
    const uint32_t nx = (uint32_t)g.nx, ny = (uint32_t)g.ny, y = n / nx, x = n - y * nx;
    // the neighbours x + v and x - v, v = (j != 1, 0 / 1 / 1 / -1)
    const uint32_t xp = j == 1 ? x : x + 1u == nx ? 0u : x + 1u, xm = j == 1 ? x : x == 0u ? nx - 1u : x - 1u;
    const uint32_t yu = y + 1u == ny ? 0u : y + 1u, yd = y == 0u ? ny - 1u : y - 1u;
    const uint32_t yp = j == 0 ? y : j == 3 ? yd : yu, ym = j == 0 ? y : j == 3 ? yu : yd;
    const uint32_t plus = xp + nx * yp, minus = xm + nx * ym;
    const size_t N = g.N, pf = (size_t)(2 * j + 1) * N, pg = pf + N;  // planes of +v and -v
    double rest = src[n];
    double f = LAYOUT == LAYOUT_PULL ? src[pf + minus] : LAYOUT == LAYOUT_LOCAL ? src[pf + n] : src[pg + minus];
    double h = LAYOUT == LAYOUT_PULL ? src[pg + plus] : LAYOUT == LAYOUT_LOCAL ? src[pg + n] : src[pf + plus];
    double rho, usum;
    bgk_lane(cf, j, rest, f, h, rho, usum);
    __syncwarp();  // in place, lane 0 writes the rest population that the cell's other lanes have read
    if (!in) return;
    if (!(rho > 0.0) || !isfinite(usum)) *flag = 1;
    if (j == 0) dst[n] = rest;
    dst[LAYOUT == LAYOUT_PULL ? pf + n : LAYOUT == LAYOUT_LOCAL ? pg + n : pf + plus] = f;
    dst[LAYOUT == LAYOUT_PULL ? pg + n : LAYOUT == LAYOUT_LOCAL ? pf + n : pg + minus] = h;
}

}  // namespace LBM_VARIANT
}  // namespace lbm
