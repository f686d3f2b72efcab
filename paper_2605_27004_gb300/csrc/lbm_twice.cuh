// Two time steps per launch for FP32 storage on D3Q19 without walls (pull scheme).
//
// One step per launch is bound by DRAM: every population is read and written once per step (the
// one-cell kernels run at 1.03 of the copy bandwidth at 256^3). Here a block owns up to 64 x 9 cells
// of x and y and walks along z. For each plane it first computes the collided populations of the
// intermediate step on its cells and one ring of neighbours, straight into shared memory, and then
// the second step from there, so the intermediate state never reaches DRAM: at 256^3 one launch of
// two steps moves 2.56 GB, as much as one step did.
//
// Rows: one warp per row of the ring-extended tile, lane l holding the cells l and l + 32 as one
// packed pair (consecutive lanes are consecutive cells, so that every access is coalesced and free
// of bank conflicts at any alignment of the row); one more warp computes the two cells left and
// right of every row. Shared memory keeps, per direction, the planes the second step still needs:
// one of c_z = -1, two of c_z = 0, three of c_z = +1; directions along z stay in registers. The
// loads of the next plane are in flight (in registers) while the second step works on this one.
//
// What bounds it now: the FP32 pipe (49 % busy) and the latency of the two collisions between the
// two barriers a plane takes, at three warps per scheduler; DRAM is 51 % busy. One block of 12 warps
// at 164 registers measured best: with 16 rows the loads in flight no longer fit the L1 beside the
// shared memory (256^3: 355 us a step), two blocks of 8 warps 346 us, one barrier a plane with
// deeper buffers 327 us, this form 308 us; one step a launch 368 us. 384^3: 1239 -> 1017 us,
// 512^3: 2952 -> 2309 us a step. D3Q27 (7 rows at 254 registers, 507 to 529 against 521 us) gains
// nothing and stays at one step a launch.
//
// The arithmetic is that of the one-cell kernels operation for operation (bgk), so that two
// steps in one launch give the bits of two launches.
#pragma once
#include "lbm_cells2.cuh"

namespace lbm {
inline namespace LBM_VARIANT {

constexpr int TWICE_ROWS = 11;        // rows of a block's ring-extended tile
constexpr int TWICE_W = 64;           // cells of a row of the tile, at most
constexpr int TWICE_P = TWICE_W + 2;  // a row in shared memory: the ring's left cell, the row, the right cell
constexpr int TWICE_THREADS = 32 * (TWICE_ROWS + 1);
// Directions along the z axis (and rest): they stay in the registers of the thread that owns the column.
template <int Q>
__host__ __device__ constexpr bool twice_column(int i) {
    return vel<Q>(i).x == 0 && vel<Q>(i).y == 0;
}
// Slot of direction i among the directions of its c_z, and the planes kept per c_z.
template <int Q>
__host__ __device__ constexpr int twice_slot(int i) {
    int n = 0;
    for (int k = 0; k < i; ++k) n += vel<Q>(k).z == vel<Q>(i).z && !twice_column<Q>(k);
    return n;
}
template <int Q>
__host__ __device__ constexpr int twice_count(int cz) {
    int n = 0;
    for (int k = 0; k < Q; ++k) n += vel<Q>(k).z == cz && !twice_column<Q>(k);
    return n;
}
// first row-slot of (c_z, plane buffer)
template <int Q>
__host__ __device__ constexpr int twice_base(int cz) {
    return cz < 0 ? 0 : cz == 0 ? twice_count<Q>(-1) : twice_count<Q>(-1) + 2 * twice_count<Q>(0);
}
template <int Q>
__host__ __device__ constexpr int twice_smem() {
    return (twice_count<Q>(-1) + 2 * twice_count<Q>(0) + 3 * twice_count<Q>(1)) * TWICE_ROWS * TWICE_P *
           (int)sizeof(float);
}

template <int Q, int S>
__global__ void __launch_bounds__(TWICE_THREADS, 1)
    k_step_twice(Geom g, Coef<float> cf, Tiles t, const Planes<const float> src, const Planes<float> dst,
                 int* __restrict__ flag) {
    constexpr int R = TWICE_ROWS, TY = R - 2, P = TWICE_P, RP = R * P;
    extern __shared__ float sh[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t nx = (uint32_t)g.nx, ny = (uint32_t)g.ny, nxy = nx * ny;
    const bool ring = warp == R;
    const int r = ring ? min(lane, R - 1) : warp;
    bool bad = false;
    int b2 = 0, b3 = 0;  // buffers (c_z = 0, +1) of the plane the first step writes
    long long at = (long long)blockIdx.x * t.run, stop = min(at + t.run, (long long)t.tiles * g.nz);
    if (t.chunks) {
        const int za = (int)(blockIdx.x % t.chunks) * t.run;
        at = (long long)(blockIdx.x / t.chunks) * g.nz + za;
        stop = at + min(t.run, g.nz - za);
    }
    while (at < stop) {
        const int tile = (int)(at / g.nz), za = (int)(at - (long long)tile * g.nz);
        const int zb = (int)min((long long)g.nz, za + (stop - at));
        at += zb - za;
        const int x0 = (tile % t.tx) * t.w, y0 = (tile / t.tx) * TY;
        const int w = min(t.w, g.nx - x0), h = min(TY, g.ny - y0);
        // first step: the thread's row r of the extended tile and its cells at columns ca and cb
        const int ca = ring ? 0 : lane + 1, cb = ring ? w + 1 : lane + 33;
        const bool on = r < h + 2 && (!ring || lane < R);
        const bool va = on && (ring || lane < w), vb = on && (ring || lane + 32 < w);
        uint32_t XA[3], XB[3], Y[3];  // wrapped x + 1, x, x - 1 of the cells; row offsets of y + 1, y, y - 1
        {
            // cells that do not exist take those of the tile's first cell, and write nothing
            int xa = x0 + (va ? ca - 1 : 0), xb = x0 + (vb ? cb - 1 : 0);
            xa = xa < 0 ? g.nx - 1 : xa;
            xb = xb >= g.nx ? xb - g.nx : xb;
            XA[0] = xa + 1 == g.nx ? 0u : (uint32_t)(xa + 1);
            XA[1] = (uint32_t)xa;
            XA[2] = (uint32_t)(xa == 0 ? g.nx - 1 : xa - 1);
            XB[0] = xb + 1 == g.nx ? 0u : (uint32_t)(xb + 1);
            XB[1] = (uint32_t)xb;
            XB[2] = (uint32_t)(xb == 0 ? g.nx - 1 : xb - 1);
            int y = y0 - 1 + (on ? r : 0);
            y = y < 0 ? y + g.ny : y >= g.ny ? y - g.ny : y;
            Y[0] = nx * (uint32_t)(y + 1 == g.ny ? 0 : y + 1);
            Y[1] = nx * (uint32_t)y;
            Y[2] = nx * (uint32_t)(y == 0 ? g.ny - 1 : y - 1);
        }
        // second step: the same cells of the rows inside the ring (the first cell again where there
        // is no second)
        const bool inner = warp >= 1 && warp <= h;
        const bool wa = inner && lane < w, wb = inner && lane + 32 < w;
        const uint32_t row_out = (uint32_t)(x0 + lane) + nx * (uint32_t)(y0 + warp - 1);
        const int second = wb ? 32 : 0;

        F2 e[Q];  // the gathered populations of the next plane of the first step
        auto load = [&](int p) {
            const int z = p < 0 ? p + g.nz : p >= g.nz ? p - g.nz : p;
            const uint32_t Z[3] = {nxy * (uint32_t)(z + 1 == g.nz ? 0 : z + 1), nxy * (uint32_t)z,
                                   nxy * (uint32_t)(z == 0 ? g.nz - 1 : z - 1)};
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                const Vec3 v = vel<Q>(i);
                const uint32_t row = Y[v.y + 1] + Z[v.z + 1];
                e[i] = f2(__ldg(src.p[i] + (XA[v.x + 1] + row)), __ldg(src.p[i] + (XB[v.x + 1] + row)));
            }
        };
        // the column's own populations: c_z = 0 of planes p, p - 1; +1 of p, p - 1, p - 2; -1 of p
        F2 h0[2] = {f2(0.f), f2(0.f)}, hu[3] = {f2(0.f), f2(0.f), f2(0.f)}, hd = f2(0.f);
        if (on) load(za - 1);
        for (int p = za - 1; p <= zb; ++p) {
            if (on) {
                F2 d[Q];
#pragma unroll
                for (int i = 0; i < Q; ++i) d[i] = to_shifted2<S>(e[i], cf.so[i]);
                const Macro2 m = bgk<Q, S>(cf, d);
                bad |= bad_pair(m, true, true);
                float* o = sh + r * P;
                float* of = o + b2 * (twice_count<Q>(0) * RP);
                float* ou = o + b3 * (twice_count<Q>(1) * RP);
#pragma unroll
                for (int i = 0; i < Q; ++i) {
                    const int cz = vel<Q>(i).z;
                    float* q = (cz == 0 ? of : cz > 0 ? ou : o) + (twice_base<Q>(cz) + twice_slot<Q>(i)) * RP;
                    const F2 s = from_shifted2<S>(d[i], cf.so[i]);
                    if (twice_column<Q>(i)) {
                        if (cz == 0) h0[0] = s;
                        if (cz < 0) hd = s;
                        if (cz > 0) hu[0] = s;
                        continue;
                    }
                    if (va) q[ca] = s.v.x;
                    if (vb) q[cb] = s.v.y;
                }
                if (p < zb) load(p + 1);
            }
            __syncthreads();
            if (p > za && wa) {
                // plane p - 1: c_z = +1 from plane p - 2, c_z = 0 from its own, c_z = -1 from p
                const float* o = sh + warp * P + lane + 1;
                const float* of = o + (b2 ^ 1) * (twice_count<Q>(0) * RP);
                const float* ou = o + (b3 == 2 ? 0 : b3 + 1) * (twice_count<Q>(1) * RP);
                F2 d[Q];
#pragma unroll
                for (int i = 0; i < Q; ++i) {
                    const Vec3 v = vel<Q>(i);
                    const float* q = (v.z == 0 ? of : v.z > 0 ? ou : o) + (twice_base<Q>(v.z) + twice_slot<Q>(i)) * RP -
                                     v.y * P - v.x;
                    if (twice_column<Q>(i))
                        d[i] = to_shifted2<S>(v.z == 0 ? h0[1] : v.z > 0 ? hu[2] : hd, cf.so[i]);
                    else
                        d[i] = to_shifted2<S>(f2(q[0], q[second]), cf.so[i]);
                }
                const Macro2 m = bgk<Q, S>(cf, d);
                bad |= bad_pair(m, true, wb);  // without a second cell its half mixes cells that are no neighbours
                const uint32_t n = row_out + nxy * (uint32_t)(p - 1);
#pragma unroll
                for (int i = 0; i < Q; ++i) {
                    const F2 s = from_shifted2<S>(d[i], cf.so[i]);
                    float* q = dst.p[i] + n;
                    q[0] = s.v.x;
                    if (wb) q[32] = s.v.y;
                }
            }
            hu[2] = hu[1];
            hu[1] = hu[0];
            h0[1] = h0[0];
            __syncthreads();
            b2 ^= 1;
            b3 = b3 == 2 ? 0 : b3 + 1;
        }
    }
    if (bad) *flag = 1;
}

// The split with the fewest plane walks of the busiest block (one block per SM of `slots`), two more
// than it owns for every tile it works on; `walks` returns them.
inline Tiles twice_tiles(const Geom& g, int slots, long long& walks) {
    constexpr int TY = TWICE_ROWS - 2;
    Tiles t;
    t.tx = (g.nx + TWICE_W - 1) / TWICE_W;
    t.w = ((g.nx + t.tx - 1) / t.tx + 7) & ~7;  // whole sectors: 160 = 56 + 56 + 48 cells
    t.tiles = t.tx * ((g.ny + TY - 1) / TY);
    t.run = (int)(((long long)t.tiles * g.nz + slots - 1) / slots);
    t.chunks = 0;
    walks = t.run + 2 * (2 + (t.run - 2) / g.nz);
    for (int nc = 1; nc <= g.nz; ++nc) {
        const int zc = (g.nz + nc - 1) / nc, chunks = (g.nz + zc - 1) / zc;
        const long long c = (((long long)t.tiles * chunks + slots - 1) / slots) * (zc + 2);
        if (c < walks) {
            walks = c;
            t.run = zc;
            t.chunks = chunks;
        }
    }
    return t;
}

// Whether two steps in one launch are faster than two launches. A plane walk of a block takes 3.1 us
// (9 x 64 cells, two steps) while one step a launch runs at the copy bandwidth, so the split has to
// fill the SMs: measured ratio of a step's time against the share `full` of the walks that own cells,
// 512^3 1.28 (0.99), 256^3 1.20 (0.96), 128^3 1.10 (0.86), 176^3 1.11 (0.84), 224^3 1.04 (0.85),
// 160^3 1.00 (0.77), 144^3 0.94 (0.68). Rows that are no multiple of 8 cells make the tiles' edges
// share sectors: 130 x 128^2 0.92, 132^3 0.97, 196^3 0.94, 252^3 0.89, 257^3 0.96, 258 x 256^2 0.86,
// 260^3 0.95, 300^3 0.89, 380^3 0.92, 508 x 256^2 0.86. Boxes whose two states stay in L2 in good part are
// faster in single steps where they are cubes (96^3 0.74, 104^3 0.89, 112^3 0.90, 120^3 0.97); some of
// them would gain (128^2 x 96 1.06, 64 x 144 x 128 1.06), so the line at 1.9M cells is on the safe side.
inline bool twice_pays(const Geom& g, int slots, Tiles& t) {
    if (g.nx % 8 != 0 || g.N < 1900000u || slots < 1) return false;
    long long walks = 0;
    t = twice_tiles(g, slots, walks);
    const double full = (double)g.N / ((double)walks * slots * TWICE_W * (TWICE_ROWS - 2));
    return full >= 0.82;
}

}  // namespace LBM_VARIANT
}  // namespace lbm
