// step_small.cuh -- two time steps of a small FP32 D3Q19 A/B lattice in one
// launch.
//
// Why: below 100,000 nodes a step is latency: one kernel edge (1.15 us inside a
// graph, 1.5 us or more outside) and one wave of load, collide, store, with few
// warps per scheduler (16 x 32 x 32: 2.2 us a step, 0.07 of them arithmetic at
// full rate). Two steps per launch halve the edges and the trips to L2; the
// nodes they compute twice ride in issue slots that would stay empty.
//
// How: a block owns a brick of nodes. Stage 1 steps the brick grown by one node
// on each side (not along axes the brick spans), one thread per node, as
// k_step does, and keeps the 19 post-collision values in shared memory; stage 2
// steps the brick itself from there and stores. The intermediate values are
// the FP32 values a single step would store: the same bits as two steps.
#pragma once

#include "cascaded.cuh"
#include "kernels.cuh"
#include "step_kernels.cuh"

namespace clbm {

template <int FM, bool WALLS>
__global__ void __launch_bounds__(1024) k_step_small2(const float *src, float *__restrict__ dst, Geom g, Rates r,
                                                      ForceArgs F, float scale2, int *__restrict__ flag, SmallPlan p) {
    extern __shared__ float small_smem[];  // [kQ][p.ext]
    grid_dependency_wait();
    const int tid = threadIdx.x;
    // the brick
    int b = blockIdx.x;
    const int kz = b / (p.nbx * p.nby);
    b -= kz * p.nbx * p.nby;
    const int ky = b / p.nbx, kx = b - ky * p.nbx;
    const int x0 = kx * p.bx, y0 = ky * p.by, z0 = kz * p.bz;
    const int w = min(p.bx, g.nx - x0), h = min(p.by, g.ny - y0), d = min(p.bz, g.nz - z0);
    {  // stage 1: extended node (ex, ey, ez)
        const int ez = (int)__umulhi((uint32_t)tid, p.exydiv), q = tid - ez * p.ex * p.ey;
        const int ey = (int)__umulhi((uint32_t)q, p.exdiv), ex = q - ey * p.ex;
        int x = x0 - p.hx + ex, y = y0 - p.hy + ey, z = z0 - p.hz + ez;
        bool on = tid < p.ext && ex < w + 2 * p.hx && ey < h + 2 * p.hy && ez < d + 2 * p.hz;
        if (x < 0 || x >= g.nx) {  // across a face: the periodic image, or nothing beyond a wall
            if (WALLS && (g.walls & 1u)) on = false;
            x = x < 0 ? x + g.nx : x - g.nx;
        }
        if (y < 0 || y >= g.ny) {
            if (WALLS && (g.walls & 2u)) on = false;
            y = y < 0 ? y + g.ny : y - g.ny;
        }
        if (z < 0 || z >= g.nz) {
            if (WALLS && (g.walls & 4u)) on = false;
            z = z < 0 ? z + g.nz : z - g.nz;
        }
        if (on) {
            uint32_t off[kQ];
            int pop[kQ];
            pull_sources<WALLS>(g, x, y, z, off, pop);
            float f[kQ];
#pragma unroll
            for (int i = 0; i < kQ; ++i) f[i] = ld_state(src + CLBM_IDX(g, (size_t)pop[i] * g.stride + off[i]));
            float fx, fy, fz;
            force_at<FM>(F, g, z, off[0], fx, fy, fz);
            const float drho = Cascaded::run<false>(f, fx, fy, fz, r);
            if (!(fabsf(drho) < 0.9f)) *flag = 1;
#pragma unroll
            for (int i = 0; i < kQ; ++i) small_smem[i * p.ext + tid] = f[i];
        }
    }
    __syncthreads();
    {  // stage 2: node (ox, oy, oz) of the brick
        const int oz = (int)__umulhi((uint32_t)tid, p.bxydiv), q = tid - oz * p.bx * p.by;
        const int oy = (int)__umulhi((uint32_t)q, p.bxdiv), ox = q - oy * p.bx;
        if (ox >= w || oy >= h || oz >= d) return;
        const int x = x0 + ox, y = y0 + oy, z = z0 + oz;
        const int sy = p.ex, sz = p.ex * p.ey;
        const int e = ((oz + p.hz) * p.ey + oy + p.hy) * p.ex + ox + p.hx;
        // steps to the neighbours; along an axis that the brick spans they wrap inside it
        const int xm = p.hx == 0 && x == 0 ? g.nx - 1 : -1, xp = p.hx == 0 && x == g.nx - 1 ? 1 - g.nx : 1;
        const int ym = p.hy == 0 && y == 0 ? (g.ny - 1) * sy : -sy, yp = p.hy == 0 && y == g.ny - 1 ? (1 - g.ny) * sy : sy;
        const int zm = p.hz == 0 && z == 0 ? (g.nz - 1) * sz : -sz, zp = p.hz == 0 && z == g.nz - 1 ? (1 - g.nz) * sz : sz;
        bool xl = false, xh = false, yl = false, yh = false, zl = false, zh = false;
        if (WALLS) {
            xl = (g.walls & 1u) && x == 0; xh = (g.walls & 1u) && x == g.nx - 1;
            yl = (g.walls & 2u) && y == 0; yh = (g.walls & 2u) && y == g.ny - 1;
            zl = (g.walls & 4u) && z == 0; zh = (g.walls & 4u) && z == g.nz - 1;
        }
        float f[kQ];
#pragma unroll
        for (int i = 0; i < kQ; ++i) {
            const int dx = ex19(i) > 0 ? xm : (ex19(i) < 0 ? xp : 0), dy = ey19(i) > 0 ? ym : (ey19(i) < 0 ? yp : 0),
                      dz = ez19(i) > 0 ? zm : (ez19(i) < 0 ? zp : 0);
            const bool bb = WALLS && ((ex19(i) > 0 && xl) || (ex19(i) < 0 && xh) || (ey19(i) > 0 && yl) ||
                                      (ey19(i) < 0 && yh) || (ez19(i) > 0 && zl) || (ez19(i) < 0 && zh));
            const int o = bb ? opposite(i) * p.ext + e : i * p.ext + e + dx + dy + dz;
            f[i] = small_smem[CLBM_SIDX(g, o, kQ * p.ext)];
        }
        const uint32_t self = ((uint32_t)z * g.ny + y) * g.nx + x;
        ForceArgs F2 = F;
        F2.scale = scale2;
        float fx, fy, fz;
        force_at<FM>(F2, g, z, self, fx, fy, fz);
        const float drho = Cascaded::run<false>(f, fx, fy, fz, r);
        if (!(fabsf(drho) < 0.9f)) *flag = 1;
        store_node<float>(dst + CLBM_SLOTS(g, self, (kQ - 1) * g.stride), g.stride, f, self, 0u);
    }
}

}  // namespace clbm
