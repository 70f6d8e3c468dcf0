// step_pair.cuh -- the D3Q19 A/B step with two adjacent nodes per thread,
// collided together in the lanes of f2 (FP32x2 instructions).
//
// Why: with the populations in L2 (up to some 80^3) the one-node step is bound
// by instruction issue and by the last wave of its blocks; above, it runs at
// the DRAM rate only as long as enough of its warps are loading. A pair halves
// the arithmetic's issue slots (f2 rounds like the one-node collision, so the
// results are the same bits), forms each address once for two nodes and moves
// 9 of 19 populations by 64-bit loads and all of them by 64-bit stores. 78-80
// registers for the pair (96 and 88 with odd rows) keep six blocks of 128, 24
// warps of pairs, in flight on an SM. 256^3: 368.6 us a
// step against 379.2 (6.92 TB/s algorithmic, 1.03 of the copy rate), on other
// days 361 against 371; 80^3 in L2: 9.2 against 13.5.
//
// (A pass of two steps over a column kept in shared memory, which halves the
// DRAM traffic, measured 38-45k MLUPS in six forms, no more than the single
// step's 45.5-46.4k: 16 warps per SM do not hide its phases.)
#pragma once

#include "cascaded.cuh"
#include "kernels.cuh"
#include "step_kernels.cuh"

namespace clbm {

constexpr int kPairThreads = 128;

// The wall faces a node touches, and whether population i arrives from beyond
// one of them (halfway bounce-back).
struct WallFaces {
    bool xl, xh, yl, yh, zl, zh;
    __device__ __forceinline__ bool any() const { return xl || xh || yl || yh || zl || zh; }
    __device__ __forceinline__ bool bounces(int i) const {
        return (ex19(i) > 0 && xl) || (ex19(i) < 0 && xh) || (ey19(i) > 0 && yl) || (ey19(i) < 0 && yh) ||
               (ez19(i) > 0 && zl) || (ez19(i) < 0 && zh);
    }
};
__device__ __forceinline__ WallFaces wall_faces(const Geom &g, int x, int y, int z) {
    const bool wx = g.walls & 1u, wy = g.walls & 2u, wz = g.walls & 4u;
    return WallFaces{wx && x == 0, wx && x == g.nx - 1, wy && y == 0, wy && y == g.ny - 1, wz && z == 0,
                     wz && z == g.nz - 1};
}

// An aligned pair of adjacent values (global memory, as ld_state).
__device__ __forceinline__ float2 ld_state2(const float *p) {
    float2 v;
    asm volatile("ld.global.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
    return v;
}

// The FP32 step. VEC: nx even, so that a pair x, x + 1 (x even) is 8-byte aligned in every
// row. Thread t of plane z takes pair t of the plane's rows of (nx + 1) / 2
// pairs: no lane idles whatever nx is. rdiv = ceil(2^32 / pairs per row).
template <int FM, bool WALLS, bool VEC>
__global__ void __launch_bounds__(kPairThreads) k_step_pair(const float *src, float *__restrict__ dst, Geom g, Rates r,
                                                            ForceArgs F, int *__restrict__ flag, uint32_t npx,
                                                            uint32_t rdiv) {
    grid_dependency_wait();
    const uint32_t t = blockIdx.x * kPairThreads + threadIdx.x;
    if (t >= npx * (uint32_t)g.ny) return;
    const int y = (int)__umulhi(t, rdiv), z = blockIdx.y;
    const int x = 2 * (int)(t - (uint32_t)y * npx);
    const bool two = VEC || x + 1 < g.nx;
    const uint32_t unx = (uint32_t)g.nx, plane = unx * (uint32_t)g.ny;
    const uint32_t rc = (uint32_t)y * unx, rm = (uint32_t)(y == 0 ? g.ny - 1 : y - 1) * unx,
                   rp = (uint32_t)(y == g.ny - 1 ? 0 : y + 1) * unx;
    const uint32_t zc = (uint32_t)z * plane, zm = (uint32_t)(z == 0 ? g.nz - 1 : z - 1) * plane,
                   zp = (uint32_t)(z == g.nz - 1 ? 0 : z + 1) * plane;
    const uint32_t xa = (uint32_t)x, xb = two ? xa + 1u : xa;  // the pair (odd nx: a row's last pair is one node)
    const uint32_t xam = xa == 0u ? unx - 1u : xa - 1u, xbp = xb == unx - 1u ? 0u : xb + 1u;
    const uint32_t self = zc + rc + xa;
    f2 h[kQ];
#pragma unroll
    for (int i = 0; i < kQ; ++i) {
        const float *base = src + (size_t)i * g.stride;
        const uint32_t row = (ez19(i) > 0 ? zm : (ez19(i) < 0 ? zp : zc)) + (ey19(i) > 0 ? rm : (ey19(i) < 0 ? rp : rc));
        if (ex19(i) == 0 && VEC)
            h[i] = f2{ld_state2(CLBM_AT(g, src, base, row + xa, 1u))};
        else if (ex19(i) == 0)
            h[i] = mk2(ld_state(CLBM_AT(g, src, base, row + xa, 0u)), ld_state(CLBM_AT(g, src, base, row + xb, 0u)));
        else if (ex19(i) > 0)
            h[i] = mk2(ld_state(CLBM_AT(g, src, base, row + xam, 0u)), ld_state(CLBM_AT(g, src, base, row + (two ? xa : xam), 0u)));
        else
            h[i] = mk2(ld_state(CLBM_AT(g, src, base, row + (two ? xb : xbp), 0u)), ld_state(CLBM_AT(g, src, base, row + xbp, 0u)));
    }
    if (WALLS) {
        const WallFaces wa = wall_faces(g, (int)xa, y, z), wb = wall_faces(g, (int)xb, y, z);
        if (wa.any() || wb.any()) {
#pragma unroll
            for (int i = 1; i < kQ; ++i) {
                const float *base = src + (size_t)opposite(i) * g.stride;
                if (wa.bounces(i)) h[i].v.x = ld_state(CLBM_AT(g, src, base, self, 0u));
                if (wb.bounces(i)) h[i].v.y = ld_state(CLBM_AT(g, src, base, self + (xb - xa), 0u));
            }
        }
    }
    f2 fx, fy, fz;
    {
        float ax, ay, az;
        force_at<FM>(F, g, z, self, ax, ay, az);
        fx = mk2(ax); fy = mk2(ay); fz = mk2(az);
        if (FM == kForceField) force_at<FM>(F, g, z, self + (xb - xa), fx.v.y, fy.v.y, fz.v.y);
    }
    const f2 drho = Cascaded::run<false>(h, fx, fy, fz, r);
    if (!(fabsf(drho.v.x) < 0.9f) || !(fabsf(drho.v.y) < 0.9f)) *flag = 1;
#pragma unroll
    for (int i = 0; i < kQ; ++i) {
        float *to = dst + (size_t)i * g.stride + CLBM_SLOTS(g, self, (kQ - 1) * g.stride + (xb - xa));
        if (VEC) {
            *reinterpret_cast<float2 *>(to) = h[i].v;
        } else {
            to[0] = h[i].v.x;
            if (two) to[1] = h[i].v.y;
        }
    }
}

// The in-place (AA) step with FP32 storage in node pairs (the kinds of
// k_step_aa, step_kernels.cuh, with its bits).
//   even kind: no node looks at a neighbour, so the pairs are 2t and 2t + 1 in
//              the lattice's linear order, aligned whatever nx is;
//   odd kind:  pairs of a row as k_step_pair; population i of both nodes is
//              read from array ibar at x - e_i (from array i at a wall) and
//              pushed to (i, x + e_i) (to array ibar at a wall): with e_x = 0
//              both are one aligned pair, otherwise two values.
// One node per thread, the odd kind's pushes and the idle lanes of rows that no
// block width divides cost 12-30 % over the even kind. us a step, mean of both
// kinds, one node / pairs: 256^3 399 / 366 (6.97 TB/s algorithmic), 200 x 180 x
// 160 with z walls 158 / 131, 150 x 91 x 61 with a force field 21.0 / 15.7,
// 80^3 14.3 / 10.3.
template <int FM>
__global__ void __launch_bounds__(kPairThreads) k_step_aa_pair_even(float *f, Geom g, Rates r, ForceArgs F,
                                                                    int *__restrict__ flag, uint32_t n) {
    grid_dependency_wait();
    const uint32_t self = 2u * (blockIdx.x * kPairThreads + threadIdx.x);
    if (self >= n) return;
    const bool two = self + 1u < n;  // (the slot after an odd lattice's last node is padding of the array)
    f2 h[kQ];
#pragma unroll
    for (int i = 0; i < kQ; ++i) h[i] = f2{ld_state2(CLBM_AT(g, f, f + (size_t)i * g.stride, self, 1u))};
    const uint32_t last = two ? self + 1u : self, plane = (uint32_t)g.nx * (uint32_t)g.ny;
    const int za = FM == kForceProfileZ ? (int)(self / plane) : 0, zb = FM == kForceProfileZ ? (int)(last / plane) : 0;
    f2 fx, fy, fz;
    force_at<FM>(F, g, za, self, fx.v.x, fy.v.x, fz.v.x);
    force_at<FM>(F, g, zb, last, fx.v.y, fy.v.y, fz.v.y);
    const f2 drho = Cascaded::run<false>(h, fx, fy, fz, r);
    if (!(fabsf(drho.v.x) < 0.9f) || (two && !(fabsf(drho.v.y) < 0.9f))) *flag = 1;
#pragma unroll
    for (int i = 0; i < kQ; ++i) {
        float *to = CLBM_AT(g, f, f + (size_t)opposite(i) * g.stride, self, two ? 1u : 0u);
        if (two)
            *reinterpret_cast<float2 *>(to) = h[i].v;
        else
            to[0] = h[i].v.x;
    }
}

template <int FM, bool WALLS, bool VEC>
__global__ void __launch_bounds__(kPairThreads) k_step_aa_pair_odd(float *f, Geom g, Rates r, ForceArgs F,
                                                                   int *__restrict__ flag, uint32_t npx,
                                                                   uint32_t rdiv) {
    grid_dependency_wait();
    const uint32_t t = blockIdx.x * kPairThreads + threadIdx.x;
    if (t >= npx * (uint32_t)g.ny) return;
    int y = (int)__umulhi(t, rdiv), z = blockIdx.y;
    int x = 2 * (int)(t - (uint32_t)y * npx);
    const bool two = VEC || x + 1 < g.nx;
    const uint32_t unx = (uint32_t)g.nx, plane = unx * (uint32_t)g.ny;
    f2 h[kQ];
    WallFaces wa, wb;
    bool any = false;
    if (WALLS) {
        wa = wall_faces(g, x, y, z);
        wb = wall_faces(g, two ? x + 1 : x, y, z);
        any = wa.any() || wb.any();
    }
    uint32_t self;
    {
        const uint32_t rc = (uint32_t)y * unx, rm = (uint32_t)(y == 0 ? g.ny - 1 : y - 1) * unx,
                       rp = (uint32_t)(y == g.ny - 1 ? 0 : y + 1) * unx;
        const uint32_t zc = (uint32_t)z * plane, zm = (uint32_t)(z == 0 ? g.nz - 1 : z - 1) * plane,
                       zp = (uint32_t)(z == g.nz - 1 ? 0 : z + 1) * plane;
        const uint32_t xa = (uint32_t)x, xb = two ? xa + 1u : xa;
        const uint32_t xam = xa == 0u ? unx - 1u : xa - 1u, xbp = xb == unx - 1u ? 0u : xb + 1u;
        self = zc + rc + xa;
#pragma unroll
        for (int i = 0; i < kQ; ++i) {
            const float *base = f + (size_t)opposite(i) * g.stride;
            const uint32_t row =
                (ez19(i) > 0 ? zm : (ez19(i) < 0 ? zp : zc)) + (ey19(i) > 0 ? rm : (ey19(i) < 0 ? rp : rc));
            if (ex19(i) == 0 && VEC)
                h[i] = f2{ld_state2(CLBM_AT(g, f, base, row + xa, 1u))};
            else if (ex19(i) == 0)
                h[i] = mk2(ld_state(CLBM_AT(g, f, base, row + xa, 0u)), ld_state(CLBM_AT(g, f, base, row + xb, 0u)));
            else if (ex19(i) > 0)
                h[i] = mk2(ld_state(CLBM_AT(g, f, base, row + xam, 0u)), ld_state(CLBM_AT(g, f, base, row + (two ? xa : xam), 0u)));
            else
                h[i] = mk2(ld_state(CLBM_AT(g, f, base, row + (two ? xb : xbp), 0u)), ld_state(CLBM_AT(g, f, base, row + xbp, 0u)));
        }
        if (WALLS && any) {
#pragma unroll
            for (int i = 1; i < kQ; ++i) {
                const float *base = f + (size_t)i * g.stride;
                if (wa.bounces(i)) h[i].v.x = ld_state(CLBM_AT(g, f, base, self, 0u));
                if (wb.bounces(i)) h[i].v.y = ld_state(CLBM_AT(g, f, base, self + (xb - xa), 0u));
            }
        }
    }
    f2 fx, fy, fz;
    force_at<FM>(F, g, z, self, fx.v.x, fy.v.x, fz.v.x);
    if (FM == kForceField)
        force_at<FM>(F, g, z, self + (two ? 1u : 0u), fx.v.y, fy.v.y, fz.v.y);
    else
        fx.v.y = fx.v.x, fy.v.y = fy.v.x, fz.v.y = fz.v.x;
    const f2 drho = Cascaded::run<false>(h, fx, fy, fz, r);
    if (!(fabsf(drho.v.x) < 0.9f) || !(fabsf(drho.v.y) < 0.9f)) *flag = 1;
    // push targets, from coordinates the compiler must treat as new, so that the offsets above do not stay live
    asm volatile("" : "+r"(x), "+r"(y), "+r"(z) : "f"(h[0].v.x), "f"(h[kQ - 1].v.x));
    const uint32_t rc = (uint32_t)y * unx, rm = (uint32_t)(y == 0 ? g.ny - 1 : y - 1) * unx,
                   rp = (uint32_t)(y == g.ny - 1 ? 0 : y + 1) * unx;
    const uint32_t zc = (uint32_t)z * plane, zm = (uint32_t)(z == 0 ? g.nz - 1 : z - 1) * plane,
                   zp = (uint32_t)(z == g.nz - 1 ? 0 : z + 1) * plane;
    const uint32_t xa = (uint32_t)x, xb = two ? xa + 1u : xa;
    const uint32_t xam = xa == 0u ? unx - 1u : xa - 1u, xbp = xb == unx - 1u ? 0u : xb + 1u;
#pragma unroll
    for (int i = 0; i < kQ; ++i) {
        float *base = f + (size_t)i * g.stride;
        const uint32_t row = (ez19(i) > 0 ? zp : (ez19(i) < 0 ? zm : zc)) + (ey19(i) > 0 ? rp : (ey19(i) < 0 ? rm : rc));
        bool ba = false, bb = false;  // leaving through a wall: the direction that arrives from it is ibar
        if (WALLS && any) {
            ba = wa.bounces(opposite(i));
            bb = wb.bounces(opposite(i));
        }
        if (ex19(i) == 0 && VEC && !(WALLS && any)) {
            *reinterpret_cast<float2 *>(CLBM_AT(g, f, base, row + xa, 1u)) = h[i].v;
        } else {
            float *back = CLBM_AT(g, f, f + (size_t)opposite(i) * g.stride, self, two ? 1u : 0u);
            const uint32_t oa = row + (ex19(i) > 0 ? (two ? xb : xbp) : (ex19(i) < 0 ? xam : xa));
            const uint32_t ob = row + (ex19(i) > 0 ? xbp : (ex19(i) < 0 ? xa : xb));
            *(ba ? back : CLBM_AT(g, f, base, oa, 0u)) = h[i].v.x;
            if (two) *(bb ? back + 1 : CLBM_AT(g, f, base, ob, 0u)) = h[i].v.y;
        }
    }
}

template <typename S>
__device__ __forceinline__ float2 ld_state2(const S *p) {  // 16-bit formats: one word
    uint32_t w;
    asm volatile("ld.global.u32 %0, [%1];" : "=r"(w) : "l"(p));
    return Codec<S>::unpack2(w);
}

// 16-bit formats: load what arrives at the nodes x and x + 1 (x even) of row y, plane z under
// Eq. 8; returns the first one's offset. VEC: nx even, so that such a pair is
// aligned in every row; otherwise two says whether x + 1 is a node (a row's
// last pair of an odd row is one node: its second lane repeats the first).
template <typename S, bool WALLS, bool VEC>
__device__ __forceinline__ uint32_t pair_load(const S *src, const Geom &g, int x, int y, int z, bool two,
                                              f2 (&h)[kQ]) {
    const uint32_t unx = (uint32_t)g.nx, plane = unx * (uint32_t)g.ny;
    const uint32_t rc = (uint32_t)y * unx, rm = (uint32_t)(y == 0 ? g.ny - 1 : y - 1) * unx,
                   rp = (uint32_t)(y == g.ny - 1 ? 0 : y + 1) * unx;
    const uint32_t zc = (uint32_t)z * plane, zm = (uint32_t)(z == 0 ? g.nz - 1 : z - 1) * plane,
                   zp = (uint32_t)(z == g.nz - 1 ? 0 : z + 1) * plane;
    const uint32_t xa = (uint32_t)x, xb = two ? xa + 1u : xa;
    const uint32_t xam = xa == 0u ? unx - 1u : xa - 1u, xbp = xb == unx - 1u ? 0u : xb + 1u;
    const uint32_t self = zc + rc + xa;
#pragma unroll
    for (int i = 0; i < kQ; ++i) {
        const size_t pop = (size_t)i * g.stride;
        const uint32_t row = (ez19(i) > 0 ? zm : (ez19(i) < 0 ? zp : zc)) + (ey19(i) > 0 ? rm : (ey19(i) < 0 ? rp : rc));
        if (ex19(i) == 0 && VEC) {
            h[i] = f2{ld_state2(src + CLBM_SLOTS(g, pop + (row + xa), 1u))};
        } else {
            const uint32_t oa = row + (ex19(i) > 0 ? xam : (ex19(i) < 0 ? (two ? xb : xbp) : xa));
            const uint32_t ob = row + (ex19(i) > 0 ? (two ? xa : xam) : (ex19(i) < 0 ? xbp : xb));
            h[i] = mk2(Codec<S>::load(src + CLBM_IDX(g, pop + oa)), Codec<S>::load(src + CLBM_IDX(g, pop + ob)));
        }
    }
    if (WALLS) {
        const WallFaces wa = wall_faces(g, (int)xa, y, z), wb = wall_faces(g, (int)xb, y, z);
        if (wa.any() || wb.any()) {
#pragma unroll
            for (int i = 1; i < kQ; ++i) {
                const size_t b = (size_t)opposite(i) * g.stride + self;
                if (wa.bounces(i)) h[i].v.x = Codec<S>::load(src + CLBM_IDX(g, b));
                if (wb.bounces(i)) h[i].v.y = Codec<S>::load(src + CLBM_IDX(g, b + (xb - xa)));
            }
        }
    }
    return self;
}

// Store the pair's post-collision values at its own slots: a pair of an even
// row is one conversion and one word; in odd rows each node converts on its own (the dither is drawn per even-odd pair of node indices).
template <typename S, bool VEC>
__device__ __forceinline__ void pair_store(S *dst, const Geom &g, uint32_t self, bool two, const f2 (&h)[kQ],
                                           uint32_t key) {
    S *at = dst + CLBM_SLOTS(g, self, (kQ - 1) * g.stride + (two ? 1u : 0u));
    if constexpr (VEC) {
        const uint32_t hb = Codec<S>::kStochastic ? pair_hash(self >> 1, key) : 0u;
#pragma unroll
        for (int i = 0; i < kQ; ++i) {
            uint32_t w;
            if constexpr (Codec<S>::kStochastic)
                w = Codec<S>::pair_sr(h[i].v.y, h[i].v.x, pop_bits(hb, i));
            else
                w = Codec<S>::pair_rn(h[i].v.y, h[i].v.x);
            *reinterpret_cast<uint32_t *>(at + (size_t)i * g.stride) = w;
        }
    } else {
        const uint32_t ha = Codec<S>::kStochastic ? pair_hash(self >> 1, key) : 0u;
        const uint32_t hb = Codec<S>::kStochastic ? pair_hash((self + 1u) >> 1, key) : 0u;
#pragma unroll
        for (int i = 0; i < kQ; ++i) {
            S *to = at + (size_t)i * g.stride;
            if constexpr (Codec<S>::kStochastic) {
                to[0] = Codec<S>::from_f_sr(h[i].v.x, pop_bits(ha, i), self & 1u);
                if (two) to[1] = Codec<S>::from_f_sr(h[i].v.y, pop_bits(hb, i), (self + 1u) & 1u);
            } else {
                to[0] = Codec<S>::from_f(h[i].v.x);
                if (two) to[1] = Codec<S>::from_f(h[i].v.y);
            }
        }
    }
}

// The 16-bit A/B step in node pairs, for lattices that the staged step
// (step_tma.cuh) does not take or does not pay for. Without walls the pair is
// capped at five blocks of 128 per SM (96 registers): FP16 at 151 x 90 x 61
// 17.3 -> 14.5 us a step (17.6 one node per thread); with walls it keeps its
// 104-122 registers (150 x 91 x 61: 15.0 us, 15.4 capped, 19.9 one node).
template <typename S, int FM, bool WALLS, bool VEC>
__global__ void __launch_bounds__(kPairThreads, WALLS ? 1 : 5)
    k_step_pair16(const S *src, S *__restrict__ dst, Geom g, Rates r, ForceArgs F, int *__restrict__ flag,
                  uint32_t key, uint32_t npx, uint32_t rdiv) {
    grid_dependency_wait();
    const uint32_t t = blockIdx.x * kPairThreads + threadIdx.x;
    if (t >= npx * (uint32_t)g.ny) return;
    const int y = (int)__umulhi(t, rdiv), z = blockIdx.y;
    const int x = 2 * (int)(t - (uint32_t)y * npx);
    const bool two = VEC || x + 1 < g.nx;
    f2 h[kQ];
    const uint32_t self = pair_load<S, WALLS, VEC>(src, g, x, y, z, two, h);
    f2 fx, fy, fz;
    {
        float ax, ay, az;
        force_at<FM>(F, g, z, self, ax, ay, az);
        fx = mk2(ax); fy = mk2(ay); fz = mk2(az);
        if (FM == kForceField) force_at<FM>(F, g, z, self + (two ? 1u : 0u), fx.v.y, fy.v.y, fz.v.y);
    }
    const f2 drho = Cascaded::run<true>(h, fx, fy, fz, r);
    if (!(fabsf(drho.v.x) < 0.9f) || !(fabsf(drho.v.y) < 0.9f)) *flag = 1;
    pair_store<S, VEC>(dst, g, self, two, h, key);
}

}  // namespace clbm
