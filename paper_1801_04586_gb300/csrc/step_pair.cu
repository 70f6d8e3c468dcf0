// step_pair.cu -- launch of the FP32 node-pair step (step_pair.cuh).
#include "step_pair.cuh"

namespace clbm {

// From 100,000 nodes on: two to three warps of pairs for each of the 608
// schedulers. Below that a scheduler's one warp of pairs runs longer than its two warps of
// single nodes (us a step from a graph, one node / pairs: 16 x 32 x 32 2.08 /
// 2.59, 32^3 2.34 / 2.71, 128 x 128 x 5 3.36 / 3.30 and
// 4.13 / 4.18 launched one by one, 48^3 4.06 / 3.36, 64^3
// 6.27 / 5.41, 80^3 13.5 / 9.2, 150 x 91 x 61 with a force field 22.5 / 20.6,
// 200 x 180 x 160 137 / 128, 256^3 379 / 369).
bool step_pairs(const Geom &g) {
    const int64_t npx = (g.nx + 1) / 2;
    // the row of a pair by one multiplication: exact while pairs of a plane x pairs of a row < 2^32
    return npx >= 2 && npx * npx * g.ny < ((int64_t)1 << 32) && (int64_t)g.nx * g.ny * g.nz >= 100000;
}

template <typename S, int FM>
static cudaError_t pair_t(const Launch &L, const void *src, void *dst, const Rates &r, const ForceArgs &F, int *flag,
                          uint32_t key) {
    const Geom &g = L.g;
    const uint32_t npx = (uint32_t)(g.nx + 1) / 2u, rdiv = 0xffffffffu / npx + 1u;
    const dim3 grid((npx * (uint32_t)g.ny + kPairThreads - 1u) / kPairThreads, (unsigned)g.nz);
    const bool vec = g.nx % 2 == 0 && (((uintptr_t)src | (uintptr_t)dst) & (2 * sizeof(S) - 1u)) == 0;
    auto go = [&](auto kern, auto... keys) {
        return launch_overlapped(kern, grid, dim3(kPairThreads), 0, L.stream, L.overlap, (const S *)src, (S *)dst, g, r,
                                 F, flag, keys..., npx, rdiv);
    };
    if constexpr (sizeof(S) == 4) {
        if (g.walls) return vec ? go(k_step_pair<FM, true, true>) : go(k_step_pair<FM, true, false>);
        return vec ? go(k_step_pair<FM, false, true>) : go(k_step_pair<FM, false, false>);
    } else {
        if (g.walls) return vec ? go(k_step_pair16<S, FM, true, true>, key) : go(k_step_pair16<S, FM, true, false>, key);
        return vec ? go(k_step_pair16<S, FM, false, true>, key) : go(k_step_pair16<S, FM, false, false>, key);
    }
}

template <typename S>
static cudaError_t pair_force_t(const Launch &L, const void *src, void *dst, const Rates &r, const ForceArgs &F,
                                int *flag, uint32_t key) {
    switch (F.mode) {
        case kForceUniform: return pair_t<S, kForceUniform>(L, src, dst, r, F, flag, key);
        case kForceProfileZ: return pair_t<S, kForceProfileZ>(L, src, dst, r, F, flag, key);
        default: return pair_t<S, kForceField>(L, src, dst, r, F, flag, key);
    }
}

template <int FM>
static cudaError_t aa_pair_t(const Launch &L, void *f, const Rates &r, const ForceArgs &F, int *flag, bool odd) {
    const Geom &g = L.g;
    if (!odd) {
        const uint32_t n = (uint32_t)g.nx * (uint32_t)g.ny * (uint32_t)g.nz;
        const dim3 grid(((n + 1u) / 2u + kPairThreads - 1u) / kPairThreads);
        return launch_overlapped(k_step_aa_pair_even<FM>, grid, dim3(kPairThreads), 0, L.stream, L.overlap, (float *)f,
                                 g, r, F, flag, n);
    }
    const uint32_t npx = (uint32_t)(g.nx + 1) / 2u, rdiv = 0xffffffffu / npx + 1u;
    const dim3 grid((npx * (uint32_t)g.ny + kPairThreads - 1u) / kPairThreads, (unsigned)g.nz);
    auto go = [&](auto kern) {
        return launch_overlapped(kern, grid, dim3(kPairThreads), 0, L.stream, L.overlap, (float *)f, g, r, F, flag, npx,
                                 rdiv);
    };
    const bool vec = g.nx % 2 == 0;
    if (g.walls) return vec ? go(k_step_aa_pair_odd<FM, true, true>) : go(k_step_aa_pair_odd<FM, true, false>);
    return vec ? go(k_step_aa_pair_odd<FM, false, true>) : go(k_step_aa_pair_odd<FM, false, false>);
}

cudaError_t launch_step_aa_pair(const Launch &L, void *f, const Rates &r, const ForceArgs &F, int *flag, bool odd) {
    switch (F.mode) {
        case kForceUniform: return aa_pair_t<kForceUniform>(L, f, r, F, flag, odd);
        case kForceProfileZ: return aa_pair_t<kForceProfileZ>(L, f, r, F, flag, odd);
        default: return aa_pair_t<kForceField>(L, f, r, F, flag, odd);
    }
}

cudaError_t launch_step_pair(int storage, const Launch &L, const void *src, void *dst, const Rates &r,
                             const ForceArgs &F, int *flag, uint32_t key) {
    switch (storage) {
        case 0: return pair_force_t<float>(L, src, dst, r, F, flag, key);
        case 1: return pair_force_t<__half>(L, src, dst, r, F, flag, key);
        case 2: return pair_force_t<__nv_bfloat16>(L, src, dst, r, F, flag, key);
        case 3: return pair_force_t<HalfSR>(L, src, dst, r, F, flag, key);
        default: return pair_force_t<BF16SR>(L, src, dst, r, F, flag, key);
    }
}

}  // namespace clbm
