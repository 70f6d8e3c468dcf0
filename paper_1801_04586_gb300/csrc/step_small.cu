// step_small.cu -- plan and launch of the two-step kernel of small lattices
// (step_small.cuh).
#include <algorithm>
#include <atomic>
#include <cmath>
#include <type_traits>

#include "step_small.cuh"

namespace clbm {

// The brick that minimises a model of the launch, in cycles: 2100 of latency
// and 190 per warp and stage on the SM that has most of them, fitted to
// measured launches (8^3 to 128 x 128 x 5) to some 8 %. Only plans whose blocks
// are all resident at once (on the sms SMs of the device) are taken: 46^3 (two rounds of 800-thread blocks)
// measured 5.95 us a step against 4.13 one step per launch. A single step, in
// the same fit, costs 1150 + 165 per warp, and each launch its edge: 2240
// cycles (1.15 us) in a graph, 0.9 us more outside. Two steps per launch run
// where the model finds them cheaper, which may hold only outside a graph.
// us a step (graph / launched one by one), one step per launch -> two: 8^3
// 1.80 / 2.12 -> 1.31 / 1.45, 16 x 32 x 32 2.08 / 2.67 -> 1.69 / 2.44,
// 64 x 64 x 5 2.18 / 2.45 -> 1.82 / 2.27, 128 x 128 x 5 3.27 / 4.18 -> 3.23 /
// 3.16, 32^3 2.32 / 2.89 -> 2.45 / 2.61.
bool small_plan(const Geom &g, int sms, SmallPlan &p) {
    const int64_t n = (int64_t)g.nx * g.ny * g.nz;
    if (g.slab || n >= 100000) return false;
    double best = 1e300;
    auto sizes = [](int n, int most, auto use) {  // the axis whole, or its even splits
        for (int k = (n + most - 1) / most;;) {
            const int s = (n + k - 1) / k;  // the largest part of k even ones
            use(s, (n + s - 1) / s);
            if (s == 1) return;
            k = (n + s - 2) / (s - 1);  // the fewest parts that are smaller
        }
    };
    sizes(g.nx, 1024, [&](int bx, int nbx) {
        const int hx = nbx > 1, ex = bx + 2 * hx;
        if (ex > 1024 || (nbx > 1 && bx < 8)) return;
        sizes(g.ny, 1024 / ex, [&](int by, int nby) {
            const int hy = nby > 1, ey = by + 2 * hy;
            if (ex * ey > 1024) return;
            sizes(g.nz, 1024 / (ex * ey), [&](int bz, int nbz) {
                const int hz = nbz > 1, ez = bz + 2 * hz, ext = ex * ey * ez;
                if (ext > 1024) return;
                const int we = (ext + 31) / 32, wo = (bx * by * bz + 31) / 32;
                const int resident = std::min(32 / we, (int)(220 * 1024 / (ext * kQ * 4 + 1024)));
                if (resident < 1) return;
                const double blocks = (double)nbx * nby * nbz, per_sm = std::ceil(blocks / sms);
                if (per_sm > resident) return;
                const double cost = 2100.0 + per_sm * 190.0 * (we + wo);
                if (cost < best) {
                    best = cost;
                    p.bx = bx; p.by = by; p.bz = bz;
                    p.nbx = nbx; p.nby = nby; p.nbz = nbz;
                    p.hx = hx; p.hy = hy; p.hz = hz;
                    p.ex = ex; p.ey = ey; p.ext = ext;
                    p.threads = we * 32;
                }
            });
        });
    });
    const double edge = 2240.0, more = 1750.0, single = 1150.0 + 165.0 * std::ceil((double)n / ((double)sms * 32));
    if (best + edge + more >= 2.0 * (single + edge + more)) return false;
    p.in_graph = best + edge < 2.0 * (single + edge);
    // quotients of thread indices below 1024 by multiplication; a divisor of 1 has no such factor
    if (p.ex < 2 || p.bx < 2) return false;
    auto magic = [](int v) { return 0xffffffffu / (uint32_t)v + 1u; };
    p.exdiv = magic(p.ex);
    p.exydiv = magic(p.ex * p.ey);
    p.bxdiv = magic(p.bx);
    p.bxydiv = magic(p.bx * p.by);
    return true;
}

template <int FM, bool WALLS>
static cudaError_t small_t(const Launch &L, const SmallPlan &p, const float *src, float *dst, const Rates &r,
                           const ForceArgs &F, float scale2, int *flag) {
    const size_t smem = (size_t)kQ * p.ext * sizeof(float);
    if (smem > 48 * 1024) {
        // the shared-memory opt-in, once per device for this kernel; host threads
        // may race to set it, which repeats a harmless call
        static std::atomic<int> opted_in[64] = {};
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        if (dev >= 64 || !opted_in[dev].load(std::memory_order_relaxed)) {
            e = cudaFuncSetAttribute(k_step_small2<FM, WALLS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     kQ * 1024 * (int)sizeof(float));
            if (e != cudaSuccess) return e;
            if (dev < 64) opted_in[dev].store(1, std::memory_order_relaxed);
        }
    }
    return launch_overlapped(k_step_small2<FM, WALLS>, dim3(p.nbx * p.nby * p.nbz), dim3(p.threads), smem, L.stream,
                             L.overlap, src, dst, L.g, r, F, scale2, flag, p);
}

cudaError_t launch_step_small2(const Launch &L, const SmallPlan &p, const void *src, void *dst, const Rates &r,
                               const ForceArgs &F, float scale2, int *flag) {
    const float *s = (const float *)src;
    float *d = (float *)dst;
    auto walls = [&](auto fm) {
        constexpr int FM = decltype(fm)::value;
        return L.g.walls ? small_t<FM, true>(L, p, s, d, r, F, scale2, flag)
                         : small_t<FM, false>(L, p, s, d, r, F, scale2, flag);
    };
    switch (F.mode) {
        case kForceUniform: return walls(std::integral_constant<int, kForceUniform>{});
        case kForceProfileZ: return walls(std::integral_constant<int, kForceProfileZ>{});
        default: return walls(std::integral_constant<int, kForceField>{});
    }
}

}  // namespace clbm
