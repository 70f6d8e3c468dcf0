// step_small.cu -- plan and launch of the two-step kernel of small lattices
// (step_small.cuh).
#include <algorithm>
#include <cmath>

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
                const int resident = std::min({32 / we, 64 / we, (int)(220 * 1024 / (ext * kQ * 4 + 1024))});
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

template <int FM>
static cudaError_t small_t(const Launch &L, const SmallPlan &p, const float *src, float *dst, const Rates &r,
                           const ForceArgs &F, float scale2, int *flag) {
    auto go = [&](auto kern) -> cudaError_t {
        const size_t smem = (size_t)kQ * p.ext * sizeof(float);
        if (smem > 48 * 1024) {
            const cudaError_t e =
                cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kQ * 1024 * (int)sizeof(float));
            if (e != cudaSuccess) return e;
        }
        return launch_overlapped(kern, dim3(p.nbx * p.nby * p.nbz), dim3(p.threads), smem, L.stream, L.overlap, src,
                                 dst, L.g, r, F, scale2, flag, p);
    };
    return L.g.walls ? go(k_step_small2<FM, true>) : go(k_step_small2<FM, false>);
}

cudaError_t launch_step_small2(const Launch &L, const SmallPlan &p, const void *src, void *dst, const Rates &r,
                               const ForceArgs &F, float scale2, int *flag) {
    const float *s = (const float *)src;
    float *d = (float *)dst;
    switch (F.mode) {
        case kForceUniform: return small_t<kForceUniform>(L, p, s, d, r, F, scale2, flag);
        case kForceProfileZ: return small_t<kForceProfileZ>(L, p, s, d, r, F, scale2, flag);
        default: return small_t<kForceField>(L, p, s, d, r, F, scale2, flag);
    }
}

}  // namespace clbm
