// batch.cu -- many independent lattices of uneven sizes and parameters stepped
// by one launch per time step.
//
// Every domain is a complete D3Q19 lattice (its own extents, walls, relaxation
// rates and uniform body force) with the per-node update of the single-lattice
// kernel (pull, Eqs. 5, 7, 8, 9 in deviation form; see d3q19.cuh). The
// domains' populations share two A/B allocations, domain after domain, each in
// the single-lattice layout. A host-built work list cuts every domain into
// tiles of T consecutive nodes, or pairs of adjacent nodes, in its linear index
// (T = threads per block), so every lane has a node whatever the domain's
// extents, a warp reads contiguous memory, and only a domain's last tile is
// partial. One block takes one tile, or a grid of (SMs x resident blocks) walks
// the list with a stride (form_for): one launch covers all domains. Steps are
// replayed from a captured CUDA graph.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "../../include/clbm.h"
#include "kernels.cuh"
#include "step_pair.cuh"

using namespace clbm;

namespace clbm {

// Does the pull of node (x, y, z) meet a wall (a node on a wall face)?
__device__ __forceinline__ bool on_wall_face(const Geom &g, int x, int y, int z) {
    return ((g.walls & 1u) && (x == 0 || x == g.nx - 1)) || ((g.walls & 2u) && (y == 0 || y == g.ny - 1)) ||
           ((g.walls & 4u) && (z == 0 || z == g.nz - 1));
}

// Load the 19 populations arriving at (x, y, z) (pull map of Eq. 8). With
// walls, a warp none of whose nodes lies on a wall face takes the periodic
// map, whose array indices are constants; only warps that touch a wall face
// evaluate the bounce-back substitutions. Returns the node's offset. (On the
// single-lattice step the two code paths measured 2 % slower than the
// bounce-back map alone; on the batched step, whose domains all have walls,
// 1 % faster.)
template <typename S, bool WALLS>
__device__ __forceinline__ uint32_t pull_load(const S *src, const Geom &g, int x, int y, int z,
                                              float (&h)[kQ]) {
    uint32_t off[kQ];
    int pop[kQ];
    if (WALLS && __any_sync(__activemask(), on_wall_face(g, x, y, z))) {
        pull_sources<true>(g, x, y, z, off, pop);
#pragma unroll
        for (int i = 0; i < kQ; ++i) h[i] = Codec<S>::load(src + (size_t)pop[i] * g.stride + off[i]);
    } else {
        pull_sources<false>(g, x, y, z, off, pop);
#pragma unroll
        for (int i = 0; i < kQ; ++i) h[i] = Codec<S>::load(src + (size_t)i * g.stride + off[i]);
    }
    return off[0];
}

struct DomainDesc {
    Geom g;
    Rates r;
    float fx, fy, fz;
    float inv_nx, inv_ny;  // 1/nx, 1/ny (FP32) for the tile coordinate decode
    float inv_npx;         // 1/npx, npx = (nx + 1) / 2 node pairs per row
    int64_t offset;        // element offset of the domain's 19 x stride block in A and in B
};

// Blocks of 128 threads of the node-pair kernel that an SM holds (its launch bounds).
__host__ __device__ constexpr int pair_blocks(bool f32) { return f32 ? 6 : 5; }

// SMEM: the domain table is staged in shared memory once per launch (the
// usual case); otherwise it is read through the read-only cache. The next
// tile's entry is fetched while the current tile is processed. A tile is
// blockDim.x consecutive nodes of the domain, or pairs of adjacent nodes in
// the order of rows of (nx + 1) / 2 pairs, one per thread.
template <typename S, int NODES, bool SMEM>
__global__ void __launch_bounds__(512) k_batch_step(const S *A, S *__restrict__ B,
                                                    const DomainDesc *__restrict__ doms, int ndom,
                                                    const int4 *__restrict__ tiles, int ntiles,
                                                    int *__restrict__ flag) {
    extern __shared__ DomainDesc sdom[];
    int t = blockIdx.x;
    if (t >= ntiles) return;
    // the domain table and the work list stay unchanged while steps run; the first tile's entry is on its way while
    // the table is staged
    int4 tile = __ldg(tiles + t);  // (domain, x or pair of the row, y, z) of the tile's first node or pair
    if (SMEM) {
        for (int i = threadIdx.x; i < ndom; i += blockDim.x) sdom[i] = doms[i];
        __syncthreads();
    }
    grid_dependency_wait();
    for (; t < ntiles; t += gridDim.x) {
        const int tn = t + gridDim.x;
        const int4 next = tn < ntiles ? __ldg(tiles + tn) : tile;
        const DomainDesc *D = SMEM ? sdom + tile.x : doms + tile.x;
        const Geom g = D->g;
        // entry tile_start + threadIdx.x: carry x into y and y into z. The
        // quotients are below 2^17, so floor((v + 0.5) * (1/n)) in FP32 is exact.
        const int row = NODES == 2 ? (g.nx + 1) >> 1 : g.nx;
        const int xt = tile.y + (int)threadIdx.x;
        const int cy = (int)(((float)xt + 0.5f) * (NODES == 2 ? D->inv_npx : D->inv_nx));
        const int yt = tile.z + cy;
        const int cz = (int)(((float)yt + 0.5f) * D->inv_ny);
        const int x = NODES * (xt - cy * row), y = yt - cz * g.ny, z = tile.w + cz;
        if (z < g.nz) {
            const S *src = A + D->offset;
            S *dst = B + D->offset;
            if constexpr (NODES == 2) {
                const bool even = (g.nx & 1) == 0, two = x + 1 < g.nx;
                f2 h[kQ];
                const uint32_t self = even ? pair_load<S, true, true>(src, g, x, y, z, true, h)
                                           : pair_load<S, true, false>(src, g, x, y, z, two, h);
                const f2 drho = collide<true>(h, mk2(D->fx), mk2(D->fy), mk2(D->fz), D->r);
                if (!(fabsf(drho.v.x) < 0.9f) || !(fabsf(drho.v.y) < 0.9f)) *flag = 1;
                if (even)
                    pair_store<S, true>(dst, g, self, true, h, 0u);
                else
                    pair_store<S, false>(dst, g, self, two, h, 0u);
            } else {
                float h[kQ];
                const uint32_t self = pull_load<S, true>(src, g, x, y, z, h);
                const float drho = collide<sizeof(S) == 2>(h, D->fx, D->fy, D->fz, D->r);
                if (!(fabsf(drho) < 0.9f)) *flag = 1;
                store_node<S>(dst + self, g.stride, h, self, 0u);
            }
        }
        tile = next;
    }
}

// The A/B batch in node pairs, one block per tile (small tiles, see
// form_for): no loop state and no shared domain table, so that the FP32 pair
// keeps the 80 registers of six blocks of 128 per SM (12 bytes spilled).
template <typename S, int MAXT>
__global__ void __launch_bounds__(MAXT, pair_blocks(sizeof(S) == 4) * 128 / MAXT)
    k_batch_pair(const S *A, S *__restrict__ B, const DomainDesc *__restrict__ doms, const int4 *__restrict__ tiles,
                 int *__restrict__ flag) {
    const int4 tile = __ldg(tiles + blockIdx.x);  // (domain, pair of the row, y, z) of the tile's first pair
    const DomainDesc *D = doms + tile.x;
    const Geom g = D->g;
    const float inv_npx = D->inv_npx, inv_ny = D->inv_ny;
    const int64_t off = D->offset;
    grid_dependency_wait();  // (the domain table and the work list stay unchanged while steps run)
    const int npx = (g.nx + 1) >> 1;
    const int xt = tile.y + (int)threadIdx.x;
    const int cy = (int)(((float)xt + 0.5f) * inv_npx);
    const int yt = tile.z + cy;
    const int cz = (int)(((float)yt + 0.5f) * inv_ny);
    const int x = 2 * (xt - cy * npx), y = yt - cz * g.ny, z = tile.w + cz;
    if (z >= g.nz) return;
    const S *src = A + off;
    S *dst = B + off;
    const bool even = (g.nx & 1) == 0, two = x + 1 < g.nx;
    f2 h[kQ];
    if constexpr (sizeof(S) == 2) {
        const uint32_t self = even ? pair_load<S, true, true>(src, g, x, y, z, true, h)
                                   : pair_load<S, true, false>(src, g, x, y, z, two, h);
        const f2 drho = collide<true>(h, mk2(D->fx), mk2(D->fy), mk2(D->fz), D->r);
        if (!(fabsf(drho.v.x) < 0.9f) || !(fabsf(drho.v.y) < 0.9f)) *flag = 1;
        if (even)
            pair_store<S, true>(dst, g, self, true, h, 0u);
        else
            pair_store<S, false>(dst, g, self, two, h, 0u);
    } else {  // the pull of k_step_pair, rows of either parity
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
            const float *base = src + (size_t)i * g.stride;
            const uint32_t row =
                (ez19(i) > 0 ? zm : (ez19(i) < 0 ? zp : zc)) + (ey19(i) > 0 ? rm : (ey19(i) < 0 ? rp : rc));
            if (ex19(i) > 0)
                h[i] = mk2(ld_state(CLBM_AT(g, src, base, row + xam, 0u)), ld_state(CLBM_AT(g, src, base, row + (two ? xa : xam), 0u)));
            else if (ex19(i) < 0)
                h[i] = mk2(ld_state(CLBM_AT(g, src, base, row + (two ? xb : xbp), 0u)), ld_state(CLBM_AT(g, src, base, row + xbp, 0u)));
            else if (even)
                h[i] = f2{ld_state2(CLBM_AT(g, src, base, row + xa, 1u))};
            else
                h[i] = mk2(ld_state(CLBM_AT(g, src, base, row + xa, 0u)), ld_state(CLBM_AT(g, src, base, row + xb, 0u)));
        }
        const WallFaces wa = wall_faces(g, (int)xa, y, z), wb = wall_faces(g, (int)xb, y, z);
        if (wa.any() || wb.any()) {
#pragma unroll
            for (int i = 1; i < kQ; ++i) {
                const float *base = src + (size_t)opposite(i) * g.stride;
                if (wa.bounces(i)) h[i].v.x = ld_state(CLBM_AT(g, src, base, self, 0u));
                if (wb.bounces(i)) h[i].v.y = ld_state(CLBM_AT(g, src, base, self + (xb - xa), 0u));
            }
        }
        const f2 drho = collide<false>(h, mk2(D->fx), mk2(D->fy), mk2(D->fz), D->r);
        if (!(fabsf(drho.v.x) < 0.9f) || !(fabsf(drho.v.y) < 0.9f)) *flag = 1;
#pragma unroll
        for (int i = 0; i < kQ; ++i) {
            float *to = dst + (size_t)i * g.stride + CLBM_SLOTS(g, self, (kQ - 1) * g.stride + (xb - xa));
            if (even) {
                *reinterpret_cast<float2 *>(to) = h[i].v;
            } else {
                to[0] = h[i].v.x;
                if (two) to[1] = h[i].v.y;
            }
        }
    }
}

// The in-place (AA) pattern over the batch: every domain's one population
// array, even and odd step kinds as k_step_aa (step_kernels.cuh): the even
// kind reads a node's own slots and writes population i into the slot of
// ibar; the odd kind reads (ibar, x - e_i), or (i, x) across a wall, and writes
// population i to (i, x + e_i), or (ibar, x) across a wall. The same tiles,
// domain table and collision as k_batch_step, so the batch stores the bits of
// the A/B batch and of each domain stepped alone.
// The even kind with FP32 wants 84 registers: capped at two blocks of 512 (64)
// an in-place step of the benchmark's 64 domains takes 946 instead of 977 us
// (tile of 128; with a table too large for shared memory the cap spills 24
// bytes, 390 us for 600 small domains either way).
template <typename S, bool SMEM, bool ODD>
__global__ void __launch_bounds__(512, ODD || sizeof(S) == 2 ? 0 : 2) k_batch_step_aa(S *A, const DomainDesc *__restrict__ doms, int ndom,
                                                       const int4 *__restrict__ tiles, int ntiles,
                                                       int *__restrict__ flag) {
    extern __shared__ DomainDesc sdom[];
    int t = blockIdx.x;
    if (t >= ntiles) return;
    // the domain table and the work list stay unchanged while steps run; the first tile's entry is on its way while
    // the table is staged
    int4 tile = __ldg(tiles + t);
    if (SMEM) {
        for (int i = threadIdx.x; i < ndom; i += blockDim.x) sdom[i] = doms[i];
        __syncthreads();
    }
    grid_dependency_wait();
    for (; t < ntiles; t += gridDim.x) {
        const int tn = t + gridDim.x;
        const int4 next = tn < ntiles ? __ldg(tiles + tn) : tile;
        const DomainDesc *D = SMEM ? sdom + tile.x : doms + tile.x;
        const Geom g = D->g;
        const int xt = tile.y + (int)threadIdx.x;
        const int cy = (int)(((float)xt + 0.5f) * D->inv_nx);
        const int yt = tile.z + cy;
        const int cz = (int)(((float)yt + 0.5f) * D->inv_ny);
        const int x = xt - cy * g.nx, y = yt - cz * g.ny, z = tile.w + cz;
        if (z < g.nz) {
            S *f = A + D->offset;
            const uint32_t self = ((uint32_t)z * g.ny + y) * g.nx + x;
            float h[kQ];
            if (ODD) {
                uint32_t off[kQ];
                int pop[kQ];
                pull_sources<true, true>(g, x, y, z, off, pop);
#pragma unroll
                for (int i = 0; i < kQ; ++i) h[i] = Codec<S>::load(f + CLBM_IDX(g, (size_t)pop[i] * g.stride + off[i]));
                const float drho = collide<sizeof(S) == 2>(h, D->fx, D->fy, D->fz, D->r);
                if (!(fabsf(drho) < 0.9f)) *flag = 1;
                // the push targets from coordinates the compiler must treat as new (as in k_step_aa)
                int xs = x, ys = y, zs = z;
                asm volatile("" : "+r"(xs), "+r"(ys), "+r"(zs) : "f"(h[0]), "f"(h[kQ - 1]));
                push_targets<true>(g, xs, ys, zs, off, pop);
                store_each<S, kQ>(h, self, 0u,
                                  [&](int i) { return f + CLBM_IDX(g, (size_t)pop[i] * g.stride + off[i]); });
            } else {
#pragma unroll
                for (int i = 0; i < kQ; ++i) h[i] = Codec<S>::load(f + CLBM_IDX(g, (size_t)i * g.stride + self));
                const float drho = collide<sizeof(S) == 2>(h, D->fx, D->fy, D->fz, D->r);
                if (!(fabsf(drho) < 0.9f)) *flag = 1;
                store_each<S, kQ>(h, self, 0u,
                                  [&](int i) { return f + CLBM_IDX(g, (size_t)opposite(i) * g.stride + self); });
            }
        }
        tile = next;
    }
}

constexpr int kSmemDomains = 512;  // domain tables up to this size are staged in shared memory

// The kernel of one step: how a batch's work list is cut and walked.
struct BatchForm {
    int threads = 0;
    bool pairs = false;     // A/B: a thread takes two adjacent nodes instead of one
    bool per_tile = false;  // ... and a block one tile (k_batch_pair); otherwise resident blocks walk the tiles
};

// The step kernel of a form (A/B; in place, of one kind) through `use`.
template <typename S, typename Use>
static auto with_kernel(const BatchForm &f, int ndom, Use use) {
    const bool sm = ndom <= kSmemDomains;
    if constexpr (sizeof(S) == 2)  // (FP32 pairs take one block per tile)
        if (f.pairs) return use(sm ? k_batch_step<S, 2, true> : k_batch_step<S, 2, false>);
    return use(sm ? k_batch_step<S, 1, true> : k_batch_step<S, 1, false>);
}
template <typename S, typename Use>
static auto with_kernel_aa(bool odd, int ndom, Use use) {
    const bool sm = ndom <= kSmemDomains;
    if (odd) return use(sm ? k_batch_step_aa<S, true, true> : k_batch_step_aa<S, false, true>);
    return use(sm ? k_batch_step_aa<S, true, false> : k_batch_step_aa<S, false, false>);
}

static size_t table_bytes(int ndom) { return ndom <= kSmemDomains ? sizeof(DomainDesc) * ndom : 0; }

template <typename S>
static cudaError_t batch_launch_t(const BatchForm &f, const void *A, void *B, const DomainDesc *doms, int ndom,
                                  const int4 *tiles, int ntiles, int grid, int *flag, cudaStream_t s, bool overlap) {
    const dim3 block(f.threads);
    if (f.per_tile) {
        auto go = [&](auto kern) {
            return launch_overlapped(kern, dim3(ntiles), block, 0, s, overlap, (const S *)A, (S *)B, doms, tiles, flag);
        };
        if constexpr (sizeof(S) == 4)
            if (f.threads > 128) return go(k_batch_pair<S, 256>);
        return go(k_batch_pair<S, 128>);
    }
    return with_kernel<S>(f, ndom, [&](auto kern) {
        return launch_overlapped(kern, dim3(grid), block, table_bytes(ndom), s, overlap, (const S *)A, (S *)B, doms,
                                 ndom, tiles, ntiles, flag);
    });
}

template <typename S>
static cudaError_t batch_launch_aa_t(const BatchForm &f, void *A, const DomainDesc *doms, int ndom, const int4 *tiles,
                                     int ntiles, int grid, int *flag, cudaStream_t s, bool overlap, bool odd) {
    return with_kernel_aa<S>(odd, ndom, [&](auto kern) {
        return launch_overlapped(kern, dim3(grid), dim3(f.threads), table_bytes(ndom), s, overlap, (S *)A, doms, ndom,
                                 tiles, ntiles, flag);
    });
}

template <typename Use>
static auto with_storage(int storage, Use use) {
    switch (storage) {
        case 0: return use(float{});
        case 1: return use(__half{});
        default: return use(__nv_bfloat16{});
    }
}

// Resident blocks per SM of the kernel that walks the tiles (in place: of the kind `odd`).
static int resident_blocks(int storage, const BatchForm &f, bool aa, bool odd, int ndom) {
    auto ask = [&](auto kern) {
        int per_sm = 0;
        const cudaError_t e =
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, f.threads, table_bytes(ndom));
        return e == cudaSuccess && per_sm > 0 ? per_sm : 1;
    };
    return with_storage(storage, [&](auto s) {
        using S = decltype(s);
        return aa ? with_kernel_aa<S>(odd, ndom, ask) : with_kernel<S>(f, ndom, ask);
    });
}

}  // namespace clbm

struct clbm_batch {
    std::vector<clbm_domain> host;
    std::vector<DomainDesc> descs;
    int ndom;
    int storage;
    size_t elem;
    int64_t total_nodes, total_elems;
    void *buf[2];
    int cur;
    cudaStream_t stream, capture_stream;
    DomainDesc *d_descs;
    int4 *d_tiles;
    int ntiles, tiles_cap;
    BatchForm form;
    int grid[2];  // of a step; in place: of the even and of the odd kind
    int *d_flag;
    cudaGraphExec_t graph;
    int graph_steps;
    int64_t steps_done;
    int sms;  // of the device
    bool aa;  // in-place pattern: one buffer (buf[1] == buf[0]), step kind by the parity of steps_done
};

namespace {

int bfail(int code, const std::string &msg) { return clbm::set_error(code, msg.c_str()); }

int bcuda(cudaError_t e, const char *where) {
    return bfail(CLBM_ERR_CUDA, std::string(where) + ": " + cudaGetErrorString(e));
}

Launch domain_launch(const clbm_batch *b, int d) {
    const Geom &g = b->descs[d].g;
    Launch L;
    L.g = g;
    const int bx = default_block_x(g.nx);
    const int by = std::max(1, std::min(g.ny, 128 / bx));
    L.block = dim3(bx, by, 1);
    L.grid = dim3((g.nx + bx - 1) / bx, (g.ny + by - 1) / by, g.nz);
    L.stream = b->stream;
    L.overlap = stream_overlaps(b->stream);
    L.packed = false;
    L.staged = false;  // the per-domain schedule runs the one-node kernels
    // state maps: A/B pull map; in place, natural slots after an even number of steps, the odd map after an odd
    L.map = b->aa ? ((b->steps_done & 1) ? 2 : 1) : 0;
    return L;
}

ForceArgs domain_force(const clbm_batch *b, int d) {
    ForceArgs F;
    F.mode = kForceUniform;
    F.fx = b->descs[d].fx; F.fy = b->descs[d].fy; F.fz = b->descs[d].fz;
    F.profile = nullptr;
    F.field = nullptr;
    F.n = (int64_t)b->descs[d].g.nx * b->descs[d].g.ny * b->descs[d].g.nz;
    F.scale = 1.0f;
    return F;
}

void *domain_ptr(const clbm_batch *b, int which, int d) {
    return (char *)b->buf[which] + (size_t)b->descs[d].offset * b->elem;
}

// The form a batch steps in with tiles of T threads (us a step of batches of
// channels and ducts):
// A/B, by size (nodes): below 1.2 rounds of resident pair blocks (FP32 280,000,
//   16-bit 233,000) one node per thread: half as many warps of pairs leave
//   schedulers idle (T = 128, one node / pairs: FP16 45k 2.97 / 3.49, 94k 4.14
//   / 4.75, 234k 6.94 / 6.95, 352k 9.76 / 9.00; FP32 94k 4.24 / 4.64, 234k 6.70
//   / 7.25, 352k 9.45 / 8.92);
// above that by T:
//   up to 256 (FP32) or 128 (16-bit): pairs, one block per tile: FP32 897 (T =
//     128) and 929 (256) on 39 M nodes, FP16 708 (128);
//   larger: resident blocks walk the tiles, one node per thread with FP32 (976
//     at 512; a walking pair takes 108 registers), pairs with 16 bits (726 at
//     256, 667 at 512).
BatchForm form_for(const clbm_batch &b, int T) {
    BatchForm f;
    f.threads = T;
    const bool f32 = b.storage == CLBM_STORAGE_F32;
    if (b.aa || (double)b.total_nodes < 1.2 * b.sms * pair_blocks(f32) * 256) return f;
    f.per_tile = T <= (f32 ? 256 : 128);
    f.pairs = f.per_tile || !f32;
    return f;
}

// Build and upload the work list for T threads per block: tiles of T
// consecutive nodes, or pairs of nodes, domain after domain.
int build_tiles(clbm_batch *b, int T) {
    const BatchForm form = form_for(*b, T);
    std::vector<int4> tiles;
    for (int d = 0; d < b->ndom; ++d) {
        const Geom &g = b->descs[d].g;
        const int64_t row = form.pairs ? (g.nx + 1) / 2 : g.nx;
        const int64_t n = row * g.ny * g.nz;
        for (int64_t s0 = 0; s0 < n; s0 += T) {
            const int x = (int)(s0 % row);
            const int64_t r = s0 / row;
            tiles.push_back(make_int4(d, x, (int)(r % g.ny), (int)(r / g.ny)));
        }
    }
    if (tiles.size() > (size_t)INT32_MAX) return bfail(CLBM_ERR_ARG, "clbm_batch: too many tiles");
    if ((int)tiles.size() > b->tiles_cap) {
        if (b->d_tiles) cudaFree(b->d_tiles);
        b->d_tiles = nullptr;
        cudaError_t e = cudaMalloc(&b->d_tiles, tiles.size() * sizeof(int4));
        if (e != cudaSuccess) {
            b->tiles_cap = 0;
            cudaGetLastError();
            return bfail(CLBM_ERR_OOM, "clbm_batch: cudaMalloc of the work list failed");
        }
        b->tiles_cap = (int)tiles.size();
    }
    cudaError_t e = cudaMemcpyAsync(b->d_tiles, tiles.data(), tiles.size() * sizeof(int4), cudaMemcpyHostToDevice,
                                    b->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) return bcuda(e, "clbm_batch: work list upload");
    b->ntiles = (int)tiles.size();
    b->form = form;
    for (int odd = 0; odd < 2; ++odd)
        b->grid[odd] = form.per_tile
                           ? b->ntiles
                           : std::min(b->ntiles, b->sms * resident_blocks(b->storage, form, b->aa, odd, b->ndom));
    if (b->graph) {
        cudaGraphExecDestroy(b->graph);
        b->graph = nullptr;
    }
    return CLBM_OK;
}

// The tile size a batch starts with (clbm_batch_autotune finds its own), us a step:
// A/B: 128; 512 for 16-bit batches of 30 rounds of resident 512-thread blocks or
//   more (one block per SM, 1024-node tiles: 4.7 M nodes), whose last round no
//   longer counts: FP16 128 / 512: 0.5 M nodes 12.0 / 15.0, 2.2 M 46.1 / 47.1,
//   4.5 M 88.7 / 88.5, 36 M 657 / 617.
// In place: 128; 16-bit batches 512 from 700,000 nodes on and 256 from 3 M on,
//   where the populations no longer fit the L2: FP16 128 / 256 / 512: 0.5 M
//   14.7 / 15.2 / 15.3, 1.7 M 45.1 / 43.9 / 43.6, 4.5 M 126.7 / 127.3 / 130.4,
//   36 M 981 / 972 / 981 (FP32 36 M 1036 / 1063 / 1151).
int default_tile(const clbm_batch &b) {
    if (b.storage == CLBM_STORAGE_F32) return 128;
    if (b.aa) return b.total_nodes < 700000 ? 128 : (b.total_nodes < 3000000 ? 512 : 256);
    return b.total_nodes < (int64_t)30 * b.sms * 1024 ? 128 : 512;
}

// One step of every domain: A/B from buffer `from`; in place, the odd kind when
// `from` is 1 (the parity of the step).
cudaError_t launch_all(clbm_batch *b, cudaStream_t s, int from) {
    const bool overlap = stream_overlaps(s);
    return with_storage(b->storage, [&](auto v) {
        using S = decltype(v);
        return b->aa ? batch_launch_aa_t<S>(b->form, b->buf[0], b->d_descs, b->ndom, b->d_tiles, b->ntiles,
                                            b->grid[from], b->d_flag, s, overlap, from == 1)
                     : batch_launch_t<S>(b->form, b->buf[from], b->buf[from ^ 1], b->d_descs, b->ndom, b->d_tiles,
                                         b->ntiles, b->grid[0], b->d_flag, s, overlap);
    });
}

// Capture graph_steps steps starting from buffer 0 (in place: from an even
// step); graph_steps is even, so the replay ends there again.
int ensure_graph(clbm_batch *b) {
    if (b->graph) return CLBM_OK;
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaStreamBeginCapture(b->capture_stream, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return bcuda(e, "clbm_batch: begin capture");
    for (int k = 0; k < b->graph_steps && e == cudaSuccess; ++k) e = launch_all(b, b->capture_stream, k & 1);
    cudaError_t e2 = cudaStreamEndCapture(b->capture_stream, &g);
    if (e == cudaSuccess) e = e2;
    if (e == cudaSuccess) e = cudaGraphInstantiate(&b->graph, g, 0);
    if (g) cudaGraphDestroy(g);
    if (e != cudaSuccess) {
        b->graph = nullptr;
        return bcuda(e, "clbm_batch: graph capture");
    }
    return CLBM_OK;
}

}  // namespace

extern "C" {

int clbm_batch_create(const clbm_domain *doms, int32_t ndomains, int32_t storage, void *stream, clbm_batch **out) {
    return clbm_batch_create_pattern(doms, ndomains, storage, CLBM_PATTERN_AB, stream, out);
}

int clbm_batch_create_pattern(const clbm_domain *doms, int32_t ndomains, int32_t storage, int32_t pattern,
                              void *stream, clbm_batch **out) {
    if (!doms || !out || ndomains < 1) return bfail(CLBM_ERR_ARG, "clbm_batch_create: bad argument");
    *out = nullptr;
    if (pattern != CLBM_PATTERN_AB && pattern != CLBM_PATTERN_AA)
        return bfail(CLBM_ERR_ARG, "clbm_batch_create: pattern must be CLBM_PATTERN_AB or CLBM_PATTERN_AA");
    if (storage < CLBM_STORAGE_F32 || storage > CLBM_STORAGE_BF16)
        return bfail(CLBM_ERR_ARG, "clbm_batch_create: storage must be f32, f16 or bf16 (round to nearest)");
    clbm_batch *b = new (std::nothrow) clbm_batch();
    if (!b) return bfail(CLBM_ERR_OOM, "clbm_batch_create: host allocation failed");
    b->ndom = ndomains;
    b->storage = storage;
    b->aa = pattern == CLBM_PATTERN_AA;
    b->elem = storage == CLBM_STORAGE_F32 ? 4 : 2;
    b->stream = (cudaStream_t)stream;
    b->graph_steps = 16;
    int64_t off = 0, nodes = 0;
    for (int d = 0; d < ndomains; ++d) {
        const clbm_domain &p = doms[d];
        const double s2 = 1.0 / (3.0 * p.nu + 0.5);
        auto ok = [](double s) { return std::isfinite(s) && s > 0.0 && s < 2.0; };
        const int64_t n = (int64_t)p.nx * p.ny * p.nz;
        if (p.nx < 1 || p.ny < 1 || p.nz < 1 || p.nx > 65535 || p.ny > 65535 || p.nz > 65535 ||
            n > ((int64_t)1 << 31) - 1 || (p.walls & ~7u) || !(std::isfinite(p.nu) && p.nu > 0.0) || !ok(s2) ||
            !ok(p.s2b) || !ok(p.s3) || !ok(p.s4) || !std::isfinite(p.fx) || !std::isfinite(p.fy) ||
            !std::isfinite(p.fz)) {
            delete b;
            return bfail(CLBM_ERR_ARG, "clbm_batch_create: invalid domain " + std::to_string(d));
        }
        DomainDesc D;
        std::memset(&D, 0, sizeof(D));
        D.g.nx = p.nx; D.g.ny = p.ny; D.g.nz = p.nz;
        D.g.walls = p.walls;
        D.g.stride = (n + 63) / 64 * 64;
#ifdef CLBM_BOUNDS_CHECK
        D.g.bc_limit = (uint64_t)kQ * D.g.stride;  // the domain's own arrays
#endif
        D.r.om2 = (float)(1.0 - s2);
        D.r.cb = (float)((p.s2b - s2) / 3.0);
        D.r.om3 = (float)(1.0 - p.s3);
        D.r.c3 = (float)((1.0 - 0.5 * p.s3) / 3.0);
        D.r.om4 = (float)(1.0 - p.s4);
        D.fx = (float)p.fx; D.fy = (float)p.fy; D.fz = (float)p.fz;
        D.inv_nx = 1.0f / (float)p.nx;
        D.inv_ny = 1.0f / (float)p.ny;
        D.inv_npx = 1.0f / (float)((p.nx + 1) / 2);
        D.offset = off;
        off += (int64_t)kQ * D.g.stride;
        nodes += n;
        b->descs.push_back(D);
        b->host.push_back(p);
    }
    b->total_nodes = nodes;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&b->sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || b->sms < 1) {
        cudaGetLastError();
        b->sms = 1;
    }
    b->total_elems = off;
    const size_t nbuf = b->aa ? 1 : 2;
    cudaError_t e = cudaMalloc(&b->buf[0], nbuf * (size_t)off * b->elem);
    if (e != cudaSuccess) {
        delete b;
        cudaGetLastError();
        return bfail(CLBM_ERR_OOM, "clbm_batch_create: cudaMalloc of the populations failed");
    }
    b->buf[1] = b->aa ? b->buf[0] : (char *)b->buf[0] + (size_t)off * b->elem;
    if ((e = cudaMalloc(&b->d_descs, sizeof(DomainDesc) * ndomains + 256)) != cudaSuccess) {
        cudaFree(b->buf[0]);
        delete b;
        cudaGetLastError();
        return bfail(CLBM_ERR_OOM, "clbm_batch_create: cudaMalloc failed");
    }
    b->d_flag = (int *)((char *)b->d_descs + sizeof(DomainDesc) * ndomains);
    b->d_flag = (int *)(((uintptr_t)b->d_flag + 15) & ~(uintptr_t)15);
    if ((e = cudaStreamCreateWithFlags(&b->capture_stream, cudaStreamNonBlocking)) != cudaSuccess) {
        cudaFree(b->d_descs);
        cudaFree(b->buf[0]);
        delete b;
        return bcuda(e, "clbm_batch_create: stream");
    }
#ifdef CLBM_BOUNDS_CHECK
    for (DomainDesc &D : b->descs) D.g.bc = (BoundsRecord *)((char *)b->d_flag + 64);  // the flag block's bytes 64-79
#endif
    e = cudaMemcpyAsync(b->d_descs, b->descs.data(), sizeof(DomainDesc) * ndomains, cudaMemcpyHostToDevice,
                        b->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(b->d_flag, 0, 128, b->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(b->buf[0], 0, nbuf * (size_t)off * b->elem, b->stream);
    int rc = e == cudaSuccess ? build_tiles(b, default_tile(*b)) : bcuda(e, "clbm_batch_create");
    if (rc != CLBM_OK) {
        clbm_batch_destroy(b);
        return rc;
    }
    *out = b;
    return CLBM_OK;
}

int clbm_batch_destroy(clbm_batch *b) {
    if (!b) return CLBM_OK;
    cudaStreamSynchronize(b->stream);
    if (b->graph) cudaGraphExecDestroy(b->graph);
    if (b->capture_stream) cudaStreamDestroy(b->capture_stream);
    if (b->d_tiles) cudaFree(b->d_tiles);
    if (b->d_descs) cudaFree(b->d_descs);
    if (b->buf[0]) cudaFree(b->buf[0]);
    delete b;
    return CLBM_OK;
}

int clbm_batch_get_info(const clbm_batch *b, clbm_batch_info *info) {
    if (!b || !info) return bfail(CLBM_ERR_ARG, "clbm_batch_get_info: null pointer");
    info->ndomains = b->ndom;
    info->total_nodes = b->total_nodes;
    info->state_bytes = (int64_t)b->total_elems * (int64_t)b->elem;
    info->ntiles = b->ntiles;
    info->grid = b->grid[0];
    info->threads = b->form.threads;
    info->graph_steps = b->graph_steps;
    info->steps_done = b->steps_done;
    info->pattern = b->aa ? CLBM_PATTERN_AA : CLBM_PATTERN_AB;
    info->buffers = b->aa ? 1 : 2;
    return CLBM_OK;
}

int clbm_batch_set_tile(clbm_batch *b, int32_t threads) {
    if (!b || threads < 32 || threads % 32 != 0 || threads > 512)
        return bfail(CLBM_ERR_ARG, "clbm_batch_set_tile: threads must be a multiple of 32 in [32, 512]");
    return build_tiles(b, threads);
}

int clbm_batch_autotune(clbm_batch *b, int32_t trial_steps, int32_t *threads_out) {
    if (!b || trial_steps < 1) return bfail(CLBM_ERR_ARG, "clbm_batch_autotune: bad argument");
    static const int cand[] = {64, 128, 192, 256, 384, 512};
    // in place, a trial step overwrites the state: keep a copy and put it back after the trials
    void *saved = nullptr;
    const size_t sbytes = (size_t)b->total_elems * b->elem;
    if (b->aa) {
        cudaError_t e = cudaMalloc(&saved, sbytes);
        if (e != cudaSuccess) {
            cudaGetLastError();
            return bfail(CLBM_ERR_OOM, "clbm_batch_autotune: no room for the copy of an in-place state");
        }
        if ((e = cudaMemcpyAsync(saved, b->buf[0], sbytes, cudaMemcpyDeviceToDevice, b->stream)) != cudaSuccess) {
            cudaFree(saved);
            return bcuda(e, "clbm_batch_autotune: save");
        }
    }
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    float best = 1e30f;
    int bt = 256;
    int rc = CLBM_OK;
    for (int T : cand) {
        if ((rc = build_tiles(b, T)) != CLBM_OK) break;
        // A/B trials read the current buffer and write the other one: the state is unchanged. In place they
        // are steps of alternating kind from the current parity on the saved state, restored afterwards.
        int ph = b->aa ? (int)(b->steps_done & 1) : b->cur;
        auto trial = [&]() {
            cudaError_t r = launch_all(b, b->stream, ph);
            if (b->aa) ph ^= 1;
            return r;
        };
        cudaError_t e = trial();
        if (e == cudaSuccess) e = cudaEventRecord(e0, b->stream);
        for (int k = 0; k < trial_steps && e == cudaSuccess; ++k) e = trial();
        if (e == cudaSuccess) e = cudaEventRecord(e1, b->stream);
        if (e == cudaSuccess) e = cudaEventSynchronize(e1);
        float ms = 0.f;
        if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
        if (e != cudaSuccess) {
            rc = bcuda(e, "clbm_batch_autotune");
            break;
        }
        if (ms < best) {
            best = ms;
            bt = T;
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (saved) {
        cudaError_t e = cudaMemcpyAsync(b->buf[0], saved, sbytes, cudaMemcpyDeviceToDevice, b->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
        cudaFree(saved);
        if (e != cudaSuccess && rc == CLBM_OK) rc = bcuda(e, "clbm_batch_autotune: restore");
    }
    if (rc != CLBM_OK) return rc;
    if ((rc = build_tiles(b, bt)) != CLBM_OK) return rc;
    if (threads_out) *threads_out = bt;
    return CLBM_OK;
}

int clbm_batch_init_equilibrium(clbm_batch *b) {
    if (!b) return bfail(CLBM_ERR_ARG, "clbm_batch_init_equilibrium: null pointer");
    b->steps_done = 0;  // before domain_launch: the in-place pattern starts in natural order
    for (int d = 0; d < b->ndom; ++d) {
        cudaError_t e = launch_init_eq(b->storage, domain_launch(b, d), domain_ptr(b, b->cur, d), nullptr, nullptr,
                                       domain_force(b, d).n, domain_force(b, d));
        if (e != cudaSuccess) return bcuda(e, "clbm_batch_init_equilibrium");
    }
    b->steps_done = 0;
    return CLBM_OK;
}

int clbm_batch_step(clbm_batch *b, int64_t nsteps, int32_t mode) {
    if (!b || nsteps < 0 || mode < 0 || mode > 2) return bfail(CLBM_ERR_ARG, "clbm_batch_step: bad argument");
    Range range("clbm_batch_step");
    cudaError_t e = cudaSuccess;
    int64_t t = 0;
    // the phase of the next step: the buffer (A/B) or the parity of the step (in place)
    auto phase = [&]() { return b->aa ? (int)((b->steps_done + t) & 1) : b->cur; };
    if (mode == CLBM_BATCH_GRAPH && nsteps >= b->graph_steps) {
        int rc = ensure_graph(b);
        if (rc != CLBM_OK) return rc;
        if (phase() == 1) {  // the graph starts from phase 0
            if ((e = launch_all(b, b->stream, 1)) != cudaSuccess) return bcuda(e, "clbm_batch_step");
            if (!b->aa) b->cur = 0;
            ++t;
        }
        for (; t + b->graph_steps <= nsteps; t += b->graph_steps)
            if ((e = cudaGraphLaunch(b->graph, b->stream)) != cudaSuccess) return bcuda(e, "clbm_batch_step: graph");
    }
    for (; t < nsteps; ++t) {
        if (mode == CLBM_BATCH_PER_DOMAIN) {
            const bool odd = phase() == 1;
            for (int d = 0; d < b->ndom && e == cudaSuccess; ++d) {
                Rates r = b->descs[d].r;
                if (b->aa)
                    e = launch_step_aa(b->storage, domain_launch(b, d), domain_ptr(b, 0, d), r, domain_force(b, d),
                                       b->d_flag, 0u, odd);
                else
                    e = launch_step(b->storage, domain_launch(b, d), domain_ptr(b, b->cur, d),
                                    domain_ptr(b, b->cur ^ 1, d), r, domain_force(b, d), b->d_flag, 0u);
            }
        } else {
            e = launch_all(b, b->stream, phase());
        }
        if (e != cudaSuccess) return bcuda(e, "clbm_batch_step");
        if (!b->aa) b->cur ^= 1;
    }
    b->steps_done += nsteps;
    return CLBM_OK;
}

int clbm_batch_get_macros(clbm_batch *b, int32_t d, float *rho, float *u) {
    if (!b || d < 0 || d >= b->ndom) return bfail(CLBM_ERR_ARG, "clbm_batch_get_macros: bad domain");
    if (!rho && !u) return CLBM_OK;
    cudaError_t e = launch_macros(b->storage, domain_launch(b, d), domain_ptr(b, b->cur, d), domain_force(b, d),
                                  rho, u, domain_force(b, d).n);
    if (e != cudaSuccess) return bcuda(e, "clbm_batch_get_macros");
    return CLBM_OK;
}

int clbm_batch_get_populations(clbm_batch *b, int32_t d, float *f, int deviation) {
    if (!b || !f || d < 0 || d >= b->ndom) return bfail(CLBM_ERR_ARG, "clbm_batch_get_populations: bad argument");
    cudaError_t e =
        launch_gather(b->storage, domain_launch(b, d), domain_ptr(b, b->cur, d), f, domain_force(b, d).n, deviation);
    if (e != cudaSuccess) return bcuda(e, "clbm_batch_get_populations");
    return CLBM_OK;
}

int clbm_batch_set_populations(clbm_batch *b, int32_t d, const float *f, int deviation) {
    if (!b || !f || d < 0 || d >= b->ndom) return bfail(CLBM_ERR_ARG, "clbm_batch_set_populations: bad argument");
    cudaError_t e = launch_scatter(b->storage, domain_launch(b, d), domain_ptr(b, b->cur, d), f,
                                   domain_force(b, d).n, deviation);
    if (e != cudaSuccess) return bcuda(e, "clbm_batch_set_populations");
    return CLBM_OK;
}

int clbm_batch_check(clbm_batch *b, int clear) {
    if (!b) return bfail(CLBM_ERR_ARG, "clbm_batch_check: null pointer");
    int h = 0;
    cudaError_t e = cudaMemcpyAsync(&h, b->d_flag, sizeof(int), cudaMemcpyDeviceToHost, b->stream);
#ifdef CLBM_BOUNDS_CHECK
    BoundsRecord rec = {0ull, 0ull};
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(&rec, (char *)b->d_flag + 64, sizeof(rec), cudaMemcpyDeviceToHost, b->stream);
#endif
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
    if (e == cudaSuccess && clear) e = cudaMemsetAsync(b->d_flag, 0, 128, b->stream);
    if (e != cudaSuccess) return bcuda(e, "clbm_batch_check");
#ifdef CLBM_BOUNDS_CHECK
    if (rec.count)
        return bfail(CLBM_ERR_BOUNDS, "clbm_batch_check: " + std::to_string(rec.count) +
                                          " out-of-range indices; the first: kind " + std::to_string(rec.first >> 56) +
                                          ", index " + std::to_string(rec.first & 0x00ffffffffffffffull));
#endif
    if (h) return bfail(CLBM_ERR_UNSTABLE, "clbm_batch_check: a node's density left (0.1, 1.9) or became non-finite");
    return CLBM_OK;
}

}  // extern "C"
