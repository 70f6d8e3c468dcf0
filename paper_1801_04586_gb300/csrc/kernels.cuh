// kernels.cuh -- launch interface between the C ABI (capi.cu) and the kernel
// translation units. Plain structs only.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "d3q19.cuh"

namespace clbm {

// Every kernel of the step path starts with this: it lets the next launch of
// the stream be set up while this one runs, and waits until the grids it
// depends on have completed and their writes are visible. Nothing before it
// may touch global memory, and no load of the kernel may go through the
// read-only path (__ldg, const __restrict__): what it reads can have been
// written while it was already resident.
__device__ __forceinline__ void grid_dependency_wait() {
    asm volatile("griddepcontrol.launch_dependents;\n\tgriddepcontrol.wait;" ::: "memory");
}

// Launch a kernel that begins with grid_dependency_wait() so that it may
// become resident while its predecessor in the stream drains (programmatic
// stream serialization) if overlap is set. From kernel to kernel in a stream
// that takes about 1.5 us instead of 4.1 (144 blocks of 128 threads that move
// one float each). Launches captured into a graph, the library's or a
// caller's, do without (stream_overlaps): there a plain edge takes 1.15 us, and
// early-resident blocks crowd onto the SMs that the running kernel leaves free
// (the 16 x 32 x 32 channel: 2.7 against 2.2 us a step).
inline bool stream_overlaps(cudaStream_t stream) {
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(stream, &st) == cudaSuccess) return st == cudaStreamCaptureStatusNone;
    cudaGetLastError();  // (the launch itself reports what is wrong with the stream)
    return false;
}

template <typename... P, typename... A>
cudaError_t launch_overlapped(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                              bool overlap, A &&...args) {
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = overlap ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

enum ForceMode : int { kForceUniform = 0, kForceProfileZ = 1, kForceField = 2 };

struct ForceArgs {
    int mode;
    float fx, fy, fz;        // uniform
    const float *profile;    // 3 x nz
    const float *field;      // 3 x N
    int64_t n;               // N, component stride of `field`
    float scale;             // time factor e^{-gamma t} of the step (1 for a static force)
};

// Default block of the one-node kernels: about 128 threads, of the width
// (a multiple of 32, at most 224) that leaves the fewest idle lanes in a row
// of nx nodes; 128 among equals, else the widest. Against a fixed 128 x 2
// (us a step, FP32): 150 x 91 x 61 with y walls and a force field 25.4 -> 22.5
// (160 x 1; half of 256 lanes were idle), 200 x 180 x 160 with z walls 149 ->
// 139 (224 x 1), D3Q27 at 192 x 176 x 160 192 -> 181 (192 x 1), 256^3 380.6 ->
// 376 (128 x 1: smaller blocks leave less idle while the last one finishes).
inline int default_block_x(int nx) {
    int best = 32;
    int64_t pad = INT64_MAX;
    for (int bx = 32; bx <= 224; bx += 32) {
        const int64_t w = ((int64_t)nx + bx - 1) / bx * bx;
        if (w < pad || (w == pad && best != 128)) {
            pad = w;
            best = bx;
        }
    }
    return best;
}

struct Launch {
    Geom g;
    dim3 block, grid;  // grid of the one-node-per-thread kernels
    cudaStream_t stream;
    bool overlap = true;  // launch_overlapped: not inside a graph capture (stream_overlaps)
    bool pairs = false;   // launch_step, where the staged form does not apply: two adjacent nodes per thread (step_pair.cu)
    bool packed;       // launch_step: two nodes per thread (grid.x halved)
    bool staged;       // launch_step (A/B) and launch_step_aa (16-bit, cascaded): rows staged by bulk copies
                       // where they apply (step_tma.cuh)
    int map;           // state kernels: slots of the post-streaming state (0 A/B pull map,
                       // 1 in-place pattern after even steps, 2 after odd steps, 3 the A/B pull
                       // map of a z-slab with halo faces)
    long long wait_cycles = 0;  // staged step: bound of a wait for a tile's copies (0: kWaitCycles)
    bool drop_first_tile = false;  // staged step, failure injection: tile 0's copies are not issued
    int z0 = 0, zs = 1, nplanes = -1;  // staged and fused-sums steps, init, read-out: the planes z0, z0 + zs, ...
                                       // (nplanes of them; -1: all)
};

// storage: 0 = f32, 1 = f16, 2 = bf16, 3 = f16 stochastic, 4 = bf16 stochastic
// (CLBM_STORAGE_*). key: per-step dither key (stochastic formats).
cudaError_t launch_step(int storage, const Launch &L, const void *src, void *dst, const Rates &r,
                        const ForceArgs &F, int *flag, uint32_t key);
// One cascaded A/B step with two adjacent nodes per thread (step_pair.cu):
// whether a lattice takes it by default, and its launch (the bits of
// launch_step's one-node kernel).
bool step_pairs(const Geom &g);
cudaError_t launch_step_pair(int storage, const Launch &L, const void *src, void *dst, const Rates &r,
                             const ForceArgs &F, int *flag, uint32_t key);
// The in-place FP32 step in node pairs, as launch_step_aa.
cudaError_t launch_step_aa_pair(const Launch &L, void *f, const Rates &r, const ForceArgs &F, int *flag, bool odd);
// Two cascaded FP32 A/B steps of a small lattice in one launch (step_small.cu):
// bricks of bx x by x bz nodes, grown by hx, hy, hz to ext = ex x ey x ez.
struct SmallPlan {
    int bx, by, bz, nbx, nby, nbz, hx, hy, hz;
    int ex, ey, ext, threads;
    int in_graph;  // pays inside a captured graph too
    uint32_t exdiv, exydiv, bxdiv, bxydiv;  // ceil(2^32 / divisor)
};
bool small_plan(const Geom &g, int sms, SmallPlan &p);  // sms: SMs of the device
// F carries the first step's force factor, scale2 is the second step's.
cudaError_t launch_step_small2(const Launch &L, const SmallPlan &p, const void *src, void *dst, const Rates &r,
                               const ForceArgs &F, float scale2, int *flag);
// The cascaded step on a z-slab (Geom::slab halo faces): the planes z0,
// z0 + zs, ... (nplanes of them) from src into dst (step.cu).
cudaError_t launch_step_slab(int storage, const Launch &L, const void *src, void *dst, const Rates &r,
                             const ForceArgs &F, int *flag, uint32_t key, int z0, int zs, int nplanes);
// Whether an A/B step of a q-population lattice from a state buffer at src
// (elem bytes per value) with force F runs the shared-memory staged kernel
// (step_tma.cuh) when the launch asks for it.
bool step_staged(const Geom &g, size_t elem, const void *src, int q, const ForceArgs &F);
// The rounds of tiles of a 16-bit staged step on a device of sms SMs, and the
// nodes that a round of full tiles holds; pairs: a collision in node pairs (the
// cascaded one). False where the geometry is not staged.
bool staged_rounds(const Geom &g, int q, bool pairs, int sms, int &rounds, int64_t &capacity);
// In-place (AA) pattern: one step on the single population array f; odd
// selects the odd step kind (step.cu).
cudaError_t launch_step_aa(int storage, const Launch &L, void *f, const Rates &r, const ForceArgs &F, int *flag,
                           uint32_t key, bool odd);
// The cascaded in-place step with 16-bit storage staged in node pairs, if it
// applies (step_aa.cu); false: nothing launched.
bool launch_step_aa_staged(int storage, const Launch &L, void *f, const Rates &r, const ForceArgs &F, int *flag,
                           uint32_t key, bool odd, cudaError_t &err);
// The comparison collision models (models.cuh): SRT-LBM and non-orthogonal
// MRT, A/B and in-place forms (step_srt.cu, step_mrt.cu).
cudaError_t launch_step_srt(int storage, const Launch &L, const void *src, void *dst, const Rates &r,
                            const ForceArgs &F, int *flag, uint32_t key);
cudaError_t launch_step_mrt(int storage, const Launch &L, const void *src, void *dst, const Rates &r,
                            const ForceArgs &F, int *flag, uint32_t key);
cudaError_t launch_step_aa_srt(int storage, const Launch &L, void *f, const Rates &r, const ForceArgs &F, int *flag,
                               uint32_t key, bool odd);
cudaError_t launch_step_aa_mrt(int storage, const Launch &L, void *f, const Rates &r, const ForceArgs &F, int *flag,
                               uint32_t key, bool odd);
// Fused step + fixed-point conservation sums of the pulled state into the
// kDiagSlots x 4 accumulators acc (zero on entry). If acc_prev is not null,
// the launch first drains that set (the previous step's) into out_prev[0..3]
// (FP64 totals, add0 added to the first) and clears it. launch_drain4 drains a set on its own (step_diag.cu).
// With L.nplanes >= 0 it steps the planes L.z0 .. L.z0 + L.nplanes - 1 only
// (L.zs = 1); the launches of one step's plane ranges add into the same set.
constexpr int kDiagSlots = 1024;
struct DiagSums {
    unsigned long long *acc;
    unsigned long long *acc_prev;
    double *out_prev;
    double add0;
};
cudaError_t launch_step_diag(int storage, const Launch &L, const void *src, void *dst, const Rates &r,
                             const ForceArgs &F, int *flag, const DiagSums &d, uint32_t key);
cudaError_t launch_drain4(unsigned long long *acc, double *out, double add0, cudaStream_t stream);
cudaError_t launch_fixed_final4(const long long *partials, int nblocks, double *out, double add0,
                                cudaStream_t stream);
cudaError_t launch_scatter(int storage, const Launch &L, void *dst, const float *f, int64_t n, int deviation);
cudaError_t launch_init_eq(int storage, const Launch &L, void *dst, const float *rho, const float *u, int64_t n,
                           const ForceArgs &F);
cudaError_t launch_gather(int storage, const Launch &L, const void *src, float *f, int64_t n, int deviation);
cudaError_t launch_macros(int storage, const Launch &L, const void *src, const ForceArgs &F, float *rho, float *u,
                          int64_t n);
cudaError_t launch_reduce_moments(int storage, const Launch &L, const void *src, const ForceArgs &F,
                                  long long *partials, int nblocks, double *out);
cudaError_t launch_adjoint_step(int storage, const Launch &L, const void *state, const float *lam_next, float *lam,
                                float *gF, const Rates &r, const ForceArgs &F, int64_t n);
cudaError_t launch_adjoint_seed(int storage, const Launch &L, const void *state, const float *gu, float *lam,
                                float *gF, const ForceArgs &F, int64_t n);
cudaError_t launch_reduce_pair(const float *a, const float *b, int64_t n, double *partials, int nblocks,
                               double *out, cudaStream_t stream);

// D3Q27 (step27.cu); Rates27 in d3q27.cuh.
struct Rates27;
cudaError_t launch_step27(int storage, const Launch &L, const void *src, void *dst, const Rates27 &r,
                          const ForceArgs &F, int *flag, uint32_t key);
cudaError_t launch_init27(int storage, const Launch &L, void *dst, const float *rho, const float *u, int64_t n,
                          const ForceArgs &F);
cudaError_t launch_scatter27(int storage, const Launch &L, void *dst, const float *f, int64_t n, int deviation);
cudaError_t launch_gather27(int storage, const Launch &L, const void *src, float *f, int64_t n, int deviation);
cudaError_t launch_macros27(int storage, const Launch &L, const void *src, const ForceArgs &F, float *rho, float *u,
                            int64_t n);
cudaError_t launch_step27_aa(int storage, const Launch &L, void *f, const Rates27 &r, const ForceArgs &F, int *flag,
                             uint32_t key, bool odd);
// The comparison models on D3Q27 (models27.cuh; step27_srt.cu, step27_mrt.cu).
cudaError_t launch_step27_srt(int storage, const Launch &L, const void *src, void *dst, const Rates27 &r,
                              const ForceArgs &F, int *flag, uint32_t key);
cudaError_t launch_step27_mrt(int storage, const Launch &L, const void *src, void *dst, const Rates27 &r,
                              const ForceArgs &F, int *flag, uint32_t key);
cudaError_t launch_step27_aa_srt(int storage, const Launch &L, void *f, const Rates27 &r, const ForceArgs &F,
                                 int *flag, uint32_t key, bool odd);
cudaError_t launch_step27_aa_mrt(int storage, const Launch &L, void *f, const Rates27 &r, const ForceArgs &F,
                                 int *flag, uint32_t key, bool odd);
cudaError_t launch_moments27(int storage, const Launch &L, const void *src, const ForceArgs &F, long long *partials,
                             int nblocks, double *out);

// Record `msg` as the calling thread's last error (clbm_last_error) and return code.
int set_error(int code, const char *msg);

// NVTX range for the span of one entry point (shown by profilers that
// record NVTX; a no-op otherwise), in the "clbm" domain.
struct Range {
    explicit Range(const char *name);
    ~Range();
    Range(const Range &) = delete;
    Range &operator=(const Range &) = delete;
};

}  // namespace clbm
