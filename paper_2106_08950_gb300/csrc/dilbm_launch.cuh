// Launch shapes of the lattice sweep and the launchers that take them.
//
// A shape is numerics-neutral: it only decides how many row segments a block
// keeps in flight (warps per block, one row segment per warp) and how many
// blocks the persistent grid holds per SM.  Every node is swept by the same
// code in the same arithmetic whatever the shape, so the autotuner may pick
// any shape without changing a single result bit.
//
// The launchers are compiled once per storage type, each in its own
// translation unit (dilbm_launch_f32.cu, _f16.cu, _bf16.cu).
#pragma once
#include "dilbm_grid.h"
#include "dilbm_kernels.cuh"

namespace dilbm {

constexpr SweepShape SWEEP_SHAPE{SWEEP_WARPS, 0};  // of the sweep alone until another is set, and of the fields
constexpr SweepShape PS_SHAPE = SWEEP_SHAPE;       // the one shape that a PS-LBM context takes and reports; its
constexpr int PS_WARPS = 4;                        // fused steps run with this many warps per block all the same

// row_of's multiplier: floor(2^32 / ntx) + 1 (unused for ntx == 1).
inline unsigned ntx_inverse(int ntx) {
    return ntx > 1 ? (unsigned)((1ull << 32) / (unsigned long long)ntx) + 1u : 0u;
}

// Blocks of `kern` (W warps, `smem` bytes of dynamic shared memory) resident
// per SM, after opting in to that shared memory; cached per device.
template <typename K>
cudaError_t occupancy_of(K kern, int warps, size_t smem, int *cache, int *per_sm) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 64) return cudaErrorInvalidDevice;
    if (cache[dev] == 0) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        int n = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, warps * 32, smem);
        if (e != cudaSuccess) return e;
        cache[dev] = n > 0 ? n : 1;
    }
    *per_sm = cache[dev];
    return cudaSuccess;
}

// Several steps: the blocks wait for one another (particle blocks for the
// sweeping ones, and all of them between steps), so the launch is cooperative:
// the driver starts it only with every block resident.  One step (`alone`):
// particle blocks wait for the sweeping ones, which are then first in the grid
// and wait for no block, so an ordinary launch makes progress on whatever SMs
// are free.  (us per call of one step, cooperative and ordinary: 512^2 FP32 14.6
// both, 1024^2 FP16 28.9 and 26.9, 200 small lattices 77.2 and 74.4; PS-LBM on
// 512^2 20.9 and 22.6, so PS steps stay cooperative.)
inline cudaError_t launch_steps(const void *kern, void **args, StepRun *run, const FusedGrid &g, bool alone, int warps,
                                size_t smem, cudaStream_t st) {
    const dim3 blocks((unsigned)g.blocks), threads(warps * 32);
    run->pblocks = g.pblocks;
    run->ahead = alone ? 0 : g.pblocks;
    return alone ? cudaLaunchKernel(kern, blocks, threads, args, smem, st)
                 : cudaLaunchCooperativeKernel(kern, blocks, threads, args, smem, st);
}

template <typename T, bool EDGES, int W, bool PS, bool HALVES = false>
cudaError_t step_variant(const SweepArgs<T> &a, const PartArgs &pa, StepRun run, const SweepShape &sh, int num_sms,
                         cudaStream_t st, int *per_sm_out) {
    static int cache[64] = {};
    constexpr size_t smem = sweep_smem_bytes<T, W>();
    auto *kern = step_kernel<T, EDGES, W, PS, HALVES>;
    int per_sm = 1;
    cudaError_t e = occupancy_of(kern, W, smem, cache, &per_sm);
    if (e != cudaSuccess || per_sm_out) {
        if (per_sm_out) *per_sm_out = per_sm;
        return e;
    }
    const long long items = (long long)a.L.ny * a.L.ntx;
    if constexpr (W == 4 && !PS && !HALVES) {
        // two warps to a segment, where every warp still has at most one (in
        // the default shape)
        static int halves_cache[64] = {};
        int fit = 1;
        e = occupancy_of(step_kernel<T, EDGES, W, PS, true>, W, smem, halves_cache, &fit);
        if (e != cudaSuccess) return e;
        if (one_item_per_warp(2 * items, a.np, W, fit, num_sms, sh))
            return step_variant<T, EDGES, W, PS, true>(a, pa, run, sh, num_sms, st, per_sm_out);
    }
    const FusedGrid g = fused_grid(HALVES ? 2 * items : items, a.np, W, per_sm, num_sms, sh);
    void *p[3] = {const_cast<SweepArgs<T> *>(&a), const_cast<PartArgs *>(&pa), &run};
    return launch_steps((const void *)kern, p, &run, g, run.nsteps == 1 && !PS, W, smem, st);
}

template <typename T, int W>
cudaError_t batch_variant(const BatchArgs<T> &ba, StepRun run, const SweepShape &sh, int num_sms, cudaStream_t st,
                          int *per_sm_out) {
    static int cache[64] = {};
    constexpr size_t smem = sweep_smem_bytes<T, W>();
    auto *kern = step_batch_kernel<T, W>;
    int per_sm = 1;
    cudaError_t e = occupancy_of(kern, W, smem, cache, &per_sm);
    if (e != cudaSuccess || per_sm_out) {
        if (per_sm_out) *per_sm_out = per_sm;
        return e;
    }
    const FusedGrid g = fused_grid(ba.item_start[ba.n], ba.part_start[ba.n], W, per_sm, num_sms, sh);
    void *p[2] = {const_cast<BatchArgs<T> *>(&ba), &run};
    return launch_steps((const void *)kern, p, &run, g, run.nsteps == 1, W, smem, st);
}

// The sweep without the particle update (a step of a strip or of a small lattice
// without particles, in its shape; MODE_FIELDS: the macroscopic fields instead
// of a step).  `chained`: the launch before it on the stream is such a step too,
// and this one may come before its end (it waits for it: a microsecond less
// between steps).
template <typename T, int MODE, bool EDGES, bool PS, int W = SWEEP_WARPS>
cudaError_t sweep_variant(const SweepArgs<T> &a, const FieldsOut &fo, int num_sms, cudaStream_t st,
                          const SweepShape &sh = SWEEP_SHAPE, bool chained = false, int *per_sm_out = nullptr) {
    static int cache[64] = {};
    constexpr size_t smem = sweep_smem_bytes<T, W>();
    int per_sm = 1;
    cudaError_t e = occupancy_of(sweep_kernel<T, MODE, EDGES, PS, W>, W, smem, cache, &per_sm);
    if (e != cudaSuccess || per_sm_out) {
        if (per_sm_out) *per_sm_out = per_sm;
        return e;
    }
    const long long blocks = persistent_grid((long long)a.L.ny * a.L.ntx, W, per_sm, num_sms, sh);
    cudaLaunchAttribute early{};
    early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    early.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(W * 32);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &early;
    cfg.numAttrs = chained ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, sweep_kernel<T, MODE, EDGES, PS, W>, a, fo);
}

// Per-storage launchers, instantiated in dilbm_launch_f32.cu, _f16.cu and
// _bf16.cu.  per_sm != NULL: launch nothing, return the kernel's resident
// blocks per SM there.
template <typename T>
struct Launch {
    // fused steps of one lattice (PS-LBM: in the default shape)
    static cudaError_t steps(const SweepArgs<T> &a, const PartArgs &pa, const StepRun &run, bool edges, bool ps, const SweepShape &sh,
                             int num_sms, cudaStream_t st, int *per_sm = nullptr);
    // fused steps of a batch
    static cudaError_t batch(const BatchArgs<T> &ba, const StepRun &run, const SweepShape &sh, int num_sms,
                             cudaStream_t st, int *per_sm = nullptr);
    // a sweep alone (PS-LBM: in the default shape)
    static cudaError_t sweep(const SweepArgs<T> &a, bool edges, bool ps, const SweepShape &sh, int num_sms,
                             cudaStream_t st, bool chained = false, int *per_sm = nullptr);
    static cudaError_t fields(const SweepArgs<T> &a, const FieldsOut &fo, bool edges, bool ps, int num_sms,
                              cudaStream_t st);
};

}  // namespace dilbm
