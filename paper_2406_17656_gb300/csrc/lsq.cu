// lsq.cu -- the batched column least-squares solves of SAM construction
// (arXiv 2406.17656, Sec. 2), FP32 register tiles with FP64 refinement, the
// dispatch over the size classes, and the refinement guard's FP64 re-solve
// and outcome counts.  The kernel is described in lsq_kernel.cuh.
#include "lsq_kernel.cuh"

namespace sam {

cudaError_t launch_lsq_bin(sam_handle h, int precision, const LsqArgs &args, int bin) {
    if (bin == kBinBig && precision == SAM_FP32_REFINE && args.refine_steps != 0)
        return launch_lsq_dense(h, args, bin);
    if (bin == kBinBig) return launch_lsq_big(h, args, bin, true, precision == SAM_FP32_REFINE);
    if (precision == SAM_FP64) return launch_lsq_fp64_bin(h, args, bin);
    if (bin < kSimtBins && args.kev) {
        const cudaError_t e = launch_lsq_simt_bin(h, args, bin);
        if (e != cudaSuccess || !args.longest) return e;
        LsqArgs t = args;
        t.kev = nullptr;
        t.tile_gate = args.longest;
        return launch_lsq_bin(h, precision, t, bin);
    }
    // FP32 tiles: the shape of each size class comes from the handle (sam_tune)
    const bool b = handle_variant(h, bin) != 0;
    switch (bin) {
        case 0: return launch_one<F0, false>(h, args, 0);
        case 1: return b ? launch_one<F1b, false>(h, args, 1) : launch_one<F1, false>(h, args, 1);
        case 2: return b ? launch_one<F2b, false>(h, args, 2) : launch_one<F2, false>(h, args, 2);
        case 3: return b ? launch_one<F3b, false>(h, args, 3) : launch_one<F3, false>(h, args, 3);
        default: return b ? launch_one<F4b, false>(h, args, 4) : launch_one<F4, false>(h, args, 4);
    }
}

cudaError_t launch_lsq(sam_handle h, int precision, const LsqArgs &args) {
    for (int b = 0; b < kNumBins; ++b) {
        cudaError_t e = launch_lsq_bin(h, precision, args, b);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

namespace {
// the columns flagged for the FP64 re-solve, in any order: those of the large
// class into big, the others into list; off[1] and off[3] receive their
// numbers (off[0] = off[2] = 0: the lists as work-list ranges);
// counts (nullable): the columns that took s = 1..kAutoSteps steps, and the
// FP64 re-solves (per-thread counts, one shared atomic per warp)
__global__ void __launch_bounds__(256) flag_list_kernel(int N, const int32_t *colstat, const uint8_t *used,
                                                        const uint8_t *bin, int32_t *list, int32_t *big, int32_t *off,
                                                        unsigned long long *counts) {
    __shared__ unsigned sh[kAutoSteps + 1];
    if (threadIdx.x <= kAutoSteps) sh[threadIdx.x] = 0u;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    unsigned c[kAutoSteps + 1] = {};
    for (int64_t j0 = (int64_t)blockIdx.x * 256; j0 < N; j0 += (int64_t)gridDim.x * 256) {
        const int64_t j = j0 + threadIdx.x;
        const bool f = j < N && colstat[j] == kStRefine;
        const int u = counts && j < N ? used[j] : 0;
#pragma unroll
        for (int v = 0; v <= kAutoSteps; ++v) c[v] += (u == v + 1) ? 1u : 0u;
        if (!__any_sync(0xffffffffu, f)) continue;
        const bool large = f && bin[j] >= kBinBig;
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            const bool mine = f && large == (t == 1);
            const unsigned m = __ballot_sync(0xffffffffu, mine);
            if (!m) continue;
            const int leader = __ffs(m) - 1;
            int base = 0;
            if (lane == leader) base = atomicAdd(&off[2 * t + 1], __popc(m));
            base = __shfl_sync(0xffffffffu, base, leader);
            if (mine) (t ? big : list)[base + __popc(m & ((1u << lane) - 1u))] = (int)j;
        }
    }
    if (!counts) return;
#pragma unroll
    for (int v = 0; v <= kAutoSteps; ++v) {
        const unsigned t = __reduce_add_sync(0xffffffffu, c[v]);
        if (lane == 0 && t) atomicAdd(&sh[v], t);
    }
    __syncthreads();
    if (threadIdx.x <= kAutoSteps && sh[threadIdx.x]) atomicAdd(&counts[threadIdx.x], (unsigned long long)sh[threadIdx.x]);
}
}  // namespace

cudaError_t launch_refine_fallback(sam_handle h, const LsqArgs &args, int N, int32_t *list, int32_t *list_off,
                                   int64_t *counts, const RedoLists &redo) {
    cudaStream_t st = handle_stream(h);
    cudaError_t e;
    if (!redo.bin || !args.dense_list) return cudaErrorInvalidValue;
    if (args.refine_steps < 0) {
        // automatic refinement: the columns whose first step asked for a
        // second, solved again from the start with two steps, by their size
        // classes' kernels (the guard after the second step sends a miss to
        // the FP64 re-solve below)
        if (!redo.bins2 || !redo.work || !redo.bin_off || !redo.ws) return cudaErrorInvalidValue;
        if ((e = flagged_bins(h, N, redo.bin, args.colstat, kStStep2, redo.bins2)) != cudaSuccess ||
            (e = build_work_list(h, N, redo.bins2, redo.work, redo.bin_off, redo.ws)) != cudaSuccess)
            return e;
        LsqArgs a2 = args;
        a2.work = redo.work;
        a2.bin_off = redo.bin_off;
        a2.item_lo = a2.item_hi = 0;
        a2.refine_steps = kAutoSteps;
        // (the large class never flags a column: its kernel takes its own steps)
        for (int b = 0; b < kBinBig; ++b)
            if ((e = launch_lsq_bin(h, SAM_FP32_REFINE, a2, b)) != cudaSuccess) return e;
    }
    // (list_off is zero: cleared with the batch's other counters)
    if (counts && (e = cudaMemsetAsync(counts, 0, sizeof(int64_t) * (kAutoSteps + 1), st)) != cudaSuccess) return e;
    if (N > 0) {
        int blocks = (N + 255) / 256;
        if (blocks > handle_sms(h) * 8) blocks = handle_sms(h) * 8;
        flag_list_kernel<<<blocks, 256, 0, st>>>(N, args.colstat, args.refine_used, redo.bin, list, args.dense_list,
                                                 list_off,
                                                 reinterpret_cast<unsigned long long *>(counts));
        count_launch(h);
    }
    // the flagged columns in FP64, by the large class's kernel; those of the
    // classes 0-4 in two blocks per SM instead of one, since their tiles are
    // small (results do not depend on the lists' order).  A warp per column
    // through class 4's register tile was faster for thousands of columns but
    // slower by 35 us for a few, and a rule on their number would make a
    // column's bits depend on the others.
    LsqArgs a = args;
    a.work = list;
    a.bin_off = list_off;
    a.item_lo = a.item_hi = 0;
    if ((e = launch_lsq_small_fp64(h, a)) != cudaSuccess) return e;
    a.work = args.dense_list;
    a.bin_off = list_off + 2;
    if ((e = launch_lsq_big(h, a, 0, false)) != cudaSuccess) return e;
    return cudaGetLastError();
}

}  // namespace sam
