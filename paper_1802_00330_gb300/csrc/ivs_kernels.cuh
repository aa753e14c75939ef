// ivs_kernels.cuh -- kernels of one sweep over the device queue, and their launchers.
//
// One sweep ("wave") pops up to K parent boxes from the top of the queue and runs:
//   k_wave_begin  : chooses K so that the worst case (every child kept) fits
//   k_eval        : a warp (many children, or few parents: a block) per parent; Algorithm 2's split
//                   is implicit: child c takes the upper half of coordinate j when bit j of
//                   c is set; FP32 outward evaluation, or FP64 without the FP32 stage
//                   (Definition 1-2); survivors compacted with warp ballots into a list
//                   per dimension n, undecided children into one for
//   k_eval64      : the FP64 evaluation of those
//   k_screen<N>   : decides in FP32 what the contraction would drop or leave unchanged
//   k_hs<N>       : 32 survivors per block (narrow sweeps: 8 per block,
//   k_hs_narrow<N>  k_hs_narrow): Hansen-Sengupta sweeps (Algorithm 3) or Krawczyk steps
//                   (eq 15-16), then accept (Algorithm 1 (II)) or write the box as a
//                   new parent
//   k_commit      : moves the new parents onto the queue where the popped ones were
#pragma once
#include <cuda_runtime.h>

#include "ivs_internal.h"

namespace ivs {

struct SweepArgs {
    DevTables tb;
    DevQueue q;        // the queue
    DevQueue stage;    // new parents of this sweep
    DevOut out;
    WaveCtl *ctl;
    Surv *surv;        // survivor list of dimension n at surv + n * surv_cap
    int64_t surv_cap;
    Surv *cand;        // FP32 survivors (capacity surv_cap)
    unsigned long long *stats;   // [n_sys][ST_COUNT]
    int64_t wave_children;       // children a sweep may evaluate
    int32_t max_fan_shift;       // max n over the plan's systems
    int32_t n_sys;
    int32_t single;              // 1: one system (closed-form pop, in k_commit after the first sweep)
    int32_t blob_smem;           // bytes of its blob when k_eval caches it in shared memory, else 0
    int32_t head_smem;           // bytes of the blob's head when the other kernels cache it, else 0
    int32_t tv_entries;          // table entries of a block of k_eval (0: no tables)
    int32_t eval_forms;          // bit 0: some system's parents go to warps, bit 1: to blocks;
                                 // bit 2: every parent has few children (a warp also in narrow sweeps)
    int32_t screen;              // 1: some system may be screened in FP32 (ivs_screen.cuh)
    DevRegions rg;               // serving: per-system queue regions (rg.n == 0: shared stack)
};

// dynamic shared memory of k_eval (blob cache + the warps' combination tables) and the
// kernels' limits
size_t eval_smem_bytes(const SweepArgs &a);
cudaError_t configure_eval_kernels(const SweepArgs &a);
// raises a kernel's dynamic shared memory limit to the device maximum (idempotent)
cudaError_t allow_max_dynamic_smem(const void *func);
// k_eval's table region: eight warps' tables where they fit 56 KB (three blocks per SM with
// the blob of an n = 8 system beside them), else one table per block; a table has at most
// 2048 entries.  sys == nullptr: any systems (the server).
constexpr int kTvEntries = 3584;
inline bool eval_uses_table(const DevSys &d) { return d.n_tv > 0 && (d.shadow || !d.prefilter); }
inline void choose_eval_layout(SweepArgs &a, const DevSys *sys, int n_sys) {
    a.tv_entries = sys ? 0 : kTvEntries;
    a.eval_forms = sys ? 0 : 3;
    for (int s = 0; s < n_sys; s++) {
        const DevSys &d = sys[s];
        if (!eval_uses_table(d)) continue;
        const int need = (!d.eval_block && d.n_tv * 8 <= kTvEntries) ? d.n_tv * 8 : d.n_tv;
        if (need > a.tv_entries) a.tv_entries = need;
    }
    bool few = sys != nullptr;
    for (int s = 0; s < n_sys; s++) {
        a.eval_forms |= (sys[s].eval_block || sys[s].n_tv > a.tv_entries / 8) ? 2 : 1;
        few = few && (sys[s].bisect || sys[s].n <= 3) && sys[s].n_tv <= 64 && sys[s].m <= 8;
    }
    if (few && a.eval_forms == 1) a.eval_forms |= 4;
}
// one sweep; ev (nullable) receives n_hs_dims + 5 stage events; *kernels (nullable) the
// number of kernels launched
cudaError_t launch_sweep(const SweepArgs &a, const int *hs_dims, int n_hs_dims, int eval_blocks,
                         int eval_threads, int num_sms, cudaStream_t st, cudaEvent_t *ev, int *kernels = nullptr);
// The sweep loop as one CUDA graph: a conditional WHILE node whose body is one sweep; its
// commit kernel keeps the condition set while the queue is non-empty, no error occurred
// and ctl->waves < ctl->wave_limit.  *kernels_per_sweep: kernels per iteration (plans of one system
// pop in the commit and have no k_wave_begin in it).
cudaError_t build_sweep_graph(const SweepArgs &a, const int *hs_dims, int n_hs_dims, int eval_blocks,
                              int eval_threads, int num_sms, cudaGraph_t *out, int *kernels_per_sweep = nullptr);
// directed-rounding rate microbenchmark (kind 0 FP64, 1 FP32); returns ops and fills ms
cudaError_t run_probe(int kind, int num_sms, double *ops, float *ms);
cudaError_t launch_seed_roots(const SweepArgs &a, const double *d_box_lo, const double *d_box_hi,
                              const int32_t *d_root_depth, int n_sys, int n_max, cudaStream_t st);
// serving with regions: empties the regions of the slots with d_cancel[s] != 0 (between
// sweeps) and lowers the queue total accordingly
cudaError_t launch_cancel_regions(const SweepArgs &a, const int32_t *d_cancel, cudaStream_t st);
// One system's results in a packed buffer: n x count lower ends, n x count upper ends
// (coordinate-major), then count flags and count depths (int32), from `off` (doubles) on.
struct PackDesc {
    int64_t base, count, off;
    int64_t n;
};
// packs the results of n_sys systems, at most `most` of one; desc in device memory, or `one` when n_sys == 1
cudaError_t launch_pack_results(const DevOut &o, const PackDesc *desc, PackDesc one, int n_sys, int64_t most, double *dst,
                                cudaStream_t st);
// appends initial boxes of newly admitted systems (slot ids) on top of the queue, or at
// the start of each system's region
cudaError_t launch_admit(const SweepArgs &a, const double *d_lo, const double *d_hi, const int32_t *d_slot,
                         const int32_t *d_depth, int count, int n_max, cudaStream_t st);
// Hansen-Sengupta + accept/split kernels for dimension n (ivs_hs_*.cu); *kernels receives
// how many kernels the call launched (2, one more with the screen)
cudaError_t launch_hs_dim1(const SweepArgs &a, int num_sms, cudaStream_t st, int *kernels);
cudaError_t launch_hs_dim2(const SweepArgs &a, int num_sms, cudaStream_t st, int *kernels);
cudaError_t launch_hs_dim3(const SweepArgs &a, int num_sms, cudaStream_t st, int *kernels);
cudaError_t launch_hs_dim4(const SweepArgs &a, int num_sms, cudaStream_t st, int *kernels);
cudaError_t launch_hs_dim5(const SweepArgs &a, int num_sms, cudaStream_t st, int *kernels);
cudaError_t launch_hs_dim6(const SweepArgs &a, int num_sms, cudaStream_t st, int *kernels);
cudaError_t launch_hs_dim7(const SweepArgs &a, int num_sms, cudaStream_t st, int *kernels);
cudaError_t launch_hs_dim8(const SweepArgs &a, int num_sms, cudaStream_t st, int *kernels);
cudaError_t launch_hs_dim9(const SweepArgs &a, int num_sms, cudaStream_t st, int *kernels);
cudaError_t launch_hs_dim10(const SweepArgs &a, int num_sms, cudaStream_t st, int *kernels);
cudaError_t launch_hs_dim11(const SweepArgs &a, int num_sms, cudaStream_t st, int *kernels);
cudaError_t launch_hs_dim12(const SweepArgs &a, int num_sms, cudaStream_t st, int *kernels);
cudaError_t launch_hs_dim13(const SweepArgs &a, int num_sms, cudaStream_t st, int *kernels);
cudaError_t launch_hs_dim14(const SweepArgs &a, int num_sms, cudaStream_t st, int *kernels);
cudaError_t launch_hs_dim15(const SweepArgs &a, int num_sms, cudaStream_t st, int *kernels);
cudaError_t launch_hs_dim16(const SweepArgs &a, int num_sms, cudaStream_t st, int *kernels);

}  // namespace ivs
