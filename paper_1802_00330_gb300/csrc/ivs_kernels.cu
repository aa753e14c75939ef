// ivs_kernels.cu -- the per-box sweep over the device queue (sm_103a): control,
// evaluation stages, and the sweep loop as one CUDA graph.
//
// Paper map: Definition 1-2 and Algorithm 2 (evaluation and exclusion of the 2^n children
// of each parent); Algorithm 1 (the loop M_k -> M_{k+1} until the queue is empty).  The
// Hansen-Sengupta stage and the accept / split step are in ivs_hs.cuh.  Every operation
// sequence matches the serial definition step for step (same fold orders, same
// roundings), so the sorted result set is identical to the serial solver's.
#include <cuda_runtime.h>

#include "ivs_internal.h"
#include "ivs_interval.cuh"
#include "ivs_kernels.cuh"
#include "ivs_tab.cuh"

namespace ivs {

constexpr unsigned kFull = 0xFFFFFFFFu;
constexpr int kEvalThreads = 256;
constexpr int kEvalWarps = kEvalThreads / 32;
constexpr int kEval64Threads = 128;

__device__ __forceinline__ unsigned lane_id() { return threadIdx.x & 31u; }
__device__ __forceinline__ unsigned lanemask_lt() { return (1u << lane_id()) - 1u; }

__device__ __forceinline__ unsigned long long *stat_ptr(const SweepArgs &a, int sys, int slot) {
    return a.stats + (size_t)sys * ST_COUNT + slot;
}

// ------------------------------------------------------------------------------------
// sweep control
// ------------------------------------------------------------------------------------

// Pops K parents from the top of the queue, as many as fit: the K popped parents'
// children (2^n each, 1 for an initial box) must fit the sweep's budget W, and in the
// worst case (every child kept and split again) the queue must hold them:
// top - K + children <= cap.  One block scans the fan-outs of the top entries.
constexpr int kBeginThreads = 1024;
constexpr int kBeginPer = 64;       // entries per thread: a window of 65536 parents
constexpr size_t kBeginSmem = (size_t)kBeginThreads * kBeginPer;   // one byte per window entry
// Serving with per-system regions, one block.  Least attained service first (the
// default): the regions with entries are taken in order of the boxes their request has
// processed so far (fewest first; a bitonic sort of up to kLasMax slots in shared memory),
// and each pops as many parents as its region allows until the sweep's W children are
// used up -- requests that need little work finish in few sweeps, whatever else is in
// flight.  Fair share (rg.fair_share, or more than kLasMax slots): every region gets W
// divided by the regions with entries (at least one parent), in an order that rotates
// with the sweep count.  Either way a region pops breadth first while under half full
// and one parent at a time beyond; the schedule never changes a result.
constexpr int kLasMax = 4096;
__device__ __forceinline__ void reset_lists(WaveCtl *c) {
    for (int n = 0; n <= kMaxVars; n++) {
        c->surv_count[n] = 0;
        c->hs_cursor[n] = 0;
        c->screen_cursor[n] = 0;
        c->open_count[n] = 0;
    }
}
__device__ void wave_begin_regions(const SweepArgs &a, unsigned long long *s_key) {
    __shared__ long long s_red[kBeginThreads];
    __shared__ long long s_active, s_total, s_run;
    const DevRegions &rg = a.rg;
    WaveCtl *c = a.ctl;
    const int t = threadIdx.x, S = rg.n;
    const int64_t waves = c->waves;
    if (t == 0) { s_active = 0; s_total = 0; s_run = 0; }
    __syncthreads();
    // entries each region holds after the last sweep
    long long act = 0, tot = 0;
    for (int sl = t; sl < S; sl += kBeginThreads) {
        const int64_t held = rg.rem[sl] + (int64_t)rg.cursor[sl];
        rg.rem[sl] = held;
        rg.cursor[sl] = 0;
        act += held > 0 ? 1 : 0;
        tot += held;
    }
    atomicAdd((unsigned long long *)&s_active, (unsigned long long)act);
    atomicAdd((unsigned long long *)&s_total, (unsigned long long)tot);
    __syncthreads();
    const bool las = !rg.fair_share && S <= kLasMax;
    const long long share = las ? a.wave_children : a.wave_children / (s_active > 0 ? s_active : 1);
    if (las) {
        // keys (boxes processed, slot), slots without entries last; sorted ascending
        int n2 = 1;
        while (n2 < S) n2 <<= 1;
        for (int q = t; q < n2; q += kBeginThreads) {
            unsigned long long key = ~0ull;
            if (q < S) {
                const unsigned long long done = a.stats[(size_t)q * ST_COUNT + ST_BOXES];
                const unsigned long long cap = 1ull << 40;
                key = ((rg.rem[q] > 0 ? (done < cap ? done : cap) : 2 * cap) << 13) | (unsigned long long)q;
            }
            s_key[q] = key;
        }
        __syncthreads();
        for (int kk = 2; kk <= n2; kk <<= 1)
            for (int j = kk >> 1; j > 0; j >>= 1) {
                for (int q = t; q < n2; q += kBeginThreads) {
                    const int l = q ^ j;
                    if (l > q) {
                        const unsigned long long x = s_key[q], y = s_key[l];
                        if (((q & kk) == 0) ? (y < x) : (x < y)) {
                            s_key[q] = y;
                            s_key[l] = x;
                        }
                    }
                }
                __syncthreads();
            }
    }
    // position q serves slot order[q] (least served first) or (q + waves) % S (rotating);
    // chunks of kBeginThreads positions are scanned in order with a running total of children
    for (int q0 = 0; q0 < S; q0 += kBeginThreads) {
        const int q = q0 + t;
        long long want = 0, fan = 1, k = 0;
        int sl = -1;
        if (q < S) {
            sl = las ? (int)(s_key[q] & 8191ull) : (int)(((int64_t)q + waves) % S);
            const int64_t held = rg.rem[sl];
            if (held > 0) {
                const bool root = held == 1 && (a.q.meta[rg.base[sl]] & kRootFlag) != 0;
                fan = fan_out(a.tb.sys[sl], root ? kRootFlag : 0u);
                k = share / fan;
                if (k < 1) k = 1;
                if (k > held) k = held;
                if (fan > 1) {
                    // breadth while the region is less than half full, one parent at a time
                    // (depth first) beyond: a region of R entries then still holds about
                    // R / (2 fan) more levels of the depth-first walk
                    const long long breadth = (rg.cap[sl] / 2 - held) / (fan - 1);
                    if (k > breadth) k = breadth > 1 ? breadth : 1;
                    if (held + k * (fan - 1) > rg.cap[sl]) k = 0;   // even one parent may not fit
                }
                want = k * fan;
            }
        }
        // inclusive scan of the children wanted (Hillis-Steele over the block)
        s_red[t] = want;
        __syncthreads();
        for (int off = 1; off < kBeginThreads; off <<= 1) {
            const long long v = t >= off ? s_red[t - off] : 0;
            __syncthreads();
            s_red[t] += v;
            __syncthreads();
        }
        const long long before = s_run + s_red[t] - want;
        if (sl >= 0) {
            long long give = k;
            if (before + want > a.wave_children) {
                const long long left = a.wave_children - before;
                give = left > 0 ? left / fan : 0;
            }
            rg.prefix[sl] = give;   // parents popped; turned into a prefix below
            if (rg.rem[sl] > 0 && give == 0 && s_active == 1) c->error = 1;   // cannot progress
        }
        __syncthreads();
        if (t == kBeginThreads - 1) s_run += s_red[t];
        __syncthreads();
    }
    // prefix over slots in slot order; rem = entries left below the popped parents
    if (t == 0) {
        long long run = 0, kids = 0;
        for (int sl = 0; sl < S; sl++) {
            const long long k = rg.prefix[sl];
            rg.prefix[sl] = run;
            run += k;
            const bool root = rg.rem[sl] == 1 && (a.q.meta[rg.base[sl]] & kRootFlag) != 0;
            kids += k * fan_out(a.tb.sys[sl], root ? kRootFlag : 0u);
            rg.rem[sl] -= k;
        }
        rg.prefix[S] = run;
        if (run == 0 && s_total > 0) c->error = 1;
        c->top = s_total;
        c->base = s_total - run;
        c->k = run;
        c->children = kids;
        c->cursor = 0;
        c->staged = 0;
        reset_lists(c);
        c->cand_count = 0;
        c->cand_cursor = 0;
        c->waves += 1;
    }
}

// queue index of the sweep's parent p
__device__ __forceinline__ int64_t parent_index(const SweepArgs &a, int64_t base, int64_t p) {
    if (a.rg.n == 0) return base + p;
    int lo = 0, hi = a.rg.n;   // the slot s with prefix[s] <= p < prefix[s + 1]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (a.rg.prefix[mid] <= p) lo = mid;
        else hi = mid;
    }
    return a.rg.base[lo] + a.rg.rem[lo] + (p - a.rg.prefix[lo]);
}

// One system: every entry has the fan-out F = 2^n (2 when bisected) except the initial box
// (fan-out 1, alone in the queue when popped), so the pop is a closed form.
__device__ __forceinline__ void begin_single(const SweepArgs &a, WaveCtl *c, int64_t top, bool root) {
    int64_t k = 0, children = 0;
    if (top > 0) {
        if (root) {
            k = 1;
            children = 1;
        } else {
            const int64_t F = fan_out(a.tb.sys[0], 0u);
            k = a.wave_children / F;
            const int64_t by_room = (a.q.cap - top) / (F - 1);
            k = k < by_room ? k : by_room;
            k = k < top ? k : top;
            children = k * F;
        }
    }
    if (k <= 0 && top > 0) c->error = 1;
    c->base = top - k;
    c->k = k;
    c->children = children;
    c->cursor = 0;
    c->staged = 0;
    reset_lists(c);
    c->cand_count = 0;
    c->cand_cursor = 0;
    c->waves += 1;
}

__global__ void __launch_bounds__(kBeginThreads) k_wave_begin(SweepArgs a) {
    // log2 children of the window's entries; serving: the sort keys of the slots
    extern __shared__ __align__(8) unsigned char s_fan[];
    __shared__ long long s_sum[kBeginThreads];
    __shared__ long long s_first;
    if (a.rg.n > 0) {
        wave_begin_regions(a, reinterpret_cast<unsigned long long *>(s_fan));
        return;
    }
    WaveCtl *c = a.ctl;
    const int64_t top = c->top;
    const int t = threadIdx.x;
    if (a.single) {
        if (t == 0) begin_single(a, c, top, top > 0 && (a.q.meta[top - 1] & kRootFlag) != 0);
        return;
    }
    const int64_t window = top < (int64_t)kBeginThreads * kBeginPer ? top : (int64_t)kBeginThreads * kBeginPer;
    // entry i (0-based from the top) is queue index top - 1 - i; its log2 children come
    // from its meta word (0 for an initial box), read once with coalesced loads
    for (int q = 0; q < kBeginPer; q++) {
        const int64_t i = (int64_t)q * kBeginThreads + t;
        if (i < window) {
            const uint32_t m = a.q.meta[top - 1 - i];
            s_fan[i] = (m & kRootFlag) ? 0 : (unsigned char)((m >> kFanShift) & kFanMask);
        }
    }
    __syncthreads();
    auto fan_of = [&](int64_t i) -> long long { return 1ll << s_fan[i]; };
    long long local = 0;
    for (int q = 0; q < kBeginPer; q++) {
        const int64_t i = (int64_t)t * kBeginPer + q;
        if (i < window) local += fan_of(i);
    }
    // inclusive scan of the per-thread sums (Hillis-Steele over the block)
    s_sum[t] = local;
    if (t == 0) s_first = window;
    __syncthreads();
    for (int off = 1; off < kBeginThreads; off <<= 1) {
        const long long v = t >= off ? s_sum[t - off] : 0;
        __syncthreads();
        s_sum[t] += v;
        __syncthreads();
    }
    long long pre = s_sum[t] - local;   // children of the entries before this thread's
    const long long room = a.q.cap - top;
    for (int q = 0; q < kBeginPer; q++) {
        const int64_t i = (int64_t)t * kBeginPer + q;
        if (i >= window) break;
        pre += fan_of(i);
        if (pre > a.wave_children || pre - (i + 1) > room) {
            atomicMin(&s_first, (long long)i);
            break;
        }
    }
    __syncthreads();
    if (t != 0) return;
    const int64_t k = s_first;
    int64_t children = 0;
    if (k > 0) {
        // children of the first k entries: recompute from the scan
        const int tk = (int)((k - 1) / kBeginPer), qk = (int)((k - 1) % kBeginPer);
        long long pre2 = tk > 0 ? s_sum[tk - 1] : 0;
        for (int q = 0; q <= qk; q++) pre2 += fan_of((int64_t)tk * kBeginPer + q);
        children = pre2;
    }
    if (k <= 0 && top > 0) c->error = 1;
    c->base = top - k;
    c->k = k;
    c->children = children;
    c->cursor = 0;
    c->staged = 0;
    reset_lists(c);
    c->cand_count = 0;
    c->cand_cursor = 0;
    c->waves += 1;
}

// Moves the sweep's new parents onto the queue.  In the sweep graph (use_cond) it also sets
// the WHILE condition: more sweeps while the queue is non-empty after this commit, no error
// occurred and the sweep limit is not reached (nothing after the commit changes any of
// them).  use_cond 2 (plans of one system): when there are more, the last block that has
// read this sweep's bounds also pops the next sweep's parents, a closed form that reads no
// queue entry, so the sweep needs no k_wave_begin of its own (n = 5 bisection, 35 sweeps: 2217 ->
// 2173 us; n = 6 plan: 1081 -> 1070).
__global__ void k_commit(SweepArgs a, int n_max, cudaGraphConditionalHandle h, int use_cond) {
    WaveCtl *c = a.ctl;
    const int64_t staged = c->staged, base = c->base;
    if (use_cond == 2) {
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            if (atomicAdd(&c->ticket, 1) == (int)gridDim.x - 1) {
                __threadfence();
                const int64_t top = base + staged;
                const bool more = top > 0 && c->error == 0 && c->waves < c->wave_limit;
                c->ticket = 0;
                c->top = top;
                if (more) begin_single(a, c, top, false);
                cudaGraphSetConditional(h, more ? 1u : 0u);
            }
        }
    } else if (use_cond && blockIdx.x == 0 && threadIdx.x == 0) {
        const bool more = base + staged > 0 && c->error == 0 && c->waves < c->wave_limit;
        cudaGraphSetConditional(h, more ? 1u : 0u);
    }
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < staged; i += stride) {
        int64_t d = base + i;
        if (a.rg.n > 0) {   // into the parent's own region, above what stays there
            const int sl = a.stage.sys[i];
            d = a.rg.base[sl] + a.rg.rem[sl] + (int64_t)atomicAdd(&a.rg.cursor[sl], 1ull);
        }
        for (int j = 0; j < n_max; j++) {
            a.q.lo[j * a.q.cap + d] = a.stage.lo[j * a.stage.cap + i];
            a.q.mid[j * a.q.cap + d] = a.stage.mid[j * a.stage.cap + i];
            a.q.hi[j * a.q.cap + d] = a.stage.hi[j * a.stage.cap + i];
        }
        a.q.sys[d] = a.stage.sys[i];
        a.q.meta[d] = a.stage.meta[i];
    }
    if (use_cond != 2 && blockIdx.x == 0 && threadIdx.x == 0) c->top = base + staged;
}

__global__ void k_seed_roots(SweepArgs a, const double *box_lo, const double *box_hi,
                             const int32_t *root_depth, int n_sys, int n_max) {
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < n_sys; s += gridDim.x * blockDim.x) {
        for (int j = 0; j < n_max; j++) {
            a.q.lo[j * a.q.cap + s] = box_lo[(size_t)s * n_max + j];
            a.q.mid[j * a.q.cap + s] = box_hi[(size_t)s * n_max + j];   // a root's only
            a.q.hi[j * a.q.cap + s] = box_hi[(size_t)s * n_max + j];    // child is itself
        }
        a.q.sys[s] = s;
        a.q.meta[s] = kRootFlag | ((uint32_t)root_depth[s] & kDepthMask);
        a.stats[(size_t)s * ST_COUNT + ST_LIVE] = 1;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        WaveCtl *c = a.ctl;
        c->top = n_sys;
        c->base = 0;
        c->k = 0;
        c->staged = 0;
        c->out_count = 0;
        c->cursor = 0;
        c->error = 0;
        c->ticket = 0;
        c->waves = 0;
        c->cand_count = 0;
        c->cand_cursor = 0;
        c->wave_limit = 0x7FFFFFFFFFFFFFFFLL;
        reset_lists(c);
    }
}

// Serving: appends `count` initial boxes (one per newly admitted system) on top of the
// queue between sweeps; one block.
__global__ void k_admit(SweepArgs a, const double *box_lo, const double *box_hi, const int32_t *slot,
                        const int32_t *root_depth, int count, int n_max) {
    const int64_t top = a.ctl->top;
    for (int i = threadIdx.x; i < count; i += blockDim.x) {
        int64_t e = top + i;
        if (a.rg.n > 0) {   // the start of the system's own region
            const int sl = slot[i];
            e = a.rg.base[sl];
            a.rg.rem[sl] = 1;
            a.rg.cursor[sl] = 0;
        }
        for (int j = 0; j < n_max; j++) {
            a.q.lo[j * a.q.cap + e] = box_lo[(size_t)i * n_max + j];
            a.q.mid[j * a.q.cap + e] = box_hi[(size_t)i * n_max + j];
            a.q.hi[j * a.q.cap + e] = box_hi[(size_t)i * n_max + j];
        }
        a.q.sys[e] = slot[i];
        a.q.meta[e] = kRootFlag | ((uint32_t)root_depth[i] & kDepthMask);
        a.stats[(size_t)slot[i] * ST_COUNT + ST_LIVE] = 1;
    }
    __syncthreads();
    if (threadIdx.x == 0) a.ctl->top = top + count;
}

// Serving with regions: a cancelled slot's region is emptied (its entries leave the total).
__global__ void k_cancel_regions(SweepArgs a, const int32_t *cancel) {
    for (int sl = threadIdx.x; sl < a.rg.n; sl += blockDim.x) {
        if (!cancel[sl]) continue;
        const int64_t held = a.rg.rem[sl] + (int64_t)a.rg.cursor[sl];
        if (held) atomicAdd((unsigned long long *)&a.ctl->top, (unsigned long long)(-held));
        a.rg.rem[sl] = 0;
        a.rg.cursor[sl] = 0;
    }
}

// ------------------------------------------------------------------------------------
// evaluation of the children of each parent
// ------------------------------------------------------------------------------------

// Child c of the warp's parent: coordinate j is [lo_j, mid_j] when bit j of c is clear,
// [mid_j, hi_j] when set.  p[0|1|2][j] = lo / mid / hi in FP64; f[0..3][j] = rd32(lo),
// rd32(mid), ru32(mid), ru32(hi); e[0..5][j] = rd32 / ru32 of lo, mid, hi.
struct ChildCoord64 {
    const double (*p)[kMaxVars];
    unsigned c;
    __device__ __forceinline__ ivd operator()(unsigned j) const {
        const unsigned up = (c >> j) & 1u;
        return ivd{p[up][j], p[up + 1][j]};
    }
};
struct ChildCoord32 {
    const float (*f)[kMaxVars];
    unsigned c;
    __device__ __forceinline__ ivf operator()(unsigned j) const {
        const unsigned up = (c >> j) & 1u;
        return ivf{f[up][j], f[up + 2][j]};
    }
};
struct ChildCoordShadow {
    const float (*e)[kMaxVars];
    unsigned c;
    __device__ __forceinline__ shv operator()(unsigned j) const {
        const unsigned up = (c >> j) & 1u;
        return shv{e[2 * up][j], e[2 * up + 1][j], e[2 * up + 2][j], e[2 * up + 3][j]};
    }
};
// box held in shared memory, structure of arrays with the given stride
struct BoxCoord {
    const double *X;
    int stride;
    __device__ __forceinline__ ivd operator()(unsigned j) const {
        return ivd{X[(2 * j) * stride], X[(2 * j + 1) * stride]};
    }
};

__device__ __forceinline__ void push_surv(const SweepArgs &a, WaveCtl *ctl, int n, bool keep, Surv sv) {
    const unsigned km = __ballot_sync(kFull, keep);
    if (!km) return;
    unsigned long long pos = 0;
    if (lane_id() == 0) pos = atomicAdd((unsigned long long *)&ctl->surv_count[n], (unsigned long long)__popc(km));
    pos = __shfl_sync(kFull, pos, 0);
    if (keep) {
        const unsigned long long k = pos + __popc(km & lanemask_lt());
        if ((long long)k < a.surv_cap) a.surv[(size_t)n * a.surv_cap + k] = sv;
        else ctl->error = 1;
    }
}

// undecided children for k_eval64 (warp-aggregated append)
__device__ __forceinline__ void push_cand(const SweepArgs &a, WaveCtl *ctl, bool cand, Surv sv) {
    const unsigned cm = __ballot_sync(kFull, cand);
    if (!cm) return;
    unsigned long long pos = 0;
    if (lane_id() == 0) pos = atomicAdd((unsigned long long *)&ctl->cand_count, (unsigned long long)__popc(cm));
    pos = __shfl_sync(kFull, pos, 0);
    if (cand) {
        const unsigned long long k = pos + __popc(cm & lanemask_lt());
        if ((long long)k < a.surv_cap) a.cand[k] = sv;
        else ctl->error = 1;
    }
}

// ---- decisions from a parent's table -------------------------------------------------------
// A term's value over a child depends only on the child's halves in the term's variables,
// so a parent's children share a table of the terms' values (ivs_tab.cuh): FP32 shadows, or
// FP64 intervals when the system has no FP32 stage.  Both take 16 bytes an entry and hold
// exactly what the per-child evaluation computes for the term.

// states of a child: bit 0 some equation excludes 0, bit 1 some equation is open (shadow)
enum : unsigned { CH_OUT = 1u, CH_OPEN = 2u };

// coordinate of factor f of a table entry: bit f of q is the half (the split coordinate's
// half alone for a bisected parent, whose other coordinates are not split)
struct ComboCoordShadow {
    const float (*e)[kMaxVars];
    unsigned q;
    int only;
    __device__ __forceinline__ shv operator()(unsigned j, int f) const {
        const unsigned up = only < 0 ? (q >> f) & 1u : (j == (unsigned)only ? q : 0u);
        return shv{e[2 * up][j], e[2 * up + 1][j], e[2 * up + 2][j], e[2 * up + 3][j]};
    }
};
struct ComboCoord64 {
    const double (*p)[kMaxVars];
    unsigned q;
    int only;
    __device__ __forceinline__ ivd operator()(unsigned j, int f) const {
        const unsigned up = only < 0 ? (q >> f) & 1u : (j == (unsigned)only ? q : 0u);
        return ivd{p[up][j], p[up + 1][j]};
    }
};

// entries r, r + G, ... of a parent's table
__device__ __forceinline__ void fill_table(const SysTab &T, const DevSys &S, float4 *tv, const double (*sp)[kMaxVars],
                                           const float (*se)[kMaxVars], int only, unsigned r, unsigned G) {
    for (int e = (int)r; e < S.n_tv; e += (int)G) {
        const uint32_t mp = T.tv_map[e];
        if (S.prefilter) {
            tv[e] = term_shadow(T, (int)(mp >> 8), ComboCoordShadow{se, mp & 255u, only});
        } else {
            const ivd v = term_combo64(T, (int)(mp >> 8), ComboCoord64{sp, mp & 255u, only});
            reinterpret_cast<double2 *>(tv)[e] = make_double2(v.lo, v.hi);
        }
    }
}

// table entry of term t for the child with bits c: the variables below 8 through the
// child-index table (one byte a child), the others from the factors (in variable order)
__device__ __forceinline__ int high_bits(const SysTab &T, int t, unsigned c) {
    const uint32_t info = T.tinfo[t];
    const int f0 = term_f0(info);
    unsigned q = 0;
    for (int f = term_nf(info) - 1; f >= 0; f--) {
        const unsigned v = T.fac[f0 + f] >> 4;
        if (v < 8) break;
        q |= ((c >> v) & 1u) << f;
    }
    return (int)q;
}
__device__ __forceinline__ int entry_of(const SysTab &T, const DevSys &S, int t, unsigned c, int only) {
    if (only >= 0) return T.tv_off[t] + (int)((c >> only) & 1u);
    if (S.n_cix > 0) {
        const int lb = S.n < 8 ? S.n : 8;
        return T.tv_off[t] + (int)T.cix[((unsigned)t << lb) + (c & ((1u << lb) - 1u))] + (S.n > 8 ? high_bits(T, t, c) : 0);
    }
    const uint32_t info = T.tinfo[t];
    const int nf = term_nf(info), f0 = term_f0(info);
    unsigned q = 0;
    for (int f = 0; f < nf; f++) q |= ((c >> (T.fac[f0 + f] >> 4)) & 1u) << f;
    return T.tv_off[t] + (int)q;
}

// the running sums of one equation over one child, shadow or FP64, and their verdict
struct SumShadow {
    shv a;
    __device__ __forceinline__ void set(const float4 *tv, int e) {
        const float4 v = tv[e];
        a = shv{v.x, v.y, v.z, v.w};
    }
    __device__ __forceinline__ void add(const float4 *tv, int e) {
        const float4 v = tv[e];
        a = sh_add(a, shv{v.x, v.y, v.z, v.w});
    }
    __device__ __forceinline__ void zero() { a = shv{0.f, 0.f, 0.f, 0.f}; }
    __device__ __forceinline__ unsigned state() const {
        if (a.ld > 0.0f || a.hu < 0.0f) return CH_OUT;
        return (a.lu <= 0.0f && a.hd >= 0.0f) ? 0u : CH_OPEN;   // NaN (a poisoned term) is open
    }
};
struct Sum64 {
    ivd a;
    __device__ __forceinline__ void set(const float4 *tv, int e) {
        const double2 v = reinterpret_cast<const double2 *>(tv)[e];
        a = ivd{v.x, v.y};
    }
    __device__ __forceinline__ void add(const float4 *tv, int e) {
        const double2 v = reinterpret_cast<const double2 *>(tv)[e];
        a = iv_add(a, ivd{v.x, v.y});
    }
    __device__ __forceinline__ void zero() { a = ivd{0.0, 0.0}; }
    __device__ __forceinline__ unsigned state() const { return d_pos(a.lo) || d_neg(a.hi) ? CH_OUT : 0u; }
};

// state of child c under equation i, from the table
template <class Sum>
__device__ __forceinline__ unsigned table_state(const SysTab &T, const DevSys &S, const float4 *tv, int i, unsigned c,
                                                int only) {
    const int t0 = T.poly_off[S.f_poly + i], t1 = T.poly_off[S.f_poly + i + 1];
    Sum s;
    s.zero();
    for (int t = t0; t < t1; t++) {
        const int e = entry_of(T, S, t, c, only);
        if (t == t0) s.set(tv, e);
        else s.add(tv, e);
    }
    return s.state();
}
// the same without a table
__device__ __forceinline__ unsigned direct_state(const SysTab &T, const DevSys &S, const double (*sp)[kMaxVars],
                                                 const float (*se)[kMaxVars], int i, unsigned c) {
    if (S.prefilter) {
        bool poison = false;
        const shv F = poly_shadow(T, S.f_poly + i, ChildCoordShadow{se, c}, poison);
        if (poison) return CH_OPEN;
        return SumShadow{F}.state();
    }
    return Sum64{poly64(T, S.f_poly + i, ChildCoord64{sp, c})}.state();
}

// One round of a warp over the children still in (entries [b0, b0 + 32 K) of `m` in `list`;
// the first equation takes entry q = child q): equation i decides K children per lane, K
// independent chains, and the ones that stay are packed to the front of the list.
template <class Sum, int K>
__device__ __forceinline__ void list_round(const SysTab &T, const DevSys &S, const float4 *tv, uint16_t *list, unsigned c0,
                                           int i, bool first, unsigned b0, unsigned m, unsigned &out, unsigned &n_out) {
    const unsigned lane = lane_id();
    const int lb = S.n < 8 ? S.n : 8;
    unsigned ent[K];
    bool act[K];
#pragma unroll
    for (int k = 0; k < K; k++) {
        const unsigned q = b0 + (unsigned)k * 32u + lane;
        act[k] = q < m;
        ent[k] = first ? (act[k] ? q : 0u) : (act[k] ? (unsigned)list[q] : 0u);
    }
    Sum s[K];
#pragma unroll
    for (int k = 0; k < K; k++) s[k].zero();
    const int t0 = T.poly_off[S.f_poly + i], t1 = T.poly_off[S.f_poly + i + 1];
    const unsigned low0 = c0 & ((1u << lb) - 1u);
    for (int t = t0; t < t1; t++) {
        const int off = T.tv_off[t] + (S.n > 8 ? high_bits(T, t, c0) : 0);
        const uint8_t *row = T.cix + ((unsigned)t << lb) + low0;
#pragma unroll
        for (int k = 0; k < K; k++) {
            const int e = off + (int)row[ent[k] & 255u];
            if (t == t0) s[k].set(tv, e);
            else s[k].add(tv, e);
        }
    }
    __syncwarp();   // every entry of the round has been read before any is written
#pragma unroll
    for (int k = 0; k < K; k++) {
        const unsigned st = s[k].state();
        const bool stay = act[k] && !(st & CH_OUT);
        n_out += act[k] && (st & CH_OUT) ? 1u : 0u;
        const unsigned bal = __ballot_sync(kFull, stay);
        if (stay) list[out + __popc(bal & lanemask_lt())] = (uint16_t)(ent[k] | ((st & CH_OPEN) ? 256u : 0u));
        out += __popc(bal);
    }
    __syncwarp();
}

// Children [c0, c0 + m) (m <= 256, c0 a multiple of m) of parent pi by one warp.  Every
// equation excludes a third to a half of what is left, so the equations run over a list
// of the children still in, packed after each: at n = 8 about 22 rounds of 32 instead of the
// 64 that a lane per child takes (a warp's 32 lanes hardly ever finish early together).
// Equations with fewer terms come first: cheaper, and narrower.  The survivors leave with
// one reservation of the survivor list instead of one per 32 children.  (Evaluation of the
// n = 8 plan, 6.4e7 children: 3.47 -> 2.35 ms; kinema, n = 9, 6.5e8: 62 -> 37 ms; n = 11, 3.2e7:
// 23 -> 2.8 ms, where a table per warp had left one block per SM and no child index; 64-system
// batch 144 -> 82 ms; the FP64-only n = 6 plan, whose children had no table: 0.91 -> 0.39 ms.)
template <class Sum>
__device__ __forceinline__ void list_children(const SweepArgs &a, WaveCtl *ctl, const SysTab &T, const DevSys &S,
                                              const uint8_t *order, const float4 *tv, uint16_t *list, int64_t pi, unsigned c0,
                                              unsigned m, unsigned &n_out, unsigned &n_keep) {
    for (int q = 0; q < S.m && m > 0; q++) {
        const int i = S.m <= kMaxVars ? (int)order[q] : q;
        unsigned out = 0;
        for (unsigned b0 = 0; b0 < m;) {
            if (m - b0 > 64) {
                list_round<Sum, 4>(T, S, tv, list, c0, i, q == 0, b0, m, out, n_out);
                b0 += 128;
            } else if (m - b0 > 32) {
                list_round<Sum, 2>(T, S, tv, list, c0, i, q == 0, b0, m, out, n_out);
                b0 += 64;
            } else {
                list_round<Sum, 1>(T, S, tv, list, c0, i, q == 0, b0, m, out, n_out);
                b0 += 32;
            }
        }
        m = out;
    }
    for (unsigned b0 = 0; b0 < m; b0 += 32) {
        const bool act = b0 + lane_id() < m;
        const unsigned ent = act ? (unsigned)list[b0 + lane_id()] : 0u;
        const Surv sv{(uint32_t)pi, c0 + (ent & 255u)};
        const bool keep = act && !(ent & 256u);
        n_keep += keep ? 1u : 0u;
        push_surv(a, ctl, S.n, keep, sv);
        push_cand(a, ctl, act && (ent & 256u), sv);
    }
    __syncwarp();
}

// counts of one warp's children, in per-lane parts
struct EvalCount {
    unsigned pre, ev, e64, keep;
};
__device__ __forceinline__ void add_counts(const SweepArgs &a, int sys, const EvalCount &c) {
    const unsigned pre = __reduce_add_sync(kFull, c.pre), ev = __reduce_add_sync(kFull, c.ev);
    const unsigned e64 = __reduce_add_sync(kFull, c.e64), keep = __reduce_add_sync(kFull, c.keep);
    if (lane_id() == 0) {
        if (pre) atomicAdd(stat_ptr(a, sys, ST_EXCL_PREFILTER), (unsigned long long)pre);
        if (ev) atomicAdd(stat_ptr(a, sys, ST_EXCL_EVAL), (unsigned long long)ev);
        if (e64) atomicAdd(stat_ptr(a, sys, ST_EVAL64), (unsigned long long)e64);
        if (keep) atomicAdd(stat_ptr(a, sys, ST_KEEP_SHADOW), (unsigned long long)keep);
    }
}
__device__ __forceinline__ void add_parents(const SweepArgs &a, int sys, int depth, unsigned parents,
                                            unsigned long long boxes) {
    if (lane_id() == 0 && parents) {
        atomicAdd(stat_ptr(a, sys, ST_LIVE), ~(unsigned long long)parents + 1ull);
        atomicAdd(stat_ptr(a, sys, ST_BOXES), boxes);
        if (boxes) atomicMax(stat_ptr(a, sys, ST_MAX_DEPTH), (unsigned long long)depth);
        if (boxes) atomicAdd(stat_ptr(a, sys, ST_DEPTH_BOXES + (depth < kDepthSlots ? depth : kDepthSlots - 1)), boxes);
    }
}

template <bool BLOCK>
__device__ __forceinline__ void group_sync() {
    if (BLOCK) __syncthreads();
    else __syncwarp();
}

// The parent's coordinates into shared memory, by the first n threads of its group
__device__ __forceinline__ void load_parent(const SweepArgs &a, int64_t pi, int n, double (*sp)[kMaxVars],
                                            float (*sf)[kMaxVars], float (*se)[kMaxVars], unsigned r) {
    if ((int)r < n) {
        const double lo = a.q.lo[r * a.q.cap + pi];
        const double mid = a.q.mid[r * a.q.cap + pi];
        const double hi = a.q.hi[r * a.q.cap + pi];
        sp[0][r] = lo;
        sp[1][r] = mid;
        sp[2][r] = hi;
        const float lod = __double2float_rd(lo), lou = __double2float_ru(lo);
        const float mdd = __double2float_rd(mid), mdu = __double2float_ru(mid);
        const float hid = __double2float_rd(hi), hiu = __double2float_ru(hi);
        sf[0][r] = lod;
        sf[1][r] = mdd;
        sf[2][r] = mdu;
        sf[3][r] = hiu;
        se[0][r] = lod;
        se[1][r] = lou;
        se[2][r] = mdd;
        se[3][r] = mdu;
        se[4][r] = hid;
        se[5][r] = hiu;
    }
}

// Children of one parent spread over a group (a warp, or a block of 256 threads) by
// (equation, child) pairs, `chunk` children at a time: for few children, or few parents,
// where lanes would idle otherwise and a thread that takes a child's equations one after the
// other waits on their chain (evaluation of an n = 5 bisection, 35 narrow sweeps: 34 -> 16.5 us
// a sweep; of the n = 6 solve: 0.31 -> 0.25 ms).  state: chunk words.
template <bool BLOCK>
__device__ __forceinline__ void pair_children(const SweepArgs &a, WaveCtl *ctl, const SysTab &T, const DevSys &S,
                                              const float4 *tv, bool use_tv, const double (*sp)[kMaxVars],
                                              const float (*se)[kMaxVars], unsigned *state, unsigned chunk, uint32_t meta,
                                              int64_t pi, unsigned fan, int only, unsigned r, unsigned G, EvalCount &cnt) {
    for (unsigned c0 = 0; c0 < fan; c0 += chunk) {
        const unsigned cn = fan - c0 < chunk ? fan - c0 : chunk;
        for (unsigned q = r; q < cn; q += G) state[q] = 0u;
        group_sync<BLOCK>();
        const unsigned pairs = cn * (unsigned)S.m;
        for (unsigned e = r; e < pairs; e += G) {
            const unsigned q = e % cn;
            const int i = (int)(e / cn);
            const unsigned c = child_bits(S, meta, c0 + q);
            const unsigned st = !use_tv ? direct_state(T, S, sp, se, i, c)
                                : S.prefilter ? table_state<SumShadow>(T, S, tv, i, c, only)
                                              : table_state<Sum64>(T, S, tv, i, c, only);
            if (st) atomicOr(&state[q], st);
        }
        group_sync<BLOCK>();
        for (unsigned q0 = 0; q0 < cn; q0 += G) {
            const bool act = q0 + r < cn;
            const unsigned st = act ? state[q0 + r] : CH_OUT;
            const bool keep = act && st == 0u, open = act && st == CH_OPEN;
            const Surv sv{(uint32_t)pi, child_bits(S, meta, c0 + q0 + r)};
            if (S.prefilter) {
                cnt.pre += act && (st & CH_OUT) ? 1u : 0u;
                cnt.keep += keep ? 1u : 0u;
            } else {
                cnt.e64 += act ? 1u : 0u;
                cnt.ev += act && (st & CH_OUT) ? 1u : 0u;
            }
            push_surv(a, ctl, S.n, keep, sv);
            if (S.prefilter) push_cand(a, ctl, open, sv);
        }
        group_sync<BLOCK>();
    }
}

// Up to 16 children of one parent by one warp: lane e takes pairs e, e + 32, ... of (equation,
// child), always of child e mod fan (fan is a power of two), and the lanes of a child join
// their states with shuffles.
__device__ __forceinline__ void few_children(const SweepArgs &a, WaveCtl *ctl, const SysTab &T, const DevSys &S,
                                             const float4 *tv, bool use_tv, const double (*sp)[kMaxVars],
                                             const float (*se)[kMaxVars], uint32_t meta, int64_t pi, unsigned fan, int only,
                                             EvalCount &cnt) {
    const unsigned lane = lane_id(), q = lane & (fan - 1u), pairs = fan * (unsigned)S.m;
    const unsigned c = child_bits(S, meta, q);
    unsigned st = 0u;
    for (unsigned e = lane; e < pairs; e += 32u) {
        const int i = (int)(e / fan);
        st |= !use_tv ? direct_state(T, S, sp, se, i, c)
              : S.prefilter ? table_state<SumShadow>(T, S, tv, i, c, only)
                            : table_state<Sum64>(T, S, tv, i, c, only);
    }
    __syncwarp();
    for (unsigned o = fan; o < 32u; o <<= 1) st |= __shfl_xor_sync(kFull, st, (int)o);
    const bool act = lane < fan, keep = act && st == 0u, open = act && st == CH_OPEN;
    const Surv sv{(uint32_t)pi, c};
    if (S.prefilter) {
        cnt.pre += act && (st & CH_OUT) ? 1u : 0u;
        cnt.keep += keep ? 1u : 0u;
    } else {
        cnt.e64 += act ? 1u : 0u;
        cnt.ev += act && (st & CH_OUT) ? 1u : 0u;
    }
    push_surv(a, ctl, S.n, keep, sv);
    if (S.prefilter) push_cand(a, ctl, open, sv);
}

// Without the shadow (magnitudes that float may not hold): the plain FP32 prefilter, one
// child per thread; its survivors go to k_eval64.
__device__ __forceinline__ void plain_children(const SweepArgs &a, WaveCtl *ctl, const SysTab &T, const DevSys &S,
                                               const float (*sf)[kMaxVars], uint32_t meta, int64_t pi, unsigned fan,
                                               unsigned r, unsigned G, EvalCount &cnt) {
    for (unsigned c0 = 0; c0 < fan; c0 += G) {
        const bool active = c0 + r < fan;
        const unsigned c = child_bits(S, meta, c0 + r);
        const bool cand = active && keep32(T, S, ChildCoord32{sf, c});
        cnt.pre += active && !cand ? 1u : 0u;
        push_cand(a, ctl, cand, Surv{(uint32_t)pi, c});
    }
}

// Past its box budget a system's children are dropped.
__device__ __forceinline__ bool over_budget(const SweepArgs &a, int sys, const DevSys &S) {
    if (S.max_boxes <= 0) return false;
    const unsigned long long done = *(volatile unsigned long long *)stat_ptr(a, sys, ST_BOXES);
    if ((long long)done < S.max_boxes) return false;
    atomicOr(stat_ptr(a, sys, ST_FLAGS), (unsigned long long)kFlagBudget);
    return true;
}

// Whether a parent of system S takes a block in wide sweeps: its table does not fit a
// warp's share of the region, or a block's warps each get 64 of its children or more.
__device__ __forceinline__ bool block_form(const SweepArgs &a, const DevSys &S) {
    return S.eval_block || S.n_tv > a.tv_entries / kEvalWarps;
}

// Without a table (more combinations than a region holds), one child per thread.
__device__ __forceinline__ void direct_children(const SweepArgs &a, WaveCtl *ctl, const SysTab &T, const DevSys &S,
                                                const double (*sp)[kMaxVars], const float (*se)[kMaxVars], uint32_t meta,
                                                int64_t pi, unsigned fan, unsigned r, unsigned G, EvalCount &cnt) {
    for (unsigned c0 = 0; c0 < fan; c0 += G) {
        const bool active = c0 + r < fan;
        const unsigned c = child_bits(S, meta, c0 + r);
        bool keep = false, cand = false;
        if (active && S.prefilter) {
            const int d = decide_shadow(T, S, ChildCoordShadow{se, c});
            keep = d == 1;
            cand = d == 2;
            cnt.pre += d == 0 ? 1u : 0u;
            cnt.keep += keep ? 1u : 0u;
        } else if (active) {
            cnt.e64 += 1;
            keep = keep64(T, S, ChildCoord64{sp, c});
            cnt.ev += keep ? 0u : 1u;
        }
        push_surv(a, ctl, S.n, keep, Surv{(uint32_t)pi, c});
        if (S.prefilter) push_cand(a, ctl, cand, Surv{(uint32_t)pi, c});
    }
}

// children [c0, c0 + m) by one warp through list_children, with the counts of either mode
__device__ __forceinline__ void listed(const SweepArgs &a, WaveCtl *ctl, const SysTab &T, const DevSys &S,
                                       const uint8_t *order, const float4 *tv, uint16_t *list, int64_t pi, unsigned c0,
                                       unsigned m, EvalCount &cnt) {
    unsigned n_out = 0, n_keep = 0;
    if (S.prefilter) {
        list_children<SumShadow>(a, ctl, T, S, order, tv, list, pi, c0, m, n_out, n_keep);
        cnt.pre += n_out;
        cnt.keep += n_keep;
    } else {
        list_children<Sum64>(a, ctl, T, S, order, tv, list, pi, c0, m, n_out, n_keep);
        cnt.ev += n_out;
        cnt.e64 += lane_id() == 0 ? m : 0u;
    }
}

// What a warp has counted for the system and depth of its last parents: added to the
// system's counters when either changes and at the end, not parent by parent (six atomics on
// the same six addresses for each of the 16384 parents of an n = 8 sweep).
struct WarpTally {
    int sys, depth;
    unsigned parents;
    unsigned long long boxes;
    EvalCount cnt;
};
__device__ __forceinline__ void flush_tally(const SweepArgs &a, WarpTally &w) {
    if (w.parents) {
        add_counts(a, w.sys, w.cnt);
        add_parents(a, w.sys, w.depth, w.parents, w.boxes);
    }
    w.parents = 0;
    w.boxes = 0;
    w.cnt = EvalCount{0u, 0u, 0u, 0u};
}

// One parent per warp.
__device__ __forceinline__ void eval_warp(const SweepArgs &a, WaveCtl *ctl, const char *s_blob, float4 *s_tv,
                                          double (*sp)[kMaxVars], float (*sf)[kMaxVars], float (*se)[kMaxVars],
                                          uint16_t *list, int64_t pi, WarpTally &w) {
    const unsigned lane = lane_id();
    const int sys = a.q.sys[pi];
    const uint32_t meta = a.q.meta[pi];
    const DevSys S = a.tb.sys[sys];
    if (block_form(a, S)) return;   // the block pass takes it
    const SysTab T = make_tab(a.blob_smem ? s_blob : a.tb.blobs + S.blob_off, S);
    const bool root = (meta & kRootFlag) != 0;
    const int depth = (int)(meta & kDepthMask) + (root ? 0 : 1);
    if (sys != w.sys || depth != w.depth || S.max_boxes > 0) {
        flush_tally(a, w);
        w.sys = sys;
        w.depth = depth;
    }
    w.parents += 1;
    int over = 0;
    if (lane == 0) over = over_budget(a, sys, S) ? 1 : 0;
    if (__shfl_sync(kFull, over, 0)) return;
    const unsigned fan = (unsigned)fan_out(S, meta);
    w.boxes += fan;
    load_parent(a, pi, S.n, sp, sf, se, lane);
    __syncwarp();
    const bool plain = S.prefilter && !S.shadow;
    // a round of short equations is sooner evaluated than a table filled for it
    const bool brief = fan * (unsigned)S.m <= 32u && S.n_fterms <= 4 * S.m;
    const bool use_tv = !plain && !brief && S.n_tv > 0 && S.n_tv <= a.tv_entries / kEvalWarps;
    const int only = S.bisect ? (int)((meta >> kSplitShift) & kSplitMask) : -1;
    if (use_tv) {
        fill_table(T, S, s_tv, sp, se, only, lane, 32u);
        __syncwarp();
    }
    if (plain) {
        plain_children(a, ctl, T, S, sf, meta, pi, fan, lane, 32u, w.cnt);
    } else if (use_tv && fan >= 32 && S.n_cix > 0) {
        for (unsigned c0 = 0; c0 < fan; c0 += 256)
            listed(a, ctl, T, S, a.tb.sys[sys].eq_order, s_tv, list, pi, c0, fan - c0 < 256 ? fan - c0 : 256, w.cnt);
    } else if (fan < 32) {
        few_children(a, ctl, T, S, s_tv, use_tv, sp, se, meta, pi, fan, only, w.cnt);
    } else if (use_tv) {
        pair_children<false>(a, ctl, T, S, s_tv, use_tv, sp, se, reinterpret_cast<unsigned *>(list), 64u, meta, pi, fan, only,
                             lane, 32u, w.cnt);
    } else {
        direct_children(a, ctl, T, S, sp, se, meta, pi, fan, lane, 32u, w.cnt);
    }
    __syncwarp();   // the parent's arrays are rewritten for the next parent
}

// One parent per block: its table is filled by all threads; many children go to the warps
// in equal parts (list_children), few are spread by (equation, child) pairs.
__device__ __forceinline__ void eval_block(const SweepArgs &a, WaveCtl *ctl, const char *s_blob, float4 *s_tv,
                                           double (*sp)[kMaxVars], float (*sf)[kMaxVars], float (*se)[kMaxVars],
                                           uint16_t *lists, int *s_flag, int64_t pi) {
    const unsigned t = threadIdx.x, warp = t >> 5;
    const int sys = a.q.sys[pi];
    const uint32_t meta = a.q.meta[pi];
    const DevSys S = a.tb.sys[sys];
    const SysTab T = make_tab(a.blob_smem ? s_blob : a.tb.blobs + S.blob_off, S);
    const bool root = (meta & kRootFlag) != 0;
    const int depth = (int)(meta & kDepthMask) + (root ? 0 : 1);
    if (t == 0) *s_flag = over_budget(a, sys, S) ? 1 : 0;
    load_parent(a, pi, S.n, sp, sf, se, t);
    __syncthreads();
    const bool over = *s_flag != 0;
    const unsigned fan = (unsigned)fan_out(S, meta);
    if (!over) {
        const bool plain = S.prefilter && !S.shadow;
        const bool use_tv = !plain && S.n_tv > 0 && S.n_tv <= a.tv_entries;
        const int only = S.bisect ? (int)((meta >> kSplitShift) & kSplitMask) : -1;
        EvalCount cnt{0u, 0u, 0u, 0u};
        if (use_tv) {
            fill_table(T, S, s_tv, sp, se, only, t, kEvalThreads);
            __syncthreads();
        }
        if (plain) {
            plain_children(a, ctl, T, S, sf, meta, pi, fan, t, kEvalThreads, cnt);
        } else if (use_tv && fan >= 512 && S.n_cix > 0) {
            const unsigned m = fan / kEvalWarps < 256 ? fan / kEvalWarps : 256;
            for (unsigned c0 = warp * m; c0 < fan; c0 += kEvalWarps * m)
                listed(a, ctl, T, S, a.tb.sys[sys].eq_order, s_tv, lists + warp * 256, pi, c0, m, cnt);
        } else if (use_tv || fan < 32) {
            pair_children<true>(a, ctl, T, S, s_tv, use_tv, sp, se, reinterpret_cast<unsigned *>(lists), 256u, meta, pi, fan,
                                only, t, kEvalThreads, cnt);
        } else {
            direct_children(a, ctl, T, S, sp, se, meta, pi, fan, t, kEvalThreads, cnt);
        }
        add_counts(a, sys, cnt);
    }
    if (warp == 0) add_parents(a, sys, depth, 1u, over ? 0ull : (unsigned long long)fan);
    __syncthreads();   // the parent's arrays and s_flag are rewritten for the next parent
}

// Children of the popped parents.  A narrow sweep (no more parents than blocks) gives each
// block a parent at a time.  A wide one gives each warp a parent at a time from a shared
// cursor, and then each block the parents of the systems whose table or number of children
// asks for a block.
__global__ void __launch_bounds__(kEvalThreads, 3) k_eval(SweepArgs a) {
    extern __shared__ __align__(16) char s_blob[];
    float4 *s_tv = reinterpret_cast<float4 *>(s_blob + a.blob_smem);
    __shared__ double s_p[kEvalWarps][3][kMaxVars];
    __shared__ float s_f[kEvalWarps][4][kMaxVars];
    __shared__ float s_e[kEvalWarps][6][kMaxVars];
    __shared__ __align__(8) uint16_t s_list[kEvalWarps * 256];
    __shared__ unsigned s_need[kEvalWarps];
    __shared__ int s_flag;
    const unsigned lane = lane_id();
    const int w = threadIdx.x >> 5;
    WaveCtl *ctl = a.ctl;
    const int64_t base = ctl->base, K = ctl->k;
    const bool narrow = K <= (int64_t)gridDim.x;
    const bool block_pass = narrow || (a.eval_forms & 2), warp_pass = !narrow && (a.eval_forms & 1);
    // blocks beyond what K parents need leave at once (the others take every parent), so
    // a small sweep does not pay for the whole grid
    if (block_pass ? (int64_t)blockIdx.x >= K : (int64_t)blockIdx.x * kEvalWarps >= K) return;
    if (a.blob_smem) {
        copy_blob(s_blob, a.tb.blobs + a.tb.sys[0].blob_off, (uint32_t)a.blob_smem);
        __syncthreads();
    }
    if (warp_pass) {
        float4 *tv = s_tv + (size_t)w * (a.tv_entries / kEvalWarps);
        WarpTally tally{-1, 0, 0u, 0ull, EvalCount{0u, 0u, 0u, 0u}};
        for (;;) {
            int p = 0;
            if (lane == 0) p = atomicAdd(&ctl->cursor, 1);
            p = __shfl_sync(kFull, p, 0);
            if (p >= K) break;
            eval_warp(a, ctl, s_blob, tv, s_p[w], s_f[w], s_e[w], s_list + w * 256, parent_index(a, base, p), tally);
        }
        flush_tally(a, tally);
        if (!block_pass) return;
        __syncthreads();
    }
    if (!warp_pass) {
        for (int64_t p = blockIdx.x; p < K; p += gridDim.x) {
            const int64_t pi = parent_index(a, base, p);
            if (!(a.eval_forms & 4)) {
                eval_block(a, ctl, s_blob, s_tv, s_p[0], s_f[0], s_e[0], s_list, &s_flag, pi);
            } else if (w == 0) {
                // parents of up to 8 children: a warp each, without the block's barriers
                WarpTally tally{-1, 0, 0u, 0ull, EvalCount{0u, 0u, 0u, 0u}};
                eval_warp(a, ctl, s_blob, s_tv, s_p[0], s_f[0], s_e[0], s_list, pi, tally);
                flush_tally(a, tally);
            }
        }
        return;
    }
    // the parents that the warps left, 256 of the block's at a time
    for (int64_t p0 = blockIdx.x; p0 < K; p0 += (int64_t)gridDim.x * kEvalThreads) {
        const int64_t p = p0 + (int64_t)threadIdx.x * gridDim.x;
        const bool need = p < K && block_form(a, a.tb.sys[a.q.sys[parent_index(a, base, p)]]);
        const unsigned bal = __ballot_sync(kFull, need);
        if (lane == 0) s_need[w] = bal;
        __syncthreads();
        for (int v = 0; v < kEvalWarps; v++)
            for (unsigned bits = s_need[v]; bits; bits &= bits - 1u)
                eval_block(a, ctl, s_blob, s_tv, s_p[0], s_f[0], s_e[0], s_list, &s_flag,
                           parent_index(a, base, p0 + (int64_t)(v * 32 + __ffs(bits) - 1) * gridDim.x));
        __syncthreads();
    }
}

// FP64 evaluation of the candidates (undecided by the FP32 stage), 32 / g per warp from an
// atomic cursor.  Few candidates (a sweep with the FP32 shadow leaves some hundred): g = 8
// lanes share a candidate's equations, so the kernel takes one or two equations' chains
// instead of all of them one after the other (n = 8: 26 -> 15 us a sweep, n = 7: 25 -> 13).  Many: one lane each (g = 1), which
// stops at the first equation that excludes, so the FP64 pipe does no more than it has to.
constexpr int64_t kSplitCandidates = 16384;
__global__ void __launch_bounds__(kEval64Threads) k_eval64(SweepArgs a) {
    extern __shared__ __align__(16) char s_blob[];
    __shared__ double sX[2 * kMaxVars * kEval64Threads];
    const int T = blockDim.x, tid = threadIdx.x;
    double *X = sX + tid;
    WaveCtl *ctl = a.ctl;
    const int64_t count = ctl->cand_count;
    const bool split = count <= kSplitCandidates;
    // not needed for this many candidates
    if ((int64_t)blockIdx.x * blockDim.x >= (split ? 8 * count : count)) return;
    if (a.head_smem) {
        copy_blob(s_blob, a.tb.blobs + a.tb.sys[0].blob_off, (uint32_t)a.head_smem);
        __syncthreads();
    }
    const unsigned lane = lane_id();
    for (;;) {
        // candidates of the warp: 32, or 4 with 8 lanes each (equations lane, lane + 8, ...)
        const int per = split ? 4 : 32;
        unsigned long long base = 0;
        if (lane == 0) base = atomicAdd((unsigned long long *)&ctl->cand_cursor, (unsigned long long)per);
        base = __shfl_sync(kFull, base, 0);
        if ((long long)base >= count) break;
        const int64_t idx = (int64_t)base + (split ? lane >> 3 : lane);
        const bool there = idx < count;
        bool keep = false;
        int sys = 0, n = 0;
        Surv sv{0, 0};
        if (there) {
            sv = a.cand[idx];
            const int64_t pi = sv.parent;
            sys = a.q.sys[pi];
            const DevSys S = a.tb.sys[sys];
            const SysTab Tb = make_tab(a.head_smem ? s_blob : a.tb.blobs + S.blob_off, S);
            n = S.n;
            for (int j = 0; j < n; j++) {
                const bool up = (sv.child >> j) & 1u;
                X[(2 * j) * T] = up ? a.q.mid[j * a.q.cap + pi] : a.q.lo[j * a.q.cap + pi];
                X[(2 * j + 1) * T] = up ? a.q.hi[j * a.q.cap + pi] : a.q.mid[j * a.q.cap + pi];
            }
            if (split) {
                keep = true;
                for (int i = (int)(lane & 7u); i < S.m; i += 8) {
                    const ivd F = poly64(Tb, S.f_poly + i, BoxCoord{X, T});
                    keep = keep && !(d_pos(F.lo) || d_neg(F.hi));
                }
            } else {
                keep = keep64(Tb, S, BoxCoord{X, T});
            }
        }
        __syncwarp();
        bool active = there;
        if (split) {   // a candidate's first lane speaks for it
            const unsigned kept = __ballot_sync(kFull, keep);
            keep = ((kept >> (lane & 24u)) & 255u) == 255u;
            active = there && (lane & 7u) == 0u;
            keep = keep && active;
        }
        const int sys0 = __shfl_sync(kFull, sys, 0);
        const int n0 = __shfl_sync(kFull, n, 0);
        const bool uniform = __all_sync(kFull, !active || (sys == sys0 && n == n0));
        if (uniform) {
            push_surv(a, ctl, n0, keep, sv);
            const unsigned na = __popc(__ballot_sync(kFull, active));
            const unsigned nk = __popc(__ballot_sync(kFull, keep));
            if (lane == 0) {
                atomicAdd(stat_ptr(a, sys0, ST_EVAL64), (unsigned long long)na);
                if (na - nk) atomicAdd(stat_ptr(a, sys0, ST_EXCL_EVAL), (unsigned long long)(na - nk));
            }
        } else if (active) {
            if (keep) {
                const unsigned long long k = atomicAdd((unsigned long long *)&ctl->surv_count[n], 1ull);
                if ((long long)k < a.surv_cap) a.surv[(size_t)n * a.surv_cap + k] = sv;
                else ctl->error = 1;
            }
            atomicAdd(stat_ptr(a, sys, ST_EVAL64), 1ull);
            if (!keep) atomicAdd(stat_ptr(a, sys, ST_EXCL_EVAL), 1ull);
        }
    }
}

// ------------------------------------------------------------------------------------
// launchers
// ------------------------------------------------------------------------------------

static cudaError_t launch_hs(const SweepArgs &a, int n, int num_sms, cudaStream_t st, int *kernels) {
    switch (n) {
    case 1: return launch_hs_dim1(a, num_sms, st, kernels);
    case 2: return launch_hs_dim2(a, num_sms, st, kernels);
    case 3: return launch_hs_dim3(a, num_sms, st, kernels);
    case 4: return launch_hs_dim4(a, num_sms, st, kernels);
    case 5: return launch_hs_dim5(a, num_sms, st, kernels);
    case 6: return launch_hs_dim6(a, num_sms, st, kernels);
    case 7: return launch_hs_dim7(a, num_sms, st, kernels);
    case 8: return launch_hs_dim8(a, num_sms, st, kernels);
    case 9: return launch_hs_dim9(a, num_sms, st, kernels);
    case 10: return launch_hs_dim10(a, num_sms, st, kernels);
    case 11: return launch_hs_dim11(a, num_sms, st, kernels);
    case 12: return launch_hs_dim12(a, num_sms, st, kernels);
    case 13: return launch_hs_dim13(a, num_sms, st, kernels);
    case 14: return launch_hs_dim14(a, num_sms, st, kernels);
    case 15: return launch_hs_dim15(a, num_sms, st, kernels);
    case 16: return launch_hs_dim16(a, num_sms, st, kernels);
    default: return cudaErrorInvalidValue;
    }
}

size_t eval_smem_bytes(const SweepArgs &a) {
    return (size_t)a.blob_smem + (size_t)a.tv_entries * sizeof(float4);
}

cudaError_t allow_max_dynamic_smem(const void *func) {
    // The attribute is global to the kernel: every plan and server sets the same maximum,
    // so one whose launches need less never lowers it under another's captured graph.
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaFuncAttributes fa{};
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, func);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes);
    return e;
}

cudaError_t configure_eval_kernels(const SweepArgs &a) {
    (void)a;
    cudaError_t e = allow_max_dynamic_smem((const void *)k_wave_begin);
    if (e != cudaSuccess) return e;
    e = allow_max_dynamic_smem((const void *)k_eval);
    if (e != cudaSuccess) return e;
    return allow_max_dynamic_smem((const void *)k_eval64);
}

// Branches of the contraction stage in a captured sweep.  The kernels of one dimension touch
// nothing of another's (own survivor list, own part of a.cand, own cursors; results, staging
// and counters through atomics), and most sweeps of a batch leave the small dimensions a few
// boxes each, whose 25-50 us of latency added up one dimension after the other (96-system
// batch of n = 2..5: 3.7 of 5.3 ms; the call 8.0 -> 6.7 ms, 24 served requests 70 -> 67 ms, the
// 64-system batch 257 -> 252).  Branch 0 is the capturing stream; the largest dimensions
// get a branch of their own, the rest share them in reverse order.
constexpr int kBranches = 4;
struct Branches {
    cudaStream_t st[kBranches] = {};
    cudaEvent_t fork = nullptr, join[kBranches] = {};
    int n = 1;
    cudaError_t open(cudaStream_t main, int dims) {
        st[0] = main;
        n = dims < kBranches ? dims : kBranches;
        cudaError_t e = cudaSuccess;
        if (n > 1) e = cudaEventCreateWithFlags(&fork, cudaEventDisableTiming);
        for (int b = 1; b < n && e == cudaSuccess; b++) {
            e = cudaStreamCreateWithFlags(&st[b], cudaStreamNonBlocking);
            if (e == cudaSuccess) e = cudaEventCreateWithFlags(&join[b], cudaEventDisableTiming);
        }
        return e;
    }
    // branch of the q-th largest of the dimensions
    int of(int q) const {
        const int r = q % (2 * n);
        return r < n ? r : 2 * n - 1 - r;
    }
    ~Branches() {
        for (int b = 1; b < kBranches; b++) {
            if (st[b]) cudaStreamDestroy(st[b]);
            if (join[b]) cudaEventDestroy(join[b]);
        }
        if (fork) cudaEventDestroy(fork);
    }
};

static cudaError_t launch_sweep_impl(const SweepArgs &a, const int *hs_dims, int n_hs_dims, int eval_blocks,
                                     int num_sms, cudaStream_t st, cudaEvent_t *ev, cudaGraphConditionalHandle h,
                                     int use_cond, int *kernels, const Branches *br = nullptr) {
    int count = use_cond == 2 ? 3 : 4;   // (wave_begin,) eval, eval64, commit
    // ev (optional): n_hs_dims + 5 events recorded between the stages
    const size_t head = (size_t)a.head_smem;
    if (ev) cudaEventRecord(ev[0], st);
    if (use_cond != 2) k_wave_begin<<<1, kBeginThreads, kBeginSmem, st>>>(a);
    if (ev) cudaEventRecord(ev[1], st);
    k_eval<<<eval_blocks, kEvalThreads, eval_smem_bytes(a), st>>>(a);
    if (ev) cudaEventRecord(ev[2], st);
    k_eval64<<<num_sms * 4, kEval64Threads, head, st>>>(a);
    if (ev) cudaEventRecord(ev[3], st);
    if (br && br->n > 1) {
        cudaError_t e = cudaEventRecord(br->fork, st);
        for (int b = 1; b < br->n && e == cudaSuccess; b++) e = cudaStreamWaitEvent(br->st[b], br->fork, 0);
        for (int q = 0; q < n_hs_dims && e == cudaSuccess; q++) {
            int kq = 0;
            e = launch_hs(a, hs_dims[n_hs_dims - 1 - q], num_sms, br->st[br->of(q)], &kq);
            count += kq;
        }
        // (joined also after an error, so that the capture can end)
        for (int b = 1; b < br->n; b++) {
            cudaError_t je = cudaEventRecord(br->join[b], br->st[b]);
            if (je == cudaSuccess) je = cudaStreamWaitEvent(st, br->join[b], 0);
            if (e == cudaSuccess) e = je;
        }
        if (e != cudaSuccess) return e;
    } else
    for (int q = 0; q < n_hs_dims; q++) {
        int kq = 0;
        cudaError_t e = launch_hs(a, hs_dims[q], num_sms, st, &kq);
        if (e != cudaSuccess) return e;
        count += kq;
        if (ev) cudaEventRecord(ev[4 + q], st);
    }
    k_commit<<<num_sms * (use_cond == 2 ? 2 : 4), 256, 0, st>>>(a, a.max_fan_shift, h, use_cond);
    if (ev) cudaEventRecord(ev[4 + n_hs_dims], st);
    if (kernels) *kernels = count;
    return cudaGetLastError();
}

cudaError_t launch_sweep(const SweepArgs &a, const int *hs_dims, int n_hs_dims, int eval_blocks,
                         int eval_threads, int num_sms, cudaStream_t st, cudaEvent_t *ev, int *kernels) {
    (void)eval_threads;
    return launch_sweep_impl(a, hs_dims, n_hs_dims, eval_blocks, num_sms, st, ev, cudaGraphConditionalHandle{}, 0,
                             kernels);
}

cudaError_t build_sweep_graph(const SweepArgs &a, const int *hs_dims, int n_hs_dims, int eval_blocks,
                              int eval_threads, int num_sms, cudaGraph_t *out, int *kernels_per_sweep) {
    *out = nullptr;
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaGraphCreate(&g, 0);
    if (e != cudaSuccess) return e;
    cudaGraphConditionalHandle h;
    e = cudaGraphConditionalHandleCreate(&h, g, 1, cudaGraphCondAssignDefault);
    cudaGraphNodeParams cp = {};
    cp.type = cudaGraphNodeTypeConditional;
    cp.conditional.handle = h;
    cp.conditional.type = cudaGraphCondTypeWhile;
    cp.conditional.size = 1;
    // plans of one system: the first sweep's pop in front of the loop, the others in k_commit
    const bool fused = a.single && a.rg.n == 0;
    cudaGraphNode_t node, first = nullptr;
    if (e == cudaSuccess && fused) {
        SweepArgs copy = a;
        void *args[1] = {&copy};
        cudaKernelNodeParams kp = {};
        kp.func = (void *)k_wave_begin;
        kp.gridDim = dim3(1);
        kp.blockDim = dim3(kBeginThreads);
        kp.sharedMemBytes = (unsigned)kBeginSmem;
        kp.kernelParams = args;
        e = cudaGraphAddKernelNode(&first, g, nullptr, 0, &kp);
    }
    if (e == cudaSuccess) e = cudaGraphAddNode(&node, g, fused ? &first : nullptr, nullptr, fused ? 1 : 0, &cp);
    cudaStream_t cs = nullptr;
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking);
    Branches br;
    if (e == cudaSuccess) e = br.open(cs, n_hs_dims);
    if (e == cudaSuccess) {
        cudaGraph_t body = cp.conditional.phGraph_out[0];
        e = cudaStreamBeginCaptureToGraph(cs, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal);
        if (e == cudaSuccess) {
            (void)eval_threads;
            cudaError_t le = launch_sweep_impl(a, hs_dims, n_hs_dims, eval_blocks, num_sms, cs, nullptr, h, fused ? 2 : 1,
                                               kernels_per_sweep, &br);
            cudaGraph_t captured = nullptr;
            e = cudaStreamEndCapture(cs, &captured);
            if (e == cudaSuccess && le != cudaSuccess) e = le;
        }
    }
    if (cs) cudaStreamDestroy(cs);
    if (e != cudaSuccess) {
        cudaGraphDestroy(g);
        return e;
    }
    *out = g;
    return cudaSuccess;
}

cudaError_t launch_admit(const SweepArgs &a, const double *d_lo, const double *d_hi, const int32_t *d_slot,
                         const int32_t *d_depth, int count, int n_max, cudaStream_t st) {
    k_admit<<<1, 256, 0, st>>>(a, d_lo, d_hi, d_slot, d_depth, count, n_max);
    return cudaGetLastError();
}

// blockIdx.x: the system (see PackDesc), blockIdx.y: which of its rows, so that one system with
// many results is packed by many blocks: 2.0e5 boxes of 4 variables come to the host, sorted, in 45.3 ms
// (47.6 with a block per system and a division per element).  Many systems' results leave in
// one copy, where four copies and a wait per system took 4 of the 14 ms of a 96-system call.
__global__ void k_pack_results(DevOut o, const PackDesc *desc, PackDesc one, double *dst) {
    const PackDesc d = desc ? desc[blockIdx.x] : one;
    double *lo = dst + d.off, *hi = lo + d.n * d.count;
    int32_t *flags = reinterpret_cast<int32_t *>(hi + d.n * d.count), *depth = flags + d.count;
    for (int64_t k = (int64_t)blockIdx.y * blockDim.x + threadIdx.x; k < d.count; k += (int64_t)gridDim.y * blockDim.x) {
        for (int64_t j = 0; j < d.n; j++) {
            const int64_t at = j * o.cap + d.base + k;
            lo[j * d.count + k] = o.lo[at];
            hi[j * d.count + k] = o.hi[at];
        }
        flags[k] = o.flags[d.base + k];
        depth[k] = o.depth[d.base + k];
    }
}

cudaError_t launch_pack_results(const DevOut &o, const PackDesc *desc, PackDesc one, int n_sys, int64_t most, double *dst,
                                cudaStream_t st) {
    const int64_t rows = (most + 255) / 256;
    k_pack_results<<<dim3((unsigned)n_sys, (unsigned)(rows < 1 ? 1 : rows > 64 ? 64 : rows)), 256, 0, st>>>(o, desc, one, dst);
    return cudaGetLastError();
}

cudaError_t launch_cancel_regions(const SweepArgs &a, const int32_t *d_cancel, cudaStream_t st) {
    k_cancel_regions<<<1, 1024, 0, st>>>(a, d_cancel);
    return cudaGetLastError();
}

cudaError_t launch_seed_roots(const SweepArgs &a, const double *d_box_lo, const double *d_box_hi,
                              const int32_t *d_root_depth, int n_sys, int n_max, cudaStream_t st) {
    int blocks = (n_sys + 255) / 256;
    if (blocks < 1) blocks = 1;
    k_seed_roots<<<blocks, 256, 0, st>>>(a, d_box_lo, d_box_hi, d_root_depth, n_sys, n_max);
    return cudaGetLastError();
}

}  // namespace ivs
