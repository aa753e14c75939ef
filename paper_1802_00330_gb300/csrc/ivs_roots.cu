// ivs_roots.cu -- root isolation and Algorithm 5 backtracking on the GPU.
//
// Section 3.4: the last round leaves many tiny configurations; merging them isolates the
// real roots.  Two device pipelines over a solve's accepted boxes (a plan's result region,
// or host rows copied in), with the same results as the host versions in ivs_clusters.cu:
//
// backtracking (Algorithm 5, read on the dyadic grid of the initial box): per box the cell
//   ranges of level L per coordinate (t = (x - d_lo) / w in round to nearest, cells
//   floor(t_lo) .. ceil(t_hi) - 1, swapped when they cross, clamped), a scan of the cell
//   counts, one 128-bit key per (box, cell) (coordinate 0 in the most significant bits),
//   a bitonic sort, unique -> the distinct cells; then the groups (connected components of
//   cells whose indices differ by at most 1 in every coordinate): in key order every
//   neighbour of a cell with a larger key has coordinate 0 at most one above, so each
//   cell tests the cells after it up to that bound (binary search) and unites with the
//   touching ones (lock-free union-find, roots = smallest index).
// clusters (connected components of touching boxes): boxes sorted by (lo_0, index); a box
//   can only touch the later boxes whose lo_0 <= its hi_0 (binary search), so each tests
//   those; clusters are numbered in the order of their first box (a scan over the
//   "first box of its component" flags) and their hulls taken with atomic min / max.
//
// Every loop that waits on other threads' progress (the union-find retry loop) has an
// iteration limit after which the kernel sets an error flag and returns.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <vector>

#include "../../include/ivsolve.h"
#include "ivs_hostcore.h"

using namespace ivs;
using namespace ivs::host;

// the plan's device-resident result region of one system (ivs_host.cu)
int plan_result_view(ivs_plan *p, int32_t s, const double **lo, const double **hi, int64_t *count, int64_t *stride,
                     int *n, const double **box_lo, const double **box_hi, cudaStream_t *st, int *device);

namespace {

constexpr double kMaxPairTests = 4e9;
constexpr int kUfIters = 1 << 20;   // retries of one union before the kernel gives up

// A set of boxes in device memory: coordinate j of box i at lo[i * rs + j * cs].
struct BoxView {
    const double *lo, *hi;
    int64_t rs, cs, count;
    int n;
    __device__ __forceinline__ double l(int64_t i, int j) const { return lo[i * rs + (int64_t)j * cs]; }
    __device__ __forceinline__ double h(int64_t i, int j) const { return hi[i * rs + (int64_t)j * cs]; }
};

struct Key {
    unsigned long long a, b;   // a: high word
};
__device__ __forceinline__ bool key_less(Key x, Key y) { return x.a < y.a || (x.a == y.a && x.b < y.b); }

// Device memory of one call, given back at its end.  What a stage is known to need is reserved
// in one piece of that size, and its buffers are cut from it; a buffer that does not fit takes
// an allocation of its own.  An allocation and its release cost 55 us when the driver has to map
// memory, a few us when it holds a part of 2 MB that it can cut, so a small set must ask for
// little and a large one seldom: components and cells of 2e3 boxes of 2 variables 0.87 ms with a dozen
// buffers of their own, 0.98 with blocks of 16 MB, 0.82 with these pieces; 2e4 of 5 1.66, 1.31 and
// 1.22; 2e5 of 9 21.4, 9.4 and 8.8.
struct Scratch {
    std::vector<void *> v;
    char *cur = nullptr;
    size_t left = 0;
    ~Scratch() {
        for (void *p : v) cudaFree(p);
    }
    static size_t up(size_t bytes) { return (std::max<size_t>(bytes, 1) + 255) & ~(size_t)255; }
    cudaError_t piece(void **p, size_t bytes) {
        *p = nullptr;
        v.reserve(v.size() + 1);
        cudaError_t e = cudaMalloc(p, bytes);
        if (e == cudaSuccess) v.push_back(*p);
        return e;
    }
    // (when the piece cannot be had the buffers are allocated one by one)
    void reserve(size_t bytes) {
        void *q;
        if (bytes <= left) return;
        if (piece(&q, bytes) == cudaSuccess) {
            cur = (char *)q;
            left = bytes;
        } else {
            cudaGetLastError();
        }
    }
    template <class T>
    cudaError_t get(T **p, size_t n) {
        const size_t bytes = up(n * sizeof(T));
        if (bytes <= left) {
            *p = (T *)cur;
            cur += bytes;
            left -= bytes;
            return cudaSuccess;
        }
        void *q;
        cudaError_t e = piece(&q, bytes);
        *p = (T *)q;
        return e;
    }
};

// ---- scan (exclusive, int64) -------------------------------------------------------------
constexpr int kScanThreads = 1024;

__global__ void k_scan_blocks(const int64_t *in, int64_t *out, int64_t count, int64_t *sums) {
    __shared__ int64_t s[kScanThreads];
    const int t = threadIdx.x;
    const int64_t i = (int64_t)blockIdx.x * kScanThreads + t;
    const int64_t v = i < count ? in[i] : 0;
    s[t] = v;
    __syncthreads();
    for (int off = 1; off < kScanThreads; off <<= 1) {
        const int64_t x = t >= off ? s[t - off] : 0;
        __syncthreads();
        s[t] += x;
        __syncthreads();
    }
    if (i < count) out[i] = s[t] - v;
    if (t == kScanThreads - 1) sums[blockIdx.x] = s[t];
}

__global__ void k_scan_add(int64_t *out, int64_t count, const int64_t *offs) {
    const int64_t i = (int64_t)blockIdx.x * kScanThreads + threadIdx.x;
    if (i < count) out[i] += offs[blockIdx.x];
}

// exclusive scan of count values; *total (device) receives their sum
cudaError_t scan_exclusive(const int64_t *in, int64_t *out, int64_t count, int64_t *total, cudaStream_t st,
                           Scratch &scratch) {
    if (count <= 0) return cudaMemsetAsync(total, 0, sizeof(int64_t), st);
    const int64_t nb = (count + kScanThreads - 1) / kScanThreads;
    int64_t *sums = nullptr, *offs = nullptr;
    cudaError_t e = scratch.get(&sums, (size_t)nb);
    if (e == cudaSuccess) e = scratch.get(&offs, (size_t)nb);
    if (e != cudaSuccess) return e;
    k_scan_blocks<<<(unsigned)nb, kScanThreads, 0, st>>>(in, out, count, sums);
    if (nb == 1) return cudaMemcpyAsync(total, sums, sizeof(int64_t), cudaMemcpyDeviceToDevice, st);
    e = scan_exclusive(sums, offs, nb, total, st, scratch);
    if (e != cudaSuccess) return e;
    k_scan_add<<<(unsigned)nb, kScanThreads, 0, st>>>(out, count, offs);
    return cudaGetLastError();
}

// what a scan takes from its scratch
size_t scan_bytes(int64_t count) {
    size_t bytes = 0;
    while (count > 1) {
        count = (count + kScanThreads - 1) / kScanThreads;
        bytes += 2 * Scratch::up((size_t)count * sizeof(int64_t));
    }
    return bytes;
}

// ---- bitonic sort of 128-bit keys ----------------------------------------------------------
// 2^18 keys: 0.44 -> 0.31 ms a sort.  Every thread of a step holds a pair (element index from
// the pair index), blocks of 1024 keys sort in shared memory (2048 made
// sets of a few thousand boxes 0.1 ms slower), and a global pass does two
// steps on four keys per thread, so a merge of 2^18 keys reads the keys 4 times, not 8.
constexpr int kSortBlock = 1024;     // elements per shared-memory stage
constexpr int kSortThreads = kSortBlock / 2;

// element x of a pair / quad with its partner at distance j: bit log2(j) of the index is 0
__device__ __forceinline__ int64_t pair_low(int64_t p, int64_t j) { return 2 * p - (p & (j - 1)); }
__device__ __forceinline__ void order_keys(Key &x, Key &y, bool up) {
    if (up ? key_less(y, x) : key_less(x, y)) {
        const Key t = x;
        x = y;
        y = t;
    }
}

__global__ void k_bitonic_global(Key *k, int64_t N, int64_t j, int64_t kk) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= N / 2) return;
    const int64_t i = pair_low(p, j);
    Key x = k[i], y = k[i + j];
    order_keys(x, y, (i & kk) == 0);
    k[i] = x;
    k[i + j] = y;
}

// steps j and j / 2 of merge size kk
__global__ void k_bitonic_global2(Key *k, int64_t N, int64_t j, int64_t kk) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= N / 4) return;
    const int64_t h = j / 2, i = pair_low(pair_low(p, h), j);
    const bool up = (i & kk) == 0;
    Key a = k[i], b = k[i + h], c = k[i + j], d = k[i + j + h];
    order_keys(a, c, up);
    order_keys(b, d, up);
    order_keys(a, b, up);
    order_keys(c, d, up);
    k[i] = a;
    k[i + h] = b;
    k[i + j] = c;
    k[i + j + h] = d;
}

// stages j = jmax .. 1 of merge size kk inside blocks of kSortBlock elements; with
// kk = 0 the whole sort of every block (kk = 2 .. kSortBlock)
__global__ void __launch_bounds__(kSortThreads) k_bitonic_shared(Key *k, int64_t kk, int64_t jmax) {
    __shared__ Key s[kSortBlock];
    const int64_t base = (int64_t)blockIdx.x * kSortBlock;
    const int t = threadIdx.x;
    s[t] = k[base + t];
    s[t + kSortThreads] = k[base + t + kSortThreads];
    __syncthreads();
    const int64_t k0 = kk ? kk : 2, k1 = kk ? kk : kSortBlock;
    for (int64_t q = k0; q <= k1; q <<= 1) {
        for (int64_t j = kk ? jmax : q / 2; j > 0; j >>= 1) {
            const int i = (int)pair_low(t, j), l = i + (int)j;
            Key x = s[i], y = s[l];
            order_keys(x, y, ((base + i) & q) == 0);
            s[i] = x;
            s[l] = y;
            __syncthreads();
        }
    }
    k[base + t] = s[t];
    k[base + t + kSortThreads] = s[t + kSortThreads];
}

// sorts N keys (N a power of two >= kSortBlock) ascending
cudaError_t bitonic_sort(Key *k, int64_t N, cudaStream_t st) {
    const unsigned blocks = (unsigned)(N / kSortBlock);
    k_bitonic_shared<<<blocks, kSortThreads, 0, st>>>(k, 0, 0);
    for (int64_t kk = 2 * kSortBlock; kk <= N; kk <<= 1) {
        int64_t j = kk / 2;
        for (; j >= 2 * kSortBlock; j >>= 2)
            k_bitonic_global2<<<(unsigned)((N / 4 + 255) / 256), 256, 0, st>>>(k, N, j, kk);
        if (j >= kSortBlock) {
            k_bitonic_global<<<(unsigned)((N / 2 + 255) / 256), 256, 0, st>>>(k, N, j, kk);
            j >>= 1;
        }
        k_bitonic_shared<<<blocks, kSortThreads, 0, st>>>(k, kk, j);
    }
    return cudaGetLastError();
}

__global__ void k_fill_keys(Key *k, int64_t from, int64_t to) {
    for (int64_t i = from + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < to; i += (int64_t)gridDim.x * blockDim.x)
        k[i] = Key{~0ull, ~0ull};
}

// ---- union-find -----------------------------------------------------------------------------
// Path halving by plain stores: an item that is not a root never becomes one again, its
// parent only ever moves to an ancestor, and every ancestor is a valid parent, so racing
// stores are harmless (the intermediate pointer jumping of ECL-CC, Jaiganesh and Burtscher
// 2018).  As compare-and-swaps they queued up on the parents of a cluster's few top items.
__device__ __forceinline__ int64_t uf_load(const int64_t *par, int64_t x) {
    return (int64_t)*reinterpret_cast<const volatile long long *>(par + x);
}
__device__ __forceinline__ int64_t uf_find(int64_t *par, int64_t x) {
    int64_t p = uf_load(par, x);
    for (int it = 0; it < kUfIters; it++) {
        if (p == x) return x;
        const int64_t gp = uf_load(par, p);
        if (gp == p) return p;
        *reinterpret_cast<volatile long long *>(par + x) = (long long)gp;
        x = gp;
        p = uf_load(par, x);
    }
    return -1;
}

// the root of x without halving: k_uf_flatten's own stores must stay the last ones
__device__ __forceinline__ int64_t uf_root(const int64_t *par, int64_t x) {
    for (int it = 0; it < kUfIters; it++) {
        const int64_t p = uf_load(par, x);
        if (p == x) return x;
        x = p;
    }
    return -1;
}

// unites the sets of a and b; the root with the larger index is hooked under the smaller.
// (false: it gave up)
__device__ __forceinline__ bool uf_union(int64_t *par, int64_t a, int64_t b) {
    for (int it = 0; it < kUfIters; it++) {
        a = uf_find(par, a);
        b = uf_find(par, b);
        if (a < 0 || b < 0) return false;
        if (a == b) return true;
        if (a < b) {
            const int64_t t = a;
            a = b;
            b = t;
        }
        if (atomicCAS((unsigned long long *)&par[a], (unsigned long long)a, (unsigned long long)b) ==
            (unsigned long long)a)
            return true;
    }
    return false;
}

__global__ void k_iota(int64_t *par, int64_t count) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x)
        par[i] = i;
}

// Unites touching items.  Items lie in sorted order, coordinate j of item p as integer keys
// [lo, hi] at key[(2 j) * count + p], key[(2 j + 1) * count + p] (order-preserving images of
// a box's ends; a cell's index c and c + 1); item p may only touch the items p + 1 .. end[p] - 1.
// A block takes 32 items, one per lane of every warp, and its warps share the range that
// follows them: an item of the range is read by a warp once (a broadcast) and tested against
// 32, coordinate 1 first.  Integer compares: FP64 ones would run at 1/64 of their rate.
// id: what the union-find calls item p (nullptr: p).  (A warp per item, its lanes gathering
// the candidates' rows through the sorted keys, took 6.3 ms for 2e5 boxes of 6 coordinates,
// and 1.1 ms for their 8.9e4 cells; this 1.4 and 0.47.)
// Touching pairs queue up in shared memory and are united 32 at a time: a union is a chain
// of dependent loads, which the lanes that found a pair would go through on their own.
constexpr int kUniteWarps = 8;
__device__ __forceinline__ void unite_pair(int64_t *par, const Key *id, longlong2 w, int *err) {
    if (!uf_union(par, id ? (int64_t)id[w.x].b : w.x, id ? (int64_t)id[w.y].b : w.y)) atomicExch(err, 1);
}
template <class K, int N>
__global__ void __launch_bounds__(kUniteWarps * 32) k_unite(const K *key, int64_t count, const int64_t *end, const Key *id,
                                                            int64_t *par, int *err) {
    __shared__ longlong2 s_pair[kUniteWarps][64];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int64_t p0 = (int64_t)blockIdx.x * 32; p0 < count; p0 += (int64_t)gridDim.x * 32) {
        const int64_t p = p0 + lane;
        const bool on = p < count;
        K l[N], h[N];
#pragma unroll
        for (int j = 0; j < N; j++) {
            l[j] = on ? key[(int64_t)(2 * j) * count + p] : K(0);
            h[j] = on ? key[(int64_t)(2 * j + 1) * count + p] : K(0);
        }
        const int64_t stop = on ? end[p] : 0;
        int64_t last = stop;
        for (int o = 16; o > 0; o >>= 1) {
            const int64_t x = __shfl_xor_sync(0xFFFFFFFFu, last, o);
            last = x > last ? x : last;
        }
        constexpr int J = N > 1 ? 1 : 0;   // the coordinate tested first
        const K *kl = key + (int64_t)(2 * J) * count, *kh = key + (int64_t)(2 * J + 1) * count;
        int held = 0;   // pairs in the warp's queue
        for (int64_t q = p0 + 1 + blockIdx.y * kUniteWarps + warp; q < last; q += kUniteWarps * gridDim.y) {
            bool touch = kl[q] <= h[J] && l[J] <= kh[q] && q > p && q < stop;
            if (!__any_sync(0xFFFFFFFFu, touch)) continue;
#pragma unroll
            for (int j = 0; j < N; j++)
                touch = touch && key[(int64_t)(2 * j) * count + q] <= h[j] && l[j] <= key[(int64_t)(2 * j + 1) * count + q];
            const unsigned bal = __ballot_sync(0xFFFFFFFFu, touch);
            if (!bal) continue;
            if (touch) s_pair[warp][held + __popc(bal & ((1u << lane) - 1u))] = make_longlong2(p, q);
            held += __popc(bal);
            __syncwarp();
            if (held >= 32) {
                const longlong2 w = s_pair[warp][held - 32 + lane];
                held -= 32;
                unite_pair(par, id, w, err);
                __syncwarp();
            }
        }
        if (lane < held) unite_pair(par, id, s_pair[warp][lane], err);
        __syncwarp();
    }
}
template <class K>
cudaError_t launch_unite(int n, const K *key, int64_t count, const int64_t *end, const Key *id, int64_t *par, int *err,
                         cudaStream_t st) {
    // small sets: the ranges are split over more blocks, so that the chip has a few per SM
    const unsigned gx = (unsigned)std::max<int64_t>(1, std::min<int64_t>((count + 31) / 32, 1 << 20));
    const dim3 grid(gx, (unsigned)std::max<int64_t>(1, std::min<int64_t>(32, 2432 / (int64_t)gx)));
    switch (n) {
#define IVS_UNITE(N) case N: k_unite<K, N><<<grid, kUniteWarps * 32, 0, st>>>(key, count, end, id, par, err); break;
        IVS_UNITE(1) IVS_UNITE(2) IVS_UNITE(3) IVS_UNITE(4) IVS_UNITE(5) IVS_UNITE(6) IVS_UNITE(7) IVS_UNITE(8)
        IVS_UNITE(9) IVS_UNITE(10) IVS_UNITE(11) IVS_UNITE(12) IVS_UNITE(13) IVS_UNITE(14) IVS_UNITE(15) IVS_UNITE(16)
#undef IVS_UNITE
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

// full compression; roots[i] = 1 when i is a root
__global__ void k_uf_flatten(int64_t *par, int64_t count, int64_t *is_root, int *err) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = uf_root(par, i);
        if (r < 0) {
            atomicExch(err, 1);
            continue;
        }
        par[i] = r;
        if (is_root) is_root[i] = r == i ? 1 : 0;
    }
}

// ---- backtracking kernels -------------------------------------------------------------------
struct Grid {
    double d_lo[kMaxVars], w[kMaxVars];
    int64_t side;
    int level, bits;   // bits = n * level (<= 127)
};

// cell index range of box i in coordinate j (the host rule, operation for operation)
__device__ __forceinline__ void cell_range(const BoxView &v, const Grid &g, int64_t i, int j, int32_t &a, int32_t &b) {
    const double tl = __ddiv_rn(__dsub_rn(v.l(i, j), g.d_lo[j]), g.w[j]);
    const double th = __ddiv_rn(__dsub_rn(v.h(i, j), g.d_lo[j]), g.w[j]);
    const double fa = floor(tl), fb = __dsub_rn(ceil(th), 1.0);
    double x = fa < fb ? fa : fb, y = fa < fb ? fb : fa;
    const double top = (double)(g.side - 1);
    if (x < 0) x = 0;
    if (y > top) y = top;
    if (y < x) y = x;
    if (x > top) x = y = top;
    a = (int32_t)x;
    b = (int32_t)y;
}

// the cells per box; the ranges stay for k_bt_emit (coordinate j of box i at j * count + i):
// their divisions are the FP64 part of both
__global__ void k_bt_count(BoxView v, Grid g, int64_t max_cells, int64_t *m, int2 *range, int *over) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < v.count; i += (int64_t)gridDim.x * blockDim.x) {
        int64_t c = 1;
        for (int j = 0; j < v.n; j++) {
            int32_t a, b;
            cell_range(v, g, i, j, a, b);
            range[(int64_t)j * v.count + i] = make_int2(a, b);
            c *= (int64_t)(b - a + 1);
            if (c > max_cells) {
                atomicExch(over, 1);
                c = 0;
                break;
            }
        }
        m[i] = c;
    }
}

// places field value c of coordinate j into the key (coordinate 0 most significant)
__device__ __forceinline__ void key_put(Key &k, const Grid &g, int n, int j, uint64_t c) {
    const int lsb = (n - 1 - j) * g.level;   // bit position of the field's lowest bit
    if (lsb >= 64) {
        k.a |= c << (lsb - 64);
    } else {
        k.b |= c << lsb;
        if (lsb + g.level > 64 && lsb > 0) k.a |= c >> (64 - lsb);
    }
}
__device__ __forceinline__ int32_t key_get(Key k, const Grid &g, int n, int j) {
    const int lsb = (n - 1 - j) * g.level;
    const uint64_t mask = (g.level >= 64) ? ~0ull : ((1ull << g.level) - 1ull);
    uint64_t v;
    if (lsb >= 64) v = k.a >> (lsb - 64);
    else if (lsb == 0) v = k.b;
    else v = (k.b >> lsb) | (k.a << (64 - lsb));
    return (int32_t)(v & mask);
}

__global__ void k_bt_emit(BoxView v, Grid g, const int64_t *offs, const int2 *range, Key *keys) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < v.count; i += (int64_t)gridDim.x * blockDim.x) {
        int32_t a[kMaxVars], b[kMaxVars], cur[kMaxVars];
        int64_t m = 1;
        for (int j = 0; j < v.n; j++) {
            const int2 r = range[(int64_t)j * v.count + i];
            a[j] = r.x;
            b[j] = r.y;
            cur[j] = a[j];
            m *= (int64_t)(b[j] - a[j] + 1);
        }
        int64_t o = offs[i];
        for (int64_t q = 0; q < m; q++) {
            Key k{0ull, 0ull};
            for (int j = 0; j < v.n; j++) key_put(k, g, v.n, j, (uint64_t)cur[j]);
            keys[o + q] = k;
            for (int j = 0; j < v.n; j++) {   // next cell of the box's ranges
                if (cur[j] < b[j]) {
                    cur[j]++;
                    break;
                }
                cur[j] = a[j];
            }
        }
    }
}

__global__ void k_flag_distinct(const Key *k, int64_t total, int64_t *flag) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x)
        flag[i] = (i == 0 || k[i].a != k[i - 1].a || k[i].b != k[i - 1].b) ? 1 : 0;
}

__global__ void k_compact(const Key *k, int64_t total, const int64_t *flag, const int64_t *pos, Key *out) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x)
        if (flag[i]) out[pos[i]] = k[i];
}

// first position in [lo, hi) whose key is >= x
__device__ __forceinline__ int64_t lower_bound(const Key *k, int64_t lo, int64_t hi, Key x) {
    while (lo < hi) {
        const int64_t mid = lo + (hi - lo) / 2;
        if (key_less(k[mid], x)) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// the key just above every cell whose coordinate 0 is c0 + 1 (c0 + 2 in field 0, rest 0)
__device__ __forceinline__ Key field0_bound(const Grid &g, int n, int32_t c0) {
    Key k{0ull, 0ull};
    const uint64_t c = (uint64_t)c0 + 2ull;
    if (c >= (1ull << g.level)) return Key{~0ull, ~0ull};
    key_put(k, g, n, 0, c);
    return k;
}

// candidates of each distinct cell: the cells after it up to coordinate 0 + 1
__global__ void k_bt_ranges(const Key *u, int64_t d, Grid g, int n, int64_t *end, int64_t *work) {
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < d; p += (int64_t)gridDim.x * blockDim.x) {
        const int32_t c0 = key_get(u[p], g, n, 0);
        const int64_t e = lower_bound(u, p + 1, d, field0_bound(g, n, c0));
        end[p] = e;
        work[p] = e - p - 1;
    }
}

// the cells' indices as k_unite's keys: cells touch when their indices differ by <= 1
// everywhere, i.e. when the closed intervals [c, c + 1] meet
__global__ void k_bt_planes(const Key *u, int64_t d, Grid g, int n, int32_t *key) {
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < d; p += (int64_t)gridDim.x * blockDim.x) {
        const Key k = u[p];
        for (int j = 0; j < n; j++) {
            const int32_t c = key_get(k, g, n, j);
            key[(int64_t)(2 * j) * d + p] = c;
            key[(int64_t)(2 * j + 1) * d + p] = c + 1;
        }
    }
}

__global__ void k_sum(const int64_t *v, int64_t count, unsigned long long *out) {
    unsigned long long s = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x)
        s += (unsigned long long)v[i];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xFFFFFFFFu, s, o);
    if ((threadIdx.x & 31) == 0 && s) atomicAdd(out, s);
}

// ---- cluster kernels ---------------------------------------------------------------------------
// ordered integer image of a double (numeric order; -0 and +0 map to the same value)
__device__ __forceinline__ unsigned long long dkey(double x) {
    if (x == 0.0) x = 0.0;
    const unsigned long long u = (unsigned long long)__double_as_longlong(x);
    return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}
__device__ __forceinline__ double dkey_inv(unsigned long long k) {
    const unsigned long long u = (k >> 63) ? (k & 0x7FFFFFFFFFFFFFFFull) : ~k;
    return __longlong_as_double((long long)u);
}

__global__ void k_cl_keys(BoxView v, Key *k) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < v.count; i += (int64_t)gridDim.x * blockDim.x)
        k[i] = Key{dkey(v.l(i, 0)), (unsigned long long)i};
}

// candidates of the box at sorted position p: the later positions with lo_0 <= its hi_0
__global__ void k_cl_ranges(BoxView v, const Key *k, int64_t *end, int64_t *work) {
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < v.count; p += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = (int64_t)k[p].b;
        const Key bound{dkey(v.h(i, 0)), ~0ull};
        int64_t lo = p + 1, hi = v.count;   // first position with key > (hi_0, any index)
        while (lo < hi) {
            const int64_t mid = lo + (hi - lo) / 2;
            if (!key_less(bound, k[mid])) lo = mid + 1;
            else hi = mid;
        }
        end[p] = lo;
        work[p] = lo - p - 1;
    }
}

// the boxes' ends in sorted order as k_unite's keys; a NaN end compares with nothing
__global__ void k_cl_planes(BoxView v, const Key *k, unsigned long long *key) {
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < v.count; p += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = (int64_t)k[p].b;
        for (int j = 0; j < v.n; j++) {
            const double l = v.l(i, j), h = v.h(i, j);
            key[(int64_t)(2 * j) * v.count + p] = isnan(l) ? ~0ull : dkey(l);
            key[(int64_t)(2 * j + 1) * v.count + p] = isnan(h) ? 0ull : dkey(h);
        }
    }
}

// first[i] = 1 when box i is the smallest index of its component (par[i] is its root, and
// the root is the smallest index: unions hook larger roots under smaller ones)
__global__ void k_cl_first(const int64_t *par, int64_t count, int64_t *first) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x)
        first[i] = par[i] == i ? 1 : 0;
}

__global__ void k_cl_label(BoxView v, const int64_t *par, const int64_t *num, int64_t *label, int64_t cl_cap,
                           unsigned long long *hlo, unsigned long long *hhi) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < v.count; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t c = num[par[i]];
        label[i] = c;
        if (c < cl_cap)
            for (int j = 0; j < v.n; j++) {
                atomicMin(&hlo[c * v.n + j], dkey(v.l(i, j)));
                atomicMax(&hhi[c * v.n + j], dkey(v.h(i, j)));
            }
    }
}

__global__ void k_cl_hull_init(unsigned long long *hlo, unsigned long long *hhi, int64_t m) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
        hlo[i] = ~0ull;
        hhi[i] = 0ull;
    }
}

__global__ void k_cl_hull_out(const unsigned long long *hlo, const unsigned long long *hhi, int64_t m, double *lo,
                              double *hi) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
        lo[i] = dkey_inv(hlo[i]);
        hi[i] = dkey_inv(hhi[i]);
    }
}

// ---- host drivers -----------------------------------------------------------------------------
unsigned grid_for(int64_t n) { return (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 152 * 32)); }

#define RT_TRY(x)                                                                                   \
    do {                                                                                            \
        cudaError_t e_ = (x);                                                                       \
        if (e_ != cudaSuccess) return fail(IVS_ERR_CUDA, std::string(#x) + ": " + cudaGetErrorString(e_)); \
    } while (0)

int64_t pow2_at_least(int64_t x) {
    int64_t p = kSortBlock;
    while (p < x) p <<= 1;
    return p;
}

// bytes of the rows of a set in device memory (upload_rows)
size_t rows_bytes(int n, int64_t count) { return 2 * Scratch::up((size_t)count * n * sizeof(double)); }

// what backtrack_device needs per box
size_t box_cells_bytes(int n, int64_t count) {
    const size_t c = (size_t)count;
    return 2 * Scratch::up(8 * c) + Scratch::up(8 * c * n) + scan_bytes(count) + 1024;
}

int backtrack_device(Scratch &sc, const BoxView &v, const double *box_lo, const double *box_hi, int32_t level,
                     int64_t max_cells, int64_t *n_cells, int64_t *n_groups, cudaStream_t st) {
    *n_cells = 0;
    if (n_groups) *n_groups = 0;
    const int n = v.n;
    if (level < 0 || level > 30) return fail(IVS_ERR_INVALID, "ivs_backtrack: level must be in 0..30");
    if ((int64_t)n * level > 127) return fail(IVS_ERR_INVALID, "backtracking on the GPU: n_vars * level must be <= 127");
    Grid g{};
    for (int j = 0; j < n; j++) {
        if (!(box_hi[j] > box_lo[j])) return fail(IVS_ERR_INVALID, "ivs_backtrack: empty initial box");
        g.d_lo[j] = box_lo[j];
        g.w[j] = std::ldexp(box_hi[j] - box_lo[j], -level);
    }
    g.side = (int64_t)1 << level;
    g.level = level;
    g.bits = n * level;
    if (v.count == 0) return IVS_OK;
    sc.reserve(box_cells_bytes(n, v.count));
    int64_t *m = nullptr, *offs = nullptr, *tot = nullptr;
    int *flags = nullptr;   // [0] over budget, [1] union-find gave up
    RT_TRY(sc.get(&m, v.count));
    RT_TRY(sc.get(&offs, v.count));
    RT_TRY(sc.get(&tot, 2));
    RT_TRY(sc.get(&flags, 2));
    int2 *range = nullptr;
    RT_TRY(sc.get(&range, (size_t)v.count * n));
    RT_TRY(cudaMemsetAsync(flags, 0, 2 * sizeof(int), st));
    k_bt_count<<<grid_for(v.count), 256, 0, st>>>(v, g, max_cells, m, range, flags);
    RT_TRY(cudaGetLastError());
    RT_TRY(scan_exclusive(m, offs, v.count, tot, st, sc));
    int64_t total = 0;
    int hf[2] = {0, 0};
    RT_TRY(cudaMemcpyAsync(&total, tot, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
    RT_TRY(cudaMemcpyAsync(hf, flags, sizeof(hf), cudaMemcpyDeviceToHost, st));
    RT_TRY(cudaStreamSynchronize(st));
    if (hf[0] || total > max_cells) return fail(IVS_ERR_BUDGET, "ivs_backtrack: too many cells");
    const int64_t N = pow2_at_least(total);
    Key *keys = nullptr, *uniq = nullptr;
    // the cells' keys, distinct cells, and what joins the cells into groups: in the same piece when it is
    // small, else once the number of distinct cells is known
    const size_t key_bytes = Scratch::up(16 * N) + Scratch::up(16 * total) + 2 * Scratch::up(8 * total) + scan_bytes(total);
    auto group_bytes = [&](int64_t cells) { return 3 * Scratch::up(8 * cells) + Scratch::up(8 * cells * n) + 256; };
    const bool together = n_groups && group_bytes(total) <= ((size_t)16 << 20);
    sc.reserve(key_bytes + (together ? group_bytes(total) : 0));
    int64_t *fl = nullptr, *pos = nullptr;
    RT_TRY(sc.get(&keys, N));
    k_bt_emit<<<grid_for(v.count), 128, 0, st>>>(v, g, offs, range, keys);
    k_fill_keys<<<grid_for(N - total), 256, 0, st>>>(keys, total, N);
    RT_TRY(cudaGetLastError());
    RT_TRY(bitonic_sort(keys, N, st));
    RT_TRY(sc.get(&fl, total));
    RT_TRY(sc.get(&pos, total));
    k_flag_distinct<<<grid_for(total), 256, 0, st>>>(keys, total, fl);
    RT_TRY(scan_exclusive(fl, pos, total, tot, st, sc));
    int64_t d = 0;
    RT_TRY(cudaMemcpyAsync(&d, tot, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
    RT_TRY(sc.get(&uniq, total));
    k_compact<<<grid_for(total), 256, 0, st>>>(keys, total, fl, pos, uniq);
    RT_TRY(cudaGetLastError());
    RT_TRY(cudaStreamSynchronize(st));
    *n_cells = d;
    if (!n_groups || d == 0) return IVS_OK;
    if (!together) sc.reserve(group_bytes(d));
    int64_t *end = nullptr, *work = nullptr, *par = nullptr;
    unsigned long long *wsum = nullptr;
    RT_TRY(sc.get(&end, d));
    RT_TRY(sc.get(&work, d));
    RT_TRY(sc.get(&par, d));
    RT_TRY(sc.get(&wsum, 1));
    RT_TRY(cudaMemsetAsync(wsum, 0, sizeof(unsigned long long), st));
    k_bt_ranges<<<grid_for(d), 256, 0, st>>>(uniq, d, g, n, end, work);
    k_sum<<<grid_for(d), 256, 0, st>>>(work, d, wsum);
    unsigned long long hw = 0;
    RT_TRY(cudaMemcpyAsync(&hw, wsum, sizeof(hw), cudaMemcpyDeviceToHost, st));
    RT_TRY(cudaStreamSynchronize(st));
    if ((double)hw > kMaxPairTests) return fail(IVS_ERR_BUDGET, "ivs_backtrack: too many cells to group");
    int32_t *key = nullptr;
    RT_TRY(sc.get(&key, (size_t)d * 2 * n));
    k_iota<<<grid_for(d), 256, 0, st>>>(par, d);
    k_bt_planes<<<grid_for(d), 256, 0, st>>>(uniq, d, g, n, key);
    RT_TRY(launch_unite<int32_t>(n, key, d, end, nullptr, par, flags + 1, st));
    int64_t *root = work;   // reused
    k_uf_flatten<<<grid_for(d), 256, 0, st>>>(par, d, root, flags + 1);
    RT_TRY(cudaGetLastError());
    RT_TRY(cudaMemsetAsync(wsum, 0, sizeof(unsigned long long), st));
    k_sum<<<grid_for(d), 256, 0, st>>>(root, d, wsum);
    RT_TRY(cudaMemcpyAsync(&hw, wsum, sizeof(hw), cudaMemcpyDeviceToHost, st));
    RT_TRY(cudaMemcpyAsync(hf, flags, sizeof(hf), cudaMemcpyDeviceToHost, st));
    RT_TRY(cudaStreamSynchronize(st));
    if (hf[1]) return fail(IVS_ERR_CUDA, "ivs_backtrack: union-find did not settle");
    *n_groups = (int64_t)hw;
    return IVS_OK;
}

// what clusters_device needs for count boxes (more when it returns many hulls)
size_t clusters_bytes(int n, int64_t count) {
    const size_t c = (size_t)count;
    return Scratch::up(16 * (size_t)pow2_at_least(count)) + 5 * Scratch::up(8 * c) + Scratch::up(16 * c * n) +
           scan_bytes(count) + 8192;
}

int clusters_device(Scratch &sc, const BoxView &v, int64_t *n_clusters, int64_t *label_h, double *cl_lo, double *cl_hi,
                    int64_t cl_cap, cudaStream_t st) {
    *n_clusters = 0;
    if (v.count == 0) return IVS_OK;
    sc.reserve(clusters_bytes(v.n, v.count));
    const int64_t N = pow2_at_least(v.count);
    Key *keys = nullptr;
    int64_t *end = nullptr, *work = nullptr, *par = nullptr, *num = nullptr, *tot = nullptr, *label = nullptr;
    unsigned long long *wsum = nullptr, *hlo = nullptr, *hhi = nullptr;
    int *err = nullptr;
    RT_TRY(sc.get(&keys, N));
    RT_TRY(sc.get(&end, v.count));
    RT_TRY(sc.get(&work, v.count));
    RT_TRY(sc.get(&par, v.count));
    RT_TRY(sc.get(&wsum, 1));
    RT_TRY(sc.get(&err, 1));
    RT_TRY(cudaMemsetAsync(err, 0, sizeof(int), st));
    RT_TRY(cudaMemsetAsync(wsum, 0, sizeof(unsigned long long), st));
    k_cl_keys<<<grid_for(v.count), 256, 0, st>>>(v, keys);
    k_fill_keys<<<grid_for(N - v.count), 256, 0, st>>>(keys, v.count, N);
    RT_TRY(cudaGetLastError());
    RT_TRY(bitonic_sort(keys, N, st));
    k_cl_ranges<<<grid_for(v.count), 256, 0, st>>>(v, keys, end, work);
    k_sum<<<grid_for(v.count), 256, 0, st>>>(work, v.count, wsum);
    unsigned long long hw = 0;
    RT_TRY(cudaMemcpyAsync(&hw, wsum, sizeof(hw), cudaMemcpyDeviceToHost, st));
    RT_TRY(cudaStreamSynchronize(st));
    if ((double)hw > kMaxPairTests) return fail(IVS_ERR_BUDGET, "ivs_clusters: too many overlapping boxes");
    unsigned long long *key = nullptr;
    RT_TRY(sc.get(&key, (size_t)v.count * 2 * v.n));
    k_iota<<<grid_for(v.count), 256, 0, st>>>(par, v.count);
    k_cl_planes<<<grid_for(v.count), 256, 0, st>>>(v, keys, key);
    RT_TRY(launch_unite<unsigned long long>(v.n, key, v.count, end, keys, par, err, st));
    k_uf_flatten<<<grid_for(v.count), 256, 0, st>>>(par, v.count, nullptr, err);
    // clusters numbered in the order of their first box
    RT_TRY(sc.get(&num, v.count));
    RT_TRY(sc.get(&tot, 1));
    k_cl_first<<<grid_for(v.count), 256, 0, st>>>(par, v.count, work);
    RT_TRY(scan_exclusive(work, num, v.count, tot, st, sc));
    int64_t nc = 0;
    int he = 0;
    RT_TRY(cudaMemcpyAsync(&nc, tot, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
    RT_TRY(cudaMemcpyAsync(&he, err, sizeof(int), cudaMemcpyDeviceToHost, st));
    RT_TRY(cudaStreamSynchronize(st));
    if (he) return fail(IVS_ERR_CUDA, "ivs_clusters: union-find did not settle");
    *n_clusters = nc;
    if (!label_h && !(cl_lo && cl_hi && cl_cap > 0)) return IVS_OK;
    const int64_t cap = (cl_lo && cl_hi) ? std::min<int64_t>(cl_cap, nc) : 0;
    RT_TRY(sc.get(&label, v.count));
    RT_TRY(sc.get(&hlo, std::max<int64_t>(cap * v.n, 1)));
    RT_TRY(sc.get(&hhi, std::max<int64_t>(cap * v.n, 1)));
    k_cl_hull_init<<<grid_for(cap * v.n), 256, 0, st>>>(hlo, hhi, cap * v.n);
    k_cl_label<<<grid_for(v.count), 256, 0, st>>>(v, par, num, label, cap, hlo, hhi);
    RT_TRY(cudaGetLastError());
    if (label_h) RT_TRY(cudaMemcpyAsync(label_h, label, (size_t)v.count * sizeof(int64_t), cudaMemcpyDeviceToHost, st));
    if (cap > 0) {
        double *dl = (double *)end, *dh = (double *)work;   // reused (count >= cap * n? not always)
        if (cap * v.n > v.count) {
            RT_TRY(sc.get(&dl, cap * v.n));
            RT_TRY(sc.get(&dh, cap * v.n));
        }
        k_cl_hull_out<<<grid_for(cap * v.n), 256, 0, st>>>(hlo, hhi, cap * v.n, dl, dh);
        RT_TRY(cudaMemcpyAsync(cl_lo, dl, (size_t)(cap * v.n) * sizeof(double), cudaMemcpyDeviceToHost, st));
        RT_TRY(cudaMemcpyAsync(cl_hi, dh, (size_t)(cap * v.n) * sizeof(double), cudaMemcpyDeviceToHost, st));
    }
    RT_TRY(cudaStreamSynchronize(st));
    return IVS_OK;
}

// host rows (count x n, row-major) copied to the device
int upload_rows(Scratch &sc, int n, int64_t count, const double *lo, const double *hi, BoxView *v, cudaStream_t st) {
    double *dl = nullptr, *dh = nullptr;
    RT_TRY(sc.get(&dl, (size_t)count * n));
    RT_TRY(sc.get(&dh, (size_t)count * n));
    if (count > 0) {
        RT_TRY(cudaMemcpyAsync(dl, lo, (size_t)count * n * sizeof(double), cudaMemcpyHostToDevice, st));
        RT_TRY(cudaMemcpyAsync(dh, hi, (size_t)count * n * sizeof(double), cudaMemcpyHostToDevice, st));
    }
    *v = BoxView{dl, dh, n, 1, count, n};
    return IVS_OK;
}

}  // namespace

extern "C" {

int ivs_clusters_gpu(int32_t n_vars, int64_t count, const double *lo, const double *hi, int64_t *n_clusters,
                     int64_t *label, double *cl_lo, double *cl_hi, int64_t cl_cap, int32_t device) {
    if (!n_clusters || n_vars <= 0 || n_vars > kMaxVars || count < 0 || (count > 0 && (!lo || !hi)))
        return fail(IVS_ERR_INVALID, "ivs_clusters_gpu: bad arguments");
    *n_clusters = 0;
    RT_TRY(cudaSetDevice(device));
    cudaStream_t st = nullptr;
    RT_TRY(cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking));
    int rc;
    {
        Scratch sc;
        BoxView v{};
        if (count > 0) sc.reserve(rows_bytes(n_vars, count) + clusters_bytes(n_vars, count));
        rc = upload_rows(sc, n_vars, count, lo, hi, &v, st);
        if (rc == IVS_OK) rc = clusters_device(sc, v, n_clusters, label, cl_lo, cl_hi, cl_cap, st);
        cudaStreamSynchronize(st);
    }
    cudaStreamDestroy(st);
    return rc;
}

int ivs_backtrack_gpu(int32_t n_vars, int64_t count, const double *lo, const double *hi, const double *box_lo,
                      const double *box_hi, int32_t level, int64_t max_cells, int64_t *n_cells, int64_t *n_groups,
                      int32_t device) {
    if (!n_cells || n_vars <= 0 || n_vars > kMaxVars || count < 0 || !box_lo || !box_hi ||
        (count > 0 && (!lo || !hi)))
        return fail(IVS_ERR_INVALID, "ivs_backtrack_gpu: bad arguments");
    *n_cells = 0;
    if (n_groups) *n_groups = 0;
    RT_TRY(cudaSetDevice(device));
    cudaStream_t st = nullptr;
    RT_TRY(cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking));
    int rc;
    {
        Scratch sc;
        BoxView v{};
        if (count > 0) sc.reserve(rows_bytes(n_vars, count) + box_cells_bytes(n_vars, count));
        rc = upload_rows(sc, n_vars, count, lo, hi, &v, st);
        if (rc == IVS_OK) rc = backtrack_device(sc, v, box_lo, box_hi, level, max_cells, n_cells, n_groups, st);
        cudaStreamSynchronize(st);
    }
    cudaStreamDestroy(st);
    return rc;
}

int ivs_plan_backtrack(ivs_plan *p, int32_t s, int32_t level, int64_t max_cells, int64_t *n_cells,
                       int64_t *n_groups) {
    if (!p || !n_cells) return fail(IVS_ERR_INVALID, "ivs_plan_backtrack: bad arguments");
    const double *lo, *hi, *blo, *bhi;
    int64_t count, stride;
    int n, dev;
    cudaStream_t st;
    int rc = plan_result_view(p, s, &lo, &hi, &count, &stride, &n, &blo, &bhi, &st, &dev);
    if (rc) return rc;
    RT_TRY(cudaSetDevice(dev));
    BoxView v{lo, hi, 1, stride, count, n};
    Scratch sc;
    return backtrack_device(sc, v, blo, bhi, level, max_cells, n_cells, n_groups, st);
}

int ivs_plan_clusters(ivs_plan *p, int32_t s, int64_t *n_clusters) {
    if (!p || !n_clusters) return fail(IVS_ERR_INVALID, "ivs_plan_clusters: bad arguments");
    const double *lo, *hi, *blo, *bhi;
    int64_t count, stride;
    int n, dev;
    cudaStream_t st;
    int rc = plan_result_view(p, s, &lo, &hi, &count, &stride, &n, &blo, &bhi, &st, &dev);
    if (rc) return rc;
    RT_TRY(cudaSetDevice(dev));
    BoxView v{lo, hi, 1, stride, count, n};
    Scratch sc;
    return clusters_device(sc, v, n_clusters, nullptr, nullptr, nullptr, 0, st);
}

}  // extern "C"
