// ivs_screen.cuh -- FP32 screen of the boxes that enter the contraction: decides in FP32
// what the FP64 sweep (ivs_hs.cuh) would do with a box when it would either drop it or
// leave it as it is, and passes only the other boxes on to it.
//
// Why: FP64 runs at 1/74 of the FP32 rate here and the sweep is bound by it, while on the
// recipes' systems 70-95% of the swept boxes come out empty or unchanged.  Deciding those
// needs no FP64 bit, only a proof of what the FP64 operations give; the boxes that the
// sweep shrinks (and the few that the proof misses) still take the FP64 sweep, so every
// result is bit for bit what it was.
//
// The proof.  For a box X with centre x (its split midpoint) and half widths h_j, let
// J(X) = [C - W, C + W], A = mid J(X) and B = A^-1 as the FP64 sweep computes them (its
// Gauss-Jordan, operation by operation), f = f(x), r = B f, M = B J(X) = [BC - |B|W, BC + |B|W].
// Each of these is carried as a float value and a float radius that encloses the FP64
// value: the radius takes the float roundings, the FP64 roundings (below 2^-50 of the
// magnitudes, far below the float ones) and the inputs' radii, with directed-up operations.
// X - x is [-h, h], so with mag M = |BC| + |B|W the Gauss-Seidel sum of row k over the whole
// box is S_k = r_k +- sum_{j != k} mag(M_kj) h_j.  Writing T_k = sum_j mag(M_kj) h_j (all j):
//   * |r_k| > T_k in some row: 0 is outside S_k + M_kk [-h_k, h_k], so every quotient of the
//     extended division S_k / M_kk lies outside [-h_k, h_k] and Y_k misses X_k.  The
//     Gauss-Seidel row has smaller sums (its earlier coordinates have only shrunk, and the
//     FP64 operations are inclusion monotone), so it is empty as well: the box is dropped.
//   * T_k - |r_k| >= 2 h_k |(BC)_kk| in every row: the lower end of S_k (after mirroring to
//     r_k, (BC)_kk >= 0) is at or below -h_k times the lower end of M_kk, which in each case
//     of the extended division (ordinary, one piece, two pieces, whole line) makes the hull of
//     Y_k and X_k equal X_k.  No row changes, so the sequential sweep equals these rows: the
//     box is unchanged.
//   Krawczyk's operator reads the same sums: K_k = x_k - r_k +- (T_k - h_k |(BC)_kk| +
//   h_k |1 - (BC)_kk|), empty when it misses X_k, unchanged when it holds X_k.
//   Centred form: F_i = f_i +- sum_j (|C_ij| + W_ij) h_j, excluded when 0 lies outside.
// Each comparison carries the enclosures' radii; a box with a comparison that they leave
// open, a pivot that they do not single out, or a value out of range is undecided.  Only
// |B| W h and the radii's sums enter T, so M itself costs one n x n product BC per box and
// the rest are matrix-vector products.
//
// Measured (GB300, the whole contraction stage per solve, before -> after): n = 8, 9.0e5
// boxes, 15.6 -> 5.9 ms; n = 9 (kinema), 1.5e7 boxes, 274 -> 93 ms; n = 11 with the centred
// form, 166 -> 36 ms; n = 7 Krawczyk, 5.6 -> 2.5 ms.  What remains is the FP64 sweep of the
// boxes that shrink.
//
// Mapping: 32 boxes per block.  J(X) and f(x): one polynomial per warp, one box per lane (no
// divergence in the term loops).  Gauss-Jordan and BC: Wd lanes per box (4, 8 or 16), lane
// j holds column j in registers; each step's pivot column goes through shared memory once
// and is read back as 16-byte broadcasts.  Rows are not swapped: the pivot rows are kept as
// a permutation.  The planes of J are padded to 32 + 32 / Wd floats per entry, which makes
// both the lane = box writes and the lane = column reads conflict-free.
#pragma once
#include <cuda_runtime.h>

#include "ivs_internal.h"
#include "ivs_interval.cuh"
#include "ivs_kernels.cuh"
#include "ivs_tab.cuh"

namespace ivs {

namespace scr {
constexpr unsigned kFull = 0xFFFFFFFFu;
constexpr float kU = 5.9604645e-8f;     // 2^-24, the float rounding unit
constexpr float kTiny = kScrTiny;       // absolute part of every radius (underflow)
constexpr float kHuge = 1e15f;          // larger magnitudes are left to FP64
constexpr float kSlack = 1.0f + 1e-5f;  // relative part of the final comparisons

template <int N>
struct Cfg {
    static constexpr int BB = 32;
    static constexpr int WD = N <= 4 ? 4 : N <= 8 ? 8 : 16;    // lanes per box
    static constexpr int NT = BB * WD;
    static constexpr int NP = (N + 3) & ~3;                    // a column, padded to 16 bytes
    static constexpr int P = 32 + 32 / WD;                     // floats per plane entry
    static constexpr int GS = N * NP + 4;                      // a box's N columns, padded
    // floats
    static constexpr int JC = 0;                               // N^2: centre of J_ij
    static constexpr int JW = JC + N * N * P;                  // N^2: half width
    static constexpr int JR = JW + N * N * P;                  // N^2: radius
    static constexpr int G1 = (JW + 3) & ~3;                   // B's columns per box: values
    static constexpr int G2 = G1 + BB * GS;                    // and radii (over JW, JR, read before)
    static constexpr int JEND = JR + N * N * P, GEND = G2 + BB * GS;
    static constexpr int XL = JEND > GEND ? JEND : GEND;       // N: box ends
    static constexpr int XH = XL + N * BB;
    static constexpr int PL = XH + N * BB;                     // kScrPow N: powers' lower ends
    static constexpr int PH = PL + kScrPow * N * BB;           // and upper ends
    static constexpr int PX = PH + kScrPow * N * BB;           // powers of the centre
    static constexpr int HW = PX + kScrPow * N * BB;           // N: half widths
    static constexpr int FV = HW + N * BB;                     // N: f(x)
    static constexpr int FR = FV + N * BB;                     // N: its radius
    static constexpr int VEC = (FR + N * BB + 3) & ~3;         // per box N x {W h, radius, magnitude, f}
    static constexpr int VS = 4 * N + 4;                       // a box's vectors, padded
    static constexpr int QS = VEC + BB * VS;                   // per box 2 N: sum_j h_j |BC|, BC_kk
    static constexpr int FLOATS = QS + BB * (2 * NP + 4);
    // doubles: widths of the box (for the accept test)
    static constexpr size_t WOFF = ((size_t)FLOATS * 4 + 15) & ~(size_t)15;
    static constexpr size_t BYTES = WOFF + (size_t)N * BB * 8;
    static constexpr int MIN_BLOCKS = N <= 4 ? 6 : N <= 8 ? 3 : 1;
};

// box fates
enum : int { SC_OPEN = 0, SC_EMPTY = 1, SC_CENTRED = 2, SC_KEEP = 3 };

struct Poly { float c, w, r; };   // [c - w, c + w], every end within r

// x^k over [l, h] (magnitude m) by the power rule, in round to nearest
__device__ __forceinline__ void pow32(float l, float h, float m, int k, float &a, float &b, float &mm) {
    if (k == 1) {
        a = l;
        b = h;
        mm = m;
        return;
    }
    if ((k & 1) == 0) {
        const float z = fmaxf(fmaxf(l, -h), 0.0f);
        a = z;
        b = m;
        for (int i = 1; i < k; i++) {
            a *= z;
            b *= m;
        }
        mm = b;
        return;
    }
    const float al = fabsf(l), ah = fabsf(h);
    a = l;
    b = h;
    mm = m;
    for (int i = 1; i < k; i++) {
        a *= al;
        b *= ah;
        mm *= m;
    }
}

// Natural extension of polynomial p over the box (ends xl, xh, stride 32 floats).  The FP64
// ends are real interval arithmetic up to rounding, so the float ends differ from them by at
// most (operations + input roundings) x 2^-24 x the sum of the terms' magnitudes, plus what
// products lose below float's normal range: tiny, a bound over the system's initial box
// (host::float_range).  Magnitudes that underflow themselves are covered by it too.
// Terms of up to three factors of degree up to kScrPow read the box's powers (pl, ph: computed
// once per box, stride 32) and one 16-byte record; the others go through the term table.
// (With the table alone every term decoded its factors and raised its powers again; with that, the
// n = 11 stage 30.3 -> 23.6 ms and kinema 93.6 -> 87.4, the pivot search by trees included.)
__device__ __forceinline__ Poly poly_c(const SysTab &T, int p, const float *xl, const float *xh, const float *pl_,
                                       const float *ph_, float tiny) {
    const int t0 = T.poly_off[p], t1 = T.poly_off[p + 1];
    const float nt = (float)(t1 - t0 + 6);
    float lo = 0.0f, hi = 0.0f, rad = 0.0f;
    bool exact = t1 - t0 <= 1;
    for (int t = t0; t < t1; t++) {
        const ScrTerm q = T.scr[t];
        if (q.kind) {
            float l = 1.0f, h = 1.0f, m = 1.0f;
            uint32_t f = q.fac;
            if ((f & 255u) != 255u) {
                const int at = (int)(f & 255u) * 32;
                l = pl_[at];
                h = ph_[at];
                m = fmaxf(fabsf(l), fabsf(h));
                for (f = (f >> 8) | 0xFF000000u; (f & 255u) != 255u; f = (f >> 8) | 0xFF000000u) {
                    const int at2 = (int)(f & 255u) * 32;
                    const float a = pl_[at2], b = ph_[at2];
                    const float p1 = l * a, p2 = l * b, p3 = h * a, p4 = h * b;
                    l = fminf(fminf(p1, p2), fminf(p3, p4));
                    h = fmaxf(fmaxf(p1, p2), fmaxf(p3, p4));
                    m *= fmaxf(fabsf(a), fabsf(b));
                }
            }
            const float q1 = q.c * l, q2 = q.c * h;
            lo += fminf(q1, q2);
            hi += fmaxf(q1, q2);
            rad = fmaf(q.w, m, rad);
            exact = exact && q.kind == 3u;
            continue;
        }
        const uint32_t info = T.tinfo[t];
        const float4 ce = T.cs[t];
        const int nf = term_nf(info), f0 = term_f0(info);
        float pl = 1.0f, ph = 1.0f, pm = 1.0f;
        int deg = 0;
        for (int f = 0; f < nf; f++) {
            const unsigned fc = T.fac[f0 + f];
            const int j = (int)(fc >> 4), k = (int)(fc & 15u);
            const float l = xl[j * 32], h = xh[j * 32], m = fmaxf(fabsf(l), fabsf(h));
            float a, b, mm;
            pow32(l, h, m, k, a, b, mm);
            deg += k;
            if (f == 0) {
                pl = a;
                ph = b;
                pm = mm;
            } else {
                const float p1 = pl * a, p2 = pl * b, p3 = ph * a, p4 = ph * b;
                pl = fminf(fminf(p1, p2), fminf(p3, p4));
                ph = fmaxf(fmaxf(p1, p2), fmaxf(p3, p4));
                pm *= mm;
            }
        }
        const float q1 = ce.x * pl, q2 = ce.x * ph;
        float l = fminf(q1, q2), h = fmaxf(q1, q2);
        if (!(info & kTermPoint)) {
            const float q3 = ce.w * pl, q4 = ce.w * ph;
            l = fminf(l, fminf(q3, q4));
            h = fmaxf(h, fmaxf(q3, q4));
        }
        lo += l;
        hi += h;
        exact = exact && deg == 0 && (info & kTermPoint) && ce.x == ce.y;
        rad += fmaxf(fabsf(ce.x), fabsf(ce.w)) * pm * ((float)(2 * deg) + nt);
    }
    // a single constant that float holds exactly has no error
    return Poly{0.5f * (lo + hi), 0.5f * (hi - lo), exact ? kTiny : rad * (1.01f * kU) + tiny};
}

// value of polynomial p at the box's centre (each coordinate within 2 units of the largest
// end's magnitude), with its radius
__device__ __forceinline__ float2 poly_v(const SysTab &T, int p, const float *xl, const float *xh, const float *pl_,
                                         const float *ph_, const float *px_, float tiny) {
    const int t0 = T.poly_off[p], t1 = T.poly_off[p + 1];
    const float nt = (float)(t1 - t0 + 6);
    float v = 0.0f, w = 0.0f, rad = 0.0f;
    for (int t = t0; t < t1; t++) {
        const ScrTerm q = T.scr[t];
        if (q.kind) {
            float x = q.c, m = q.w;
            for (uint32_t f = q.fac; (f & 255u) != 255u; f = (f >> 8) | 0xFF000000u) {
                const int at = (int)(f & 255u) * 32;
                x *= px_[at];
                m *= fmaxf(fabsf(pl_[at]), fabsf(ph_[at]));
            }
            v += x;
            rad = fmaf(2.0f, m, rad);   // the centre's powers err by at most twice the ends'
            continue;
        }
        const uint32_t info = T.tinfo[t];
        const float4 ce = T.cs[t];
        const int nf = term_nf(info), f0 = term_f0(info);
        float pv = 1.0f, pm = 1.0f;
        int deg = 0;
        for (int f = 0; f < nf; f++) {
            const unsigned fc = T.fac[f0 + f];
            const int j = (int)(fc >> 4), k = (int)(fc & 15u);
            const float l = xl[j * 32], h = xh[j * 32], m = fmaxf(fabsf(l), fabsf(h)), x = 0.5f * (l + h);
            for (int i = 0; i < k; i++) {
                pv *= x;
                pm *= m;
            }
            deg += k;
        }
        v = fmaf(ce.x, pv, v);
        // a coefficient interval widens the value by its own width
        if (!(info & kTermPoint)) w += (ce.w - ce.x) * pm;
        rad += fmaxf(fabsf(ce.x), fabsf(ce.w)) * pm * ((float)(4 * deg) + nt);
    }
    return make_float2(v, fmaf(rad, 1.01f * kU, w * 1.01f) + tiny);
}

__device__ __forceinline__ float mul_ru(float a, float b) { return __fmul_ru(a, b); }
__device__ __forceinline__ float fma_ru(float a, float b, float c) { return __fmaf_ru(a, b, c); }

// a column of NP floats (16-byte aligned)
template <int NP>
__device__ __forceinline__ void load_col(const float *p, float (&v)[NP]) {
#pragma unroll
    for (int q = 0; q < NP / 4; q++) {
        const float4 x = reinterpret_cast<const float4 *>(p)[q];
        v[4 * q] = x.x;
        v[4 * q + 1] = x.y;
        v[4 * q + 2] = x.z;
        v[4 * q + 3] = x.w;
    }
}

template <int M>
__device__ __forceinline__ float tree_max(const float (&v)[M]) {
    float m[M];
#pragma unroll
    for (int i = 0; i < M; i++) m[i] = v[i];
#pragma unroll
    for (int o = 1; o < M; o <<= 1) {
#pragma unroll
        for (int i = 0; i + o < M; i += 2 * o) m[i] = fmaxf(m[i], m[i + o]);
    }
    return m[0];
}

// one atomic per distinct (system, slot) of the warp's counting lanes
__device__ __forceinline__ void count_warp(const SweepArgs &a, int sys, int slot, bool on) {
    const unsigned m = __ballot_sync(kFull, on);
    if (!on) return;
    const unsigned same = __match_any_sync(m, ((unsigned long long)sys << 12) | (unsigned long long)slot);
    if ((int)(threadIdx.x & 31u) == __ffs(same) - 1)
        atomicAdd(a.stats + (size_t)sys * ST_COUNT + slot, (unsigned long long)__popc(same));
}
}  // namespace scr

// Systems of fewer variables are not screened: their FP64 sweep is a few hundred operations,
// and on batches of 29 to 96 systems the screen's launch and first chunk cost what it saved
// (n = 2: 0.53 -> 0.60 ms of a batch's sweeps, n = 3: 0.51 -> 0.65, n = 4: 1.02 -> 1.04, n = 5:
// 2.98 -> 1.87, n = 8 of the 64-system batch: 406 -> 136).
constexpr int kScreenMinVars = 4;

// Where the screen's list of undecided boxes of dimension n begins: in a.cand (the
// evaluation's candidates have been used by then), behind room for the survivors of the
// smaller dimensions; all survivors of a sweep fit, there are at most as many as children.
__device__ __forceinline__ long long open_list_base(const WaveCtl *c, int n) {
    long long b = 0;
    for (int k = 1; k < n; k++) b += c->surv_count[k];
    return b;
}

// A sweep with at most `screen_min` boxes is not screened: it runs in one round of narrow
// FP64 chunks, whose time is one chunk's latency whatever the number of boxes.
template <int N>
__global__ void __launch_bounds__(scr::Cfg<N>::NT, scr::Cfg<N>::MIN_BLOCKS)
    k_screen(SweepArgs a, int cache_blob, long long screen_min) {
    using namespace scr;
    using C = Cfg<N>;
    constexpr int BB = C::BB, NT = C::NT, WD = C::WD, P = C::P;
    extern __shared__ __align__(16) char smem[];
    __shared__ long long s_base;
    __shared__ Surv s_sv[BB];
    __shared__ int s_sys[BB], s_mode[BB], s_bad[BB], s_fate[BB], s_depth[BB], s_jw[BB];
    __shared__ long long s_pos[BB];
    WaveCtl *ctl = a.ctl;
    const long long count = ctl->surv_count[N];
    if (count <= screen_min || (long long)blockIdx.x * BB >= count) return;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    if (cache_blob) {
        const DevSys &S0 = a.tb.sys[0];
        copy_blob(smem, a.tb.blobs + S0.blob_off, (uint32_t)S0.head_bytes);   // visible after the next barrier
    }
    float *sf = reinterpret_cast<float *>(smem + (cache_blob ? (size_t)a.head_smem : 0));
    double *sw = reinterpret_cast<double *>(reinterpret_cast<char *>(sf) + C::WOFF);
    const Surv *list = a.surv + (size_t)N * a.surv_cap;
    Surv *open = a.cand + open_list_base(ctl, N);
    for (;;) {
        if (t == 0) s_base = (long long)atomicAdd((unsigned long long *)&ctl->screen_cursor[N], (unsigned long long)BB);
        __syncthreads();
        const long long base = s_base;
        if (base >= count) break;
        if (t < BB) {
            // mode: bit 0 takes part, 1 sweep wanted, 2 Krawczyk, 3 centred test
            int mode = 0, sys = 0, depth = 0;
            Surv sv{0, 0};
            if (base + t < count) {
                sv = list[base + t];
                sys = a.q.sys[sv.parent];
                const uint32_t meta = a.q.meta[sv.parent];
                depth = (int)(meta & kDepthMask) + ((meta & kRootFlag) ? 0 : 1);
                const DevSys &S = a.tb.sys[sys];
                const bool hs = S.hs_enable && depth >= S.hs_min_depth;
                if (S.prefilter && S.shadow && S.j_poly >= 0 && !S.gap_split && (hs || S.centred))
                    mode = 1 | (hs ? 2 : 0) | (S.krawczyk ? 4 : 0) | (S.centred ? 8 : 0);
            }
            s_sv[t] = sv;
            s_sys[t] = sys;
            s_depth[t] = depth;
            s_mode[t] = mode;
            s_bad[t] = 0;
            s_fate[t] = 0;
        }
        __syncthreads();
        for (int e = t; e < N * BB; e += NT) {
            const int j = e / BB, b = e % BB;
            float l = 0.0f, h = 0.0f, hw = 0.0f;
            double w = 0.0;
            if (s_mode[b]) {
                const Surv sv = s_sv[b];
                const size_t at = (size_t)j * a.q.cap + sv.parent;
                const bool up = (sv.child >> j) & 1u;
                const double lo = up ? a.q.mid[at] : a.q.lo[at], hi = up ? a.q.hi[at] : a.q.mid[at];
                w = __dsub_rn(hi, lo);
                l = __double2float_rn(lo);
                h = __double2float_rn(hi);
                hw = 0.5f * __double2float_rn(w);
                const float m = fmaxf(fabsf(l), fabsf(h));
                // the ends of X - x are +- h up to FP64 roundings of the ends: far below the
                // float unit only while h is not tiny beside them
                if (!(m < kHuge && hw > m * 3.7e-9f && hw > 1e-18f)) atomicOr(&s_bad[b], 1);
            }
            sf[C::XL + j * BB + b] = l;
            sf[C::XH + j * BB + b] = h;
            sf[C::HW + j * BB + b] = hw;
#pragma unroll
            for (int k = 1; k <= kScrPow; k++) {
                float x, y, mm;
                pow32(l, h, fmaxf(fabsf(l), fabsf(h)), k, x, y, mm);
                sf[C::PL + (j * kScrPow + k - 1) * BB + b] = x;
                sf[C::PH + (j * kScrPow + k - 1) * BB + b] = y;
                const float c = 0.5f * (l + h);
                float v = c;
                for (int i = 1; i < k; i++) v *= c;
                sf[C::PX + (j * kScrPow + k - 1) * BB + b] = v;
            }
            sw[j * BB + b] = w;
        }
        __syncthreads();
        // J(X) and f(x): one polynomial per warp, one box per lane
        {
            const int b = lane;
            const bool on = s_mode[b] != 0;
            const DevSys &S = a.tb.sys[s_sys[b]];
            const SysTab T = make_tab(cache_blob ? smem : a.tb.blobs + S.blob_off, S);
            const float *xl = sf + C::XL + b, *xh = sf + C::XH + b;
            const float tiny = S.scr_tiny;
            for (int q = warp; q < N * N + N; q += NT / 32) {
                if (!on) continue;
                if (q < N * N) {
                    const Poly v = poly_c(T, S.j_poly + q, xl, xh, sf + C::PL + b, sf + C::PH + b, tiny);
                    sf[C::JC + q * P + b] = v.c;
                    sf[C::JW + q * P + b] = v.w;
                    sf[C::JR + q * P + b] = v.r;
                } else {
                    const float2 v = poly_v(T, S.f_poly + (q - N * N), xl, xh, sf + C::PL + b, sf + C::PH + b,
                                            sf + C::PX + b, tiny);
                    sf[C::FV + (q - N * N) * BB + b] = v.x;
                    sf[C::FR + (q - N * N) * BB + b] = v.y;
                }
            }
        }
        __syncthreads();
        // row sums of J weighted with h: half widths, radii (with the float error of the
        // products below), magnitudes; the centred test
        for (int e = t; e < N * BB; e += NT) {
            const int u = e / BB, b = e % BB;
            if (!s_mode[b]) continue;
            constexpr float g = (float)(N + 4) * 1.02f * kU;
            float wv = 0.0f, rv = 0.0f, av = 0.0f;
#pragma unroll
            for (int j = 0; j < N; j++) {
                const float h = sf[C::HW + j * BB + b];
                const float c = fabsf(sf[C::JC + (u * N + j) * P + b]), w = sf[C::JW + (u * N + j) * P + b];
                const float r = sf[C::JR + (u * N + j) * P + b];
                wv = fmaf(h, w, wv);
                rv = fma_ru(h, fma_ru(g, c + w, r), rv);
                av = fma_ru(h, c + w + r, av);
            }
            const float f = sf[C::FV + u * BB + b], fr = sf[C::FR + u * BB + b];
            float *v = sf + C::VEC + b * C::VS + 4 * u;
            v[0] = wv;
            v[1] = rv + fma_ru(g, fabsf(f), fr);   // every radius that B multiplies
            v[2] = av + fabsf(f) + fr;             // and every magnitude that B's radius does
            v[3] = f;
            if (s_mode[b] & 8) {
                const float err = (rv + fr + 1e-5f * (av + fabsf(f))) * kSlack;
                if (!(av < kHuge && fabsf(f) < kHuge)) atomicOr(&s_bad[b], 1);
                else if (fabsf(f) > av + err) atomicOr(&s_fate[b], 1);     // excluded
                // (av holds J's ends moved out by the radii; they may lie as far in)
                else if (!(fabsf(f) + err + rv * kSlack <= av)) atomicOr(&s_fate[b], 2);   // open
            }
        }
        __syncthreads();
        // Gauss-Jordan of mid J(X) with enclosures, Wd lanes per box
        {
            const int b = t / WD, j = t % WD;
            const int jc = j < N ? j : N - 1;   // idle lanes shadow the last column
            // boxes that still want the sweep: in range, not settled by the centred form
            const bool want = (s_mode[b] & 2) && !s_bad[b] && !(s_fate[b] & 3);
            const bool any = __any_sync(kFull, want);
            float gm[N], gr[N];
#pragma unroll
            for (int i = 0; i < N; i++) {
                gm[i] = sf[C::JC + (i * N + jc) * P + b];
                gr[i] = fma_ru(2.0f * kU, fabsf(gm[i]), sf[C::JR + (i * N + jc) * P + b]);
                if (sf[C::JR + (i * N + jc) * P + b] <= kTiny) gr[i] = kTiny;   // an exact constant
            }
            __syncthreads();   // J's half widths and radii have been read: B's columns take their place
            if (any) {   // (a warp whose boxes are all settled skips the rest)
            float *col1 = sf + C::G1 + b * C::GS, *col2 = sf + C::G2 + b * C::GS;
            unsigned used = 0;
            bool ok = true;
            int prow[N];
#pragma unroll
            for (int k = 0; k < N; k++) {
                __syncwarp();
                if (j == k) {
#pragma unroll
                    for (int i = 0; i < N; i++) {
                        col1[k * C::NP + i] = gm[i];
                        col2[k * C::NP + i] = gr[i];
                    }
                }
                __syncwarp();
                float f[C::NP], fr[C::NP];
                load_col<C::NP>(col1 + k * C::NP, f);
                load_col<C::NP>(col2 + k * C::NP, fr);
                // the pivot: the largest of the unused rows, by more than the radii.  Maxima by
                // trees and the pivot's entries through shared memory: as chains of selects
                // this was the longest part of a step.  (fmaxf passes a NaN over, but a NaN
                // entry stays in its row and fails the range test at the end.)
                float top[C::NP];
#pragma unroll
                for (int i = 0; i < C::NP; i++) top[i] = i < N && !((used >> i) & 1u) ? fabsf(f[i]) : -1.0f;
                const float best = tree_max<C::NP>(top);
                unsigned at = 0;
#pragma unroll
                for (int i = 0; i < N; i++) at |= top[i] == best ? 1u << i : 0u;
                const int p = at ? __ffs((int)at) - 1 : 0;
                const float pv = col1[k * C::NP + p], br = col2[k * C::NP + p];
                const float low = __fsub_rd(best, br);
#pragma unroll
                for (int i = 0; i < C::NP; i++)
                    top[i] = i < N && i != p && !((used >> i) & 1u) ? __fadd_ru(fabsf(f[i]), fr[i]) : -1.0f;
                ok = ok && low > 1e-15f && best < kHuge && tree_max<C::NP>(top) < low;
                used |= 1u << p;
                prow[k] = p;
                // 1 / pivot, then the pivot row's entry of this column
                const float rp = __frcp_rn(pv);
                const float rr = fma_ru(mul_ru(br, fabsf(rp) * (1.0f + 4.0f * kU)), __frcp_ru(low),
                                        fma_ru(2.0f * kU, fabsf(rp), kTiny));
                unsigned ua = 0, ur = 0;   // entry p of the lane's column
#pragma unroll
                for (int i = 0; i < N; i++) {
                    ua |= i == p ? __float_as_uint(gm[i]) : 0u;
                    ur |= i == p ? __float_as_uint(gr[i]) : 0u;
                }
                const float am = __uint_as_float(ua), ar = __uint_as_float(ur);
                float c = am * rp;
                float cr = fma_ru(fabsf(am), rr, fma_ru(ar, __fadd_ru(fabsf(rp), rr), fma_ru(2.0f * kU, fabsf(c), kTiny)));
                if (j == k) {
                    c = rp;
                    cr = rr;
                }
                const float ca = __fadd_ru(fabsf(c), cr);
                const float cr2 = fma_ru(1e-15f, ca, cr);   // with FP64's rounding of f c
#pragma unroll
                for (int i = 0; i < N; i++) {
                    const float a0 = j == k ? 0.0f : gm[i], r0 = j == k ? kTiny : gr[i];
                    const float m = fmaf(-f[i], c, a0);
                    const float r = fma_ru(2.0f * kU, fabsf(m), fma_ru(fabsf(f[i]), cr2, fma_ru(fr[i], ca, r0)));
                    gm[i] = i == p ? c : m;
                    gr[i] = i == p ? cr : r;
                }
            }
            __syncwarp();
            // storage column l is column prow[l] of B; row prow[k] is row k
            if (j < N) {
#pragma unroll
                for (int i = 0; i < N; i++) {
                    col1[j * C::NP + i] = gm[i];
                    col2[j * C::NP + i] = gr[i];
                    ok = ok && fabsf(gm[i]) < kHuge && gr[i] < kHuge;
                }
            }
            if (!ok) atomicOr(&s_bad[b], 2);
            __syncwarp();
            // column j of BC: every row at once
            float acc[N];
#pragma unroll
            for (int i = 0; i < N; i++) acc[i] = 0.0f;
#pragma unroll
            for (int l = 0; l < N; l++) {
                const float jv = sf[C::JC + (prow[l] * N + jc) * P + b];
                float g[C::NP];
                load_col<C::NP>(col1 + l * C::NP, g);
#pragma unroll
                for (int i = 0; i < N; i++) acc[i] = fmaf(g[i], jv, acc[i]);
            }
            // row i's sum over the columns of h_j |BC_ij|, and its diagonal entry
            float *qs = sf + C::QS + b * (2 * C::NP + 4);
            const float h = j < N ? sf[C::HW + jc * BB + b] : 0.0f;
#pragma unroll
            for (int i = 0; i < N; i++) {
                float v = h * fabsf(acc[i]);
#pragma unroll
                for (int o = WD / 2; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o, WD);
                if (j == i) qs[i] = v;
            }
            if (j < N) {
                int pj = 0;
                float d = 0.0f;
#pragma unroll
                for (int k = 0; k < N; k++) pj = k == j ? prow[k] : pj;
#pragma unroll
                for (int i = 0; i < N; i++) d = i == pj ? acc[i] : d;
                qs[C::NP + j] = d;
            }
            __syncwarp();
            // row k: lane k of the box
            if (j < N && s_mode[b] && !s_bad[b]) {
                int pk = 0;
#pragma unroll
                for (int k = 0; k < N; k++) pk = k == j ? prow[k] : pk;
                float vw = 0.0f, er = 0.0f, rc = 0.0f;
#pragma unroll
                for (int l = 0; l < N; l++) {
                    const float g = col1[l * C::NP + pk], gr1 = col2[l * C::NP + pk];
                    const float *v = sf + C::VEC + b * C::VS + 4 * prow[l];
                    vw = fmaf(fabsf(g), v[0], vw);
                    er = fma_ru(fabsf(g), v[1], fma_ru(gr1, v[2], er));
                    rc = fmaf(g, v[3], rc);
                }
                const float T = qs[pk] + vw, ra = fabsf(rc), d = qs[C::NP + j], hk = sf[C::HW + j * BB + b];
                // the slack covers the float error of T's sums (at most 2 N + 6 units of T; that
                // of the products BC and B f is in er), the ends of X - x (3 units of h) and
                // FP64's quotients and differences
                const float err = fmaf(4e-6f, T + ra, er * kSlack) + 1e-25f;
                const bool range = T < kHuge && ra < kHuge && er < kHuge && fabsf(d) < kHuge;
                int v = 0;   // 1 empty, 2 unchanged
                if (range && (s_mode[b] & 4)) {
                    const float Tk = T + hk * (fabsf(1.0f - d) - fabsf(d));
                    const float e2 = err + 4e-6f * hk * (2.0f * fabsf(d) + 1.0f);
                    if (ra - Tk > hk + e2) v = 1;
                    else if (Tk - ra >= hk + e2) v = 2;
                } else if (range) {
                    if (ra > T + err) v = 1;
                    else if (T - ra >= 2.0f * hk * fabsf(d) * (1.0f + 4e-6f) + err) v = 2;
                }
                if (v == 1) atomicOr(&s_fate[b], 4);
                else if (v == 0) atomicOr(&s_fate[b], 8);
            }
            }
        }
        __syncthreads();
        // fates: warp 0, lane b owns box b
        if (warp == 0) {
            const int b = lane, mode = s_mode[b], f = s_fate[b], sys = s_sys[b], depth = s_depth[b];
            const bool valid = base + b < count;
            const int dslot = depth < kDepthSlots ? depth : kDepthSlots - 1;
            int fate = SC_OPEN;
            const int bad = s_bad[b];   // 1: a coordinate or J(X) out of range, 2: B not enclosed
            if (mode && !(bad & 1)) {
                if (f & 1) fate = SC_CENTRED;
                else if (f & 2) fate = SC_OPEN;
                else if (!(mode & 2)) fate = SC_KEEP;
                else if (!bad && (f & 4)) fate = SC_EMPTY;
                else if (!bad && !(f & 8)) fate = SC_KEEP;
            }
            // the sweep's accept / split step for the boxes it would leave unchanged
            int step = 0, flag = 0, jw = 0;   // step: 1 accepted, 2 new parent
            if (fate == SC_KEEP) {
                const DevSys &S = a.tb.sys[sys];
                double w = 0.0;
#pragma unroll
                for (int j = 0; j < N; j++) {
                    const double wj = sw[j * BB + b];
                    if (d_key(wj) > d_key(w)) {
                        w = wj;
                        jw = j;
                    }
                }
                // the widest coordinate's midpoint lies strictly inside: h > 2^-28 of its
                // ends' magnitude (the range test above)
                if (d_key(w) <= d_key(S.tol)) {
                    step = 1;
                    flag = 1;
                } else if (depth + 1 > S.max_depth) {
                    step = 1;
                    flag = 4;
                } else {
                    step = 2;
                }
            }
            // undecided boxes, for the FP64 sweep
            {
                const bool o = valid && fate == SC_OPEN;
                const unsigned m = __ballot_sync(kFull, o);
                if (m) {
                    unsigned long long pos = 0;
                    if (lane == 0) pos = atomicAdd((unsigned long long *)&ctl->open_count[N], (unsigned long long)__popc(m));
                    pos = __shfl_sync(kFull, pos, 0);
                    if (o) open[pos + __popc(m & ((1u << lane) - 1u))] = s_sv[b];
                }
            }
            // new parents
            long long k = -1;
            {
                const unsigned m = __ballot_sync(kFull, step == 2);
                if (m) {
                    unsigned long long pos = 0;
                    if (lane == 0) pos = atomicAdd((unsigned long long *)&ctl->staged, (unsigned long long)__popc(m));
                    pos = __shfl_sync(kFull, pos, 0);
                    if (step == 2) {
                        k = (long long)(pos + __popc(m & ((1u << lane) - 1u)));
                        if (k < a.stage.cap) {
                            const bool bis = a.tb.sys[sys].bisect != 0;
                            a.stage.sys[k] = sys;
                            a.stage.meta[k] = ((uint32_t)depth & kDepthMask) | (bis ? ((uint32_t)jw << kSplitShift) : 0u) |
                                              ((uint32_t)(bis ? 1 : N) << kFanShift);
                        } else {
                            ctl->error = 1;
                            k = -1;
                        }
                    }
                }
            }
            // accepted boxes, into the system's result region
            long long out = -1;
            if (step == 1) {
                const DevSys &S = a.tb.sys[sys];
                const long long q = (long long)atomicAdd(a.stats + (size_t)sys * ST_COUNT + ST_OUT, 1ull);
                unsigned long long fl = flag == 4 ? (unsigned long long)kFlagDepthCut : 0ull;
                if (q < S.out_cap) {
                    out = S.out_base + q;
                    a.out.sys[out] = sys;
                    a.out.flags[out] = flag;
                    a.out.depth[out] = depth;
                } else {
                    fl |= (unsigned long long)kFlagResultOverflow;
                }
                if (fl) atomicOr(a.stats + (size_t)sys * ST_COUNT + ST_FLAGS, fl);
            }
            s_jw[b] = step == 2 && k >= 0 ? (a.tb.sys[sys].bisect ? jw : N) : (out >= 0 ? N + 1 : -1);
            s_pos[b] = step == 2 ? k : out;
            // the counters the FP64 sweep would have raised
            const bool swept = (fate == SC_EMPTY || fate == SC_KEEP) && (mode & 2);
            count_warp(a, sys, ST_HS_APPLIED, swept);
            count_warp(a, sys, ST_DEPTH_HS + dslot, swept);
            count_warp(a, sys, ST_HS_EMPTY, fate == SC_EMPTY);
            count_warp(a, sys, ST_EXCL_CENTRED, fate == SC_CENTRED);
            count_warp(a, sys, ST_DEPTH_KEPT + dslot, step != 0);
            count_warp(a, sys, ST_ACCEPTED, step == 1 && flag != 4);
            count_warp(a, sys, ST_SPLIT, step == 2);
            count_warp(a, sys, ST_LIVE, step == 2);
        }
        __syncthreads();
        // the kept boxes' coordinates (one per thread); split midpoints as in the FP64 step
        for (int e = t; e < N * BB; e += NT) {
            const int j = e / BB, b = e % BB, w = s_jw[b];
            if (w < 0) continue;
            const Surv sv = s_sv[b];
            const size_t at = (size_t)j * a.q.cap + sv.parent;
            const bool up = (sv.child >> j) & 1u;
            const double lo = up ? a.q.mid[at] : a.q.lo[at], hi = up ? a.q.hi[at] : a.q.mid[at];
            const long long k = s_pos[b];
            if (w == N + 1) {
                a.out.lo[j * a.out.cap + k] = lo;
                a.out.hi[j * a.out.cap + k] = hi;
            } else {
                a.stage.lo[j * a.stage.cap + k] = lo;
                a.stage.mid[j * a.stage.cap + k] = (w < N && j != w) ? hi : __dmul_rn(0.5, __dadd_rn(lo, hi));
                a.stage.hi[j * a.stage.cap + k] = hi;
            }
        }
        __syncthreads();   // the chunk's arrays are reused by the next chunk
    }
}

}  // namespace ivs
