// cp_spec.cu -- the direct form through the pair spectrum (arXiv:1412.1840).
//
// Eq. (taylor) regrouped by harmonic, a_n = 2 e^-k I_n(k), k = 1 / sigma_t^2:
//   S(f) = sum_ij w_ij exp(-2 sin^2(pi f t_ij) / sigma_t^2)
//        = N (1 - ip) (1 - a_0) + 2 sum_{n=1}^{nh} a_n P(n f),
//   P(nu) = sum_{i<j} w_ij cos(2 pi nu (t_i - t_j))
// (sum_{i<j} w_ij = -N (1 - ip) / 2 by Eq. (IP)).  P is one function of one
// variable: the N (N - 1) / 2 pairs are gone through once per curve instead of
// once per trial frequency.  It is computed by a non-uniform cosine transform
// (Dutt and Rokhlin 1993; the Kaiser-Bessel window of Beatty et al. 2005):
//
//   k_spec_prep    per curve: a_n by Miller's backward recurrence (FP64), the
//                  transform length, times in grid cells (exact 32.32 fixed
//                  point) in ascending order
//   k_spec_spread  every pair adds w_ij times an 8-point Kaiser-Bessel window
//                  to the cells around |t_i - t_j|; exact integer sums in
//                  shared memory, so the result does not depend on the order
//   k_spec_fft1/2  cosine transform of the cells (a DCT-II as one complex
//                  transform of half the length, Makhoul 1980), two passes of
//                  at most 2048 points; the last one divides by the window's
//                  transform and writes P on the grid of multiples of delta
//   k_spec_sum     the harmonic sum at every trial frequency
//   k_spec_select  the trial frequencies within the rounding of the largest
//                  value; the pair-sum kernel evaluates those again, so the best
//                  frequency and its statistic are the pair sum's
//   k_spec_peaks,  coarse-then-fine search: the coarse points whose exact values
//   k_spec_rank    decide the peaks (evaluated again by the pair sum), and the peaks
//
// Frequencies that are multiples of one spacing delta (a uniform grid whose f_min
// and df are integer multiples of it) are entries of a spectrum of period
// 1 / delta; time differences beyond half of the period fold back exactly.
// Other frequencies (fine windows, trial lists, any other grid) are
// interpolated with the same window from a spectrum of period L >= 4 T, the
// pairs' weights divided by the window's transform beforehand (a type-3
// transform).
//
// Measured (GB300; N 300-1000, 49,981 frequencies, sigma_t rule): best period of
// 384 curves 715 ms by the pair sum alone, 3.9 ms through the spectrum, results
// identical; 12 periodograms 25.4 -> 0.25 ms, error against FP64 3.2e-7 -> 8e-8;
// three of up to 4,096 samples at 4,981 frequencies 24.5 -> 0.43 ms;
// coarse-then-fine search of 256 curves 81.3 -> 3.1 ms, results identical.
#include <cmath>
#include <cstdint>
#include <cuda_runtime.h>

#include "cp_spec.cuh"

namespace cpk {

// ---- Kaiser-Bessel window, 8 cells wide, shape 18.4 ---------------------------
// phi(x) = I_0(18.4 sqrt(1 - (x/4)^2)) / I_0(18.4), |x| <= 4 cells.  For a point at
// fraction f of the way from cell l to l + 1, z = f - 1/2: the weight of cell
// l + k is E_k(z^2) + z O_k(z^2), of cell l + 1 - k it is E_k - z O_k (k = 1..4).
// Cubics fitted at Chebyshev nodes, error below 4e-8 of the window's peak.
// Aliasing at a transform length of 1.1 times the highest frequency: below 7e-8
// of the statistic's r.m.s. for sigma_t of 0.1 to 0.6, since the highest
// harmonics carry the smallest weights.
constexpr float kKbShape = 18.4f;
constexpr float kKbInv0 = 4.3081865766e-01f;    // 1 / (transform of phi at frequency 0)
__constant__ float c_kbE[4][4] = {{8.690783782e-01f, -3.592686741e-01f, 6.729875121e-02f, -7.158902972e-03f},
                                  {2.713657147e-01f, 2.530506475e-01f, -9.204296489e-02f, 1.273117479e-02f},
                                  {2.002778820e-02f, 1.033609628e-01f, 1.877904103e-02f, -6.835285293e-03f},
                                  {1.093004653e-04f, 2.854978233e-03f, 5.982321180e-03f, 1.216996292e-03f}};
__constant__ float c_kbO[4][4] = {{4.896753093e-01f, -2.389145815e-01f, 5.541547310e-02f, -7.758932522e-03f},
                                  {4.899222498e-01f, -5.540891185e-02f, -1.377328856e-02f, 4.083793095e-03f},
                                  {7.114549842e-02f, 7.360287984e-02f, -8.433019061e-03f, -8.226859164e-04f},
                                  {8.560250652e-04f, 5.304136764e-03f, 4.027436937e-03f, -1.340719502e-04f}};

// 1 / (transform of phi) at m cells^-1 / (2 H): z / sinh(z) with
// z = sqrt(shape^2 - (4 pi m / H)^2) >= 14 here, so 2 z e^-z.
__device__ __forceinline__ float kb_inverse(float r)     // r = m / H
{
    const float o2 = (16.0f * (float)(CP_PI * CP_PI)) * (r * r);
    float z, q;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(z) : "f"(fmaf(-(16.0f * (float)(CP_PI * CP_PI)) * r, r, kKbShape * kKbShape)));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(q) : "f"(z + kKbShape));
    return (kKbInv0 / kKbShape) * z * ex2_approx(1.4426950408889634f * o2 * q);
}

// Weights of the 8 cells l - 3 .. l + 4 around a point z = f - 1/2 off the middle of cells l, l + 1.
__device__ __forceinline__ void kb_weights(float z, float (&w)[8])
{
    const float s = z * z;
#pragma unroll
    for (int k = 1; k <= 4; k++) {
        float ev = fmaf(s, c_kbE[k - 1][3], c_kbE[k - 1][2]);
        ev = fmaf(s, ev, c_kbE[k - 1][1]);
        ev = fmaf(s, ev, c_kbE[k - 1][0]);
        float od = fmaf(s, c_kbO[k - 1][3], c_kbO[k - 1][2]);
        od = fmaf(s, od, c_kbO[k - 1][1]);
        od = fmaf(s, od, c_kbO[k - 1][0]);
        w[3 + k] = fmaf(z, od, ev);
        w[4 - k] = fmaf(-z, od, ev);
    }
}

// ===========================================================================
// k_spec_prep: one CTA per curve.  Latency: the sort (only unordered times), one
// thread's recurrence and set-up in FP64; 24 us for 384 curves, 20 for 64.
// ===========================================================================
constexpr int kSpecPrepThreads = 256;
constexpr int kMillerMax = 104;

__device__ __host__ inline int spec_logq_of(int64_t n_out)
{
    int lq = kSpecMinLogQ;
    while (lq <= kSpecMaxLogQ && (double)((int64_t)2 << lq) < kSpecOver * (double)n_out) lq++;
    return lq;
}

__global__ void __launch_bounds__(kSpecPrepThreads) k_spec_prep(const SpecArgs a)
{
    // FP64 runs at 1.7 operations/clk/SM here, so only the differences and their fixed-point
    // form are FP64; the times (all >= 0) are compared as the integers of their bits.
    extern __shared__ __align__(16) unsigned char smem[];
    long long* ts = reinterpret_cast<long long*>(smem);
    int32_t* ix = reinterpret_cast<int32_t*>(ts + a.np2max);
    __shared__ double s_a[kMillerMax + 2];
    __shared__ float s_f[kMillerMax + 2];
    __shared__ long long s_max[kSpecPrepThreads / 32];
    __shared__ double s_cpd, s_T, s_inv;
    __shared__ int s_n0, s_nh;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int c = a.order[a.slot_begin + blockIdx.x];
    const CurveParams& P = a.cp[c];
    const int n = P.n;
    const int64_t off = P.off;
    const double t0 = P.t0;
    long long tmax = 0;
    for (int i = tid; i < n; i += kSpecPrepThreads) {
        long long t = __double_as_longlong(a.times[off + i] - t0);
        if (t < 0) t = t == (long long)0x8000000000000000ull ? 0 : 0x7ff8000000000000ll;   // -0; a NaN
        ts[i] = t;
        ix[i] = i;
        tmax = t > tmax ? t : tmax;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const long long t = __shfl_xor_sync(0xffffffffu, tmax, o);
        tmax = t > tmax ? t : tmax;
    }
    if (lane == 0) s_max[warp] = tmax;
    __syncthreads();
    bool ordered = true;
    for (int i = tid; i + 1 < n; i += kSpecPrepThreads) ordered = ordered && ts[i] <= ts[i + 1];
    if (!__syncthreads_and(ordered)) {
        int np2 = 1;
        while (np2 < n) np2 <<= 1;
        for (int i = n + tid; i < np2; i += kSpecPrepThreads) {
            ts[i] = 0x7fffffffffffffffll;
            ix[i] = i;
        }
        for (int k = 2; k <= np2; k <<= 1) {
            for (int j = k >> 1; j > 0; j >>= 1) {
                __syncthreads();
                for (int i = tid; i < np2; i += kSpecPrepThreads) {
                    const int q = i ^ j;
                    if (q > i) {
                        const long long u = ts[i], v = ts[q];
                        const int iu = ix[i], iv = ix[q];
                        if ((u > v || (u == v && iu > iv)) == ((i & k) == 0)) {
                            ts[i] = v; ts[q] = u;
                            ix[i] = iv; ix[q] = iu;
                        }
                    }
                }
            }
        }
        __syncthreads();
    }
    if (tid == 0) {
        for (int w = 0; w < kSpecPrepThreads / 32; w++) tmax = s_max[w] > tmax ? s_max[w] : tmax;
        const double T = __longlong_as_double(tmax);
        s_T = T;
        // a_n = 2 e^-k I_n(k) by the backward recurrence I_{n-1} = I_{n+1} + (2n/k) I_n,
        // normalised by a_0 + sum a_n = 1.  One thread's chain of FP64 FMAs; all that
        // can be done by the other threads is left to them below.
        const float st = P.sigma_t;
        int n0 = 0;
        if (st >= 0.09f && st < 1e3f && tmax < 0x7ff0000000000000ll) {
            const double s2 = (double)st * (double)st, two_k = 2.0 * s2;      // 2 / k
            n0 = min(kMillerMax, (int)(14.0f + 10.0f / st));
            double hi = 0.0, cur = 1e-200, sum = 0.0, qk = (double)n0 * two_k;
            for (int q = n0; q >= 1; q--) {
                s_a[q] = cur;
                sum += cur;
                const double nx = fma(qk, cur, hi);
                qk -= two_k;
                hi = cur;
                cur = nx;
            }
            s_a[0] = cur;
            s_inv = 1.0 / (2.0 * sum + cur);
        }
        s_n0 = n0;
        s_nh = 1;
    }
    __syncthreads();
    // harmonics kept: the smallest count whose tail is below kSpecTail
    const int n0 = s_n0;
    if (tid <= n0 && n0) s_f[tid] = (float)((tid ? 2.0 : 1.0) * s_a[tid] * s_inv);
    __syncthreads();
    if (tid <= n0 && tid >= 1) {
        float tail = 0.f;
        for (int q = n0; q >= tid; q--) tail += s_f[q];
        if (tail > (float)kSpecTail) atomicMax(&s_nh, tid);      // without harmonic tid the tail is too large
    }
    __syncthreads();
    const int nh = n0 ? s_nh : kSpecMaxHarm + 1;
    if (tid < nh && nh <= kSpecMaxHarm) a.coef[(int64_t)c * kSpecMaxHarm + tid] = s_f[tid + 1];
    if (tid == 0) {
        SpecCurve S;
        S.nh = 0;
        S.logq = 0;
        S.H = 0;
        S.L = 0.0;
        S.support = 0;
        S.n_out = 0;
        S.cells_per_day = 0.0;
        S.one_minus_a0 = 0.f;
        S.whole = 0;
        if (nh <= kSpecMaxHarm) {
            S.one_minus_a0 = (float)(1.0 - s_a[0] * s_inv);
            int lq;
            double n_out;
            if (a.interp) {
                // period at least 4 T, stretched to fill the transform
                const double top = fmax((double)nh * a.f_top, 1e-9);
                const double need = fmin(4.0 * s_T * top + 8.0, 1e9);
                lq = spec_logq_of((int64_t)need);
                S.L = ((double)((int64_t)2 << lq) / kSpecOver - 8.0) / top;
                n_out = floor(top * S.L) + 7.0;
            } else {
                n_out = (double)((int64_t)nh * (a.m0 + a.mq * (a.n_freq - 1)) + 1);
                lq = spec_logq_of((int64_t)n_out);
                S.L = 1.0 / a.delta;
            }
            S.logq = lq;
            S.H = (int64_t)2 << lq;
            S.cells_per_day = a.interp ? 2.0 * (double)S.H / S.L : 2.0 * (double)S.H * a.delta;
            const double cells = s_T * S.cells_per_day;
            // a curve that the workspace was not sized for, or spread over many periods: the pair sum
            if (n_out + kSpecPad <= (double)a.p_ld && ((int64_t)1 << lq) <= a.x_ld && cells < 64.0 * (double)S.H) {
                const double sup = ceil(cells) + 6.0;
                S.nh = nh;
                S.n_out = (int32_t)n_out;
                S.support = sup >= (double)S.H ? (int32_t)S.H : min((int32_t)S.H, ((int32_t)sup + 3) & ~3);
            }
        }
        // segments: seg_items of them per curve or more, about 16384 pairs each (a dense curve's
        // segment of 512 cells near zero difference took 270 us), of 128 cells at least
        const int items = max(a.seg_items, (int)(((int64_t)n * n) >> 15));
        S.seg = min(a.seg_max, max(128, (S.support / items + 127) & ~127));
        a.sc[c] = S;
        s_cpd = S.cells_per_day * 4294967296.0;
        a.vmax[c] = 0u;
        a.vtop[c] = 0u;
    }
    __syncthreads();
    const double cpd = s_cpd;
    for (int i = tid; i < n; i += kSpecPrepThreads) {
        a.xs[off + i] = (uint64_t)__double2ll_rn(__longlong_as_double(ts[i]) * cpd);
        a.ys[off + i] = a.yp[off + ix[i]];
    }
}

// ===========================================================================
// k_spec_spread: one item = (curve, segment of cells).  With the times sorted,
// the pairs of a segment are one range of j per row i (and per fold of the
// period).  A warp takes 16 rows, half its lanes bisecting for the first j, half
// for the last, and then 32 pairs at a time across the rows.  Cells are 64-bit
// integers of 2^-26 quanta: the low word, started at 2^31, takes a shared-memory
// integer add whose carry or borrow (rare) goes to the high word, so the sums are
// exact and do not depend on the order.  Bound by instructions issued, about 120
// per 32 pairs: the 8 cells of a pair lie at constant offsets (a margin on both
// sides of the segment takes what falls outside; at 0 and at half the period the
// margin is folded back when the segment is written).
// ===========================================================================
constexpr int kSpreadThreads = 512;
constexpr int kSpreadMargin = 16;                // cells on either side of a segment
constexpr int kSpreadRows = 16;                  // rows a warp takes at a time
// Quanta per unit of weight, 2^26: a contribution is rounded by 4e-9 r.m.s., below the
// 1.7e-8 of w itself, and the low word spans +-32, which even thousands of pairs on a
// cell rarely leave.
constexpr float kQuanta = 67108864.0f;

// First index in [lo, n) whose cell (high word of x) is at least v; steps: a power of two above n / 2.
__device__ __forceinline__ int lower_bound_cell(const uint64_t* x, int lo, int n, int steps, uint32_t v)
{
    const uint32_t* h = reinterpret_cast<const uint32_t*>(x) + 1;
    int pos = lo - 1;
    for (int s = steps; s > 0; s >>= 1)
        if (pos + s < n && h[2 * (pos + s)] < v) pos += s;
    return pos + 1;
}

// Items of a launch: counts per curve as a prefix in shared memory.
template <typename F>
__device__ __forceinline__ void item_prefix(int* pre, int nc, F count)
{
    if (threadIdx.x < 32) {
        int base = 0;
        for (int c0 = 0; c0 < nc; c0 += 32) {
            const int i = c0 + (int)threadIdx.x;
            int v = i < nc ? count(i) : 0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(0xffffffffu, v, o);
                if ((int)threadIdx.x >= o) v += t;
            }
            if (i < nc) pre[i + 1] = base + v;
            base += __shfl_sync(0xffffffffu, v, 31);
        }
        if (threadIdx.x == 0) pre[0] = 0;
    }
    __syncthreads();
}

__device__ __forceinline__ int item_curve(const int* pre, int nc, int item)
{
    int lo = 0, hi = nc - 1;
    while (lo < hi) {
        const int m = (lo + hi + 1) >> 1;
        if (pre[m] <= item) lo = m; else hi = m - 1;
    }
    return lo;
}

// A block's largest admissible value and largest magnitude: into the curve's maxima, the first
// also into the block's.  All threads call it.
template <int WARPS>
__device__ __forceinline__ void block_maxima(const SpecArgs& a, int c, int64_t blk, unsigned int key, unsigned int top,
                                             unsigned int (&s_key)[WARPS], unsigned int (&s_top)[WARPS])
{
    key = __reduce_max_sync(0xffffffffu, key);
    top = __reduce_max_sync(0xffffffffu, top);
    if ((threadIdx.x & 31) == 0) {
        s_key[threadIdx.x >> 5] = key;
        s_top[threadIdx.x >> 5] = top;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll
        for (int w = 1; w < WARPS; w++) {
            key = max(key, s_key[w]);
            top = max(top, s_top[w]);
        }
        if (key) atomicMax(a.vmax + c, key);
        if (top) atomicMax(a.vtop + c, top);
        a.vblk[blk] = key;
    }
    __syncthreads();
}

// INTERP: the weights are divided by the interpolation window's transform at the
// pair's time difference (all differences lie below half of the half period).
template <bool INTERP>
__global__ void __launch_bounds__(kSpreadThreads, 2) k_spec_spread(const SpecArgs a, int max_n)
{
    extern __shared__ __align__(16) unsigned char smem[];
    // low and high words of the cells A - margin .. A + seg + margin, then the curve's samples
    uint32_t* cl = reinterpret_cast<uint32_t*>(smem);
    const int words = a.seg_max + 2 * kSpreadMargin;
    int32_t* ch = reinterpret_cast<int32_t*>(cl + words);
    uint64_t* X = reinterpret_cast<uint64_t*>(ch + words);
    float* Y = reinterpret_cast<float*>(X + max_n);
    __shared__ int s_item, s_group;
    __shared__ int s_pre[kSpecMaxChunk + 1];
    const int tid = threadIdx.x, lane = tid & 31;
    const int nc = a.slot_end - a.slot_begin;
    item_prefix(s_pre, nc, [&](int i) {
        const SpecCurve& S = a.sc[a.order[a.slot_begin + i]];
        return S.nh ? (S.support + S.seg - 1) / S.seg : 0;
    });
    const int total = s_pre[nc];
    int loaded = -1;
    for (;;) {
        __syncthreads();
        if (tid == 0) s_item = (int)atomicAdd(a.queue, 1ull);
        __syncthreads();
        const int item = s_item;
        if (item >= total) break;
        const int ci = item_curve(s_pre, nc, item);
        const int c = a.order[a.slot_begin + ci];
        const SpecCurve S = a.sc[c];
        const CurveParams& P = a.cp[c];
        const int n = P.n;
        if (ci != loaded) {
            for (int i = tid; i < n; i += kSpreadThreads) {
                X[i] = a.xs[P.off + i];
                Y[i] = a.ys[P.off + i];
            }
            loaded = ci;
        }
        const int H = (int)S.H;
        const int A = (item - s_pre[ci]) * S.seg, B = min(A + S.seg, S.support), len = B - A;
        if (tid == 0) s_group = 0;
        for (int i = tid; i < (len + 2 * kSpreadMargin) / 4; i += kSpreadThreads) {
            reinterpret_cast<uint4*>(cl)[i] = make_uint4(0x80000000u, 0x80000000u, 0x80000000u, 0x80000000u);
            reinterpret_cast<int4*>(ch)[i] = make_int4(0, 0, 0, 0);
        }
        __syncthreads();
        const float iph = P.ip_hi, ipl = P.ip_lo;
        const float inv_h = 1.0f / (float)H;
        const uint64_t span = X[n - 1];
        // folded interval of the differences that touch the segment (window half-width 4, half-cell
        // centres, differences of whole cells off by one at most; a pair that whole cells put on the
        // wrong side of a fold lands in the margin there, which folds it back)
        const int flo = A - 6 > 0 ? A - 6 : 0, fhi = B + 6 < H ? B + 6 : H;
        int steps = 1;
        while (steps < n) steps <<= 1;
        // (fold, row group) go to the warps as they become free
        const int groups = (n + kSpreadRows - 1) / kSpreadRows;
        const int folds = (int)(span / ((uint64_t)H << 32)) + 1;
        const uint64_t shift = ((uint64_t)(uint32_t)(kSpreadMargin - A) << 32) - 0x80000000ull;
        for (;;) {
            int ticket = 0;
            if (lane == 0) ticket = atomicAdd(&s_group, 1);
            ticket = __shfl_sync(0xffffffffu, ticket, 0);
            if (ticket >= folds * groups) break;
            const int r = ticket / groups, g = ticket - r * groups;
            const bool odd = r & 1;
            const uint32_t ulo = odd ? (uint32_t)(r + 1) * H - fhi : (uint32_t)r * H + flo;
            const uint32_t uhi = odd ? (uint32_t)(r + 1) * H - flo : (uint32_t)r * H + fhi;
            if (ulo > (uint32_t)(span >> 32) + 1u) continue;
            // cell position of a difference d: +-(d - fold) less half a cell, relative to A - margin
            const uint64_t fold = (uint64_t)(odd ? r + 1 : r) * (uint64_t)H << 32;
            {
                const int row = min(g * kSpreadRows + (lane & (kSpreadRows - 1)), n - 1);
                const int bound = lower_bound_cell(X, row + 1, n, steps, (uint32_t)(X[row] >> 32) + (lane < kSpreadRows ? ulo : uhi));
                int cnt = __shfl_down_sync(0xffffffffu, bound, kSpreadRows) - bound;   // lanes below kSpreadRows
                if (lane >= kSpreadRows || g * kSpreadRows + lane >= n) cnt = 0;
                int incl = cnt;
#pragma unroll
                for (int o = 1; o < kSpreadRows; o <<= 1) {
                    const int t = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += t;
                }
                const int np = __shfl_sync(0xffffffffu, incl, kSpreadRows - 1);
                const int start = bound - (incl - cnt);      // j of pair p of this row: start + p
                for (int p0 = 0; p0 < np; p0 += 32) {
                    const int p = p0 + lane;
                    // row of pair p: how many rows end at or before it
                    int q = 0;
#pragma unroll
                    for (int o = kSpreadRows / 2; o > 0; o >>= 1) {
                        const int e = __shfl_sync(0xffffffffu, incl, q + o - 1);
                        if (e <= p) q += o;
                    }
                    const int j = __shfl_sync(0xffffffffu, start, q) + p;
                    if (p < np) {
                        const int i = g * kSpreadRows + q;
                        const uint64_t d = X[j] - X[i];
                        const uint64_t u = (odd ? fold - d : d - fold) + shift;
                        const int t = (int)(u >> 32);
                        const float z = (float)(uint32_t)u * 2.3283064365386963e-10f - 0.5f;
                        float w = ((gauss_g(Y[i], Y[j]) - iph) - ipl) * kQuanta;
                        if (INTERP) w *= kb_inverse(((float)(t + A - kSpreadMargin) + (z + 1.0f)) * inv_h);
                        float k[8];
                        kb_weights(z, k);
                        if ((unsigned)(t - 3) <= (unsigned)(len + 2 * kSpreadMargin - 8)) {
                            uint32_t* at = cl + (t - 3);
                            int up[8], any = 0;
#pragma unroll
                            for (int m = 0; m < 8; m++) {
                                const int v = __float2int_rn(w * k[m]);
                                const uint32_t old = atomicAdd(at + m, (uint32_t)v);
                                up[m] = (v >> 31) + (old + (uint32_t)v < old ? 1 : 0);
                                any |= up[m];
                            }
                            if (any) {
#pragma unroll
                                for (int m = 0; m < 8; m++)
                                    if (up[m]) atomicAdd(ch + (t - 3) + m, up[m]);
                            }
                        }
                    }
                }
            }
        }
        __syncthreads();
        // cells 4b .. 4b + 3 in the order of the half-length transform: g[2j] at j, g[2j+1] from the
        // end, two reals per complex value
        float2* x = a.x + (int64_t)ci * a.x_ld;
        const int Q = H >> 1;
        auto cell = [&](int t) {
            return fmaf((float)ch[t], 64.0f, (float)(int)(cl[t] - 0x80000000u) * (1.0f / kQuanta));
        };
        for (int b = tid; b < len >> 2; b += kSpreadThreads) {
            const int4 h = reinterpret_cast<const int4*>(ch + kSpreadMargin)[b];
            const uint4 l = reinterpret_cast<const uint4*>(cl + kSpreadMargin)[b];
            float g[4] = {fmaf((float)h.x, 64.0f, (float)(int)(l.x - 0x80000000u) * (1.0f / kQuanta)),
                          fmaf((float)h.y, 64.0f, (float)(int)(l.y - 0x80000000u) * (1.0f / kQuanta)),
                          fmaf((float)h.z, 64.0f, (float)(int)(l.z - 0x80000000u) * (1.0f / kQuanta)),
                          fmaf((float)h.w, 64.0f, (float)(int)(l.w - 0x80000000u) * (1.0f / kQuanta))};
            if (A == 0 && b < kSpreadMargin / 4) {            // cell -1 - i folds to cell i
#pragma unroll
                for (int m = 0; m < 4; m++) g[m] += cell(kSpreadMargin - 1 - (4 * b + m));
            }
            if (B == H && 4 * b + 4 > len - kSpreadMargin) {  // cell H + i folds to cell H - 1 - i
#pragma unroll
                for (int m = 0; m < 4; m++) g[m] += cell(kSpreadMargin + 2 * len - 1 - (4 * b + m));
            }
            const int bb = (A >> 2) + b;
            x[bb] = make_float2(g[0], g[2]);
            x[Q - 1 - bb] = make_float2(g[3], g[1]);
        }
    }
}

// ===========================================================================
// Complex transforms in registers and shared memory.  512 threads hold 8192
// points, 16 each: radix-16 steps, the last one 2, 4 or 8.  Complex values are
// f32x2 pairs, so an addition is one instruction; 64 registers a thread let two
// CTAs share an SM, one's loads and barriers under the other's arithmetic.
// 64 curves of 300 to 1,000 samples at 49,981 frequencies: first pass 149 us
// (2.8 TB/s, ALU 34 %, FMA 21 %), second 190 us (2.5 TB/s, ALU 40 %, FMA 34 %): held by
// the chain load, steps with their barriers, store of two blocks an SM, not by one unit.
// ===========================================================================
constexpr int kFftThreads = 512;
constexpr int kFftPoints = 16 * kFftThreads;

typedef f2 cx;                                   // (re, im)
__device__ __forceinline__ cx cadd(cx a, cx b) { return add2(a, b); }
__device__ __forceinline__ cx csub(cx a, cx b) { return fma2(b, pk(-1.f, -1.f), a); }
__device__ __forceinline__ cx cmul(cx a, cx b)
{
    float ax, ay, bx, by;
    upk(a, ax, ay);
    upk(b, bx, by);
    return fma2(pk(ax, ax), b, mul2(pk(ay, ay), pk(-by, bx)));
}
__device__ __forceinline__ cx cmi(cx a)          // times -i
{
    float x, y;
    upk(a, x, y);
    return pk(y, -x);
}

__device__ __forceinline__ void dft4(cx& a, cx& b, cx& c, cx& d)
{
    const cx s0 = cadd(a, c), s1 = csub(a, c), s2 = cadd(b, d), s3 = csub(b, d);
    a = cadd(s0, s2);
    c = csub(s0, s2);
    float x1, y1, x3, y3;
    upk(s1, x1, y1);
    upk(s3, x3, y3);
    b = pk(x1 + y3, y1 - x3);                    // s1 - i s3
    d = pk(x1 - y3, y1 + x3);
}

template <int R>
__device__ __forceinline__ void dft(cx* v)
{
    constexpr float h = 0.70710678118654752f;
    if constexpr (R == 2) {
        const cx t = csub(v[0], v[1]);
        v[0] = cadd(v[0], v[1]);
        v[1] = t;
    } else if constexpr (R == 4) {
        dft4(v[0], v[1], v[2], v[3]);
    } else if constexpr (R == 8) {
        dft4(v[0], v[2], v[4], v[6]);
        dft4(v[1], v[3], v[5], v[7]);
        // even part E_k = v[2k], odd part O_k = v[2k + 1]
        const cx o0 = v[1], o1 = cmul(v[3], pk(h, -h)), o2 = cmi(v[5]), o3 = cmul(v[7], pk(-h, -h));
        const cx e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6];
        v[0] = cadd(e0, o0); v[4] = csub(e0, o0);
        v[1] = cadd(e1, o1); v[5] = csub(e1, o1);
        v[2] = cadd(e2, o2); v[6] = csub(e2, o2);
        v[3] = cadd(e3, o3); v[7] = csub(e3, o3);
    } else {
        constexpr float c1 = 0.92387953251128674f, s1 = 0.38268343236508977f;
#pragma unroll
        for (int k = 0; k < 4; k++) dft4(v[k], v[k + 4], v[k + 8], v[k + 12]);
        // v[k + 4 q] holds part q of column k: twiddle exp(-2 pi i k q / 16), then across the columns
        v[5] = cmul(v[5], pk(c1, -s1));
        v[9] = cmul(v[9], pk(h, -h));
        v[13] = cmul(v[13], pk(s1, -c1));
        v[6] = cmul(v[6], pk(h, -h));
        v[10] = cmi(v[10]);
        v[14] = cmul(v[14], pk(-h, -h));
        v[7] = cmul(v[7], pk(s1, -c1));
        v[11] = cmul(v[11], pk(-h, -h));
        v[15] = cmul(v[15], pk(-c1, s1));
#pragma unroll
        for (int q = 0; q < 4; q++) dft4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
        // transpose: output q + 4 k from v[4 q + k]
#pragma unroll
        for (int q = 0; q < 4; q++)
#pragma unroll
            for (int k = q + 1; k < 4; k++) {
                const cx t = v[4 * q + k];
                v[4 * q + k] = v[4 * k + q];
                v[4 * k + q] = t;
            }
    }
}

// Twiddle factors exp(-2 pi i r k / (NS R)) of a step of radix R after NS points:
// [r - 1][k], k < NS, so that a warp's loads are consecutive.  Tables in one
// array: (16, 16), (16, 8), (256, 2), (256, 4), (256, 8), (256, 16), (4096, 2).
__host__ __device__ constexpr int tw_offset(int ns, int r)
{
    return ns == 16    ? (r == 16 ? 0 : 240)
           : ns == 256 ? 352 + 256 * (r == 2 ? 0 : r == 4 ? 1 : r == 8 ? 4 : 11)
                       : 352 + 256 * 26;
}

// Column c, element i of the block's 8192 points in shared memory (a pad every
// 16 elements; columns fastest in the first pass, elements in the second, whose
// columns start 4 elements apart in the banks).
template <int LOGN, bool CFAST>
__device__ __forceinline__ int fft_addr(int c, int i)
{
    constexpr int N = 1 << LOGN, C = kFftPoints / N;
    return CFAST ? (i + (i >> 4)) * C + c : c * (N + N / 16 + 4) + i + (i >> 4);
}

// On entry v[r] = element j + r N/16 of column c (j < N/16).  On return v[b R + r]
// = element j + b N/16 + r N/R of the transform, R the last radix.  `on` masks
// idle threads (every thread takes the barriers).
template <int LOGN, int DONE, bool CFAST>
__device__ __forceinline__ void fft_rest(cx* v, cx* sm, const cx* __restrict__ tw, int c, int j, bool on)
{
    constexpr int N = 1 << LOGN, NT = N / 16;
    constexpr int LEFT = LOGN - DONE;                 // bits still to do
    if constexpr (LEFT > 0) {
        constexpr int R = LEFT >= 4 ? 16 : (1 << LEFT);
        constexpr int NS = 1 << DONE, B = 16 / R;
        __syncthreads();
        if (on) {
#pragma unroll
            for (int b = 0; b < B; b++)
#pragma unroll
                for (int r = 0; r < R; r++) v[b * R + r] = sm[fft_addr<LOGN, CFAST>(c, j + b * NT + r * (N / R))];
        }
#pragma unroll
        for (int b = 0; b < B; b++) {
            const int k = (j + b * NT) & (NS - 1);
#pragma unroll
            for (int r = 1; r < R; r++)
                v[b * R + r] = cmul(v[b * R + r], __ldg(tw + tw_offset(NS, R) + (r - 1) * NS + k));
            dft<R>(v + b * R);
        }
        if constexpr (LEFT > 4) {
            __syncthreads();
            if (on) {
#pragma unroll
                for (int b = 0; b < B; b++) {
                    const int jj = j + b * NT, k = jj & (NS - 1);
#pragma unroll
                    for (int r = 0; r < R; r++) sm[fft_addr<LOGN, CFAST>(c, (jj - k) * R + k + r * NS)] = v[b * R + r];
                }
            }
            fft_rest<LOGN, DONE + 4, CFAST>(v, sm, tw, c, j, on);
        }
    }
}

template <int LOGN, bool CFAST>
__device__ __forceinline__ void fft_block(cx* v, cx* sm, const cx* __restrict__ tw, int c, int j, bool on)
{
    dft<16>(v);
    if (on) {
#pragma unroll
        for (int r = 0; r < 16; r++) sm[fft_addr<LOGN, CFAST>(c, j * 16 + r)] = v[r];
    }
    fft_rest<LOGN, 4, CFAST>(v, sm, tw, c, j, on);
}

// exp(-2 pi i U / 2^32)
__device__ __forceinline__ cx cis_neg(uint32_t U)
{
    float s, c;
    sincos2pi_turns(U, s, c);
    return pk(c, -s);
}

// sin and cos of x, |x| <= pi / 4, by Taylor polynomials (remainders below 2e-9)
__device__ __forceinline__ void sincos_small(float x, float& s, float& c)
{
    const float x2 = x * x;
    float p = fmaf(x2, 1.0f / 362880.0f, -1.0f / 5040.0f);
    p = fmaf(x2, p, 1.0f / 120.0f);
    p = fmaf(x2, p, -1.0f / 6.0f);
    s = fmaf(x2 * x, p, x);
    float q = fmaf(x2, -1.0f / 3628800.0f, 1.0f / 40320.0f);
    q = fmaf(x2, q, -1.0f / 720.0f);
    q = fmaf(x2, q, 1.0f / 24.0f);
    q = fmaf(x2, q, -0.5f);
    c = fmaf(x2, q, 1.0f);
}

// Bits of the second pass's length.  512 points make 16 rows of a block, so its
// eight mirror pairs write 32-byte runs; longer ones only where the first pass
// would exceed 2048.
__host__ __device__ constexpr int spec_log2(int logq)
{
    return logq >= 20 ? (logq - 11 > 9 ? logq - 11 : 9) : logq >= 18 ? 9 : logq >> 1;
}

constexpr int fft_smem_floats2() { return kFftPoints + kFftPoints / 16 + 4 * 64; }

template <int LOGN>
__device__ __forceinline__ void fft1_item(const SpecArgs& a, const SpecCurve& S, cx* x, int blk, cx* sm)
{
    constexpr int N = 1 << LOGN, C = kFftPoints / N, NT = N / 16;
    constexpr int LEFT = (LOGN & 3) == 0 ? 4 : (LOGN & 3);
    constexpr int R = 1 << LEFT, B = 16 / R;
    const int tid = threadIdx.x, c = tid % C, j = tid / C;
    const int Q = 1 << S.logq, log2q = S.logq - LOGN;
    const int col = blk * C + c;
    const int zlo = S.support >> 2, zhi = Q - zlo;       // x is zero in [zlo, zhi)
    cx v[16];
#pragma unroll
    for (int r = 0; r < 16; r++) {
        const int l = ((j + r * NT) << log2q) + col;
        v[r] = l < zlo || l >= zhi ? x[l] : 0ull;
    }
    fft_block<LOGN, true>(v, sm, reinterpret_cast<const cx*>(a.tw), c, j, true);
    // times exp(-2 pi i k1 col / Q), k1 = j + b NT + r N/R: one sine and cosine each for j, NT and N/R,
    // the others by products
    const int sh = 32 - S.logq;
    const cx sr = cis_neg((uint32_t)((N / R) * col) << sh);
    const cx sb = B > 1 ? cis_neg((uint32_t)(NT * col) << sh) : 0ull;
    cx wb = cis_neg((uint32_t)(j * col) << sh);
    cx* xo = x + ((int64_t)j << log2q) + col;
#pragma unroll
    for (int b = 0; b < B; b++) {
        cx w = wb;
#pragma unroll
        for (int r = 0; r < R; r++) {
            xo[(b * NT + r * (N / R)) << log2q] = cmul(v[b * R + r], w);
            if (r + 1 < R)      // every fourth afresh: products of at most three roundings
                w = (r & 3) == 3 ? cis_neg((uint32_t)((j + b * NT + (r + 1) * (N / R)) * col) << sh) : cmul(w, sr);
        }
        if (b + 1 < B) wb = cmul(wb, sb);
    }
}

__global__ void __launch_bounds__(kFftThreads, 2) k_spec_fft1(const SpecArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    cx* sm = reinterpret_cast<cx*>(smem);
    __shared__ int s_pre[kSpecMaxChunk + 1];
    const int nc = a.slot_end - a.slot_begin;
    item_prefix(s_pre, nc, [&](int i) {
        const SpecCurve& S = a.sc[a.order[a.slot_begin + i]];
        return S.nh && S.logq > kSpecOneLogQ ? 1 << (S.logq - 13) : 0;
    });
    for (int item = blockIdx.x; item < s_pre[nc]; item += gridDim.x) {
        const int ci = item_curve(s_pre, nc, item);
        const SpecCurve S = a.sc[a.order[a.slot_begin + ci]];
        cx* x = reinterpret_cast<cx*>(a.x + (int64_t)ci * a.x_ld);
        const int blk = item - s_pre[ci];
        switch (S.logq - spec_log2(S.logq)) {
        case 7: fft1_item<7>(a, S, x, blk, sm); break;
        case 8: fft1_item<8>(a, S, x, blk, sm); break;
        case 9: fft1_item<9>(a, S, x, blk, sm); break;
        case 10: fft1_item<10>(a, S, x, blk, sm); break;
        default: fft1_item<11>(a, S, x, blk, sm); break;
        }
        __syncthreads();
    }
}

// The four pair-spectrum values of X[m] and X[Q - m] (x the transform of the
// packed reals): V the half-length real transform, C[m] = Re(c_m V[m]),
// C[H - m] = -Im(c_m V[m]), c_m = exp(-i pi m / (2 H)).
__device__ __forceinline__ void spec_emit(const SpecCurve& S, float* P, int m, cx pa, cx pb)
{
    const int Q = 1 << S.logq, H = 2 * Q;
    const float inv_h = 1.0f / (float)H, fm = (float)m;      // m <= Q / 2 (or the row Q1 / 2's up to Q)
    float xa, ya, xb, yb;
    upk(pa, xa, ya);
    upk(pb, xb, yb);
    const float ex = 0.5f * (xa + xb), ey = 0.5f * (ya - yb), ox = 0.5f * (ya + yb), oy = -0.5f * (xa - xb);
    float s4, c4, sm_, cm;
    sincos2pi_turns((uint32_t)m << (31 - S.logq), s4, c4);
    sincos_small((float)(0.5 * CP_PI) * fm * inv_h, sm_, cm);                // pi m / (2 H) <= pi / 4
    const float wx = fmaf(c4, ox, s4 * oy), wy = fmaf(c4, oy, -s4 * ox);     // exp(-i a) O
    // V[m] = E + W O times c_m = exp(-i pi m / (2 H)); V[Q - m] = conj(E - W O), c_{Q-m} = exp(-i pi/4) conj(c_m)
    const float h = 0.70710678118654752f;
    const float ux = ex + wx, uy = ey + wy, dx = ex - wx, dy = wy - ey;
    const float qx = h * (cm + sm_), qy = h * (sm_ - cm);
    const int m2 = Q - m, m3 = H - m, m4 = Q + m;
    if (m < S.n_out) {
        const float p = fmaf(cm, ux, sm_ * uy) * kb_inverse(fm * inv_h);
        P[m] = p;
        if (m <= 4) P[-m] = p;                            // the interpolation reads across 0
    }
    if (m2 < S.n_out) P[m2] = fmaf(qx, dx, -qy * dy) * kb_inverse((float)m2 * inv_h);
    if (m3 < S.n_out) P[m3] = fmaf(sm_, ux, -cm * uy) * kb_inverse((float)m3 * inv_h);
    if (m4 < S.n_out) P[m4] = -fmaf(qx, dy, qy * dx) * kb_inverse((float)m4 * inv_h);
}

template <int LOGN>
__device__ __forceinline__ void fft2_item(const SpecArgs& a, const SpecCurve& S, const cx* x, float* P, int blk, cx* sm)
{
    constexpr int N = 1 << LOGN, C = kFftPoints / N, NT = N / 16;
    constexpr int LEFT = (LOGN & 3) == 0 ? 4 : (LOGN & 3);
    constexpr int R = 1 << LEFT, B = 16 / R;
    const int tid = threadIdx.x, c = tid / NT, j = tid % NT;
    const int Q1 = 1 << (S.logq - LOGN);
    const int a0 = blk * (C / 2);
    // rows a0 .. a0 + C/2 - 1 and their mirror rows Q1 - a (row 0 with row Q1 / 2: each its own mirror)
    const int ar = a0 + (c < C / 2 ? c : c - C / 2);
    const int row = c < C / 2 ? ar : (ar == 0 ? Q1 >> 1 : Q1 - ar);
    cx v[16];
#pragma unroll
    for (int r = 0; r < 16; r++) v[r] = x[((int64_t)row << LOGN) + j + r * NT];
    fft_block<LOGN, false>(v, sm, reinterpret_cast<const cx*>(a.tw), c, j, true);
    __syncthreads();
#pragma unroll
    for (int b = 0; b < B; b++)
#pragma unroll
        for (int r = 0; r < R; r++) sm[fft_addr<LOGN, false>(c, j + b * NT + r * (N / R))] = v[b * R + r];
    __syncthreads();
    for (int it = tid; it < (C / 2) * N; it += kFftThreads) {
        const int ca = it % (C / 2), k2 = it / (C / 2);
        const int aa = a0 + ca;
        if (aa > 0) {
            spec_emit(S, P, aa + Q1 * k2, sm[fft_addr<LOGN, false>(ca, k2)],
                      sm[fft_addr<LOGN, false>(ca + C / 2, N - 1 - k2)]);
        } else if (k2 <= N / 2) {
            spec_emit(S, P, Q1 * k2, sm[fft_addr<LOGN, false>(0, k2)],
                      sm[fft_addr<LOGN, false>(0, (N - k2) & (N - 1))]);
            if (k2 < N / 2)
                spec_emit(S, P, (Q1 >> 1) + Q1 * k2, sm[fft_addr<LOGN, false>(C / 2, k2)],
                          sm[fft_addr<LOGN, false>(C / 2, N - 1 - k2)]);
        }
    }
}

__global__ void __launch_bounds__(kFftThreads, 2) k_spec_fft2(const SpecArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    cx* sm = reinterpret_cast<cx*>(smem);
    __shared__ int s_pre[kSpecMaxChunk + 1];
    __shared__ int s_next;
    const int nc = a.slot_end - a.slot_begin;
    item_prefix(s_pre, nc, [&](int i) {
        const SpecCurve& S = a.sc[a.order[a.slot_begin + i]];
        return S.nh && S.logq > kSpecOneLogQ ? 1 << (S.logq - 13) : 0;
    });
    // Items are started in order, by ticket: the runs that neighbouring items write are half a sector
    // each above 2^19 points, and meet in L2 only if their blocks keep together (71 curves of 2^20
    // points in one launch: 1400 us with a fixed stride of the grid, against 960 in three launches).
    int item = blockIdx.x;
    while (item < s_pre[nc]) {
        int next = 0;
        if (threadIdx.x == 0) next = (int)gridDim.x + (int)atomicAdd(a.queue + 1, 1ull);
        const int ci = item_curve(s_pre, nc, item);
        const SpecCurve S = a.sc[a.order[a.slot_begin + ci]];
        const cx* x = reinterpret_cast<const cx*>(a.x + (int64_t)ci * a.x_ld);
        float* P = a.P + (int64_t)ci * a.p_ld + kSpecPad;
        const int blk = item - s_pre[ci];
        switch (spec_log2(S.logq)) {
        case 7: fft2_item<7>(a, S, x, P, blk, sm); break;
        case 8: fft2_item<8>(a, S, x, P, blk, sm); break;
        case 9: fft2_item<9>(a, S, x, P, blk, sm); break;
        case 10: fft2_item<10>(a, S, x, P, blk, sm); break;
        default: fft2_item<11>(a, S, x, P, blk, sm); break;
        }
        __syncthreads();
        if (threadIdx.x == 0) s_next = next;
        __syncthreads();
        item = s_next;
    }
}

// Short transforms (Q <= 8192): one CTA per curve, both passes in one.
template <int LOGN>
__device__ __forceinline__ void fft_one(const SpecArgs& a, const SpecCurve& S, const cx* x, float* P, cx* sm)
{
    constexpr int N = 1 << LOGN, NT = N / 16;
    constexpr int LEFT = (LOGN & 3) == 0 ? 4 : (LOGN & 3);
    constexpr int R = 1 << LEFT, B = 16 / R;
    const int tid = threadIdx.x;
    const bool on = tid < NT;
    const int j = on ? tid : 0;
    const int zlo = S.support >> 2, zhi = N - zlo;
    cx v[16];
#pragma unroll
    for (int r = 0; r < 16; r++) {
        const int l = j + r * NT;
        v[r] = l < zlo || l >= zhi ? x[l] : 0ull;
    }
    fft_block<LOGN, false>(v, sm, reinterpret_cast<const cx*>(a.tw), 0, j, on);
    __syncthreads();
    if (on) {
#pragma unroll
        for (int b = 0; b < B; b++)
#pragma unroll
            for (int r = 0; r < R; r++) sm[fft_addr<LOGN, false>(0, j + b * NT + r * (N / R))] = v[b * R + r];
    }
    __syncthreads();
    for (int k = tid; k <= N / 2; k += kFftThreads)
        spec_emit(S, P, k, sm[fft_addr<LOGN, false>(0, k)], sm[fft_addr<LOGN, false>(0, (N - k) & (N - 1))]);
}

__global__ void __launch_bounds__(kFftThreads, 2) k_spec_fft_one(const SpecArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    cx* sm = reinterpret_cast<cx*>(smem);
    const int ci = blockIdx.x;
    const SpecCurve S = a.sc[a.order[a.slot_begin + ci]];
    if (!S.nh || S.logq > kSpecOneLogQ) return;
    const cx* x = reinterpret_cast<const cx*>(a.x + (int64_t)ci * a.x_ld);
    float* P = a.P + (int64_t)ci * a.p_ld + kSpecPad;
    switch (S.logq) {
    case 8: fft_one<8>(a, S, x, P, sm); break;
    case 9: fft_one<9>(a, S, x, P, sm); break;
    case 10: fft_one<10>(a, S, x, P, sm); break;
    case 11: fft_one<11>(a, S, x, P, sm); break;
    case 12: fft_one<12>(a, S, x, P, sm); break;
    default: fft_one<13>(a, S, x, P, sm); break;
    }
}

// ===========================================================================
// k_spec_sum: nCKP at every trial frequency from the pair spectrum.  The n-th
// harmonic of neighbouring frequencies lies n entries apart: bound by the sectors
// these gathers move through L2 (57 % of its rate) and their latency, four
// frequencies a thread and four harmonics in flight (64 curves at 49,981: 74 us).
// ===========================================================================
constexpr int kSumThreads = 256;
constexpr int kSumPer = 4;                        // frequencies per thread

__global__ void __launch_bounds__(kSumThreads) k_spec_sum(const SpecArgs a)
{
    __shared__ int s_pre[kSpecMaxChunk + 1];
    __shared__ float s_a[kSpecMaxHarm];
    __shared__ unsigned int s_key[kSumThreads / 32], s_top[kSumThreads / 32];
    const int tid = threadIdx.x;
    const int nc = a.slot_end - a.slot_begin;
    const int blocks = (int)((a.n_freq + kSumThreads * kSumPer - 1) / (kSumThreads * kSumPer));
    item_prefix(s_pre, nc, [&](int i) { return a.sc[a.order[a.slot_begin + i]].nh ? blocks : 0; });
    for (int item = blockIdx.x; item < s_pre[nc]; item += gridDim.x) {
        const int ci = item_curve(s_pre, nc, item);
        const int c = a.order[a.slot_begin + ci];
        const SpecCurve S = a.sc[c];
        const CurveParams& P = a.cp[c];
        if (tid < S.nh) s_a[tid] = a.coef[(int64_t)c * kSpecMaxHarm + tid];
        __syncthreads();
        const float* Ps = a.P + (int64_t)ci * a.p_ld + kSpecPad;
        const int64_t k0 = (int64_t)(item - s_pre[ci]) * (kSumThreads * kSumPer) + tid;
        int m[kSumPer];
        float s[kSumPer];
        int at[kSumPer];
#pragma unroll
        for (int q = 0; q < kSumPer; q++) {
            const int64_t k = min(k0 + q * kSumThreads, a.n_freq - 1);
            m[q] = (int)(a.m0 + a.mq * k);
            at[q] = 0;
            s[q] = 0.f;
        }
#pragma unroll 4
        for (int h = 0; h < S.nh; h++) {
            const float an = s_a[h];
#pragma unroll
            for (int q = 0; q < kSumPer; q++) {
                at[q] += m[q];
                s[q] = fmaf(an, Ps[at[q]], s[q]);
            }
        }
        unsigned int key = 0u, top = 0u;
        float* row = a.rows + (a.rows_by_curve ? (int64_t)c : (int64_t)ci) * a.row_ld;
#pragma unroll
        for (int q = 0; q < kSumPer; q++) {
            const int64_t k = k0 + q * kSumThreads;
            if (k < a.n_freq) {
                const float v = fmaf(2.0f, s[q], P.diag * S.one_minus_a0) * P.norm;
                row[k] = v;
                top = max(top, __float_as_uint(fabsf(v)));
                if (!excluded_k(a.ex.full_k, a.ex.n, k)) key = max(key, orderable(v));
            }
        }
        block_maxima(a, c, (int64_t)ci * a.vb_ld + (item - s_pre[ci]), key, top, s_key, s_top);
    }
}

// ===========================================================================
// k_spec_interp: the same at any frequencies (a uniform grid, fine windows, the
// trial list), each harmonic interpolated from 8 pair-spectrum values.  The
// position n f L is an integer multiple of the fixed-point f L (32.32).
// ===========================================================================
constexpr int kInterpBlock = kSumThreads / 4;      // frequencies per block of the interpolation
static_assert(kInterpBlock == kSpecBlock, "block maxima");

__device__ __forceinline__ int spec_count(const SpecArgs& a, int c)
{
    return a.stage == kSpecFine ? a.n_peaks[c] * (2 * a.fine_half + 1) : a.stage == kSpecList ? a.n_trials : (int)a.n_freq;
}

__global__ void __launch_bounds__(kSumThreads) k_spec_interp(const SpecArgs a)
{
    __shared__ int s_pre[kSpecMaxChunk + 1];
    __shared__ float s_a[kSpecMaxHarm];
    __shared__ unsigned int s_key[kSumThreads / 32], s_top[kSumThreads / 32];
    const int tid = threadIdx.x;
    const int nc = a.slot_end - a.slot_begin;
    item_prefix(s_pre, nc, [&](int i) {
        const int c = a.order[a.slot_begin + i];
        return a.sc[c].nh && !a.sc[c].whole ? (spec_count(a, c) + kInterpBlock - 1) / kInterpBlock : 0;
    });
    for (int item = blockIdx.x; item < s_pre[nc]; item += gridDim.x) {
        const int ci = item_curve(s_pre, nc, item);
        const int c = a.order[a.slot_begin + ci];
        const SpecCurve S = a.sc[c];
        const CurveParams& P = a.cp[c];
        if (tid < S.nh) s_a[tid] = a.coef[(int64_t)c * kSpecMaxHarm + tid];
        __syncthreads();
        const float* Ps = a.P + (int64_t)ci * a.p_ld + kSpecPad;
        // four threads a frequency, each every fourth harmonic (one thread's chain of up to 64
        // dependent fetches took 55 us a launch, however few the frequencies)
        const int q = (item - s_pre[ci]) * kInterpBlock + (tid >> 2), part = tid & 3;
        unsigned int key = 0u, top = 0u;
        const bool in = q < spec_count(a, c);
        bool ok = in, live = in;                  // admissible as the best; evaluated at all
        double f = 0.0;
        if (in) {
            if (a.stage == kSpecFine) {
                const int W = 2 * a.fine_half + 1, pk = q / W;
                const double fpk = grid_freq(a.f_min, (double)a.peaks[(int64_t)c * a.top_k + pk], a.coarse_df);
                f = grid_freq(fpk, (double)(q - pk * W - a.fine_half), a.step);
                live = f >= a.f_min && f <= a.f_max;
                ok = live && !excluded_f(a.ex, f);
            } else if (a.stage == kSpecList) {
                const int k = a.trials[(int64_t)c * a.n_trials + q];
                live = k >= 0;
                ok = live && !excluded_k(a.ex.full_k, a.ex.n, k);
                f = grid_freq(a.f_min, (double)max(k, 0), a.step);
            } else {
                f = grid_freq(a.f_min, (double)q, a.step);
                ok = a.stage == kSpecFull && !excluded_k(a.ex.full_k, a.ex.n, q);
            }
        }
        float s = 0.f;
        if (live) {
            const uint64_t step = (uint64_t)__double2ll_rn(f * S.L * 4294967296.0);
            uint64_t pos = step * (uint64_t)(part + 1);
#pragma unroll 2
            for (int h = part; h < S.nh; h += 4, pos += 4 * step) {
                    float w[8];
                    kb_weights((float)(uint32_t)pos * 2.3283064365386963e-10f - 0.5f, w);
                    const float* p = Ps + ((int)(pos >> 32) - 3);
                    float t = 0.f;
#pragma unroll
                    for (int k = 0; k < 8; k++) t = fmaf(w[k], p[k], t);
                    s = fmaf(s_a[h], t, s);
            }
        }
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        s += __shfl_xor_sync(0xffffffffu, s, 2);
        if (in && part == 0) {
            float v = live ? fmaf(2.0f, s, P.diag * S.one_minus_a0) * P.norm : 0.f;
            top = __float_as_uint(fabsf(v));
            if (a.stage == kSpecFine && !ok) v = -INFINITY;
            if (a.stage == kSpecList && !live) v = __int_as_float(0x7fc00000);
            a.rows[(a.rows_by_curve ? (int64_t)c : (int64_t)ci) * a.row_ld + q] = v;
            if (ok) key = orderable(v);
        }
        block_maxima(a, c, (int64_t)ci * a.vb_ld + (item - s_pre[ci]), key, top, s_key, s_top);
    }
}

// Margin below which two values of a curve are not told apart by the spectrum:
// 1e-5 of the largest magnitude in the row, admissible or not (an excluded peak
// carries its error to the values beside it), plus 4e-6 + 7e-7 sqrt(N) of norm N, the
// scale of a noise curve.  The second part decides where the curve covers so little
// of a cycle that the whole row lies below that scale: the sums cancel there, and
// spectrum and pair sum drift apart near the top by up to 5e-6, 1.5e-5, 2.0e-5 and
// 2.9e-5 of norm N for N up to 100, 500, 1,500 and 4,096 (198,000 rows of random
// batches below norm N); above it by at most 0.76 of the first part alone.
__device__ __forceinline__ float spec_margin(float vtop, const CurveParams& P)
{
    const float n = (float)P.n;
    return 1e-5f * vtop + (4e-6f + 7e-7f * sqrtf(n)) * P.norm * n;
}

// ===========================================================================
// k_spec_select: the admissible entries (grid points, fine candidates, list
// positions) within the margin of the largest value, in ascending order: the pair
// sum's own best is among them.  A curve with more than kSpecCand of them (a
// constant curve), or without a spectrum, is evaluated whole by the pair sum.
// ===========================================================================
constexpr int kSelThreads = 256;

// Writes the n entries of s_k (distinct, any order) in ascending order, -1 after them.
__device__ __forceinline__ void write_sorted(const int32_t* s_k, int n, int32_t* out)
{
    const int tid = threadIdx.x;
    if (tid < kSpecCand) {
        if (tid >= n) {
            out[tid] = -1;
        } else {
            const int32_t k = s_k[tid];
            int rank = 0;
            for (int q = 0; q < n; q++) rank += s_k[q] < k;
            out[rank] = k;
        }
    }
}

__global__ void __launch_bounds__(kSelThreads) k_spec_select(const SpecArgs a)
{
    __shared__ int s_n, s_hot;
    __shared__ int32_t s_k[kSpecCand], s_blk[kSpecCand];
    const int ci = blockIdx.x, tid = threadIdx.x;
    const int c = a.order[a.slot_begin + ci];
    const CurveParams& P = a.cp[c];
    int32_t* out = a.cand + (int64_t)c * kSpecCand;
    if (tid == 0) s_n = 0;
    __syncthreads();
    const bool spec = a.sc[c].nh != 0 && !a.sc[c].whole;
    const unsigned int top = a.vmax[c];
    if (tid == 0) s_hot = 0;
    __syncthreads();
    if (spec && top) {
        const float thr = from_orderable(top) - spec_margin(__uint_as_float(a.vtop[c]), P);
        const unsigned int othr = orderable(thr);
        const float* row = a.rows + (a.rows_by_curve ? (int64_t)c : (int64_t)ci) * a.row_ld;
        const int count = spec_count(a, c), per = a.interp ? kInterpBlock : kSumThreads * kSumPer;
        // only the blocks whose largest admissible value reaches the threshold are read again
        for (int b = tid; b * per < count; b += kSelThreads)
            if (a.vblk[(int64_t)ci * a.vb_ld + b] >= othr) {
                const int pos = atomicAdd(&s_hot, 1);
                if (pos < kSpecCand) s_blk[pos] = b;
            }
        __syncthreads();
        const int hot = s_hot;
        if (hot > kSpecCand) {                       // at least as many entries
            if (tid == 0) s_n = hot;
        } else {
            for (int h = 0; h < hot; h++) {
                const int k1 = min(count, (s_blk[h] + 1) * per);
                for (int k = s_blk[h] * per + tid; k < k1; k += kSelThreads) {
                    if (row[k] >= thr) {
                        const int g = a.stage == kSpecList ? a.trials[(int64_t)c * a.n_trials + k] : k;
                        if (a.stage != kSpecFine && excluded_k(a.ex.full_k, a.ex.n, g)) continue;
                        const int pos = atomicAdd(&s_n, 1);
                        if (pos < kSpecCand) s_k[pos] = k;
                    }
                }
            }
        }
    }
    __syncthreads();
    const int n = s_n;
    const bool whole = !spec || n > kSpecCand || (top && n == 0);
    write_sorted(s_k, whole ? 0 : n, out);
    if (tid == 0 && whole) a.fb_slots[atomicAdd(a.fb_count, 1)] = a.slot_begin + ci;
}

// ===========================================================================
// k_spec_peaks: the coarse points whose exact values decide the top_k peaks.
// With m the margin: T = the top_k-th largest value that is a local maximum by
// more than m (radix select on the value bits); every point that may be a local
// maximum within m and lies above T - m, and any neighbour within m of it.  The
// pair sum evaluates them again, and k_spec_rank ranks them from exact values;
// every other comparison is decided by more than the margin.
// ===========================================================================
constexpr int kPeakRaw = 256;
constexpr int kPeakThreads = 1024;
constexpr int kPeakRow = 24576;                  // row points kept in shared memory

__global__ void __launch_bounds__(kPeakThreads) k_spec_peaks(const SpecArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ unsigned int s_hist[256], s_prefix, s_need;
    __shared__ int s_n, s_m;
    __shared__ int32_t s_raw[kPeakRaw], s_k[kSpecCand];
    const int ci = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int c = a.order[a.slot_begin + ci];
    const CurveParams& P = a.cp[c];
    int32_t* out = a.cand + (int64_t)c * kSpecCand;
    const int K = (int)a.n_freq;
    const float* v = a.rows + (int64_t)c * a.row_ld;
    if (a.sc[c].nh == 0) {
        if (tid < kSpecCand) out[tid] = -1;
        if (tid == 0) {
            a.n_peaks[c] = 0;
            a.fb_slots[atomicAdd(a.fb_count, 1)] = a.slot_begin + ci;
        }
        return;
    }
    if (K <= kPeakRow) {
        float* row = reinterpret_cast<float*>(smem);
        for (int k = tid; k < K; k += kPeakThreads) row[k] = v[k];
        v = row;
    }
    const float vm = __uint_as_float(a.vtop[c]);         // the row's largest magnitude
    if (tid == 0) {
        s_n = 0;
        s_m = 0;
        s_prefix = 0u;
        s_need = (unsigned)a.top_k;
    }
    __syncthreads();
    const float m = spec_margin(vm, P);
    auto sure = [&](int k) {
        const float x = v[k];
        return (k == 0 || x > v[k - 1] + m) && (k == K - 1 || x > v[k + 1] + m) && !excluded_k(a.ex.coarse_k, a.ex.n, k);
    };
    // the value of the top_k-th sure maximum (none so far down: every possible maximum counts)
    bool enough = true;
    for (int pass = 0; pass < 4 && enough; pass++) {
        const int shift = 24 - 8 * pass;
        for (int i = tid; i < 256; i += kPeakThreads) s_hist[i] = 0u;
        __syncthreads();
        const unsigned int prefix = s_prefix, need = s_need;
        for (int k = tid; k < K; k += kPeakThreads) {
            const unsigned int u = orderable(v[k]);
            if ((pass == 0 || (u >> (shift + 8)) == prefix) && sure(k)) atomicAdd(&s_hist[(u >> shift) & 255u], 1u);
        }
        __syncthreads();
        if (warp == 0) {
            // lane l owns digits 255 - 8l .. 248 - 8l; the one holding the need-th largest
            unsigned int h[8], sum = 0;
#pragma unroll
            for (int x = 0; x < 8; x++) sum += h[x] = s_hist[255 - 8 * lane - x];
            unsigned int incl = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned int y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            unsigned int cum = incl - sum;
            if (cum < need && need <= incl) {
                bool found = false;
#pragma unroll
                for (int x = 0; x < 8; x++) {
                    if (!found && cum + h[x] >= need) {
                        found = true;
                        s_prefix = (prefix << 8) | (255u - 8u * lane - x);
                        s_need = need - cum;
                    }
                    cum += h[x];
                }
            }
            if (lane == 31 && incl < need) s_need = 0u;      // fewer than top_k (first pass only)
        }
        __syncthreads();
        enough = s_need != 0u;
    }
    const float floor_v = enough ? from_orderable(s_prefix) - m : -INFINITY;
    for (int k = tid; k < K; k += kPeakThreads) {
        const float x = v[k];
        if (!(x >= floor_v) || excluded_k(a.ex.coarse_k, a.ex.n, k)) continue;
        const float l = k > 0 ? v[k - 1] : -INFINITY, h = k < K - 1 ? v[k + 1] : -INFINITY;
        if (x >= l - m && x >= h - m) {
            const int add = 1 + (x - l <= m ? 1 : 0) + (x - h <= m ? 1 : 0);
            int pos = atomicAdd(&s_n, add);
            if (pos + add <= kPeakRaw) {
                s_raw[pos++] = k;
                if (x - l <= m) s_raw[pos++] = k - 1;
                if (x - h <= m) s_raw[pos++] = k + 1;
            }
        }
    }
    __syncthreads();
    const int raw = s_n;
    if (raw <= kPeakRaw && tid < raw) {                  // distinct entries: the first of equal ones stays
        const int32_t k = s_raw[tid];
        bool first = true;
        for (int q = 0; q < tid; q++) first = first && s_raw[q] != k;
        if (first) {
            const int pos = atomicAdd(&s_m, 1);
            if (pos < kSpecCand) s_k[pos] = k;
        }
    }
    __syncthreads();
    const bool whole = raw > kPeakRaw || s_m > kSpecCand || !(vm < INFINITY);
    write_sorted(s_k, whole ? 0 : s_m, out);
    if (tid == 0 && whole) {
        a.sc[c].whole = 1;
        a.fb_slots[atomicAdd(a.fb_count, 1)] = a.slot_begin + ci;
    }
}

// k_spec_rank: the peaks of a curve from its candidates' exact values (the rule
// and order of k_topk).  One CTA of kSpecCand threads per curve.
__global__ void __launch_bounds__(kSpecCand) k_spec_rank(const SpecArgs a)
{
    __shared__ unsigned long long s_key[kSpecCand];
    const int tid = threadIdx.x;
    const int c = a.order[a.slot_begin + blockIdx.x];
    const float* v = a.rows + (int64_t)c * a.row_ld;
    const int K = (int)a.n_freq;
    const int k = a.cand[(int64_t)c * kSpecCand + tid];
    unsigned long long key = 0ull;
    if (k >= 0) {
        const float x = v[k];
        if ((k == 0 || x > v[k - 1]) && (k == K - 1 || x >= v[k + 1]) && !excluded_k(a.ex.coarse_k, a.ex.n, k))
            key = make_key(x, (uint32_t)k);
    }
    s_key[tid] = key;
    const int found = __syncthreads_count(key != 0ull);
    if (key) {
        int rank = 0;
        for (int q = 0; q < kSpecCand; q++) rank += s_key[q] > key;
        if (rank < a.top_k) a.peaks_out[(int64_t)c * a.top_k + rank] = k;
    }
    if (tid == 0) a.n_peaks[c] = min(found, a.top_k);
}

// ---------------------------------------------------------------------------
__global__ void k_spec_twiddle(float2* tw)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int ns[7] = {16, 16, 256, 256, 256, 256, 4096}, rr[7] = {16, 8, 2, 4, 8, 16, 2};
    for (int t = 0; t < 7; t++) {
        const int e = i - tw_offset(ns[t], rr[t]);
        if (e >= 0 && e < (rr[t] - 1) * ns[t]) {
            const int r = e / ns[t] + 1, k = e % ns[t];
            double s, c;
            sincospi(-2.0 * (double)(r * k) / (double)(ns[t] * rr[t]), &s, &c);
            tw[i] = make_float2((float)c, (float)s);
        }
    }
}

cudaError_t launch_spec_twiddle(float2* tw, cudaStream_t s)
{
    static_assert(tw_offset(4096, 2) + 4096 <= kSpecTwiddles, "twiddle tables");
    k_spec_twiddle<<<kSpecTwiddles / 256, 256, 0, s>>>(tw);
    return cudaGetLastError();
}

static size_t prep_smem(int np2max) { return (size_t)np2max * (sizeof(double) + sizeof(int32_t)); }
static size_t fft_smem() { return (size_t)fft_smem_floats2() * sizeof(float2); }

// Shared memory of the spreading kernel: two CTAs share an SM where the curve
// leaves room for at least 4096 cells each.
size_t spec_spread_smem(int max_n, int seg)
{
    return (size_t)max_n * (sizeof(uint64_t) + sizeof(float)) + 8 * (size_t)(seg + 2 * kSpreadMargin);
}

int spec_seg_max(int max_n)
{
    const size_t half = 112 * 1024;
    int seg = 4096;
    while (seg < 16384 && spec_spread_smem(max_n, seg + 512) <= half) seg += 512;
    return seg;
}

cudaError_t spec_prepare(int np2max, int max_n, int seg_max)
{
    cudaError_t e = raise_dyn_smem((const void*)k_spec_prep, prep_smem(np2max));
    if (e == cudaSuccess) e = raise_dyn_smem((const void*)k_spec_spread<false>, spec_spread_smem(max_n, seg_max));
    if (e == cudaSuccess) e = raise_dyn_smem((const void*)k_spec_spread<true>, spec_spread_smem(max_n, seg_max));
    if (e == cudaSuccess) e = raise_dyn_smem((const void*)k_spec_fft1, fft_smem());
    if (e == cudaSuccess) e = raise_dyn_smem((const void*)k_spec_fft2, fft_smem());
    if (e == cudaSuccess) e = raise_dyn_smem((const void*)k_spec_fft_one, fft_smem());
    if (e == cudaSuccess) e = raise_dyn_smem((const void*)k_spec_peaks, kPeakRow * sizeof(float));
    return e;
}

cudaError_t launch_spec_prep(const SpecArgs& a, cudaStream_t s)
{
    const int n = a.slot_end - a.slot_begin;
    if (n <= 0) return cudaSuccess;
    k_spec_prep<<<n, kSpecPrepThreads, prep_smem(a.np2max), s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_spec_transform(const SpecArgs& a, int n_sm, int max_n, bool one_pass, bool two_pass, cudaStream_t s)
{
    const int n = a.slot_end - a.slot_begin;
    if (n <= 0) return cudaSuccess;
    if (n > kSpecMaxChunk) return cudaErrorInvalidValue;
    const size_t smem = spec_spread_smem(max_n, a.seg_max);
    if (a.interp) k_spec_spread<true><<<2 * n_sm, kSpreadThreads, smem, s>>>(a, max_n);
    else k_spec_spread<false><<<2 * n_sm, kSpreadThreads, smem, s>>>(a, max_n);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess && two_pass) {
        k_spec_fft1<<<2 * n_sm, kFftThreads, fft_smem(), s>>>(a);
        e = cudaGetLastError();
        if (e == cudaSuccess) {
            k_spec_fft2<<<2 * n_sm, kFftThreads, fft_smem(), s>>>(a);
            e = cudaGetLastError();
        }
    }
    if (e == cudaSuccess && one_pass) {
        k_spec_fft_one<<<n, kFftThreads, fft_smem(), s>>>(a);
        e = cudaGetLastError();
    }
    return e;
}

cudaError_t launch_spec_values(const SpecArgs& a, int n_sm, cudaStream_t s)
{
    if (a.interp) k_spec_interp<<<8 * n_sm, kSumThreads, 0, s>>>(a);
    else k_spec_sum<<<8 * n_sm, kSumThreads, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_spec_select(const SpecArgs& a, cudaStream_t s)
{
    k_spec_select<<<a.slot_end - a.slot_begin, kSelThreads, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_spec_peaks(const SpecArgs& a, cudaStream_t s)
{
    k_spec_peaks<<<a.slot_end - a.slot_begin, kPeakThreads, a.n_freq <= kPeakRow ? (size_t)a.n_freq * sizeof(float) : 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_spec_rank(const SpecArgs& a, cudaStream_t s)
{
    k_spec_rank<<<a.slot_end - a.slot_begin, kSpecCand, 0, s>>>(a);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
int spec_harmonics(double sigma_t)
{
    if (!(sigma_t >= 0.09) || !(sigma_t < 1e3)) return 0;
    const double kap = 1.0 / (sigma_t * sigma_t);
    double a[kMillerMax + 2];
    int n0 = (int)(14.0 + 10.0 * std::sqrt(kap));
    n0 = n0 < kMillerMax ? n0 : kMillerMax;
    double hi = 0.0, cur = 1e-200, sum = 0.0;
    for (int q = n0; q >= 1; q--) {
        a[q] = cur;
        sum += 2.0 * cur;
        const double nx = (double)q * 2.0 / kap * cur + hi;
        hi = cur;
        cur = nx;
    }
    sum += cur;
    double tail = 0.0;
    int nh = n0;
    while (nh > 1 && tail + 2.0 * a[nh] / sum <= kSpecTail) {
        tail += 2.0 * a[nh] / sum;
        nh--;
    }
    return nh <= kSpecMaxHarm ? nh : 0;
}

int spec_logq(int64_t n_out)
{
    const int lq = spec_logq_of(n_out);
    return lq <= kSpecMaxLogQ ? lq : 0;
}

}  // namespace cpk
