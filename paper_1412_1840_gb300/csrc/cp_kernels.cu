// cp_kernels.cu -- sm_103a kernels of the correntropy kernelized periodogram.
//
// Hot path (arXiv:1412.1840, Section 3, Eq. (HP), (IP), (CKP)):
//   k_stats        per-curve scalars (sigma_y = med(e), pSNR, sigma_t, IP),
//                  scaled magnitudes y' and 64-bit fixed-point phase steps
//   k_build_w      period-independent magnitude-kernel tiles w_ij = g_ij - ip
//   k_pair_direct  persistent pair-sum kernel over (curve, frequency-chunk)
//                  work units: the N(N-1)/2 interactions of Section 8 per
//                  trial frequency, FP32 with packed f32x2 arithmetic
//   k_topk         coarse-grid local maxima for the coarse-then-fine search
//                  (the bands method of Section 3.1 is in cp_bands.cu)
//   k_finalize     best frequency, nCKP and Table tab:th discriminator
#include <algorithm>
#include <cstdint>
#include <map>
#include <mutex>
#include <type_traits>
#include <utility>
#include <cuda_runtime.h>

#include "cp_internal.cuh"

namespace cpk {

// Table "tab:th" of Section 4.1: pSNR bin lower edges and thresholds.
__constant__ double c_bin_lo[8] = {0.0, 1.5, 2.0, 2.5, 3.5, 5.0, 10.0, 20.0};
__constant__ float c_th[8] = {0.4584f, 0.4565f, 0.4537f, 0.4581f, 0.5875f, 1.1153f, 1.6464f, 2.4112f};

// ===========================================================================
// k_stats: one CTA per curve.
// ===========================================================================

constexpr int kStatsThreads = 256;

__device__ __forceinline__ double median_sorted(const float* s, int n) { return median_of_sorted(s, n); }

// Quantile by linear interpolation between order statistics at q*(n-1).
__device__ __forceinline__ double quantile_sorted(const float* s, int n, double q)
{
    const double pos = q * (double)(n - 1);
    const int lo = (int)floor(pos);
    const int hi = lo + 1 < n ? lo + 1 : n - 1;
    return (double)s[lo] + (pos - (double)lo) * ((double)s[hi] - (double)s[lo]);
}

__device__ __forceinline__ int snr_bin(double p)
{
    int b = 0;
#pragma unroll
    for (int k = 0; k < 8; k++)
        if (p >= c_bin_lo[k]) b = k;
    return b;
}

// Ascending bitonic sort of np2 floats (a power of two, at least 32) by T threads
// of whole warps: strides below 32 stay in a warp's registers, a barrier separates
// only the longer ones (15 instead of 55 at 1024).  Other is a second array
// sorted alike (or the same pointer: one array).
template <int T>
__device__ __forceinline__ void sort_floats(float* a, float* other, int np2)
{
    const int tid = threadIdx.x, lane = tid & 31;
    const bool two = other != a;
    for (int k = 32; k <= np2; k <<= 1) {
        for (int j = k >> 1; j >= 32; j >>= 1) {
            __syncthreads();
            for (int p = tid; p < np2 >> 1; p += T) {
                const int i = ((p & ~(j - 1)) << 1) | (p & (j - 1)), o = i | j;
                const bool up = (i & k) == 0;
                float u = a[i], v = a[o];
                if ((u > v) == up) { a[i] = v; a[o] = u; }
                if (two) {
                    u = other[i];
                    v = other[o];
                    if ((u > v) == up) { other[i] = v; other[o] = u; }
                }
            }
        }
        __syncthreads();
        for (int i = tid; i < np2; i += T) {
            float u = a[i], v = two ? other[i] : 0.f;
            for (int kk = k == 32 ? 2 : k; kk <= k; kk <<= 1) {
#pragma unroll
                for (int j = 16; j > 0; j >>= 1) {
                    if (j >= kk) continue;
                    const bool low = ((i & kk) == 0) == ((lane & j) == 0);     // keeps the smaller
                    const float u2 = __shfl_xor_sync(0xffffffffu, u, j);
                    u = (u2 < u) == low ? u2 : u;
                    if (two) {
                        const float v2 = __shfl_xor_sync(0xffffffffu, v, j);
                        v = (v2 < v) == low ? v2 : v;
                    }
                }
            }
            a[i] = u;
            if (two) other[i] = v;
        }
    }
    __syncthreads();
}

// Block sum of one double per thread in a fixed order (lanes, then warps); thread 0 gets it.
template <int T>
__device__ __forceinline__ double stats_sum(double v, double* s_red)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if (lane == 0) s_red[warp] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < T / 32; w++) t += s_red[w];
    return t;
}

// This block's part of sum_{i<j} g_ij: rows block, block + blocks, ... dealt to the
// warps, lanes along j, each lane a compensated (Kahan) FP32 sum whose remainder is
// kept, so that nothing is lost beyond FP32's second order; FP64 only at the end.
template <int T>
__device__ __forceinline__ double ip_part(const float* y, int n, int block, int blocks)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float s0 = 0.f, c0 = 0.f, s1 = 0.f, c1 = 0.f;
    for (int i = block + blocks * warp; i < n; i += blocks * (T / 32)) {
        const float yi = y[i];
        int j = i + 1 + lane;
        for (; j + 32 < n; j += 64) {
            float d = gauss_g(yi, y[j]) - c0, t = s0 + d;
            c0 = (t - s0) - d;
            s0 = t;
            d = gauss_g(yi, y[j + 32]) - c1;
            t = s1 + d;
            c1 = (t - s1) - d;
            s1 = t;
        }
        if (j < n) {
            const float d = gauss_g(yi, y[j]) - c0, t = s0 + d;
            c0 = (t - s0) - d;
            s0 = t;
        }
    }
    return ((double)s0 - (double)c0) + ((double)s1 - (double)c1);
}

// IP and what follows from it: ip = (N + 2 sum_{i<j} g_ij) / N^2.
__device__ __forceinline__ void set_ip(CurveParams* P, double s2)
{
    const double nn = (double)P->n;
    const double ip = (nn + 2.0 * s2) / (nn * nn);
    const float iph = (float)ip;
    P->ip = ip;
    P->ip_hi = iph;
    P->ip_lo = (float)(ip - (double)iph);
    P->norm = (float)(sqrt(nn) / (nn * nn * ip * sqrt(2.0 * CP_PI) * sqrt((double)P->sigma_t)));
    P->diag = (float)(nn * (1.0 - ip));
}

// One CTA per curve.  FP64 runs at 1.7 operations/clk/SM: the phase steps are
// integer products of the significands, the scalars are dealt to three warps, and
// the pair sum of IP is FP32.  With few long curves the pair sum is left to k_ip
// (a.ip_blocks blocks a curve).  With k_ip: 12 curves of up to 1,000 samples 70 ->
// 28 us, three of up to 4,096 568 -> 41 us (and 18 in k_ip); a curve of 150 samples 18 -> 14 us.
template <int T>
__global__ void __launch_bounds__(T) k_stats(const StatsArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    double* ts = reinterpret_cast<double*>(smem);
    float* ys = reinterpret_cast<float*>(ts + a.np2max);
    float* es = ys + a.np2max;
    float* ypl = es + a.np2max;
    __shared__ double s_red[T / 32];
    __shared__ double s_t0;
    __shared__ float s_yref, s_gamma;
    __shared__ int s_bad;

    const int c = blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    CurveParams* P = a.cp + c;
    const int64_t off = P->off;
    const int n = P->n;
    int np2 = 32;
    while (np2 < n) np2 <<= 1;
    if (tid == 0) s_bad = 0;
    __syncthreads();

    // 1. load, validate, min t
    double tmin = INFINITY;
    for (int i = tid; i < np2; i += T) {
        if (i < n) {
            const double t = a.times[off + i];
            const float y = a.mags[off + i];
            const float e = a.errs[off + i];
            if ((__double2hiint(t) & 0x7ff00000) == 0x7ff00000 || !isfinite(y) || !isfinite(e)) s_bad = 1;
            ts[i] = t;
            ys[i] = y;
            es[i] = e;
            ypl[i] = y;
            tmin = t < tmin ? t : tmin;
        } else {
            ys[i] = INFINITY;
            es[i] = INFINITY;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double t = __shfl_xor_sync(0xffffffffu, tmin, o);
        tmin = t < tmin ? t : tmin;
    }
    if (lane == 0) s_red[warp] = tmin;

    // 2. magnitudes and error bars in ascending order
    sort_floats<T>(ys, es, np2);

    // 3. per-curve scalars (FP64), one thread of three warps
    if (tid == 0) {
        double m = s_red[0];
        for (int w = 1; w < T / 32; w++) m = s_red[w] < m ? s_red[w] : m;
        s_t0 = m;
        P->t0 = m;
        const double sy = median_sorted(es, n);
        if (!(sy > 0.0) || !isfinite(sy)) s_bad = 1;
        const double gamma = sqrt(1.4426950408889634 / (2.0 * sy * sy));
        P->sigma_y = (float)sy;
        s_yref = (float)median_sorted(ys, n);
        s_gamma = (float)gamma;
        P->gamma = (float)gamma;
    } else if (tid == 32) {
        double st;
        if (a.sigma_t_mode == 1) {
            st = (double)a.sigma_t_per_curve[c];
        } else if (a.sigma_t_mode == 2) {
            st = sigma_t_rule(ys, n);
        } else {
            st = (double)a.sigma_t;
        }
        if (!(st > 0.0) || !isfinite(st)) s_bad = 1;
        const float stf = (float)st;
        // the planned harmonic count no longer covers this sigma_t: the host re-plans
        if (stf < P->st_floor) atomicOr(a.status, 4);
        P->sigma_t = stf;
        // sqrt(beta), beta = sqrt(2 log2 e) / sigma_t
        P->tscale = (float)sqrt(sqrt(2.0 * 1.4426950408889634) / (double)stf);
    } else if (tid == 64) {
        const double sy = median_sorted(es, n);
        const double q1 = quantile_sorted(ys, n, 0.25), q3 = quantile_sorted(ys, n, 0.75);
        const double psnr = 0.7413 * (q3 - q1) / ((double)a.alpha * sy);
        P->psnr = (float)psnr;
        P->th = c_th[snr_bin(psnr)];
    }
    __syncthreads();

    // 4. scaled magnitudes y' = (y - y_ref) * gamma (same values feed IP and W)
    const float yref = s_yref, gamma = s_gamma;
    for (int i = tid; i < n; i += T) {
        const float v = (ypl[i] - yref) * gamma;
        ypl[i] = v;
        a.yp[off + i] = v;
    }
    __syncthreads();

    // 5. IP
    if (a.ip_blocks == 0) {
        const double s2 = stats_sum<T>(ip_part<T>(ypl, n, 0, 1), s_red);
        if (tid == 0) set_ip(P, s2);
    }
    if (tid == 0 && s_bad) atomicOr(a.status, 1);

    // 6. fixed-point phase steps of t - t0 for each grid the search uses
    const double t0 = s_t0;
    for (int i = tid; i < n; i += T) {
        const double tp = ts[i] - t0;
        a.ph_base[off + i] = fixfrac(a.f_min, tp);
        a.ph_full[off + i] = fixfrac(a.df, tp);
        if (a.hierarchical) {
            a.ph_coarse[off + i] = fixfrac(a.coarse_df, tp);
            a.ph_fine[off + i] = fixfrac(a.fine_df, tp);
        }
    }
}

// Adds the blocks' parts of a curve in the last block to arrive (*last, all threads
// agree), in a fixed order; thread 0 gets the sum.  At most kStatsThreads blocks.
__device__ __forceinline__ double last_block_sum(double part, double* parts, unsigned int* count, int blocks,
                                                 double* s_red, int* last)
{
    if (threadIdx.x == 0) {
        parts[blockIdx.y] = part;
        __threadfence();
        *last = atomicAdd(count, 1u) == (unsigned)blocks - 1u;
        __threadfence();
    }
    __syncthreads();
    if (!*last) return 0.0;
    return stats_sum<kStatsThreads>((int)threadIdx.x < blocks ? __ldcg(parts + threadIdx.x) : 0.0, s_red);
}

// IP of few curves: a.ip_blocks CTAs a curve; the last to finish adds the parts in
// order and takes the steps that follow.
__global__ void __launch_bounds__(kStatsThreads) k_ip(const StatsArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    float* y = reinterpret_cast<float*>(smem);
    __shared__ double s_red[kStatsThreads / 32];
    __shared__ int s_last;
    const int c = blockIdx.x, tid = threadIdx.x, nb = a.ip_blocks;
    CurveParams* P = a.cp + c;
    const int n = P->n;
    for (int i = tid; i < n; i += kStatsThreads) y[i] = a.yp[P->off + i];
    __syncthreads();
    const double part = stats_sum<kStatsThreads>(ip_part<kStatsThreads>(y, n, blockIdx.y, nb), s_red);
    const double s2 = last_block_sum(part, a.ip_parts + (int64_t)c * nb, a.ip_count + c, nb, s_red, &s_last);
    if (tid == 0 && s_last) set_ip(P, s2);
}

// Tensor form: per sample i, the sum over j of the rounding error of the 16-bit
// operand w_ij = (g_ij - ip_hi) - ip_lo (the same FP32 values the tile builder
// rounds), and its total.  With these the tensor epilogue removes the error's
// coherent part: for a Z column x with mean xm the operand error adds
// xm^2 sum(dW) + 2 xm drho^T (x - xm), which does not average out where x is nearly
// constant over the samples (low f T, or aliases of the sampling).  A warp per row,
// a.rho_blocks CTAs per curve; fixed order: deterministic.
__global__ void __launch_bounds__(kStatsThreads) k_wrho(const StatsArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    float* y = reinterpret_cast<float*>(smem);
    __shared__ double s_red[kStatsThreads / 32];
    __shared__ int s_last;
    const int c = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nb = a.rho_blocks;
    CurveParams* P = a.cp + c;
    const int n = P->n;
    const int64_t off = P->off;
    for (int i = tid; i < n; i += kStatsThreads) y[i] = a.yp[off + i];
    __syncthreads();
    const float iph = P->ip_hi, ipl = P->ip_lo;
    const bool bf = a.wrho_bf16 != 0;
    double tot = 0.0;
    for (int i = blockIdx.y + nb * warp; i < n; i += nb * (kStatsThreads / 32)) {
        const float yi = y[i];
        float s = 0.f;
        for (int j = lane; j < n; j += 32) s += w16_err((gauss_g(yi, y[j]) - iph) - ipl, bf);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) {
            a.wrho[off + i] = s;
            tot += (double)s;
        }
    }
    const double part = stats_sum<kStatsThreads>(tot, s_red);
    const double t = last_block_sum(part, a.rho_parts + (int64_t)c * nb, a.rho_count + c, nb, s_red, &s_last);
    if (tid == 0 && s_last) P->dwsum = (float)t;
}

// ===========================================================================
// k_sigma_t_rule: sigma_t of the skewness rule per curve (one CTA per curve),
// the same sort and the same FP64 arithmetic as k_stats.
// ===========================================================================
__global__ void __launch_bounds__(kStatsThreads) k_sigma_t_rule(const float* mags, const int64_t* offsets,
                                                               int np2max, float* out)
{
    extern __shared__ __align__(16) unsigned char smem[];
    float* ys = reinterpret_cast<float*>(smem);
    const int c = blockIdx.x, tid = threadIdx.x;
    const int64_t off = offsets[c];
    const int n = (int)(offsets[c + 1] - off);
    int np2 = 32;
    while (np2 < n) np2 <<= 1;
    for (int i = tid; i < np2; i += kStatsThreads) ys[i] = i < n ? mags[off + i] : INFINITY;
    sort_floats<kStatsThreads>(ys, ys, np2);
    if (tid == 0) out[c] = (float)sigma_t_rule(ys, n);
}

// Curves with sigma_t at or above this take the exponent in the cos form (see
// pair_item); below it the sin form keeps the exponent's rounding relative.
constexpr float kCosFormMinSigma = 0.3f;

// ===========================================================================
// k_build_w: one warp per 32x32 tile of the upper block triangle.
// Layout per tile: [k][lane][m] floats, k < 8 rows, m < 4 columns per lane.
// ===========================================================================

__device__ __forceinline__ void decode_tile(int t, int nb, int& bi, int& bj)
{
    int b = 0, rem = t;
    while (rem >= nb - b) { rem -= nb - b; ++b; }
    bi = b;
    bj = b + rem;
}

// The constant 2^(-beta/2) that the cos form's w carries (see pair_item); 1 in the sin form.
__device__ __forceinline__ float w_scale(const CurveParams& P)
{
    const float tsc = P.tscale * P.tscale * 0.70710678f;
    return P.sigma_t >= kCosFormMinSigma ? exp2f(-(tsc * tsc)) : 1.0f;
}

__device__ __forceinline__ float w_of(float ypi, float ypj, float ip_hi, float ip_lo, float scale)
{
    return ((gauss_g(ypi, ypj) - ip_hi) - ip_lo) * scale;
}

__global__ void __launch_bounds__(256) k_build_w(const BuildWArgs a)
{
    const int lane = threadIdx.x & 31;
    const int64_t T = a.tile_begin + (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (T >= a.tile_end) return;
    int lo = a.slot_begin, hi = a.slot_end - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (a.wtile_start[mid] <= T) lo = mid; else hi = mid - 1;
    }
    const int c = a.order[lo];
    const CurveParams P = a.cp[c];
    const int n = P.n;
    const int nb = (n + kTile - 1) / kTile;
    int bi, bj;
    decode_tile((int)(T - a.wtile_start[lo]), nb, bi, bj);
    const int la = lane >> 3, lb = lane & 7;
    // cos-form curves: w carries the exponent's constant term, w 2^(-beta/2), so
    // that the pair kernel's exponent is the bare product sum (see pair_item)
    const float wscale = w_scale(P);
    float ypc[kColsPerLane];
    int jj[kColsPerLane];
#pragma unroll
    for (int m = 0; m < kColsPerLane; m++) {
        jj[m] = bj * kTile + lb + 8 * m;
        ypc[m] = jj[m] < n ? a.yp[P.off + jj[m]] : 0.f;
    }
    float* dst = a.W + (T - a.tile_begin) * kTileFloats;
#pragma unroll
    for (int k = 0; k < kRowsPerLane; k++) {
        const int i = bi * kTile + la + 4 * k;
        const float ypr = i < n ? a.yp[P.off + i] : 0.f;
        float w[kColsPerLane];
#pragma unroll
        for (int m = 0; m < kColsPerLane; m++) {
            w[m] = (i < jj[m] && jj[m] < n) ? w_of(ypr, ypc[m], P.ip_hi, P.ip_lo, wscale) : 0.f;
        }
        reinterpret_cast<float4*>(dst)[k * 32 + lane] = make_float4(w[0], w[1], w[2], w[3]);
    }
}

// ===========================================================================
// k_pair_direct: persistent CTAs pop (curve, frequency-chunk) units.
// ===========================================================================
constexpr int kPairThreads = 512;
// Rows per lane in one warp work item: 8 = a whole 32 x 32 tile (each lane 8
// rows x 4 columns), 4 = half a tile.  Every trig value a lane loads from
// shared memory serves (rows x columns) / (rows + columns) evaluations, so the
// whole-tile item needs a third fewer shared-memory loads per evaluation.
constexpr int kItemRows = 8;
static_assert(kItemRows == kRowsPerLane && kFcMax == 16, "whole-tile items, 16 sums per share");
// The unit's trig table is built by one thread per (point, half of the
// frequency pairs): each point's phase and step are loaded twice per unit
// instead of once per frequency pair, and the threads' shares stay even
// (one thread per point leaves a few threads with twice the work).
constexpr int kTableGroups = 2;

// One work item (4 kItemRows rows x 32 columns of a tile) at every frequency
// pair of the unit.  The exponent of the periodic kernel (Eq. (periodickernel)),
// -beta sin^2(pi dphi) with beta = 2 log2(e) / sigma_t^2, is taken in one of
// two forms from the trig table of the unit:
//   sin form  -(c_i s_j - s_i c_j)^2 with (s, c) = (sin, cos)(pi phi) sqrt(beta)
//             (three f32x2 operations per two frequencies);
//   cos form  C_i C_j + S_i S_j - beta/2 with (S, C) = (sin, cos)(2 pi phi)
//             sqrt(beta/2), from sin^2 x = (1 - cos 2x)/2; the constant
//             2^(-beta/2) is carried by the tile's w (k_build_w), so the
//             exponent is the bare sum, a multiply and an FMA (two operations,
//             one of them with two operands).
// The cos form's rounding is absolute, about beta 2^-24 in the exponent, so it
// is used only for sigma_t >= kCosFormMinSigma (beta <= 32: below 3e-6 per term;
// the exponent then lies in [-beta/2, beta/2], within FP32 range).
// The item's sum at one frequency pair (SCf, NSf: that pair's table): (f, f').
template <bool COSF>
__device__ __forceinline__ f2 pair_item_at(const ulonglong2* SCf, const f2* NSf, int rbase, int cbase,
                                           const f2 (&w01)[kItemRows], const f2 (&w23)[kItemRows])
{
    ulonglong2 col[kColsPerLane];
#pragma unroll
    for (int m = 0; m < kColsPerLane; m++) col[m] = SCf[cbase + 8 * m];
    f2 tf0 = 0ull, tf1 = 0ull, tg0 = 0ull, tg1 = 0ull;
#pragma unroll
    for (int k = 0; k < kItemRows; k++) {
        const int i = rbase + 4 * k;
        float e[kColsPerLane][2];
        if (COSF) {
            const ulonglong2 R = SCf[i];   // ((S_i(f), S_i(f')), (C_i(f), C_i(f')))
#pragma unroll
            for (int m = 0; m < kColsPerLane; m++) {
                const f2 a2 = fma2(R.y, col[m].y, mul2(R.x, col[m].x));
                float a0, a1;
                upk(a2, a0, a1);
                e[m][0] = ex2_approx(a0);
                e[m][1] = ex2_approx(a1);
            }
        } else {
            const f2 A = SCf[i].y;   // (c_i(f), c_i(f'))
            const f2 B = NSf[i];     // (-s_i(f), -s_i(f'))
#pragma unroll
            for (int m = 0; m < kColsPerLane; m++) {
                const f2 t2 = mul2(B, col[m].y);
                const f2 d2 = fma2(A, col[m].x, t2);
                const f2 q2 = mul2(d2, d2);
                float q0, q1;
                upk(q2, q0, q1);
                e[m][0] = ex2_approx(-q0);
                e[m][1] = ex2_approx(-q1);
            }
        }
        tf0 = fma2(w01[k], pk(e[0][0], e[1][0]), tf0);
        tf1 = fma2(w23[k], pk(e[2][0], e[3][0]), tf1);
        tg0 = fma2(w01[k], pk(e[0][1], e[1][1]), tg0);
        tg1 = fma2(w23[k], pk(e[2][1], e[3][1]), tg1);
    }
    float fx, fy, gx, gy;
    upk(add2(tf0, tf1), fx, fy);
    upk(add2(tg0, tg1), gx, gy);
    return pk(fx + fy, gx + gy);
}

template <bool COSF>
__device__ __forceinline__ void pair_item(const ulonglong2* SC, const f2* NS, int npad, int nfp, int rbase,
                                          int cbase, const f2 (&w01)[kItemRows],
                                          const f2 (&w23)[kItemRows], f2 (&acc)[kFcMax / 2])
{
#pragma unroll
    for (int fp = 0; fp < kFcMax / 2; fp++)
        if (fp < nfp)
            acc[fp] = add2(acc[fp], pair_item_at<COSF>(SC + fp * npad, NS + fp * npad, rbase, cbase, w01, w23));
}

// The item's w from the curve's scaled magnitudes (as k_build_w stores them).
__device__ __forceinline__ void item_w(const float* Y, int n, int rbase, int cbase, float ip_hi, float ip_lo, float scale,
                                       f2 (&w01)[kItemRows], f2 (&w23)[kItemRows])
{
    float yc[kColsPerLane];
#pragma unroll
    for (int m = 0; m < kColsPerLane; m++) yc[m] = Y[cbase + 8 * m];
#pragma unroll
    for (int k = 0; k < kItemRows; k++) {
        const int i = rbase + 4 * k;
        const float yr = Y[i];
        float w[kColsPerLane];
#pragma unroll
        for (int m = 0; m < kColsPerLane; m++) {
            const int j = cbase + 8 * m;
            w[m] = (i < j && j < n) ? w_of(yr, yc[m], ip_hi, ip_lo, scale) : 0.f;
        }
        w01[k] = pk(w[0], w[1]);
        w23[k] = pk(w[2], w[3]);
    }
}

// Trig table entry of one point at a frequency pair (phases p0, p1).
__device__ __forceinline__ void table_entry(bool cosf, float ts, uint64_t p0, uint64_t p1, ulonglong2& sc, f2& ns)
{
    float s0, c0, s1, c1;
    if (cosf) {
        sincos2pi_turns((uint32_t)(p0 >> 32), s0, c0);
        sincos2pi_turns((uint32_t)(p1 >> 32), s1, c1);
    } else {
        sincospi_turns((uint32_t)(p0 >> 32), s0, c0);
        sincospi_turns((uint32_t)(p1 >> 32), s1, c1);
    }
    s0 *= ts; c0 *= ts; s1 *= ts; c1 *= ts;
    sc = make_ulonglong2(pk(s0, s1), pk(c0, c1));
    ns = pk(-s0, -s1);
}

// Phase of point `at` (index in the CSR arrays) at candidate entry e.
__device__ __forceinline__ uint64_t cand_phase(const PairArgs& a, const int32_t* tl, int c, int64_t at, int e)
{
    const uint64_t base = a.ph_base[at], st = a.ph_step[at];
    if (a.candidates == kCandTrial) return base + (uint64_t)max(tl[e], 0) * st;
    if (a.candidates != kCandFine) return base + (uint64_t)e * st;
    const int W = 2 * a.fine_half + 1, pk_ = e / W;
    return base + (uint64_t)a.peaks[(int64_t)c * a.top_k + pk_] * a.ph_coarse[at] +
           (uint64_t)(int64_t)(e - pk_ * W - a.fine_half) * st;
}

// The value at candidate entry e (admissible already) replaces the spectrum's; its key.
__device__ __forceinline__ unsigned long long cand_emit(const PairArgs& a, int c, int e, float v)
{
    if (a.candidates == kCandGrid && a.out) a.out[(int64_t)c * a.out_ld + e] = v;
    if (a.candidates == kCandCoarse) a.coarse_out[(int64_t)c * a.n_freq + e] = v;
    if (a.candidates == kCandTrial && a.trial_stat) a.trial_stat[(int64_t)c * a.n_trials + e] = v;
    return a.candidates == kCandCoarse ? 0ull : make_key(v, (uint32_t)e);
}

// Butterfly reduce-scatter of 16 values: on return lane l holds the warp's sum of
// x[l >> 1] (the same pairs in the same order as 16 separate butterflies).
__device__ __forceinline__ float reduce_scatter16(float (&x)[16], int lane)
{
#pragma unroll
    for (int half = 8, bit = 4; half > 0; half >>= 1, bit--) {
        const bool upper = (lane >> bit) & 1;
#pragma unroll
        for (int q = 0; q < half; q++) {
            const float recv = __shfl_xor_sync(0xffffffffu, upper ? x[q] : x[q + half], 1 << bit);
            x[q] = (upper ? x[q + half] : x[q]) + recv;
        }
    }
    return x[0] + __shfl_xor_sync(0xffffffffu, x[0], 1);
}

// SEL: a launch over chosen curves (fb_slots), those that the pair-spectrum path
// leaves to the pair sum; its own instantiation, so that the units of a plain
// launch carry none of it.  Its w come from the magnitudes
// instead of stored tiles (one more exponential per pair and unit), so that
// plans whose every pass goes through the spectrum keep no tiles.
// WARPS: a unit's tiles are always summed as by kPairThreads / 32 warps (each
// every 16th tile, then lanes, then warps); a block of fewer warps takes several
// of these shares in turn, with the same result.
// Each form has its own loop, the tile's loads before the search for its place, and
// on 16 warps the cos form its own butterflies (the same additions): with one loop
// whose form is chosen inside, the place found first and one reduction for both,
// 256 curves of 300 to 1,000 samples at 2,048 frequencies took 20.64 instead of
// 20.31 ms, 16 of 3,000 to 4,000 at 600 frequencies 13.46 instead of 12.78; the sin
// form with butterflies takes 22.6 instead of 22.1.
template <bool SEL, int WARPS>
__global__ void __launch_bounds__(32 * WARPS, 16 / WARPS) k_pair_direct(const PairArgs a)
{
    constexpr int NW = kPairThreads / 32;
    constexpr int T = 32 * WARPS;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ long long s_unit;
    __shared__ float s_red[NW][kFcMax];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int la = lane >> 3, lb = lane & 7;

    for (;;) {
        __syncthreads();
        if (tid == 0) s_unit = (long long)atomicAdd(a.queue, 1ull) + a.unit_begin;
        __syncthreads();
        const long long u = s_unit;
        if (u >= (SEL ? (long long)*a.fb_count * a.upc : a.unit_end)) break;

        int slot;
        long long chunk;
        if (SEL) {
            const int64_t q = u / a.upc;
            chunk = u - q * a.upc;
            slot = a.fb_slots[q];
        } else {
            int lo = a.slot_begin, hi = a.slot_end - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (a.unit_start[mid] <= u) lo = mid; else hi = mid - 1;
            }
            slot = lo;
            chunk = u - a.unit_start[slot];
        }
        const int c = a.order[slot];
        const CurveParams& P = a.cp[c];
        const int n = P.n, fc = P.fc;
        const int npad = (n + kTile - 1) & ~(kTile - 1);
        const int64_t off = P.off;

        // frequencies of this unit: phase(i, kk) = base_i + mult0 * step_i + kk * step_i
        long long kfirst;      // full/coarse: first grid index; fine: first j
        int count;
        int peak = 0;
        uint64_t peak_mult = 0;  // fine: coarse peak index (phase offset kpeak * coarse_i)
        if (a.stage == kStageFine) {
            const int W = 2 * a.fine_half + 1;
            const int upp = (W + fc - 1) / fc;
            peak = (int)(chunk / upp);
            const int sub = (int)(chunk - (long long)peak * upp);
            if (peak >= a.n_peaks[c]) continue;   // (also a chunk beyond the curve's own units)
            peak_mult = (uint64_t)a.peaks[(int64_t)c * a.top_k + peak];
            kfirst = -a.fine_half + (long long)sub * fc;
            count = (int)min((long long)fc, (long long)a.fine_half - kfirst + 1);
        } else if (a.stage == kStageList) {
            kfirst = chunk * fc;     // first list position
            count = (int)min((long long)fc, (long long)a.n_trials - kfirst);
            if (SEL && count <= 0) continue;
        } else {
            kfirst = chunk * fc;
            count = (int)min((long long)fc, a.n_freq - kfirst);
            if (SEL && count <= 0) continue;   // fewer units than the launch gives a curve
        }
        const int32_t* tl = a.trials + (int64_t)c * a.n_trials;   // list stage only
        const int nfp = SEL ? (count + 1) >> 1 : fc >> 1;   // frequency pairs of the unit

        // trig table: SC[fp][i] = {(s_f, s_f'), (c_f, c_f')} * sqrt(beta), NS[fp][i] = -(s_f, s_f')
        // (sin form), or the sines and cosines of the doubled angle * sqrt(beta / 2) (cos form)
        ulonglong2* SC = reinterpret_cast<ulonglong2*>(smem);
        f2* NS = reinterpret_cast<f2*>(SC + nfp * npad);
        const bool cosf = P.sigma_t >= kCosFormMinSigma;
        const float ts = cosf ? P.tscale * P.tscale * 0.70710678f : P.tscale;   // tscale^4 = beta
        // One thread per (point, group of frequency pairs): the point's phase and
        // step are loaded once for the whole group, and the phase advances by two
        // grid steps per pair (exact in the 2^-64 fixed point).
        const int gsz = (nfp + kTableGroups - 1) / kTableGroups;
        for (int it = tid; it < kTableGroups * npad; it += T) {
            const int gi = it / npad, i = it - gi * npad;
            const int fp0 = gi * gsz, fp1 = min(nfp, fp0 + gsz);
            if (i < n) {
                const uint64_t st = a.ph_step[off + i];
                const uint64_t base = a.ph_base[off + i];
                uint64_t ph = base + (uint64_t)(kfirst + 2 * fp0) * st;
                if (a.stage == kStageFine) ph += peak_mult * a.ph_coarse[off + i];
                for (int fp = fp0; fp < fp1; fp++, ph += 2 * st) {
                    uint64_t p0 = ph, p1 = ph + st;
                    if (a.stage == kStageList) {
                        // grid indices of list positions kfirst + 2 fp (+1); a missing entry evaluates k = 0
                        const long long q0 = kfirst + 2 * fp;
                        const int k0 = q0 < a.n_trials ? max(tl[q0], 0) : 0;
                        const int k1 = q0 + 1 < a.n_trials ? max(tl[q0 + 1], 0) : 0;
                        p0 = base + (uint64_t)k0 * st;
                        p1 = base + (uint64_t)k1 * st;
                    }
                    f2 ns;
                    table_entry(cosf, ts, p0, p1, SC[fp * npad + i], ns);
                    if (!cosf) NS[fp * npad + i] = ns;   // the cos form reads SC only
                }
            } else {
                for (int fp = fp0; fp < fp1; fp++) {
                    SC[fp * npad + i] = make_ulonglong2(0ull, 0ull);
                    if (!cosf) NS[fp * npad + i] = 0ull;
                }
            }
        }
        float* Y = reinterpret_cast<float*>(SC) + (size_t)(fc >> 1) * npad * 6;   // SEL: after the tables
        if (SEL)
            for (int i = tid; i < npad; i += T) Y[i] = i < n ? a.yp[off + i] : 0.f;
        const float wscale = SEL ? w_scale(P) : 1.0f;
        __syncthreads();

        const int nb = npad / kTile;
        const int ntiles = nb * (nb + 1) / 2;
        const int nitems = ntiles;                   // a warp item is a whole tile
        const float4* Wc =
            SEL ? nullptr : reinterpret_cast<const float4*>(a.W + (a.wtile_start[slot] - a.wtile_base) * kTileFloats);
#pragma unroll 1
        for (int share = warp; share < NW; share += WARPS) {
            if (share >= nitems) {                   // a short curve's shares without a tile
                if (lane < 16) s_red[share][lane] = 0.f;
                continue;
            }
            auto sum_share = [&](auto form) {
                constexpr bool COSF = decltype(form)::value;
                f2 acc[kFcMax / 2];                  // per f-pair: (sum at f, sum at f')
#pragma unroll
                for (int q = 0; q < kFcMax / 2; q++) acc[q] = 0ull;
#pragma unroll 1
                for (int item = share; item < nitems; item += NW) {
                    f2 w01[kItemRows], w23[kItemRows];
#pragma unroll
                    for (int k = 0; k < (SEL ? 0 : kItemRows); k++) {      // in flight while the tile is found
                        const float4 wv = __ldg(Wc + (int64_t)item * (kTileFloats / 4) + k * 32 + lane);
                        w01[k] = pk(wv.x, wv.y);
                        w23[k] = pk(wv.z, wv.w);
                    }
                    int bi, bj;
                    decode_tile(item, nb, bi, bj);
                    const int rbase = bi * kTile + la;
                    const int cbase = bj * kTile + lb;
                    if (SEL) item_w(Y, n, rbase, cbase, P.ip_hi, P.ip_lo, wscale, w01, w23);
                    pair_item<COSF>(SC, NS, npad, nfp, rbase, cbase, w01, w23, acc);
                }
                // the share's frequency sums over the lanes, then (below) a fixed-order sum over the shares
                if constexpr (COSF && WARPS == NW) {
#pragma unroll
                    for (int fp = 0; fp < kFcMax / 2; fp++) {
                        if (fp < nfp) {
                            float vf, vg;
                            upk(acc[fp], vf, vg);
#pragma unroll
                            for (int o = 16; o > 0; o >>= 1) {
                                vf += __shfl_xor_sync(0xffffffffu, vf, o);
                                vg += __shfl_xor_sync(0xffffffffu, vg, o);
                            }
                            if (lane == 0) {
                                s_red[share][2 * fp] = vf;
                                s_red[share][2 * fp + 1] = vg;
                            }
                        }
                    }
                } else {
                    float x[16];
#pragma unroll
                    for (int fp = 0; fp < kFcMax / 2; fp++) upk(acc[fp], x[2 * fp], x[2 * fp + 1]);
                    const float v = reduce_scatter16(x, lane);
                    if ((lane & 1) == 0) s_red[share][lane >> 1] = v;
                }
            };
            if (cosf) sum_share(std::true_type{});
            else sum_share(std::false_type{});
        }
        __syncthreads();
        if (warp == 0) {
            unsigned long long key = 0ull;
            if (lane < count) {
                float S = 0.f;
#pragma unroll
                for (int w = 0; w < NW; w++) S += s_red[w][lane];
                const float v = (2.0f * S + P.diag) * P.norm;
                const long long kk = kfirst + lane;
                if (a.stage == kStageFull) {
                    if (a.out) a.out[(int64_t)c * a.out_ld + kk] = v;
                    if (!excluded_k(a.ex.full_k, a.ex.n, kk)) key = make_key(v, (uint32_t)kk);
                } else if (a.stage == kStageCoarse) {
                    a.coarse_out[(int64_t)c * a.n_freq + kk] = v;
                } else if (a.stage == kStageList) {
                    const bool valid = tl[kk] >= 0;
                    if (a.trial_stat) a.trial_stat[(int64_t)c * a.n_trials + kk] = valid ? v : __int_as_float(0x7fc00000);
                    if (valid && !excluded_k(a.ex.full_k, a.ex.n, tl[kk])) key = make_key(v, (uint32_t)kk);
                } else {
                    const double fpk = grid_freq(a.f_min, (double)peak_mult, a.coarse_df);
                    const double f = grid_freq(fpk, (double)kk, a.step);
                    if (f >= a.f_min && f <= a.f_max && !excluded_f(a.ex, f))
                        key = make_key(v, (uint32_t)(peak * (2 * a.fine_half + 1) + (kk + a.fine_half)));
                }
            }
            if (a.stage != kStageCoarse) {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    const unsigned long long other = __shfl_xor_sync(0xffffffffu, key, o);
                    key = other > key ? other : key;
                }
                if (lane == 0 && key) atomicMax(a.best_key + c, key);
            }
        }
    }
}

// ===========================================================================
// k_confirm / k_confirm_sum: the pair sum at the candidate
// entries, for a chunk of curves.  A unit of k_pair_direct would run
// its few frequencies on one SM (0.8 ms for one frequency of a 4,000-sample
// curve, 50 us for the 12 coarse points of a 650-sample one).  Here the tiles are
// spread over the chip: k_confirm stores every tile's sum per lane, and
// k_confirm_sum adds them in k_pair_direct's order (lane by lane over the tiles
// of each of its warps, then lanes, then warps), so the value is the same to the
// last bit.
// ===========================================================================
constexpr int kConfirmThreads = 512;
constexpr int kConfirmWarps = kConfirmThreads / 32;

__global__ void __launch_bounds__(kConfirmThreads) k_confirm(const PairArgs a, f2* part, int64_t part_ld, int group,
                                                             int smem_bytes)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_pre[kConfirmMaxChunk + 1];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int la = lane >> 3, lb = lane & 7;
    const int nc = a.slot_end - a.slot_begin;
    if (warp == 0) {
        int base = 0;
        for (int c0 = 0; c0 < nc; c0 += 32) {
            int v = 0;
            if (c0 + lane < nc) {
                const int c = a.order[a.slot_begin + c0 + lane];
                if (a.cand[(int64_t)c * a.n_cand] >= 0) v = (tiles_of(a.cp[c].n) + group - 1) / group;
            }
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(0xffffffffu, v, o);
                if (lane >= o) v += t;
            }
            if (c0 + lane < nc) s_pre[c0 + lane + 1] = base + v;
            base += __shfl_sync(0xffffffffu, v, 31);
        }
        if (lane == 0) s_pre[0] = 0;
    }
    __syncthreads();
    for (int item = blockIdx.x; item < s_pre[nc]; item += gridDim.x) {
        int lo = 0, hi = nc - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (s_pre[mid] <= item) lo = mid; else hi = mid - 1;
        }
        const int c = a.order[a.slot_begin + lo];
        const CurveParams& P = a.cp[c];
        const int n = P.n, npad = (n + kTile - 1) & ~(kTile - 1), nb = npad / kTile, ntiles = nb * (nb + 1) / 2;
        const int64_t off = P.off;
        const int32_t* ce = a.cand + (int64_t)c * a.n_cand;
        const int32_t* tl = a.trials + (int64_t)c * a.n_trials;
        int count = 0;
        {
            const int e = lane < a.n_cand ? ce[lane] : -1;
            count = __popc(__ballot_sync(0xffffffffu, e >= 0));
        }
        const bool cosf = P.sigma_t >= kCosFormMinSigma;
        const float ts = cosf ? P.tscale * P.tscale * 0.70710678f : P.tscale;
        const float wscale = w_scale(P);
        // frequency pairs per pass: as many as the table holds
        const int room = (smem_bytes - npad * 4) / (npad * 24);
        const int step = min(room, (count + 1) >> 1);
        float* Y = reinterpret_cast<float*>(smem);
        ulonglong2* SC = reinterpret_cast<ulonglong2*>(Y + npad);
        f2* NS = reinterpret_cast<f2*>(SC + step * npad);
        const int t0 = (item - s_pre[lo]) * group, t1 = min(t0 + group, ntiles);
        f2* dst = part + (int64_t)lo * part_ld;
        int bi0, bi1, bj0, bj1;
        decode_tile(t0, nb, bi0, bj0);
        decode_tile(t1 - 1, nb, bi1, bj1);
        if (bi0 != bi1) {                         // several tile rows: every column from the first row on
            bj0 = bi0;
            bj1 = nb - 1;
        }
        for (int f0 = 0; 2 * f0 < count; f0 += step) {
            const int nfp = min(step, ((count + 1) >> 1) - f0);
            __syncthreads();
            for (int q = tid; q < nfp * npad; q += kConfirmThreads) {
                const int fp = q / npad, i = q - fp * npad;
                // only the points of the group's tile rows and columns
                const int b = i / kTile;
                if (!((b >= bi0 && b <= bi1) || (b >= bj0 && b <= bj1))) continue;
                if (f0 == 0 && fp == 0) Y[i] = i < n ? a.yp[off + i] : 0.f;
                ulonglong2 sc = make_ulonglong2(0ull, 0ull);
                f2 ns = 0ull;
                if (i < n) {
                    const int e0 = 2 * (f0 + fp), e1 = e0 + 1 < count ? e0 + 1 : e0;
                    table_entry(cosf, ts, cand_phase(a, tl, c, off + i, ce[e0]), cand_phase(a, tl, c, off + i, ce[e1]), sc, ns);
                }
                SC[q] = sc;
                if (!cosf) NS[q] = ns;
            }
            __syncthreads();
            for (int t = t0 + warp; t < t1; t += kConfirmWarps) {
                int bi, bj;
                decode_tile(t, nb, bi, bj);
                const int rbase = bi * kTile + la, cbase = bj * kTile + lb;
                f2 w01[kItemRows], w23[kItemRows];
                item_w(Y, n, rbase, cbase, P.ip_hi, P.ip_lo, wscale, w01, w23);
                for (int fp = 0; fp < nfp; fp++) {
                    const f2 v = cosf ? pair_item_at<true>(SC + fp * npad, NS + fp * npad, rbase, cbase, w01, w23)
                                      : pair_item_at<false>(SC + fp * npad, NS + fp * npad, rbase, cbase, w01, w23);
                    dst[((int64_t)(f0 + fp) * ntiles + t) * 32 + lane] = v;
                }
            }
        }
        __syncthreads();
    }
}

// A block per (curve, share of k_pair_direct's 16 warps): its warps load 64 tiles at
// a time, the first adds them in order; a curve's last block adds the shares.  (One
// block for all shares pulled 2 MB through one SM for a 4,000-sample curve; one
// warp a share waited for memory every 16 tiles: 56 and 44 us.)
constexpr int kSumWarps = 4, kSumLoads = 16;

__global__ void __launch_bounds__(32 * kSumWarps) k_confirm_sum(const PairArgs a, const f2* part, int64_t part_ld,
                                                                float2* shares, unsigned int* arrived)
{
    constexpr int NW = kPairThreads / 32, B = kSumWarps * kSumLoads;
    __shared__ f2 s_v[B][32];
    __shared__ int s_last;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, share = blockIdx.y;
    const int c = a.order[a.slot_begin + blockIdx.x];
    const int32_t* ce = a.cand + (int64_t)c * a.n_cand;
    const CurveParams& P = a.cp[c];
    const int nb = (P.n + kTile - 1) / kTile, ntiles = nb * (nb + 1) / 2;
    const int mine = (ntiles - share + NW - 1) / NW;           // tiles share, share + 16, ...
    float2* sums = shares + (int64_t)blockIdx.x * (kConfirmCand / 2) * NW;
    int pairs = 0;
    for (; 2 * pairs < a.n_cand && ce[2 * pairs] >= 0; pairs++) {
        const f2* src = part + (int64_t)blockIdx.x * part_ld + ((int64_t)pairs * ntiles + share) * 32 + lane;
        f2 acc = 0ull, v[kSumLoads];
        auto load = [&](int t0) {
#pragma unroll
            for (int q = 0; q < kSumLoads; q++) {
                const int t = t0 + warp * kSumLoads + q;
                v[q] = t < mine ? src[(int64_t)t * (NW * 32)] : 0ull;
            }
        };
        load(0);
        for (int t0 = 0; t0 < mine; t0 += B) {
            __syncthreads();
#pragma unroll
            for (int q = 0; q < kSumLoads; q++) s_v[warp * kSumLoads + q][lane] = v[q];
            __syncthreads();
            if (t0 + B < mine) load(t0 + B);
            if (warp == 0) {
                const int m = min(B, mine - t0);
#pragma unroll 8
                for (int q = 0; q < m; q++) acc = add2(acc, s_v[q][lane]);
            }
        }
        if (warp == 0) {
            float vf, vg;
            upk(acc, vf, vg);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                vf += __shfl_xor_sync(0xffffffffu, vf, o);
                vg += __shfl_xor_sync(0xffffffffu, vg, o);
            }
            if (lane == 0) sums[pairs * NW + share] = make_float2(vf, vg);
        }
    }
    if (pairs == 0) return;
    if (tid == 0) {
        __threadfence();
        const bool last = atomicAdd(arrived + blockIdx.x, 1u) == NW - 1u;
        if (last) arrived[blockIdx.x] = 0u;     // for the next launch
        s_last = last;
        __threadfence();
    }
    __syncthreads();
    if (!s_last) return;
    for (int e = tid; e < 2 * pairs; e += 32 * kSumWarps) {
        if (ce[e] < 0) continue;
        float S = 0.f;
#pragma unroll
        for (int w = 0; w < NW; w++) {
            const float2 v = __ldcg(sums + (e >> 1) * NW + w);
            S += (e & 1) ? v.y : v.x;
        }
        const float v = (2.0f * S + P.diag) * P.norm;
        const unsigned long long key = cand_emit(a, c, ce[e], v);
        if (key) atomicMax(a.best_key + c, key);
    }
}

// ===========================================================================
// k_topk: one CTA per curve, top_k local maxima of the coarse periodogram.
// Local maximum: v[k] > v[k-1] and v[k] >= v[k+1]; ends use one neighbour.
// Order: value descending, ties to the lower k (larger key).  The row is gone
// through once per peak; with one warp per curve that was a chain of
// top_k K / 32 dependent steps (150 us at K = 4,999, top_k = 10, however few
// curves), with 256 threads it is top_k K / 256.
// ===========================================================================
constexpr int kTopkThreads = 256;

__global__ void __launch_bounds__(kTopkThreads) k_topk(const TopkArgs a)
{
    __shared__ unsigned long long s_best[kTopkThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (a.fb_count && (int)blockIdx.x >= *a.fb_count) return;
    const int slot = a.fb_count ? a.fb_slots[blockIdx.x] : a.slot_begin + (int)blockIdx.x;
    const int c = a.order[slot];
    const float* v = a.coarse + (int64_t)c * a.n_freq;
    const int64_t K = a.n_freq;
    unsigned long long prev = ~0ull;
    int cnt = 0;
    for (int r = 0; r < a.top_k; r++) {
        unsigned long long best = 0ull;
        for (int64_t k = tid; k < K; k += kTopkThreads) {
            const float x = v[k];
            const bool lok = (k == 0) || (x > v[k - 1]);
            const bool rok = (k == K - 1) || (x >= v[k + 1]);
            if (lok && rok && !excluded_k(a.ex.coarse_k, a.ex.n, k)) {
                const unsigned long long key = make_key(x, (uint32_t)k);
                if (key < prev && key > best) best = key;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long other = __shfl_xor_sync(0xffffffffu, best, o);
            best = other > best ? other : best;
        }
        __syncthreads();
        if (lane == 0) s_best[warp] = best;
        __syncthreads();
#pragma unroll
        for (int w = 0; w < kTopkThreads / 32; w++) best = s_best[w] > best ? s_best[w] : best;
        if (best == 0ull) break;
        if (tid == 0) a.peaks[(int64_t)c * a.top_k + r] = (int32_t)(0xffffffffu - (uint32_t)(best & 0xffffffffu));
        prev = best;
        cnt++;
    }
    if (tid == 0) a.n_peaks[c] = cnt;
}

// ===========================================================================
// k_finalize: decode the best keys, apply the discriminator.
// ===========================================================================

__global__ void k_finalize(const FinalArgs a)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c == 0 && a.status_out) *a.status_out = *a.status;
    if (c >= a.n_curves) return;
    const unsigned long long key = a.best_key[c];
    int64_t kout = -1;   // no admissible candidate
    double f = __longlong_as_double(0x7ff8000000000000ll);
    float v = __int_as_float(0x7fc00000);
    if (key != 0ull) {
        v = from_orderable((uint32_t)(key >> 32));
        const uint32_t idx = 0xffffffffu - (uint32_t)(key & 0xffffffffu);
        kout = (int64_t)idx;
        if (a.hierarchical == CP_SEARCH_BANDS) {
            const uint32_t k = (uint32_t)a.trials[(int64_t)c * a.n_trials + idx];   // list position -> grid index
            kout = (int64_t)k;
            f = __dadd_rn(a.f_min, __dmul_rn((double)k, a.df));
        } else if (a.hierarchical) {
            const int W = 2 * a.fine_half + 1;
            const int p = (int)(idx / (uint32_t)W);
            const int j = (int)(idx % (uint32_t)W) - a.fine_half;
            const double fpk = __dadd_rn(a.f_min, __dmul_rn((double)a.peaks[(int64_t)c * a.top_k + p], a.coarse_df));
            f = __dadd_rn(fpk, __dmul_rn((double)j, a.fine_df));
        } else {
            f = __dadd_rn(a.f_min, __dmul_rn((double)idx, a.df));
        }
    }
    if (a.best_idx) a.best_idx[c] = kout;
    if (a.best_freq) a.best_freq[c] = f;
    if (a.best_stat) a.best_stat[c] = v;
    if (a.is_periodic) a.is_periodic[c] = v > a.cp[c].th ? 1 : 0;
    if (a.psnr) a.psnr[c] = a.cp[c].psnr;
}

__global__ void k_zero_u64(unsigned long long* p, int64_t n)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) p[i] = 0ull;
}

}  // namespace cpk

// ---------------------------------------------------------------------------
// Launchers used by the host API (C++ linkage, internal to the library).
// ---------------------------------------------------------------------------
namespace cpk {

static bool stats_wide(const StatsArgs& a, int n_curves)
{
    return (a.ip_blocks > 0 && a.np2max >= 1024) || (a.np2max >= 512 && n_curves <= 128);
}

cudaError_t launch_stats(const StatsArgs& a, int n_curves, cudaStream_t s)
{
    const size_t smem = stats_smem_bytes(a.np2max);
    // few curves, not the shortest: more threads for each curve's sort and sums
    if (stats_wide(a, n_curves)) k_stats<1024><<<n_curves, 1024, smem, s>>>(a);
    else k_stats<kStatsThreads><<<n_curves, kStatsThreads, smem, s>>>(a);
    cudaError_t e = cudaGetLastError();
    const size_t ysmem = (size_t)a.np2max * sizeof(float);
    if (e == cudaSuccess && a.ip_blocks) {
        k_ip<<<dim3(n_curves, a.ip_blocks), kStatsThreads, ysmem, s>>>(a);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess && a.wrho) {
        k_wrho<<<dim3(n_curves, a.rho_blocks), kStatsThreads, ysmem, s>>>(a);
        e = cudaGetLastError();
    }
    return e;
}

cudaError_t launch_sigma_t_rule(const float* mags, const int64_t* offsets, int n_curves, int np2max, float* out,
                                cudaStream_t s)
{
    const size_t smem = (size_t)np2max * sizeof(float);
    cudaError_t e = raise_dyn_smem((const void*)k_sigma_t_rule, smem);
    if (e != cudaSuccess) return e;
    k_sigma_t_rule<<<n_curves, kStatsThreads, smem, s>>>(mags, offsets, np2max, out);
    return cudaGetLastError();
}

cudaError_t launch_build_w(const BuildWArgs& a, cudaStream_t s)
{
    const int64_t tiles = a.tile_end - a.tile_begin;
    if (tiles <= 0) return cudaSuccess;
    k_build_w<<<(unsigned)((tiles + 7) / 8), 256, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_pair_direct(const PairArgs& a, int warps, int grid, size_t smem, cudaStream_t s)
{
    if (a.fb_count) k_pair_direct<true, 16><<<grid, kPairThreads, smem, s>>>(a);
    else if (warps == 4) k_pair_direct<false, 4><<<grid, 128, smem, s>>>(a);
    else k_pair_direct<false, 16><<<grid, kPairThreads, smem, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_topk(const TopkArgs& a, cudaStream_t s)
{
    const int n = a.slot_end - a.slot_begin;
    if (n <= 0) return cudaSuccess;
    k_topk<<<n, kTopkThreads, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_finalize(const FinalArgs& a, cudaStream_t s)
{
    k_finalize<<<(a.n_curves + 255) / 256, 256, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_confirm(const PairArgs& a, void* part, int64_t part_ld, int chunk, int n_sm, int max_n, cudaStream_t s)
{
    const int n = a.slot_end - a.slot_begin;
    if (n <= 0) return cudaSuccess;
    if (n > kConfirmMaxChunk || a.n_cand != kConfirmCand) return cudaErrorInvalidValue;
    // tiles per item: one to four a warp, so that there are a few items for every SM
    const int64_t tiles = (int64_t)n * tiles_of(max_n);
    int group = kConfirmWarps;
    while (group < 4 * kConfirmWarps && tiles / group > 4 * n_sm) group += kConfirmWarps;
    // trig table: at least one frequency pair of the longest curve
    const int npad = (max_n + kTile - 1) & ~(kTile - 1);
    const int smem = std::min(kConfirmSmem, std::max(npad * 28, 104 * 1024));
    k_confirm<<<n_sm, kConfirmThreads, smem, s>>>(a, static_cast<f2*>(part), part_ld, group, smem);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    // after the tiles' sums: the shares' sums of every slot and frequency pair, the slots' arrival counts
    float2* shares = reinterpret_cast<float2*>(static_cast<f2*>(part) + part_ld * chunk);
    unsigned int* arrived = reinterpret_cast<unsigned int*>(shares + kConfirmMaxChunk * kConfirmCand / 2 * 16);
    k_confirm_sum<<<dim3(n, kPairThreads / 32), 32 * kSumWarps, 0, s>>>(a, static_cast<const f2*>(part), part_ld, shares,
                                                                       arrived);
    return cudaGetLastError();
}

size_t confirm_extra_bytes()
{
    return (size_t)kConfirmMaxChunk * (kConfirmCand / 2) * (16 * sizeof(float2) + sizeof(unsigned int));
}

size_t confirm_bytes(int max_n) { return (size_t)tiles_of(max_n) * 32 * sizeof(f2) * (kConfirmCand / 2); }

cudaError_t prepare_selected(size_t pair_smem)
{
    cudaError_t e = raise_dyn_smem((const void*)k_confirm, kConfirmSmem);
    return e == cudaSuccess ? raise_dyn_smem((const void*)k_pair_direct<true, 16>, pair_smem) : e;
}

int pair_direct_threads() { return kPairThreads; }

size_t stats_smem_bytes(int np2max) { return (size_t)np2max * (sizeof(double) + 3 * sizeof(float)); }

namespace {
std::mutex g_smem_mutex;
std::map<std::pair<const void*, int>, size_t> g_smem_limit;   // (kernel, device) -> limit set
}  // namespace

cudaError_t raise_dyn_smem(const void* func, size_t bytes)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(g_smem_mutex);
    size_t& cur = g_smem_limit[std::make_pair(func, dev)];
    if (bytes <= cur) return cudaSuccess;
    e = cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) cur = bytes;
    return e;
}

cudaError_t prepare_kernels(int np2max, size_t pair_smem)
{
    cudaError_t e = raise_dyn_smem((const void*)k_stats<kStatsThreads>, stats_smem_bytes(np2max));
    if (e == cudaSuccess) e = raise_dyn_smem((const void*)k_stats<1024>, stats_smem_bytes(np2max));
    if (e != cudaSuccess) return e;
    e = raise_dyn_smem((const void*)k_pair_direct<false, 4>, pair_smem);
    if (e != cudaSuccess) return e;
    return raise_dyn_smem((const void*)k_pair_direct<false, 16>, pair_smem);
}

cudaError_t pair_direct_occupancy(int* blocks_per_sm, int warps, size_t smem)
{
    const void* k = warps == 4 ? (const void*)k_pair_direct<false, 4> : (const void*)k_pair_direct<false, 16>;
    cudaError_t e = raise_dyn_smem(k, smem);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k, 32 * warps, smem);
}

cudaError_t launch_zero_u64(unsigned long long* p, int64_t n, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    k_zero_u64<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(p, n);
    return cudaGetLastError();
}

}  // namespace cpk
