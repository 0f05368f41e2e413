// cp_prep.cu -- per-curve transforms around the periodogram search
// (arXiv:1412.1840):
//
//   cp_preprocess  Section 5.2: drop samples whose error bar is not below
//                  mean(e) + 3 std(e) (population std), discard curves with
//                  fewer than min_n samples left, fit x = a0 + a1 t by the
//                  weighted linear chi^2 of Eq. (chisquare) and subtract the
//                  fit when the Pearson correlation between the magnitudes and
//                  the fit exceeds 0.5.  The kept samples keep their order.
//   cp_whiten      Section 7.1 (multimodes): fold each curve at its P0
//                  (phase = frac(t / P0), equal phases by sample index),
//                  smooth the folded curve by a circular moving average of
//                  w = min(window, N) samples (folded positions k - w/2 ..
//                  k - w/2 + w - 1), subtract that template and return the
//                  samples in their original order.
//
// Every sum is FP64 in a fixed order.
#include <cmath>
#include <cstdint>
#include <cstring>
#include <memory>
#include <mutex>
#include <new>
#include <string>
#include <vector>

#include <cuda_runtime.h>

#include "cp.h"
#include "cp_internal.cuh"

namespace cpk {

constexpr int kPrepThreads = 256;

// The cleaning takes a warp per curve; two warps a block spread a field evenly.
constexpr int kCleanThreads = 64;

struct PrepStats {
    int32_t n_out, kept, detrended;
    float cut;                    // samples with e < cut are kept (the FP64 cut rounded up: the same samples)
    double a0, a1, r;
};

// FP64 runs at 1.7 operations/clk/SM here and bounds the per-curve statistics:
// with 256 threads a curve, the eleven block-wide sums cost more than the samples'
// own arithmetic (2048 curves of 60-1000 samples: 360 us).  A warp per curve, the
// count and the comparison with the cut outside FP64, and one pass for everything
// after the cut take 127 us; with the compaction (88 -> 20 us, the cut passed on
// instead of summed again), one synchronisation and pooled temporaries the call
// takes 286 us instead of 783.
__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Sum of f(i), i < n, as eight warps of a block of 256 threads would add it (each
// thread its samples, lanes by a butterfly, then the warps in order): the cut
// compares error bars that may all be equal with a sum that must not change.
template <typename F>
__device__ __forceinline__ double sum_as_256(int n, int lane, F f)
{
    double t = 0.0;
    double s[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    for (int i0 = lane; i0 < n; i0 += 256)
#pragma unroll
        for (int w = 0; w < 8; w++)
            if (i0 + 32 * w < n) s[w] = f(i0 + 32 * w, s[w]);
#pragma unroll
    for (int w = 0; w < 8; w++) t += warp_sum(s[w]);
    return t;
}

__global__ void __launch_bounds__(kCleanThreads) k_prep_stats(const double* times, const float* mags,
                                                             const float* errs, const int64_t* offsets,
                                                             int n_curves, int min_n, PrepStats* out)
{
    const int lane = threadIdx.x & 31;
    const int c = (int)blockIdx.x * (kCleanThreads / 32) + (int)(threadIdx.x >> 5);
    if (c >= n_curves) return;                  // whole warps
    const int64_t off = offsets[c];
    const int n = (int)(offsets[c + 1] - off);

    // error-bar cut: e_i < mean + 3 std (population)
    const double mean = sum_as_256(n, lane, [&](int i, double s) { return s + (double)errs[off + i]; }) / (double)n;
    const double var = sum_as_256(n, lane, [&](int i, double s) {
                           const double d = (double)errs[off + i] - mean;
                           return fma(d, d, s);
                       }) / (double)n;
    const float cutf = __double2float_ru(mean + 3.0 * sqrt(var));

    // weighted chi^2 sums (weights 1 / e^2) and unweighted moments of the kept samples, about the
    // first kept sample: single-pass sums then lose nothing to a large common offset, and a dropped
    // sample (not finite, or a sentinel value) has no part in them
    int first = 0;
    for (int i0 = 0; i0 < n; i0 += 32) {
        const int i = i0 + lane;
        const uint32_t kept = __ballot_sync(0xffffffffu, i < n && errs[off + i] < cutf);
        if (kept) {
            first = i0 + __ffs(kept) - 1;
            break;
        }
    }
    const double tref = times[off + first], xref = (double)mags[off + first];
    int cnt = 0;
    double S = 0, St = 0, Sx = 0, Stt = 0, Stx = 0, ut = 0, ux = 0, utt = 0, utx = 0, uxx = 0;
    for (int i = lane; i < n; i += 32) {
        const float ef = errs[off + i];
        if (!(ef < cutf)) continue;
        const double e = (double)ef, t = times[off + i] - tref, x = (double)mags[off + i] - xref;
        const double w = 1.0 / (e * e), wt = w * t;
        cnt++;
        S += w;
        St += wt;
        Sx = fma(w, x, Sx);
        Stt = fma(wt, t, Stt);
        Stx = fma(wt, x, Stx);
        ut += t;
        ux += x;
        utt = fma(t, t, utt);
        utx = fma(t, x, utx);
        uxx = fma(x, x, uxx);
    }
    __syncwarp();
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    S = warp_sum(S);
    St = warp_sum(St);
    Sx = warp_sum(Sx);
    Stt = warp_sum(Stt);
    Stx = warp_sum(Stx);
    ut = warp_sum(ut);
    ux = warp_sum(ux);
    utt = warp_sum(utt);
    utx = warp_sum(utx);
    uxx = warp_sum(uxx);
    if (lane == 0) {
        double a0 = 0.0, a1 = 0.0, r = 0.0;
        if (cnt >= 2) {
            const double det = S * Stt - St * St, k = (double)cnt;
            a1 = (S * Stx - St * Sx) / det;
            a0 = (Stt * Sx - St * Stx) / det + xref - a1 * tref;
            // Pearson correlation of the kept magnitudes with the fit a0 + a1 t
            const double sxt = utx - ut * ux / k, sxx = uxx - ux * ux / k, stt = utt - ut * ut / k;
            const double sff = a1 * a1 * stt;
            r = (sxx <= 0.0 || sff <= 0.0) ? 0.0 : a1 * sxt / sqrt(sxx * sff);
            if (det == 0.0) {                    // one time only: no slope, no correlation
                a0 = Sx / S + xref;
                a1 = r = 0.0;
            }
        }
        PrepStats p;
        p.n_out = cnt;
        p.kept = cnt >= min_n;
        p.detrended = r > 0.5;
        p.cut = cutf;
        p.a0 = a0;
        p.a1 = a1;
        p.r = r;
        out[c] = p;
    }
}

// First output sample of every curve (kept samples of the kept curves before it); one CTA.
__global__ void __launch_bounds__(1024) k_prep_offsets(const PrepStats* st, int n_curves, int64_t* out_off)
{
    __shared__ long long s_w[32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    long long base = 0;
    for (int c0 = 0; c0 < n_curves; c0 += 1024) {
        const int c = c0 + tid;
        const long long v = c < n_curves && st[c].kept ? st[c].n_out : 0;
        long long incl = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) s_w[warp] = incl;
        __syncthreads();
        long long before = base;
        for (int w = 0; w < 32; w++) {
            if (w < warp) before += s_w[w];
            base += s_w[w];
        }
        if (c < n_curves) out_off[c] = before + incl - v;
        __syncthreads();
    }
}

// Order-preserving compaction of the kept samples, fit removed where flagged; a warp per curve.
__global__ void __launch_bounds__(kCleanThreads) k_prep_compact(const double* times, const float* mags,
                                                               const float* errs, const int64_t* offsets,
                                                               const PrepStats* st, const int64_t* out_off,
                                                               int n_curves, double* out_t, float* out_x, float* out_e)
{
    const int lane = threadIdx.x & 31;
    const int c = (int)blockIdx.x * (kCleanThreads / 32) + (int)(threadIdx.x >> 5);
    if (c >= n_curves) return;
    const PrepStats P = st[c];
    if (!P.kept) return;
    const int64_t off = offsets[c];
    const int n = (int)(offsets[c + 1] - off);
    int64_t o = out_off[c];
    constexpr int U = 4;                         // rounds whose loads are in flight together
    for (int i0 = 0; i0 < n; i0 += 32 * U) {
        float e[U], x[U];
        double t[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int i = min(i0 + 32 * u + lane, n - 1);
            e[u] = errs[off + i];
            t[u] = times[off + i];
            x[u] = mags[off + i];
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
            const bool keep = i0 + 32 * u + lane < n && e[u] < P.cut;
            const uint32_t bal = __ballot_sync(0xffffffffu, keep);
            if (keep) {
                const int64_t pos = o + __popc(bal & ((1u << lane) - 1u));
                out_t[pos] = t[u];
                out_x[pos] = P.detrended ? (float)((double)x[u] - (P.a0 + P.a1 * t[u])) : x[u];
                out_e[pos] = e[u];
            }
            o += __popc(bal);
        }
    }
}

// Whitening: bitonic sort of (phase, sample) pairs, circular moving average
// from FP64 prefix sums, subtraction, scatter back to the sample positions.
// Phases are compared as the integers of their bits (all in [0, 1)): FP64
// comparisons, one thread's chain over all prefix sums and FP64 divisions took
// most of 550 us for 2048 curves.  Strides below 32 of the sort stay within a
// warp's registers, a block barrier separates only the longer ones: 129 us, the
// call 168 us instead of 755.
__device__ __forceinline__ void order_pair(unsigned long long& k, int& i, unsigned long long ok, int oi, bool keep_small)
{
    const bool less = ok < k || (ok == k && oi < i);     // the other comes first
    if (less == keep_small) {
        k = ok;
        i = oi;
    }
}

__global__ void __launch_bounds__(kPrepThreads) k_whiten(const double* times, const float* mags,
                                                         const int64_t* offsets, const double* p0, int window,
                                                         int np2max, float* out)
{
    extern __shared__ __align__(16) unsigned char smem[];
    unsigned long long* ph = reinterpret_cast<unsigned long long*>(smem);   // np2max
    double* pre = reinterpret_cast<double*>(ph + np2max);     // np2max + 1 prefix sums (folded order)
    int32_t* idx = reinterpret_cast<int32_t*>(pre + np2max + 1);
    float* xs = reinterpret_cast<float*>(idx + np2max);       // folded magnitudes
    constexpr int kSeg = 64;
    __shared__ double s_carry[kMaxN / kSeg];
    const int c = blockIdx.x, tid = threadIdx.x, lane = tid & 31;
    const int64_t off = offsets[c];
    const int n = (int)(offsets[c + 1] - off);
    const double P = p0[c];
    if (!(P > 0.0) || !isfinite(P)) {
        for (int i = tid; i < n; i += kPrepThreads) out[off + i] = mags[off + i];
        return;
    }
    int np2 = 32;
    while (np2 < n) np2 <<= 1;
    const double rP = 1.0 / P;
    // tiny, huge and non-finite quotients keep the plain division
    const bool easy = P > 1e-100 && P < 1e100;
    for (int i = tid; i < np2; i += kPrepThreads) {
        unsigned long long key = ~0ull;
        if (i < n) {
            const double t = times[off + i];
            const double q = easy && fabs(t) < 1e100 && fabs(t) > 1e-100 ? div_by(t, P, rP) : t / P;
            key = (unsigned long long)__double_as_longlong(q - floor(q)) & 0x7fffffffffffffffull;
        }
        ph[i] = key;
        idx[i] = i;
    }
    // ascending by (phase, sample index)
    for (int k = 32; k <= np2; k <<= 1) {
        for (int j = k >> 1; j >= 32; j >>= 1) {
            __syncthreads();
            for (int p = tid; p < np2 >> 1; p += kPrepThreads) {
                const int i = ((p & ~(j - 1)) << 1) | (p & (j - 1)), o = i | j;
                const unsigned long long u = ph[i], v = ph[o];
                const int iu = idx[i], iv = idx[o];
                if ((u > v || (u == v && iu > iv)) == ((i & k) == 0)) {
                    ph[i] = v; ph[o] = u;
                    idx[i] = iv; idx[o] = iu;
                }
            }
        }
        __syncthreads();
        for (int i = tid; i < np2; i += kPrepThreads) {       // whole warps: np2 is a multiple of 32
            unsigned long long key = ph[i];
            int ix = idx[i];
            for (int kk = k == 32 ? 2 : k; kk <= k; kk <<= 1) {
#pragma unroll
                for (int j = 16; j > 0; j >>= 1) {
                    if (j >= kk) continue;
                    const unsigned long long ok = __shfl_xor_sync(0xffffffffu, key, j);
                    const int oi = __shfl_xor_sync(0xffffffffu, ix, j);
                    order_pair(key, ix, ok, oi, ((i & kk) == 0) == ((lane & j) == 0));
                }
            }
            ph[i] = key;
            idx[i] = ix;
        }
    }
    __syncthreads();
    for (int k = tid; k < n; k += kPrepThreads) xs[k] = mags[off + idx[k]];
    __syncthreads();
    // prefix sums of the folded magnitudes: 64-sample blocks, then the blocks' carries
    const int nseg = (n + kSeg - 1) / kSeg;
    for (int sgi = tid; sgi < nseg; sgi += kPrepThreads) {
        double acc = 0.0;
        const int end = min(n, (sgi + 1) * kSeg);
        for (int k = sgi * kSeg; k < end; k++) {
            acc += (double)xs[k];
            pre[k + 1] = acc;
        }
    }
    __syncthreads();
    if (tid == 0) {
        pre[0] = 0.0;
        double carry = 0.0;
        for (int sgi = 0; sgi < nseg; sgi++) {
            s_carry[sgi] = carry;
            carry += pre[min(n, (sgi + 1) * kSeg)];
        }
    }
    __syncthreads();
    for (int k = tid; k < n; k += kPrepThreads) pre[k + 1] += s_carry[k / kSeg];
    __syncthreads();
    const int w = window < n ? window : n;
    const double total = pre[n], wd = (double)w, rw = 1.0 / wd;
    for (int k = tid; k < n; k += kPrepThreads) {
        // folded positions k - w/2 .. k - w/2 + w - 1, circular
        int a = k - w / 2, b = a + w;                          // [a, b)
        double sum;
        if (a >= 0 && b <= n) {
            sum = pre[b] - pre[a];
        } else if (a < 0) {
            sum = pre[b] + (total - pre[n + a]);
        } else {
            sum = (total - pre[a]) + pre[b - n];
        }
        out[off + idx[k]] = (float)((double)xs[k] - div_by(sum, wd, rw));
    }
}

size_t whiten_smem_bytes(int np2max)
{
    return (size_t)np2max * 8 + (size_t)(np2max + 1) * 8 + (size_t)np2max * 4 + (size_t)np2max * 4;
}

}  // namespace cpk

using namespace cpk;

namespace {

cp_status pfail(cp_status s, const std::string& m) { return cpk::set_error(s, m.c_str()); }

#define PREP_CUDA(call)                                                                 \
    do {                                                                                \
        cudaError_t e_ = (call);                                                        \
        if (e_ != cudaSuccess) {                                                        \
            cudaGetLastError();                                                         \
            st = pfail(e_ == cudaErrorMemoryAllocation ? CP_ENOMEM : CP_ECUDA,          \
                       std::string(#call) + ": " + cudaGetErrorString(e_));             \
            goto done;                                                                  \
        }                                                                               \
    } while (0)

cp_status check_csr(const int64_t* offsets, int64_t n_curves, int min_size, const char* who)
{
    if (!offsets) return pfail(CP_EINVAL, std::string(who) + ": null offsets");
    if (n_curves < 1 || n_curves > ((int64_t)1 << 30)) return pfail(CP_EINVAL, std::string(who) + ": bad n_curves");
    if (offsets[0] != 0) return pfail(CP_EINVAL, std::string(who) + ": offsets[0] must be 0");
    for (int64_t c = 0; c < n_curves; c++) {
        const int64_t n = offsets[c + 1] - offsets[c];
        if (n < min_size) return pfail(CP_EINVAL, std::string(who) + ": curve " + std::to_string(c) + " is too short");
        if (n > kMaxN) return pfail(CP_EUNSUPPORTED, std::string(who) + ": curve " + std::to_string(c) + " exceeds cp_max_points()");
    }
    return CP_OK;
}

bool on_device(const void* p)
{
    cudaPointerAttributes at{};
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

// Temporaries of the two calls come from a memory pool per device, in stream
// order: cudaMalloc and cudaFree took 0.2 to 0.3 ms a call.  The pool keeps at
// most kPoolKeep bytes between calls; freed memory beyond that goes back to the
// device at the next synchronisation.  Pools are thread safe, and an allocation is
// only handed to another stream after its own stream's work on it has completed.
constexpr uint64_t kPoolKeep = 16u << 20;

cudaError_t pool_alloc(void** p, size_t bytes, cudaStream_t s)
{
    static std::mutex mutex;
    static cudaMemPool_t pools[64];          // by device ordinal
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 64) return cudaMallocAsync(p, bytes, s);
    cudaMemPool_t pool = nullptr;
    {
        std::lock_guard<std::mutex> lock(mutex);
        if (!pools[dev]) {
            cudaMemPoolProps props{};
            props.allocType = cudaMemAllocationTypePinned;
            props.location.type = cudaMemLocationTypeDevice;
            props.location.id = dev;
            e = cudaMemPoolCreate(&pool, &props);
            if (e != cudaSuccess) return e;
            uint64_t keep = kPoolKeep;
            e = cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
            if (e != cudaSuccess) {
                cudaMemPoolDestroy(pool);
                return e;
            }
            pools[dev] = pool;
        }
        pool = pools[dev];
    }
    return cudaMallocFromPoolAsync(p, bytes, pool, s);
}

size_t up256(size_t x) { return (x + 255) & ~(size_t)255; }

}  // namespace

extern "C" cp_status cp_preprocess(const double* times, const float* mags, const float* errs, const int64_t* offsets,
                                   int64_t n_curves, int32_t min_n, double* out_times, float* out_mags,
                                   float* out_errs, int64_t* out_offsets, uint8_t* flags, double* fit,
                                   void* cuda_stream)
{
    if (!times || !mags || !errs || !out_times || !out_mags || !out_errs || !out_offsets)
        return pfail(CP_EINVAL, "cp_preprocess: null argument");
    if (min_n < 1) return pfail(CP_EINVAL, "cp_preprocess: min_n must be >= 1");
    cp_status st = check_csr(offsets, n_curves, 1, "cp_preprocess");
    if (st != CP_OK) return st;
    for (const void* p : {(const void*)times, (const void*)mags, (const void*)errs, (const void*)out_times,
                          (const void*)out_mags, (const void*)out_errs})
        if (!on_device(p)) return pfail(CP_EINVAL, "cp_preprocess: inputs and outputs must be device memory");
    const cudaStream_t s = (cudaStream_t)cuda_stream;
    const int64_t nc = n_curves;
    char* tmp = nullptr;
    const size_t ob = up256((size_t)(nc + 1) * sizeof(int64_t));
    std::vector<PrepStats> h_st((size_t)nc);
    PREP_CUDA(pool_alloc((void**)&tmp, 2 * ob + (size_t)nc * sizeof(PrepStats), s));
    {
        int64_t* d_off = reinterpret_cast<int64_t*>(tmp);
        int64_t* d_oout = reinterpret_cast<int64_t*>(tmp + ob);
        PrepStats* d_st = reinterpret_cast<PrepStats*>(tmp + 2 * ob);
        const unsigned ctas = (unsigned)((nc + kCleanThreads / 32 - 1) / (kCleanThreads / 32));
        PREP_CUDA(cudaMemcpyAsync(d_off, offsets, (nc + 1) * sizeof(int64_t), cudaMemcpyHostToDevice, s));
        k_prep_stats<<<ctas, kCleanThreads, 0, s>>>(times, mags, errs, d_off, (int)nc, min_n, d_st);
        PREP_CUDA(cudaGetLastError());
        k_prep_offsets<<<1, 1024, 0, s>>>(d_st, (int)nc, d_oout);
        PREP_CUDA(cudaGetLastError());
        k_prep_compact<<<ctas, kCleanThreads, 0, s>>>(times, mags, errs, d_off, d_st, d_oout, (int)nc, out_times, out_mags,
                                                     out_errs);
        PREP_CUDA(cudaGetLastError());
        PREP_CUDA(cudaMemcpyAsync(h_st.data(), d_st, nc * sizeof(PrepStats), cudaMemcpyDeviceToHost, s));
        PREP_CUDA(cudaStreamSynchronize(s));
    }
    out_offsets[0] = 0;
    for (int64_t c = 0; c < nc; c++) {
        out_offsets[c + 1] = out_offsets[c] + (h_st[c].kept ? h_st[c].n_out : 0);
        if (flags) flags[c] = (uint8_t)((h_st[c].kept ? 1 : 0) | (h_st[c].kept && h_st[c].detrended ? 2 : 0));
        if (fit) {
            fit[3 * c] = h_st[c].a0;
            fit[3 * c + 1] = h_st[c].a1;
            fit[3 * c + 2] = h_st[c].r;
        }
    }
done:
    if (tmp) cudaFreeAsync(tmp, s);
    return st;
}

extern "C" cp_status cp_whiten(const double* times, const float* mags, const int64_t* offsets, int64_t n_curves,
                               const double* p0, int32_t window, float* out_mags, void* cuda_stream)
{
    if (!times || !mags || !p0 || !out_mags) return pfail(CP_EINVAL, "cp_whiten: null argument");
    if (window < 1) return pfail(CP_EINVAL, "cp_whiten: window must be >= 1");
    cp_status st = check_csr(offsets, n_curves, 1, "cp_whiten");
    if (st != CP_OK) return st;
    for (const void* p : {(const void*)times, (const void*)mags, (const void*)out_mags})
        if (!on_device(p)) return pfail(CP_EINVAL, "cp_whiten: times, mags and out_mags must be device memory");
    const cudaStream_t s = (cudaStream_t)cuda_stream;
    const int64_t nc = n_curves;
    int max_n = 1;
    for (int64_t c = 0; c < nc; c++) max_n = std::max(max_n, (int)(offsets[c + 1] - offsets[c]));
    int np2 = 32;
    while (np2 < max_n) np2 <<= 1;
    const size_t smem = whiten_smem_bytes(np2);
    char* tmp = nullptr;
    // offsets and periods in one copy
    const size_t in_bytes = (size_t)(2 * nc + 1) * 8;
    const std::unique_ptr<char[]> h_in(new (std::nothrow) char[in_bytes]);
    if (!h_in) return pfail(CP_ENOMEM, "cp_whiten: host allocation failed");
    std::memcpy(h_in.get(), offsets, (size_t)(nc + 1) * 8);
    std::memcpy(h_in.get() + (nc + 1) * 8, p0, (size_t)nc * 8);
    PREP_CUDA(pool_alloc((void**)&tmp, in_bytes, s));
    PREP_CUDA(cudaMemcpyAsync(tmp, h_in.get(), in_bytes, cudaMemcpyHostToDevice, s));
    PREP_CUDA(raise_dyn_smem((const void*)k_whiten, smem));
    k_whiten<<<(unsigned)nc, kPrepThreads, smem, s>>>(times, mags, reinterpret_cast<const int64_t*>(tmp),
                                                      reinterpret_cast<const double*>(tmp + (nc + 1) * 8), window, np2,
                                                      out_mags);
    PREP_CUDA(cudaGetLastError());
    PREP_CUDA(cudaStreamSynchronize(s));
done:
    if (tmp) cudaFreeAsync(tmp, s);
    if (st != CP_OK) cudaStreamSynchronize(s);       // the copy may still read h_in
    return st;
}
