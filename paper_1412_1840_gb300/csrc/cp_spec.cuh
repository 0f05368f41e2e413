// cp_spec.cuh -- the pair-spectrum evaluation of the direct form (cp_spec.cu):
// types and launchers shared with the host API.
//
// The periodic kernel is even and periodic in the phase, so (Eq. (taylor)
// regrouped by harmonic) the pair sum of Eq. (HP) is
//   S(f) = N (1 - ip) (1 - a_0) + 2 sum_{n=1}^{nh} a_n P(n f),
//   P(nu) = sum_{i<j} w_ij cos(2 pi nu (t_i - t_j)),
// and P does not depend on the trial frequency: one cosine transform of the
// pairs' time differences serves every frequency of the grid.
#pragma once
#include "cp_internal.cuh"

namespace cpk {

constexpr int kSpecMaxHarm = 64;       // harmonics kept per curve
constexpr int kSpecMinLogQ = 8;        // complex transform length 2^logq
constexpr int kSpecMaxLogQ = 22;
constexpr int kSpecOneLogQ = 13;       // up to this length one CTA transforms a curve
constexpr int kSpecCand = kConfirmCand;// frequencies per curve evaluated again by the pair sum
constexpr int kSpecMaxChunk = kConfirmMaxChunk;   // curves per chunk
constexpr double kSpecTail = 2e-8;     // harmonics left out: at most this much of the kernel's peak
constexpr double kSpecOver = 1.1;      // transform length over the highest frequency needed, at least

constexpr int kSpecBlock = 64;         // values per block at least (one item of the value kernels)
constexpr int kSpecPad = 8;            // pair-spectrum values kept before index 0 (P(-nu) = P(nu))

// Which frequencies a launch evaluates.
enum SpecStage : int { kSpecFull = 0, kSpecCoarse = 1, kSpecFine = 2, kSpecList = 3 };

// What the device decides for one curve (its sigma_t and span are known there).
struct SpecCurve {
    double cells_per_day;   // 2 H / L: grid cells per day of time difference
    double L;               // transform period in days: the pair spectrum's spacing is 1 / L
    int64_t H;              // cells of the half period, 2 Q
    int32_t nh;             // harmonics (0: the pair sum evaluates the curve)
    int32_t logq;           // Q = 2^logq
    int32_t support;        // cells that can be non-zero, a multiple of 4 (H: all)
    int32_t n_out;          // pair-spectrum values needed
    float one_minus_a0;
    int32_t seg;            // cells per spreading item
    int32_t whole;          // set when a curve's candidates do not fit its list
};

struct SpecArgs {
    CurveParams* cp;
    SpecCurve* sc;                // [n_curves]
    float* coef;                  // [n_curves * kSpecMaxHarm] a_1..
    const int32_t* order;
    const double* times;
    const float* yp;              // scaled magnitudes, caller's order
    uint64_t* xs;                 // sorted times in cells, 32.32 fixed point
    float* ys;                    // scaled magnitudes in time order
    int stage;                    // SpecStage
    int interp;                   // 0: frequencies (m0 + mq k) delta are entries of the pair spectrum
                                  // 1: any frequency up to f_top, by interpolation
    double delta;
    int64_t m0, mq;
    double f_top;
    int64_t n_freq;               // points of the row (full, coarse), of the grid (list)
    double f_min, f_max, step;    // uniform grid of the stage (fine: step of the window)
    double coarse_df;
    const int32_t* peaks;         // coarse peaks (peaks_out: where k_spec_rank writes them)
    int32_t* peaks_out;
    int32_t* n_peaks;
    int32_t top_k, fine_half;
    const int32_t* trials;
    int32_t n_trials;
    int slot_begin, slot_end;     // curves of this launch
    int np2max;
    int seg_max;                  // cells per spreading item at most
    int seg_items;                // spreading items per curve wanted
    float2* x;                    // chunk workspace: transform data, x_ld per curve
    int64_t x_ld;
    float* P;                     // pair spectrum, p_ld per curve (index 0 at kSpecPad)
    int64_t p_ld;
    float* rows;                  // values: row index = caller's curve, or slot - slot_begin
    int64_t row_ld;
    int rows_by_curve;
    unsigned int* vmax;           // [n_curves] largest admissible value (orderable bits)
    unsigned int* vtop;           // [n_curves] largest magnitude of any value, excluded ones too (float bits)
    unsigned int* vblk;           // the same per block of a launch's values, vb_ld per curve of the chunk
    int64_t vb_ld;
    int32_t* cand;                // [n_curves * kSpecCand] candidate entries, -1 after the last
    int32_t* fb_slots;            // slots that the pair sum evaluates whole
    int* fb_count;
    unsigned long long* queue;    // two work counters of the chunk: spreading, second transform pass
    const float2* tw;             // twiddle factors, see launch_spec_twiddle
    Exclusion ex;
};

constexpr int kSpecTwiddles = 11264;
cudaError_t launch_spec_twiddle(float2* tw, cudaStream_t s);   // fills kSpecTwiddles entries
cudaError_t spec_prepare(int np2max, int max_n, int seg);
int spec_seg_max(int max_n);           // cells per spreading item that shared memory holds
cudaError_t launch_spec_prep(const SpecArgs& a, cudaStream_t s);
// pair spectrum of one chunk (slot_end - slot_begin <= kSpecMaxChunk)
cudaError_t launch_spec_transform(const SpecArgs& a, int n_sm, int max_n, bool one_pass, bool two_pass, cudaStream_t s);
cudaError_t launch_spec_values(const SpecArgs& a, int n_sm, cudaStream_t s);   // the stage's values and their largest
cudaError_t launch_spec_select(const SpecArgs& a, cudaStream_t s);             // candidates for the best
cudaError_t launch_spec_peaks(const SpecArgs& a, cudaStream_t s);              // coarse points whose exact values matter
cudaError_t launch_spec_rank(const SpecArgs& a, cudaStream_t s);               // the coarse peaks, from exact values

// Host: harmonics needed at sigma_t for a truncation tail of kSpecTail (0: more than kSpecMaxHarm).
int spec_harmonics(double sigma_t);
// Host: log2 of the complex transform length for n_out values (0: too long).
int spec_logq(int64_t n_out);

}  // namespace cpk
