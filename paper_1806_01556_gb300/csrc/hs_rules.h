// How the harmonic sums cut their work into CTAs (host code only).
#pragma once
#include "fdas_internal.cuh"

namespace fdas {
namespace {

// Rows and fundamental columns of the harmonic sum: |i| <= hs_rows, j < hs_end. All of them, or, when the
// convolution took HP_1, those with at least two planes.
inline int hs_rows(const fdas_params &p, bool hp1_done) {
    const int c = (p.n_temp - 1) / 2;
    return hp1_done ? c / 2 : c;
}

inline int hs_end(const fdas_params &p, size_t n, bool hp1_done) {
    return !hp1_done ? (int)n : p.n_harm < 2 ? 0 : (int)((n - 1) / 2 + 1);
}

// Columns per unit for `total` fundamental columns per row, on `sms` SMs. Large units amortise a CTA's start, but the
// units in flight must touch less than L2 holds. Measured at 2^21 bins, 85 rows, in us:
//   search (rows with 2 planes or more): 2048 columns 600, 4096: 600, 8192: 626;
//   all rows (where most units only stream their own row): 4096: 187, 8192: 169, 16384: 205.
// Fewer columns when that would leave less than 9 units per SM, but 512 at least. The line is one of balance, not of
// the CTAs that an SM holds (7, or 4 with more than 8 planes): all rows with 8 (16) planes take 45.0, 43.4, 43.9
// (59.4, 53.4, 62.3) us with 1024, 2048, 4096 columns at 65536 bins, where it gives 2048, and 55.0, 50.7, 51.6 (69.4,
// 65.6, 76.0) us with 2048, 4096, 8192 columns at 200003 bins, where it gives 8192. A search with 1024 (512, 256)
// columns takes 19.3 (18.5, 18.5) us at 4099 bins, 22.1 (20.9, 21.4) at 10115, 28.7 (26.6, 27.1) with 16 planes at 18248.
inline int hs_columns(int rows, long long total, bool hp1_done, int sms) {
    int cols = hp1_done ? 4096 : 8192;
    while (cols > 512 && (2 * rows + 1) * ((total + cols - 1) / cols) < 9ll * sms) cols >>= 1;
    return cols;
}

// The sum by the highest harmonic: rows per CTA for `blocks` column blocks of n_temp rows each, on `sms` SMs. A CTA's
// setup costs about as much as two rows; the work spreads over two CTAs per SM; at the end the GPU waits for CTAs that
// started late, which a last group of fewer rows, started last, makes shorter. The weights are fitted to sweeps from 4099 to 2^20 bins, where the
// choice stays within about 2% of the best. The groups interleave (but for the last), so that the rows around a
// strong signal, which all cross their thresholds, fall to different CTAs. A search with tones in us, with
// neighbouring rows and about eight CTAs per slot, and with this rule: 8 planes 4099 bins 28, 27, 27000 bins 63, 49,
// 65536 bins 98, 88, 2^20 bins 796, 788; 16 planes 9169 bins 116, 69, 95815 bins 334, 305, 262147 bins 745, 738.
// (Rows in the order of a golden-section stride: 806 and 755 at the last sizes.)
constexpr int kMaxRows = 43;
inline int rows_per_cta(int blocks, int n_temp, int sms) {
    constexpr float kSetup = 2.0f;
    const float slots = 2.0f * (float)sms;
    int best = 1;
    float best_cost = 0.0f;
    for (int r = 1; r <= kMaxRows && r <= n_temp; ++r) {
        const int groups = (n_temp + r - 1) / r, last = n_temp - (groups - 1) * r;
        if (4 * last < r) continue;  // a setup for next to nothing
        const float one = (float)r + kSetup;  // a CTA, in rows
        const float all = (float)blocks * ((float)n_temp + kSetup * (float)groups) / slots +
                          0.3f * ((float)last + kSetup) + 0.5f * one;
        const float cost = all > one ? all : one;
        if (best_cost == 0.0f || cost < best_cost) {
            best = r;
            best_cost = cost;
        }
    }
    return best;
}

}  // namespace
}  // namespace fdas
