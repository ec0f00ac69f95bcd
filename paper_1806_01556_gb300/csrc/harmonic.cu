// Harmonic summing with threshold detection (Sec. 2.2, Algorithm 1).
//
// Stretch read by fundamental (the default): HP_k(i, j) = sum_{l=1..k} P[c + l*i][l*j] on
// D_k = {|k*i| <= c, k*j <= n-1}, summed in float32 in the order l = 1, 2, ..., k. As in the
// paper's MultipleHP kernels, all planes are computed at once and no HP plane is stored: one
// thread owns one fundamental (i, j) and keeps the running sum in a register.
//
// GB300 mapping:
//   fdas_hs_reset    zeroes the per-plane crossing counters and peak keys in the workspace.
//   fdas_hs_sum      every row in one launch (the comment at the kernel says how it is split).
//                    Crossings are rare and take a separate path: a ballot, one atomicAdd per warp,
//                    and a prefix popcount for each lane's slot. Each candidate
//                    is one 64-bit key whose ascending order is the canonical order (power desc,
//                    i asc, j asc).
//                    (harmonic_highest.cu has the kernel for FDAS_INDEX_HIGHEST.)
//   fdas_hs_finalize one CTA per plane. A bitonic sort of the raw keys (2, 4 or 16 keys per thread in
//                    registers, shuffles for the middle strides, shared memory for the largest), then
//                    the top cand_cap keys decoded into fdas_cand records, the counts and the peaks.
#include "hs_keys.cuh"
#include "hs_rules.h"

namespace fdas {
namespace {

constexpr int kFinThreads = 1024;

__global__ void fdas_hs_reset(unsigned long long *counters, unsigned long long *peaks, int n_harm) {
    pdl_trigger();
    pdl_wait();
    const int t = threadIdx.x;
    if (t < n_harm) {
        counters[t] = 0ull;
        peaks[t] = 0ull;
    }
}

// ---- the harmonic sum by fundamental: fdas_hs_sum --------------------------------------------------
//
// A unit (one CTA) is one row i with `cols` consecutive fundamental columns. Its warps take strips of
// 32 J columns; lane L of a strip holds j = s + L + 32 u, u < J, so each gather P[c + l i][l j] of a
// warp is one coalesced stride-l access, and a thread issues all J T gathers of a strip before it sums
// (T = number of terms, the planes l <= K(i) with l j <= n-1). T is constant on at most K(i) column
// ranges of a row, so every range runs code compiled for its T: no tests per element.
//
// Order of the units. Fundamental (i, j) reads row l i at column l j, so (i, j) and (i', j') share a
// plane point exactly when j / i = j' / i'. The units are therefore issued in the order of j / |i|: slab
// s takes, of every row +-a, the `a` column blocks [a s, a (s + 1)), and while it runs each plane row
// p = l i is read in one window [p s cols, p (s + 1) cols) by every fundamental that needs it. With 85
// rows a slab touches 1806 cols floats (30 MB for 4096 columns), so a point comes from DRAM once and its
// other readers find it in L2. Row 0, whose terms all lie in plane row 0, goes first.
//
// Measured at 2^21 bins, 85 rows, 8 planes, against one launch per group of rows with equal plane
// counts, row after row, three launches side by side: DRAM reads 1262 -> 620 MB (the points that are
// needed at all: about 590 MB) at 6.0 TB/s, 128 -> 29 M warp instructions, the sums of a search
// 255 -> 103 us; all rows (fdas_harmonic_sum) 300 -> 145 us. What bounds it now is DRAM, at 90% of the
// measured copy rate (all rows: 800 MB, 80%).
//
// Bookkeeping. The hot path compares each running sum with one limit per plane, the smaller of the
// threshold and of the power that could still become the plane's peak (the peak key in the
// workspace, read once per unit and after each update, kept in shared memory). Only a strip that exceeds a
// limit takes hs_strip_slow, which sums it again, emits the crossings and raises the peaks.

// 128 threads and 6 CTAs per SM or more (7 with up to 8 planes): a CTA's start overlaps the others' strips (with 6, 8
// warps and 3 CTAs: 109 us, 2 warps and 12 CTAs: 104 us, against 104 us, rows with 2 planes or more at 2^21 bins).
constexpr int kSumThreads = 128;
constexpr int kSumWarps = kSumThreads / 32;

// Gathers in flight per thread: J T = 16 to 32.
__host__ __device__ constexpr int hs_j(int t) { return t == 1 ? 16 : t <= 4 ? 8 : t <= 8 ? 4 : 2; }

// What a unit's strips share, in shared memory: all but `either` is read on the rare path only. Held in registers,
// its pointers and places took the hot path from 72 to 80, and one CTA less ran on an SM: all rows of 2^21 bins
// 154.8 us, 144.7 us this way.
template <int KMAX>
struct HsUnit {
    // Per plane: the threshold (+inf: not reported), the largest sum that cannot be the peak (hs_limit), and the
    // smaller of the two.
    float ta[KMAX], peak_limit[KMAX], either[KMAX];
    unsigned long long *raw, *counters, *peaks;
    int row;
    unsigned loc;  // (row << 24) | first column of the unit
};

// Plane row c, and i * ld: term l of column j is center[l * step + l * j].
struct HsRow {
    const float *center;
    long long step;
};

// Raises plane lane + 1's peak and limits, if key (this lane's; 0: none) wins.
template <int KMAX>
__device__ __forceinline__ void hs_raise(HsUnit<KMAX> &u, int lane, unsigned long long key) {
    if (key == 0ull) return;
    unsigned long long cur = *(volatile unsigned long long *)&u.peaks[lane];
    if (key > cur) {
        atomicMax(&u.peaks[lane], key);
        cur = key;
    }
    const float peak = hs_limit(cur, u.loc);
    *(volatile float *)&u.peak_limit[lane] = peak;
    *(volatile float *)&u.either[lane] = fminf(u.ta[lane], peak);
}

// Columns [lo, hi) of the row, one strip at most with T <= TMAX terms each, by one converged warp: every crossing
// emitted, the peaks and the limits raised. A spectrum pays for this in every strip that crosses, and a short one in
// the first strip of each warp, which finds no peak yet:
//   - Lane l - 1 updates plane l's counter once for the strip; a second pass over the columns that crossed writes
//     them. The planes' reductions are left out when no sum beats a peak (one test for all: a test for each plane costs
//     the first strips of a search of 4099 bins with 16 planes 2 us). With an update for every 32 columns and plane, one
//     after the other, and all reductions, the sum of every row of 2^21 bins took 970 us at 3 sigma, 4200 us at 2
//     sigma and 680 us with loud tones, now 537, 855 and 434 us.
//   - Code for TMAX = 1, 2, 4, 8 or 16 terms. One size for all: 583, 776 and 458 us, with 16 planes 458 us instead of
//     354 (524288 bins, 3 sigma). One for each number of terms, a whole strip in registers, is slower where it
//     counts, on short spectra, whose launch first has to fetch it: 11.4 us at 4099 bins, 8.4 us this way.
template <int TMAX, int KMAX>
__device__ __noinline__ void hs_strip_slow(HsUnit<KMAX> &unit, const HsRow r, int T, int lo, int hi) {
    const int lane = threadIdx.x & 31;
    const float inf = __int_as_float(0x7f800000);
    float v[TMAX], best[TMAX];
    int bestj[TMAX];
#pragma unroll
    for (int l = 0; l < TMAX; ++l) {
        best[l] = -1.0f;
        bestj[l] = 0;
    }
    auto sums = [&](int j) {  // of column j in v; -inf, above nothing, where the column or the plane is not there
#pragma unroll
        for (int l = 1; l <= TMAX; ++l)
            v[l - 1] = j < hi && l <= T ? __ldg(r.center + (long long)l * r.step + (size_t)l * (unsigned)j) : -inf;
#pragma unroll
        for (int l = 1; l < TMAX; ++l) v[l] = __fadd_rn(v[l - 1], v[l]);
    };
    unsigned crossed = 0u;  // bit b: columns lo + 32 b .. have crossings
    int mine = 0;           // lane l - 1: crossings of plane l
#pragma unroll 1
    for (int b = 0; lo + 32 * b < hi; ++b) {
        const int j = lo + 32 * b + lane;
        sums(j);
        bool any = false;
#pragma unroll
        for (int l = 0; l < TMAX; ++l) {
            any |= l < T && v[l] > unit.ta[l];
            if (v[l] > best[l]) {
                best[l] = v[l];
                bestj[l] = j;
            }
        }
        if (!__any_sync(0xFFFFFFFFu, any)) continue;
        crossed |= 1u << b;
#pragma unroll
        for (int l = 0; l < TMAX; ++l) {
            const int n = __popc(__ballot_sync(0xFFFFFFFFu, l < T && v[l] > unit.ta[l]));
            if (lane == l) mine += n;
        }
    }
    if (crossed != 0u) {
        unsigned long long base = 0ull;
        if (mine > 0) base = atomicAdd(&unit.counters[lane], (unsigned long long)mine);
        unsigned slot = base < FDAS_RAW_CAP ? (unsigned)base : FDAS_RAW_CAP;  // lane l - 1: the next slot of plane l
        if (__any_sync(0xFFFFFFFFu, mine > 0 && slot < FDAS_RAW_CAP)) {
            for (; crossed != 0u; crossed &= crossed - 1u) {
                const int j = lo + 32 * (__ffs(crossed) - 1) + lane;
                sums(j);
#pragma unroll
                for (int l = 0; l < TMAX; ++l) {
                    const bool hit = l < T && v[l] > unit.ta[l];
                    const unsigned m = __ballot_sync(0xFFFFFFFFu, hit);
                    if (m == 0u) continue;
                    const unsigned at = __shfl_sync(0xFFFFFFFFu, slot, l) + __popc(m & ((1u << lane) - 1u));
                    if (hit && at < FDAS_RAW_CAP) unit.raw[(size_t)l * FDAS_RAW_CAP + at] = cand_key(v[l], unit.row, (unsigned)j);
                    if (lane == l) slot += __popc(m);
                }
            }
        }
    }
    bool beats = false;
#pragma unroll
    for (int l = 0; l < TMAX; ++l) beats |= l < T && best[l] > *(volatile float *)&unit.peak_limit[l];
    if (__any_sync(0xFFFFFFFFu, beats)) {
        unsigned long long key = 0ull;  // lane l - 1: the strip's peak key of plane l
#pragma unroll
        for (int l = 0; l < TMAX; ++l) {
            const unsigned long long k = warp_peak_key(best[l], bestj[l], unit.row);
            key = lane == l ? k : key;
        }
        // +inf: a plane that is not reported here, or whose peak no power beats.
        if (lane < T && unit.peak_limit[lane] < inf) hs_raise(unit, lane, key);
    }
    __syncwarp();
}

// The same for one term: the strip's 16 columns per thread at once (a sum of one plane of 65536 bins takes 14 us, 25 us
// with the loop above).
template <int KMAX>
__device__ __noinline__ void hs_strip_slow_1(HsUnit<KMAX> &unit, const HsRow r, int lo, int hi) {
    constexpr int J = hs_j(1);
    const int lane = threadIdx.x & 31;
    const float ta = unit.ta[0];
    const float *const p = r.center + r.step + lo + lane;
    float v[J], best = -1.0f;
    int bestj = 0, n = 0;
#pragma unroll
    for (int u = 0; u < J; ++u) v[u] = lo + lane + 32 * u < hi ? __ldg(p + 32 * u) : -__int_as_float(0x7f800000);
#pragma unroll
    for (int u = 0; u < J; ++u) {
        n += __popc(__ballot_sync(0xFFFFFFFFu, v[u] > ta));
        if (v[u] > best) {
            best = v[u];
            bestj = lo + lane + 32 * u;
        }
    }
    if (n != 0) {
        unsigned long long base = 0ull;
        if (lane == 0) base = atomicAdd(&unit.counters[0], (unsigned long long)n);
        base = __shfl_sync(0xFFFFFFFFu, base, 0);
        if (base < FDAS_RAW_CAP) {
            unsigned slot = (unsigned)base;
#pragma unroll
            for (int u = 0; u < J; ++u) {
                const unsigned m = __ballot_sync(0xFFFFFFFFu, v[u] > ta);
                const unsigned at = slot + __popc(m & ((1u << lane) - 1u));
                if (v[u] > ta && at < FDAS_RAW_CAP) unit.raw[at] = cand_key(v[u], unit.row, (unsigned)(lo + lane + 32 * u));
                slot += __popc(m);
            }
        }
    }
    if (__any_sync(0xFFFFFFFFu, best > *(volatile float *)&unit.peak_limit[0])) {
        const unsigned long long key = warp_peak_key(best, bestj, unit.row);
        hs_raise(unit, lane, lane == 0 ? key : 0ull);
    }
    __syncwarp();
}

// Columns [lo, hi) of the row, which all have T terms. `first` is the warp that takes the range's first
// strip, then the one for the next range: the short ranges of a small spectrum go to different warps.
template <int T, int KMAX>
__device__ __forceinline__ void hs_range(HsUnit<KMAX> &unit, const HsRow &r, int lo, int hi, bool vec, int &first) {
    constexpr int J = hs_j(T), W = 32 * J;
    const int lane = threadIdx.x & 31, warp = ((threadIdx.x >> 5) - first) & (kSumWarps - 1);
    // T = 1 (a row's own values only): strips on 16-byte boundaries, four 16-byte loads per thread. The up
    // to 3 columns before lo are compared as well, which can only send a strip to the second look.
    for (int s = (T == 1 ? lo & ~3 : lo) + warp * W; s < hi; s += kSumWarps * W) {
        float lim[T];
#pragma unroll
        for (int l = 0; l < T; ++l) lim[l] = *(volatile float *)&unit.either[l];
        bool hit = false, done = false;
        if constexpr (T == 1) {
            if (vec && s + W <= hi) {
                const float4 *p = reinterpret_cast<const float4 *>(r.center + r.step + s) + lane;
                float4 q[J / 4];
#pragma unroll
                for (int g = 0; g < J / 4; ++g) q[g] = __ldg(p + 32 * g);
#pragma unroll
                for (int g = 0; g < J / 4; ++g)
                    hit |= q[g].x > lim[0] || q[g].y > lim[0] || q[g].z > lim[0] || q[g].w > lim[0];
                done = true;
            }
        }
        if (!done) {
            const float *p[T];
#pragma unroll
            for (int l = 1; l <= T; ++l) p[l - 1] = r.center + (long long)l * r.step + (size_t)l * (unsigned)(s + lane);
            float v[J][T];
            if (s + W <= hi) {
#pragma unroll
                for (int l = 1; l <= T; ++l)
#pragma unroll
                    for (int u = 0; u < J; ++u) v[u][l - 1] = __ldg(p[l - 1] + 32 * l * u);
            } else {
#pragma unroll
                for (int l = 1; l <= T; ++l)
#pragma unroll
                    for (int u = 0; u < J; ++u)  // -inf: never above a limit
                        v[u][l - 1] = s + lane + 32 * u < hi ? __ldg(p[l - 1] + 32 * l * u) : -__int_as_float(0x7f800000);
            }
#pragma unroll
            for (int u = 0; u < J; ++u) {
                float hp = v[u][0];
                hit |= hp > lim[0];
#pragma unroll
                for (int l = 2; l <= T; ++l) {
                    hp = __fadd_rn(hp, v[u][l - 1]);
                    hit |= hp > lim[l - 1];
                }
            }
        }
        if (__any_sync(0xFFFFFFFFu, hit)) {
            if constexpr (T == 1)
                hs_strip_slow_1(unit, r, max(s, lo), min(s + W, hi));
            else
                hs_strip_slow<(T <= 2 ? 2 : T <= 4 ? 4 : T <= 8 ? 8 : KMAX)>(unit, r, T, max(s, lo), min(s + W, hi));
        }
    }
    first += (hi - lo + W - 1) / W;
}

// Unit u of a plane with rows -A..A and nb column blocks per row: row offset i and column block k. The
// first nb units are row 0's; then unit 2 h + sign, h counting the blocks of the rows 1..A slab by slab.
// Before slab s lie C(s) = sum_a min(a s, nb) blocks. The warp searches s 32 ways at a time, then
// finds the row in the slab by a prefix sum over a.
__device__ __forceinline__ void hs_locate(int u, int nb, int A, int &i, int &k) {
    if (u < nb) {
        i = 0;
        k = u;
        return;
    }
    const int lane = threadIdx.x & 31;
    u -= nb;
    int h = u >> 1;
    auto before = [&](int s) {  // C(s), s >= 1; the float quotient's floor is exact for nb < 2^20
        const int r = min(A, (int)__fdividef((float)nb + 0.5f, (float)s));
        return s * ((r * (r + 1)) >> 1) + (A - r) * nb;
    };
    int s = 0;
    for (int len = nb; len > 1;) {  // s <= slab < s + len
        const int step = (len + 31) >> 5;
        const int t = s + (lane + 1) * step;
        const unsigned m = __ballot_sync(0xFFFFFFFFu, t <= nb && before(t) <= h);
        s += __popc(m) * step;
        len = step;
    }
    h -= s > 0 ? before(s) : 0;
    for (int a0 = 0; a0 < A; a0 += 32) {
        const int a = a0 + lane + 1;
        const int cnt = a <= A ? max(0, min(a * (s + 1), nb) - a * s) : 0;
        int sum = cnt;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int o = __shfl_up_sync(0xFFFFFFFFu, sum, d);
            if (lane >= d) sum += o;
        }
        const unsigned m = __ballot_sync(0xFFFFFFFFu, sum > h);
        if (m) {
            const int f = __ffs(m) - 1;
            const int first = __shfl_sync(0xFFFFFFFFu, sum - cnt, f);
            i = a0 + f + 1;
            k = i * s + (h - first);
            i = (u & 1) ? -i : i;
            return;
        }
        h -= __shfl_sync(0xFFFFFFFFu, sum, 31);
    }
    i = 0;  // not reached: u is below the number of units
    k = 0;
}

template <int KMAX, int T>
__device__ __forceinline__ void hs_dispatch(HsUnit<KMAX> &unit, const HsRow &r, int t, int lo, int hi, bool vec, int &first) {
    if constexpr (T <= KMAX) {
        if (t == T)
            hs_range<T, KMAX>(unit, r, lo, hi, vec, first);
        else
            hs_dispatch<KMAX, T + 1>(unit, r, t, lo, hi, vec, first);
    }
}

// The planes of a launch. job_of(u): which plane unit u belongs to; job(b): that plane.
struct HsPlane {
    const float *plane;
    size_t ld;
    int n;
    int jend;   // fundamental columns [0, jend) are summed
    int unit0;  // its first unit
    unsigned long long *counters, *peaks, *raw;
};
struct HsSingle {
    HsPlane p;
    int units, cols;
    __device__ __forceinline__ int job_of(int) const { return 0; }
    __device__ __forceinline__ const HsPlane &job(int) const { return p; }
};
struct HsMany {
    HsBatch b;
    int units, cols;
    __device__ __forceinline__ int job_of(int u) const {
        int lo = 0, hi = b.count - 1;  // the last job whose first unit is <= u
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (b.job[mid].unit0 <= u) lo = mid; else hi = mid - 1;
        }
        return lo;
    }
    __device__ __forceinline__ HsPlane job(int k) const {
        const HsJob &J = b.job[k];
        return HsPlane{J.plane, (size_t)J.ld, J.n, J.jend, J.unit0, J.counters, J.peaks, J.raw};
    }
};

// One CTA per unit; warp 0 works out what the unit is, once for all warps.
template <int KMAX, class Jobs>
__global__ void __launch_bounds__(kSumThreads, KMAX <= 8 ? 6 : 4)
    fdas_hs_sum(const __grid_constant__ Jobs jobs, int A, const float *__restrict__ thresh, int n_temp, unsigned mask,
                int n_harm, int first_plane) {
    __shared__ HsUnit<KMAX> unit;
    __shared__ int s_unit[5];  // plane, row offset, first column, terms of the first and of the last column
    const int c = (n_temp - 1) / 2, cols = jobs.cols;
    if (threadIdx.x < 32) {
        const int b = jobs.job_of(blockIdx.x);
        const HsPlane P = jobs.job(b);
        int i, k;
        hs_locate(blockIdx.x - P.unit0, (P.jend + cols - 1) / cols, A, i, k);
        const int ai = i < 0 ? -i : i, j0 = k * cols, j1 = min(j0 + cols, P.jend);
        const int klast = ai == 0 ? n_harm : min(n_harm, c / ai);
        const int t = threadIdx.x;
        pdl_wait();
        if (t < klast) {
            const float inf = __int_as_float(0x7f800000);
            float ta = inf, peak = inf;
            if (t + 1 >= first_plane) {
                const unsigned long long cur = *(volatile unsigned long long *)&P.peaks[t];
                if ((mask >> t) & 1u) ta = __ldg(&thresh[(size_t)t * n_temp + c + i]);
                peak = hs_limit(cur, ((unsigned)(c + i) << 24) | (unsigned)j0);
            }
            unit.ta[t] = ta;
            unit.peak_limit[t] = peak;
            unit.either[t] = fminf(ta, peak);
        }
        if (t == 0) {
            unit.raw = P.raw;
            unit.counters = P.counters;
            unit.peaks = P.peaks;
            unit.row = c + i;
            unit.loc = ((unsigned)(c + i) << 24) | (unsigned)j0;
            s_unit[0] = b;
            s_unit[1] = i;
            s_unit[2] = j0;
            s_unit[3] = j0 == 0 ? klast : min(klast, (P.n - 1) / j0);
            s_unit[4] = j1 <= 1 ? klast : min(klast, (P.n - 1) / (j1 - 1));
        }
    } else {
        pdl_wait();
    }
    __syncthreads();
    const HsPlane P = jobs.job(s_unit[0]);
    const int i = s_unit[1], j0 = s_unit[2], tmax = s_unit[3], tmin = s_unit[4];
    const int j1 = min(j0 + cols, P.jend);
    const HsRow r{P.plane + (size_t)c * P.ld, (long long)i * (long long)P.ld};
    const bool vec = (P.ld & 3) == 0 && (reinterpret_cast<uintptr_t>(P.plane) & 15) == 0;
    int first = 0, lo = j0;
    for (int t = tmax; t >= tmin; --t) {  // T(j) = t on [lo, hi)
        const int hi = t == tmin ? j1 : (P.n - 1) / t + 1;
        if (lo < hi) hs_dispatch<KMAX, 1>(unit, r, t, lo, hi, vec, first);
        lo = hi;
    }
}

template <class Jobs>
cudaError_t launch_hs_sum(const Jobs &jobs, int rows, const fdas_params &p, const float *thresh, bool hp1_done,
                          cudaStream_t s, bool chained) {
    if (jobs.units == 0) return cudaSuccess;
    return launch_pdl(chained, p.n_harm <= 8 ? fdas_hs_sum<8, Jobs> : fdas_hs_sum<16, Jobs>,
                      dim3((unsigned)jobs.units), kSumThreads, 0, s, jobs, rows, thresh, p.n_temp, p.harm_mask, p.n_harm,
                      hp1_done ? 2 : 1);
}

__device__ __forceinline__ fdas_cand decode_cand(unsigned long long key, int c, int k) {
    fdas_cand r;
    r.power = __uint_as_float(0xFFFFFFFFu - (unsigned)(key >> 32));
    r.i = (int16_t)((int)((key >> 24) & 0xFFu) - c);
    r.j = (unsigned)(key & 0xFFFFFFu);
    r.k = (uint8_t)k;
    r.pad = 0;
    return r;
}

// One bitonic step of stride S < E between a thread's own keys (index base + e).
template <int E, int S>
__device__ __forceinline__ void fin_reg_step(unsigned long long (&r)[E], int base, int size) {
#pragma unroll
    for (int e = 0; e < E; ++e) {
        if ((e & S) != 0) continue;
        const bool up = ((base + e) & size) == 0;
        const unsigned long long a = r[e], b = r[e + S];
        const bool sw = (a > b) == up;
        r[e] = sw ? b : a;
        r[e + S] = sw ? a : b;
    }
}

// Ascending bitonic sort of the nr keys at src, padded with ~0 to np2 = 32 E 2^m >= nr, with E keys
// per thread: thread t holds keys [E t, E t + E) in registers. Strides below E are exchanges inside
// a thread, strides E..16 E warp shuffles, and only strides >= 32 E go through shared memory.
// The first nout keys are decoded to candidates of plane k.
template <int E>
__device__ __forceinline__ void fin_sort(const unsigned long long *__restrict__ src, int nr, int np2, int nout, int c,
                                         int k, int cand_cap, fdas_cand *cands, unsigned long long *keys) {
    const int nthr = np2 / E;  // active threads, whole warps
    const bool active = (int)threadIdx.x < nthr;
    const int base = (int)threadIdx.x * E;
    const int lane = threadIdx.x & 31;
    unsigned long long r[E];
    if (active) {
#pragma unroll
        for (int e = 0; e < E; ++e) r[e] = base + e < nr ? src[base + e] : ~0ull;
    }
    for (int size = 2; size <= np2; size <<= 1) {
        if ((size >> 1) >= 32 * E) {
            if (active) {
#pragma unroll
                for (int e = 0; e < E; ++e) keys[base + e] = r[e];
            }
            __syncthreads();
            for (int stride = size >> 1; stride >= 32 * E; stride >>= 1) {
                for (int x = threadIdx.x; x < (np2 >> 1); x += blockDim.x) {
                    const int lo = 2 * x - (x & (stride - 1));
                    const int hi = lo + stride;
                    const bool up = (lo & size) == 0;
                    const unsigned long long a = keys[lo], b = keys[hi];
                    if ((a > b) == up) {
                        keys[lo] = b;
                        keys[hi] = a;
                    }
                }
                __syncthreads();
            }
            if (active) {
#pragma unroll
                for (int e = 0; e < E; ++e) r[e] = keys[base + e];
            }
            __syncthreads();  // every read done before the next writes
        }
        if (active) {
            for (int stride = min(size >> 1, 16 * E); stride >= E; stride >>= 1) {
                const int lx = stride / E;            // partner lane distance
                const bool lower = (lane & lx) == 0;  // this thread holds the lower index of each pair
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const unsigned long long o = __shfl_xor_sync(0xFFFFFFFFu, r[e], lx);
                    const bool up = ((base + e) & size) == 0;
                    r[e] = (lower == up) ? (r[e] < o ? r[e] : o) : (r[e] > o ? r[e] : o);
                }
            }
            if (E > 8 && size >= 16) fin_reg_step<E, (E > 8 ? 8 : 0)>(r, base, size);
            if (E > 4 && size >= 8) fin_reg_step<E, (E > 4 ? 4 : 0)>(r, base, size);
            if (E > 2 && size >= 4) fin_reg_step<E, (E > 2 ? 2 : 0)>(r, base, size);
            fin_reg_step<E, 1>(r, base, size);
        }
    }
    if (active) {
#pragma unroll
        for (int e = 0; e < E; ++e)
            if (base + e < nout) cands[(size_t)(k - 1) * cand_cap + base + e] = decode_cand(r[e], c, k);
    }
}

// Counts, peak and the top cand_cap candidates of plane k, from its workspace.
__device__ __forceinline__ void finalize_plane(int k, const unsigned long long *__restrict__ raw,
                                               const unsigned long long *counters, const unsigned long long *peaks,
                                               int n_temp, int cand_cap, fdas_cand *cands, uint32_t *counts,
                                               fdas_cand *peak_out, unsigned long long *keys) {
    const int c = (n_temp - 1) / 2;
    const unsigned long long total = counters[k - 1];
    const int nr = (int)(total < FDAS_RAW_CAP ? total : FDAS_RAW_CAP);
    if (threadIdx.x == 0) {
        counts[k - 1] = (uint32_t)(total < 0xFFFFFFFFull ? total : 0xFFFFFFFFull);
        if (peak_out) {
            const unsigned long long pk = peaks[k - 1];
            fdas_cand r;
            r.power = __uint_as_float((unsigned)(pk >> 32));
            const unsigned loc = 0xFFFFFFFFu - (unsigned)(pk & 0xFFFFFFFFull);
            r.i = (int16_t)((int)(loc >> 24) - c);
            r.j = loc & 0xFFFFFFu;
            r.k = (uint8_t)k;
            r.pad = 0;
            peak_out[k - 1] = r;
        }
    }
    if (nr == 0) return;
    const int nout = nr < cand_cap ? nr : cand_cap;
    const unsigned long long *src = raw + (size_t)(k - 1) * FDAS_RAW_CAP;
    // Keys per thread: 2 up to 2048 keys, 4 up to 4096, 16 up to FDAS_RAW_CAP (1024 threads).
    int np2 = 64;
    while (np2 < nr) np2 <<= 1;
    if (np2 <= 2048)
        fin_sort<2>(src, nr, np2, nout, c, k, cand_cap, cands, keys);
    else if (np2 <= 4096)
        fin_sort<4>(src, nr, np2, nout, c, k, cand_cap, cands, keys);
    else
        fin_sort<16>(src, nr, np2, nout, c, k, cand_cap, cands, keys);
}

__global__ void __launch_bounds__(kFinThreads)
    fdas_hs_finalize(const unsigned long long *__restrict__ raw, const unsigned long long *counters,
                     const unsigned long long *peaks, int n_temp, int cand_cap, fdas_cand *cands, uint32_t *counts,
                     fdas_cand *peak_out) {
    extern __shared__ unsigned long long keys[];
    pdl_wait();
    finalize_plane(blockIdx.x + 1, raw, counters, peaks, n_temp, cand_cap, cands, counts, peak_out, keys);
}

// ---- batched forms: one launch per stage for every spectrum of a batch ----------------------------

__global__ void fdas_hs_reset_batch(const HsBatch B, int n_harm) {
    pdl_trigger();
    const HsJob &J = B.job[blockIdx.x];
    const int t = threadIdx.x;
    if (t < n_harm) {
        J.counters[t] = 0ull;
        J.peaks[t] = 0ull;
    }
}

__global__ void __launch_bounds__(kFinThreads) fdas_hs_finalize_batch(const HsBatch B, int n_temp, int cand_cap) {
    extern __shared__ unsigned long long keys[];
    pdl_wait();
    const HsJob &J = B.job[blockIdx.y];
    finalize_plane(blockIdx.x + 1, J.raw, J.counters, J.peaks, n_temp, cand_cap, J.cands, J.counts, J.peak_out, keys);
}

}  // namespace

cudaError_t launch_hs_reset(const fdas_params &p, const HsWorkspace &ws, cudaStream_t s, bool chained) {
    return launch_pdl(chained, fdas_hs_reset, dim3(1), 32, 0, s, ws.counters, ws.peaks, p.n_harm);
}

cudaError_t launch_harmonic(const fdas_params &p, const float *plane, size_t n, size_t ld, const float *thresh,
                            fdas_cand *cands, uint32_t *counts, fdas_cand *peaks, const HsWorkspace &ws,
                            cudaStream_t s, bool hp1_done, bool chained) {
    // hp1_done: the workspace was reset before the convolution, which also took HP_1.
    bool follows = chained || !hp1_done;  // whether finalize comes behind a kernel of this call
    cudaError_t e = cudaSuccess;
    if (!hp1_done) {
        e = launch_hs_reset(p, ws, s, chained);
        if (e != cudaSuccess) return e;
    }
    int sms = 0;
    e = sm_count(&sms);
    if (e != cudaSuccess) return e;
    if (p.harm_index == FDAS_INDEX_HIGHEST) {
        e = launch_hs_highest(p, plane, n, ld, thresh, ws, sms, s);
    } else {
        HsSingle one;
        const int rows = hs_rows(p, hp1_done);
        one.p = HsPlane{plane, ld, (int)n, hs_end(p, n, hp1_done), 0, ws.counters, ws.peaks, ws.raw};
        one.cols = hs_columns(rows, one.p.jend, hp1_done, sms);
        one.units = (2 * rows + 1) * ((one.p.jend + one.cols - 1) / one.cols);
        e = launch_hs_sum(one, rows, p, thresh, hp1_done, s, follows);
        follows = follows || one.units > 0;
    }
    if (e != cudaSuccess) return e;
    const int smem = FDAS_RAW_CAP * (int)sizeof(unsigned long long);
    e = cudaFuncSetAttribute(fdas_hs_finalize, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    return launch_pdl(follows, fdas_hs_finalize, dim3((unsigned)p.n_harm), kFinThreads, smem, s, ws.raw, ws.counters, ws.peaks,
                      p.n_temp, p.cand_cap, cands, counts, peaks);
}

int harmonic_columns(const fdas_params &p, const size_t *lengths, int count, bool hp1_done, int sms) {
    long long total = 0;
    for (int b = 0; b < count; ++b) total += hs_end(p, lengths[b], hp1_done);
    return hs_columns(hs_rows(p, hp1_done), total, hp1_done, sms);
}

int harmonic_units(const fdas_params &p, size_t n, int cols, bool hp1_done, int *jend) {
    *jend = hs_end(p, n, hp1_done);
    return (2 * hs_rows(p, hp1_done) + 1) * ((*jend + cols - 1) / cols);
}

cudaError_t prepare_harmonic_batch() {
    return cudaFuncSetAttribute(fdas_hs_finalize_batch, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                FDAS_RAW_CAP * (int)sizeof(unsigned long long));
}

cudaError_t launch_hs_reset_batch(const fdas_params &p, const HsBatch &B, cudaStream_t s) {
    fdas_hs_reset_batch<<<B.count, 32, 0, s>>>(B, p.n_harm);
    return cudaGetLastError();
}

cudaError_t launch_harmonic_batch(const fdas_params &p, const HsBatch &B, const float *thresh, cudaStream_t s,
                                  bool hp1_done) {
    cudaError_t e = cudaSuccess;
    if (!hp1_done) {
        e = launch_hs_reset_batch(p, B, s);
        if (e != cudaSuccess) return e;
    }
    e = launch_hs_sum(HsMany{B, B.units, B.cols}, hs_rows(p, hp1_done), p, thresh, hp1_done, s, true);
    if (e != cudaSuccess) return e;
    return launch_pdl(true, fdas_hs_finalize_batch, dim3((unsigned)p.n_harm, (unsigned)B.count), kFinThreads,
                      FDAS_RAW_CAP * sizeof(unsigned long long), s, B, p.n_temp, p.cand_cap);
}

}  // namespace fdas
