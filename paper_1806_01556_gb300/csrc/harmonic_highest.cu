// The harmonic sum indexed by the highest harmonic (FDAS_INDEX_HIGHEST).
//
// HP_k(i, j) = sum_{l=1..k} of P[c + rd(l i, k)][rd(l j, k)], float32 running sums in the order
// l = 1..k, rd = round half away from zero, on the whole plane. A term depends on l/k only as a rational
// number, so the terms of all planes k <= K come from the reduced fractions q = a/b, b <= K (22 for K = 8,
// 80 for K = 16): term (l, k) of fundamental (i, j) is P[c + rd(a i, b)][rd(a j, b)] with a/b = l/k in
// lowest terms.
//
// A tile is one row i with W consecutive columns. For each fraction the source columns of row c + rd(a i, b)
// that the tile needs, about W a/b of them, are copied into a shared-memory segment of their own; the
// planes are then summed from the segments. Consecutive threads take consecutive columns, so they read
// the same or consecutive words of a segment (rd(a j, b) moves by a/b <= 1 per column) and the reads
// have no bank conflicts.
//
// A CTA walks through some of the rows of one column block. Where a term of column j lies in its segment does
// not depend on the row, and nor does where each 16 bytes of a segment come from within their row, so both
// are worked out once per CTA. Two buffers: while one row is summed, the next one's segments arrive by
// cp.async. (TMA bulk copies, one per fraction, are too short here, 0.1 to 3 KB: about 20 ns each, 655 us
// and 1359 us for the two sizes below.) As in fdas_hs_sum, the hot path compares each sum with one limit
// per plane (hs_limit); a warp that exceeds one sums again, emits the crossings and raises the peaks.
//
// Measured, 85 rows, this kernel alone: 8 planes at 2^20 bins 1251 -> 574 us (983 -> 392 M warp
// instructions), 16 planes at 262147 bins 1922 -> 671 us (1351 -> 364 M), against one division per
// fraction, thread and tile, blocking copies and a best point tracked per thread and plane. No unit is
// saturated: the load-store pipe, which the 22 (80) shared reads per point and the copies of 11.5 (40.5) floats per
// point go through, is 74% (60%) busy, issue 56% (44%), and 5.3 (6.2) GB come from L2 at 9.2 TB/s (fdas_hs_sum
// reads from L2 at 14 TB/s).
#include <type_traits>

#include "hs_keys.cuh"
#include "hs_rules.h"

namespace fdas {
namespace {

__host__ __device__ constexpr int gcd_c(int x, int y) {
    while (y != 0) {
        const int t = x % y;
        x = y;
        y = t;
    }
    return x;
}
// The reduced fractions a/b (1 <= a <= b <= 16), ordered by b, then a; first[b]: the first with denominator b.
constexpr int kMaxFrac = 80;
struct Farey {
    int a[kMaxFrac], b[kMaxFrac], first[18];
    constexpr Farey() : a{}, b{}, first{} {
        int q = 0;
        for (int d = 1; d <= 16; ++d) {
            first[d] = q;
            for (int x = 1; x <= d; ++x)
                if (gcd_c(x, d) == 1) {
                    a[q] = x;
                    b[q] = d;
                    ++q;
                }
        }
        first[17] = q;
    }
    constexpr int index(int l, int k) const {  // of l/k in lowest terms
        const int g = gcd_c(l, k);
        int q = first[k / g];
        while (a[q] != l / g) ++q;
        return q;
    }
};
constexpr Farey kFarey;
static_assert(kFarey.first[9] == 22 && kFarey.first[17] == kMaxFrac, "Farey counts");

// round(x / b) for x >= 0, b > 0, halves up (away from zero).
__host__ __device__ __forceinline__ constexpr int rd_pos(int x, int b) { return (2 * x + b) / (2 * b); }
// round(a / b) for b > 0, halves away from zero, exactly in integers.
__device__ __forceinline__ int round_div(int a, int b) {
    const int m = rd_pos(a < 0 ? -a : a, b);
    return a < 0 ? -m : m;
}

// Shapes for up to KMAX planes: W columns per tile, thread t < active takes columns j0 + t + active v.
template <int KMAX>
struct Shape;
template <>
struct Shape<8> {  // active = lcm(1..7): the places of columns t and t + 420 differ by the constant 420 a/b, b <= 7
    static constexpr int threads = 448, active = 420, V = 2, W = active * V, NQ = 22;
};
template <>
struct Shape<16> {
    static constexpr int threads = 256, active = 240, V = 1, W = active * V, NQ = 80;
};

// Segment offsets in floats, segments on 16-byte boundaries. A segment starts up to 3 columns early (on a
// 16-byte boundary of the row), and its copy ends on one.
template <int KMAX>
struct Segments {
    static constexpr int NQ = Shape<KMAX>::NQ;
    int a[NQ], b[NQ], off[NQ + 1];
    constexpr Segments() : a{}, b{}, off{} {
        int o = 0;
        for (int q = 0; q < NQ; ++q) {
            a[q] = kFarey.a[q];
            b[q] = kFarey.b[q];
            off[q] = o;
            o += ((a[q] * Shape<KMAX>::W + b[q] - 1) / b[q] + 8 + 3) & ~3;
        }
        off[NQ] = o;
    }
};
template <int KMAX>
constexpr Segments<KMAX> kSeg{};
__constant__ Segments<8> c_seg8;
__constant__ Segments<16> c_seg16;
template <int KMAX>
__device__ __forceinline__ const Segments<KMAX> &segments() {
    if constexpr (KMAX == 8)
        return c_seg8;
    else
        return c_seg16;
}
template <int KMAX>
constexpr int kBufFloats = kSeg<KMAX>.off[Shape<KMAX>::NQ];
// Per CTA: two buffers and, for each 16 bytes of a buffer, where they come from (fraction, byte of its row).
template <int KMAX>
constexpr int kSmemBytes = 2 * kBufFloats<KMAX> * 4 + kBufFloats<KMAX> / 4 * 8;
static_assert(2 * kSmemBytes<8> <= 220 * 1024 && 2 * kSmemBytes<16> <= 220 * 1024, "two CTAs per SM");
// What lies below the first buffer: the kilobyte that the system keeps, and the kernel's own arrays (lim, top, src_row,
// base), each rounded up to 16 bytes at most.
template <int KMAX>
constexpr int kBelowBytes = 1024 + kMaxRows * KMAX * (int)sizeof(float) + KMAX * (int)sizeof(unsigned long long) +
                            kMaxRows * Shape<KMAX>::NQ + 2 * Shape<KMAX>::NQ * (int)sizeof(float *) + 4 * 16;
static_assert(kBelowBytes<16> + kBufFloats<16> * 4 <= 65536, "shared addresses in the first buffer fit in 16 bits");

// f(std::integral_constant<int, k>) for k = K..KMAX: loop bodies whose index must be a
// compile-time constant whatever the size of the body.
template <int K, int KMAX, class F>
__device__ __forceinline__ void for_each_k(F &&f) {
    if constexpr (K <= KMAX) {
        f(std::integral_constant<int, K>{});
        for_each_k<K + 1, KMAX>(f);
    }
}

// Shared-memory addresses of a thread's terms in the first buffer (`add` reaches the second). Up to 8
// planes: one word per fraction with b <= 7 (column v adds the constant 420 a v / b), one per column for
// b = 8. Up to 16: two addresses per word.
template <int ADD>
__device__ __forceinline__ float lds(unsigned addr) {
    float x;
    asm volatile("ld.shared.f32 %0, [%1 + %2];" : "=f"(x) : "r"(addr), "n"(ADD));
    return x;
}
template <int KMAX>
struct Places;
template <>
struct Places<8> {
    unsigned r[18 + 4 * Shape<8>::V];
    __device__ __forceinline__ void set(unsigned buf, int j0, int t, int n_harm) {
        for_each_k<0, 21>([&](auto qc) {
            constexpr int q = decltype(qc)::value, a = kFarey.a[q], b = kFarey.b[q], off = kSeg<8>.off[q];
            if (b > n_harm) return;  // uniform
            const int base = off - (rd_pos(a * j0, b) & ~3);
            if constexpr (b <= 7) {
                r[q] = buf + 4u * (unsigned)(base + (int)((unsigned)(2 * a * (j0 + t) + b) / (unsigned)(2 * b)));
            } else {
#pragma unroll
                for (int v = 0; v < Shape<8>::V; ++v)
                    r[18 + Shape<8>::V * (q - 18) + v] =
                        buf + 4u * (unsigned)(base + ((2 * a * (j0 + t + Shape<8>::active * v) + 8) >> 4));
            }
        });
    }
    template <int Q, int V, int ADD>
    __device__ __forceinline__ float at() const {
        constexpr int a = kFarey.a[Q], b = kFarey.b[Q];
        if constexpr (b <= 7)
            return lds<ADD + 4 * (Shape<8>::active * a * V / b)>(r[Q]);
        else
            return lds<ADD>(r[18 + Shape<8>::V * (Q - 18) + V]);
    }
};
template <>
struct Places<16> {
    unsigned r[kMaxFrac / 2];
    __device__ __forceinline__ void set(unsigned buf, int j0, int t, int n_harm) {
        for_each_k<0, kMaxFrac - 1>([&](auto qc) {
            constexpr int q = decltype(qc)::value, a = kFarey.a[q], b = kFarey.b[q], off = kSeg<16>.off[q];
            unsigned byte = 0u;
            if (b <= n_harm)  // uniform
                byte = buf + 4u * (unsigned)(off - (rd_pos(a * j0, b) & ~3) +
                                       (int)((unsigned)(2 * a * (j0 + t) + b) / (unsigned)(2 * b)));
            r[q / 2] = (q & 1) ? (r[q / 2] | byte << 16) : byte;
        });
    }
    template <int Q, int V, int ADD>
    __device__ __forceinline__ float at() const {
        return lds<ADD>((Q & 1) ? r[Q / 2] >> 16 : r[Q / 2] & 0xFFFFu);
    }
};

// The running sum of terms 1..L of plane K. `term(l)` for compile-time l.
template <int L, class Term>
__device__ __forceinline__ float run_sum(const Term &term) {
    const float x = term(std::integral_constant<int, L>{});
    if constexpr (L == 1)
        return x;
    else
        return __fadd_rn(run_sum<L - 1>(term), x);
}

template <int KMAX, bool FULL>
__global__ void __launch_bounds__(Shape<KMAX>::threads, 2)
    fdas_hs_highest(const float *__restrict__ plane, int n, size_t ld, bool vec, const float *__restrict__ thresh,
                    int n_temp, unsigned mask, int n_harm, int nq, int rows_per, unsigned long long *__restrict__ raw,
                    unsigned long long *counters, unsigned long long *peaks) {
    using Sh = Shape<KMAX>;
    constexpr int kWarps = Sh::threads / 32;
    constexpr int kGroups = kBufFloats<KMAX> / 4;  // 16-byte groups per buffer
    constexpr unsigned kNone = 0xFFFFFFFFu;        // a group that no segment fills
    extern __shared__ float4 hh_buf[];
    uint2 *const from = reinterpret_cast<uint2 *>(hh_buf + 2 * kGroups);  // [kGroups]: byte of the row, fraction
    __shared__ float lim[kMaxRows][KMAX];                // hs_limit of each row and plane
    __shared__ unsigned long long top[KMAX];             // peak keys behind the limits
    __shared__ unsigned char src_row[kMaxRows][Sh::NQ];  // plane row that each fraction of a row reads
    __shared__ const float *base[2][Sh::NQ];             // its address, for the row after next (copy_row)
    const int c = (n_temp - 1) / 2;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int j0 = blockIdx.x * Sh::W;
    const int jl = min(j0 + Sh::W, n) - 1;
    // The last group's rows are the last ones; the other groups interleave.
    const int others = (int)gridDim.y - 1, y0 = (int)blockIdx.y;
    const int row0 = y0 < others ? y0 : others * rows_per, step = y0 < others ? others : 1;
    const int rows = y0 < others ? rows_per : n_temp - row0;
    auto row_of = [&](int x) { return row0 + x * step; };
    const Segments<KMAX> &seg = segments<KMAX>();

    auto threshold = [&](int row, int k) {
        return ((mask >> (k - 1)) & 1u) ? __ldg(&thresh[(size_t)(k - 1) * n_temp + row]) : __int_as_float(0x7f800000);
    };
    // Limit of plane k in a row, with `cur` as the plane's peak key.
    auto limit = [&](int row, int k, unsigned long long cur) {
        return fminf(threshold(row, k), hs_limit(cur, ((unsigned)row << 24) | (unsigned)j0));
    };
    // Raises plane lane + 1's peak, and its limits in the rows x.., if key (this lane's; 0: none) wins.
    auto raise = [&](int x, unsigned long long key) {
        if (key == 0ull) return;
        unsigned long long cur = *(volatile unsigned long long *)&peaks[lane];
        if (key > cur) {
            atomicMax(&peaks[lane], key);
            cur = key;
        }
        *(volatile unsigned long long *)&top[lane] = cur;
        for (int y = x; y < rows; ++y) *(volatile float *)&lim[y][lane] = limit(row_of(y), lane + 1, cur);
    };
    auto set_base = [&](int x, int buf) {
        if (threadIdx.x < nq) base[buf][threadIdx.x] = plane + (size_t)src_row[x][threadIdx.x] * ld;
    };
    // Starts the copies of the row whose addresses are in base[buf] into buffer buf (every thread).
    auto copy_row = [&](int buf) {
        const unsigned dst = (unsigned)__cvta_generic_to_shared(hh_buf + buf * kGroups + threadIdx.x);
        for_each_k<0, (kGroups - 1) / Sh::threads>([&](auto mc) {
            constexpr int m = decltype(mc)::value;
            if ((m + 1) * Sh::threads > kGroups && threadIdx.x + m * Sh::threads >= kGroups) return;
            const uint2 f = from[threadIdx.x + m * Sh::threads];
            if (f.y == kNone) return;
            asm volatile("cp.async.cg.shared.global [%0 + %2], [%1], 16;\n" ::"r"(dst),
                         "l"(reinterpret_cast<const char *>(base[buf][f.y]) + f.x), "n"(16 * Sh::threads * m));
        });
    };
    for (int e = threadIdx.x; e < kGroups; e += Sh::threads) from[e] = make_uint2(0u, kNone);
    for (int e = threadIdx.x; e < rows * Sh::NQ; e += Sh::threads) {
        const int q = e % Sh::NQ, x = e / Sh::NQ;
        src_row[x][q] = (unsigned char)(c + round_div(seg.a[q] * (row_of(x) - c), seg.b[q]));
    }
    __syncthreads();
    if (vec) {
        for (int q = warp; q < nq; q += kWarps) {
            const int x0 = rd_pos(seg.a[q] * j0, seg.b[q]) >> 2, x1 = rd_pos(seg.a[q] * jl, seg.b[q]) >> 2;
            for (int e = lane; e <= x1 - x0; e += 32)
                from[seg.off[q] / 4 + e] = make_uint2(16u * (unsigned)(x0 + e), (unsigned)q);  // ends by the row's end
        }
        set_base(0, 0);
        if (1 < rows) set_base(1, 1);
    }
    const bool act = threadIdx.x < Sh::active;
    const int t = act ? threadIdx.x : 0;  // the other threads read inside the segments
    Places<KMAX> at;
    at.set((unsigned)__cvta_generic_to_shared(hh_buf), j0, t, n_harm);
    pdl_wait();
    for (int e = threadIdx.x; e < rows * KMAX; e += Sh::threads) {
        const int k = e % KMAX + 1, x = e / KMAX;
        if (k > n_harm) continue;
        const unsigned long long cur = *(volatile unsigned long long *)&peaks[k - 1];
        lim[x][k - 1] = limit(row_of(x), k, cur);
        if (x == 0) top[k - 1] = cur;
    }
    __syncthreads();
    if (vec) copy_row(0);

    auto tile = [&](auto bc, int x) {
        constexpr int B = decltype(bc)::value;
        constexpr int add = B * kBufFloats<KMAX> * 4;
        const int row = row_of(x);
        if (vec) {
            asm volatile("cp.async.wait_all;\n" ::: "memory");
            __syncthreads();  // the row is there, and every read of buffer B ^ 1 is done
            if (x + 1 < rows) copy_row(B ^ 1);
            if (x + 2 < rows) set_base(x + 2, B);  // base[B] was used before the barrier
        } else {  // a row stride or base without 16-byte alignment: plain loads, nothing in flight
            __syncthreads();
            for (int q = warp; q < nq; q += kWarps) {
                const int x0 = rd_pos(seg.a[q] * j0, seg.b[q]) & ~3, x1 = rd_pos(seg.a[q] * jl, seg.b[q]);
                const float *src = plane + (size_t)src_row[x][q] * ld + x0;
                float *dst = reinterpret_cast<float *>(hh_buf) + B * kBufFloats<KMAX> + seg.off[q];
                for (int e = lane; e <= x1 - x0; e += 32) dst[e] = __ldg(src + e);
            }
            __syncthreads();
        }
        float lm[KMAX];
#pragma unroll
        for (int k = 0; k < KMAX; ++k) lm[k] = *(volatile float *)&lim[x][k];
        bool hit = false;
        for_each_k<0, Sh::V - 1>([&](auto vc) {
            constexpr int v = decltype(vc)::value;
            float keep[Sh::NQ];  // fractions that a later plane uses again
            bool over = false;
            for_each_k<1, KMAX>([&](auto kc) {
                constexpr int k = decltype(kc)::value;
                if (!FULL && k > n_harm) return;  // uniform
                const float hp = run_sum<k>([&](auto lc) {
                    constexpr int l = decltype(lc)::value, q = kFarey.index(l, k);
                    if constexpr (gcd_c(l, k) == 1) {
                        const float x = at.template at<q, v, add>();
                        if constexpr (2 * k <= KMAX) keep[q] = x;
                        return x;
                    } else {
                        return keep[q];
                    }
                });
                over |= hp > lm[k - 1];
            });
            hit |= over && act && j0 + t + Sh::active * v < n;
        });
        if (!__any_sync(0xFFFFFFFFu, hit)) return;
        // Rare: the same sums again. Lane k - 1 updates plane k's counter, all planes at once, a plane whose peak no sum
        // beats takes no reduction, and limits are worked out again only when a peak may have changed. In the other form (an
        // update for every plane and 32 columns in turn, every reduction, all limits each time) the sum of 524288 bins took
        // 4870 us at 2 sigma and 985 us of a spectrum that was not whitened, 1080 and 478 us in this one; 12 planes at
        // 100003 bins 1898 and 674 us at 2 sigma, 286 and 283 us without crossings. With exactly 16 planes this form costs
        // the hot loop registers: without crossings 671 -> 690 us at 262147 bins (at 2 sigma 3357 -> 1753).
        if constexpr (KMAX <= 8 || !FULL) {
            const float inf = __int_as_float(0x7f800000);
            const float ta = lane < n_harm ? threshold(row, lane + 1) : inf;
            const float peak = lane < n_harm ? hs_limit(top[lane], ((unsigned)row << 24) | (unsigned)j0) : inf;
            auto sums = [&](auto kc, float (&hp)[Sh::V]) {  // plane k's; -inf, above nothing, past the last column
                for_each_k<0, Sh::V - 1>([&](auto vc) {
                    constexpr int k = decltype(kc)::value, v = decltype(vc)::value;
                    const float sum = run_sum<k>([&](auto lc) {
                        return at.template at<kFarey.index(decltype(lc)::value, k), v, add>();
                    });
                    hp[v] = act && j0 + t + Sh::active * v < n ? sum : -inf;
                });
            };
            float kept[FULL ? KMAX : 1][Sh::V];  // with all planes the sums fit in registers
            int mine = 0;                        // lane k - 1: crossings of plane k
            unsigned long long key = 0ull;       // and the warp's peak key, if it may win
            for_each_k<1, KMAX>([&](auto kc) {
                constexpr int k = decltype(kc)::value;
                if (!FULL && k > n_harm) return;
                float(&hp)[Sh::V] = kept[FULL ? k - 1 : 0];
                float best = -1.0f;
                int bestj = 0, count = 0;
                sums(kc, hp);
                const float tk = __shfl_sync(0xFFFFFFFFu, ta, k - 1);
#pragma unroll
                for (int v = 0; v < Sh::V; ++v) {
                    count += __popc(__ballot_sync(0xFFFFFFFFu, hp[v] > tk));
                    if (hp[v] > best) {
                        best = hp[v];
                        bestj = j0 + t + Sh::active * v;
                    }
                }
                mine = lane == k - 1 ? count : mine;
                if (!__any_sync(0xFFFFFFFFu, best > __shfl_sync(0xFFFFFFFFu, peak, k - 1))) return;
                const unsigned long long mx = warp_peak_key(best, bestj, row);
                key = lane == k - 1 ? mx : key;
            });
            unsigned long long first = 0ull;
            if (mine > 0) first = atomicAdd(&counters[lane], (unsigned long long)mine);
            const unsigned emits = __ballot_sync(0xFFFFFFFFu, mine > 0 && first < FDAS_RAW_CAP);
            if (emits != 0u)
                for_each_k<1, KMAX>([&](auto kc) {
                    constexpr int k = decltype(kc)::value;
                    if (((emits >> (k - 1)) & 1u) == 0u) return;
                    float(&hp)[Sh::V] = kept[FULL ? k - 1 : 0];
                    if constexpr (!FULL) sums(kc, hp);
                    const float tk = __shfl_sync(0xFFFFFFFFu, ta, k - 1);
                    unsigned slot = (unsigned)__shfl_sync(0xFFFFFFFFu, first, k - 1);
#pragma unroll
                    for (int v = 0; v < Sh::V; ++v) {
                        const unsigned m = __ballot_sync(0xFFFFFFFFu, hp[v] > tk);
                        const unsigned to = slot + __popc(m & ((1u << lane) - 1u));
                        if (hp[v] > tk && to < FDAS_RAW_CAP)
                            raw[(size_t)(k - 1) * FDAS_RAW_CAP + to] = cand_key(hp[v], row, (unsigned)(j0 + t + Sh::active * v));
                        slot += __popc(m);
                    }
                });
            raise(x, key);
        } else {
            unsigned long long mine = 0ull;  // lane k - 1: the warp's peak key of plane k
            for_each_k<1, KMAX>([&](auto kc) {
                constexpr int k = decltype(kc)::value;
                if (!FULL && k > n_harm) return;
                const float ta = threshold(row, k);
                float best = -1.0f;
                int bestj = 0;
                for_each_k<0, Sh::V - 1>([&](auto vc) {
                    constexpr int v = decltype(vc)::value;
                    const int j = j0 + t + Sh::active * v;
                    const bool ok = act && j < n;
                    const float hp = run_sum<k>([&](auto lc) {
                        return at.template at<kFarey.index(decltype(lc)::value, k), v, add>();
                    });
                    emit(ok && hp > ta, hp, row, (unsigned)j, k, lane, counters, raw);
                    if (ok && hp > best) {
                        best = hp;
                        bestj = j;
                    }
                });
                const unsigned long long key = warp_peak_key(best, bestj, row);
                mine = lane == k - 1 ? key : mine;
            });
            if (lane < n_harm) {
                unsigned long long cur = *(volatile unsigned long long *)&peaks[lane];
                if (mine > cur) {
                    atomicMax(&peaks[lane], mine);
                    cur = mine;
                }
                for (int y = x; y < rows; ++y) *(volatile float *)&lim[y][lane] = limit(row_of(y), lane + 1, cur);
            }
        }
    };
    for (int x = 0; x < rows; x += 2) {
        tile(std::integral_constant<int, 0>{}, x);
        if (x + 1 < rows) tile(std::integral_constant<int, 1>{}, x + 1);
    }
}

template <int KMAX, bool FULL>
cudaError_t launch(const fdas_params &p, const float *plane, size_t n, size_t ld, const float *thresh,
                   const HsWorkspace &ws, int sms, cudaStream_t s) {
    constexpr int smem = kSmemBytes<KMAX>;
    const cudaError_t e =
        cudaFuncSetAttribute(fdas_hs_highest<KMAX, FULL>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    const bool vec = (ld & 3) == 0 && (reinterpret_cast<uintptr_t>(plane) & 15) == 0;
    const int blocks = (int)((n + Shape<KMAX>::W - 1) / Shape<KMAX>::W);
    const int rows_per = rows_per_cta(blocks, p.n_temp, sms);
    const dim3 grid((unsigned)blocks, (unsigned)((p.n_temp + rows_per - 1) / rows_per));
    return launch_pdl(true, fdas_hs_highest<KMAX, FULL>, grid, Shape<KMAX>::threads, (size_t)smem, s, plane, (int)n, ld, vec,
                      thresh, p.n_temp, p.harm_mask, p.n_harm, kFarey.first[p.n_harm + 1], rows_per, ws.raw,
                      ws.counters, ws.peaks);
}

}  // namespace

cudaError_t launch_hs_highest(const fdas_params &p, const float *plane, size_t n, size_t ld, const float *thresh,
                              const HsWorkspace &ws, int sms, cudaStream_t s) {
    if (p.n_harm == 8) return launch<8, true>(p, plane, n, ld, thresh, ws, sms, s);
    if (p.n_harm < 8) return launch<8, false>(p, plane, n, ld, thresh, ws, sms, s);
    if (p.n_harm == 16) return launch<16, true>(p, plane, n, ld, thresh, ws, sms, s);
    return launch<16, false>(p, plane, n, ld, thresh, ws, sms, s);
}

}  // namespace fdas
