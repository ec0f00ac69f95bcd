// FT convolution with the tensor cores: precisions FDAS_BF16X3 and FDAS_FP16S.
//
// The overlap-save steps are those of the FP32 kernel (Sec. 2.1): segment s of F = 2048 input
// points is transformed once (FP32 FFT in registers), multiplied by each template T_t, transformed
// back, and |u|^2 of the L = F - n_tap + 1 valid outputs is stored. The inverse transform, 85 per
// segment, is factored in four steps with F = 32 x 64, m = m1 + 32 m2 and n = 64 n1 + n2:
//
//   D1[n2; t, m1] = sum_m2 e^{2 pi i m2 n2 / 64} U_t[m1 + 32 m2]   (tensor cores, two thirds of the work)
//   V [n2; t, m1] = e^{2 pi i m1 n2 / 2048} D1[n2; t, m1]           (CUDA cores, FP32)
//   u_t[64 n1 + n2] = sum_m1 e^{2 pi i m1 n1 / 32} V[n2; t, m1]     (CUDA cores, FP32, in registers)
//
// The first step is a dense GEMM on the fifth-generation tensor cores (tcgen05.mma, FP32
// accumulation in Tensor Memory), in real form: [re; im] = [[c, -s], [s, c]] [re; im], so it is a
// real GEMM with M = 128 (n2, re/im), K = 128 (m2, re/im), N = 32 m1 per template. The tensor cores
// take 16-bit operands, so each operand x is split into x = hi + lo with hi = round16(x),
// lo = round16(x - hi), and a product A B is accumulated as A_lo B_hi + A_hi B_lo + A_hi B_hi (the
// A_lo B_lo term is below FP32 rounding of the result). With BF16 halves (FDAS_BF16X3) this keeps
// about 16 significant bits per operand; with FP16 halves (FDAS_FP16S) about 22 bits, but FP16's
// range needs scaling: the product U = W * T_t is scaled by 2^k per segment, chosen from the
// largest component of W so that |U| < 2^14.5 (|T_t| is at most sqrt(n_tap) <= 32 because the taps
// have unit energy); the 64-term sums D1 are FP32 and the twiddles carry a factor 2^-6 that the
// power rescaling 2^(12 - 2k) undoes.
//
// One persistent CTA per SM runs three independent worker groups of 4 warps; each group owns a
// stream of work items (a segment with a range of templates), its own shared-memory operand and two
// TMEM accumulators, and is served by its own MMA-issue warp:
//   prep  (group)       forward FFT of the segment (W kept in shared memory); per pair of templates
//                       U = W * T_t (templates read from L2), split, stored as the GEMM's B operand
//                       (rows: 2 templates x 32 m1, K: 64 m2 x re/im);
//   MMA   (warp 12 + g) one thread issues 24 MMAs per pair (M = 128, N = 64, K = 128; A = the
//                       real-form 64-point DFT matrix, both halves, resident in Tensor Memory);
//   mid   (group)       D1 from TMEM (a thread gets both components of its n2 and template from two loads
//                       of 16 lanes), the twiddle product, a 32-point DFT in registers (radix 4 x 8),
//                       |u|^2 of the kept outputs, coalesced stores.
// A group finishes pair p - 1 (mid) while the GEMM of pair p runs, which is why there are two
// accumulators: a group that waits for its own GEMM between prep and mid leaves the CUDA cores idle
// (2^21 bins, BF16X3: 655 us; 526 us in this order). Reading both components from TMEM instead of
// exchanging them between lanes took it to 509 us, packed sums in the DFT to 488 us, equal shares of the
// work to 428 us. What bounds it now is issue: 5.7 K warp instructions per pair and group (with HP_1), issued
// at 63% of the rate; the waits left
// are for templates from L2 and for TMEM. (Copying the first template of the next pair to shared memory
// by TMA: 498 us, with spills.)
// Every wait is bounded: a wait that gives up sets the device
// status word and an abort flag, after which no role issues work or waits again; before freeing its
// TMEM the CTA waits once more, bounded, for whatever it had issued.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "hs_keys.cuh"
#include "ols_common.cuh"
#include "tc_ops.cuh"

namespace fdas {
namespace {

constexpr int kGroups = 3;                            // worker groups of 4 warps
constexpr int kMmaWarp0 = 4 * kGroups;                // MMA-issue warps 12, 13, 14
constexpr int kTcThreads = (4 * kGroups + kGroups) * 32;
constexpr uint32_t kTmemCols = 512;
// Tensor Memory columns: the DFT matrix (hi, lo), then two D1 buffers per group.
constexpr uint32_t kColAhi = 0, kColAlo = 64, kColD1 = 128;

// Shared memory (bytes), per group: region X (the forward FFT's exchange buffers, then the GEMM's
// B operand, hi and lo) and W; then the twiddle table, barriers and small state.
constexpr int kB1Term = 64 * 128 * 2;                 // rows (t_local, m1) x K (m2, re/im), 16-bit
constexpr int kXBytes = 2 * kPadded * 8;
constexpr int kGroupBytes = kXBytes + kF * 8;         // region X + W
constexpr int kTwRow = 32 * 8 + 16;                   // 32 twiddles per n2 row, padded by 16 bytes
constexpr int kOffTw = kGroups * kGroupBytes;
constexpr int kOffBar = kOffTw + 64 * kTwRow;
constexpr int kNumBars = 2 * kGroups + 1;
constexpr int kOffMisc = kOffBar + kNumBars * 8;
constexpr int kTcSmemBytes = kOffMisc + 16 + 16 * kGroups + 64 * kGroups;
static_assert(2 * kB1Term <= kXBytes, "the operand fits in the FFT's region");
static_assert(kGroupBytes % 1024 == 0 && kOffTw % 16 == 0 && kOffBar % 8 == 0, "alignment");
static_assert(kTcSmemBytes <= 227 * 1024, "shared memory per CTA");

// Byte offset of element (row, k) in a K-major operand without swizzle: 8 x 8 core matrices of
// 128 bytes, K-adjacent core matrices 128 bytes apart, row groups `sbo` bytes apart.
__host__ __device__ constexpr int kmajor_off(int row, int k, int sbo) {
    return (row >> 3) * sbo + (k >> 3) * 128 + (row & 7) * 16 + (k & 7) * 2;
}

template <bool HALF>
__device__ __forceinline__ void split2(float a, float b, uint32_t &hi, uint32_t &lo) {
    if (HALF) {
        const __half2 h = __floats2half2_rn(a, b);
        const float2 hf = __half22float2(h);
        const __half2 l = __floats2half2_rn(a - hf.x, b - hf.y);
        hi = *reinterpret_cast<const uint32_t *>(&h);
        lo = *reinterpret_cast<const uint32_t *>(&l);
    } else {
        const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
        const float2 hf = __bfloat1622float2(h);
        const __nv_bfloat162 l = __floats2bfloat162_rn(a - hf.x, b - hf.y);
        hi = *reinterpret_cast<const uint32_t *>(&h);
        lo = *reinterpret_cast<const uint32_t *>(&l);
    }
}

// Bounded mbarrier wait that also gives up at once when the CTA has already aborted.
__device__ __forceinline__ bool tc_wait(unsigned long long *bar, unsigned parity, volatile int *aborted) {
    if (*aborted) return false;
    if (mbar_wait(bar, parity)) return true;
    *aborted = 1;
    return false;
}
__device__ __forceinline__ void mbar_arrive(unsigned long long *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_init_n(unsigned long long *bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

// v * e^{2 pi i k / 32} for k known at compile time after unrolling.
__device__ __forceinline__ float2 w32(float2 v, int k) {
    constexpr float C[9] = {1.f, 0.98078528040323043f, 0.92387953251128674f, 0.83146961230254524f,
                            0.70710678118654752f, 0.55557023301960218f, 0.38268343236508977f,
                            0.19509032201612825f, 0.f};  // cos(2 pi j / 32), j = 0..8
    k &= 31;
    if (k == 0) return v;
    if (k == 8) return make_float2(-v.y, v.x);
    if (k == 16) return make_float2(-v.x, -v.y);
    if (k == 24) return make_float2(v.y, -v.x);
    const float c = k <= 8 ? C[k] : k <= 16 ? -C[16 - k] : k <= 24 ? -C[k - 16] : C[32 - k];
    const float sn = k <= 8 ? C[8 - k] : k <= 16 ? C[k - 8] : k <= 24 ? -C[24 - k] : -C[k - 24];
    return make_float2(fmaf(v.x, c, -v.y * sn), fmaf(v.x, sn, v.y * c));
}

// In-place inverse 32-point DFT, natural order: u[n] = sum_m v[m] e^{2 pi i m n / 32}. Radix 4 x 8:
// m = a + 8 b, n = 4 c + d: 4-point DFTs over b, twiddles e^{2 pi i a d / 32}, 8-point DFTs over a.
// Packed sums: 488 us at 2^21 bins, 509 us with scalar ones (while the groups still waited for their
// GEMMs the packed form was slightly slower).
__device__ __forceinline__ void idft32(float2 (&v)[32]) {
#pragma unroll
    for (int a = 0; a < 8; ++a) dft4<true>(v[a], v[a + 8], v[a + 16], v[a + 24]);
#pragma unroll
    for (int a = 1; a < 8; ++a)
#pragma unroll
        for (int d = 1; d < 4; ++d) v[a + 8 * d] = w32(v[a + 8 * d], a * d);
    float2 u[32];
#pragma unroll
    for (int d = 0; d < 4; ++d) {
        float2 x[8];
#pragma unroll
        for (int a = 0; a < 8; ++a) x[a] = v[a + 8 * d];
        dft8<true>(x);
#pragma unroll
        for (int c = 0; c < 8; ++c) u[4 * c + d] = x[c];
    }
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = u[i];
}

// Barrier indices: per group g, B1 full (4 warp arrivals) and D1 full (MMA commit).
__device__ __forceinline__ int bar_b1full(int g) { return 2 * g; }
__device__ __forceinline__ int bar_d1full(int g) { return 2 * g + 1; }
constexpr int kBarFin = 2 * kGroups;

// Named barrier of group g's four warps (ids 1..kGroups).
__device__ __forceinline__ void group_sync(int g) { asm volatile("bar.sync %0, 128;\n" ::"r"(g + 1) : "memory"); }

// HP_1 (see the FP32 form), taken here too: the harmonic sum then takes 103 us at 2^21 bins instead of 149 us, for 3 to
// 10 us in the convolution (BF16X3 search 592 -> 550 us). The rare paths are out of line. A thread's outputs are
// the columns col + 64 n1 of its row, kept where bit n1 of omask is set; every lane of the warp comes along.
// The outputs above ta go by way of the stack, with one counter update and so one latency for all. Read again from
// L2 in four steps, counted column by column, and with rows in the plain order, an FP16s search of 200003 bins
// with tones took 103 us, 88 us this way (99 us with HP_1 in the harmonic sum).
__device__ __noinline__ void tc_hp1_emit(const float *pw, float ta, int row, int col, unsigned omask, Hp1 hp1) {
    unsigned hits = 0u;
#pragma unroll 8
    for (int n1 = 0; n1 < 32; ++n1) hits |= (unsigned)(pw[n1] > ta) << n1;
    hits &= omask;
    unsigned long long slot = emit_slots(__popc(hits), threadIdx.x & 31, hp1.counters);
    for (; hits != 0u; hits &= hits - 1u, ++slot) {
        const int n1 = __ffs(hits) - 1;
        if (slot < FDAS_RAW_CAP) hp1.raw[slot] = cand_key(pw[n1], row, (unsigned)(col + 64 * n1));
    }
    __syncwarp();
}
// Place (row << 24 | column) of the first output equal to best.
__device__ __noinline__ unsigned tc_hp1_best_loc(const float *rowp, float best, int row, int col, unsigned omask) {
    unsigned loc = 0xFFFFFFFFu;
#pragma unroll 1
    for (int b = 0; b < 32; b += 16) {
        float v[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) v[q] = ((omask >> (b + q)) & 1u) ? __ldcg(rowp + 64 * (b + q)) : -1.0f;
#pragma unroll
        for (int q = 0; q < 16; ++q)
            if (v[q] == best) loc = min(loc, ((unsigned)row << 24) | (unsigned)(col + 64 * (b + q)));
    }
    return loc;
}

template <bool HALF, bool HP1, class Jobs>
__global__ void __launch_bounds__(kTcThreads, 1)
    fdas_ols_tc(Jobs jobs, const float2 *__restrict__ tmpl, int n_temp, int h, int keep, Hp1 hp1) {
    extern __shared__ __align__(1024) unsigned char smem[];
    unsigned char *const twt = smem + kOffTw;
    unsigned long long *const bars = reinterpret_cast<unsigned long long *>(smem + kOffBar);
    uint32_t *const tslot = reinterpret_cast<uint32_t *>(smem + kOffMisc);
    volatile int *const aborted = reinterpret_cast<volatile int *>(smem + kOffMisc + 4);

    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    const float2 *wtab = tmpl + (size_t)n_temp * kF;  // exp(-2 pi i k / F)

    if (tid == 0) {
        for (int g = 0; g < kGroups; ++g) {
            mbar_init_n(&bars[bar_b1full(g)], 4);
            mbar_init_n(&bars[bar_d1full(g)], 1);
        }
        mbar_init_n(&bars[kBarFin], 1);
        *aborted = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (w == 0) tc::tmem_alloc(tslot, kTmemCols);

    // Mid-stage twiddles e^{2 pi i m1 n2 / 2048} (times 2^-6 for FP16), row n2, column m1.
    for (int i = tid; i < 64 * 32; i += kTcThreads) {
        const int n2 = i >> 5, m1 = i & 31;
        const float2 e0 = __ldg(&wtab[m1 * n2]);
        const float s2 = HALF ? 0.015625f : 1.f;
        *reinterpret_cast<float2 *>(twt + n2 * kTwRow + m1 * 8) = make_float2(e0.x * s2, -e0.y * s2);
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tm = *tslot;
    const uint32_t lane_base = (uint32_t)(32 * (w & 3)) << 16;

    // The GEMM's A operand into TMEM (warps 0-3, one lane each): lane l is output row (n2, c) with
    // n2 = 16 (l >> 5) + (l & 15), c = (l >> 4) & 1; K index k = 32 wq + 2 q + c' is input
    // (m2 = wq + 4 q, c').
    if (w < 4) {
        const int n2 = 16 * w + (lane & 15), c = lane >> 4;
#pragma unroll 1
        for (int j0 = 0; j0 < 64; j0 += 16) {
            uint32_t hw[16], lw[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                float v2[2];
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    const int k = 2 * (j0 + j) + b;
                    const int m2 = (k >> 5) + 4 * ((k & 31) >> 1), cp = k & 1;
                    const float2 e0 = __ldg(&wtab[32 * ((m2 * n2) & 63)]);
                    const float er = e0.x, ei = -e0.y;  // e^{+2 pi i m2 n2 / 64}
                    v2[b] = c == 0 ? (cp == 0 ? er : -ei) : (cp == 0 ? ei : er);
                }
                split2<HALF>(v2[0], v2[1], hw[j], lw[j]);
            }
            tc::tmem_st16(tm + kColAhi + lane_base + j0, hw);
            tc::tmem_st16(tm + kColAlo + lane_base + j0, lw);
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();

    if (HP1) pdl_wait();  // the workspace has been reset
    if (w < kMmaWarp0) {
        // ------------------------------------------------------------------ worker group g
        const int g = w >> 2, gt = tid & 127;  // group and thread index within the group
        unsigned char *const region = smem + g * kGroupBytes;  // FFT buffers, then B1 (hi, lo)
        float2 *const Ws = reinterpret_cast<float2 *>(region + kXBytes);
        float2 *buf0 = reinterpret_cast<float2 *>(region);
        float2 *buf1 = buf0 + kPadded;
        unsigned *const red = reinterpret_cast<unsigned *>(smem + kOffMisc + 16 + 16 * g);  // [4]
        const uint32_t d1 = tm + kColD1 + 128 * g + lane_base;
        // Mid role: TMEM lanes 32 (w & 3) + 0..15 hold the real rows of 16 n2, the next 16 lanes the
        // imaginary rows. Threads 0..15 take template 0 of the pair, threads 16..31 template 1, and
        // each reads both components of its own.
        const int n2 = 16 * (w & 3) + (lane & 15);
        const int tlm = lane >> 4;
        const unsigned char *trow = twt + n2 * kTwRow;
        const float inv_f = 1.0f / kF;
        const int x = worker(jobs.deal, blockIdx.x, gridDim.x, g, kGroups);
        int p = 0;  // pair counter of this group
        for (int q_seg = -1, t0, t1 = 0; deal_next(jobs.deal, x, gridDim.x * kGroups, q_seg, t0, t1);) {
            const Item it = jobs.get(q_seg);
            const int n = it.n;
            const int origin = it.s * keep - h;
            const int col0 = it.s * keep - h;
            // Forward FFT of the segment: W[q] = DFT(w_s)[gt + 128 q] / F, kept in shared memory
            // (each thread reads back only what it wrote). Region X is free: this group's last
            // GEMM has completed (its D1 was read).
            float pscale = 1.f;
            {
                float2 v[16];
                {
                    float2 tw2[16];
                    const int k = gt & 15;
#pragma unroll
                    for (int q = 0; q < 16; ++q) tw2[q] = __ldg(&wtab[8 * ((k * q) & 255)]);
#pragma unroll
                    for (int q = 0; q < 16; ++q) {
                        const int idx = origin + gt + 128 * q;
                        v[q] = (idx >= 0 && idx < n) ? __ldg(&it.spec[idx]) : make_float2(0.f, 0.f);
                    }
                    fft_passes_12<false>(v, buf0, buf1, tw2, gt, [] {}, [g] { group_sync(g); });
                }
#pragma unroll
                for (int hh = 0; hh < 2; ++hh) {
                    float2 tw3[8];
#pragma unroll
                    for (int q = 0; q < 8; ++q) tw3[q] = __ldg(&wtab[(gt + 128 * hh) * q]);
                    float2 u[8];
                    fft_pass_3<false>(u, buf1, tw3, gt + 128 * hh);
#pragma unroll
                    for (int q = 0; q < 8; ++q) v[2 * q + hh] = make_float2(u[q].x * inv_f, u[q].y * inv_f);
                }
                if (HALF) {
                    float mx = 0.f;
#pragma unroll
                    for (int q = 0; q < 16; ++q) mx = fmaxf(mx, fmaxf(fabsf(v[q].x), fabsf(v[q].y)));
                    const unsigned mb = __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(mx));
                    if (lane == 0) red[w & 3] = mb;
                    group_sync(g);
                    const unsigned mall = max(max(red[0], red[1]), max(red[2], red[3]));
                    // 2^k with k = 8 - exponent(max component), so that |U| 2^k < 2^14.5.
                    int k = mall ? 8 - ((int)((mall >> 23) & 0xFF) - 127) : 0;
                    k = max(-40, min(40, k));
                    const float s1 = __uint_as_float((unsigned)(k + 127) << 23);
#pragma unroll
                    for (int q = 0; q < 16; ++q) v[q] = make_float2(v[q].x * s1, v[q].y * s1);
                    pscale = __uint_as_float((unsigned)(12 - 2 * k + 127) << 23);
                }
#pragma unroll
                for (int q = 0; q < 16; ++q) Ws[gt + 128 * q] = v[q];
            }
            group_sync(g);  // every thread of the group is done with the FFT buffers (and red[])
            uint32_t omask = 0u;  // outputs n = 64 n1 + n2 kept (h <= n < h + keep) and inside the spectrum
#pragma unroll
            for (int n1 = 0; n1 < 32; ++n1) {
                const int m = 64 * n1 + n2;
                if (m >= h && m < h + keep && col0 + m < n) omask |= 1u << n1;
            }

            // With HP1, shares number the pairs of rows in a scattered order, as the FP32 form its rows. The last
            // pair of an odd n_temp, or of an odd chunk, is one row.
            const bool scattered = HP1 && jobs.deal.per_seg > 0;
            const int row_end = scattered ? n_temp : t1;
            const int units = (n_temp + 1) >> 1;
            int r0 = scattered ? 2 * (int)((unsigned)((t0 >> 1) * jobs.deal.stride) % (unsigned)units) : t0;
            int r_prev = r0;  // first rows of this pair and the one before
            float best = -1.0f;  // HP1: this thread's largest output of the item, its row
            int best_t = -1;
            // mid: both rows of the pair (r, r + 1) whose sums are in D1 buffer `buf`.
            auto mid = [&](int r, int buf) {
                float2 v[32];
#pragma unroll
                for (int hh = 0; hh < 2; ++hh) {
                    uint32_t re[16], im[16];  // of this lane's template
                    const uint32_t d = d1 + 64 * buf + 16 * hh;
                    tc::tmem_ld16_halves<32>(d, re, d + (16u << 16), im);
#pragma unroll
                    for (int i = 0; i < 16; i += 2) {
                        const int m1 = 16 * hh + i;
                        const float4 tw = *reinterpret_cast<const float4 *>(trow + 8 * m1);
                        v[m1] = cmul(make_float2(__uint_as_float(re[i]), __uint_as_float(im[i])), make_float2(tw.x, tw.y));
                        v[m1 + 1] = cmul(make_float2(__uint_as_float(re[i + 1]), __uint_as_float(im[i + 1])),
                                         make_float2(tw.z, tw.w));
                    }
                }
                idft32(v);  // v[n1] = u[64 n1 + n2]
                const int row = r + tlm;
                const bool have = row < row_end;
                float mx = -1.0f;  // HP1: largest kept output of this row
                float *const dst = it.plane + (size_t)row * it.ld + col0 + n2;
                if (have) {
#pragma unroll
                    for (int n1 = 0; n1 < 32; ++n1) {
                        const float pw = HALF ? fmaf(v[n1].x, v[n1].x, v[n1].y * v[n1].y) * pscale
                                              : fmaf(v[n1].x, v[n1].x, v[n1].y * v[n1].y);
                        if ((omask >> n1) & 1u) {
                            dst[64 * n1] = pw;
                            if (HP1) mx = fmaxf(mx, pw);
                        }
                        if (HP1) v[n1].x = pw;
                    }
                }
                if (HP1) {
                    const float ta = have && hp1.ta ? __ldg(&hp1.ta[row]) : __int_as_float(0x7f800000);
                    if (__any_sync(0xFFFFFFFFu, mx > ta)) {  // rare
                        float pw[32];
#pragma unroll
                        for (int n1 = 0; n1 < 32; ++n1) pw[n1] = v[n1].x;
                        tc_hp1_emit(pw, ta, row, col0 + n2, have ? omask : 0u, jobs.hp1(hp1, it.job));
                    }
                    if (mx > best || (mx == best && row < best_t)) {  // the first row wins ties
                        best = mx;
                        best_t = row;
                    }
                }
            };
            for (int t = t0; t < t1; t += 2, ++p) {
                if (t > t0) {  // the GEMM of the pair before has read the operand, and its sums are there
                    tc_wait(&bars[bar_d1full(g)], (p - 1) & 1, aborted);
                    tc::fence_after_sync();
                }
                // prep: U = W T_t; B1 row 32 tl + lane, K chunk 4 (w & 3) + i holds q = 4 i .. 4 i + 3.
                const int tb = min(2, row_end - r0);
                for (int tl = 0; tl < tb; ++tl) {
                    const float2 *T = tmpl + (size_t)(r0 + tl) * kF + gt;
                    float2 tv[16];
#pragma unroll
                    for (int q = 0; q < 16; ++q) tv[q] = __ldg(&T[128 * q]);
                    uint32_t hw[16], lw[16];
#pragma unroll
                    for (int q = 0; q < 16; ++q) {
                        const float2 u = cmul(Ws[gt + 128 * q], tv[q]);
                        split2<HALF>(u.x, u.y, hw[q], lw[q]);
                    }
                    unsigned char *row = region + kmajor_off(32 * tl + lane, 32 * (w & 3), 2048);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        *reinterpret_cast<uint4 *>(row + 128 * i) =
                            make_uint4(hw[4 * i], hw[4 * i + 1], hw[4 * i + 2], hw[4 * i + 3]);
                        *reinterpret_cast<uint4 *>(row + kB1Term + 128 * i) =
                            make_uint4(lw[4 * i], lw[4 * i + 1], lw[4 * i + 2], lw[4 * i + 3]);
                    }
                }
                tc::fence_before_sync();  // this warp's reads of this D1 buffer (two pairs ago) are done
                tc::fence_proxy_async();
                __syncwarp();
                if (lane == 0) mbar_arrive(&bars[bar_b1full(g)]);
                if (t > t0) mid(r_prev, (p - 1) & 1);  // while the GEMM of this pair runs
                r_prev = r0;
                r0 += scattered ? 2 * jobs.deal.stride : 2;
                if (scattered && r0 >= 2 * units) r0 -= 2 * units;
            }
            tc_wait(&bars[bar_d1full(g)], (p - 1) & 1, aborted);
            tc::fence_after_sync();
            mid(r_prev, (p - 1) & 1);
            if (HP1) {  // the item's HP_1 peak, as in the FP32 form
                const Hp1 h1 = jobs.hp1(hp1, it.job);
                const unsigned wmax = __reduce_max_sync(0xFFFFFFFFu, best >= 0.0f ? __float_as_uint(best) : 0u);
                const unsigned cur = (unsigned)(*(volatile unsigned long long *)&h1.peaks[0] >> 32);
                if (wmax >= cur) {  // warp-uniform
                    const unsigned loc = best_t >= 0 ? tc_hp1_best_loc(it.plane + (size_t)best_t * it.ld + col0 + n2,
                                                                       best, best_t, col0 + n2, omask)
                                                     : 0xFFFFFFFFu;
                    const unsigned long long key = warp_peak_key_loc(best, loc);
                    if (lane == 0 && key != 0ull) atomicMax(&h1.peaks[0], key);
                }
            }
        }
    } else {
        // ------------------------------------------------------------------ MMA issue for group g
        const int g = w - kMmaWarp0;
        if (lane == 0) {
            constexpr uint32_t id1 = tc::idesc_f16(128, 64, !HALF);
            const uint32_t bs = smem_u32(smem + g * kGroupBytes);
            const uint32_t d1g = tm + kColD1 + 128 * g;
            const int x = worker(jobs.deal, blockIdx.x, gridDim.x, g, kGroups);
            int p = 0;
            for (int q_seg = -1, t0, t1 = 0; deal_next(jobs.deal, x, gridDim.x * kGroups, q_seg, t0, t1);) {
                for (int t = t0; t < t1; t += 2, ++p) {
                    tc_wait(&bars[bar_b1full(g)], p & 1, aborted);
                    if (*aborted) continue;
                    tc::fence_after_sync();
                    const uint32_t d1 = d1g + 64 * (p & 1);
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk) {
                        const uint64_t bh = tc::desc_kmajor(bs + 256 * kk, 128, 2048);
                        const uint64_t bl = tc::desc_kmajor(bs + kB1Term + 256 * kk, 128, 2048);
                        tc::mma_ts(d1, tm + kColAlo + 8 * kk, bh, id1, kk > 0);
                        tc::mma_ts(d1, tm + kColAhi + 8 * kk, bl, id1, 1u);
                        tc::mma_ts(d1, tm + kColAhi + 8 * kk, bh, id1, 1u);
                    }
                    tc::commit(reinterpret_cast<uint64_t *>(&bars[bar_d1full(g)]));
                }
            }
        }
        __syncwarp();
    }

    // Teardown: nothing of this CTA may be in flight when its TMEM is freed. Without an abort
    // every MMA was waited for; after one, wait (bounded) for the MMAs each issuer issued.
    tc::fence_before_sync();
    __syncthreads();
    if (*aborted) {
        for (int g = 0; g < kGroups; ++g) {
            if (tid == (kMmaWarp0 + g) * 32) tc::commit(reinterpret_cast<uint64_t *>(&bars[kBarFin]));
            mbar_wait(&bars[kBarFin], (unsigned)(g & 1));
            __syncthreads();
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (w == 0) tc::tmem_dealloc(tm, kTmemCols);
}

template <bool HALF, bool HP1, class Jobs>
cudaError_t set_smem() {
    return cudaFuncSetAttribute(fdas_ols_tc<HALF, HP1, Jobs>, cudaFuncAttributeMaxDynamicSharedMemorySize, kTcSmemBytes);
}

// With HP1 the launch follows the workspace's reset of this call.
template <bool HALF, bool HP1, class Jobs>
cudaError_t launch(const Geometry &g, const Jobs &jobs, int workers, int sms, const float2 *tmpl, const Hp1 &hp1,
                   cudaStream_t s) {
    const dim3 grid((unsigned)(workers < sms ? workers : sms));
    return launch_pdl(HP1, fdas_ols_tc<HALF, HP1, Jobs>, grid, kTcThreads, (size_t)kTcSmemBytes, s, jobs, tmpl, g.n_temp, g.h,
                      g.keep, hp1);
}

}  // namespace

cudaError_t launch_convolve_tc(const Geometry &g, const float2 *spec, size_t n, const float2 *tmpl, float *plane,
                               size_t ld, int ctas_per_sm, int templates_per_item, cudaStream_t s, const float *thresh,
                               unsigned harm_mask, const HsWorkspace *ws) {
    (void)ctas_per_sm;  // one CTA per SM
    int sms = 0, workers = 0;
    cudaError_t e = sm_count(&sms);
    if (e != cudaSuccess) return e;
    const SingleJobs jobs{spec, plane, ld, (int)n,
                          make_deal(g, segment_count(g, n), templates_per_item, sms, kGroups, &workers)};
    const bool half = g.precision == FDAS_FP16S;
    e = ws ? (half ? set_smem<true, true, SingleJobs>() : set_smem<false, true, SingleJobs>())
           : (half ? set_smem<true, false, SingleJobs>() : set_smem<false, false, SingleJobs>());
    if (e != cudaSuccess) return e;
    if (!ws)
        return half ? launch<true, false>(g, jobs, workers, sms, tmpl, Hp1{}, s)
                    : launch<false, false>(g, jobs, workers, sms, tmpl, Hp1{}, s);
    const Hp1 hp1{(harm_mask & 1u) ? thresh : nullptr, ws->raw, ws->counters, ws->peaks};
    return half ? launch<true, true>(g, jobs, workers, sms, tmpl, hp1, s)
                : launch<false, true>(g, jobs, workers, sms, tmpl, hp1, s);
}

cudaError_t prepare_convolve_batch_tc() {
    const cudaError_t e = set_smem<true, true, BatchJobs>();
    return e != cudaSuccess ? e : set_smem<false, true, BatchJobs>();
}

cudaError_t launch_convolve_batch_tc(const Geometry &g, const ConvBatch &batch, const float2 *tmpl,
                                     int templates_per_item, int sms, const float *thresh, unsigned harm_mask,
                                     cudaStream_t s) {
    int workers = 0;
    const BatchJobs jobs{batch, make_deal(g, batch.total_segments, templates_per_item, sms, kGroups, &workers)};
    // The workspace pointers come from each item.
    const Hp1 hp1{(harm_mask & 1u) ? thresh : nullptr, nullptr, nullptr, nullptr};
    return g.precision == FDAS_FP16S ? launch<true, true>(g, jobs, workers, sms, tmpl, hp1, s)
                                     : launch<false, true>(g, jobs, workers, sms, tmpl, hp1, s);
}

cudaError_t device_status_tc(unsigned *flags, bool clear) {
    cudaError_t e = cudaMemcpyFromSymbol(flags, g_device_status, sizeof(unsigned));
    if (e == cudaSuccess && clear) {
        const unsigned zero = 0u;
        e = cudaMemcpyToSymbol(g_device_status, &zero, sizeof(unsigned));
    }
    return e;
}

cudaError_t device_status_tc_async(unsigned *h_flags, cudaStream_t s) {
    return cudaMemcpyFromSymbolAsync(h_flags, g_device_status, sizeof(unsigned), 0, cudaMemcpyDeviceToHost, s);
}

}  // namespace fdas
