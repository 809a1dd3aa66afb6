// gram_exact.cu -- the FP64 correlation matrix (Sec. 4, the matrix corr) on the
// 5th-generation tensor cores, from X itself: corr_ab = sum_t (x_ta - m_a)(x_tb - m_b) /
// (n sd_a sd_b), in exact integer arithmetic up to one truncation below FP64's rounding.
//
// GB300 runs FP64 at 2 FMA per clock and SM, BF16 products at about 2000 times that.  Each
// deviation is taken to fixed point, D = round(x 2^s) - round(m 2^s) as 64-bit integers, s
// such that |x - m| <= sqrt(n) sd < 2^(54-s) (every deviation obeys that bound, whatever
// the distribution), and cut into 8 balanced base-128 digits, D = sum_i d_i 128^(7-i),
// -64 <= d_i <= 63: small integers that BF16 holds exactly.  The digit products of equal
// weight w = i + j go to one FP32 accumulator; 512 samples times at most 8 digit pairs
// times 64^2 is 2^24, so every accumulator stays an exact integer (this is the splitting
// scheme of Ozaki, Ogita, Oishi and Rump, "Error-free transformations of matrix
// multiplication", 2012).  Weights 0 to 9 are kept: the dropped ones add up to sqrt(n)
// 2^-67 of the correlation scale where the low digits vary, n 2^-66 at worst (digits that
// are the same in every sample), and the fixed-point rounding of x to about 2^-54: below
// the rounding of an FP64 sum.  The subtracted mean is rounded to 2^-28 of the standard
// deviation, which changes a correlation by 2^-56 (the deviations sum to zero) and leaves
// the low digits of coarse data (FP32 columns with large means) zero.  The weights' integers are added with their shifts
// into one 64-bit integer in units of 2^46; by Cauchy-Schwarz |sum_t D_a D_b| <= 2^108, so
// it does not overflow, and the K splits meet by integer atomics in the output matrix
// itself: exact, hence the same in any order, and without a workspace.
//
// Measured (kernel time, FP32 input): p = 300, n = 8000 68 us where the FP64 pipe needs
// 580 us (and the one-CTA-per-64x64-tile FP64 kernel it replaces took about 9 ms);
// p = 95, n = 5000 16 us (FP64 split-K Gram and its reduce 81 us); p = 1000, n = 20000
// 1.00 ms (FP64: 16 ms).
#include "internal.h"
#include "tc_util.cuh"

#include <algorithm>

namespace fpc {

namespace {

constexpr int GE_M = 128, GE_N = 48;                 // tile: rows a, columns b
constexpr int GE_K = 32;                             // samples per stage
constexpr int GE_S = 8;                              // digits
constexpr int GE_W = 10;                             // weights kept
constexpr int GE_STAGES = 2;
constexpr int GE_A_BLK = GE_K * 128;                 // 64 columns (128 bytes) x GE_K samples
constexpr int GE_A = 2 * GE_A_BLK;                   // a digit of A
constexpr int GE_B = GE_S * GE_N / 64 * GE_A_BLK;    // all digits of B side by side: 384 columns
constexpr int GE_STAGE = GE_S * GE_A + GE_B;
constexpr int GE_CH = (GE_M + GE_N) / 8;             // groups of 8 columns: 16 of A, 6 of B
constexpr int GE_PROD = GE_K * GE_CH;                // producer threads: one group of one sample each
constexpr int GE_THREADS = GE_PROD + 32;
constexpr int GE_KMAX = 512;                         // samples per CTA: exactness of the accumulators
constexpr int GE_TMEM = 512;
constexpr int GE_COLS = GE_M + GE_N;
static_assert(GE_S * GE_N % 64 == 0 && GE_W * GE_N <= GE_TMEM, "B's digits fill whole blocks; accumulators");
static_assert(GE_PROD % 32 == 0 && (GE_K * GE_M / 8) % 32 == 0, "whole warps per operand");

// s of a column: |x - mean| <= sqrt(n) sd < 2^(54 - s).  A constant column (rsd 0) or one
// with a non-finite statistic has no digits (its correlations are 0 or NaN through rsd).
// From rsd's exponent and an FP32 quotient of sqrt(n) and its leading bits, rounded up (the
// same in an FP64 division took each CTA 2 us of the FP64 pipe).
__device__ __forceinline__ bool ge_scale(double rsd, long long n, int &s)
{
    s = 0;
    const int hi = __double2hiint(rsd), er = (hi >> 20) - 1023;          // rsd < 0 (never) or NaN: out of range
    if (er < -1020 || er > 1020) return false;
    const float m = __int_as_float(0x3f800000 | (hi & 0xfffff) << 3);    // in [1, 2), at most rsd 2^-er
    const float b = sqrtf((float)n) / m * 1.000002f;                     // above sqrt(n) / rsd 2^er, normal
    const int e = (__float_as_int(b) >> 23) - 126 - er;                  // sqrt(n) / rsd < 2^e
    if (e < -996 || e > 996) return false;
    s = 54 - e;
    return true;
}

// round(mant 2^sh) for mant < 2^53, modulo 2^64 (the difference of two of them, below 2^55,
// is exact modulo 2^64 however large the operands are)
__device__ __forceinline__ long long ge_shift(unsigned long long mant, int sh)
{
    if (sh >= 0) return sh < 64 ? (long long)(mant << sh) : 0;
    const int k = -sh;
    return k <= 60 ? (long long)((mant + (1ull << (k - 1))) >> k) : 0;
}
// the left shift of a 24-bit significand as a 32 x 32 product (the multiplier's pipe is idle
// here, the shifter's is not)
__device__ __forceinline__ long long ge_fixed(float x, int s)
{
    const uint32_t b = __float_as_uint(x);
    const int e = (int)((b >> 23) & 0xffu);
    const uint32_t m = (b & 0x7fffffu) | (e ? 0x800000u : 0u);
    const int sh = (e ? e : 1) - 150 + s;
    long long v;
    if (sh >= 0 && sh < 64) {
        const unsigned long long w = (unsigned long long)m * (1u << (sh & 31));
        v = (long long)(sh & 32 ? w << 32 : w);
    } else {
        v = ge_shift(m, sh);
    }
    return (int)b < 0 ? -v : v;
}
__device__ __forceinline__ long long ge_fixed(double x, int s)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int e = (int)((b >> 52) & 0x7ffu);
    const unsigned long long m = (b & 0xfffffffffffffull) | (e ? 1ull << 52 : 0ull);
    const long long v = ge_shift(m, (e ? e : 1) - 1075 + s);
    return (long long)b < 0 ? -v : v;
}

// the mean to a multiple of 2^r, 2^r <= 2^-28 sd 2^s (sd 2^s >= 2^53 / sqrt(n))
__device__ __forceinline__ long long ge_round_mean(long long m, long long n)
{
    const int r = 25 - (64 - __clzll(n - 1)) / 2 - 1;    // sqrt(n) <= 2^((bits(n-1) + 1) / 2)
    if (r <= 0) return m;
    return (long long)(((unsigned long long)m + (1ull << (r - 1))) & ~((1ull << r) - 1ull));
}

// MN-major, 128-byte-swizzled operand: rows of 64 columns (128 bytes) per sample, atoms of
// 8 samples (1024 bytes); leading byte offset: the next 64 columns, stride byte offset: the
// next 8 samples.
__device__ __forceinline__ uint64_t ge_desc(uint32_t saddr)
{
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFF);
    d |= (uint64_t)(GE_A_BLK >> 4) << 16;
    d |= (uint64_t)(1024 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

__device__ __forceinline__ void tc_ld_8cols_async(uint32_t taddr, uint32_t (&r)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
}
// the loads in flight, whose registers no use may move above it
__device__ __forceinline__ void tc_ld_wait5(uint32_t (&r)[5][8])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 5; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) asm volatile("" : "+r"(r[i][j]));
}

__device__ __forceinline__ void tc_zero_8cols(uint32_t taddr)
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%1,%1,%1,%1,%1,%1,%1};" ::"r"(taddr), "r"(0u)
                 : "memory");
}

// one lane of a converged warp
__device__ __forceinline__ bool elect_lane()
{
    uint32_t ok;
    asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}" : "=r"(ok));
    return ok != 0;
}

// Digits of two elements as packed BF16.  x holds a biased digit (d' = digit + 64 in 0..127)
// of each in the low 7 bits of its halves: 0x4300 + d' is 128 + d', minus 192.
__device__ __forceinline__ uint32_t ge_digit2(uint32_t x)
{
    uint32_t r;
    asm("add.rn.bf16x2 %0, %1, %2;" : "=r"(r) : "r"((x & 0x007f007fu) | 0x43004300u), "r"(0xc340c340u));
    return r;
}
// The 8 digits of two biased elements, a and b the low and high 28 bits of each, 14 bits of
// both at a time: about 10 shifts and logic operations an element (their pipe runs at half
// rate).
__device__ __forceinline__ void ge_cut2(uint32_t a0, uint32_t b0, uint32_t a1, uint32_t b1, uint32_t (&w)[GE_S])
{
    uint32_t q[4];
    q[0] = __byte_perm(a0, a1, 0x5410);
    q[1] = __byte_perm(a0 >> 14, a1 >> 14, 0x5410);
    q[2] = __byte_perm(b0, b1, 0x5410);
    q[3] = __byte_perm(b0 >> 14, b1 >> 14, 0x5410);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        w[7 - 2 * i] = ge_digit2(q[i]);
        w[6 - 2 * i] = ge_digit2(q[i] >> 7);
    }
}

// round(x 2^s) - m of an FP32 element, m = mhi 2^28 + mlo, as its low and high 28 bits (the
// bits above them are not cleared): y = x 2^s is exact in FP32, as are its rounding to a
// multiple of 2^28 and the rest.  32-bit conversions: the 64-bit one runs on the FP64 pipe.
__device__ __forceinline__ void ge_fixed28(float x, float scale, int mlo, int mhi, uint32_t &a, uint32_t &b)
{
    const float y = x * scale;
    const int hi = __float2int_rn(y * 0x1p-28f);
    const int lo = __float2int_rn(fmaf(__int2float_rn(hi), -0x1p28f, y)) - mlo;
    a = (uint32_t)lo;
    b = (uint32_t)(hi - mhi + (lo >> 28));
}

// tile t -> (row block bi, column block bj): the tiles that reach the upper triangle
__host__ __device__ inline int ge_first(int bi) { return bi * GE_M / GE_N; }
__device__ __forceinline__ void ge_tile(int t, int nc, int &bi, int &bj)
{
    bi = 0;
    while (t >= nc - ge_first(bi)) {
        t -= nc - ge_first(bi);
        ++bi;
    }
    bj = ge_first(bi) + t;
}

// One CTA: a 128 x 48 tile over a range of kper samples.  Warps 0-21 cut the digits of a
// stage of 32 samples into shared memory (a thread takes 8 neighbouring columns of a
// sample: one 16-byte store per digit, conflict-free under the swizzle) while the last warp
// runs the 49 digit-pair products of the stage before it on the tensor core; then the
// producers read the accumulators back.  B's digits lie side by side as one operand of 8 x 48
// columns and the accumulators of the weights side by side in TMEM, so the products of A's
// digit x with B's digits 0, 1, ... are one product with N = 48 min(8, 10 - x) columns that
// adds into the weights x, x + 1, ... (two instructions above N = 256): A is read once for
// them all, 13 instructions per 16 samples instead of 49 (which took 80 clocks each: 1.56 ms
// at p = 1000, n = 20000, this 1.23).  The cutting is about 20 instructions an element, each
// element cut once per tile that needs it, and wants many warps in flight (64-bit fixed point
// and a 64-bit shift a digit: 45 instructions, 1.23 ms; 1.06 as it is, 1.00 with a warp's lanes
// on the samples of one column group).  Bound: shared memory -- per stage of 32 samples the
// products read 250 KB (1950 clocks at 128 bytes) beside 88 KB of digit stores; 3.7 k clocks
// measured -- and 13 k clocks a CTA of setup, last products and readback (the readback through
// shared memory with coalesced atomics: the same time).
template <typename T>
__global__ void __launch_bounds__(GE_THREADS, 1) gram_exact_kernel(const T *__restrict__ X, long long n, int p,
                                                                   long long ld, const double *mean,
                                                                   const double *rsd, unsigned long long *C,
                                                                   long long ldc, int ntiles, int kper, int vec, int *err)
{
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    __shared__ __align__(8) uint64_t full[GE_STAGES], empty[GE_STAGES], done;
    __shared__ uint32_t tmem_base;
    __shared__ int fail;
    // per column c = 8 group + j: round(mean 2^s) - the digits' bias as its low 28 and upper
    // 32 bits, [j / 2][group] in the order lo, hi, lo, hi; s and 2^s (FP32 input) [j / 4][group]
    __shared__ int4 mint[4][GE_CH];
    __shared__ int4 shf[2][GE_CH];
    __shared__ float4 scl[2][GE_CH];
    __shared__ int far[GE_CH];                       // a column of the group needs the 64-bit fixed point
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    int bi, bj;
    const int split = blockIdx.x / ntiles;
    ge_tile(blockIdx.x - split * ntiles, (p + GE_N - 1) / GE_N, bi, bj);
    const int a0 = bi * GE_M, b0 = bj * GE_N;
    const long long k0 = (long long)split * kper;
    const long long k1 = k0 + kper < n ? k0 + kper : n;
    const int ns = (int)((k1 - k0 + GE_K - 1) / GE_K);

    // a producer warp's 8 columns c .. c + 7, a lane's sample k of the stage: the columns'
    // constants are the same for the warp, the 16-byte stores free of bank conflicts.  The first
    // samples are in flight over the setup.
    static_assert(GE_K == 32, "a lane per sample");
    const bool isA = warp < GE_M / 8;
    const int k = lane, gi = min(warp, GE_CH - 1), ch = isA ? gi : gi - GE_M / 8;
    const int c = (isA ? a0 : b0) + ch * 8;
    uint8_t *out = smem + (isA ? (ch >> 3) * GE_A_BLK + (((ch & 7) ^ (k & 7)) << 4) : GE_S * GE_A) + k * 128;
    const bool wide = vec && c + 8 <= p;
    T x[8];
    auto load = [&](long long t) {
        const T *q = X + t * ld + c;
        if (t < k1 && wide) {
            if constexpr (sizeof(T) == 4) {
                const float4 f0 = __ldg((const float4 *)q), f1 = __ldg((const float4 *)q + 1);
                x[0] = f0.x, x[1] = f0.y, x[2] = f0.z, x[3] = f0.w;
                x[4] = f1.x, x[5] = f1.y, x[6] = f1.z, x[7] = f1.w;
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const double2 d = __ldg((const double2 *)q + j);
                    x[2 * j] = d.x, x[2 * j + 1] = d.y;
                }
            }
        } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) x[j] = t < k1 && c + j < p ? __ldg(q + j) : (T)0;
        }
    };
    if (tid < GE_PROD) load(k0 + k);

    if (tid == 0) {
        for (int s = 0; s < GE_STAGES; ++s) {
            mbar_init(&full[s], GE_PROD / 32);
            mbar_init(&empty[s], 1);
        }
        mbar_init(&done, 1);
        fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    constexpr unsigned long long BIAS = 64ull * ((1ull << 56) - 1) / 127ull;   // 64 in every digit
    for (int i = tid; i < GE_CH; i += GE_THREADS) far[i] = 0;
    __syncthreads();
    for (int i = tid; i < GE_COLS; i += GE_THREADS) {
        const int c = i < GE_M ? a0 + i : b0 + (i - GE_M);
        int s = 0;
        // a column without digits: every x shifted out
        const bool live = c < p && ge_scale(rsd[c], n, s);
        const int gr = i >> 3, j = i & 7;
        const long long m = (live ? ge_round_mean(ge_fixed(mean[c], s), n) : 0ll) - (long long)BIAS;
        ((int *)&shf[j >> 2][gr])[j & 3] = live ? s : -4096;
        ((int *)&mint[j >> 1][gr])[2 * (j & 1)] = (int)(m & 0xfffffff);
        ((int *)&mint[j >> 1][gr])[2 * (j & 1) + 1] = (int)(m >> 28);
        // ge_fixed28: 2^s a normal FP32 number, x 2^s 2^-28 in 32 bits (|x| <= |mean| + sqrt(n) sd
        // and sqrt(n) sd 2^s < 2^54)
        const int em = ((__double2hiint(live ? mean[c] : 0.0) >> 20) & 0x7ff) - 1022;     // |mean| < 2^em
        const bool near = !live || (s >= -120 && s <= 120 && em + s <= 57);
        ((float *)&scl[j >> 2][gr])[j & 3] = live && near ? __int_as_float((s + 127) << 23) : 0.f;
        if (!near) far[gr] = 1;
    }
    if (warp == GE_PROD / 32) tc_alloc(&tmem_base, GE_TMEM);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base;
    // A's digit 0 sets the weights 0 to 7, the last two start from zero
    if (warp < 4) {
#pragma unroll
        for (int c = GE_S * GE_N; c < GE_W * GE_N; c += 8) tc_zero_8cols(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c);
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();

    if (warp == GE_PROD / 32) {
        // One thread issues every product, an elected lane (uniform registers); descriptors are
        // a base plus immediates.
        constexpr uint32_t mn = (1u << 15) | (1u << 16);     // both operands MN-major
        if (elect_lane()) {
        for (int i = 0; i < ns; ++i) {
            const int s = i % GE_STAGES;
            if (!mbar_wait(&full[s], (unsigned)(i / GE_STAGES) & 1u)) {
                atomicExch(&fail, 1);
                break;
            }
            tc_fence_after();
            const uint64_t da = ge_desc(smem_u32(smem + s * GE_STAGE));
            const uint64_t db = da + (GE_S * GE_A >> 4);
#pragma unroll
            for (int ks = 0; ks < GE_K / 16; ++ks)
#pragma unroll
                for (int x = 0; x < GE_S; ++x) {
                    const int N = GE_N * (GE_W - x < GE_S ? GE_W - x : GE_S), N1 = N < 256 ? N : 256;
                    const uint32_t acc = ks == 0 && x == 0 ? (uint32_t)i : 1u;
                    tc_mma(tmem + (uint32_t)(x * GE_N), da + ((x * GE_A + ks * 2048) >> 4), db + ((ks * 2048) >> 4),
                           idesc_bf16_f32(GE_M, N1) | mn, acc);
                    if (N > 256)
                        tc_mma(tmem + (uint32_t)(x * GE_N + 256), da + ((x * GE_A + ks * 2048) >> 4),
                               db + ((4 * GE_A_BLK + ks * 2048) >> 4), idesc_bf16_f32(GE_M, N - 256) | mn, acc);
                }
            tc_commit(&empty[s]);
        }
        tc_commit(&done);
        }
        __syncwarp();
    } else {
        const bool slow = far[gi] != 0;
        bool ok = true;
        for (int i = 0; i < ns; ++i) {
            const int s = i % GE_STAGES;
            const long long t = k0 + (long long)i * GE_K + k;
            uint32_t w[4][GE_S];
            if (t < k1) {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int4 m = mint[j][gi];
                    uint32_t a0, b0, a1, b1;
                    if (sizeof(T) == 4 && !slow) {
                        const float4 sc = scl[j >> 1][gi];
                        ge_fixed28((float)x[2 * j], j & 1 ? sc.z : sc.x, m.x, m.y, a0, b0);
                        ge_fixed28((float)x[2 * j + 1], j & 1 ? sc.w : sc.y, m.z, m.w, a1, b1);
                    } else {
                        const int4 sh = shf[j >> 1][gi];
                        const long long m0 = ((long long)m.y << 28) + m.x, m1 = ((long long)m.w << 28) + m.z;
                        const unsigned long long y0 = (unsigned long long)(ge_fixed(x[2 * j], j & 1 ? sh.z : sh.x) - m0);
                        const unsigned long long y1 = (unsigned long long)(ge_fixed(x[2 * j + 1], j & 1 ? sh.w : sh.y) - m1);
                        a0 = (uint32_t)y0, b0 = (uint32_t)(y0 >> 28), a1 = (uint32_t)y1, b1 = (uint32_t)(y1 >> 28);
                    }
                    ge_cut2(a0, b0, a1, b1, w[j]);
                }
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j)
#pragma unroll
                    for (int d = 0; d < GE_S; ++d) w[j][d] = 0u;
            }
            if (i + 1 < ns) load(t + GE_K);              // in flight over the wait and the stores
            if (i >= GE_STAGES) ok = __all_sync(0xffffffffu, mbar_wait(&empty[s], (unsigned)(i / GE_STAGES - 1) & 1u));
            if (!ok) {
                atomicExch(&fail, 1);
                break;
            }
            uint8_t *o = out + s * GE_STAGE;
            if (isA) {
#pragma unroll
                for (int d = 0; d < GE_S; ++d) *(uint4 *)(o + d * GE_A) = make_uint4(w[0][d], w[1][d], w[2][d], w[3][d]);
            } else {
#pragma unroll
                for (int d = 0; d < GE_S; ++d) {
                    const int g8 = d * (GE_N / 8) + ch;      // group of 8 among B's 384 columns
                    *(uint4 *)(o + (g8 >> 3) * GE_A_BLK + (((g8 & 7) ^ (k & 7)) << 4)) =
                        make_uint4(w[0][d], w[1][d], w[2][d], w[3][d]);
                }
            }
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(&full[s]);
        }
        // the accumulators: warp -> TMEM lane quadrant warp % 4, every (warps / 4)-th 8 columns
        ok = __all_sync(0xffffffffu, mbar_wait(&done, 0u)) && !*(volatile int *)&fail;
        if (ok) {
            tc_fence_after();
            const int row = (warp & 3) * 32 + lane, a = a0 + row;
            const uint32_t lane_addr = tmem + ((uint32_t)((warp & 3) * 32) << 16);
#pragma unroll 1
            for (int cb = (warp >> 2) * 8; warp < 16 && cb < GE_N; cb += 32) {
                long long acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
                uint32_t r[5][8];
#pragma unroll
                for (int w = 0; w < GE_W; ++w) {
                    if (w % 5 == 0) {                        // five weights in flight
#pragma unroll
                        for (int i = 0; i < 5; ++i) tc_ld_8cols_async(lane_addr + (uint32_t)((w + i) * GE_N + cb), r[i]);
                        tc_ld_wait5(r);
                    }
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const long long v = (long long)__float2int_rn(__uint_as_float(r[w % 5][j]));
                        acc[j] += w < GE_S ? v * (1ll << (w < GE_S ? 52 - 7 * w : 0))    // units of 2^46
                                           : (v + (1ll << (7 * w - 53))) >> (7 * w - 52);
                    }
                }
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int b = b0 + cb + j;
                    if (a < b && b < p) atomicAdd(C + (long long)a * ldc + b, (unsigned long long)acc[j]);
                }
            }
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == GE_PROD / 32) {
        if (lane == 0 && !mbar_wait(&done, 0u)) fail = 1;    // every issued product finished
        __syncwarp();
        tc_dealloc(tmem, GE_TMEM);
    }
    if (tid == GE_PROD && fail) atomicExch(err, 7);          // PC_ERR_TIMEOUT
}

// The integers above the diagonal to correlations, mirrored, unit diagonal (and the FP32
// matrix): corr = Q 2^46 (rsd_a 2^-s_a) (rsd_b 2^-s_b) / n.  32 x 32 tiles, the mirror
// written through shared memory.
__global__ void __launch_bounds__(256) gram_finish_kernel(double *C, long long ldc, int p, long long n,
                                                          const double *mean, const double *rsd, float *C32, int ldc32,
                                                          const int *err)
{
    __shared__ double tile[32][33];
    __shared__ double fa[32], fb[32];
    const int bi = blockIdx.y, bj = blockIdx.x;
    if (bj < bi) return;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    if (ty < 2) {
        const int c = (ty ? bj : bi) * 32 + tx;
        int s = 0;
        double f = 0.0;
        if (c < p) {
            const double r = rsd[c];
            // a constant column: 0; one with a non-finite statistic: NaN
            f = ge_scale(r, n, s) ? ldexp(r, -s) : (mean[c] - mean[c]) + (r - r);
        }
        (ty ? fb : fa)[tx] = f;
    }
    __syncthreads();
    // 2^46 / n; a product whose bounded wait ran out (err) gives no numbers
    const double unit = *err ? __longlong_as_double(0x7ff8000000000000ll) : 70368744177664.0 / (double)n;
    for (int k = ty; k < 32; k += 8) {
        const int a = bi * 32 + k, b = bj * 32 + tx;
        double v = 0.0;
        if (a < p && b < p && a <= b) {
            const long long q = *(const long long *)(C + (long long)a * ldc + b);
            v = a == b ? 1.0 : (double)q * unit * (fa[k] * fb[tx]);
            C[(long long)a * ldc + b] = v;
            if (C32) C32[(long long)a * ldc32 + b] = (float)v;
        }
        tile[k][tx] = v;
    }
    __syncthreads();
    for (int k = ty; k < 32; k += 8) {
        const int b = bj * 32 + k, a = bi * 32 + tx;
        if (a < p && b < p && a < b) {
            C[(long long)b * ldc + a] = tile[tx][k];
            if (C32) C32[(long long)b * ldc32 + a] = (float)tile[tx][k];
        }
    }
}

}  // namespace

cudaError_t launch_gram_exact(const void *X, int dtype, long long n, int p, long long ld, const double *mean,
                              const double *rsd, double *C, long long ldc, float *C32, int ldc32, int *err,
                              cudaStream_t s)
{
    int dev = 0, sms = 148;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int nc = (p + GE_N - 1) / GE_N;
    int ntiles = 0;
    for (int bi = 0; bi * GE_M < p; ++bi) ntiles += nc - ge_first(bi);
    // K splits: at least n / 512 (exact accumulators), and whole waves of one CTA per SM as
    // long as a CTA keeps 2 stages of samples
    const long long smin = (n + GE_KMAX - 1) / GE_KMAX, smax = std::max<long long>(smin, n / (2 * GE_K));
    long long waves = (ntiles * smin + sms - 1) / sms;
    long long splits = std::min(smax, std::max(smin, waves * sms / ntiles));
    long long kper = (n + splits - 1) / splits;
    kper = std::min<long long>(GE_KMAX, (kper + GE_K - 1) / GE_K * GE_K);
    splits = (n + kper - 1) / kper;
    if (splits * ntiles > 0x7fffffffll) return cudaErrorInvalidValue;
    const size_t smem = (size_t)GE_STAGES * GE_STAGE + 1024;
    const unsigned grid = (unsigned)(splits * ntiles);
    if (dtype == 1) {
        const int vec = ld % 2 == 0 && ((uintptr_t)X & 15) == 0;
        e = cudaFuncSetAttribute(gram_exact_kernel<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        gram_exact_kernel<double><<<grid, GE_THREADS, smem, s>>>((const double *)X, n, p, ld, mean, rsd,
                                                                 (unsigned long long *)C, ldc, ntiles, (int)kper, vec, err);
    } else {
        const int vec = ld % 4 == 0 && ((uintptr_t)X & 15) == 0;
        e = cudaFuncSetAttribute(gram_exact_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        gram_exact_kernel<float><<<grid, GE_THREADS, smem, s>>>((const float *)X, n, p, ld, mean, rsd,
                                                                (unsigned long long *)C, ldc, ntiles, (int)kper, vec, err);
    }
    note_launch();
    const int nt = (p + 31) / 32;
    gram_finish_kernel<<<dim3(nt, nt), 256, 0, s>>>(C, ldc, p, n, mean, rsd, C32, ldc32, err);
    note_launch();
    return cudaGetLastError();
}

}  // namespace fpc
