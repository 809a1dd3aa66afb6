// mlp.cu -- the conditioning-set proposal network (not in the paper): a
// member score s(u, v, k) for every candidate k of an ordered pair (u, v) at
// stage l, used to enumerate the likeliest separating sets first.
//
//   h1 = relu(W1 x + b1)  (16 -> 128),  h2 = relu(W2 h1 + b2)  (128 -> 128),
//   s = w3 . h2 + b3;     training loss: mean BCE(sigmoid(s), y).
//
// Forward and gradient on the tensor cores (tcgen05, BF16 operands, FP32 accumulators in
// TMEM): 128-row tiles of features go to a swizzled shared tile, D1 = X W1^T (K = 16), the
// epilogue applies bias + ReLU and writes h1 (BF16) into the A operand of D2 = h1 W2^T
// (K = 128), and the second epilogue reduces h2 against w3; the gradient kernel goes on to
// the backward products of the same tile.  Adam, and an FP32 backward kept as an option,
// run on the CUDA cores.
#include "internal.h"
#include "device_util.cuh"
#include "tc_util.cuh"

#include <cuda_bf16.h>

#include <algorithm>

namespace fpc {

constexpr int NF = 16, NH = 128;
constexpr int NPARAM = NH * NF + NH + NH * NH + NH + NH + 1;   // 18817
constexpr int OFF_W1 = 0, OFF_B1 = NH * NF, OFF_W2 = OFF_B1 + NH, OFF_B2 = OFF_W2 + NH * NH;
constexpr int OFF_W3 = OFF_B2 + NH, OFF_B3 = OFF_W3 + NH;
constexpr int T_ROWS = 128;
constexpr int W1_TILE = 128 * 128;            // bytes: 128 rows x 64 bf16 (features in the first 16, b2 behind)
constexpr int A1_TILE = 128 * 128;
constexpr int W2_TILE = 128 * 128;            // bytes per 64-wide K tile

// byte offset of element (row, col) of a 128-byte-row K-major tile with the
// 128-byte swizzle: the 16-byte chunk index is XORed with row mod 8
__device__ __forceinline__ int sw128_off(int row, int col_bf16)
{
    const int chunk = col_bf16 >> 3, within = col_bf16 & 7;
    return row * 128 + (((chunk ^ (row & 7)) << 4) | (within << 1));
}

// Member features of candidate k for the ordered pair (u, v) at stage l, from
// the FP32 correlation matrix: marginal correlations, first-order partial
// correlations, the first-order test statistic relative to the threshold,
// and the stage shape.
__device__ __forceinline__ void member_features_of(float cuv, float cuk, float cvk, int l, int d, float sqn_over_q,
                                                   float *f)
{
    const float e = 1e-6f;
    const float ruv_k = (cuv - cuk * cvk) * rsqrtf(fmaxf((1.f - cuk * cuk) * (1.f - cvk * cvk), e));
    const float ruk_v = (cuk - cuv * cvk) * rsqrtf(fmaxf((1.f - cuv * cuv) * (1.f - cvk * cvk), e));
    const float rvk_u = (cvk - cuv * cuk) * rsqrtf(fmaxf((1.f - cuv * cuv) * (1.f - cuk * cuk), e));
    f[0] = fabsf(cuv);
    f[1] = fabsf(cuk);
    f[2] = fabsf(cvk);
    f[3] = fabsf(cuk * cvk);
    f[4] = fabsf(ruv_k);
    f[5] = fabsf(ruk_v);
    f[6] = fabsf(rvk_u);
    f[7] = fminf(sqn_over_q * fabsf(ruv_k), 4.f);
    f[8] = fminf(sqn_over_q * fabsf(cuv), 4.f);
    f[9] = fminf(fmaxf(sqn_over_q * (fabsf(cuv) - fabsf(ruv_k)), -4.f), 4.f);
    f[10] = d > 0 ? (float)l / (float)d : 0.f;
    f[11] = log2f((float)d + 1.f) * 0.125f;
    f[12] = (float)l * (1.f / 16.f);
    f[13] = (cuv * cuk * cvk > 0.f) ? 1.f : 0.f;
    f[14] = 1.f;
    f[15] = 0.f;
}

__device__ __forceinline__ void member_features(const float *C, int ldc, const long long *prow, int u, int v, int k,
                                                int l, int d, float sqn_over_q, float *f)
{
    member_features_of(C[cidx(prow, ldc, u, v)], C[cidx(prow, ldc, u, k)], C[cidx(prow, ldc, v, k)], l, d,
                       sqn_over_q, f);
}

// Packs the FP32 master parameters into the swizzled BF16 B-operand tiles of
// W1 (128 x 64, features zero-padded) and W2 (two 128 x 64 K tiles).
// ... and W2 transposed (rows i, K = o) as the B operand of the backward
// product dL/dh1 = dL/da2 W2, after the forward's tiles.
__global__ void mlp_pack_kernel(const float *theta, uint8_t *wpack)
{
    const int o = blockIdx.x;            // output unit (row of the B operand)
    for (int c = threadIdx.x; c < 64; c += blockDim.x) {
        float w = c < NF ? theta[OFF_W1 + o * NF + c] : 0.f;
        if (c >= NF && c < NF + 3) {                     // b2 in three BF16 parts
            w = theta[OFF_B2 + o];
            for (int k = NF; k < c; ++k) w -= __bfloat162float(__float2bfloat16_rn(w));
        }
        *(__nv_bfloat16 *)(wpack + sw128_off(o, c)) = __float2bfloat16_rn(w);
    }
    for (int c = threadIdx.x; c < NH; c += blockDim.x) {
        const int t = c >> 6;
        const __nv_bfloat16 w = __float2bfloat16_rn(theta[OFF_W2 + o * NH + c]);
        *(__nv_bfloat16 *)(wpack + W1_TILE + t * W2_TILE + sw128_off(o, c & 63)) = w;
        // element (i = c, K = o) of W2^T
        *(__nv_bfloat16 *)(wpack + W1_TILE + 2 * W2_TILE + (o >> 6) * W2_TILE + sw128_off(c, o & 63)) = w;
    }
}

// Where the rows of a forward pass come from.
struct MlpRows {
    // explicit features (R x 16 FP32), or ...
    const float *feats;
    long long R;
    // ... the candidates of the current stage: node u owns deg_u * (deg_u - 1)
    // rows starting at row_off[u] (pair j, candidate position x)
    const GraphDev *gp;
    const unsigned long long *row_off;
    const float *C32;
    int ldc;
    float sqn_over_q;
    const long long *nvec;   // batched problems: per-node samples (sqrt(n_u)/q per row)
    float inv_q;
};

// A candidate row of the current stage: node u (tracked by the caller, which
// walks it forward over consecutive rows), the pair's v, the candidate k.
struct RowRef {
    int u, v, k, d;
    bool ok;
};

__device__ __forceinline__ RowRef locate_row(const MlpRows &R, const GraphDev &g, long long row, long long nrows,
                                             int &ucur)
{
    RowRef r{0, 0, 0, 0, row < nrows};
    if (!r.ok) return r;
    while ((long long)R.row_off[ucur + 1] <= row) ++ucur;
    const int u = ucur, d = g.deg[u] - 1;
    const long long w = row - (long long)R.row_off[u];
    const int j = (int)(w / d), x = (int)(w - (long long)j * d);
    const int *nb = g.nbr + nidx(g, u);
    r.u = u;
    r.d = d;
    r.v = nb[j];
    r.k = nb[x + (x >= j)];
    return r;
}

// The correlations a row's features need (loaded one tile ahead of use).
struct RowVals {
    float cuv, cuk, cvk, sq;
    int d;
    bool ok;
};

__device__ __forceinline__ RowVals fetch_row(const MlpRows &R, const GraphDev &g, const RowRef &r)
{
    RowVals x{0.f, 0.f, 0.f, 0.f, r.d, r.ok};
    if (!r.ok) return x;
    x.cuv = R.C32[cidx(g.prow, R.ldc, r.u, r.v)];
    x.cuk = R.C32[cidx(g.prow, R.ldc, r.u, r.k)];
    x.cvk = R.C32[cidx(g.prow, R.ldc, r.v, r.k)];
    x.sq = R.nvec ? sqrtf((float)R.nvec[r.u]) * R.inv_q : R.sqn_over_q;
    return x;
}

// ---- epilogue pieces shared by the forward and the gradient kernels
// a + b and a * b + c on two FP32 values at once
__device__ __forceinline__ float2 add2(float2 a, float2 b)
{
    float2 r;
    asm("{\n .reg .b64 x, y, z;\n mov.b64 x, {%2, %3};\n mov.b64 y, {%4, %5};\n add.rn.f32x2 z, x, y;\n"
        " mov.b64 {%0, %1}, z;\n}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c)
{
    float2 r;
    asm("{\n .reg .b64 x, y, z, w;\n mov.b64 x, {%2, %3};\n mov.b64 y, {%4, %5};\n mov.b64 z, {%6, %7};\n"
        " fma.rn.f32x2 w, x, y, z;\n mov.b64 {%0, %1}, w;\n}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return r;
}
// relu(bf16(a)), relu(bf16(b)) packed (rounding and the maximum with 0 commute)
__device__ __forceinline__ uint32_t relu_pack(float2 v)
{
    __nv_bfloat162 h = __hmax2(__floats2bfloat162_rn(v.x, v.y), __floats2bfloat162_rn(0.f, 0.f));
    return *(uint32_t *)&h;
}
// barrier of the N threads of group gi
template <int N>
__device__ __forceinline__ void group_sync(int gi)
{
    asm volatile("bar.sync %0, %1;" ::"r"(gi + 1), "n"(N) : "memory");
}

// a row's features as BF16, into the first 16 columns of row r of a swizzled tile
__device__ __forceinline__ void store_features(uint8_t *tile, int r, const float (&f)[NF])
{
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        uint32_t w[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            __nv_bfloat162 h = __floats2bfloat162_rn(f[8 * q + 2 * k], f[8 * q + 2 * k + 1]);
            w[k] = *(uint32_t *)&h;
        }
        *(uint4 *)(tile + sw128_off(r, 8 * q)) = make_uint4(w[0], w[1], w[2], w[3]);
    }
}
__device__ __forceinline__ void load_features(const float *feats, long long row, bool ok, int vec, float (&f)[NF])
{
    if (ok && vec) {
        const float4 *q = (const float4 *)(feats + row * NF);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float4 x = __ldg(q + k);
            f[4 * k] = x.x, f[4 * k + 1] = x.y, f[4 * k + 2] = x.z, f[4 * k + 3] = x.w;
        }
    } else {
#pragma unroll
        for (int i = 0; i < NF; ++i) f[i] = ok ? feats[row * NF + i] : 0.f;
    }
}

// fn(c0, v) over the 128 columns of this warp's TMEM lanes, 32 at a time, the next 32 in
// flight meanwhile.
template <class F>
__device__ __forceinline__ void tmem_columns(uint32_t taddr, const F &fn)
{
    uint32_t a[32], b[32];
    tc_ld_32cols_async(taddr, a);
    tc_ld_wait(a);
    tc_ld_32cols_async(taddr + 32, b);
    fn(0, a);
    tc_ld_wait(b);
    tc_ld_32cols_async(taddr + 64, a);
    fn(32, b);
    tc_ld_wait(a);
    tc_ld_32cols_async(taddr + 96, b);
    fn(64, a);
    tc_ld_wait(b);
    fn(96, b);
}
__device__ __forceinline__ float2 pair_of(const uint32_t (&v)[32], int c)
{
    return make_float2(__uint_as_float(v[c]), __uint_as_float(v[c + 1]));
}

// h1 = relu(D1 + b1) of this thread's row (TMEM lane) -> BF16 into the K-major operand
// tile sA2 (and to out when given); mask: its positive entries, 32 columns per word.
template <bool MASK>
__device__ __forceinline__ void epilogue_h1(uint32_t taddr, uint8_t *sA2, int r, const float *b1, uint32_t *mask,
                                            __nv_bfloat16 *out)
{
    tmem_columns(taddr, [&](int c0, const uint32_t (&v)[32]) {
        uint32_t m = 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            uint32_t w[4];
#pragma unroll
            for (int k = 0; k < 4; k += 2) {
                const int c = q * 8 + 2 * k;
                const float4 b = *(const float4 *)(b1 + c0 + c);
                w[k] = relu_pack(add2(pair_of(v, c), make_float2(b.x, b.y)));
                w[k + 1] = relu_pack(add2(pair_of(v, c + 2), make_float2(b.z, b.w)));
            }
            if (MASK) {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if (w[k] & 0xffffu) m |= 1u << (q * 8 + 2 * k);
                    if (w[k] >> 16) m |= 2u << (q * 8 + 2 * k);
                }
            }
            const int c = c0 + q * 8;
            const uint4 x = make_uint4(w[0], w[1], w[2], w[3]);
            *(uint4 *)(sA2 + (c >> 6) * W2_TILE + sw128_off(r, c & 63)) = x;
            if (out) *(uint4 *)(out + c) = x;
        }
        if (MASK) mask[c0 >> 5] = m;
    });
}

// s = w3 . relu(D2) of this thread's row (D2 holds b2 already), h2 = relu(D2) to out when given
__device__ __forceinline__ float epilogue_score(uint32_t taddr, const float *w3, float *out)
{
    float2 s[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
    tmem_columns(taddr, [&](int c0, const uint32_t (&v)[32]) {
#pragma unroll
        for (int c = 0; c < 32; c += 4) {
            const float4 w = *(const float4 *)(w3 + c0 + c);
            float2 h = pair_of(v, c), g = pair_of(v, c + 2);
            h.x = fmaxf(h.x, 0.f);
            h.y = fmaxf(h.y, 0.f);
            g.x = fmaxf(g.x, 0.f);
            g.y = fmaxf(g.y, 0.f);
            if (out) *(float4 *)(out + c0 + c) = make_float4(h.x, h.y, g.x, g.y);
            s[0] = fma2(make_float2(w.x, w.y), h, s[0]);
            s[1] = fma2(make_float2(w.z, w.w), g, s[1]);
        }
    });
    const float2 t = add2(s[0], s[1]);
    return t.x + t.y;
}

// A constant operand: every row 1, 1, 1, 0, ... in columns 16..31 of a swizzled tile.  The
// product with the same columns of the W1 tile, which hold b2 in three BF16 parts (24 bits:
// exactly), starts the accumulator of the second layer at b2, so that its epilogue adds no
// bias.  (b1 is added in FP32 by the epilogue: h1 is rounded to BF16 right behind it.)
__device__ __forceinline__ void store_ones(uint8_t *tile, int t, int nthreads)
{
    for (int r = t; r < T_ROWS; r += nthreads) {
        *(uint4 *)(tile + sw128_off(r, 16)) = make_uint4(0x3f803f80u, 0x00003f80u, 0u, 0u);
        *(uint4 *)(tile + sw128_off(r, 24)) = make_uint4(0u, 0u, 0u, 0u);
    }
}

// D2 = b2 + h1 W2^T: the issue of the second layer's products (one thread)
__device__ __forceinline__ void issue_layer2(uint32_t d, const uint8_t *sOnes, const uint8_t *sW1, const uint8_t *sA2,
                                             const uint8_t *sW2, uint32_t idesc)
{
    tc_mma(d, sw128_desc(smem_u32(sOnes)) + 2, sw128_desc(smem_u32(sW1)) + 2, idesc, 0u);   // 32 bytes on: columns 16..31
    const uint64_t a = sw128_desc(smem_u32(sA2)), b = sw128_desc(smem_u32(sW2));
#pragma unroll
    for (int tt = 0; tt < 2; ++tt)
#pragma unroll
        for (int ks = 0; ks < 4; ++ks)
            tc_mma(d, a + (uint64_t)((tt * W2_TILE + ks * 32) >> 4), b + (uint64_t)((tt * W2_TILE + ks * 32) >> 4), idesc,
                   1u);
}

// Forward pass over rows [0, R): scores s, and for the CUDA-core backward h1 (BF16), h2
// (FP32).  A tile of 128 rows is a chain -- features, product, ReLU, product, score -- run by
// a group of 128 threads, one to a row; four groups per CTA, independent of one another,
// fill each other's waits (each has 128 TMEM columns,
// which D1 and D2 use in turn, and one 32 KB operand tile, whose first columns hold the
// features until h1 replaces them).  The next tile's features (or, for the rows of the
// current stage, its indices and correlations) are fetched while the products run.
// Measured, 1 M rows, the whole call: 170 us with one chain per CTA, two CTAs per SM and a
// scalar epilogue, 97 us now; 256 threads a chain, two to a row, took 111 (64 registers a
// thread spill).  Bound by shared memory -- the products' operands (640 clocks a tile), the
// epilogues' reads of b1 and w3 (384) and stores of h1 (256) -- and the chains' latency.
constexpr int FW_G = 4, FW_GT = 128, FW_THREADS = FW_G * FW_GT;
constexpr int FW_SMEM = W1_TILE + 2 * W2_TILE + A1_TILE + FW_G * 2 * W2_TILE + 1024;
__global__ void __launch_bounds__(FW_THREADS, 1) mlp_forward_kernel(MlpRows rows, GraphDev g, const uint8_t *wpack,
                                                                    const float *theta, float *scores,
                                                                    __nv_bfloat16 *h1_out, float *h2_out, int vec,
                                                                    int *err)
{
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    __shared__ __align__(8) uint64_t bars[FW_G];
    __shared__ uint32_t tmem_base;
    __shared__ __align__(16) float b1[NH], w3[NH];
    const int gi = threadIdx.x / FW_GT, tid = threadIdx.x % FW_GT, warp = threadIdx.x >> 5;
    if (!rows.feats && (g.info->done || g.info->halt)) return;
    const long long R = rows.feats ? rows.R : (long long)rows.row_off[g.p];
    const long long ntiles = (R + T_ROWS - 1) / T_ROWS;
    // this group's tiles: with few tiles one group per SM first
    const long long ng = ntiles < (long long)gridDim.x * FW_G ? ntiles : (long long)gridDim.x * FW_G;
    const long long id = (long long)gi * gridDim.x + blockIdx.x;
    if ((long long)blockIdx.x >= ng) return;             // no group of this CTA has a tile
    const long long tb = id < ng ? ntiles * id / ng : 0, te = id < ng ? ntiles * (id + 1) / ng : 0;
    uint8_t *sW1 = smem, *sW2 = smem + W1_TILE, *sOnes = sW2 + 2 * W2_TILE;
    uint8_t *sA = sOnes + A1_TILE + gi * 2 * W2_TILE;
    uint64_t *bar = &bars[gi];
    if (threadIdx.x == 0) {
        for (int w = 0; w < FW_G; ++w) mbar_init(&bars[w], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int i = threadIdx.x; i < (W1_TILE + 2 * W2_TILE) / 16; i += FW_THREADS)
        ((uint4 *)smem)[i] = ((const uint4 *)wpack)[i];
    for (int i = threadIdx.x; i < NH; i += FW_THREADS) {
        b1[i] = theta[OFF_B1 + i];
        w3[i] = theta[OFF_W3 + i];
    }
    store_ones(sOnes, threadIdx.x, FW_THREADS);
    const float b3 = theta[OFF_B3];
    if (warp == 0) tc_alloc(&tmem_base, 512);
    fence_proxy_async_smem();                            // the weights, written by every thread
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t d = tmem_base + (uint32_t)(gi * 128), dl = d + ((uint32_t)((warp & 3) * 32) << 16);
    constexpr uint32_t idesc = idesc_bf16_f32(128, 128);
    const int l = rows.feats ? 0 : g.info->l;
    unsigned phase = 0;
    bool ok = true;
    // the row this thread feeds into the first tile, located and fetched
    int ucur = 0;
    RowVals cur{};
    float f[NF];
    if (!rows.feats && tb < te) {
        const long long r0 = tb * T_ROWS + tid;
        if (r0 < R) ucur = (int)(upper_bound_dev(rows.row_off, (long long)g.p + 1, (unsigned long long)r0) - 1);
        cur = fetch_row(rows, g, locate_row(rows, g, r0, R, ucur));
    } else if (tb < te) {
        load_features(rows.feats, tb * T_ROWS + tid, tb * T_ROWS + tid < R, vec, f);
    }
    for (long long t = tb; t < te; ++t) {
        const long long row = t * T_ROWS + tid;
        if (!rows.feats) {
#pragma unroll
            for (int i = 0; i < NF; ++i) f[i] = 0.f;
            if (cur.ok) member_features_of(cur.cuv, cur.cuk, cur.cvk, l, cur.d, cur.sq, f);
        }
        store_features(sA, tid, f);
        fence_proxy_async_smem();
        group_sync<FW_GT>(gi);
        if (tid == 0) {
            tc_fence_after();
            tc_mma(d, sw128_desc(smem_u32(sA)), sw128_desc(smem_u32(sW1)), idesc, 0u);
            tc_commit(bar);
        }
        __syncwarp();
        // the next tile's row: features or indices now, correlations before the second wait
        RowRef nxt{0, 0, 0, 0, false};
        if (t + 1 < te) {
            if (rows.feats) load_features(rows.feats, row + T_ROWS, row + T_ROWS < R, vec, f);
            else nxt = locate_row(rows, g, row + T_ROWS, R, ucur);
        }
        ok = ok && mbar_wait(bar, phase);
        phase ^= 1u;
        tc_fence_after();
        epilogue_h1<false>(dl, sA, tid, b1, nullptr, h1_out && row < R ? h1_out + row * NH : nullptr);
        tc_fence_before();
        fence_proxy_async_smem();
        group_sync<FW_GT>(gi);
        if (tid == 0) {
            tc_fence_after();
            issue_layer2(d, sOnes, sW1, sA, sW2, idesc);
            tc_commit(bar);
        }
        __syncwarp();
        if (!rows.feats && t + 1 < te) cur = fetch_row(rows, g, nxt);
        ok = ok && mbar_wait(bar, phase);
        phase ^= 1u;
        tc_fence_after();
        const float s = b3 + epilogue_score(dl, w3, h2_out && row < R ? h2_out + row * NH : nullptr);
        if (row < R) scores[row] = s;
        tc_fence_before();                               // before the next tile's product into d
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tc_dealloc(tmem_base, 512);
    if (!ok && tid == 0) atomicExch(err, 7);             // a bounded wait expired
}

// Backward pass for rows [0, R) of a batch: per-CTA FP32 partial gradients in
// registers, added into grad (atomics once per CTA).  Uses the activations the
// forward pass saved (h1 BF16 as consumed by layer 2, h2 FP32) and the BF16
// weights the forward pass used.
__global__ void __launch_bounds__(256) mlp_backward_kernel(const float *feats, const float *labels,
                                                           const float *scores, const __nv_bfloat16 *h1,
                                                           const float *h2, long long R, float inv_b,
                                                           const float *theta, float *grad, double *loss)
{
    extern __shared__ float bsm[];
    float(*sdh2)[NH + 1] = (float(*)[NH + 1])bsm;                       // dL/dh2 (masked) of the tile
    float(*sh1)[NH + 1] = (float(*)[NH + 1])(bsm + T_ROWS * (NH + 1));   // h1, then dL/dh1
    float(*sW2)[NH + 1] = (float(*)[NH + 1])(bsm + 2 * T_ROWS * (NH + 1)); // W2 rounded to BF16
    float(*sx)[NF] = (float(*)[NF])(bsm + 2 * T_ROWS * (NH + 1) + NH * (NH + 1));
    float *sds = bsm + 2 * T_ROWS * (NH + 1) + NH * (NH + 1) + T_ROWS * NF;
    const int tid = threadIdx.x;
    for (int e = tid; e < NH * NH; e += blockDim.x)
        sW2[e / NH][e % NH] = __bfloat162float(__float2bfloat16_rn(theta[OFF_W2 + e]));
    // per-thread partials: dW2 entries (o, i) with o = tid/2, i in the half tid&1
    float gW2[64];
#pragma unroll
    for (int i = 0; i < 64; ++i) gW2[i] = 0.f;
    float gW1[8], gb1 = 0.f, gb2 = 0.f, gw3 = 0.f, gb3 = 0.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) gW1[i] = 0.f;
    double lsum = 0.0;
    const int o = tid >> 1, ih = (tid & 1) * 64;
    __syncthreads();
    for (long long t0 = (long long)blockIdx.x * T_ROWS; t0 < R; t0 += (long long)gridDim.x * T_ROWS) {
        const int nr = (int)(R - t0 < T_ROWS ? R - t0 : T_ROWS);
        for (int r = tid; r < T_ROWS; r += blockDim.x) {
            float ds = 0.f;
            if (r < nr) {
                const float s = scores[t0 + r], y = labels[t0 + r];
                ds = (1.f / (1.f + __expf(-s)) - y) * inv_b;
                lsum += (double)(fmaxf(s, 0.f) + log1pf(__expf(-fabsf(s))) - y * s);
            }
            sds[r] = ds;
        }
        for (int e = tid; e < T_ROWS * NH; e += blockDim.x) {
            const int r = e / NH, c = e % NH;
            float hv1 = 0.f, d2 = 0.f;
            if (r < nr) {
                hv1 = __bfloat162float(h1[(t0 + r) * NH + c]);
                const float hv2 = h2[(t0 + r) * NH + c];
                d2 = hv2 > 0.f ? 1.f : 0.f;
            }
            sh1[r][c] = hv1;
            sdh2[r][c] = d2;                     // mask for now; scaled below
        }
        for (int e = tid; e < T_ROWS * NF; e += blockDim.x) {
            const int r = e / NF, c = e % NF;
            sx[r][c] = r < nr ? __bfloat162float(__float2bfloat16_rn(feats[(t0 + r) * NF + c])) : 0.f;
        }
        __syncthreads();
        // dW3 / db3 (threads 0..127 own one unit each) and the masked dh2
        for (int e = tid; e < T_ROWS * NH; e += blockDim.x) {
            const int r = e / NH, c = e % NH;
            sdh2[r][c] *= sds[r] * theta[OFF_W3 + c];
        }
        if (tid < NH) {
            float a = 0.f;
            for (int r = 0; r < nr; ++r) a = fmaf(sds[r], h2[(t0 + r) * NH + tid], a);
            gw3 += a;
        }
        if (tid == 0)
            for (int r = 0; r < nr; ++r) gb3 += sds[r];
        __syncthreads();
        // dW2[o][i] += sum_r dh2[r][o] h1[r][i]; db2[o]
#pragma unroll 4
        for (int r = 0; r < nr; ++r) {
            const float a = sdh2[r][o];
#pragma unroll
            for (int i = 0; i < 64; ++i) gW2[i] = fmaf(a, sh1[r][ih + i], gW2[i]);
        }
        if ((tid & 1) == 0)
            for (int r = 0; r < nr; ++r) gb2 += sdh2[r][o];
        __syncthreads();
        // dh1[r][i] = sum_o dh2[r][o] W2[o][i], masked by h1 > 0 (stored into sh1)
        for (int e = tid; e < T_ROWS * NH; e += blockDim.x) {
            const int r = e / NH, i = e % NH;
            float a = 0.f;
            if (r < nr && sh1[r][i] > 0.f)
                for (int q = 0; q < NH; ++q) a = fmaf(sdh2[r][q], sW2[q][i], a);
            sh1[r][i] = a;                   // sh1 now holds dh1 (masked); each (r, i) is read and
                                             // written by the same thread only
        }
        __syncthreads();
        // dW1[i][f] += sum_r dh1[r][i] x[r][f]; db1[i]   (thread -> unit i = tid/2, 8 features)
        {
            const int iu = tid >> 1, f0 = (tid & 1) * 8;
            for (int r = 0; r < nr; ++r) {
                const float a = sh1[r][iu];
#pragma unroll
                for (int q = 0; q < 8; ++q) gW1[q] = fmaf(a, sx[r][f0 + q], gW1[q]);
                if ((tid & 1) == 0) gb1 += a;
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 64; ++i) atomicAdd(&grad[OFF_W2 + o * NH + ih + i], gW2[i]);
    if ((tid & 1) == 0) atomicAdd(&grad[OFF_B2 + o], gb2);
    {
        const int iu = tid >> 1, f0 = (tid & 1) * 8;
#pragma unroll
        for (int q = 0; q < 8; ++q) atomicAdd(&grad[OFF_W1 + iu * NF + f0 + q], gW1[q]);
        if ((tid & 1) == 0) atomicAdd(&grad[OFF_B1 + iu], gb1);
    }
    if (tid < NH) atomicAdd(&grad[OFF_W3 + tid], gw3);
    if (tid == 0) atomicAdd(&grad[OFF_B3], gb3);
    if (loss) {
        // block-level sum of the loss terms
        __shared__ double red[256];
        red[tid] = lsum;
        __syncthreads();
        for (int s = 128; s > 0; s >>= 1) {
            if (tid < s) red[tid] += red[tid + s];
            __syncthreads();
        }
        if (tid == 0) atomicAdd(loss, red[0]);
    }
}

// Gradient of the mean loss, forward and backward in one kernel: BF16 operands, FP32
// accumulators in TMEM, nothing but features and labels read.  A group of 128 threads runs
// the chain of a 128-row tile, thread t owning row t (its TMEM lane):
//   D1 = x W1^T -> h1 = relu(D1 + b1)             D2 = b2 + h1 W2^T -> s = w3 . relu(D2) + b3
//   ds = (sigmoid(s) - y) / B,  da2 = ds w3 (h2 > 0)                  (FP32, then BF16)
//   D = da2 W2,  dW2 += da2^T h1                                      (one pair of products)
//   da1 = D (h1 > 0)                                                  (BF16)
//   D = da1^T [x | 1] -> dW1, db1
// The products that contract over the rows read the same tiles as the others, row-major with
// the units contiguous, as MN-major operands: nothing is transposed.  D1, D2, dL/dh1 and dW1
// use one set of 128 TMEM columns in turn, dW2 stays in another; two groups per CTA fill
// each other's waits.  dw3 and db2 (of the BF16 signals) are column sums over the rows:
// lanes exchange halves (31 shuffles for 32 columns instead of 5 for each).  db3 and the
// loss in FP32 and FP64.  Each group writes its sums to its own part of a workspace;
// mlp_reduce_kernel adds the parts in order.
// Measured, 100 thousand rows, the whole call: 666 us with the activations (77 MB) through
// memory, 2-byte transposing stores and three allocations a call; 87 us now.
constexpr int GR_G = 2, GR_THREADS = 128 * GR_G;
constexpr int GR_X = 128 * 64;                       // x tile: 128 rows x 32 columns (features, then 1 1 1 0 ...)
constexpr int GR_GROUP = GR_X + 4 * W2_TILE;
constexpr int GR_SMEM = W1_TILE + 4 * W2_TILE + GR_G * GR_GROUP + 1024;
constexpr int GR_PART = (NPARAM + 3) / 4 * 4 + 4;    // floats of a group's part: gradient, then the loss (double)

// shared-memory descriptor: leading and stride byte offsets, swizzle (2: 128 bytes, 4: 64)
__device__ __forceinline__ uint64_t smem_desc(const void *p, uint32_t lbo, uint32_t sbo, uint32_t swizzle)
{
    return (uint64_t)((smem_u32(p) >> 4) & 0x3FFF) | (uint64_t)(lbo >> 4) << 16 | (uint64_t)(sbo >> 4) << 32 |
           (uint64_t)1 << 46 | (uint64_t)swizzle << 61;
}
// byte offset of 16-byte chunk q of row r in the 64-byte-swizzled x tile
__device__ __forceinline__ int sw64_off(int r, int q) { return r * 64 + ((q ^ ((r >> 1) & 3)) << 4); }

// v[j] of lane i -> in v[0] of lane c the sum over the lanes of v[c]
__device__ __forceinline__ float column_sums(float (&v)[32])
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const bool up = lane & off;
#pragma unroll
        for (int j = 0; j < off; ++j) {
            const float send = up ? v[j] : v[j + off], keep = up ? v[j + off] : v[j];
            v[j] = keep + __shfl_xor_sync(0xffffffffu, send, off);
        }
    }
    return v[0];
}

__global__ void __launch_bounds__(GR_THREADS, 1) mlp_grad_kernel(const float *feats, const float *labels, long long R,
                                                                 float inv_b, const float *theta,
                                                                 const uint8_t *wpack, float *part, int vec, int *err)
{
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    __shared__ __align__(8) uint64_t bars[GR_G];
    __shared__ uint32_t tmem_base;
    __shared__ __align__(16) float b1[NH], w3[NH];
    const int gi = threadIdx.x >> 7, tid = threadIdx.x & 127, warp = threadIdx.x >> 5, lane = tid & 31;
    const long long ntiles = (R + T_ROWS - 1) / T_ROWS;
    const long long ng = ntiles < (long long)gridDim.x * GR_G ? ntiles : (long long)gridDim.x * GR_G;
    const long long id = (long long)gi * gridDim.x + blockIdx.x;    // parts 0 .. ng - 1 are written
    const long long tb = id < ng ? ntiles * id / ng : 0, te = id < ng ? ntiles * (id + 1) / ng : 0;
    const uint8_t *sW1 = smem, *sW2 = smem + W1_TILE, *sW2T = sW2 + 2 * W2_TILE;
    uint8_t *sX = smem + W1_TILE + 4 * W2_TILE + gi * GR_GROUP, *sH = sX + GR_X, *sD = sH + 2 * W2_TILE;
    uint64_t *bar = &bars[gi];
    if (threadIdx.x == 0) {
        for (int w = 0; w < GR_G; ++w) mbar_init(&bars[w], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int i = threadIdx.x; i < (W1_TILE + 4 * W2_TILE) / 16; i += GR_THREADS)
        ((uint4 *)smem)[i] = ((const uint4 *)wpack)[i];
    for (int i = threadIdx.x; i < NH; i += GR_THREADS) {
        b1[i] = theta[OFF_B1 + i];
        w3[i] = theta[OFF_W3 + i];
    }
    *(uint4 *)(sX + sw64_off(tid, 2)) = make_uint4(0x3f803f80u, 0x00003f80u, 0u, 0u);
    *(uint4 *)(sX + sw64_off(tid, 3)) = make_uint4(0u, 0u, 0u, 0u);
    const float b3 = theta[OFF_B3];
    if (warp == 0) tc_alloc(&tmem_base, 512);
    fence_proxy_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t d = tmem_base + (uint32_t)(gi * 256), dW2 = d + 128;
    const uint32_t lanes = (uint32_t)((warp & 3) * 32) << 16;
    constexpr uint32_t idesc = idesc_bf16_f32(128, 128);
    constexpr uint32_t idesc_t = idesc | (1u << 15) | (1u << 16);                // both operands MN-major
    constexpr uint32_t idesc_x = idesc_bf16_f32(128, 32) | (1u << 15) | (1u << 16);
    unsigned phase = 0;
    bool ok = true;
    auto wait = [&]() {
        ok = ok && mbar_wait(bar, phase);
        phase ^= 1u;
        tc_fence_after();
    };
    // operand tiles written (or accumulators read) by every thread of the group: on to the products
    auto meet = [&]() {
        tc_fence_before();
        fence_proxy_async_smem();
        group_sync<128>(gi);
    };
    float gW1[NF], gb1 = 0.f, gb3 = 0.f, gw3[4] = {0.f, 0.f, 0.f, 0.f}, gb2[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int i = 0; i < NF; ++i) gW1[i] = 0.f;
    double lsum = 0.0;
    float f[NF], y = 0.f;
    if (tb < te) {
        const long long row = tb * T_ROWS + tid;
        load_features(feats, row, row < R, vec, f);
        y = row < R ? labels[row] : 0.f;
    }
    for (long long t = tb; t < te; ++t) {
        const long long row = t * T_ROWS + tid;
        const bool valid = row < R;
        // layer 1
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            uint32_t w[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                __nv_bfloat162 h = __floats2bfloat162_rn(f[8 * q + 2 * k], f[8 * q + 2 * k + 1]);
                w[k] = *(uint32_t *)&h;
            }
            *(uint4 *)(sX + sw64_off(tid, q)) = make_uint4(w[0], w[1], w[2], w[3]);
        }
        meet();
        if (tid == 0) {
            tc_fence_after();
            tc_mma(d, smem_desc(sX, 16, 512, 4), sw128_desc(smem_u32(sW1)), idesc, 0u);
            tc_commit(bar);
        }
        __syncwarp();
        const float yr = y;
        if (t + 1 < te) {                                // the next tile's rows
            load_features(feats, row + T_ROWS, row + T_ROWS < R, vec, f);
            y = row + T_ROWS < R ? labels[row + T_ROWS] : 0.f;
        }
        wait();
        uint32_t mask[4];
        epilogue_h1<true>(d + lanes, sH, tid, b1, mask, nullptr);
        meet();
        // layer 2
        if (tid == 0) {
            tc_fence_after();
            tc_mma(d, smem_desc(sX, 16, 512, 4) + 2, sw128_desc(smem_u32(sW1)) + 2, idesc, 0u);   // 1 1 1 with b2's parts
            const uint64_t a = sw128_desc(smem_u32(sH)), b = sw128_desc(smem_u32(sW2));
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const uint64_t o = (uint64_t)(((k >> 2) * W2_TILE + (k & 3) * 32) >> 4);
                tc_mma(d, a + o, b + o, idesc, 1u);
            }
            tc_commit(bar);
        }
        __syncwarp();
        wait();
        const float s = b3 + epilogue_score(d + lanes, w3, nullptr);
        float ds = 0.f;
        if (valid) {
            ds = (1.f / (1.f + __expf(-s)) - yr) * inv_b;
            lsum += (double)(fmaxf(s, 0.f) + log1pf(__expf(-fabsf(s))) - yr * s);
        }
        gb3 += ds;
        // da2 into its tile, the column sums of ds h2 and of the BF16 da2
#pragma unroll
        for (int c0 = 0; c0 < NH; c0 += 32) {
            uint32_t v[32];
            tc_ld_32cols_async(d + lanes + (uint32_t)c0, v);
            tc_ld_wait(v);
            float a[32], b[32];
#pragma unroll
            for (int c = 0; c < 32; c += 8) {
                uint32_t w[4];
#pragma unroll
                for (int k = 0; k < 8; k += 2) {
                    const float2 w2 = *(const float2 *)(w3 + c0 + c + k);
                    const float h0 = fmaxf(__uint_as_float(v[c + k]), 0.f), h1 = fmaxf(__uint_as_float(v[c + k + 1]), 0.f);
                    a[c + k] = ds * h0;
                    a[c + k + 1] = ds * h1;
                    const __nv_bfloat162 g = __floats2bfloat162_rn(h0 > 0.f ? ds * w2.x : 0.f, h1 > 0.f ? ds * w2.y : 0.f);
                    const float2 gf = __bfloat1622float2(g);
                    b[c + k] = gf.x;
                    b[c + k + 1] = gf.y;
                    w[k >> 1] = *(const uint32_t *)&g;
                }
                *(uint4 *)(sD + ((c0 + c) >> 6) * W2_TILE + sw128_off(tid, (c0 + c) & 63)) =
                    make_uint4(w[0], w[1], w[2], w[3]);
            }
            gw3[c0 >> 5] += column_sums(a);
            gb2[c0 >> 5] += column_sums(b);
        }
        meet();
        // dL/dh1 = da2 W2 and dW2 += da2^T h1
        if (tid == 0) {
            tc_fence_after();
            const uint64_t a = sw128_desc(smem_u32(sD)), b = sw128_desc(smem_u32(sW2T));
            const uint64_t at = smem_desc(sD, W2_TILE, 1024, 2), bt = smem_desc(sH, W2_TILE, 1024, 2);
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const uint64_t o = (uint64_t)(((k >> 2) * W2_TILE + (k & 3) * 32) >> 4);
                tc_mma(d, a + o, b + o, idesc, k ? 1u : 0u);
                tc_mma(dW2, at + (uint64_t)(k * 2048 >> 4), bt + (uint64_t)(k * 2048 >> 4), idesc_t,
                       t > tb || k ? 1u : 0u);
            }
            tc_commit(bar);
        }
        __syncwarp();
        wait();
        // da1 over da2's tile
        tmem_columns(d + lanes, [&](int c0, const uint32_t (&v)[32]) {
            const uint32_t m = mask[c0 >> 5];
#pragma unroll
            for (int c = 0; c < 32; c += 8) {
                uint32_t w[4];
#pragma unroll
                for (int k = 0; k < 8; k += 2) {
                    const __nv_bfloat162 g =
                        __floats2bfloat162_rn((m >> (c + k)) & 1u ? __uint_as_float(v[c + k]) : 0.f,
                                              (m >> (c + k + 1)) & 1u ? __uint_as_float(v[c + k + 1]) : 0.f);
                    w[k >> 1] = *(const uint32_t *)&g;
                }
                *(uint4 *)(sD + ((c0 + c) >> 6) * W2_TILE + sw128_off(tid, (c0 + c) & 63)) =
                    make_uint4(w[0], w[1], w[2], w[3]);
            }
        });
        meet();
        if (tid == 0) {
            tc_fence_after();
            const uint64_t at = smem_desc(sD, W2_TILE, 1024, 2), bt = smem_desc(sX, 16, 512, 4);
#pragma unroll
            for (int k = 0; k < 8; ++k)
                tc_mma(d, at + (uint64_t)(k * 2048 >> 4), bt + (uint64_t)(k * 1024 >> 4), idesc_x, k ? 1u : 0u);
            tc_commit(bar);
        }
        __syncwarp();
        wait();
        // dW1 and db1 of unit i = this lane
        {
            uint32_t v[32];
            tc_ld_32cols_async(d + lanes, v);
            tc_ld_wait(v);
#pragma unroll
            for (int i = 0; i < NF; ++i) gW1[i] += __uint_as_float(v[i]);
            gb1 += __uint_as_float(v[NF]);
        }
        tc_fence_before();
    }
    // this group's part; the sums over its four warps meet in shared memory (sX is free)
    if (tb < te) {
        float *p = part + id * GR_PART;
        tmem_columns(dW2 + lanes, [&](int c0, const uint32_t (&v)[32]) {
#pragma unroll
            for (int c = 0; c < 32; c += 4)
                *(uint4 *)(p + OFF_W2 + tid * NH + c0 + c) = make_uint4(v[c], v[c + 1], v[c + 2], v[c + 3]);
        });
#pragma unroll
        for (int i = 0; i < NF; i += 4)
            *(float4 *)(p + OFF_W1 + tid * NF + i) = make_float4(gW1[i], gW1[i + 1], gW1[i + 2], gW1[i + 3]);
        p[OFF_B1 + tid] = gb1;
        float *sum = (float *)sX;                        // 4 warps x (128 db2, 128 dw3), then 4 db3
        double *lsm = (double *)(sX + 6144);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            sum[(warp & 3) * 256 + k * 32 + lane] = gb2[k];
            sum[(warp & 3) * 256 + 128 + k * 32 + lane] = gw3[k];
        }
        for (int off = 16; off > 0; off >>= 1) {
            gb3 += __shfl_xor_sync(0xffffffffu, gb3, off);
            lsum += __shfl_xor_sync(0xffffffffu, lsum, off);
        }
        if (lane == 0) {
            sum[1024 + (warp & 3)] = gb3;
            lsm[warp & 3] = lsum;
        }
        group_sync<128>(gi);
        p[OFF_B2 + tid] = (sum[tid] + sum[256 + tid]) + (sum[512 + tid] + sum[768 + tid]);
        p[OFF_W3 + tid] = (sum[128 + tid] + sum[384 + tid]) + (sum[640 + tid] + sum[896 + tid]);
        if (tid == 0) {
            p[OFF_B3] = (sum[1024] + sum[1025]) + (sum[1026] + sum[1027]);
            *(double *)(p + GR_PART - 4) = (lsm[0] + lsm[1]) + (lsm[2] + lsm[3]);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tc_dealloc(tmem_base, 512);
    if (!ok && tid == 0) atomicExch(err, 7);             // a bounded wait expired
}

// grad = the sum of the groups' parts (and *loss += theirs), in a fixed order: 64 parameters
// per CTA, 4 threads a parameter
__global__ void __launch_bounds__(256) mlp_reduce_kernel(const float *part, int ng, float *grad, double *loss)
{
    __shared__ float sum[4][64];
    const int c = threadIdx.x & 63, q = threadIdx.x >> 6, i = blockIdx.x * 64 + c;
    float s = 0.f;
    if (i < NPARAM) {
#pragma unroll 8
        for (int g = q; g < ng; g += 4) s += __ldg(part + (size_t)g * GR_PART + i);
    }
    sum[q][c] = s;
    __syncthreads();
    if (q == 0 && i < NPARAM) grad[i] = (sum[0][c] + sum[1][c]) + (sum[2][c] + sum[3][c]);
    if (loss && blockIdx.x == 0 && threadIdx.x == 0) {
        double l = 0.0;
        for (int g = 0; g < ng; ++g) l += *(const double *)(part + (size_t)g * GR_PART + GR_PART - 4);
        *loss += l;
    }
}

// Adam (Kingma & Ba): m = b1 m + (1-b1) g, v = b2 v + (1-b2) g^2,
// theta -= lr * mhat / (sqrt(vhat) + eps).
__global__ void adam_kernel(float *theta, const float *grad, float *m, float *v, int n, float lr, float bc1,
                            float bc2)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float g = grad[i];
    const float mi = 0.9f * m[i] + 0.1f * g, vi = 0.999f * v[i] + 0.001f * g * g;
    m[i] = mi;
    v[i] = vi;
    theta[i] -= lr * (mi / bc1) / (sqrtf(vi / bc2) + 1e-8f);
}

// Per ordered pair (u, j) of a node with scored candidates: the permutation of
// its d candidate positions in descending score (ties: ascending position), as
// indices into nbr[u].  One warp per pair (its node from the stage's owner
// table): each lane holds the scores of positions lane, lane + 32, ... and
// counts, for each of them, the larger scores broadcast from the other lanes.
__global__ void perm_kernel(GraphDev g, const unsigned long long *row_off, const float *scores, short *perm)
{
    if (g.info->done || g.info->halt) return;
    if (row_off[g.p] == 0) return;                     // this stage runs in plain order
    const long long npairs = g.info->n_opairs;
    const int lane = threadIdx.x & 31;
    for (long long o = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5; o < npairs;
         o += ((long long)gridDim.x * blockDim.x) >> 5) {
        const int u = g.opu[o];
        if (row_off[u + 1] == row_off[u]) continue;
        const int j = (int)(o - g.ooff[u]);
        const int d = g.deg[u] - 1;
        const long long base = (long long)row_off[u] + (long long)j * d;
        for (int x0 = 0; x0 < d; x0 += 32) {
            const int x = x0 + lane;
            const float sx = x < d ? scores[base + x] : 0.f;
            int rank = 0;
            for (int y0 = 0; y0 < d; y0 += 32) {
                const float sl = y0 + lane < d ? scores[base + y0 + lane] : 0.f;
                const int ny = d - y0 < 32 ? d - y0 : 32;
                for (int t = 0; t < ny; ++t) {
                    const float sy = __shfl_sync(0xffffffffu, sl, t);
                    const int y = y0 + t;
                    rank += (sy > sx) || (sy == sx && y < x);
                }
            }
            if (x < d) perm[base + rank] = (short)(x + (x >= j));   // index into nbr[u]
        }
    }
}

// ---------------------------------------------------------------- host side
int mlp_nparam() { return NPARAM; }
size_t mlp_pack_bytes() { return (size_t)W1_TILE + 4 * W2_TILE; }

cudaError_t launch_mlp_pack(const float *theta, uint8_t *wpack, cudaStream_t s)
{
    mlp_pack_kernel<<<NH, 64, 0, s>>>(theta, wpack);
    note_launch();
    return cudaGetLastError();
}

static int mlp_ctas(long long rows)
{
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    long long tiles = (rows + T_ROWS - 1) / T_ROWS;
    long long c = tiles < (long long)sms ? tiles : (long long)sms;
    return (int)(c < 1 ? 1 : c);
}

cudaError_t launch_mlp_forward_feats(const float *feats, long long R, const uint8_t *wpack, const float *theta,
                                     float *scores, __nv_bfloat16 *h1, float *h2, int *err, GraphDev g,
                                     cudaStream_t s)
{
    MlpRows rows{};
    rows.feats = feats;
    rows.R = R;
    cudaError_t e = cudaFuncSetAttribute(mlp_forward_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, FW_SMEM);
    if (e != cudaSuccess) return e;
    mlp_forward_kernel<<<mlp_ctas(R), FW_THREADS, FW_SMEM, s>>>(rows, g, wpack, theta, scores, h1, h2,
                                                               ((uintptr_t)feats & 15) == 0, err);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_mlp_score_stage(GraphDev g, const unsigned long long *row_off, long long rows_cap,
                                   const float *C32, int ldc, float sqn_over_q, float inv_q, const uint8_t *wpack,
                                   const float *theta, float *scores, short *perm, int *err, cudaStream_t s)
{
    MlpRows rows{};
    rows.feats = nullptr;
    rows.row_off = row_off;
    rows.C32 = C32;
    rows.ldc = ldc;
    rows.sqn_over_q = sqn_over_q;
    rows.nvec = g.nvec;
    rows.inv_q = inv_q;
    cudaError_t e = cudaFuncSetAttribute(mlp_forward_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, FW_SMEM);
    if (e != cudaSuccess) return e;
    mlp_forward_kernel<<<mlp_ctas(rows_cap), FW_THREADS, FW_SMEM, s>>>(rows, g, wpack, theta, scores, nullptr, nullptr,
                                                                      0, err);
    note_launch();
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    perm_kernel<<<sms * 4, 256, 0, s>>>(g, row_off, scores, perm);
    note_launch();
    return cudaGetLastError();
}

size_t mlp_grad_ws_bytes() { return (size_t)mlp_ctas(1ll << 40) * GR_G * GR_PART * sizeof(float); }

cudaError_t launch_mlp_grad(const float *feats, const float *labels, long long R, float inv_b, const float *theta,
                            const uint8_t *wpack, float *ws, float *grad, double *loss, int *err, cudaStream_t s)
{
    cudaError_t e = cudaFuncSetAttribute(mlp_grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, GR_SMEM);
    if (e != cudaSuccess) return e;
    const int ctas = mlp_ctas(R);
    const long long tiles = (R + T_ROWS - 1) / T_ROWS;
    const int ng = (int)std::min<long long>(tiles, (long long)ctas * GR_G);
    mlp_grad_kernel<<<ctas, GR_THREADS, GR_SMEM, s>>>(feats, labels, R, inv_b, theta, wpack, ws,
                                                      ((uintptr_t)feats & 15) == 0, err);
    note_launch();
    mlp_reduce_kernel<<<(NPARAM + 63) / 64, 256, 0, s>>>(ws, ng, grad, loss);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_mlp_backward(const float *feats, const float *labels, const float *scores,
                                const __nv_bfloat16 *h1, const float *h2, long long R, float inv_b,
                                const float *theta, float *grad, double *loss, cudaStream_t s)
{
    cudaError_t e = cudaMemsetAsync(grad, 0, NPARAM * sizeof(float), s);
    if (e != cudaSuccess) return e;
    const size_t smem = (size_t)(2 * T_ROWS * (NH + 1) + NH * (NH + 1) + T_ROWS * NF + T_ROWS) * sizeof(float);
    e = cudaFuncSetAttribute(mlp_backward_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    mlp_backward_kernel<<<mlp_ctas(R), 256, smem, s>>>(feats, labels, scores, h1, h2, R, inv_b, theta, grad, loss);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_adam(float *theta, const float *grad, float *m, float *v, float lr, int step, cudaStream_t s)
{
    const float bc1 = 1.f - powf(0.9f, (float)step), bc2 = 1.f - powf(0.999f, (float)step);
    adam_kernel<<<(NPARAM + 255) / 256, 256, 0, s>>>(theta, grad, m, v, NPARAM, lr, bc1, bc2);
    note_launch();
    return cudaGetLastError();
}

// Member features for explicit quadruples (u, v, k, l | d << 16): candidate k
// of the ordered pair (u, v) at stage l with candidate-set size d.
__global__ void mlp_features_kernel(const int *quads, long long R, const float *C32, int ldc, const long long *prow,
                                    int p, long long n, const long long *nvec, float inv_q, float *feats, int *err)
{
    const long long r = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (r >= R) return;
    const int u = quads[4 * r], v = quads[4 * r + 1], k = quads[4 * r + 2];
    const int l = quads[4 * r + 3] & 0xffff, d = (int)((unsigned)quads[4 * r + 3] >> 16);
    if (u < 0 || u >= p || v < 0 || v >= p || k < 0 || k >= p || u == v || k == u || k == v) {
        *err = 1;
        return;
    }
    float f[NF];
    member_features(C32, ldc, prow, u, v, k, l, d, sqrtf((float)(nvec ? nvec[u] : n)) * inv_q, f);
    for (int i = 0; i < NF; ++i) feats[r * NF + i] = f[i];
}

cudaError_t launch_mlp_features(const int *quads, long long R, const float *C32, int ldc, const long long *prow,
                                int p, long long n, const long long *nvec, double q, float *feats, int *err,
                                cudaStream_t s)
{
    mlp_features_kernel<<<(unsigned)((R + 255) / 256), 256, 0, s>>>(quads, R, C32, ldc, prow, p, n, nvec,
                                                                      (float)(1.0 / q), feats, err);
    note_launch();
    return cudaGetLastError();
}

}  // namespace fpc
