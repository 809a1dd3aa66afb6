// ci_test.cuh -- one CI test on the GPU: the warp-per-test evaluation in FP32 under
// the trust rule and in FP64, the FP64 correlations formed on demand, and the
// predicates the stage kernels share (level.cu, node_loop.cu).
#pragma once
#include "internal.h"
#include "device_util.cuh"

namespace fpc {

typedef unsigned long long ull;

__device__ __forceinline__ ull sat_add(ull a, ull b)
{
    ull c = a + b;
    return c < a ? KEY_NONE : c;
}

// samples behind the tests of node u (batched problems: its instance's n)
__device__ __forceinline__ long long n_of(const TestParams &tp, int u)
{
    return tp.nvec ? __ldg(tp.nvec + u) : tp.n;
}

// node u has tests at stage l only while n_u - l - 3 > 0 (one problem: the
// stage cap n - 4 already ensures it; batched problems differ in n)
__device__ __forceinline__ bool dof_ok(const TestParams &tp, int u, int l)
{
    return !tp.nvec || n_of(tp, u) - l - 3 > 0;
}

// the stage loop has finished or has been halted: nothing to do
__device__ __forceinline__ bool stopped(const LevelInfo *I) { return I->done || I->halt; }

__device__ __forceinline__ bool comp_eligible(int d, int l, const TestParams &tp)
{
    const int k = d - l;
    return tp.reversed && tp.complement && d >= l && k <= KC_MAX && k < l && d + 2 <= PREC_MAX;
}

// ---------------------------------------------------------------- warp test
// Cholesky of the leading l x l block of the (l+2) x (l+2) lower triangle M
// (row stride ms; order S..., u, v).  Lanes own rows.  After l steps the
// trailing 2x2 holds H = H0 - H1 H2^{-1} H1^T (Sec. 4).  pmin is the smallest
// of the l pivots (conditional variances of S_k given S_1..S_{k-1}), h11, h22.
// bad: a pivot, h11 or h22 <= DEGEN (the FP64 degeneracy rule) or not finite.
template <typename T>
__device__ __forceinline__ void warp_chol_test(T *M, int m, int ms, int l, T &r, T &pmin, bool &bad)
{
    const int lane = threadIdx.x & 31;
    pmin = (T)1e30;
    bad = false;
    for (int k = 0; k < l; ++k) {
        const T piv = M[k * ms + k];
        pmin = piv < pmin ? piv : pmin;
        if (!(piv > (T)DEGEN)) {
            bad = true;
            break;
        }
        const T rl = (T)1 / sqrt(piv);
        for (int i = k + 1 + lane; i < m; i += 32) M[i * ms + k] *= rl;
        __syncwarp();
        for (int i = k + 1 + lane; i < m; i += 32) {
            const T lik = M[i * ms + k];
            for (int c = k + 1; c <= i; ++c) M[i * ms + c] -= lik * M[c * ms + k];
        }
        __syncwarp();
    }
    if (bad) {
        r = (T)0;
        return;
    }
    const T h11 = M[l * ms + l], h22 = M[(l + 1) * ms + l + 1], h12 = M[(l + 1) * ms + l];
    pmin = h11 < pmin ? h11 : pmin;
    pmin = h22 < pmin ? h22 : pmin;
    if (!(h11 > (T)DEGEN) || !(h22 > (T)DEGEN)) {
        bad = true;
        r = (T)0;
        return;
    }
    r = h12 / sqrt(h11 * h22);
}

// warp_chol_test in FP32 for m <= MX <= 32: a lane holds its row in registers and the column of
// the step reaches it by shuffles, instead of chains of shared-memory loads and stores (the same
// operations in the same order, the factor left in M).  Stage 13 of the 1000-node sparse
// graph: 335 us through shared memory, 233 so (127 registers, half the warps in flight).
template <int MX>
__device__ __forceinline__ void warp_chol_reg(float *M, int m, int ms, int l, float &r, float &pmin, bool &bad)
{
    const int lane = threadIdx.x & 31;
    float a[MX];
#pragma unroll
    for (int c = 0; c < MX; ++c) a[c] = lane < m && c <= lane ? M[lane * ms + c] : 0.f;
    pmin = 1e30f;
    bad = false;
#pragma unroll
    for (int k = 0; k < MX - 2; ++k) {
        if (k >= l || bad) continue;                     // the same in all lanes
        const float piv = __shfl_sync(0xffffffffu, a[k], k);
        pmin = piv < pmin ? piv : pmin;
        if (!(piv > (float)DEGEN)) {
            bad = true;
            continue;
        }
        const float rl = 1.0f / sqrtf(piv), lik = a[k] * rl;
        if (lane > k) a[k] = lik;
#pragma unroll
        for (int c = k + 1; c < MX; ++c) a[c] = fmaf(-lik, __shfl_sync(0xffffffffu, lik, c), a[c]);
    }
    float h11 = 0.f, h12 = 0.f, h22 = 0.f;
#pragma unroll
    for (int c = 0; c < MX - 1; ++c)
        if (c == l) {
            h11 = __shfl_sync(0xffffffffu, a[c], c);
            h12 = __shfl_sync(0xffffffffu, a[c], c + 1);
            h22 = __shfl_sync(0xffffffffu, a[c + 1], c + 1);
        }
#pragma unroll
    for (int c = 0; c < MX; ++c)
        if (lane < m && c <= lane) M[lane * ms + c] = a[c];
    __syncwarp();
    r = 0.f;
    if (bad) return;
    pmin = h11 < pmin ? h11 : pmin;
    pmin = h22 < pmin ? h22 : pmin;
    if (!(h11 > (float)DEGEN) || !(h22 > (float)DEGEN)) {
        bad = true;
        return;
    }
    r = h12 / sqrtf(h11 * h22);
}

struct WarpAcc {
    ull tests, red, band, guard, degen, fl32, fl64;
    float maxdz;
};

__device__ __forceinline__ ull flops_direct(int l)
{
    ull L = (ull)l;
    return (L * L * L) / 3 + 2 * L * L + 6 * L + 10;
}

// Fills the FP64 correlations the lower triangle of corr[nd, nd] needs (lazy
// mode): every missing entry is computed once by a whole warp -- lane t sums
// samples t, t+32, ... in order, a fixed butterfly adds the lanes -- and
// published with a fence before its flag, so racing warps write equal values.
static __device__ __noinline__ void ensure_c64(const int *nd, int m, const TestParams &tp, double *C64, int ldc)
{
    const int lane = threadIdx.x & 31;
    const int ne = m * (m + 1) / 2;
    volatile unsigned char *valid = tp.c64_valid;
    for (int e0 = 0; e0 < ne; e0 += 32) {
        const int e = e0 + lane;
        bool miss = false;
        int a = 0, b = 0;
        if (e < ne) {
            int i = (int)((sqrtf(8.f * (float)e + 1.f) - 1.f) * 0.5f);
            while (i * (i + 1) / 2 > e) --i;
            while ((i + 1) * (i + 2) / 2 <= e) ++i;
            const int c = e - i * (i + 1) / 2;
            a = nd[i];
            b = nd[c];
            miss = a != b && valid[cidx(tp.prow, tp.p, a, b)] != 1;
        }
        unsigned bal = __ballot_sync(0xffffffffu, miss);
        while (bal) {
            const int src = __ffs(bal) - 1;
            const int aa = __shfl_sync(0xffffffffu, a, src), bb = __shfl_sync(0xffffffffu, b, src);
            const double *xa = tp.xs64 + (long long)aa * tp.ldk, *xb = tp.xs64 + (long long)bb * tp.ldk;
            const long long na = n_of(tp, aa);
            // rows start 512-byte aligned (ldk is a multiple of 64): 16-byte loads,
            // four independent FMA chains per lane
            const double2 *xa2 = (const double2 *)xa, *xb2 = (const double2 *)xb;
            const long long nh = na >> 1;
            double acc0 = 0.0, acc1 = 0.0, acc2 = 0.0, acc3 = 0.0;
            long long t = lane;
            for (; t + 32 < nh; t += 64) {
                const double2 a0 = __ldg(xa2 + t), b0 = __ldg(xb2 + t);
                const double2 a1 = __ldg(xa2 + t + 32), b1 = __ldg(xb2 + t + 32);
                acc0 = fma(a0.x, b0.x, acc0);
                acc1 = fma(a0.y, b0.y, acc1);
                acc2 = fma(a1.x, b1.x, acc2);
                acc3 = fma(a1.y, b1.y, acc3);
            }
            if (t < nh) {
                const double2 a0 = __ldg(xa2 + t), b0 = __ldg(xb2 + t);
                acc0 = fma(a0.x, b0.x, acc0);
                acc1 = fma(a0.y, b0.y, acc1);
            }
            if ((na & 1) && lane == 0) acc0 = fma(xa[na - 1], xb[na - 1], acc0);
            double acc = (acc0 + acc1) + (acc2 + acc3);
            for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
            if (lane == 0) {
                const double v = acc / (double)na;
                C64[cidx(tp.prow, ldc, aa, bb)] = v;
                C64[cidx(tp.prow, ldc, bb, aa)] = v;
                __threadfence();
                valid[cidx(tp.prow, tp.p, aa, bb)] = 1;
                valid[cidx(tp.prow, tp.p, bb, aa)] = 1;
            }
            bal &= bal - 1;
        }
        __syncwarp();
    }
    __threadfence_block();
    __syncwarp();
}

// ---------------------------------------------------------------- FP32 trust rule
// The FP32 trailing block (h11, h12, h22) of a test is the exact Schur
// complement of corr + E, where E holds the correlation step's entry errors
// (|E_ij| <= eps_c) and the backward error of the FP32 factorisation (every
// row of the Cholesky factor of a correlation matrix has unit norm, so each
// entry of that backward error is below a few m eps32; 4 m eps32 is taken).
// With b_u = corr_SS^{-1} corr_Su and b_v the regression coefficients of u
// and v on S, to first order in eps = eps_c + 4 m eps32
//   |dh12| <= eps A_u A_v,  |dh11| <= eps A_u^2,  |dh22| <= eps A_v^2,
//   A_u = 1 + |b_u|_1,  A_v = 1 + |b_v|_1,
// hence |dr| <= eps (A_u A_v / sqrt(h11 h22) + |r|/2 (A_u^2/h11 + A_v^2/h22)).
// The expansion is used only while eps A_u^2/h11, eps A_v^2/h22 and
// m eps |corr_SS^{-1}| (kap) stay below 0.05, and the bound is doubled to
// cover the higher-order terms and the rounding of the final ratio.  A test
// is trusted when |r| clears the threshold r_q = tanh(q / sqrt(n-l-3)) by
// more than that bound (then the FP64 decision of Eq. 1 is the same) and the
// statistic lies at least `band` from q; otherwise it is re-decided in FP64.
// Returns 0 trusted, 1 band (re-decide), 2 guard (re-decide); dr_out: the bound.
constexpr float EPS32 = 5.96e-8f;

__device__ __forceinline__ int fp32_trust(const TestParams &tp, int m, float sqf, float rq, float a, float h11,
                                          float h22, float ih, float Au, float Av, float kap, float &dr_out)
{
    const float eps = tp.eps_c + (4.0f * (float)m) * EPS32;
    const float i11 = __frcp_rn(h11), i22 = __frcp_rn(h22);
    const float qu = eps * Au * Au * i11, qv = eps * Av * Av * i22;
    dr_out = INFINITY;
    if (fmaxf(fmaxf(qu, qv), kap) > 0.05f) return 2;
    const float dr = 2.0f * eps * (Au * Av * ih + 0.5f * a * (Au * Au * i11 + Av * Av * i22)) + 8.0f * EPS32;
    dr_out = dr;
    if (dr > tp.dr_max) return 2;
    // |z - q| >= sqf |a - rq| / (1 - min(a, rq)^2) (mean-value theorem on atanh)
    const float gap = fabsf(a - rq), mn = fminf(a, rq);
    if (gap <= dr || sqf * gap < tp.band_f * (1.0f - mn * mn)) return 1;
    return 0;
}

// l1 norms of the regression coefficients b_u = corr_SS^{-1} corr_Su and b_v
// from the factor warp_chol_test left in M (column k below the diagonal holds
// L_ik, the diagonal the pivots L_kk^2, rows l and l+1 hold L^{-1} corr_Su and
// L^{-1} corr_Sv): back substitution L^T b = y by the warp, column by column.
// Overwrites the first l entries of rows l and l+1.
__device__ __forceinline__ void warp_beta_l1(float *M, int ms, int l, float &bu, float &bv)
{
    const int lane = threadIdx.x & 31;
    float *yu = M + (long long)l * ms, *yv = M + (long long)(l + 1) * ms;
    float su = 0.f, sv = 0.f;
    for (int k = l - 1; k >= 0; --k) {
        __syncwarp();
        const float rl = rsqrtf(M[k * ms + k]);
        const float b_u = yu[k] * rl, b_v = yv[k] * rl;
        su += fabsf(b_u);
        sv += fabsf(b_v);
        for (int j = lane; j < k; j += 32) {
            const float lkj = M[k * ms + j];
            yu[j] -= lkj * b_u;
            yv[j] -= lkj * b_v;
        }
    }
    __syncwarp();
    bu = su;
    bv = sv;
}

// One CI test for node ids nd[0..m) (S..., u, v) by the calling warp.
// Returns independent; writes r and z (of the path that decided).
template <bool F64>
__device__ __forceinline__ bool warp_test(const int *nd, int m, int l, const float *C32,
                                          const double *C64, int ldc, const TestParams &tp,
                                          double sq, float sqf, void *Mbuf, int ms, WarpAcc &acc,
                                          double &r_out, float &z_out)
{
    const int lane = threadIdx.x & 31;
    bool need64 = F64, indep = false;
    float zf = 0.f, rf = 0.f;
    bool f32ok = false;
    if (!F64) {
        float *M = (float *)Mbuf;
        for (int i = 0; i < m; ++i)
            for (int c = lane; c <= i; c += 32) M[i * ms + c] = C32[cidx(tp.prow, ldc, nd[i], nd[c])];
        __syncwarp();
        float pmin;
        bool bad;
        if (m <= 16) warp_chol_reg<16>(M, m, ms, l, rf, pmin, bad);
        else if (m <= 24) warp_chol_reg<24>(M, m, ms, l, rf, pmin, bad);
        else warp_chol_test<float>(M, m, ms, l, rf, pmin, bad);
        __syncwarp();
        acc.fl32 += flops_direct(l);
        if (bad || pmin < (float)tp.guard) {
            need64 = true;
            ++acc.guard;
        } else {
            const float h11 = M[l * ms + l], h22 = M[(l + 1) * ms + l + 1];
            float bu, bv, dr;
            warp_beta_l1(M, ms, l, bu, bv);
            const float ih = rsqrtf(h11 * h22);
            const float a = fabsf(rf);
            const float rq = tanhf(tp.qf / sqf);
            // kap is not formed here (it would need corr_SS^{-1}); the pivot guard
            // and the two first-order ratios bound the expansion instead
            const int t = fp32_trust(tp, m, sqf, rq, a, h11, h22, ih, 1.0f + bu, 1.0f + bv, 0.0f, dr);
            zf = a < 1.0f ? sqf * atanhf(a) : INFINITY;
            if (t == 2) {
                need64 = true;
                ++acc.guard;
            } else if (t == 1) {
                need64 = true;
                ++acc.band;
            } else {
                indep = a <= rq;
                f32ok = true;
            }
        }
    }
    double r = rf;
    float z = zf;
    if (need64) {
        double *M = (double *)Mbuf;
        if (tp.lazy) ensure_c64(nd, m, tp, (double *)C64, ldc);
        for (int i = 0; i < m; ++i)
            for (int c = lane; c <= i; c += 32) {
                const long long o = cidx(tp.prow, ldc, nd[i], nd[c]);
                M[i * ms + c] = tp.lazy ? ((volatile const double *)C64)[o] : C64[o];
            }
        __syncwarp();
        double pmin;
        bool bad;
        warp_chol_test<double>(M, m, ms, l, r, pmin, bad);
        __syncwarp();
        acc.fl64 += flops_direct(l);
        if (bad) {
            indep = true;
            r = 0.0;
            z = 0.f;
            ++acc.degen;
        } else {
            double z64 = fabs(r) < 1.0 ? sq * fabs(atanh(r)) : INFINITY;
            indep = z64 <= tp.q;
            if (!F64 && isfinite(zf) && zf > 0.f) acc.maxdz = fmaxf(acc.maxdz, (float)fabs(zf - z64));
            z = (float)z64;
        }
        if (!F64) ++acc.red;
    }
    (void)f32ok;
    r_out = r;
    z_out = z;
    return indep;
}

__device__ __forceinline__ void flush_acc(const WarpAcc &acc, DevCounters *ctr)
{
    if (acc.tests) atomicAdd(&ctr->tests_executed, acc.tests);
    if (acc.red) atomicAdd(&ctr->redecided, acc.red);
    if (acc.band) atomicAdd(&ctr->band_hits, acc.band);
    if (acc.guard) atomicAdd(&ctr->guard_hits, acc.guard);
    if (acc.degen) atomicAdd(&ctr->degenerate, acc.degen);
    if (acc.fl32) atomicAdd(&ctr->flops, acc.fl32);
    if (acc.fl64) atomicAdd(&ctr->flops64_direct, acc.fl64);
    if (acc.maxdz > 0.f) atomic_max_float_pos(&ctr->max_dz_bits, acc.maxdz);
}

}  // namespace fpc
