// node_loop.cu -- the whole skeleton search of a small problem (p <= NL_PMAX) in one
// cooperative kernel, one CTA per node.
//
// What bounds such a search is latency: the reversed order (Algorithm 2) visits up to
// p stages of a few thousand tests each, one after the other.  A stage that passes its
// state through global memory (plan, tests, commit, degrees, block downdates, a grid
// barrier between each) spends its time on chains of L2 loads.  Here CTA u keeps what
// the tests and the deletions of node u need in its shared memory for the whole
// search:
//   * the neighbourhood precision block P = corr[F,F]^{-1}, F = adj(u) u {u} (FP64,
//     packed lower triangle, and its FP32 rounding for the FP32-first tests);
//   * the FP32 correlation matrix (the direct tests of any set in adj(u));
//   * the adjacency bitset of the whole graph, every degree and C(d, l).
// Each stage, CTA u runs every test of its ordered pairs (u, v) and publishes one
// word per 32 nodes: the v it found separated.  The words of all CTAs are the only
// thing exchanged (a 64-bit store of word and stage number, polled by the readers: data
// and barrier in one L2 round trip).  Every CTA then applies the same deletions to its
// copy of the graph, and so knows the next stage and its tests without a plan; CTA u
// drops the lost members from its own block by rank-1 updates in shared memory, and
// the CTA whose side separated a pair first records the separating set.
// A CTA without tests in the next stage publishes at once and does its block work
// (the build of its first block, the drops) while it waits.
//
// Measured (skeleton search alone, us, against one cooperative kernel whose stages went
// through global memory with three grid barriers, the closed-form stage and the captured
// loop's launch around it): p = 95 dense reversed 4578 -> 945 (79 stages, 9 us each, and
// about 190 us for the closed-form stage), p = 95 hub graph reversed 1777 -> 461, p = 55
// hub graph conventional 629 -> 281, p = 20 583 -> 137.  A stage is about 2.5 us of tests,
// 1.5 us of drops, 2-3 us of exchange (a store and a polled load through L2, and the
// slowest CTA) and 2 us of applying the deletions.
#include "internal.h"
#include "device_util.cuh"
#include "ci_test.cuh"

#include <algorithm>

namespace fpc {

namespace {

constexpr int NL_THREADS = 256;
constexpr int NL_W = NL_PMAX / 32;
constexpr int NL_BR = LANE_LMAX + 1;                     // columns of the binomial table: r = 0 .. 12
constexpr int NL_QCAP = 1024;                            // untrusted direct tests of one stage of one node
// a stage in which some node has more tests than this runs on the captured loop, whose
// kernels spread one node's tests over the GPU (64 tests per thread here)
constexpr uint32_t NL_TESTS_MAX = 64u * NL_THREADS;
constexpr uint32_t NL_SAT = 0xffffffffu;
constexpr uint32_t NL_NONE = 0xffffffffu;                // no separating set yet
constexpr uint32_t NL_EXIT = 0x80000000u;                // stage-number bit: this CTA cannot run the stage
constexpr long long NL_WAIT = 4000000000ll;              // bounded waits: about 2 s at 2 GHz
constexpr int NL_MMAX = LANE_LMAX + 2;
constexpr int NL_DIRECT_BYTES = (NL_MMAX * (NL_MMAX + 1) * 8 + NL_MMAX * 4 + 15) / 16 * 16;

enum { BLK_NONE = 0, BLK_OK = 1, BLK_BUILD = 2, BLK_SINGULAR = -1 };

struct NlShared {
    uint32_t A[NL_PMAX][NL_W];       // frozen graph of the stage
    uint32_t M[NL_PMAX][NL_W];       // the stage's separated pairs as each node's CTA found them
    uint32_t own[NL_W];              // this CTA's, while the tests run
    int deg[NL_PMAX];
    uint32_t T[NL_PMAX];             // C(deg - 1, l), saturating
    uint32_t bin[NL_PMAX * NL_BR];   // C(x, r), saturating
    uint32_t best[NL_PMAX];          // rank of the first separating set per neighbour
    short nbr[NL_PMAX];              // adj(u), ascending
    short nbr0[NL_PMAX];             // adj(u) of the stage whose separating sets are still to be recorded
    short nslot[NL_PMAX];            // their slots in the block
    short slot[NL_PMAX];             // node -> slot of the block (at its build)
    short snode[NL_PMAX];            // slot -> node
    short list[NL_PMAX + 1];         // live slots: kept members ascending, then members to drop
    double colk[NL_PMAX], cols[NL_PMAX], z[NL_PMAX];
    double rD;                       // reciprocal of the next pivot
    int bad;
    uint32_t queue[NL_QCAP];
    int qn;
    int red[16];
    int flag;
};

__device__ __forceinline__ int tri(int i, int j) { return i * (i + 1) / 2 + j; }          // i >= j
__device__ __forceinline__ int tri2(int i, int j) { return i >= j ? tri(i, j) : tri(j, i); }

// row of entry e of a packed lower triangle
__device__ __forceinline__ int tri_row(int e)
{
    int r = (int)((sqrtf(8.f * (float)e + 1.f) - 1.f) * 0.5f);
    if (tri(r, 0) > e) --r;
    else if (tri(r + 1, 0) <= e) ++r;
    return r;
}

// clocks of dropping a block's members from nl down to nt one by one (two barriers and
// n^2/2 FMAs at 2 per clock each), and of a sweep build of m members
__device__ __forceinline__ float drop_clocks(int nt, int nl)
{
    const float a = (float)nt, b = (float)nl;
    return 300.f * (b - a) + (b * b * b - a * a * a) * (1.f / 12.f);
}
__device__ __forceinline__ float build_clocks(int m)
{
    const float x = (float)m;
    return 1000.f + 300.f * x + 0.25f * x * x * x;
}

__device__ __forceinline__ uint32_t nl_binom(const NlShared &S, int x, int r)
{
    return r < NL_BR ? S.bin[x * NL_BR + r] : NL_SAT;
}

// C(d, l) through the smaller of l and d - l; saturated when both exceed the table
__device__ __forceinline__ uint32_t nl_sets(const NlShared &S, int d, int l)
{
    return d < l ? 0u : nl_binom(S, d, min(l, d - l));
}

// positions of the rank-th L-subset of d items in lexicographic order (see unrank_lex)
template <int L>
__device__ __forceinline__ void nl_unrank(const NlShared &S, uint32_t rank, int d, int (&pos)[L > 0 ? L : 1])
{
    int x = 0;
#pragma unroll
    for (int i = 0; i < L; ++i) {
        const int r1 = L - i;
        if (r1 == 1) {
            pos[i] = x + (int)rank;
            break;
        }
        const uint32_t base = S.bin[(d - x) * NL_BR + r1], target = base - rank;
        int lo = x, hi = d - r1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (S.bin[(d - mid) * NL_BR + r1] >= target) lo = mid;
            else hi = mid - 1;
        }
        pos[i] = lo;
        rank -= base - S.bin[(d - lo) * NL_BR + r1];
        x = lo + 1;
    }
}

struct NlAcc {
    unsigned tests, comp, band, guard, red, degen;
    ull canon, fl32, fl64, flc;
};

// ---------------------------------------------------------------- direct tests
// One test, FP32, the whole set factored in registers (order s_0 < ... < s_{L-1}, u, v),
// with the trust rule's terms exact: |b_u|_1 and |b_v|_1 by back substitution,
// |L_S^{-1}|_F^2 >= |corr_SS^{-1}|_2 by forward substitution.
// 0 dependent, 1 independent, 2 band, 3 guard (the FP64 evaluation decides 2 and 3).
template <int L>
__device__ __forceinline__ int nl_direct(const float *C, int ld, int u, int v, const int (&s)[L > 0 ? L : 1],
                                         const TestParams &tp, float sqf, float rq)
{
    constexpr int LA = L > 0 ? L : 1;
    float Lp[LA * (LA + 1) / 2], rd[LA], lu[LA], lv[LA];
    float h11 = 1.f, h22 = 1.f, h12 = C[u * ld + v], pmin = 1e30f;
    bool bad = false;
#pragma unroll
    for (int i = 0; i < L; ++i) {
        const float *Ci = C + s[i] * ld;
        float dd = 1.f;
#pragma unroll
        for (int c = 0; c < i; ++c) {
            float t = Ci[s[c]];
#pragma unroll
            for (int q = 0; q < c; ++q) t = fmaf(-Lp[i * (i + 1) / 2 + q], Lp[c * (c + 1) / 2 + q], t);
            t *= rd[c];
            Lp[i * (i + 1) / 2 + c] = t;
            dd = fmaf(-t, t, dd);
        }
        pmin = fminf(pmin, dd);
        bad |= !(dd > 1e-12f);
        rd[i] = rsqrtf(fmaxf(dd, 1e-30f));
        float a = Ci[u], b = Ci[v];
#pragma unroll
        for (int c = 0; c < i; ++c) {
            a = fmaf(-lu[c], Lp[i * (i + 1) / 2 + c], a);
            b = fmaf(-lv[c], Lp[i * (i + 1) / 2 + c], b);
        }
        lu[i] = a * rd[i];
        lv[i] = b * rd[i];
        h11 = fmaf(-lu[i], lu[i], h11);
        h22 = fmaf(-lv[i], lv[i], h22);
        h12 = fmaf(-lu[i], lv[i], h12);
    }
    pmin = fminf(pmin, fminf(h11, h22));
    bad |= !(h11 > 1e-12f) || !(h22 > 1e-12f);
    if (bad || pmin < (float)tp.guard) return 3;
    float F = 0.f;
#pragma unroll
    for (int c = 0; c < L; ++c) {
        float z[LA];
        z[c] = rd[c];
        F = fmaf(z[c], z[c], F);
#pragma unroll
        for (int k = c + 1; k < L; ++k) {
            float t = 0.f;
#pragma unroll
            for (int j = c; j < k; ++j) t = fmaf(Lp[k * (k + 1) / 2 + j], z[j], t);
            z[k] = -t * rd[k];
            F = fmaf(z[k], z[k], F);
        }
    }
    float Au = 1.f, Av = 1.f;
#pragma unroll
    for (int k = L - 1; k >= 0; --k) {
        float a = lu[k], b = lv[k];
#pragma unroll
        for (int j = k + 1; j < L; ++j) {
            a = fmaf(-Lp[j * (j + 1) / 2 + k], lu[j], a);
            b = fmaf(-Lp[j * (j + 1) / 2 + k], lv[j], b);
        }
        lu[k] = a * rd[k];                               // regression coefficients, in place
        lv[k] = b * rd[k];
        Au += fabsf(lu[k]);
        Av += fabsf(lv[k]);
    }
    const float ih = rsqrtf(h11 * h22), a = fabsf(h12 * ih);
    const float kap = (float)(L + 2) * (tp.eps_c + (4.0f * (float)(L + 2)) * EPS32) * F;
    float dr;
    const int t = fp32_trust(tp, L + 2, sqf, rq, a, h11, h22, ih, Au, Av, kap, dr);
    if (t) return t == 1 ? 2 : 3;
    return a <= rq ? 1 : 0;
}

__device__ __forceinline__ void nl_found(NlShared &S, int j, uint32_t rank)
{
    atomicMin(&S.best[j], rank);
    const int v = S.nbr[j];
    atomicOr(&S.own[v >> 5], 1u << (v & 31));
}

// The direct tests of node u at stage L: test t is the set of rank t / deg of pair t % deg,
// so the early ranks of every pair run first and a separated pair skips the rest.
template <int L>
__device__ __noinline__ void nl_direct_stage(NlShared &S, const TestParams &tp, const float *C, int ld, int u,
                                             NlAcc &acc)
{
    const int dg = S.deg[u], d = dg - 1;
    const uint32_t total = S.T[u] * (uint32_t)dg;
    const float sqf = sqrtf((float)(tp.n - L - 3)), rq = tanhf(tp.qf / sqf);
    unsigned run = 0;
    for (uint32_t t = threadIdx.x; t < total; t += NL_THREADS) {
        const uint32_t rank = t / (uint32_t)dg;
        const int j = (int)(t - rank * (uint32_t)dg);
        if (*(volatile uint32_t *)&S.best[j] < rank) continue;
        int s[L > 0 ? L : 1];
        nl_unrank<L>(S, rank, d, s);
#pragma unroll
        for (int i = 0; i < L; ++i) s[i] = S.nbr[s[i] + (s[i] >= j)];
        ++run;
        const int r = nl_direct<L>(C, ld, u, S.nbr[j], s, tp, sqf, rq);
        if (r == 1) {
            nl_found(S, j, rank);
        } else if (r) {
            if (r == 2) ++acc.band;
            else ++acc.guard;
            const int q = atomicAdd(&S.qn, 1);
            if (q < NL_QCAP) S.queue[q] = t;
        }
    }
    acc.tests += run;
    acc.fl32 += (ull)run * flops_direct(L);
}

// FP64 evaluation of the tests of the queue (all: of every test of the stage), a warp each.
__device__ __noinline__ void nl_direct_fp64(NlShared &S, const TestParams &tp, const double *C64, int ldc, int u, int l,
                                            bool all, unsigned char *buf, NlAcc &acc)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, m = l + 2;
    unsigned char *mine = buf + (size_t)w * NL_DIRECT_BYTES;
    double *Mbuf = (double *)mine;
    int *nd = (int *)(mine + NL_MMAX * (NL_MMAX + 1) * 8);
    const int dg = S.deg[u], d = dg - 1;
    const uint32_t total = all ? S.T[u] * (uint32_t)dg : (uint32_t)min(S.qn, NL_QCAP);
    const double sq = sqrt((double)(tp.n - l - 3));
    WarpAcc wa = {0, 0, 0, 0, 0, 0, 0, 0.f};
    unsigned run = 0;
    for (uint32_t i = w; i < total; i += NL_THREADS / 32) {
        const uint32_t t = all ? i : S.queue[i];
        uint32_t rank = t / (uint32_t)dg;
        const int j = (int)(t - rank * (uint32_t)dg);
        const uint32_t rank0 = rank;
        if (*(volatile uint32_t *)&S.best[j] < rank) continue;
        if (lane == 0) {
            int x = 0;
            for (int k = 0; k < l; ++k) {
                const int r1 = l - k;
                const uint32_t base = S.bin[(d - x) * NL_BR + r1], target = base - rank;
                int lo = x, hi = d - r1;
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (S.bin[(d - mid) * NL_BR + r1] >= target) lo = mid;
                    else hi = mid - 1;
                }
                rank -= base - S.bin[(d - lo) * NL_BR + r1];
                nd[k] = S.nbr[lo + (lo >= j)];
                x = lo + 1;
            }
            nd[l] = u;
            nd[l + 1] = S.nbr[j];
        }
        __syncwarp();
        double r;
        float z;
        ++run;
        const bool ind = warp_test<true>(nd, m, l, nullptr, C64, ldc, tp, sq, (float)sq, Mbuf, NL_MMAX + 1, wa, r, z);
        if (ind && lane == 0) nl_found(S, j, rank0);
        __syncwarp();
    }
    if (lane == 0) {
        if (all) acc.tests += run;
        else acc.red += run;
        acc.degen += (unsigned)wa.degen;
        acc.fl64 += wa.fl64;
    }
}

// ---------------------------------------------------------------- complement tests
// FP32 evaluation from the FP32 rounding of the block (packed), the trust rule of
// comp_test_fp32 (level.cu): 0 trusted (indep set), 1 band, 2 guard.
template <int K>
__device__ __forceinline__ int nl_comp_fp32(const float *P, const int (&sr)[K > 0 ? K : 1], int su, int sv,
                                            const TestParams &tp, float sqf, float rq, bool &indep)
{
    constexpr int KA = K > 0 ? K : 1;
    float L[KA][KA], yu[KA], yv[KA], sd[KA], ri[KA];
#pragma unroll
    for (int i = 0; i < K; ++i) {
#pragma unroll
        for (int c = 0; c <= i; ++c) L[i][c] = P[tri(sr[i], sr[c])];
        yu[i] = P[tri2(sr[i], su)];
        yv[i] = P[tri2(sr[i], sv)];
        sd[i] = sqrtf(fmaxf(L[i][i], 0.f));
    }
    const float Puu = P[tri(su, su)], Pvv = P[tri(sv, sv)];
    float Quu = Puu, Qvv = Pvv, Quv = P[tri2(su, sv)];
    bool bad = false;
#pragma unroll
    for (int i = 0; i < K; ++i) {
#pragma unroll
        for (int c = 0; c < i; ++c) {
            float t = L[i][c];
#pragma unroll
            for (int q = 0; q < c; ++q) t = fmaf(-L[i][q], L[c][q], t);
            L[i][c] = t * ri[c];
        }
        float t = L[i][i];
#pragma unroll
        for (int q = 0; q < i; ++q) t = fmaf(-L[i][q], L[i][q], t);
        bad |= !(t > 0.f);
        ri[i] = rsqrtf(t);
        float a = yu[i], b = yv[i];
#pragma unroll
        for (int q = 0; q < i; ++q) {
            a = fmaf(-L[i][q], yu[q], a);
            b = fmaf(-L[i][q], yv[q], b);
        }
        yu[i] = a * ri[i];
        yv[i] = b * ri[i];
        Quu = fmaf(-yu[i], yu[i], Quu);
        Qvv = fmaf(-yv[i], yv[i], Qvv);
        Quv = fmaf(-yu[i], yv[i], Quv);
    }
    if (bad || !(Quu > 0.f) || !(Qvv > 0.f)) return 2;
    float Wu = sqrtf(Puu), Wv = sqrtf(Pvv);
#pragma unroll
    for (int i = K - 1; i >= 0; --i) {
        float a = yu[i], b = yv[i];
#pragma unroll
        for (int q = i + 1; q < K; ++q) {
            a = fmaf(-L[q][i], yu[q], a);
            b = fmaf(-L[q][i], yv[q], b);
        }
        yu[i] = a * ri[i];
        yv[i] = b * ri[i];
        Wu = fmaf(sd[i], fabsf(yu[i]), Wu);
        Wv = fmaf(sd[i], fabsf(yv[i]), Wv);
    }
    float tr = 0.f;
#pragma unroll
    for (int j = 0; j < K; ++j) {
        float m[KA], nj = 0.f;
#pragma unroll
        for (int i = j; i < K; ++i) {
            float t = i == j ? 1.f : 0.f;
#pragma unroll
            for (int q = j; q < i; ++q) t = fmaf(-L[i][q], m[q], t);
            m[i] = t * ri[i];
            nj = fmaf(m[i], m[i], nj);
        }
        tr = fmaf(sd[j] * sd[j], nj, tr);
    }
    const float eps = (4.0f * (float)K + 8.0f) * EPS32;
    const float kap = (float)K * eps * tr;
    const float iu = __frcp_rn(Quu), iv = __frcp_rn(Qvv);
    const float qu = eps * Wu * Wu * iu, qv = eps * Wv * Wv * iv;
    if (!(fmaxf(fmaxf(qu, qv), kap) <= 0.05f)) return 2;
    const float ih = rsqrtf(Quu * Qvv);
    const float a = fabsf(Quv * ih);
    const float dr = 2.0f * eps * (Wu * Wv * ih + 0.5f * a * (Wu * Wu * iu + Wv * Wv * iv)) + 8.0f * EPS32;
    if (!(dr <= tp.dr_max)) return 2;
    const float om = 1.0f - a * a;
    if (!(om > 8.0f * dr) || Quu * om > 1e9f || Qvv * om > 1e9f) return 2;
    const float gap = fabsf(a - rq), mn = fminf(a, rq);
    if (gap <= dr || sqf * gap < (float)tp.band * (1.0f - mn * mn)) return 1;
    indep = a <= rq;
    return 0;
}

// FP64 evaluation (the decision of complement_body, level.cu)
template <int K>
__device__ __noinline__ bool nl_comp_fp64(const double *P, const int (&sr)[K > 0 ? K : 1], int su, int sv, int l,
                                          const TestParams &tp, double rq, unsigned &degen)
{
    constexpr int KA = K > 0 ? K : 1;
    double L[KA][KA], ri[KA], yu[KA], yv[KA];
    double Quu = P[tri(su, su)], Qvv = P[tri(sv, sv)], Quv = P[tri2(su, sv)];
#pragma unroll
    for (int i = 0; i < K; ++i) {
#pragma unroll
        for (int c = 0; c <= i; ++c) L[i][c] = P[tri(sr[i], sr[c])];
        yu[i] = P[tri2(sr[i], su)];
        yv[i] = P[tri2(sr[i], sv)];
    }
    bool bad = false;
#pragma unroll
    for (int i = 0; i < K; ++i) {
#pragma unroll
        for (int c = 0; c < i; ++c) {
            double s = L[i][c];
#pragma unroll
            for (int q = 0; q < c; ++q) s = fma(-L[i][q], L[c][q], s);
            L[i][c] = s * ri[c];
        }
        double s = L[i][i];
#pragma unroll
        for (int q = 0; q < i; ++q) s = fma(-L[i][q], L[i][q], s);
        bad |= !(s > 0.0);
        ri[i] = rsqrt(s);
        double a = yu[i], b = yv[i];
#pragma unroll
        for (int q = 0; q < i; ++q) {
            a = fma(-L[i][q], yu[q], a);
            b = fma(-L[i][q], yv[q], b);
        }
        yu[i] = a * ri[i];
        yv[i] = b * ri[i];
        Quu = fma(-yu[i], yu[i], Quu);
        Qvv = fma(-yv[i], yv[i], Qvv);
        Quv = fma(-yu[i], yv[i], Quv);
    }
    const double det = Quu * Qvv - Quv * Quv;
    const double h11 = Qvv / det, h22 = Quu / det;
    if (bad || !(h11 > DEGEN) || !(h22 > DEGEN) || !(det > 0.0)) {
        ++degen;
        return true;
    }
    const double r = -Quv * rsqrt(Quu * Qvv), ar = fabs(r);
    if (fabs(ar - rq) > 1e-12 * rq) return ar < rq;
    const double z = ar < 1.0 ? sqrt((double)(tp.n - l - 3)) * fabs(atanh(r)) : INFINITY;
    return z <= tp.q;
}

// The complement tests of node u at stage l: |R| = K dropped neighbours (the same for
// every pair of u); complement of lex order is reverse lex order.
template <int K>
__device__ __noinline__ void nl_comp_stage(NlShared &S, const TestParams &tp, const double *P, const float *Pf, int u,
                                           int l, bool f32, NlAcc &acc)
{
    const int dg = S.deg[u], d = dg - 1, su = S.slot[u];
    const uint32_t T = S.T[u], total = T * (uint32_t)dg;
    const double rq = tp.rq_tab[l];
    const float sqf = sqrtf((float)(tp.n - l - 3)), rqf = (float)rq;
    unsigned run = 0;
    for (uint32_t t = threadIdx.x; t < total; t += NL_THREADS) {
        const uint32_t rank = t / (uint32_t)dg;
        const int j = (int)(t - rank * (uint32_t)dg);
        if (*(volatile uint32_t *)&S.best[j] < rank) continue;
        int sr[K > 0 ? K : 1];
        nl_unrank<K>(S, T - 1 - rank, d, sr);
#pragma unroll
        for (int i = 0; i < K; ++i) sr[i] = S.nslot[sr[i] + (sr[i] >= j)];
        const int sv = S.nslot[j];
        ++run;
        bool ind = false;
        if (f32) {
            const int r = nl_comp_fp32<K>(Pf, sr, su, sv, tp, sqf, rqf, ind);
            if (r) {
                if (r == 1) ++acc.band;
                else ++acc.guard;
                ++acc.red;
                ind = nl_comp_fp64<K>(P, sr, su, sv, l, tp, rq, acc.degen);
            }
        } else {
            ind = nl_comp_fp64<K>(P, sr, su, sv, l, tp, rq, acc.degen);
        }
        if (ind) nl_found(S, j, rank);
    }
    acc.comp += run;
    acc.flc += (ull)run * ((ull)(K * K * K) / 3 + 2ull * K * K + 6ull * K + 20);
}

// ---------------------------------------------------------------- block work
// The triangle updates below give thread (ty, tx) of a 16 x 16 grid the rows i = ty (mod
// 16) and columns j = tx (mod 16): the column's factors stay in registers over the rows
// and the row's loads are independent of one another.  A pivot costs about 0.6 us of
// dependent FP64 latency (the reciprocal, the scaled column, the update; measured at
// p = 20) plus its FMAs at 2 per clock and SM.
constexpr int NL_Q = NL_PMAX / 16;

// One pivot of the symmetric sweep A <- -A^{-1} of the m x m packed block (pivots in
// order: see sweep_inverse_block).  S.rD holds 1/pivot (formed by the thread that wrote
// the pivot last).  Sets S.bad when the next pivot is at the degeneracy floor.
__device__ __forceinline__ void nl_sweep_step(NlShared &S, double *P, int m, int k)
{
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const double iD = S.rD;
    for (int i = threadIdx.x; i < m; i += NL_THREADS) {
        const double c = P[tri2(i, k)];
        S.colk[i] = c;
        S.cols[i] = c * iD;
    }
    __syncthreads();
    double cj[NL_Q];
#pragma unroll
    for (int q = 0; q < NL_Q; ++q) cj[q] = tx + 16 * q < m ? S.colk[tx + 16 * q] : 0.0;
    const int nxt = k + 1;
    // the row of the next pivot first
    const int a0 = nxt < m && (nxt & 15) == ty ? nxt >> 4 : 0;
    for (int a = 0; 16 * a < m; ++a) {
        const int i = ty + 16 * (a == 0 ? a0 : (a == a0 ? 0 : a));
        if (i >= m) continue;
        const double ci = S.cols[i];
        double *row = P + tri(i, 0);
#pragma unroll
        for (int q = 0; q < NL_Q; ++q) {
            const int j = tx + 16 * q;
            if (j > i) break;
            double v;
            if (i == k) v = j == k ? -iD : S.cols[j];
            else if (j == k) v = ci;
            else v = fma(-ci, cj[q], row[j]);
            row[j] = v;
        }
        if (i == nxt && tx == (nxt & 15)) {
            const double v = row[nxt];
            if (!(v > DEGEN)) S.bad = 1;
            S.rD = rcp_newton(v);
        }
    }
    __syncthreads();
}

// Drops the last member of S.list (n members before): P_ij -= P_iw P_jw / P_ww for the
// others (the inverse of a principal submatrix), one pass over their triangle.  Work and
// time: n^2/2 FP64 FMAs at 2 per clock; each earlier member waits only for two barriers.
__device__ __forceinline__ void nl_drop_step(NlShared &S, double *P, float *Pf, int n, int nt)
{
    const int r = n - 1, w = S.list[r];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const double iD = S.rD;
    for (int i = threadIdx.x; i < r; i += NL_THREADS) {
        const double c = P[tri2(S.list[i], w)];
        S.colk[i] = c;
        S.cols[i] = c * iD;
    }
    __syncthreads();
    const bool last = r == nt;
    double cj[NL_Q];
    int sj[NL_Q];
#pragma unroll
    for (int q = 0; q < NL_Q; ++q) {
        const int j = tx + 16 * q;
        cj[q] = j < r ? S.colk[j] : 0.0;
        sj[q] = j < r ? S.list[j] : 0;
    }
    // rows from the last (the next pivot's) down
    for (int a = (r - 1) >> 4; a >= 0; --a) {
        const int i = ty + 16 * a;
        if (i >= r) continue;
        const int si = S.list[i];
        const double ci = S.cols[i];
#pragma unroll
        for (int q = 0; q < NL_Q; ++q) {
            const int j = tx + 16 * q;
            if (j > i) break;
            const int e = tri2(si, sj[q]);               // slots ascend among the kept members only
            const double v = fma(-ci, cj[q], P[e]);
            P[e] = v;
            if (last) Pf[e] = round_f32(v);
        }
        if (i == r - 1 && tx == ((r - 1) & 15) && !last) {
            const double v = P[tri(si, si)];
            if (!(v > DEGEN)) S.bad = 1;
            S.rD = rcp_newton(v);
        }
    }
    __syncthreads();
}

}  // namespace

__global__ void __launch_bounds__(NL_THREADS, 1) node_loop_kernel(GraphDev g, TestParams tp, const float *C32,
                                                                  const double *C64, int ldc, double *Pbuf,
                                                                  unsigned long long *xch, double budget, int cap,
                                                                  int stage_a)
{
    extern __shared__ __align__(16) unsigned char nl_raw[];
    __shared__ NlShared S;
    const int p = g.p, W = g.W, u = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int ntri = tri(p, 0), cs = p | 1;
    double *P = (double *)nl_raw;                        // packed block
    unsigned char *dbuf = nl_raw + (size_t)ntri * 8;     // warps' FP64 direct tests
    dbuf += (16 - ((size_t)ntri * 8 & 15)) & 15;
    float *Pf = (float *)(dbuf + (NL_THREADS / 32) * NL_DIRECT_BYTES);
    float *C = Pf + ntri;                                // FP32 correlations, row stride cs
    LevelInfo *I = g.info;
    NlAcc acc = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
    const bool blocks = tp.reversed && tp.complement;
    const bool f32 = tp.comp_fp32 != 0;

    // ---- tables, the complete graph, this node's rows of the set store
    for (int e = tid; e < NL_PMAX * NL_BR; e += NL_THREADS) {
        const int x = e / NL_BR, r = e - x * NL_BR;
        const ull b = x < g.ldb && r < g.ldb ? g.binom[(long long)x * g.ldb + r] : 0ull;
        S.bin[e] = b < NL_SAT ? (uint32_t)b : NL_SAT;
    }
    for (int e = tid; e < p * p; e += NL_THREADS) {
        const int i = e / p, j = e - i * p;
        C[i * cs + j] = C32[(long long)i * ldc + j];
    }
    if (tid < p) {
        for (int w = 0; w < NL_W; ++w) {
            const int lo = 32 * w;
            uint32_t b = p >= lo + 32 ? 0xffffffffu : (p > lo ? (1u << (p - lo)) - 1u : 0u);
            if (tid >= lo && tid < lo + 32) b &= ~(1u << (tid - lo));
            S.A[tid][w] = b;
        }
        S.deg[tid] = p - 1;
        if (tid > u) {
            g.sep_level[u * p + tid] = -1;
            g.sep_off[u * p + tid] = -1;
        }
    }
    if (tid == 0) S.bad = 0;
    __syncthreads();

    uint32_t seq = 0;
    // this node's block: state, pivots done (build), members, live members, kept members
    int blk = BLK_NONE, bk = 0, bm = 0, nl = 0, nt = 0;
    bool timeout = false;

    // adj(u) and its slots from A[u]
    auto neighbours = [&]() {
        if (tid < p) {
            const uint32_t word = S.A[u][tid >> 5];
            if ((word >> (tid & 31)) & 1u) {
                int x = __popc(word & ((1u << (tid & 31)) - 1u));
                for (int w = 0; w < (tid >> 5); ++w) x += __popc(S.A[u][w]);
                S.nbr[x] = (short)tid;
                S.nslot[x] = S.slot[tid];
            }
        }
    };
    // the block from corr[F,F]: load it, first pivot's reciprocal
    auto build_start = [&]() {
        bm = S.deg[u] + 1;
        if (tid < p) {
            const uint32_t self = (u >> 5) == (tid >> 5) ? 1u << (u & 31) : 0u;
            const uint32_t word = S.A[u][tid >> 5] | self;
            int x = __popc(word & ((1u << (tid & 31)) - 1u));
            for (int w = 0; w < (tid >> 5); ++w) x += __popc(S.A[u][w] | ((u >> 5) == w ? 1u << (u & 31) : 0u));
            if ((word >> (tid & 31)) & 1u) {
                S.slot[tid] = (short)x;
                S.snode[x] = (short)tid;
            } else {
                S.slot[tid] = -1;
            }
        }
        if (tid == 0) S.bad = 0;
        __syncthreads();
        for (int e = tid; e < tri(bm, 0); e += NL_THREADS) {
            const int i = tri_row(e), j = e - tri(i, 0);
            P[e] = __ldg(C64 + (long long)S.snode[i] * ldc + S.snode[j]);
        }
        if (tid == 0) S.rD = 1.0;                        // corr_00 = 1
        __syncthreads();
        blk = BLK_BUILD;
        bk = 0;
    };
    // live slots of the block: members still adjacent (and u), then members to drop
    auto live_list = [&]() {
        // S.slot[v] >= 0 marks a live member; a dropped one is set to -1 by drop
        uint32_t km = 0, pm = 0;                         // this warp's word of kept / to-drop nodes
        int myslot = -1;
        bool kept = false, gone = false;
        if (wid < NL_W) {
            const int v = tid;
            if (v < p) {
                myslot = S.slot[v];
                const bool adj = v == u || ((S.A[u][v >> 5] >> (v & 31)) & 1u);
                kept = myslot >= 0 && adj;
                gone = myslot >= 0 && !adj;
            }
            km = __ballot_sync(0xffffffffu, kept);
            pm = __ballot_sync(0xffffffffu, gone);
            if (lane == 0) {
                S.red[wid] = __popc(km);
                S.red[8 + wid] = __popc(pm);
            }
        }
        __syncthreads();
        int k0 = 0, p0 = 0, kt = 0, pt = 0;
        for (int w = 0; w < NL_W; ++w) {
            if (w < wid) {
                k0 += S.red[w];
                p0 += S.red[8 + w];
            }
            kt += S.red[w];
            pt += S.red[8 + w];
        }
        const uint32_t lt = (1u << lane) - 1u;
        if (kept) S.list[k0 + __popc(km & lt)] = (short)myslot;
        if (gone) S.list[kt + p0 + __popc(pm & lt)] = (short)myslot;
        nt = kt;
        nl = kt + pt;
        __syncthreads();
        if (tid == 0 && nl > nt) {
            const double v = P[tri(S.list[nl - 1], S.list[nl - 1])];
            S.bad = !(v > DEGEN);
            S.rD = rcp_newton(v);
        }
        __syncthreads();
    };
    // one step of this node's pending block work; false: none left
    auto block_step = [&]() -> bool {
        if (blk == BLK_BUILD) {
            if (bk < bm) {
                if (S.bad) {                             // a pivot at the floor: no block for this node
                    blk = BLK_SINGULAR;
                    return false;
                }
                nl_sweep_step(S, P, bm, bk);
                ++bk;
                return true;
            }
            for (int e = tid; e < tri(bm, 0); e += NL_THREADS) {
                const double v = -P[e];
                P[e] = v;
                Pf[e] = round_f32(v);
            }
            __syncthreads();
            blk = BLK_OK;
            if (tid == 0) {
                atomicAdd(&g.ctr->prec_builds, 1ull);
                atomicAdd(&g.ctr->flops_prec, (ull)bm * bm * bm);
            }
            live_list();
            return true;
        }
        if (blk == BLK_OK && nl > nt) {
            if (S.bad) {                                 // the block has lost accuracy: again from corr
                __syncthreads();
                build_start();
                return true;
            }
            nl_drop_step(S, P, Pf, nl, nt);
            --nl;
            if (tid == 0) S.slot[S.snode[S.list[nl]]] = -1;
            __syncthreads();
            return true;
        }
        return false;
    };
    // after the graph changed: what is pending, or a new block where one is due
    auto block_plan = [&]() {
        if (!blocks) return;
        const int dg = S.deg[u];
        if (blk == BLK_OK) {
            live_list();
            if (nl > nt) {
                // clocks of dropping nl - nt members one by one against a sweep of the nt left
                const float drop = drop_clocks(nt, nl), build = build_clocks(nt);
                if (tid == 0) {
                    atomicAdd(&g.ctr->prec_downdates, 1ull);
                    atomicAdd(&g.ctr->flops_prec, (ull)(nl - nt) * nl * nl);
                }
                if (build < drop && dg >= 2) build_start();
            }
        } else if (blk == BLK_BUILD && 2 * (dg + 1) < bm) {
            build_start();                               // the neighbourhood has shrunk far below the one being swept
        } else if (blk == BLK_NONE && dg >= 2) {
            build_start();
        }
    };
    // The separating sets this CTA records for the last stage applied (thread j: its pair
    // with neighbour j), kept in registers until the CTA waits for the others: the pool's
    // atomic and the stores are then off the stage's critical path.
    bool rec = false, rec_any = false;
    int rec_l = 0, rec_d = 0, rec_v = 0;
    uint32_t rec_rank = 0, rec_T = 0;
    bool rec_explicit = false;
    auto record = [&]() {
        if (!rec_any) return;
        rec_any = false;
        if (wid >= NL_W) return;
        const uint32_t bal = __ballot_sync(0xffffffffu, rec);
        if (!bal) return;
        const int l = rec_l;
        ull base = 0;
        if (lane == 0) {
            atomicAdd(&g.ctr->edges_removed, (ull)__popc(bal));
            if (rec_explicit && l > 0) base = atomicAdd(&g.ctr->pool_len, (ull)__popc(bal) * (ull)l);
        }
        base = __shfl_sync(0xffffffffu, base, 0);
        if (rec) {
            const int v = rec_v, a = min(u, v), b = max(u, v);
            const long long e = (long long)a * p + b;
            const ull off = base + (ull)__popc(bal & ((1u << lane) - 1u)) * (ull)l;
            g.sep_level[e] = l;
            g.sep_side[e] = rec_explicit && u > v;
            g.sep_rank[e] = (long long)rec_rank;
            g.sep_off[e] = rec_explicit ? (long long)off : -1ll;
            if (rec_explicit && (long long)(off + l) > g.pool_cap) {
                g.info->pool_overflow = 1;               // the host enlarges the pool and reruns
                g.info->halt = 1;
            } else if (rec_explicit) {
                // the set by the table's columns: its members, or the d - l dropped ones
                const int d = rec_d, j = tid, k = d - l;
                const bool cmpl = k < l;
                uint32_t r = cmpl ? rec_T - 1u - rec_rank : rec_rank;
                const int cnt = cmpl ? k : l;
                int x = 0, out = 0;
                for (int i = 0; i < cnt; ++i) {
                    const int r1 = cnt - i;
                    const uint32_t bs = S.bin[(d - x) * NL_BR + r1], target = bs - r;
                    int lo = x, hi = d - r1;
                    while (lo < hi) {
                        const int mid = (lo + hi + 1) >> 1;
                        if (S.bin[(d - mid) * NL_BR + r1] >= target) lo = mid;
                        else hi = mid - 1;
                    }
                    r -= bs - S.bin[(d - lo) * NL_BR + r1];
                    if (cmpl)
                        for (; x < lo; ++x) g.pool[off + out++] = S.nbr0[x + (x >= j)];
                    else
                        g.pool[off + out++] = S.nbr0[lo + (lo >= j)];
                    x = lo + 1;
                }
                if (cmpl)
                    for (; x < d; ++x) g.pool[off + out++] = S.nbr0[x + (x >= j)];
            }
        }
    };
    // publish this CTA's words (and `mark`) for stage number seq
    auto publish = [&](bool release, uint32_t mark) {
        if (tid < W) {
            const ull x = ((ull)(seq | mark) << 32) | S.own[tid];
            ull *to = xch + ((size_t)(seq & 1u) * p + u) * W + tid;
            if (release) asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(to), "l"(x) : "memory");
            else asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(to), "l"(x) : "memory");
        }
    };
    // wait for every CTA's words of stage number seq (block work meanwhile); true when
    // some CTA could not run the stage
    auto gather = [&](bool acquire) -> bool {
        const int ne = p * W;
        bool h0 = tid >= ne, h1 = tid + NL_THREADS >= ne, ex = false;
        const ull *src = xch + (size_t)(seq & 1u) * ne;
        const long long t0 = clock64();
        int tries = 0;
        auto poll = [&](int e) -> bool {
            ull x;
            if (acquire) asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(x) : "l"(src + e) : "memory");
            else asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(x) : "l"(src + e) : "memory");
            const uint32_t s = (uint32_t)(x >> 32);
            if ((s & ~NL_EXIT) != seq) return false;
            ex |= (s & NL_EXIT) != 0;
            S.M[e / W][e % W] = (uint32_t)x;
            return true;
        };
        for (;;) {
            if (!h0) h0 = poll(tid);
            if (!h1) h1 = poll(tid + NL_THREADS);
            if (__syncthreads_and(h0 && h1)) break;
            if ((++tries & 63) == 0 && __syncthreads_or(clock64() - t0 > NL_WAIT)) {
                timeout = true;
                return true;
            }
            if (rec_any) record();
            else block_step();
        }
        return __syncthreads_or(ex);
    };
    // apply the stage's deletions to the graph: this node's canonical count and the sets to
    // record, then the new rows, degrees and adj(u).  l: the stage (rank from S.best);
    // explicit_sets 0: the closed-form stage (one test per pair, the set is all others).
    auto apply = [&](int l, bool explicit_sets) {
        record();                                        // the stage before, if no wait gave room for it
        __syncthreads();
        const int dg = S.deg[u];
        rec = false;
        if (tid < dg) {
            const int v = S.nbr[tid];
            const bool mine = (S.M[u][v >> 5] >> (v & 31)) & 1u, its = (S.M[v][u >> 5] >> (u & 31)) & 1u;
            rec_rank = explicit_sets ? S.best[tid] : 0u;
            if (explicit_sets) {
                if (u < v || !its) acc.canon += mine ? (ull)rec_rank + 1ull : (ull)S.T[u];
                rec = mine && (u < v || !its);
            } else {
                acc.canon += u < v;
                rec = u < v && (mine || its);
            }
            rec_v = v;
            S.nbr0[tid] = (short)v;
        }
        rec_any = true;
        rec_l = l;
        rec_d = dg - 1;
        rec_T = S.T[u];
        rec_explicit = explicit_sets;
        __syncthreads();
        // the transpose of M by ballots (32 x 32 tiles), merged into the rows' deletions
        for (int t = wid; t < W * W; t += NL_THREADS / 32) {
            const int wb = t / W, kv = t - wb * W;       // rows 32 wb .. of M, word kv
            const int row = wb * 32 + lane;
            const uint32_t x = row < p ? S.M[row][kv] : 0u;
            if (!__any_sync(0xffffffffu, x != 0u)) continue;
            uint32_t mine = 0;
#pragma unroll
            for (int b = 0; b < 32; ++b) {
                const uint32_t y = __ballot_sync(0xffffffffu, (x >> b) & 1u);
                if (lane == b) mine = y;
            }
            if (mine) atomicAnd(&S.A[kv * 32 + lane][wb], ~mine);   // column bits -> rows
            if (x) atomicAnd(&S.A[row][kv], ~x);
        }
        __syncthreads();
        if (tid < p) {
            int d = 0;
            for (int w = 0; w < W; ++w) d += __popc(S.A[tid][w]);
            S.deg[tid] = d;
        }
        if (tid < NL_W) S.own[tid] = 0u;
        __syncthreads();
        neighbours();
        __syncthreads();
    };
    // largest degree
    auto max_degree = [&]() -> int {
        const int d = tid < p ? S.deg[tid] : 0;
        const int m = __reduce_max_sync(0xffffffffu, d);
        if (lane == 0) S.red[wid] = m;
        __syncthreads();
        int r = 0;
        for (int w = 0; w < NL_THREADS / 32; ++w) r = max(r, S.red[w]);
        __syncthreads();
        return r;
    };

    if (tid < NL_W) S.own[tid] = 0u;
    if (tid < p) S.slot[tid] = -1;
    __syncthreads();
    neighbours();
    __syncthreads();

    // ---- stage l = p - 2 in closed form: corr = L D L^T in every CTA (the pivots are the
    // conditional variances in node order), row u of corr^{-1} by the two solves, the rows
    // exchanged through Pbuf
    int ran_a = 0, levels = 0;
    if (stage_a) {
        for (int e = tid; e < ntri; e += NL_THREADS) {
            const int i = tri_row(e), j = e - tri(i, 0);
            P[e] = __ldg(C64 + (long long)i * ldc + j);
        }
        if (tid == 0) S.rD = 1.0;
        __syncthreads();
        bool sing = false;
        for (int k = 0; k < p; ++k) {
            if (S.bad) {
                sing = true;
                break;
            }
            const double iD = S.rD;
            for (int i = k + 1 + tid; i < p; i += NL_THREADS) {
                const double c = P[tri(i, k)];
                S.colk[i] = c;
                const double s = c * iD;
                S.cols[i] = s;
                P[tri(i, k)] = s;                        // L
            }
            if (tid == 0) S.z[k] = iD;                   // 1/D
            __syncthreads();
            const int tx = tid & 15, ty = tid >> 4;
            double cj[NL_Q];
#pragma unroll
            for (int q = 0; q < NL_Q; ++q) {
                const int j = tx + 16 * q;
                cj[q] = j > k && j < p ? S.colk[j] : 0.0;
            }
            for (int a = (k + 1) >> 4; 16 * a < p; ++a) {   // the next pivot's row is among the first
                const int i = ty + 16 * a;
                if (i <= k || i >= p) continue;
                const double ci = S.cols[i];
                double *row = P + tri(i, 0);
#pragma unroll
                for (int q = 0; q < NL_Q; ++q) {
                    const int j = tx + 16 * q;
                    if (j > i) break;
                    if (j > k) row[j] = fma(-ci, cj[q], row[j]);
                }
                if (i == k + 1 && tx == (i & 15)) {
                    const double v = row[i];
                    if (!(v > DEGEN)) S.bad = 1;
                    S.rD = rcp_newton(v);
                }
            }
            __syncthreads();
        }
        if (!sing) {
            // L z = e_u, x = L^{-T} D^{-1} z: thread i holds entry i, one broadcast per column
            double x = tid == u ? 1.0 : 0.0;
            for (int j = u; j < p; ++j) {
                if (tid == j) S.colk[j & 1] = x;
                __syncthreads();
                if (tid > j && tid < p) x = fma(-P[tri(tid, j)], S.colk[j & 1], x);
            }
            if (tid < p) x *= S.z[tid];
            __syncthreads();
            for (int j = p - 1; j > 0; --j) {
                if (tid == j) S.colk[j & 1] = x;
                __syncthreads();
                if (tid < j) x = fma(-P[tri(j, tid)], S.colk[j & 1], x);
            }
            if (tid < p) Pbuf[(long long)u * ldc + tid] = x;
            ran_a = 1;
        }
        ++seq;
        __syncthreads();
        publish(true, 0u);
        gather(true);
        if (ran_a && !timeout) {
            // pair {a < b}: the entry of row a; the decision of Eq. 1 (one test per pair)
            const double sq = sqrt((double)(tp.n - p - 1));
            if (tid < p && tid != u) {
                const int a = min(u, tid), b = max(u, tid);
                const double paa = __ldcg(Pbuf + (long long)a * ldc + a), pbb = __ldcg(Pbuf + (long long)b * ldc + b);
                const double pab = __ldcg(Pbuf + (long long)a * ldc + b);
                const double det = paa * pbb - pab * pab;
                const double h11 = pbb / det, h22 = paa / det;
                bool ind;
                if (!(h11 > DEGEN) || !(h22 > DEGEN)) {
                    ind = true;
                    if (u < tid) ++acc.degen;
                } else {
                    const double r = -pab / sqrt(paa * pbb);
                    const double z = fabs(r) < 1.0 ? sq * fabs(atanh(r)) : INFINITY;
                    ind = z <= tp.q;
                }
                if (u < tid) ++acc.tests;
                if (ind) atomicOr(&S.own[tid >> 5], 1u << (tid & 31));
            }
            ++seq;
            __syncthreads();
            publish(true, 0u);
            gather(true);
            if (!timeout) {
                apply(p - 2, false);
                levels = 1;
                if (blocks && S.deg[u] >= 2) {
                    // the first block from the inverse: all nodes members, the non-neighbours
                    // dropped, where that is less work than a sweep of corr[F,F]
                    const int m = S.deg[u] + 1;
                    if (drop_clocks(m, p) + 1000.f < build_clocks(m)) {
                        for (int e = tid; e < ntri; e += NL_THREADS) {
                            const int i = tri_row(e), j = e - tri(i, 0);
                            const double v = __ldcg(Pbuf + (long long)j * ldc + i);
                            P[e] = v;
                            Pf[e] = round_f32(v);
                        }
                        if (tid < p) {
                            S.slot[tid] = (short)tid;
                            S.snode[tid] = (short)tid;
                        }
                        bm = p;
                        blk = BLK_OK;
                        if (tid == 0) atomicAdd(&g.ctr->prec_builds, 1ull);
                        __syncthreads();
                        live_list();
                        neighbours();
                        __syncthreads();
                    } else {
                        build_start();
                    }
                }
            }
        }
    }

    // ---- the first stage (Algorithm 1: 0 upwards; Algorithm 2: from the largest degree down)
    int lmax = max_degree() - 1, l = 0;
    bool go;
    if (tp.reversed) {
        l = cap;
        if (ran_a && l > p - 3) l = p - 3;
        l = min(l, lmax);
        go = l >= 0;
    } else {
        go = cap >= 0 && lmax >= 0;
    }
    const int first = go ? l : -1;
    if (blocks && !ran_a && go && S.deg[u] >= 2) build_start();

    // ---- the stages
    bool handover = false;
    while (go && !timeout) {
        // every node's tests; the whole stage's against the budget and the size this kernel takes
        uint32_t my = 0;
        bool big = false;
        if (tid < p) {
            const int dg = S.deg[tid], d = dg - 1;
            const uint32_t T = dg > 0 ? nl_sets(S, d, l) : 0u;
            S.T[tid] = T;
            big = T > NL_TESTS_MAX || T * (uint32_t)dg > NL_TESTS_MAX;
            my = big ? 0u : T * (uint32_t)dg;
        }
        const uint32_t ws = __reduce_add_sync(0xffffffffu, my);
        if (lane == 0) S.red[wid] = (int)ws;
        if (tid == 0) S.qn = 0;
        if (tid < NL_PMAX) S.best[tid] = NL_NONE;
        big = __syncthreads_or(big);
        uint32_t total = 0;
        for (int w = 0; w < NL_THREADS / 32; ++w) total += (uint32_t)S.red[w];
        if (big || (double)total > budget) {             // the same in every CTA
            handover = true;
            break;
        }
        const int dg = S.deg[u], d = dg - 1;
        const NlAcc before = acc;
        uint32_t mark = 0;
        if (S.T[u] > 0) {
            const bool elig = blocks && comp_eligible(d, l, tp);
            if (elig)
                while (block_step()) {
                }
            if (elig && blk == BLK_OK) {
                if (dg > 0) neighbours();                // slots of a block built since the graph changed
                __syncthreads();
                switch (d - l) {
                case 0: nl_comp_stage<0>(S, tp, P, Pf, u, l, f32, acc); break;
                case 1: nl_comp_stage<1>(S, tp, P, Pf, u, l, f32, acc); break;
                case 2: nl_comp_stage<2>(S, tp, P, Pf, u, l, f32, acc); break;
                case 3: nl_comp_stage<3>(S, tp, P, Pf, u, l, f32, acc); break;
                case 4: nl_comp_stage<4>(S, tp, P, Pf, u, l, f32, acc); break;
                case 5: nl_comp_stage<5>(S, tp, P, Pf, u, l, f32, acc); break;
                case 6: nl_comp_stage<6>(S, tp, P, Pf, u, l, f32, acc); break;
                case 7: nl_comp_stage<7>(S, tp, P, Pf, u, l, f32, acc); break;
                default: nl_comp_stage<8>(S, tp, P, Pf, u, l, f32, acc); break;
                }
            } else if (l > LANE_LMAX || (g.row_off && l >= 1 && l <= tp.learned_lmax)) {
                mark = NL_EXIT;                          // larger sets, or a stage the proposal may score
            } else if (tp.precision == 0) {
                nl_direct_fp64(S, tp, C64, ldc, u, l, true, dbuf, acc);
            } else {
                switch (l) {
                case 0: nl_direct_stage<0>(S, tp, C, cs, u, acc); break;
                case 1: nl_direct_stage<1>(S, tp, C, cs, u, acc); break;
                case 2: nl_direct_stage<2>(S, tp, C, cs, u, acc); break;
                case 3: nl_direct_stage<3>(S, tp, C, cs, u, acc); break;
                case 4: nl_direct_stage<4>(S, tp, C, cs, u, acc); break;
                case 5: nl_direct_stage<5>(S, tp, C, cs, u, acc); break;
                case 6: nl_direct_stage<6>(S, tp, C, cs, u, acc); break;
                case 7: nl_direct_stage<7>(S, tp, C, cs, u, acc); break;
                case 8: nl_direct_stage<8>(S, tp, C, cs, u, acc); break;
                case 9: nl_direct_stage<9>(S, tp, C, cs, u, acc); break;
                case 10: nl_direct_stage<10>(S, tp, C, cs, u, acc); break;
                case 11: nl_direct_stage<11>(S, tp, C, cs, u, acc); break;
                default: nl_direct_stage<12>(S, tp, C, cs, u, acc); break;
                }
                __syncthreads();
                if (S.qn > NL_QCAP) mark = NL_EXIT;      // more FP64 tests than the queue holds
                else if (S.qn > 0) nl_direct_fp64(S, tp, C64, ldc, u, l, false, dbuf, acc);
            }
        }
        ++seq;
        __syncthreads();
        publish(seq <= 2u, mark);
        if (gather(seq <= 2u)) {
            handover = !timeout;
            acc = before;                                // the other driver runs, and counts, the whole stage
            break;
        }
        apply(l, true);
        ++levels;
        lmax = max_degree() - 1;
        if (tp.reversed) {
            l = min(l - 1, lmax);
            go = l >= 0;
        } else {
            ++l;
            go = l <= cap && lmax >= l;
        }
        if (go) block_plan();
    }

    record();
    // ---- results; when another driver goes on from stage l, its state as well
    const bool more = handover && !timeout;
    if (more && blocks)
        while (block_step()) {
        }
    if (tid < W) g.adj[(long long)u * W + tid] = S.A[u][tid];
    const int dg = S.deg[u];
    if (tid < dg) g.nbr[(long long)u * p + tid] = S.nbr[tid];
    if (tid == 0) {
        g.deg[u] = dg;
        g.dchg[u] = 0;
        g.prec_need[u] = 0;
        g.prec_m[u] = more && blocks ? (blk == BLK_OK ? nt : (blk == BLK_SINGULAR ? -1 : 0)) : 0;
        long long off = 0;
        for (int v = 0; v < u; ++v) off += S.deg[v];
        g.ooff[u] = off;
        if (u == p - 1) g.ooff[p] = off + dg;
    }
    if (more) {
        for (int v = tid; v < p; v += NL_THREADS) {
            g.best[(long long)u * p + v] = KEY_NONE;
            g.prec_pos[(long long)u * p + v] = -1;
        }
        __syncthreads();
        if (blocks && blk == BLK_OK) {
            double *B = g.prec + (long long)u * PREC_MAX * PREC_MAX;
            for (int e = tid; e < nt * nt; e += NL_THREADS) {
                const int i = e / nt, j = e - i * nt;
                B[i * PREC_MAX + j] = P[tri2(S.list[i], S.list[j])];
            }
            for (int i = tid; i < nt; i += NL_THREADS) {
                const int v = S.snode[S.list[i]];
                g.prec_mem[(long long)u * PREC_MAX + i] = v;
                g.prec_pos[(long long)u * p + v] = (short)i;
            }
        }
    }
    // counters: warp sums, one atomic each
    ull vals[9] = {acc.tests + acc.comp, acc.comp, acc.band, acc.guard, acc.red, acc.degen, acc.canon, acc.fl32 , acc.fl64};
    ull flc = acc.flc;
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int k = 0; k < 9; ++k) vals[k] += __shfl_xor_sync(0xffffffffu, vals[k], o);
        flc += __shfl_xor_sync(0xffffffffu, flc, o);
    }
    if (lane == 0) {
        DevCounters *c = g.ctr;
        if (vals[0]) atomicAdd(&c->tests_executed, vals[0]);
        if (vals[1]) atomicAdd(&c->complement_tests, vals[1]);
        if (vals[2]) atomicAdd(&c->band_hits, vals[2]);
        if (vals[3]) atomicAdd(&c->guard_hits, vals[3]);
        if (vals[4]) atomicAdd(&c->redecided, vals[4]);
        if (vals[5]) atomicAdd(&c->degenerate, vals[5]);
        if (vals[6]) atomicAdd(&c->tests_canonical, vals[6]);
        if (vals[7]) atomicAdd(&c->flops, vals[7]);
        if (vals[8]) atomicAdd(&c->flops64_direct, vals[8]);
        if (flc) atomicAdd(&c->flops_comp, flc);
    }
    if (u == 0 && tid == 0) {
        long long edges = 0;
        for (int v = 0; v < p; ++v) edges += S.deg[v];
        I->l = l;
        I->lstar = lmax;
        I->n_opairs = edges;
        I->edges = (ull)edges;
        I->done = !go && !timeout;
        I->levels_run = levels;
        I->first_level = first;
        I->stage_a_ran = ran_a;
        if (ran_a) g.ctr->flops_stagea = (ull)p * (p - 1) / 2 * 12ull;
    }
    if (timeout && tid == 0) {
        I->error = 7;                                    // PC_ERR_TIMEOUT
        I->halt = 1;
    }
}

static size_t node_loop_smem(int p)
{
    const size_t ntri = (size_t)p * (p + 1) / 2;
    return (ntri * 8 + 15) / 16 * 16 + (size_t)(NL_THREADS / 32) * NL_DIRECT_BYTES + ntri * 4 +
           (size_t)p * (p | 1) * 4;
}

size_t node_loop_xch_bytes(int p) { return (size_t)2 * p * ((p + 31) / 32) * sizeof(unsigned long long); }

cudaError_t launch_node_loop(GraphDev g, TestParams tp, const float *C32, const double *C64, int ldc, double *Pbuf,
                             unsigned long long *xch, double budget, int cap, int stage_a, cudaStream_t s)
{
    if (g.p > NL_PMAX) return cudaErrorInvalidValue;
    const size_t smem = node_loop_smem(g.p);
    cudaError_t e = cudaFuncSetAttribute(node_loop_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    e = cudaMemsetAsync(xch, 0, node_loop_xch_bytes(g.p), s);    // stage number 0: nothing published
    if (e != cudaSuccess) return e;
    void *args[] = {&g, &tp, (void *)&C32, (void *)&C64, &ldc, &Pbuf, &xch, &budget, &cap, &stage_a};
    e = cudaLaunchCooperativeKernel((const void *)node_loop_kernel, dim3(g.p), dim3(NL_THREADS), args, smem, s);
    note_launch();
    return e;
}

}  // namespace fpc
