// orient.cu -- Phase II of Algorithm 1 (Algorithm 2 leaves it unchanged,
// Sec. 3.3): the skeleton is oriented from the separation sets.  First the
// unshielded colliders (i - k - j, i and j non-adjacent, k not in S(i,j):
// i -> k <- j), then rules R1-R4 repeated until none orients an edge.
//
// Order-free reading (the listing orders neither loop): every collider marks
// both of its edges at once, and the rules run in rounds -- each round tests
// every undirected edge against the marks of the previous round and applies all
// orientations it finds together.  An edge marked from both ends (two colliders,
// or both directions in one round) is bidirected.  R4 is read with X_k and X_j
// non-adjacent (the printed "X_k and X_l" contradicts its own X_k -> X_l).
//
// Marks are per-node bitsets over the instance's nodes:
//   AH[x] = {y : the edge {x,y} has an arrowhead at y}
//   AT[x] = {y : the edge {x,y} has an arrowhead at x}   (the transpose of AH)
// so that, with ADJ the skeleton's rows,
//   parents PA[x] = ADJ & AT & ~AH, children CH[x] = ADJ & AH & ~AT,
//   undirected UN[x] = ADJ & ~AH & ~AT,
// and each rule is a few word operations per 32 candidate nodes.
#include "internal.h"
#include "device_util.cuh"

#include <algorithm>

namespace fpc {

namespace {

__device__ __forceinline__ void inst_words(const GraphDev &g, int x, int &lo, int &hi, int &w0, int &w1)
{
    lo = g.blk_lo ? g.blk_lo[x] : 0;
    hi = g.blk_hi ? g.blk_hi[x] : g.p;
    w0 = lo >> 5;
    w1 = (hi - 1) >> 5;
}

// A barrier over the CTAs of a cooperative launch (all resident): the k-th one waits for
// k * gridDim.x arrivals.  Bounded: false after about 2 s. 
__device__ bool grid_wait(unsigned *count, unsigned &target)
{
    __shared__ int ok_s;
    __syncthreads();
    if (threadIdx.x == 0) {
        target += gridDim.x;
        __threadfence();
        atomicAdd(count, 1u);
        const long long t0 = clock64();
        int ok = 1;
        for (;;) {
            unsigned c;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(c) : "l"(count) : "memory");
            if (c >= target) break;
            if (clock64() - t0 > 4000000000ll) {
                ok = 0;
                break;
            }
        }
        ok_s = ok;
    }
    __syncthreads();
    return ok_s != 0;
}

// The neighbours of node k (ascending) into nb by a warp, from its adjacency row; the degree.
__device__ int warp_neighbours(const GraphDev &g, int k, int w0, int w1, int *nb)
{
    const int lane = threadIdx.x & 31;
    const uint32_t *row = g.adj + (long long)k * g.W;
    int base = 0;
    for (int v0 = w0; v0 <= w1; v0 += 32) {
        const int w = v0 + lane;
        uint32_t bits = w <= w1 ? row[w] : 0u;
        const int c = __popc(bits);
        int incl = c;
        for (int off = 1; off < 32; off <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, off);
            if (lane >= off) incl += t;
        }
        int pos = base + incl - c;
        while (bits) {
            nb[pos++] = w * 32 + __ffs(bits) - 1;
            bits &= bits - 1;
        }
        base += __shfl_sync(0xffffffffu, incl, 31);
    }
    __syncwarp();
    return base;
}

// The unshielded triples i - k - j of node k, pairs t, t + step, ... of its dg neighbours:
// a collider unless k lies in S(i, j) (ascending: binary search; a pair without a record or
// with the set of all other nodes, l = p-2, has none).
__device__ __forceinline__ void colliders_of(const GraphDev &g, uint32_t *ah, uint32_t *at, int k, const int *nb,
                                             int dg, int t, int step)
{
    const int W = g.W;
    const long long np = (long long)dg * (dg - 1) / 2;
    for (long long q = t; q < np; q += step) {
        int y = (int)((sqrtf(8.f * (float)q + 1.f) + 1.f) * 0.5f);    // pair x < y, q = y (y-1) / 2 + x
        while ((long long)y * (y - 1) / 2 > q) --y;
        while ((long long)(y + 1) * y / 2 <= q) ++y;
        const int i = nb[q - (long long)y * (y - 1) / 2], j = nb[y];
        if ((g.adj[(long long)i * W + (j >> 5)] >> (j & 31)) & 1u) continue;
        const long long e = pidx(g, i, j);
        const int len = g.sep_level[e];
        const long long off = g.sep_off[e];
        if (len < 0 || off < 0) continue;
        const int *S = g.pool + off;
        int l0 = 0, l1 = len;
        while (l0 < l1) {
            const int mid = (l0 + l1) >> 1;
            if (S[mid] < k) l0 = mid + 1;
            else l1 = mid;
        }
        if (l0 < len && S[l0] == k) continue;            // k separates i and j
        atomicOr(ah + (long long)i * W + (k >> 5), 1u << (k & 31));
        atomicOr(ah + (long long)j * W + (k >> 5), 1u << (k & 31));
        atomicOr(at + (long long)k * W + (i >> 5), 1u << (i & 31));
        atomicOr(at + (long long)k * W + (j >> 5), 1u << (j & 31));
    }
}

// Is one of R1-R4 orienting the undirected edge a - b into a -> b?  One thread, over the
// words [w0, w1] of the instance: an edge is a few word operations per 32 candidates, and a
// node's edges (lanes of a warp) run side by side.  Ab, Hb, ...: rows of W words.
template <class Row>
__device__ bool rule_orients(const Row &A, const Row &H, const Row &T, int a, int b, int w0, int w1)
{
    const int wb = b >> 5;
    const uint32_t bbit = 1u << (b & 31);
    const uint32_t *Aa = A(a), *Ha = H(a), *Ta = T(a), *Ab = A(b), *Hb = H(b), *Tb = T(b);
    // R1: some c -> a with c and b non-adjacent;  R2: a -> c -> b
    bool more = false;
    for (int w = w0; w <= w1; ++w) {
        const uint32_t aa = Aa[w], ha = Ha[w], ta = Ta[w], ab = Ab[w];
        const uint32_t pb = ab & Tb[w] & ~Hb[w];
        uint32_t r1 = aa & ta & ~ha & ~ab;
        if (w == wb) r1 &= ~bbit;
        if (r1 | (aa & ha & ~ta & pb)) return true;
        more |= pb != 0u;
    }
    if (!more) return false;                             // no parent of b: R3 and R4 need one
    // R3: a - c -> b and a - d -> b with c, d non-adjacent;
    // R4: a - c -> d -> b with c and b non-adjacent
    for (int w = w0; w <= w1; ++w) {
        const uint32_t una = Aa[w] & ~Ha[w] & ~Ta[w];
        uint32_t C = una & Ab[w] & Tb[w] & ~Hb[w];
        uint32_t K = una & ~Ab[w];
        if (w == wb) K &= ~bbit;
        while (C) {
            const int cb = __ffs(C) - 1;
            C &= C - 1;
            const uint32_t *Ac = A((w << 5) + cb);
            for (int v = w0; v <= w1; ++v) {
                uint32_t x = Aa[v] & ~Ha[v] & ~Ta[v] & Ab[v] & Tb[v] & ~Hb[v] & ~Ac[v];
                if (v == w) x &= ~(1u << cb);
                if (x) return true;
            }
        }
        while (K) {
            const int cb = __ffs(K) - 1;
            K &= K - 1;
            const int c = (w << 5) + cb;
            const uint32_t *Ac = A(c), *Hc = H(c), *Tc = T(c);
            for (int v = w0; v <= w1; ++v)
                if (Ac[v] & Hc[v] & ~Tc[v] & Ab[v] & Tb[v] & ~Hb[v]) return true;
        }
    }
    return false;
}

struct GlobalRows {
    const uint32_t *base;
    int W;
    __device__ __forceinline__ const uint32_t *operator()(int x) const { return base + (long long)x * W; }
};

// codes per ordered pair: 0 no edge, 1 a - b, 2 a -> b, 3 a <- b, 4 a <-> b; four b from b0
// on (bits of the words A, AH, AT already shifted to b0)
__device__ __forceinline__ uint32_t codes4(uint32_t A, uint32_t H, uint32_t T)
{
    uint32_t c4 = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const uint32_t h = (H >> q) & 1u, t = (T >> q) & 1u;
        c4 |= ((A >> q) & 1u ? (h ? (t ? 4u : 2u) : (t ? 3u : 1u)) : 0u) << (8 * q);
    }
    return c4;
}

// The phases, over the nodes of the whole grid (a warp or a CTA each).
constexpr int OR_DEG_WARP = 64;          // nodes of larger degree: their triples by the whole CTA
struct Marks {
    uint32_t *ah, *at, *add;
};
__device__ __forceinline__ int grid_warp() { return (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); }
__device__ __forceinline__ int grid_warps() { return (int)((gridDim.x * blockDim.x) >> 5); }

__device__ __forceinline__ void phase_triples_warp(const GraphDev &g, const Marks &m)
{
    for (int k = grid_warp(); k < g.p; k += grid_warps()) {
        int lo, hi, w0, w1;
        inst_words(g, k, lo, hi, w0, w1);
        int *nb = g.nbr + nidx(g, k);
        const int dg = warp_neighbours(g, k, w0, w1, nb);
        if ((threadIdx.x & 31) == 0) g.deg[k] = dg;
        if (dg <= OR_DEG_WARP) colliders_of(g, m.ah, m.at, k, nb, dg, threadIdx.x & 31, 32);
    }
}
__device__ __forceinline__ void phase_triples_cta(const GraphDev &g, const Marks &m)
{
    for (int k = blockIdx.x; k < g.p; k += gridDim.x) {
        const int dg = __ldcg(g.deg + k);
        if (dg > OR_DEG_WARP) colliders_of(g, m.ah, m.at, k, g.nbr + nidx(g, k), dg, threadIdx.x, blockDim.x);
    }
}
// the orientations that the marks imply, into each node's row of add; did this thread find one?
__device__ __forceinline__ bool phase_find(const GraphDev &g, const Marks &m)
{
    const int lane = threadIdx.x & 31, W = g.W;
    const GlobalRows A{g.adj, W}, H{m.ah, W}, T{m.at, W};
    bool any = false;
    for (int a = grid_warp(); a < g.p; a += grid_warps()) {
        int lo, hi, w0, w1;
        inst_words(g, a, lo, hi, w0, w1);
        const long long row = (long long)a * W;
        for (int w = w0 + lane; w <= w1; w += 32) m.add[row + w] = 0u;
        __syncwarp();
        const int dg = __ldcg(g.deg + a);
        const int *nb = g.nbr + nidx(g, a);
        for (int x = lane; x < dg; x += 32) {
            const int b = nb[x], w = b >> 5;
            const uint32_t bit = 1u << (b & 31);
            if ((m.ah[row + w] | m.at[row + w]) & bit) continue;
            if (!rule_orients(A, H, T, a, b, w0, w1)) continue;
            atomicOr(m.add + row + w, bit);
            any = true;
        }
    }
    return any;
}
__device__ __forceinline__ void phase_apply(const GraphDev &g, const Marks &m)
{
    const int lane = threadIdx.x & 31, W = g.W;
    for (int a = grid_warp(); a < g.p; a += grid_warps()) {
        int lo, hi, w0, w1;
        inst_words(g, a, lo, hi, w0, w1);
        const long long row = (long long)a * W;
        for (int w = w0 + lane; w <= w1; w += 32) m.ah[row + w] |= __ldcg(m.add + row + w);
        const int dg = __ldcg(g.deg + a);
        const int *nb = g.nbr + nidx(g, a);
        for (int x = lane; x < dg; x += 32) {
            const int b = nb[x];
            if ((__ldcg(m.add + (long long)b * W + (a >> 5)) >> (a & 31)) & 1u)
                atomicOr(m.at + row + (b >> 5), 1u << (b & 31));
        }
    }
}
__device__ __forceinline__ void phase_codes(const GraphDev &g, const Marks &m, int8_t *out, int vec)
{
    const int p = g.p;
    for (int a = grid_warp(); a < p; a += grid_warps()) {
        const long long row = (long long)a * g.W;
        int8_t *o = out + (long long)a * p;
        for (int b0 = (threadIdx.x & 31) * 4; b0 < p; b0 += 128) {
            const int w = b0 >> 5, sh = b0 & 31;
            const uint32_t c4 = codes4(g.adj[row + w] >> sh, m.ah[row + w] >> sh, m.at[row + w] >> sh);
            if (vec) *(uint32_t *)(o + b0) = c4;
            else
                for (int q = 0; q < 4 && b0 + q < p; ++q) o[b0 + q] = (int8_t)(c4 >> (8 * q));
        }
    }
}

// Phase II in one cooperative launch: colliders, the rounds of R1-R4, the codes.  A round
// is two phases with a barrier after each: every node's warp finds the orientations
// a -> b of its undirected edges (a lane each) from the marks as they stand, into its own
// row of `add`, then every node's warp takes them into its rows of AH and AT.  The
// colliders walk the unshielded triples of each node k, sum deg^2/2 of them, instead of
// the common neighbours of all p^2/2 pairs.
// Measured (pc_orient from the call to its return, us): p = 1000, 1 round 177 -> 63,
// p = 500, 2 rounds 156 -> 63 (a round was two copies, a fill, a launch and a host round
// trip, about 35 us, and an edge a whole warp's turn).
// ctl: [0] barrier count, [1], [2] changed flags of even and odd rounds, [3] rounds, [4] error.
__global__ void __launch_bounds__(256) orient_kernel(GraphDev g, Marks m, int *ctl, long long max_rounds, int8_t *out,
                                                     int vec)
{
    unsigned target = 0;
    phase_triples_warp(g, m);
    bool ok = grid_wait((unsigned *)ctl, target);
    if (ok) phase_triples_cta(g, m);
    ok = ok && grid_wait((unsigned *)ctl, target);
    int rounds = 0;
    for (long long r = 0; ok && r <= max_rounds; ++r) {
        if (phase_find(g, m)) *(volatile int *)(ctl + 1 + (r & 1)) = 1;
        if (!(ok = grid_wait((unsigned *)ctl, target))) break;
        if (!*(volatile int *)(ctl + 1 + (r & 1))) break;      // the same in every CTA
        ++rounds;
        if (blockIdx.x == 0 && threadIdx.x == 0) *(volatile int *)(ctl + 1 + ((r + 1) & 1)) = 0;
        phase_apply(g, m);
        ok = grid_wait((unsigned *)ctl, target);
    }
    phase_codes(g, m, out, vec);
    if (blockIdx.x == 0 && threadIdx.x == 0) ctl[3] = rounds;
    if (!ok && threadIdx.x == 0) ctl[4] = 7;             // PC_ERR_TIMEOUT
}

// One phase a launch, for graphs whose work between two barriers could outlast the barriers'
// bound, or where the cooperative launch is not to be had.
enum { PH_TRIPLES_WARP, PH_TRIPLES_CTA, PH_FIND, PH_APPLY, PH_CODES };
__global__ void __launch_bounds__(256) orient_phase_kernel(GraphDev g, Marks m, int *ctl, int phase, int rounds,
                                                           int8_t *out, int vec)
{
    switch (phase) {
    case PH_TRIPLES_WARP: phase_triples_warp(g, m); break;
    case PH_TRIPLES_CTA: phase_triples_cta(g, m); break;
    case PH_FIND:
        if (phase_find(g, m)) ctl[1] = 1;
        break;
    case PH_APPLY: phase_apply(g, m); break;
    default:
        phase_codes(g, m, out, vec);
        if (blockIdx.x == 0 && threadIdx.x == 0) ctl[3] = rounds;
    }
}

// The same for p <= OR_ONE_P in one CTA: the three bitsets in shared memory, the rounds'
// barriers are the CTA's own, a thread per ordered adjacent pair.  Worth it while the
// triples (sum deg^2/2) and the pairs fit a few passes of its threads: mean degree <= 16;
// denser graphs take the kernel above.  Measured (pc_orient, us, before / cooperative
// kernel / this one): p = 95, 5 rounds 215 / 77 / 50, p = 95, 4 rounds 181 / 64 / 41,
// p = 20, 1 round 83 / 38 / 36.
constexpr int OR_ONE_P = 128, OR_ONE_W = OR_ONE_P / 32, OR_ONE_THREADS = 512;
struct SharedRows {
    const uint32_t (*base)[OR_ONE_W];
    __device__ __forceinline__ const uint32_t *operator()(int x) const { return base[x]; }
};
__global__ void __launch_bounds__(OR_ONE_THREADS) orient_one_kernel(GraphDev g, int *ctl, int max_rounds, int8_t *out)
{
    __shared__ uint32_t As[OR_ONE_P][OR_ONE_W], Hs[OR_ONE_P][OR_ONE_W], Ts[OR_ONE_P][OR_ONE_W];
    __shared__ int off[OR_ONE_P + 1], wsum[OR_ONE_P / 32];
    __shared__ uint16_t pair[OR_ONE_P * (OR_ONE_P - 1)];       // a << 8 | b, grouped by a
    const int tid = threadIdx.x, lane = tid & 31, p = g.p, W = g.W;
    for (int e = tid; e < OR_ONE_P * OR_ONE_W; e += OR_ONE_THREADS) {
        const int a = e / OR_ONE_W, w = e % OR_ONE_W;
        As[a][w] = a < p && w < W ? g.adj[(long long)a * W + w] : 0u;
        Hs[a][w] = Ts[a][w] = 0u;
    }
    __syncthreads();
    int dg = 0, incl = 0;
    if (tid < OR_ONE_P) {
        for (int w = 0; w < OR_ONE_W; ++w) dg += __popc(As[tid][w]);
        incl = dg;
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) wsum[tid >> 5] = incl;
    }
    __syncthreads();
    if (tid < OR_ONE_P) {
        int base = incl - dg;
        for (int w = 0; w < (tid >> 5); ++w) base += wsum[w];
        off[tid] = base;
        if (tid == OR_ONE_P - 1) off[OR_ONE_P] = base + dg;
        for (int w = 0; w < OR_ONE_W; ++w)
            for (uint32_t m = As[tid][w]; m; m &= m - 1) pair[base++] = (uint16_t)(tid << 8 | (w * 32 + __ffs(m) - 1));
    }
    __syncthreads();
    const int np = off[OR_ONE_P];
    // colliders: the triples i - k - j, a warp per k
    for (int k = tid >> 5; k < p; k += OR_ONE_THREADS / 32) {
        const int o = off[k], d = off[k + 1] - o;
        for (int q = lane; q < d * (d - 1) / 2; q += 32) {
            int y = (int)((sqrtf(8.f * (float)q + 1.f) + 1.f) * 0.5f);
            while (y * (y - 1) / 2 > q) --y;
            while ((y + 1) * y / 2 <= q) ++y;
            const int i = pair[o + q - y * (y - 1) / 2] & 255, j = pair[o + y] & 255;
            if ((As[i][j >> 5] >> (j & 31)) & 1u) continue;
            const long long e = (long long)i * p + j;
            const int len = g.sep_level[e];
            const long long so = g.sep_off[e];
            if (len < 0 || so < 0) continue;
            const int *S = g.pool + so;
            int l0 = 0, l1 = len;
            while (l0 < l1) {
                const int mid = (l0 + l1) >> 1;
                if (S[mid] < k) l0 = mid + 1;
                else l1 = mid;
            }
            if (l0 < len && S[l0] == k) continue;
            atomicOr(&Hs[i][k >> 5], 1u << (k & 31));
            atomicOr(&Hs[j][k >> 5], 1u << (k & 31));
            atomicOr(&Ts[k][i >> 5], 1u << (i & 31));
            atomicOr(&Ts[k][j >> 5], 1u << (j & 31));
        }
    }
    __syncthreads();
    const SharedRows A{As}, H{Hs}, T{Ts};
    int rounds = 0;
    for (int r = 0; r <= max_rounds; ++r) {
        // each thread's pairs in groups of 32: found orientations wait in `found` until
        // every thread has read the round's marks
        uint32_t found = 0;
        int n = 0;
        for (int e = tid; e < np; e += OR_ONE_THREADS, ++n) {
            const int a = pair[e] >> 8, b = pair[e] & 255;
            if (((Hs[a][b >> 5] | Ts[a][b >> 5]) >> (b & 31)) & 1u) continue;
            if (rule_orients(A, H, T, a, b, 0, W - 1)) found |= 1u << n;
        }
        if (!__syncthreads_or(found != 0u)) break;
        ++rounds;
        n = 0;
        for (int e = tid; found; e += OR_ONE_THREADS, ++n) {
            if (!((found >> n) & 1u)) continue;
            found &= ~(1u << n);
            const int a = pair[e] >> 8, b = pair[e] & 255;
            atomicOr(&Hs[a][b >> 5], 1u << (b & 31));
            atomicOr(&Ts[b][a >> 5], 1u << (a & 31));
        }
        __syncthreads();
    }
    for (int a = tid >> 5; a < p; a += OR_ONE_THREADS / 32) {
        const int b0 = lane * 4, w = lane >> 3, sh = b0 & 31;
        const uint32_t c4 = codes4(As[a][w] >> sh, Hs[a][w] >> sh, Ts[a][w] >> sh);
        for (int q = 0; q < 4 && b0 + q < p; ++q) out[(long long)a * p + b0 + q] = (int8_t)(c4 >> (8 * q));
    }
    if (tid == 0) ctl[3] = rounds;
}
static_assert(OR_ONE_P * (OR_ONE_P - 1) <= 32 * OR_ONE_THREADS, "a thread's pairs fit the word of found orientations");

// Word steps (each up to 8 loads) of a lane between two barriers: its nodes' edges in turns of
// 32, at most `dmax` candidates of W words for each (rule_orients).
long long lane_steps(int p, int dmax, int W, int warps)
{
    return (long long)((p + warps - 1) / warps) * ((dmax + 31) / 32) * (dmax + 2) * W;
}
// 2^20 of them at 700 clocks (L2) are 0.4 s of the barriers' 2; the triples of such nodes are
// fewer.  A sparse graph has some thousands; 1000 nodes of degree 999 are at the limit.
constexpr long long OR_STEPS_MAX = 1ll << 20;

}  // namespace

size_t orient_ws_bytes(const GraphDev &g) { return (3 * (size_t)g.p * g.W) * sizeof(uint32_t) + 8 * sizeof(int); }

// edges, dmax: of the skeleton (dmax: at least its largest degree); ws: orient_ws_bytes; ctl receives where
// the rounds ([3]) and the error ([4]) are
cudaError_t launch_orient(GraphDev g, long long edges, int dmax, void *ws, long long max_rounds, int8_t *out, int **ctl,
                          cudaStream_t s)
{
    const size_t words = (size_t)g.p * g.W;
    Marks m{(uint32_t *)ws, (uint32_t *)ws + words, (uint32_t *)ws + 2 * words};
    int *c = (int *)(m.add + words);
    *ctl = c;
    const bool one = g.p <= OR_ONE_P && !g.prow && edges <= 8ll * g.p;
    cudaError_t e = one ? cudaMemsetAsync(c, 0, 8 * sizeof(int), s) : cudaMemsetAsync(ws, 0, orient_ws_bytes(g), s);
    if (e != cudaSuccess) return e;
    int vec = g.p % 4 == 0 && ((uintptr_t)out & 3) == 0;
    if (one) {
        orient_one_kernel<<<1, OR_ONE_THREADS, 0, s>>>(g, c, (int)max_rounds, out); note_launch();
        return cudaGetLastError();
    }
    int dev = 0, sms = 0, coop = 0, per_sm = 0;
    e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, orient_kernel, 256, 0);
    if (e != cudaSuccess) return e;
    const int blocks = std::max(1, std::min((g.p + 7) / 8, sms * std::max(1, per_sm)));
    const int wi = std::min(g.W, (g.ldb + 61) / 32);     // words of the largest instance (ldb - 1 nodes, any first bit)
    if (coop && lane_steps(g.p, dmax, wi, blocks * 8) <= OR_STEPS_MAX) {
        void *args[] = {&g, &m, &c, &max_rounds, &out, &vec};
        e = cudaLaunchCooperativeKernel((const void *)orient_kernel, dim3(blocks), dim3(256), args, 0, s);
        if (e != cudaErrorCooperativeLaunchTooLarge) {
            note_launch();
            return e;
        }
        cudaGetLastError();                              // not resident: phase by phase
    }
    auto phase = [&](int k, int rounds) -> cudaError_t {
        orient_phase_kernel<<<(g.p + 7) / 8, 256, 0, s>>>(g, m, c, k, rounds, out, vec); note_launch();
        return cudaGetLastError();
    };
    e = phase(PH_TRIPLES_WARP, 0);
    if (e == cudaSuccess) e = phase(PH_TRIPLES_CTA, 0);
    int rounds = 0;
    for (long long r = 0; e == cudaSuccess && r <= max_rounds; ++r) {
        int changed = 0;
        e = cudaMemsetAsync(c + 1, 0, sizeof(int), s);
        if (e == cudaSuccess) e = phase(PH_FIND, 0);
        if (e == cudaSuccess) e = cudaMemcpyAsync(&changed, c + 1, sizeof(int), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess || !changed) break;
        ++rounds;
        e = phase(PH_APPLY, 0);
    }
    return e == cudaSuccess ? phase(PH_CODES, rounds) : e;
}

}  // namespace fpc
