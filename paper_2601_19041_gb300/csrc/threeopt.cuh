// First-improvement 3-opt with geometric neighbour lists and don't-look bits
// (Sec. III-D), one warp per tour.
//
// The search (its order defines the result):
//   cities are examined in tour-position order, skipping those whose bit is
//   set; passes repeat until one makes no move, and rounds (all bits cleared)
//   until a round whose first pass made no move; a call stops after 64n + 1024
//   moves.  For the examined city t2 = a and t1 = dir(a) (successor
//   direction, then predecessor direction), t3 runs over nbr(t2) while
//   g1 = d(t1,t2) - d(t2,t3) > 0, and t4 over dir(t3), then the other tour
//   neighbour of t3.  With t4 = dir(t3) the 2-opt closing (t4, t1) is tried
//   first, gain (g1 + d34) - d41.  Then t5 runs over nbr(t4) while
//   g2 = (g1 + d34) - d(t4,t5) > 0 (t5 = t3 skipped) and t6 over (succ t5,
//   pred t5) (t6 = t1 skipped), gain (g2 + d56) - d61.  Removed edges (t1,t2),
//   (t3,t4)[, (t5,t6)], added (t2,t3), (t4,t5)[, (t6,t1)] or (t4,t1).  The
//   first candidate in this order whose gain exceeds 1e-10 and whose
//   reconnection leaves a single cycle is applied; its cities' bits are
//   cleared and a is examined again; a city without a move gets its bit set.
//   Gains are FP64, each operation rounded once, in the order written.
//
// FP32 scan.  As in the 2-opt, gains are first estimated from FP32 distances
// (ls_da32, each within 5 units of 2^-24 of the FP64 one): with a band of 4e-6
// of the terms' sum (six terms and five additions err by less than 6.6e-7 of
// it) an estimate outside the band decides, and g1 > 0 and g2 > 0 likewise.
// ls3_scan tests one city: its (direction, t3, t4) pairs with g1 possibly
// positive are dealt to the lanes, each lane running through its pair's t5
// and t6 in order; the first pair with a possible move gives the first
// possible move of the city.  It is applied when every decision on the way
// was outside the band; otherwise ls3_examine searches the city again in
// FP64 (one t5 per lane).  FP64 is slow on this GPU (a dependent add takes about
// 100 cycles with its use, a distance several hundred): with FP64 alone one
// search took 47 ms (n = 500, 10-node lists, m = 32, start tour from the ants),
// and 8 iterations of 32 such instances 469 ms end to end; with the scan and the
// helper warps they take 30 ms.
//
// Helper warps (a block of several warps, see twoopt.cuh) test the next clear
// cities in tour order at the same time, one per warp: cities before the first
// one with a possible move have none, and testing them changes nothing.  They
// also share long middle rewrites.
//
// Applying a move: the removed edges sit at tour positions e_0 < e_1 (< e_2)
// (edge e joins tour[e] and tour[e+1 mod n]); positions outside
// [e_0 + 1, e_last] keep their cities and the middle positions receive the
// middle segments in the order and orientation in which the new cycle
// visits them after leaving tour[e_0].  The warp writes the middle through
// a scratch array (the FP32 edge array of the 2-opt, unused here).
#pragma once

#include "twoopt.cuh"

namespace hac {

__device__ __forceinline__ double ls3_d64(const float2 *xy, int u, int v)
{
    const float2 a = xy[u], b = xy[v];
    const double dx = __dsub_rn((double)b.x, (double)a.x), dy = __dsub_rn((double)b.y, (double)a.y);
    return __dsqrt_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)));
}

// A planned exchange: r removed edges at sorted positions e[], the middle
// segments j = seg[q] (positions e[j]+1 .. e[j+1]) in visiting order, rev[q]
// set when segment seg[q] is walked backwards.
struct Xchg {
    int r;
    int e[3];
    int seg[2], rev[2];
};

// position of the tour edge joining cities u and v, or -1 if they are not adjacent
__device__ __forceinline__ int ls3_edge(const LsMem &M, int n, int u, int v)
{
    const int pu = M.pos[u], pv = M.pos[v];
    if (pv == (pu + 1 == n ? 0 : pu + 1)) return pu;
    if (pu == (pv + 1 == n ? 0 : pv + 1)) return pv;
    return -1;
}

// Checks that removing the r edges {c[2k], c[2k+1]} and adding the r edges
// {c[2k+1], c[(2k+2) mod 2r]} (that is (t2,t3), (t4,t5), (t6,t1) for
// c = t1..t6, or (t2,t3), (t4,t1) for r = 2) leaves one cycle; plans it.
// The removed edges, sorted by position, have 2r endpoint slots: 2q is
// tour[e_q] and 2q + 1 is tour[e_q + 1].  The fixed part ends at slot 0 and
// starts at slot 2r - 1; middle segment j runs from slot 2j + 1 to slot 2j + 2.
// The added edges pair the slots; the pairing (a nibble per slot) is walked
// from slot 0 through every middle segment to slot 2r - 1.
template <int R>
__device__ __forceinline__ bool ls3_plan(const LsMem &M, int n, const int (&c)[2 * R], Xchg &X)
{
    int e[R];
    bool ok = true;
#pragma unroll
    for (int k = 0; k < R; ++k) {
        e[k] = ls3_edge(M, n, c[2 * k], c[2 * k + 1]);
        ok &= e[k] >= 0;
    }
    if (!ok) return false;
    int slot[2 * R];
#pragma unroll
    for (int k = 0; k < R; ++k) {
        int q = 0;
#pragma unroll
        for (int l = 0; l < R; ++l) q += e[l] < e[k];
        const int u = M.tour[e[k]];
        slot[2 * k] = 2 * q + (u == c[2 * k] ? 0 : 1);
        slot[2 * k + 1] = 2 * q + (u == c[2 * k + 1] ? 0 : 1);
    }
    unsigned pair = 0u, seen = 0u;
#pragma unroll
    for (int i = 0; i < R; ++i) {
        const int u = slot[2 * i + 1], v = slot[(2 * i + 2) % (2 * R)];
        pair |= ((unsigned)v << (4 * u)) | ((unsigned)u << (4 * v));
        seen |= (1u << u) | (1u << v);
    }
    if (seen != (1u << (2 * R)) - 1u) return false;   // equal edges, or a slot taken twice
    auto partner = [&](int s) { return (int)((pair >> (4 * s)) & 15u); };
    const int s0 = partner(0);
    if (s0 == 2 * R - 1) return false;                // the middle would be left out
    const int j0 = (s0 - 1) >> 1, x0 = ((s0 - 1) ^ 1) + 1;   // its segment and the segment's other end
    X.r = R;
    X.seg[0] = j0;
    X.rev[0] = (s0 & 1) ? 0 : 1;
    const int s1 = partner(x0);
    if constexpr (R == 2) {
        X.e[0] = min(e[0], e[1]);
        X.e[1] = max(e[0], e[1]);
        X.e[2] = 0;
        X.seg[1] = 0;
        X.rev[1] = 0;
        return s1 == 3;
    } else {
        if (s1 == 5 || ((s1 - 1) >> 1) == j0) return false;
        X.seg[1] = (s1 - 1) >> 1;
        X.rev[1] = (s1 & 1) ? 0 : 1;
        X.e[0] = min(min(e[0], e[1]), e[2]);
        X.e[2] = max(max(e[0], e[1]), e[2]);
        X.e[1] = e[0] + e[1] + e[2] - X.e[0] - X.e[2];
        return partner(((s1 - 1) ^ 1) + 1) == 5;
    }
}

// the share of thread tid of nth in rewriting the middle positions of an
// exchange: phase 0 collects the new middle in the scratch array, phase 1
// writes it back (a barrier between them)
__device__ __forceinline__ void ls3_rewrite_part(const LsMem &M, const Xchg &X, int tid, int nth, int phase)
{
    int32_t *tmp = reinterpret_cast<int32_t *>(M.el);
    const int lo = X.e[0] + 1;
    const int a0 = X.e[X.seg[0]] + 1, b0 = X.e[X.seg[0] + 1];
    const int len0 = b0 - a0 + 1;
    int a1 = 0, b1 = -1;
    if (X.r == 3) { a1 = X.e[X.seg[1]] + 1; b1 = X.e[X.seg[1] + 1]; }
    const int total = len0 + (b1 - a1 + 1);
    for (int w = tid; w < total; w += nth) {
        if (phase == 0) {
            int src;
            if (w < len0) src = X.rev[0] ? b0 - w : a0 + w;
            else src = X.rev[1] ? b1 - (w - len0) : a1 + (w - len0);
            tmp[w] = M.tour[src];
        } else {
            const int c = tmp[w];
            M.tour[lo + w] = c;
            M.pos[c] = lo + w;
        }
    }
}

// command 3, every warp of the block
__device__ __forceinline__ void ls3_coop_rewrite(const LsMem &M)
{
    const int *x = M.coop + LS_XCHG;
    Xchg X;
    X.r = x[0];
    X.e[0] = x[1]; X.e[1] = x[2]; X.e[2] = x[3];
    X.seg[0] = x[4] & 1; X.seg[1] = (x[4] >> 1) & 1;
    X.rev[0] = x[5] & 1; X.rev[1] = (x[5] >> 1) & 1;
    const int nth = 32 * M.coop_warps;
    ls3_rewrite_part(M, X, (int)threadIdx.x, nth, 0);
    ls_coop_bar(M.coop_warps);
    ls3_rewrite_part(M, X, (int)threadIdx.x, nth, 1);
    ls_coop_bar(M.coop_warps);
}

// rewrites the middle positions of the planned exchange (warp 0)
__device__ __forceinline__ void ls3_apply(const LsMem &M, const Xchg &X)
{
    const int lane = threadIdx.x & 31;
    __syncwarp();
    if (M.coop && X.e[X.r - 1] - X.e[0] >= LS_COOP_LEN) {
        if (lane == 0) {
            int *x = M.coop + LS_XCHG;
            M.coop[0] = 3;
            x[0] = X.r; x[1] = X.e[0]; x[2] = X.e[1]; x[3] = X.r == 3 ? X.e[2] : 0;
            x[4] = X.seg[0] | (X.r == 3 ? X.seg[1] << 1 : 0);
            x[5] = X.rev[0] | (X.r == 3 ? X.rev[1] << 1 : 0);
        }
        __syncwarp();
        ls_coop_bar(M.coop_warps);
        ls3_coop_rewrite(M);
        return;
    }
    ls3_rewrite_part(M, X, lane, 32, 0);
    __syncwarp();
    ls3_rewrite_part(M, X, lane, 32, 1);
    __syncwarp();
}

__device__ __forceinline__ Xchg ls3_bcast(const Xchg &X, int src)
{
    Xchg Y;
    Y.r = __shfl_sync(FULL2, X.r, src);
#pragma unroll
    for (int k = 0; k < 3; ++k) Y.e[k] = __shfl_sync(FULL2, X.e[k], src);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        Y.seg[k] = __shfl_sync(FULL2, X.seg[k], src);
        Y.rev[k] = __shfl_sync(FULL2, X.rev[k], src);
    }
    return Y;
}

// the FP64 gain of six terms from FP32 estimates of them: 0 certainly <=
// LS_GAIN, 2 certainly above, 1 undecided
__device__ __forceinline__ int ls3_gain_class(float g2, float mag2, float d56, float d61)
{
    const float est = __fsub_rn(__fadd_rn(g2, d56), d61);
    const float tol = __fadd_rn(__fmul_rn(4e-6f, __fadd_rn(mag2, __fadd_rn(d56, d61))), 1e-18f);
    if (!(est > __fsub_rn((float)LS_GAIN, tol))) return 0;
    return est > __fadd_rn((float)LS_GAIN, tol) ? 2 : 1;
}

// FP32 scan of city a (whole warp, only reads; the same result in every lane)
__device__ __forceinline__ LsMove ls3_scan(const LsMem &M, int n, int K, int a)
{
    const int lane = threadIdx.x & 31;
    const float2 *xy = M.xy;
    const int pa = M.pos[a];
    const int ts = M.tour[wrap_next(pa, n)], tp = M.tour[wrap_prev(pa, n)];
    const float2 xa = xy[a], xs = xy[ts], xp = xy[tp];
    const float ds = ls_da32(xs, xa), dp = ls_da32(xp, xa);
    const int nl = lane < K ? M.nbr[(size_t)a * K + lane] : 0;
    const float dl = lane < K ? M.nbrd32[(size_t)a * K + lane] : __int_as_float(0x7f800000);
    // t3 candidates of each direction: a prefix of the ascending list
    const float lim = __fmul_rn(dl, LS_G1_LO);
    const int Q0 = __popc(__ballot_sync(FULL2, ds > lim)), Q1 = __popc(__ballot_sync(FULL2, dp > lim));
    const int P = 2 * (Q0 + Q1);
    LsMove F;
    F.st = 0;
    F.r = 0;
#pragma unroll
    for (int k = 0; k < 6; ++k) F.c[k] = 0;
    for (int base = 0; base < P; base += 32) {
        const int pi = base + lane;
        const bool act = pi < P;
        const int dir = pi >= 2 * Q0 ? 1 : 0, qq = dir ? pi - 2 * Q0 : pi, q = qq >> 1, c4 = qq & 1;
        const int t3 = __shfl_sync(FULL2, nl, q & 31);
        const float d23 = __shfl_sync(FULL2, dl, q & 31);
        const int t1 = dir ? tp : ts, t2 = a;
        const float d12 = dir ? dp : ds;
        int st = 0, r = 0, t4 = 0, t5 = 0, t6 = 0;
        if (act && t3 != t1) {                 // t3 = t1: g1 = 0
            const int p3 = M.pos[t3];
            t4 = M.tour[c4 == dir ? wrap_next(p3, n) : wrap_prev(p3, n)];
            if (!((t3 == t1 && t4 == t2) || (t3 == t2 && t4 == t1))) {
                const float2 x1 = dir ? xp : xs, x4 = xy[t4];
                const float d34 = ls_da32(xy[t3], x4);
                const bool g1sure = __fmul_rn(d12, LS_G1_LO) > d23;
                Xchg X;
                // t4 = t2 closes to the same tour: its FP64 gain is the rounding of
                // ((d12 - d23) + d23) - d12, below 1e-10 at these lengths
                if (c4 == 0 && t4 != t1 && !(t4 == t2 && d12 + d23 < 1e4f)) {
                    const int cl = ls_gain_class(d12, d23, d34, ls_da32(x4, x1));
                    if (cl) {
                        const int c[4] = {t1, t2, t3, t4};
                        if (ls3_plan<2>(M, n, c, X)) { st = cl == 2 && g1sure ? 1 : 2; r = 2; }
                    }
                }
                const float g1b = __fadd_rn(__fsub_rn(d12, d23), d34), mag1 = __fadd_rn(__fadd_rn(d12, d23), d34);
                const int32_t *nb4 = M.nbr + (size_t)t4 * K;
                const float *nd4 = M.nbrd32 + (size_t)t4 * K;
                for (int k0 = 0; k0 < K && !st; k0 += 4) {
                    // four t5 at a time, both t6 of each: independent loads
                    int u5[4], u6[4][2];
                    float g2[4], mag2[4], d56[4][2], d61[4][2];
                    bool may[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const bool in = k0 + j < K;
                        u5[j] = in ? nb4[k0 + j] : t4;
                        const float d45 = in ? nd4[k0 + j] : __int_as_float(0x7f800000);
                        g2[j] = __fsub_rn(g1b, d45);
                        mag2[j] = __fadd_rn(mag1, d45);
                        may[j] = in && g2[j] > -__fadd_rn(__fmul_rn(4e-6f, mag2[j]), 1e-18f);
                    }
                    if (!may[0]) break;                       // the list ascends
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int p5 = M.pos[u5[j]];
                        u6[j][0] = M.tour[wrap_next(p5, n)];
                        u6[j][1] = M.tour[wrap_prev(p5, n)];
                    }
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float2 x5 = xy[u5[j]];
#pragma unroll
                        for (int c6 = 0; c6 < 2; ++c6) {
                            const float2 x6 = xy[u6[j][c6]];
                            d56[j][c6] = ls_da32(x5, x6);
                            d61[j][c6] = ls_da32(x6, x1);
                        }
                    }
                    unsigned cand = 0u, sure = 0u;
#pragma unroll
                    for (int j = 0; j < 4; ++j)
#pragma unroll
                        for (int c6 = 0; c6 < 2; ++c6) {
                            const int cl = ls3_gain_class(g2[j], mag2[j], d56[j][c6], d61[j][c6]);
                            // t4 = t2, t5 = t1 adds the edges it removes: gain 0 up to rounding, as above
                            const bool null = t4 == t2 && u5[j] == t1 && mag2[j] + d56[j][c6] < 1e4f;
                            const bool ok = may[j] && cl && u5[j] != t3 && u6[j][c6] != t1 && !null;
                            const bool g2sure = g2[j] > __fadd_rn(__fmul_rn(4e-6f, mag2[j]), 1e-18f);
                            cand |= (ok ? 1u : 0u) << (2 * j + c6);
                            sure |= (cl == 2 && g2sure ? 1u : 0u) << (2 * j + c6);
                        }
                    while (cand) {                             // rare: is the reconnection one cycle?
                        const int x = __ffs(cand) - 1;
                        cand &= cand - 1u;
                        t5 = nb4[k0 + (x >> 1)];
                        const int p5 = M.pos[t5];
                        t6 = M.tour[(x & 1) == 0 ? wrap_next(p5, n) : wrap_prev(p5, n)];
                        const int c[6] = {t1, t2, t3, t4, t5, t6};
                        if (ls3_plan<3>(M, n, c, X)) {
                            st = ((sure >> x) & 1u) && g1sure ? 1 : 2;
                            r = 3;
                            break;
                        }
                    }
                    if (!may[3]) break;
                }
            }
        }
        const unsigned hm = __ballot_sync(FULL2, st != 0);
        if (hm) {
            const int src = __ffs(hm) - 1;
            F.st = __shfl_sync(FULL2, st, src);
            F.r = __shfl_sync(FULL2, r, src);
            F.c[0] = __shfl_sync(FULL2, t1, src);
            F.c[1] = a;
            F.c[2] = __shfl_sync(FULL2, t3, src);
            F.c[3] = __shfl_sync(FULL2, t4, src);
            F.c[4] = __shfl_sync(FULL2, t5, src);
            F.c[5] = __shfl_sync(FULL2, t6, src);
            return F;
        }
    }
    return F;
}

// applies a certain move (warp 0)
__device__ __forceinline__ void ls3_apply_move(const LsMem &M, int n, const LsMove &F)
{
    const int lane = threadIdx.x & 31;
    Xchg X;
    if (F.r == 2) {
        const int c[4] = {F.c[0], F.c[1], F.c[2], F.c[3]};
        ls3_plan<2>(M, n, c, X);
    } else {
        ls3_plan<3>(M, n, F.c, X);
    }
    ls3_apply(M, X);
    if (lane < 2 * F.r) {
        int c = F.c[0];
#pragma unroll
        for (int k = 1; k < 6; ++k) c = lane == k ? F.c[k] : c;
        M.dlb[c] = 0;
    }
    __syncwarp();
}

// One examination of city a in FP64: finds and applies the first admissible
// move; true if a move was made (its cities' bits cleared).  One t5 per lane
// (both t6 of it), the first lane with an admissible move wins; the g1 values
// of all t3 are computed at once, one per lane.
static __device__ __noinline__ bool ls3_examine(const DevInst &I, const LsMem &M, int n, int K, int a)
{
    const int lane = threadIdx.x & 31;
    const float2 *xy = M.xy;
    auto succ = [&](int c) { const int p = M.pos[c]; return M.tour[p + 1 == n ? 0 : p + 1]; };
    auto pred = [&](int c) { const int p = M.pos[c]; return M.tour[p == 0 ? n - 1 : p - 1]; };
    for (int dir = 0; dir < 2; ++dir) {
        const int t2 = a, t1 = dir == 0 ? succ(a) : pred(a);
        const double d12 = ls3_d64(xy, t1, t2);
        const int t3l = lane < K ? I.nbr[(size_t)a * K + lane] : 0;
        const double g1l = lane < K ? __dsub_rn(d12, I.nbrd[(size_t)a * K + lane]) : 0.0;
        const unsigned stop = __ballot_sync(FULL2, lane >= K || !(g1l > 0.0));
        const int Q = stop ? __ffs(stop) - 1 : 32;   // t3 candidates 0..Q-1
        for (int q = 0; q < Q; ++q) {
            const int t3 = __shfl_sync(FULL2, t3l, q);
            const double g1 = __shfl_sync(FULL2, g1l, q);
            for (int c4 = 0; c4 < 2; ++c4) {
                const int t4 = (c4 == 0) == (dir == 0) ? succ(t3) : pred(t3);
                if ((t3 == t1 && t4 == t2) || (t3 == t2 && t4 == t1)) continue;
                const double d34 = ls3_d64(xy, t3, t4);
                if (c4 == 0 && t4 != t1) {
                    const double gain = __dsub_rn(__dadd_rn(g1, d34), ls3_d64(xy, t4, t1));
                    if (gain > LS_GAIN) {
                        const int c[4] = {t1, t2, t3, t4};
                        Xchg X;
                        if (ls3_plan<2>(M, n, c, X)) {
                            ls3_apply(M, X);
                            if (lane == 0) { M.dlb[t1] = 0; M.dlb[t2] = 0; M.dlb[t3] = 0; M.dlb[t4] = 0; }
                            __syncwarp();
                            return true;
                        }
                    }
                }
                const double g1b = __dadd_rn(g1, d34);
                const int t5 = lane < K ? I.nbr[(size_t)t4 * K + lane] : 0;
                const double g2 = lane < K ? __dsub_rn(g1b, I.nbrd[(size_t)t4 * K + lane]) : 0.0;
                const unsigned stop5 = __ballot_sync(FULL2, lane >= K || !(g2 > 0.0));
                const int R5 = stop5 ? __ffs(stop5) - 1 : 32;
                int hit = -1;
                Xchg X;
                if (lane < R5 && t5 != t3) {
#pragma unroll
                    for (int c6 = 0; c6 < 2 && hit < 0; ++c6) {
                        const int t6 = c6 == 0 ? succ(t5) : pred(t5);
                        if (t6 == t1) continue;
                        const double gain = __dsub_rn(__dadd_rn(g2, ls3_d64(xy, t5, t6)), ls3_d64(xy, t6, t1));
                        if (!(gain > LS_GAIN)) continue;
                        const int c[6] = {t1, t2, t3, t4, t5, t6};
                        if (ls3_plan<3>(M, n, c, X)) hit = c6;
                    }
                }
                const unsigned hm = __ballot_sync(FULL2, hit >= 0);
                if (hm) {
                    const int src = __ffs(hm) - 1;
                    const Xchg Y = ls3_bcast(X, src);
                    const int w5 = __shfl_sync(FULL2, t5, src);
                    const int w6 = __shfl_sync(FULL2, hit == 0 ? succ(t5) : hit == 1 ? pred(t5) : 0, src);
                    ls3_apply(M, Y);
                    if (lane == 0) {
                        M.dlb[t1] = 0; M.dlb[t2] = 0; M.dlb[t3] = 0; M.dlb[t4] = 0; M.dlb[w5] = 0; M.dlb[w6] = 0;
                    }
                    __syncwarp();
                    return true;
                }
            }
        }
    }
    return false;
}

// ---------------------------------------------------------------------------
// Directed 2-opt for the ATSP (Sec. III-D; the reading of the Jonker-Volgenant
// based 2-opt): the move removes two arcs, adds two arcs and reverses the
// path between them, so its gain adds the path's forward arc sum F and
// subtracts its backward sum R.  Examined city a, successor side first:
//   a+ = succ(a), b over nbr(a) while g1 = c(a,a+) - c(a,b) > 0 (b = a+ or
//   succ(b) = a skipped): remove (a,a+), (b,b+), add (a,b), (a+,b+),
//   reverse a+ .. b, gain = (((g1 + c(b,b+)) - c(a+,b+)) + F) - R;
//   predecessor side: a- = pred(a), g1 = c(a-,a) - c(a,b) (b = a- or
//   pred(b) = a skipped): remove (a-,a), (b-,b), add (a-,b-), (a,b), reverse
//   a .. b-, gain = (((g1 + c(b-,b)) - c(a-,b-)) + F) - R.
// F and R are summed in the order of the tour length (arc k of the path into
// lane k mod 32, then the pairwise tree), the path always reversed in place.

__device__ __forceinline__ double ls_arc(const DevInst &I, int n, int u, int v)
{
    return (double)I.cost[(size_t)u * n + v];
}

// forward (backward = false) or backward arc sum of the path of len cities
// starting at position i0 (whole warp, every lane gets the result)
__device__ __forceinline__ double ls_path_cost(const DevInst &I, const LsMem &M, int n, int i0, int len, bool backward)
{
    const int lane = threadIdx.x & 31;
    double P = 0.0;
    for (int k = lane; k + 1 < len; k += 32) {
        int p0 = i0 + k, p1 = i0 + k + 1;
        if (p0 >= n) p0 -= n;
        if (p1 >= n) p1 -= n;
        const int u = M.tour[p0], v = M.tour[p1];
        P = __dadd_rn(P, backward ? ls_arc(I, n, v, u) : ls_arc(I, n, u, v));
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) P = __dadd_rn(P, __shfl_xor_sync(FULL2, P, o));
    return P;
}

// reverses positions i0 .. i0+len-1 (cyclic) in place (whole warp)
__device__ __forceinline__ void ls_reverse_path(const LsMem &M, int n, int i0, int len)
{
    const int lane = threadIdx.x & 31;
    __syncwarp();
    for (int t = lane; t < len / 2; t += 32) {
        int p = i0 + t, q = i0 + len - 1 - t;
        if (p >= n) p -= n;
        if (q >= n) q -= n;
        const int u = M.tour[p], v = M.tour[q];
        M.tour[p] = v;
        M.tour[q] = u;
        M.pos[v] = p;
        M.pos[u] = q;
    }
    __syncwarp();
}

__device__ __forceinline__ bool ls2d_examine(const DevInst &I, const LsMem &M, int n, int K, int a)
{
    const int lane = threadIdx.x & 31;
    for (int dir = 0; dir < 2; ++dir) {
        const int pa = M.pos[a];
        const int x = dir == 0 ? M.tour[pa + 1 == n ? 0 : pa + 1] : M.tour[pa == 0 ? n - 1 : pa - 1];
        const double cx = dir == 0 ? ls_arc(I, n, a, x) : ls_arc(I, n, x, a);
        const int bl = lane < K ? I.nbr[(size_t)a * K + lane] : 0;
        const double g1l = lane < K ? __dsub_rn(cx, I.nbrd[(size_t)a * K + lane]) : 0.0;
        const unsigned stop = __ballot_sync(FULL2, lane >= K || !(g1l > 0.0));
        const int Q = stop ? __ffs(stop) - 1 : 32;
        for (int q = 0; q < Q; ++q) {
            const int b = __shfl_sync(FULL2, bl, q);
            const double g1 = __shfl_sync(FULL2, g1l, q);
            const int pb = M.pos[b];
            const int y = dir == 0 ? M.tour[pb + 1 == n ? 0 : pb + 1] : M.tour[pb == 0 ? n - 1 : pb - 1];
            if (b == x || y == a) continue;
            const int i0 = dir == 0 ? M.pos[x] : pa;
            const int i1 = dir == 0 ? pb : M.pos[y];
            int len = i1 - i0;
            if (len < 0) len += n;
            len += 1;
            const double F = ls_path_cost(I, M, n, i0, len, false);
            const double R = ls_path_cost(I, M, n, i0, len, true);
            const double cby = dir == 0 ? ls_arc(I, n, b, y) : ls_arc(I, n, y, b);
            const double gain = __dsub_rn(__dadd_rn(__dsub_rn(__dadd_rn(g1, cby), ls_arc(I, n, x, y)), F), R);
            if (gain > LS_GAIN) {
                ls_reverse_path(M, n, i0, len);
                if (lane == 0) { M.dlb[a] = 0; M.dlb[x] = 0; M.dlb[b] = 0; M.dlb[y] = 0; }
                __syncwarp();
                return true;
            }
        }
    }
    return false;
}

// passes and rounds of the neighbour-list searches with don't-look bits
// (as the 2-opt): examine(a) finds and applies one move of city a
template <typename Examine>
__device__ __forceinline__ void ls_rounds(const LsMem &M, int n, Examine &&examine)
{
    const int lane = threadIdx.x & 31;
    const long long max_moves = 64LL * n + 1024;
    long long moves = 0;
    int round_moves;
    do {
        round_moves = 0;
        for (int p = lane; p < n; p += 32) M.dlb[p] = 0;
        __syncwarp();
        bool improved = true;
        while (improved && moves < max_moves) {
            improved = false;
            int p = 0;
            while (p < n && moves < max_moves) {
                const int pp = p + lane;
                const bool clear = pp < n && !M.dlb[M.tour[pp]];
                const unsigned cm = __ballot_sync(FULL2, clear);
                if (!cm) { p += 32; continue; }
                p += __ffs(cm) - 1;
                const int a = M.tour[p];
                for (;;) {
                    if (!examine(a)) break;
                    improved = true;
                    ++round_moves;
                    ++moves;
                    if (moves >= max_moves) break;
                }
                if (lane == 0) M.dlb[a] = 1;
                __syncwarp();
                ++p;
            }
        }
    } while (round_moves > 0 && moves < max_moves);
}

// Improves the ATSP `tour` (global memory) in place by the directed 2-opt.
static __device__ __noinline__ void warp_two_opt_directed(const DevInst &I, int32_t *tour, const LsMem &Mref)
{
    const LsMem M = Mref;   // a local copy: see warp_two_opt_body
    const int lane = threadIdx.x & 31;
    const int n = I.n, K = I.ls_k;
    if (M.tour != tour)
        for (int p = lane; p < n; p += 32) M.tour[p] = tour[p];
    __syncwarp();
    for (int p = lane; p < n; p += 32) M.pos[M.tour[p]] = p;
    __syncwarp();
    ls_rounds(M, n, [&](int a) { return ls2d_examine(I, M, n, K, a); });
    if (M.tour != tour)
        for (int p = lane; p < n; p += 32) tour[p] = M.tour[p];
    __syncwarp();
}

// the 2-opt of the instance's kind: symmetric (twoopt.cuh) or directed
static __device__ __forceinline__ void warp_two_opt_any(const DevInst &I, int32_t *tour, const LsMem &M)
{
    if (I.kind == 1) warp_two_opt_directed(I, tour, M);
    else warp_two_opt(I, tour, M);
}

// Improves `tour` (global memory) in place; M as for warp_two_opt (its el
// array serves as the scratch of the middle rewrite).
__device__ __forceinline__ void warp_three_opt_body(const DevInst &I, int32_t *tour, const LsMem &M)
{
    const int lane = threadIdx.x & 31;
    const int n = I.n, K = I.ls_k;
    if (M.tour != tour)
        for (int p = lane; p < n; p += 32) M.tour[p] = tour[p];
    __syncwarp();
    for (int p = lane; p < n; p += 32) M.pos[M.tour[p]] = p;
    __syncwarp();
    ls_rounds_ahead<true, false>(M, n, K, 1, [&](int a) { return ls3_scan(M, n, K, a); },
                    [&](const LsMove &F) { ls3_apply_move(M, n, F); }, [&](int a) { return ls3_examine(I, M, n, K, a); });
    if (M.tour != tour)
        for (int p = lane; p < n; p += 32) tour[p] = M.tour[p];
    __syncwarp();
}

// the same as a call (the cluster kernel)
static __device__ __noinline__ void warp_three_opt(const DevInst &I, int32_t *tour, const LsMem &Mref)
{
    const LsMem M = Mref;
    warp_three_opt_body(I, tour, M);
}

// The search of a symmetric instance by a whole block (every thread calls it):
// `tour` improved in place, warp 0 in control, the other warps helping.
__device__ __forceinline__ void block_search(const DevInst &I, int32_t *tour, const LsMem &M)
{
    const int n = I.n, K = I.ls_k;
    if (M.tour != tour)
        for (int p = threadIdx.x; p < n; p += blockDim.x) M.tour[p] = tour[p];
    __syncthreads();
    for (int p = threadIdx.x; p < n; p += blockDim.x) M.pos[M.tour[p]] = p;
    __syncthreads();
    if (threadIdx.x >= 32) {
        ls_coop_help(I, M);
    } else {
        if (I.local_search >= 3)
            ls_rounds_ahead<true, true>(M, n, K, M.coop_warps, [&](int a) { return ls3_scan(M, n, K, a); },
                                  [&](const LsMove &F) { ls3_apply_move(M, n, F); },
                                  [&](int a) { return ls3_examine(I, M, n, K, a); });
        else
            ls_rounds_ahead<false, true>(M, n, K, M.coop_warps, [&](int a) { return ls2_scan(M, n, K, a); },
                                   [&](const LsMove &F) { ls2_apply(M, n, F); },
                                   [&](int a) {
                                       const LsMove F = ls2_exact(I, M, n, K, a);
                                       if (F.st) ls2_apply(M, n, F);
                                       return F.st != 0;
                                   });
        ls_coop_end(M);
    }
    __syncthreads();
    if (M.tour != tour)
        for (int p = threadIdx.x; p < n; p += blockDim.x) tour[p] = M.tour[p];
    __syncthreads();
}

// The local search of T_NN and T_ib, a block of several warps per tour, with
// its arrays in the block's shared memory where they fit.  The case that all
// of them fit has code of its own, in which the compiler knows their address
// space: through pointers that may be either, an n = 10000 search took 11.3 ms
// instead of 8.7.
__device__ __forceinline__ void block_local_search(const DevInst &I, int32_t *tour, unsigned char *sm, size_t smem_bytes,
                                                   int *coop)
{
    const int warps = (int)(blockDim.x >> 5);
    if (I.kind == 1) {                 // directed: one warp, no helpers
        if (threadIdx.x < 32) warp_two_opt_directed(I, tour, ls_shared(I, sm, smem_bytes, ls_global(I, tour)));
        __syncthreads();
    } else if (ls_smem_full(I.n) <= smem_bytes) {
        LsMem M = ls_shared_full(I, sm);
        float2 *sxy = reinterpret_cast<float2 *>(sm + ls_xy_offset(I.n));
        for (int p = threadIdx.x; p < I.n; p += blockDim.x) sxy[p] = reinterpret_cast<const float2 *>(I.xy)[p];
        M.coop = coop;
        M.coop_warps = warps;
        block_search(I, tour, M);
    } else {
        LsMem M = ls_shared(I, sm, smem_bytes, ls_global(I, tour));
        M.coop = coop;
        M.coop_warps = warps;
        block_search(I, tour, M);
    }
}

}  // namespace hac
