// First-improvement 2-opt with geometric neighbour lists and don't-look bits
// (Sec. III-D), applied to T_NN once (Algorithm 1's initialisation) and to the
// iteration-best tour or every ant's tour before they update the pheromone.
//
// Order of the search (it defines the result):
//   rounds start with all bits clear; a round repeats passes over the tour
//   positions until a pass makes no move; the search ends after a round whose
//   first pass made no move (a local optimum of the neighbour-list moves).
//   For city a, the successor direction is tried first, then the predecessor
//   direction; b runs over nbr(a) in (d, j) order while d(a, b) < d(a, dir a);
//   the first move with gain > 1e-10 is applied, the bits of a, dir a, b and
//   dir b are cleared and a is examined again; a city without a move gets its
//   bit set.  A move replacing (a, succ a), (b, succ b) by (a, b), (succ a,
//   succ b) reverses positions pos(succ a)..pos(b), or pos(succ b)..pos(a) when
//   the first range is longer than n/2; a predecessor move is the successor
//   move of (pred a, pred b).  A call stops after 64n + 1024 moves (a bound
//   that strictly decreasing tour lengths never reach in practice), so the
//   kernel always terminates.
//
// Moves follow the FP64 gain (d_ij as in the length, gain = (d(a,dir a) -
// d(a,b)) + d(b,dir b) - d(dir a,dir b)), but most candidates are decided from
// FP32 copies: el[p] holds d(tour[p], tour[p+1]) in FP32 and nbrd32 the
// neighbour distances.  Each FP32 distance is within 5 units of 2^-24 (relative) of the
// FP64 one, so the FP32 estimate of the four-term gain is within about
// 9 * 2^-24 of the sum of the four magnitudes.  With tol = 4e-6 times that
// sum (plus 1e-18 for FP32 underflow), an estimate below 1e-10 - tol means the
// FP64 gain is certainly <= 1e-10, one above 1e-10 + tol that it is certainly
// above; only estimates in between are decided in FP64.  Likewise d(a, b) is
// compared with d(a, dir a) in FP32 with a relative margin of 4e-6 on either
// side.  The moves taken are therefore exactly those of the plain FP64 search;
// the FP32 edge lengths stored for the new edges are FP32 estimates too.
//
// Parallelism inside the sequential search, on one warp (every ant's tour;
// the cluster kernel): when more than LS_FEW of the next 32 tour positions
// hold cities whose bit is clear, a pass tests them at once with the FP32 test
// only, their candidate moves spread over the lanes; the cities before the
// first one that might move have no move and get their bit at once (as they
// would one by one, since examining a city without a move changes nothing
// else).  A city that might move, or the first clear one when few are clear, is
// examined by the whole warp, one neighbour per lane (FP32 classes, then FP64
// when the first candidate is undecided).  Segment reversals swap element
// pairs across lanes.
//
// On a block of several warps (T_NN and T_ib in kernels of their own): every
// warp examines one city (ls2_scan: a neighbour per lane, both directions), the
// next clear cities in tour order at once, so that one round of the block finds
// the first city with a move and, unless FP32 leaves it undecided, the move
// itself; all warps share long reversals.  Moves are dense (4200 moves in 7300
// rounds per search of an n = 10000 iteration-best tour), so the search is a
// chain of rounds (740 cycles to find the next clear cities, 1150 to examine
// them) and moves (760), and its latency is what counts: testing 32 cities' moves
// on all warps and then examining the first candidate took 18.4 ms per search,
// this takes 8.2 ms.
#pragma once

#include "lengths.cuh"

namespace hac {

constexpr unsigned FULL2 = 0xffffffffu;
constexpr float LS_G1_LO = 0.999996f;   // FP32 margin between d(a,b) and d(a,dir a): g1 <= 0 or > 0 for certain
constexpr int LS_FEW = 4;               // at most this many clear cities in 32 positions: one at a time

__device__ __forceinline__ int wrap_next(int p, int n) { return p + 1 < n ? p + 1 : 0; }
__device__ __forceinline__ int wrap_prev(int p, int n) { return p > 0 ? p - 1 : n - 1; }

// bring the cache lines of a global row of `bytes` bytes into L1 (no result)
__device__ __forceinline__ void ls_prefetch_row(const void *row, int bytes)
{
    asm volatile("prefetch.global.L1 [%0];" ::"l"(row));
    asm volatile("prefetch.global.L1 [%0];" ::"l"(static_cast<const char *>(row) + bytes - 1));
}

// the arrays of one search: shared memory (a kernel of its own) or the workspace
struct LsMem {
    int32_t *tour;      // the tour being improved
    int32_t *pos;       // pos[city]
    uint8_t *dlb;       // don't-look bit by city
    float *el;          // el[p] ~ d(tour[p], tour[p+1 mod n]), FP32
    const float2 *xy;   // coordinates
    const int32_t *nbr = nullptr;     // neighbour lists and their FP32 distances, copied here because a
    const float *nbrd32 = nullptr;    // pointer read through the instance is read again after every store
    int *coop = nullptr;   // shared command words of the helper warps (null: warp 0 alone)
    int coop_warps = 1;    // warps of the block (warp 0 searches, the others help)
};

// Helper warps.  The search is sequential and its control runs in warp 0; in
// a block of several warps the others wait at named barrier 1 and examine
// cities and take their share of each long segment reversal (its element pairs
// are independent, so the result does not depend on who swaps which pair).
// Protocol: warp 0 writes a command to coop and every warp arrives at the
// barrier; then
//   1 (reverse i0 .. i0+len-1): every warp swaps its pairs, arrives again;
//   2 (examine up to `warps` cities): warp w examines the w-th staged city and
//     writes what it found; every warp arrives again;
//   3 (3-opt: rewrite the middle of an exchange): every warp copies its share
//     out, arrives, copies it back in, arrives;
//   0: the helpers return.
// Every path through the search ends with command 0.
constexpr int LS_COOP_LEN = 192;   // reversals of at least this many positions are shared
constexpr int LS_WARPS_MAX = 8;
// coop words: [0] command, [1] i0 or city count, [2] len; the staged cities and
// their positions; the moves found (8 words each); the exchange (8)
constexpr int LS_ST = 4, LS_POS = LS_ST + LS_WARPS_MAX + 1, LS_MOVES = LS_POS + LS_WARPS_MAX + 1,
              LS_XCHG = LS_MOVES + 8 * LS_WARPS_MAX, LS_COOP_WORDS = LS_XCHG + 8;

__device__ __forceinline__ void ls_coop_bar(int warps)
{
    asm volatile("bar.sync 1, %0;" ::"r"(32 * warps) : "memory");
}

__device__ __forceinline__ float ls_d32(const float2 *xy, int u, int v)
{
    const float2 p = xy[u], q = xy[v];
    const float dx = __fsub_rn(q.x, p.x), dy = __fsub_rn(q.y, p.y);
    return __fsqrt_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)));
}

// FP32 distance with the approximate square root (error at most 2^-23 of it):
// within 5 units of 2^-24, far inside the 4e-6 bands
__device__ __forceinline__ float ls_da32(float2 p, float2 q)
{
    const float dx = __fsub_rn(q.x, p.x), dy = __fsub_rn(q.y, p.y);
    float r;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy))));
    return r;
}

// the FP64 gain from FP32 estimates of its terms: 0 certainly <= LS_GAIN,
// 2 certainly above, 1 undecided
__device__ __forceinline__ int ls_gain_class(float da, float dab, float dbb, float dn)
{
    const float est = __fsub_rn(__fadd_rn(__fsub_rn(da, dab), dbb), dn);
    const float mag = __fadd_rn(__fadd_rn(da, dab), __fadd_rn(dbb, dn));
    const float tol = __fadd_rn(__fmul_rn(4e-6f, mag), 1e-18f);
    if (!(est > __fsub_rn((float)LS_GAIN, tol))) return 0;
    return est > __fadd_rn((float)LS_GAIN, tol) ? 2 : 1;
}

// false only if the FP64 gain is certainly <= LS_GAIN
__device__ __forceinline__ bool ls_may_improve(float da, float dab, float dbb, float dn)
{
    return ls_gain_class(da, dab, dbb, dn) != 0;
}

// the element swaps of reversing positions i0 .. i0+len-1 (mod n) that fall to
// thread `tid` of `nth`: tour/pos pairs and the inner edge lengths; the pairs
// of different t are disjoint, so each thread loads two pairs before it
// stores them (EL false: the edge lengths are not kept)
template <bool EL>
__device__ __forceinline__ void ls_reverse_part(const LsMem &M, int n, int i0, int len, int tid, int nth)
{
    const int h = len / 2;
    for (int t = tid; t < h; t += 2 * nth) {
        const bool two = t + nth < h;
        int p0 = i0 + t, q0 = i0 + len - 1 - t;
        int p1 = p0 + nth, q1 = q0 - nth;
        if (p0 >= n) p0 -= n;
        if (q0 >= n) q0 -= n;
        if (p1 >= n) p1 -= n;
        if (q1 >= n) q1 -= n;
        const int u0 = M.tour[p0], v0 = M.tour[q0];
        const int u1 = two ? M.tour[p1] : 0, v1 = two ? M.tour[q1] : 0;
        M.tour[p0] = v0;
        M.tour[q0] = u0;
        M.pos[v0] = p0;
        M.pos[u0] = q0;
        if (two) {
            M.tour[p1] = v1;
            M.tour[q1] = u1;
            M.pos[v1] = p1;
            M.pos[u1] = q1;
        }
    }
    const int he = EL ? (len - 1) / 2 : 0;
    for (int t = tid; t < he; t += 2 * nth) {
        const bool two = t + nth < he;
        int p0 = i0 + t, q0 = i0 + len - 2 - t;
        int p1 = p0 + nth, q1 = q0 - nth;
        if (p0 >= n) p0 -= n;
        if (q0 >= n) q0 -= n;
        if (p1 >= n) p1 -= n;
        if (q1 >= n) q1 -= n;
        const float u0 = M.el[p0], v0 = M.el[q0];
        const float u1 = two ? M.el[p1] : 0.0f, v1 = two ? M.el[q1] : 0.0f;
        M.el[p0] = v0;
        M.el[q0] = u0;
        if (two) {
            M.el[p1] = v1;
            M.el[q1] = u1;
        }
    }
}

// One pre-test work item: candidate move of city a in direction dir (0: succ,
// 1: pred) with its q-th neighbour; true unless the FP64 gain is certainly
// <= LS_GAIN.  an, da: the city's dir-neighbour and FP32 edge length.
__device__ __forceinline__ bool ls_item_may_improve(const LsMem &M, int n, int K, int a, int dir,
                                                   int q, int an, float da)
{
    const int b = M.nbr[(size_t)a * K + q];
    const float dab = M.nbrd32[(size_t)a * K + q];
    const int pb = M.pos[b];
    const int pe = dir == 0 ? pb : wrap_prev(pb, n);     // the edge (b, dir b)
    const int bn = M.tour[dir == 0 ? wrap_next(pb, n) : pe];
    return b != an && bn != a && ls_may_improve(da, dab, M.el[pe], ls_da32(M.xy[an], M.xy[bn]));
}

// What the examination of a city in FP32 found: st 0 no move; 1 the city's
// first move, certain; 2 a possible move, undecided.  2-opt: r is the direction
// (0 successor) and c = a, dir a, b, dir b; 3-opt: c = t1..t4 (r = 2) or t1..t6
// (r = 3).
struct LsMove {
    int st, r, c[6];
};

__device__ __forceinline__ LsMove ls3_scan(const LsMem &M, int n, int K, int a);
__device__ __forceinline__ void ls3_coop_rewrite(const LsMem &M);

// One city's 2-opt moves in FP32 (whole warp, only reads, the same result in
// every lane): a neighbour per lane, both directions.
__device__ __forceinline__ LsMove ls2_scan(const LsMem &M, int n, int K, int a)
{
    const int lane = threadIdx.x & 31;
    const int b = lane < K ? M.nbr[(size_t)a * K + lane] : a;
    const float nd = lane < K ? M.nbrd32[(size_t)a * K + lane] : __int_as_float(0x7f800000);
    const int pa = M.pos[a];
    const int an0 = M.tour[wrap_next(pa, n)], an1 = M.tour[wrap_prev(pa, n)];
    const float2 xa = M.xy[a], x0 = M.xy[an0], x1 = M.xy[an1];
    const float da0 = ls_da32(xa, x0), da1 = ls_da32(xa, x1);
    const float lim = __fmul_rn(nd, LS_G1_LO);
    const int pb = M.pos[b];
    const int bn0 = M.tour[wrap_next(pb, n)], bn1 = M.tour[wrap_prev(pb, n)];
    const float2 xb = M.xy[b], y0 = M.xy[bn0], y1 = M.xy[bn1];
    const int g0 = ls_gain_class(da0, nd, ls_da32(xb, y0), ls_da32(x0, y0));
    const int g1 = ls_gain_class(da1, nd, ls_da32(xb, y1), ls_da32(x1, y1));
    const bool c0 = (da0 > lim) & (g0 != 0) & (b != an0) & (bn0 != a);
    const bool c1 = (da1 > lim) & (g1 != 0) & (b != an1) & (bn1 != a);
    const unsigned m0 = __ballot_sync(FULL2, c0), m1 = __ballot_sync(FULL2, c1);
    LsMove F;
    F.st = 0;
    F.r = m0 ? 0 : 1;
#pragma unroll
    for (int k = 0; k < 6; ++k) F.c[k] = a;
    if (!(m0 | m1)) return F;
    const int src = __ffs(m0 ? m0 : m1) - 1;
    const bool sure = m0 ? (g0 == 2) & (__fmul_rn(da0, LS_G1_LO) > nd) : (g1 == 2) & (__fmul_rn(da1, LS_G1_LO) > nd);
    F.st = __shfl_sync(FULL2, sure ? 1 : 2, src);
    F.c[1] = m0 ? an0 : an1;
    F.c[2] = __shfl_sync(FULL2, b, src);
    F.c[3] = __shfl_sync(FULL2, m0 ? bn0 : bn1, src);
    return F;
}

// the same city in FP64, when FP32 left its first candidate undecided: the
// first improving move in order (st 0 or 1)
static __device__ __noinline__ LsMove ls2_exact(const DevInst &I, const LsMem &M, int n, int K, int a)
{
    const int lane = threadIdx.x & 31;
    const int b = lane < K ? I.nbr[(size_t)a * K + lane] : a;
    const double nd = lane < K ? I.nbrd[(size_t)a * K + lane] : 0.0;
    const int pa = M.pos[a], pb = M.pos[b];
    LsMove F;
    F.st = 0;
    F.r = 0;
#pragma unroll
    for (int k = 0; k < 6; ++k) F.c[k] = a;
    for (int dir = 0; dir < 2 && !F.st; ++dir) {
        const int an = M.tour[dir == 0 ? wrap_next(pa, n) : wrap_prev(pa, n)];
        const int bn = M.tour[dir == 0 ? wrap_next(pb, n) : wrap_prev(pb, n)];
        bool ok = false;
        if (lane < K && b != an && bn != a) {
            const double g1 = __dsub_rn(dist64(I, a, an), nd);
            if (g1 > 0.0) ok = __dsub_rn(__dadd_rn(g1, dist64(I, b, bn)), dist64(I, an, bn)) > LS_GAIN;
        }
        const unsigned m = __ballot_sync(FULL2, ok);
        if (!m) continue;
        const int src = __ffs(m) - 1;
        F.st = 1;
        F.r = dir;
        F.c[1] = an;
        F.c[2] = __shfl_sync(FULL2, b, src);
        F.c[3] = __shfl_sync(FULL2, bn, src);
    }
    return F;
}

// command 2, every warp of the block: the warp's staged city
__device__ __forceinline__ void ls_coop_scan(const LsMem &M, int n, int K, bool three)
{
    const int w = threadIdx.x >> 5;
    if (w >= M.coop[1]) return;
    const int a = M.coop[LS_ST + w];
    const LsMove F = three ? ls3_scan(M, n, K, a) : ls2_scan(M, n, K, a);
    if ((threadIdx.x & 31) == 0) {
        int *o = M.coop + LS_MOVES + 8 * w;
        o[0] = F.st;
        o[1] = F.r;
#pragma unroll
        for (int k = 0; k < 6; ++k) o[2 + k] = F.c[k];
    }
    __syncwarp();
}

// the helper warps' side of the protocol above (warps 1 .. coop_warps-1)
__device__ __forceinline__ void ls_coop_help(const DevInst &I, const LsMem &Mref)
{
    const LsMem M = Mref;
    const int n = I.n, K = I.ls_k, nth = 32 * M.coop_warps;
    const bool three = I.local_search >= 3;
    for (;;) {
        ls_coop_bar(M.coop_warps);
        const int cmd = M.coop[0];
        if (cmd == 1) {
            ls_reverse_part<false>(M, n, M.coop[1], M.coop[2], (int)threadIdx.x, nth);
            ls_coop_bar(M.coop_warps);
        } else if (cmd == 2) {
            ls_coop_scan(M, n, K, three);
            ls_coop_bar(M.coop_warps);
        } else if (cmd == 3) {
            ls3_coop_rewrite(M);
        } else {
            break;
        }
    }
}

template <int V>
struct LsInt {
    static constexpr int value = V;
};

// The passes and rounds of a search with don't-look bits, its cities examined
// W at a time by the block's warps (AHEAD), or one at a time by this warp alone.  Cities
// without a move are examined in any order with the same outcome, so the next
// W clear cities in tour order are examined at once and the first with a move
// is taken; the others are examined again after it.
//   scan(a)  the examination of one city; exact(a, F) decides an undecided one:
//   it makes the move and returns true, or returns false; apply(F) makes a
//   certain one.  Both clear the bits of the move's cities.
template <bool THREE, bool AHEAD, typename Scan, typename Apply, typename Exact>
__device__ __forceinline__ void ls_rounds_ahead(const LsMem &M, int n, int K, int W, Scan &&scan, Apply &&apply,
                                                Exact &&exact)
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
            int p = 0, cur = -1;      // next position of the pass; city to examine again after its move
            while (moves < max_moves) {
                // the next cities in order: cur, then the clear ones from position p on
                int cnt = cur >= 0 ? 1 : 0, city = cur, where = p - 1, q = p;
                if constexpr (AHEAD) {
                    // staged in coop with their positions: 64 positions first (cities are
                    // dense early in a search), then 256 at a time, the loads of a group
                    // in flight together; the slot past the last takes what is not wanted
                    if (cur >= 0 && lane == 0) { M.coop[LS_ST] = cur; M.coop[LS_POS] = p - 1; }
                    auto gather = [&](auto windows) {
                        constexpr int G = decltype(windows)::value;
                        int u[G];
                        unsigned cm[G];
#pragma unroll
                        for (int j = 0; j < G; ++j) u[j] = M.tour[min(q + 32 * j + lane, n - 1)];
#pragma unroll
                        for (int j = 0; j < G; ++j) {
                            const bool clear = (q + 32 * j + lane < n) & (u[j] != cur) & (M.dlb[u[j]] == 0);
                            cm[j] = __ballot_sync(FULL2, clear);
                        }
#pragma unroll
                        for (int j = 0; j < G; ++j)
                            if (cm[j]) {
                                const int d = cnt + __popc(cm[j] & ((1u << lane) - 1u));
                                const int slot = ((cm[j] >> lane) & 1u) && d < W ? d : LS_WARPS_MAX;
                                M.coop[LS_ST + slot] = u[j];
                                M.coop[LS_POS + slot] = q + 32 * j + lane;
                                cnt += __popc(cm[j]);
                            }
                        q += 32 * G;
                    };
                    if (cnt < W && q < n) gather(LsInt<2>{});
                    while (cnt < W && q < n) gather(LsInt<8>{});
                    __syncwarp();
                    cnt = min(cnt, W);
                    if (lane < cnt) { city = M.coop[LS_ST + lane]; where = M.coop[LS_POS + lane]; }
                } else {
                    for (; !cnt && q < n; q += 32) {
                        const int pp = q + lane;
                        const int u = pp < n ? M.tour[pp] : 0;
                        const unsigned cm = __ballot_sync(FULL2, pp < n && !M.dlb[u]);
                        if (!cm) continue;
                        where = q + __ffs(cm) - 1;
                        city = __shfl_sync(FULL2, u, __ffs(cm) - 1);
                        cnt = 1;
                    }
                }
                if (!cnt) break;
                LsMove F;
                int f = 0;            // the first of them with a possible move
                if (AHEAD && cnt > 1) {
                    if (lane == 0) { M.coop[0] = 2; M.coop[1] = cnt; }
                    __syncwarp();
                    ls_coop_bar(M.coop_warps);
                    ls_coop_scan(M, n, K, THREE);
                    ls_coop_bar(M.coop_warps);
                    const unsigned hm = __ballot_sync(FULL2, lane < cnt && M.coop[LS_MOVES + 8 * (lane < cnt ? lane : 0)] != 0);
                    f = hm ? __ffs(hm) - 1 : cnt;
                    const int *o = M.coop + LS_MOVES + 8 * (hm ? f : 0);
                    F.st = hm ? o[0] : 0;
                    F.r = o[1];
#pragma unroll
                    for (int k = 0; k < 6; ++k) F.c[k] = o[2 + k];
                } else {
                    F = scan(__shfl_sync(FULL2, city, 0));
                    f = F.st ? 0 : cnt;
                }
                if (lane < cnt && lane < f) M.dlb[city] = 1;      // examined, no move
                __syncwarp();
                if (!F.st) {          // none of them moves
                    p = __shfl_sync(FULL2, where, cnt - 1) + 1;
                    cur = -1;
                    continue;
                }
                const int a = __shfl_sync(FULL2, city, f);
                p = __shfl_sync(FULL2, where, f) + 1;
                bool moved = true;
                if (F.st == 1) apply(F);
                else moved = exact(a);
                if (moved) {
                    improved = true;
                    ++round_moves;
                    ++moves;
                    cur = a;
                } else {
                    if (lane == 0) M.dlb[a] = 1;
                    __syncwarp();
                    cur = -1;
                }
            }
        }
    } while (round_moves > 0 && moves < max_moves);
}

// warp 0: releases the helper warps (the final arrival of the protocol)
__device__ __forceinline__ void ls_coop_end(const LsMem &M)
{
    if (!M.coop) return;
    if ((threadIdx.x & 31) == 0) M.coop[0] = 0;
    __syncwarp();
    ls_coop_bar(M.coop_warps);
}

// the shorter range whose reversal turns (x, succ x), (y, succ y) into (x, y),
// (succ x, succ y)
__device__ __forceinline__ void ls_move_range(const LsMem &M, int n, int x, int y, int &i0, int &len)
{
    i0 = wrap_next(M.pos[x], n);
    len = M.pos[y] - i0;
    if (len < 0) len += n;
    len += 1;
    if (2 * len > n) {
        i0 = wrap_next(M.pos[y], n);
        len = M.pos[x] - i0;
        if (len < 0) len += n;
        len += 1;
    }
}

// one warp alone: reverses, the inner edges of the range swap, the two new
// edges get dxy, dss
__device__ __forceinline__ void apply_succ_move(const LsMem &M, int n, int x, int y, float dxy, float dss)
{
    const int lane = threadIdx.x & 31;
    int i0, len;
    ls_move_range(M, n, x, y, i0, len);
    __syncwarp();
    ls_reverse_part<true>(M, n, i0, len, lane, 32);
    __syncwarp();
    if (lane == 0) {
        M.el[wrap_prev(i0, n)] = dxy;
        int e = i0 + len - 1;
        if (e >= n) e -= n;
        M.el[e] = dss;
    }
    __syncwarp();
}

// warp 0 of a block with helpers: makes the move F (ls2_scan) and clears its
// cities' bits; no edge lengths are kept
__device__ __forceinline__ void ls2_apply(const LsMem &M, int n, const LsMove &F)
{
    const int lane = threadIdx.x & 31;
    int i0, len;
    if (F.r == 0) ls_move_range(M, n, F.c[0], F.c[2], i0, len);
    else ls_move_range(M, n, F.c[1], F.c[3], i0, len);
    __syncwarp();
    if (len >= LS_COOP_LEN) {
        if (lane == 0) { M.coop[0] = 1; M.coop[1] = i0; M.coop[2] = len; }
        __syncwarp();
        ls_coop_bar(M.coop_warps);
        ls_reverse_part<false>(M, n, i0, len, lane, 32 * M.coop_warps);
        ls_coop_bar(M.coop_warps);
    } else {
        ls_reverse_part<false>(M, n, i0, len, lane, 32);
    }
    if (lane < 4) M.dlb[lane == 0 ? F.c[0] : lane == 1 ? F.c[1] : lane == 2 ? F.c[2] : F.c[3]] = 0;
    __syncwarp();
}

// FP32 pre-test of the clear cities of 32 consecutive positions (lane l holds
// the city al at position pp = p + l): the lane of the first city that might
// move, or 32.  A work item is one candidate move of one city: a direction and
// a neighbour b while d(a, b) is below d(a, dir a) (FP32, with the margin);
// the list ascends, so each direction's items are a prefix of the list.  The
// items of all cities are dealt to the lanes in position order, 32 at a time;
// after the first group with a possible move every earlier city has been
// tested in full, so the search stops there.
__device__ __forceinline__ int ls_first_may_move(const LsMem &M, int n, int K, bool clear, int al, int pp)
{
    const int lane = threadIdx.x & 31;
    int an0 = 0, an1 = 0, c0 = 0, c1 = 0;
    float da0 = 0.0f, da1 = 0.0f;
    if (clear) {
        const int pv = wrap_prev(pp, n);
        an0 = M.tour[wrap_next(pp, n)];
        an1 = M.tour[pv];
        da0 = M.el[pp];
        da1 = M.el[pv];
        ls_prefetch_row(M.nbr + (size_t)al * K, K * 4);      // read by the work items below
        const float *nd = M.nbrd32 + (size_t)al * K;
        for (int k0 = 0; k0 < K; k0 += 4) {
            float lim[4];
#pragma unroll
            for (int q = 0; q < 4; ++q)
                lim[q] = k0 + q < K ? __fmul_rn(nd[k0 + q], LS_G1_LO) : __int_as_float(0x7f800000);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                c0 += da0 > lim[q];
                c1 += da1 > lim[q];
            }
            if (!(da0 > lim[3] || da1 > lim[3])) break;
        }
    }
    const int cnt = c0 + c1;
    int incl = cnt;     // inclusive prefix sum of the item counts over the lanes
#pragma unroll
    for (int s = 1; s < 32; s <<= 1) {
        const int v = __shfl_up_sync(FULL2, incl, s);
        if (lane >= s) incl += v;
    }
    const int excl = incl - cnt;
    const int total = __shfl_sync(FULL2, incl, 31);
    for (int base = 0; base < total; base += 32) {
        const int t = base + lane;
        int c = 0;      // the lane whose city owns item t: the number of lanes with incl <= t
#pragma unroll
        for (int s = 16; s >= 1; s >>= 1)
            if (__shfl_sync(FULL2, incl, c + s - 1) <= t) c += s;
        const int j = t - __shfl_sync(FULL2, excl, c);
        const int cc0 = __shfl_sync(FULL2, c0, c);
        const int a = __shfl_sync(FULL2, al, c);
        const int xan0 = __shfl_sync(FULL2, an0, c), xan1 = __shfl_sync(FULL2, an1, c);
        const float xda0 = __shfl_sync(FULL2, da0, c), xda1 = __shfl_sync(FULL2, da1, c);
        bool hit = false;
        if (t < total) {
            const int dir = j < cc0 ? 0 : 1;
            hit = ls_item_may_improve(M, n, K, a, dir, dir == 0 ? j : j - cc0, dir == 0 ? xan0 : xan1,
                                      dir == 0 ? xda0 : xda1);
        }
        const unsigned first = __reduce_min_sync(FULL2, hit ? (unsigned)c : 32u);
        if (first < 32u) return (int)first;
    }
    return 32;
}

// One direction of city a, one neighbour per lane: the first improving move
// in list order, decided in FP64.
__device__ __forceinline__ bool ls_find_move(const DevInst &I, const LsMem &M, int n, int K, int a, int dir,
                                             int nb, float nd32, double nd64, int &an, int &b, int &bn,
                                             float &dab, float &dn)
{
    const int lane = threadIdx.x & 31;
    const int pa = M.pos[a];
    an = dir == 0 ? M.tour[wrap_next(pa, n)] : M.tour[wrap_prev(pa, n)];
    const float da32 = M.el[dir == 0 ? pa : wrap_prev(pa, n)];
    bool cand = false, sure = false;
    int bb = 0, bbn = 0;
    float dnn = 0.0f;
    if (lane < K && da32 > __fmul_rn(nd32, LS_G1_LO)) {
        bb = nb;
        const int pb = M.pos[bb];
        bbn = dir == 0 ? M.tour[wrap_next(pb, n)] : M.tour[wrap_prev(pb, n)];
        if (!(bb == an || bbn == a)) {
            const float dbb = M.el[dir == 0 ? pb : wrap_prev(pb, n)];
            dnn = ls_da32(M.xy[an], M.xy[bbn]);
            const int g = ls_gain_class(da32, nd32, dbb, dnn);
            cand = g != 0;
            sure = g == 2 && __fmul_rn(da32, LS_G1_LO) > nd32;   // and d(a, b) < d(a, dir a) for certain
        }
    }
    const unsigned cm = __ballot_sync(FULL2, cand);
    if (!cm) return false;
    int src = __ffs(cm) - 1;
    if (!((__ballot_sync(FULL2, sure) >> src) & 1u)) {
        // the first candidate is undecided in FP32: decide all of them in FP64
        const double da = dist64(I, a, an);
        bool ok = false;
        if (cand) {
            const double g1 = __dsub_rn(da, nd64);
            if (g1 > 0.0) {
                const double gain = __dsub_rn(__dadd_rn(g1, dist64(I, bb, bbn)), dist64(I, an, bbn));
                ok = gain > LS_GAIN;
            }
        }
        const unsigned om = __ballot_sync(FULL2, ok);
        if (!om) return false;
        src = __ffs(om) - 1;
    }
    b = __shfl_sync(FULL2, bb, src);
    bn = __shfl_sync(FULL2, bbn, src);
    dab = __shfl_sync(FULL2, nd32, src);
    dn = __shfl_sync(FULL2, dnn, src);
    return true;
}

// Improves `tour` (global memory) in place.  M holds the working arrays; when
// M.tour is not `tour`, the tour is copied in and back out.  The array
// pointers are copied into a local first: the search stores through generic
// pointers, and pointers read through a reference would be reloaded after
// every store.
__device__ __forceinline__ void warp_two_opt_body(const DevInst &I, int32_t *tour, const LsMem &M)
{
    const int lane = threadIdx.x & 31;
    const int n = I.n, K = I.ls_k;
    if (M.tour != tour)
        for (int p = lane; p < n; p += 32) M.tour[p] = tour[p];
    __syncwarp();
    for (int p = lane; p < n; p += 32) M.pos[M.tour[p]] = p;
    for (int p = lane; p < n; p += 32) M.el[p] = ls_d32(M.xy, M.tour[p], M.tour[wrap_next(p, n)]);
    __syncwarp();
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
                const int al = pp < n ? M.tour[pp] : 0;
                const bool clear = pp < n && !M.dlb[al];
                const unsigned cm = __ballot_sync(FULL2, clear);
                if (!cm) { p += 32; continue; }
                if (__popc(cm) <= LS_FEW) {
                    p += __ffs(cm) - 1;     // few clear cities: the warp examines the first one
                } else {
                    // many: the next 32 positions at once, FP32 test only; the
                    // lists of the 32 positions after them are warmed for the next test
                    if (pp + 32 < n) {
                        const int ah = M.tour[pp + 32];
                        ls_prefetch_row(M.nbrd32 + (size_t)ah * K, K * 4);
                        ls_prefetch_row(M.nbr + (size_t)ah * K, K * 4);
                    }
                    const int f = ls_first_may_move(M, n, K, clear, al, pp);
                    if (clear && lane < f) M.dlb[al] = 1;   // examined, no move
                    __syncwarp();
                    if (f == 32) { p += 32; continue; }
                    p += f;
                }
                const int a = M.tour[p];
                const int nb = lane < K ? M.nbr[(size_t)a * K + lane] : 0;
                const float nd32 = lane < K ? M.nbrd32[(size_t)a * K + lane] : 0.0f;
                const double nd64 = lane < K ? I.nbrd[(size_t)a * K + lane] : 0.0;
                for (;;) {
                    bool moved = false;
                    int an = 0, b = 0, bn = 0, dir = -1;
                    float dab = 0.0f, dn = 0.0f;
                    for (int d = 0; d < 2 && dir < 0; ++d)
                        if (ls_find_move(I, M, n, K, a, d, nb, nd32, nd64, an, b, bn, dab, dn)) dir = d;
                    if (dir >= 0) {
                        if (dir == 0) apply_succ_move(M, n, a, b, dab, dn);
                        else apply_succ_move(M, n, an, bn, dn, dab);
                        if (lane == 0) { M.dlb[a] = 0; M.dlb[an] = 0; M.dlb[b] = 0; M.dlb[bn] = 0; }
                        __syncwarp();
                        moved = true;
                        improved = true;
                        ++round_moves;
                        ++moves;
                    }
                    if (!moved || moves >= max_moves) break;
                }
                if (lane == 0) M.dlb[a] = 1;
                __syncwarp();
                ++p;
            }
        }
    } while (round_moves > 0 && moves < max_moves);
    if (M.tour != tour)
        for (int p = lane; p < n; p += 32) tour[p] = M.tour[p];
    __syncwarp();
}

// the same as a call (the cluster kernel)
static __device__ __noinline__ void warp_two_opt(const DevInst &I, int32_t *tour, const LsMem &Mref)
{
    const LsMem M = Mref;
    warp_two_opt_body(I, tour, M);
}

// the workspace arrays of an instance (no shared memory)
__device__ __forceinline__ LsMem ls_global(const DevInst &I, int32_t *tour)
{
    return LsMem{tour, I.ls_pos, I.ls_dlb, I.ls_el, reinterpret_cast<const float2 *>(I.xy), I.nbr, I.nbrd32};
}

// the workspace arrays of ant a's own search (local_search = 2; ant-major tours)
__device__ __forceinline__ LsMem ls_ant(const DevInst &I, int a)
{
    const size_t o = (size_t)a * I.n;
    return LsMem{I.tours + o, I.lsa_pos + o, I.lsa_dlb + o, I.lsa_el + o, reinterpret_cast<const float2 *>(I.xy),
                 I.nbr, I.nbrd32};
}

// shared memory: tour, pos, el (4n bytes each), dlb (n bytes), then the
// coordinates at a 16-byte boundary when they fit as well
__host__ __device__ inline size_t ls_smem_core(int n) { return (size_t)n * 13; }
__host__ __device__ inline size_t ls_xy_offset(int n) { return ((size_t)n * 13 + 15) & ~(size_t)15; }
__host__ __device__ inline size_t ls_smem_full(int n) { return ls_xy_offset(n) + (size_t)n * 8; }

// every array in `sm` (ls_smem_full bytes), the coordinates not yet filled
__device__ __forceinline__ LsMem ls_shared_full(const DevInst &I, unsigned char *sm)
{
    const int n = I.n;
    LsMem M;
    M.tour = reinterpret_cast<int32_t *>(sm);
    M.pos = reinterpret_cast<int32_t *>(sm + (size_t)n * 4);
    M.el = reinterpret_cast<float *>(sm + (size_t)n * 8);
    M.dlb = sm + (size_t)n * 12;
    M.xy = reinterpret_cast<const float2 *>(sm + ls_xy_offset(n));
    M.nbr = I.nbr;
    M.nbrd32 = I.nbrd32;
    return M;
}

// where ls_shared_full's arrays do not all fit: all but the coordinates in `sm`
// (smem_bytes) if they do, else `fallback`
__device__ __forceinline__ LsMem ls_shared(const DevInst &I, unsigned char *sm, size_t smem_bytes, const LsMem &fallback)
{
    if (ls_smem_core(I.n) > smem_bytes) return fallback;
    LsMem M = ls_shared_full(I, sm);
    M.xy = reinterpret_cast<const float2 *>(I.xy);
    return M;
}

}  // namespace hac
