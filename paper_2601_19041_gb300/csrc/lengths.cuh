// Tour lengths, eq. (tour_length), in FP64.
//
// Summation order (shared with the CPU oracle): edge e joins tour[e] and
// tour[e+1] (the closing edge is e = n-1); edge e is added to partial sum
// e mod 32 in increasing e, and the 32 partials are combined by the pairwise
// tree.  A warp keeps partial l in lane l (one FP64 add per edge, all lanes
// busy) and combines the partials with a butterfly of shuffles (by
// commutativity every lane ends with the same tree value).  FP64 adds have a
// long latency on GB300, so an ant's chain is n/32 + 5 adds long instead of n.
//
// Construction records the chosen slot of every step; the d of a candidate
// step is the slot's precomputed distance.  Nearest-unvisited steps are listed
// per ant and get their d from a full-width pass, together with the closing
// edge (stored at step index 0).
#pragma once

#include "hac_internal.cuh"

namespace hac {

constexpr uint8_t SLOT_FALLBACK = 0xff;   // slot record of a nearest-unvisited step

__device__ __forceinline__ size_t step_ix(const DevInst &I, int a, int s)
{
    return (size_t)a * I.tour_sa + (size_t)s * I.tour_ss;
}

// d of ant a's listed nearest-unvisited steps and of its closing edge, into
// dstep (whole warp, an entry per lane); returns their number.  The warp that
// sums the ant's length calls it, so no barrier wider than the warp is needed.
__device__ __forceinline__ int warp_fallback_distances(const DevInst &I, int a)
{
    const int lane = threadIdx.x & 31, n = I.n, cnt = I.fbcnt[a];
    const int32_t *fbs = I.fbs + (size_t)a * n;
    for (int e = lane; e <= cnt; e += 32) {
        const int s = e < cnt ? fbs[e] : 0;            // 0: the closing edge
        const int from = I.tours[step_ix(I, a, s ? s - 1 : n - 1)], to = I.tours[step_ix(I, a, s)];
        I.dstep[step_ix(I, a, s)] = dist64(I, from, to);
    }
    return cnt;
}

// lengths of NA ants at once (whole warp; results in every lane): the loops
// of the NA ants share one body, so their FP64 chains overlap
template <int NA>
__device__ __forceinline__ void warp_ant_lengths(const DevInst &I, const int (&ants)[NA], double (&out)[NA])
{
    const int lane = threadIdx.x & 31, n = I.n, kp = I.k_pad;
    const double *cdist = I.cdist;
    double P[NA];
#pragma unroll
    for (int h = 0; h < NA; ++h) P[h] = 0.0;
    constexpr int U = 4;   // edges per ant whose loads are in flight together
    int e = lane;
    for (; e + 32 * (U - 1) < n - 1; e += 32 * U) {
        int from[NA][U];
        uint8_t c[NA][U];
#pragma unroll
        for (int h = 0; h < NA; ++h)
#pragma unroll
            for (int k = 0; k < U; ++k) {
                const int s = e + 32 * k + 1;             // the edge enters step s (< n)
                from[h][k] = I.tours[step_ix(I, ants[h], s - 1)];
                c[h][k] = I.slots[step_ix(I, ants[h], s)];
            }
        // the address of each edge's length is selected, not the load: loads behind
        // a lane-dependent branch waited for one another
        double d[NA][U];
#pragma unroll
        for (int h = 0; h < NA; ++h)
#pragma unroll
            for (int k = 0; k < U; ++k) {
                const double *src = I.dstep + step_ix(I, ants[h], e + 32 * k + 1);
                if (c[h][k] != SLOT_FALLBACK) src = cdist + ((size_t)from[h][k] * kp + c[h][k]);
                d[h][k] = *src;
            }
#pragma unroll
        for (int k = 0; k < U; ++k)
#pragma unroll
            for (int h = 0; h < NA; ++h) P[h] = __dadd_rn(P[h], d[h][k]);
    }
    for (; e < n; e += 32) {
#pragma unroll
        for (int h = 0; h < NA; ++h) {
            const int a = ants[h];
            const int s = e == n - 1 ? 0 : e + 1;          // step 0 holds the closing edge
            const uint8_t c = s ? I.slots[step_ix(I, a, s)] : SLOT_FALLBACK;
            const double *src = I.dstep + step_ix(I, a, s);
            if (c != SLOT_FALLBACK) src = cdist + ((size_t)I.tours[step_ix(I, a, e)] * kp + c);
            P[h] = __dadd_rn(P[h], *src);
        }
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1)
#pragma unroll
        for (int h = 0; h < NA; ++h) P[h] = __dadd_rn(P[h], __shfl_xor_sync(0xffffffffu, P[h], o));
#pragma unroll
    for (int h = 0; h < NA; ++h) out[h] = P[h];
}

// lengths of ants [a_lo, a_hi): one warp per ant, two ants per warp at a
// time (without `sums`, the nearest-unvisited steps are counted only: local
// search on every ant recomputes the lengths)
__device__ __forceinline__ void ant_lengths(const DevInst &I, int a_lo, int a_hi, bool sums)
{
    const int wib = threadIdx.x >> 5, nw = blockDim.x >> 5, lane = threadIdx.x & 31;
    int fb = 0;
    for (int a = a_lo + wib; a < a_hi; a += 2 * nw) {
        const int b = a + nw;
        if (!sums) {
            fb += I.fbcnt[a] + (b < a_hi ? I.fbcnt[b] : 0);
        } else if (b < a_hi) {
            const int ab[2] = {a, b};
            double L[2];
            fb += warp_fallback_distances(I, a) + warp_fallback_distances(I, b);
            __syncwarp();
            warp_ant_lengths<2>(I, ab, L);
            if (lane == 0) { I.lens[a] = L[0]; I.lens[b] = L[1]; }
        } else {
            const int a1[1] = {a};
            double L[1];
            fb += warp_fallback_distances(I, a);
            __syncwarp();
            warp_ant_lengths<1>(I, a1, L);
            if (lane == 0) I.lens[a] = L[0];
        }
    }
    if (lane == 0 && fb) atomicAdd(&I.st->n_fallback, (unsigned long long)fb);
}

// length of an explicit tour (T_NN, T_ib after 2-opt), whole warp, same order
__device__ __forceinline__ double warp_tour_length(const DevInst &I, const int32_t *tour)
{
    const int lane = threadIdx.x & 31, n = I.n;
    double P = 0.0;
    for (int e = lane; e < n; e += 32) P = __dadd_rn(P, dist64(I, tour[e], tour[e + 1 < n ? e + 1 : 0]));
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) P = __dadd_rn(P, __shfl_xor_sync(0xffffffffu, P, o));
    return P;
}

}  // namespace hac
