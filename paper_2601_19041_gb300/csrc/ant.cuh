// What the three ways to build an ant's tour (Algorithm 2) share -- one ant
// per lane quad (ant_quad.cuh), lane pair (ant_pair.cuh) or lane
// (ant_lane.cuh): candidate rows and nearest-unvisited lists in global memory
// or in the shared memory of a cluster, the second-level list lookup, and the
// scan of the group totals.
//
// Roulette (eq. transition): sequential partial sums in groups of 4 slots,
// the 8 group totals combined by an inclusive Hillis-Steele scan (offsets 1,
// 2, 4), slot prefix = exclusive group prefix + in-group partial sum;
// r = fl32(u * total) selects the first live slot with r < prefix, or the last
// live slot when rounding leaves none.
//
// Fallback (N_i empty): the nearest unvisited node by (FP32 key, index): the
// node's 32-entry list of nearest nodes in key order (the first unvisited
// entry is the exact answer when there is one), the next 256, else a scan of
// the unvisited bits of the ant's mask.
#pragma once

#include "lengths.cuh"

namespace hac {

constexpr unsigned FULL_MASK = 0xffffffffu;
constexpr int FBL = FBL1_LEN;   // fallback list length (nearest nodes in key order)

__device__ __forceinline__ uint32_t word_of(const U4 &v, int w)
{
    return w == 0 ? v.x : w == 1 ? v.y : w == 2 ? v.z : v.w;
}

// Candidate rows hand out padding slots as node n: the construction presets
// bit n of every visited mask, so a padding slot is never live and no slot
// needs a validity test of its own.

// candidate rows in global memory (int32 ids, -1 on padding; FP32 choice)
struct GlobalRows {
    const int4 *cand4;
    const float4 *ch4;
    int G, n;
    __device__ __forceinline__ void load(int cur, int g, int4 &id, float4 &ch) const
    {
        id = __ldg(cand4 + (size_t)cur * G + g);
        ch = __ldg(ch4 + (size_t)cur * G + g);
        id.x = id.x < 0 ? n : id.x;
        id.y = id.y < 0 ? n : id.y;
        id.z = id.z < 0 ? n : id.z;
        id.w = id.w < 0 ? n : id.w;
    }
};

// shared-memory loads by 32-bit shared-window address; for C > 1 the address
// is first mapped to the owning CTA of the cluster (distributed shared memory)
__device__ __forceinline__ uint32_t map_to_rank(uint32_t addr, uint32_t rank)
{
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}

__device__ __forceinline__ uint2 ld_dsmem_u2(uint32_t a)
{
    uint2 v;
    asm volatile("ld.shared::cluster.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a));
    return v;
}

__device__ __forceinline__ float4 ld_dsmem_f4(uint32_t a)
{
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a));
    return v;
}

__device__ __forceinline__ uint2 ld_smem_u2(uint32_t a)
{
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a));
    return v;
}

__device__ __forceinline__ float4 ld_smem_f4(uint32_t a)
{
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a));
    return v;
}

// candidate rows in the shared memory of the CTAs of a cluster, interleaved by
// row (row i lives in CTA i & (C-1) at local row i >> CLOG); uint16 ids with
// n for padding.  Same layout (and offsets) in every CTA.
template <int CLOG>
struct ClusterRows {
    uint32_t idx_base, ch_base;   // shared-window addresses in the calling CTA
    int kp;
    __device__ __forceinline__ void load(int cur, int g, int4 &id, float4 &chv) const
    {
        const uint32_t loc = (uint32_t)cur >> CLOG;
        const uint32_t off = loc * (uint32_t)kp + 4u * (uint32_t)g;
        uint32_t ia = idx_base + 2u * off, ca = ch_base + 4u * off;
        uint2 raw;
        if (CLOG == 0) {
            raw = ld_smem_u2(ia);
            chv = ld_smem_f4(ca);
        } else {
            const uint32_t owner = (uint32_t)cur & ((1u << CLOG) - 1u);
            raw = ld_dsmem_u2(map_to_rank(ia, owner));
            chv = ld_dsmem_f4(map_to_rank(ca, owner));
        }
        id.x = (int)(raw.x & 0xffffu);
        id.y = (int)(raw.x >> 16);
        id.z = (int)(raw.y & 0xffffu);
        id.w = (int)(raw.y >> 16);
    }
};

// nearest-unvisited lookup lists: global int32 (I.fbl) or the uint16 copy in
// the cluster's shared memory (same row interleaving as the candidate table)
struct GlobalList {
    const int32_t *fbl;
    __device__ __forceinline__ bool present() const { return fbl != nullptr; }
    __device__ __forceinline__ int get(int node, int k) const { return fbl[(size_t)node * FBL + k]; }
};

template <int CLOG>
struct ClusterList {
    uint32_t base;   // shared-window address of this CTA's list rows (0: no list)
    __device__ __forceinline__ bool present() const { return base != 0u; }
    __device__ __forceinline__ int get(int node, int k) const
    {
        const uint32_t loc = (uint32_t)node >> CLOG;
        uint32_t a = base + 2u * (loc * FBL + (uint32_t)k);
        unsigned short v;
        if (CLOG == 0) asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(a));
        else {
            a = map_to_rank(a, (uint32_t)node & ((1u << CLOG) - 1u));
            asm volatile("ld.shared::cluster.u16 %0, [%1];" : "=h"(v) : "r"(a));
        }
        return v == 0xffff ? -1 : (int)v;
    }
};

// Second-level lookup (whole warp): the next FBL2_LEN nodes of `node`'s key
// order, 8 per lane in order (lane L holds ranks 32 + 8L .. 32 + 8L + 7).
// Returns the first one that `visited` reports unvisited, or -1 (then the
// nearest unvisited node lies further out and the scan finds it).  Entries
// past the list's end (0xffff) are read as the padding node n, whose bit is
// always set, so that no load hangs on a branch.
template <typename Visited>
__device__ __forceinline__ int lookup2(const uint16_t *fbl2, int node, int lane, int n, Visited visited)
{
    const uint4 v = __ldg(reinterpret_cast<const uint4 *>(fbl2 + (size_t)node * FBL2_LEN) + lane);
    const unsigned w[4] = {v.x, v.y, v.z, v.w};
    int first = -1;
    bool vis[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) vis[k] = visited((int)min((w[k >> 1] >> (16 * (k & 1))) & 0xffffu, (unsigned)n));
#pragma unroll
    for (int k = 7; k >= 0; --k) first = vis[k] ? first : (int)((w[k >> 1] >> (16 * (k & 1))) & 0xffffu);
    const unsigned bm = __ballot_sync(FULL_MASK, first >= 0);
    return bm ? __shfl_sync(FULL_MASK, first, __ffs(bm) - 1) : -1;
}

// Hillis-Steele inclusive scan (offsets 1, 2, 4) over 8 group totals, of
// which only the first GT can be non-zero; the exclusive prefix of group g is
// ex(g) = C[g-1] and the total is C[7].  Additions of a known +0 are skipped
// (exact for non-negative operands).
template <int GT>
struct GroupScan {
    float C[8];
    __device__ __forceinline__ void run(const float (&T)[8])
    {
        float A[8], B[8];
#pragma unroll
        for (int g = 0; g < 8; ++g) {
            const bool zg = g >= GT, zp = g - 1 >= GT;   // T[g], T[g-1] known zero
            if (g == 0 || zp) A[g] = zg ? 0.0f : T[g];
            else A[g] = zg ? T[g - 1] : __fadd_rn(T[g], T[g - 1]);
        }
#pragma unroll
        for (int g = 0; g < 8; ++g) {
            const bool zg = g - 1 >= GT, zp = g - 3 >= GT;   // A[g], A[g-2] known zero
            if (g < 2 || zp) B[g] = A[g];
            else B[g] = zg ? A[g - 2] : __fadd_rn(A[g], A[g - 2]);
        }
#pragma unroll
        for (int g = 0; g < 8; ++g) {
            const bool zg = g - 3 >= GT, zp = g - 7 >= GT;   // B[g], B[g-4] known zero
            if (g < 4 || zp) C[g] = B[g];
            else C[g] = zg ? B[g - 4] : __fadd_rn(B[g], B[g - 4]);
        }
    }
};

}  // namespace hac
