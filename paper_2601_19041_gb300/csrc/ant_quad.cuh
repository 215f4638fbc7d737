// One ant per lane quad (up to 8 ants per warp): Algorithm 2 with the
// candidate row of the current node spread over 4 lanes.
//
// Lane h of a quad holds the slot groups 4j + h (j < NGL); with TAIL (five
// groups, k <= 20) the fifth group is split, lane h holding its slot 16 + h,
// so that 20 slots keep all four lanes busy.  The arithmetic is exactly that
// of the other forms (ant.cuh) and of the oracle: sequential in-group partial
// sums, the 8 group totals combined by the Hillis-Steele pattern (GroupScan),
// slot prefix = exclusive group prefix + in-group sum, r = fl32(u * total), the
// first live slot with r < prefix, or the last live slot when rounding leaves
// none.
//
// What bounds it: the dependent chain of a step (row load -> visited bits ->
// in-group sums -> group totals -> prefix -> chosen node -> next row), about
// 640 cycles with 4 warps on an SM (n = 500, m = 32, rows in shared memory), 840
// with 8 (m = 64).  The layout this replaces spread an ant over 8 or 16 lanes
// and took 1368 to 1580 cycles for 64 ants on 16 warps: the same chain, but
// four times the warp instructions for it.  Four lanes are the fewest that
// still load a row in one go; what shortened the chain besides:
//   - no value or load hangs on a divergent branch (padding slots are a node
//     whose bit is always set, lanes without a group read a padding record);
//   - the group that holds the choice is found by every lane from the group
//     prefixes, in registers, instead of a ballot, a bit scan and a shuffle;
//   - one early vote covers every step that needs more than this (no live
//     slot; rounding near the total), so the branch waits for nothing.
//
// Per-ant state in shared memory: the visited bitmask (word w of the ant's
// `stride` words) and a ring of QRING words: at the start of a window of
// QRING steps it receives the window's uniform draws (each lane evaluates
// one Philox block = 4 draws), step s reads its draw and leaves its record
// (node << 8 | slot) in the same word, and the window's end writes the
// records to the tour and slot arrays.  No register is indexed by the step.
//
// Nearest-unvisited steps (no live candidate): all quads that need one read
// their node's 32-entry list at once, 8 entries per lane; what the list does
// not answer is served by the whole warp, one ant after the other (second
// list, then a scan).
#pragma once

#include "ant.cuh"

namespace hac {

constexpr int QRING = 16;       // steps per window (4 lanes x 4 draws)
constexpr int QRING_W = 20;     // words per ring: 8 rings start in 8 different groups of 4 banks

// 8 consecutive entries (8h .. 8h+7) of a node's 32-entry lookup list; past
// its end the padding node n
__device__ __forceinline__ void list8(const GlobalList &l, int node, int h, int n, int (&u)[8])
{
    const uint4 *r = reinterpret_cast<const uint4 *>(l.fbl + (size_t)node * FBL) + 2 * h;
    const uint4 a = __ldg(r), b = __ldg(r + 1);
    const uint32_t v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
    for (int k = 0; k < 8; ++k) u[k] = (int)min(v[k], (uint32_t)n);
}

template <int CLOG>
__device__ __forceinline__ void list8(const ClusterList<CLOG> &l, int node, int h, int n, int (&u)[8])
{
    const uint32_t loc = (uint32_t)node >> CLOG;
    uint32_t a = l.base + 2u * (loc * FBL + 8u * (uint32_t)h);
    uint32_t w[4];
    if (CLOG == 0) {
        asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]) : "r"(a));
    } else {
        a = map_to_rank(a, (uint32_t)node & ((1u << CLOG) - 1u));
        asm volatile("ld.shared::cluster.v4.u32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]) : "r"(a));
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) u[k] = (int)min((w[k >> 1] >> (16 * (k & 1))) & 0xffffu, (uint32_t)n);
}

__device__ __forceinline__ uint32_t ld_smem_u1(uint32_t a)
{
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}

// the bit of node u in the mask at shared-window address `vis` is clear
__device__ __forceinline__ bool q_unvisited(uint32_t vis, int u)
{
    const uint32_t w = ld_smem_u1(vis + (((uint32_t)u >> 5) << 2));
    return !(__funnelshift_r(w, 0u, (uint32_t)u) & 1u);
}

// sets the bit of node u (one lane of the quad).  A plain conditional red: with
// the predicate inside the asm statement it took 58 cycles instead of 14.
__device__ __forceinline__ void q_visit(uint32_t vis, int u, bool on)
{
    if (on)
        asm volatile("red.shared.or.b32 [%0], %1;" ::"r"(vis + (((uint32_t)u >> 5) << 2)), "r"(1u << (u & 31)) : "memory");
}

__device__ __forceinline__ void q_store(uint32_t a, uint32_t v, bool on)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %2, 0;\n\t@p st.shared.u32 [%0], %1;\n\t}"
                 ::"r"(a), "r"(v), "r"((int)on) : "memory");
}

// Candidate rows of one lane: load(cur) -> ids and choice values of its
// groups (and of its tail slot), padding slots being node n.  No load hangs on
// a branch: a lane without a group (kp / 4 groups, fewer than the layout's)
// reads `pad`, a shared-memory record of four padding slots (16 bytes of
// zeros, then four ids n), in place of the row; from global memory it reads
// group 0 and its ids are masked.
template <int NGL, bool TAIL>
struct GlobalQuadRows {
    const int32_t *ir[NGL], *irt;
    const float *cr[NGL], *crt;
    uint32_t off[NGL], offt;      // all ones: no such group
    int kp, n;
    __device__ __forceinline__ GlobalQuadRows(const DevInst &I, int h) : kp(I.k_pad), n(I.n)
    {
        const int G = kp >> 2;
#pragma unroll
        for (int j = 0; j < NGL; ++j) {
            const int g = 4 * j + h;
            off[j] = g < G ? 0u : 0xffffffffu;
            ir[j] = I.cand + (g < G ? 4 * g : 0);
            cr[j] = I.choice + (g < G ? 4 * g : 0);
        }
        offt = G > 4 ? 0u : 0xffffffffu;
        irt = I.cand + (G > 4 ? 16 + h : 0);
        crt = I.choice + (G > 4 ? 16 + h : 0);
    }
    __device__ __forceinline__ void load(int cur, int4 (&id)[NGL], float4 (&c)[NGL], int &idt, float &ct) const
    {
        const size_t o = (size_t)(uint32_t)cur * (uint32_t)kp;
#pragma unroll
        for (int j = 0; j < NGL; ++j) {
            id[j] = __ldg(reinterpret_cast<const int4 *>(ir[j] + o));
            c[j] = __ldg(reinterpret_cast<const float4 *>(cr[j] + o));
        }
        if (TAIL) {
            idt = __ldg(irt + o);
            ct = __ldg(crt + o);
        }
#pragma unroll
        for (int j = 0; j < NGL; ++j) {
            id[j].x = (int)min((uint32_t)id[j].x | off[j], (uint32_t)n);
            id[j].y = (int)min((uint32_t)id[j].y | off[j], (uint32_t)n);
            id[j].z = (int)min((uint32_t)id[j].z | off[j], (uint32_t)n);
            id[j].w = (int)min((uint32_t)id[j].w | off[j], (uint32_t)n);
        }
        if (TAIL) idt = (int)min((uint32_t)idt | offt, (uint32_t)n);
    }
};

template <int NGL, bool TAIL, int CLOG>
struct ClusterQuadRows {
    uint32_t ib[NGL], cb[NGL], ibt, cbt;   // shared-window addresses of row 0 in the calling CTA
    uint32_t ist[NGL], cst[NGL], istt, cstt;   // bytes from row to row (0: no such group)
    __device__ __forceinline__ ClusterQuadRows(uint32_t idx_base, uint32_t ch_base, uint32_t pad, int kp, int h)
    {
        const int G = kp >> 2;
#pragma unroll
        for (int j = 0; j < NGL; ++j) {
            const int g = 4 * j + h;
            ist[j] = g < G ? 2u * kp : 0u;
            cst[j] = g < G ? 4u * kp : 0u;
            ib[j] = g < G ? idx_base + 8u * g : pad + 16u;
            cb[j] = g < G ? ch_base + 16u * g : pad;
        }
        istt = G > 4 ? 2u * kp : 0u;
        cstt = G > 4 ? 4u * kp : 0u;
        ibt = G > 4 ? idx_base + 2u * (16 + h) : pad + 16u;
        cbt = G > 4 ? ch_base + 4u * (16 + h) : pad;
    }
    __device__ __forceinline__ void load(int cur, int4 (&id)[NGL], float4 (&c)[NGL], int &idt, float &ct) const
    {
        const uint32_t loc = (uint32_t)cur >> CLOG, owner = (uint32_t)cur & ((1u << CLOG) - 1u);
        uint2 raw[NGL];
        unsigned short rt = 0;
#pragma unroll
        for (int j = 0; j < NGL; ++j) {
            const uint32_t a = ib[j] + loc * ist[j];
            raw[j] = CLOG == 0 ? ld_smem_u2(a) : ld_dsmem_u2(map_to_rank(a, owner));
        }
        if (TAIL) {
            const uint32_t a = ibt + loc * istt;
            if (CLOG == 0) asm volatile("ld.shared.u16 %0, [%1];" : "=h"(rt) : "r"(a));
            else asm volatile("ld.shared::cluster.u16 %0, [%1];" : "=h"(rt) : "r"(map_to_rank(a, owner)));
        }
#pragma unroll
        for (int j = 0; j < NGL; ++j) {
            const uint32_t a = cb[j] + loc * cst[j];
            c[j] = CLOG == 0 ? ld_smem_f4(a) : ld_dsmem_f4(map_to_rank(a, owner));
        }
        if (TAIL) {
            const uint32_t a = cbt + loc * cstt;
            if (CLOG == 0) asm volatile("ld.shared.f32 %0, [%1];" : "=f"(ct) : "r"(a));
            else asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(ct) : "r"(map_to_rank(a, owner)));
            idt = (int)rt;
        }
#pragma unroll
        for (int j = 0; j < NGL; ++j) {
            id[j].x = (int)(raw[j].x & 0xffffu);
            id[j].y = (int)(raw[j].x >> 16);
            id[j].z = (int)(raw[j].y & 0xffffu);
            id[j].w = (int)(raw[j].y >> 16);
        }
    }
};

// index of the lowest set bit (x != 0)
__device__ __forceinline__ int low_bit(unsigned x) { return 31 - __clz((int)(x & (0u - x))); }

// a & m | b, for selections by masks that do not change in the loop
__device__ __forceinline__ uint32_t and_or(float a, uint32_t m, uint32_t b) { return (__float_as_uint(a) & m) | b; }

// Nearest unvisited node of `scur` by a scan of the unvisited bits of the
// mask `sv` (whole warp): argmin of (FP32 key, index).
__device__ __forceinline__ int scan_nearest(const DevInst &I, const unsigned *sv, int scur, const float2 *xy)
{
    const int lane = threadIdx.x & 31, n = I.n, nwords = (n + 31) >> 5;
    float bk = __int_as_float(0x7f800000);
    int bu = 0x7fffffff;
    const bool euc = I.kind == 0;
    const float2 pc = euc ? xy[scur] : make_float2(0.f, 0.f);
    const float *crow = euc ? nullptr : I.cost + (size_t)scur * n;
    for (int wd = lane; wd < nwords; wd += 32) {
        unsigned um = ~sv[wd];
        if (wd == nwords - 1 && (n & 31)) um &= (1u << (n & 31)) - 1u;
        while (um) {   // two unvisited nodes per round: independent loads
            const int u0 = (wd << 5) | low_bit(um);
            um &= um - 1u;
            const int u1 = um ? (wd << 5) | low_bit(um) : u0;
            um &= um - 1u;
            const float k0 = euc ? key32_xy(pc, xy[u0]) : crow[u0];
            const float k1 = euc ? key32_xy(pc, xy[u1]) : crow[u1];
            if (key_less(k0, u0, bk, bu)) { bk = k0; bu = u0; }
            if (key_less(k1, u1, bk, bu)) { bk = k1; bu = u1; }
        }
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        const float k2 = __shfl_xor_sync(FULL_MASK, bk, o);
        const int u2 = __shfl_xor_sync(FULL_MASK, bu, o);
        if (key_less(k2, u2, bk, bu)) { bk = k2; bu = u2; }
    }
    return bu;
}

// Builds the tours of ants a_first .. a_end-1 (at most 8) in iteration t.
// vis_warp: their bitmasks, `stride` words each; ring_warp: their rings,
// QRING_W words each, 16-byte aligned.  Tours are written ant-major.  A quad
// without an ant walks along with the warp's first ant (same mask, draws and
// choices) and writes nothing.
template <int NGL, bool TAIL, typename Rows, typename List>
__device__ __forceinline__ void build_tours_quad(const DevInst &I, const Rows &rows, const List &list, int t,
                                                 int a_first, int a_end, unsigned *vis_warp, int stride,
                                                 uint32_t *ring_warp, const float2 *xy_scan)
{
    constexpr int GT = TAIL ? 5 : NGL == 1 ? 4 : 8;   // groups that may hold slots
    const int lane = threadIdx.x & 31;
    const int h = lane & 3, p = lane >> 2, qbase = lane & ~3;
    const bool real = a_first + p < a_end, writer = real && h == 0;
    const int a = a_first + (real ? p : 0), pp = real ? p : 0;
    const int n = I.n;
    const uint64_t seed = I.seed;
    unsigned *visp = vis_warp + (size_t)pp * stride;
    const uint32_t vis = (uint32_t)__cvta_generic_to_shared(visp);
    uint32_t *ring = ring_warp + pp * QRING_W;
    const uint32_t ring_a = (uint32_t)__cvta_generic_to_shared(ring);
    const uint32_t m0 = h == 0 ? ~0u : 0u, m1 = h == 1 ? ~0u : 0u, m2 = h == 2 ? ~0u : 0u, m3 = h == 3 ? ~0u : 0u;

    if (real)
        for (int w = h; w <= (n >> 5); w += 4) visp[w] = 0u;   // bits 0..n
    __syncwarp();

    int32_t *tour = I.tours + (size_t)a * n;
    uint8_t *slots = I.slots + (size_t)a * n;
    int32_t *fbs = I.fbs + (size_t)a * n;
    int nfb = 0;

    // the window's draws into the ring: lane h evaluates block (s0 >> 2) + h
    auto fill = [&](int s0) {
        const U4 x = draw_block(seed, (uint32_t)t, (uint32_t)a, (uint32_t)((s0 >> 2) + h));
        if (real)
            *reinterpret_cast<float4 *>(ring + 4 * h) =
                make_float4(unif24(x.x), unif24(x.y), unif24(x.z), unif24(x.w));
        return x.x;
    };
    const uint32_t x0 = __shfl_sync(FULL_MASK, fill(0), qbase);
    int cur = (int)__umulhi(x0, (uint32_t)n);
    q_visit(vis, n, writer);                   // padding node: never live
    q_visit(vis, cur, writer);
    __syncwarp();
    q_store(ring_a, ((uint32_t)cur << 8) | SLOT_FALLBACK, writer);

    int4 id[NGL];
    float4 ch[NGL];
    int idt = n;
    float ct = 0.0f;
    rows.load(cur, id, ch, idt, ct);
    int j0 = 1;                                // step 0 is the start node

    for (int s0 = 0; s0 < n; s0 += QRING) {
        const int je = min(QRING, n - s0);
#pragma unroll 1
        for (int j1 = j0; j1 < je; ++j1) {
            const uint32_t ra = ring_a + 4u * (uint32_t)j1;
            const float u = __uint_as_float(ld_smem_u1(ra));

            // live weights and in-group partial sums of the own groups
            float w[NGL][4], ps[NGL][4], wt = 0.0f;
#pragma unroll
            for (int j = 0; j < NGL; ++j) {
                w[j][0] = q_unvisited(vis, id[j].x) ? ch[j].x : 0.0f;
                w[j][1] = q_unvisited(vis, id[j].y) ? ch[j].y : 0.0f;
                w[j][2] = q_unvisited(vis, id[j].z) ? ch[j].z : 0.0f;
                w[j][3] = q_unvisited(vis, id[j].w) ? ch[j].w : 0.0f;
            }
            if (TAIL) wt = q_unvisited(vis, idt) ? ct : 0.0f;
#pragma unroll
            for (int j = 0; j < NGL; ++j) {
                ps[j][0] = w[j][0];
#pragma unroll
                for (int q = 1; q < 4; ++q) ps[j][q] = __fadd_rn(ps[j][q - 1], w[j][q]);
            }
            // all group totals, the tail's slots
            float T[8], tw[4] = {0.f, 0.f, 0.f, 0.f}, tp[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int g = 0; g < 8; ++g) T[g] = 0.0f;
            if (TAIL) {
#pragma unroll
                for (int q = 0; q < 4; ++q) tw[q] = __shfl_sync(FULL_MASK, wt, q, 4);
                tp[0] = tw[0];
#pragma unroll
                for (int q = 1; q < 4; ++q) tp[q] = __fadd_rn(tp[q - 1], tw[q]);
                T[4] = tp[3];
            }
#pragma unroll
            for (int j = 0; j < NGL; ++j)
#pragma unroll
                for (int g = 0; g < 4; ++g) T[4 * j + g] = __shfl_sync(FULL_MASK, ps[j][3], g, 4);
            GroupScan<GT> sc;
            sc.run(T);
            const float total = sc.C[7];
            const float r = __fmul_rn(u, total);
            // Steps whose outcome the straight path below does not cover: no live
            // slot (total = 0), or one where rounding may leave no prefix above r.
            // Prefix sums and total differ by a few units of 2^-24 of the total,
            // so r < (1 - 1e-5) total is below the last live slot's prefix, unless
            // the total is near the ends of the FP32 range.
            const bool odd = !(total > 1e-30f) | !(total < 1e37f) | (u > 0.99999f);
            const bool slow = __any_sync(FULL_MASK, odd);

            // The first group with r < its last prefix and a live slot, known to
            // every lane; a dead group or slot gets the prefix -1.
            float E[GT];
#pragma unroll
            for (int g = 0; g < GT; ++g) {
                const float e = g == 0 ? T[0] : __fadd_rn(sc.C[g - 1], T[g]);
                E[g] = T[g] > 0.0f ? e : -1.0f;
            }
            int gs = GT - 1;
#pragma unroll
            for (int g = GT - 2; g >= 0; --g) gs = r < E[g] ? g : gs;
            // the own groups' first slot with r < prefix: (node << 2) | slot in group
            int pick[NGL];
#pragma unroll
            for (int j = 0; j < NGL; ++j) {
                const uint32_t e0 = j == 0 ? 0u : and_or(sc.C[4 * j - (j > 0)], m0, 0u);
                const float ex = __uint_as_float(and_or(sc.C[4 * j], m1, and_or(sc.C[4 * j + 1], m2, and_or(sc.C[4 * j + 2], m3, e0))));
                const float S0 = w[j][0] > 0.0f ? __fadd_rn(ex, ps[j][0]) : -1.0f;
                const float S1 = w[j][1] > 0.0f ? __fadd_rn(ex, ps[j][1]) : -1.0f;
                const float S2 = w[j][2] > 0.0f ? __fadd_rn(ex, ps[j][2]) : -1.0f;
                const int k0 = id[j].x << 2, k1 = (id[j].y << 2) | 1, k2 = (id[j].z << 2) | 2, k3 = (id[j].w << 2) | 3;
                int k = r < S2 ? k2 : k3;
                k = r < S1 ? k1 : k;
                pick[j] = r < S0 ? k0 : k;
            }
            int mine = pick[0], src = gs, sbase = 4 * gs;
            if (NGL == 2) {
                mine = gs >= 4 ? pick[NGL - 1] : mine;
                src = gs & 3;
            }
            if (TAIL) {
                int tq = 3;
#pragma unroll
                for (int q = 2; q >= 0; --q) {
                    const float S = tw[q] > 0.0f ? __fadd_rn(sc.C[3], tp[q]) : -1.0f;
                    tq = r < S ? q : tq;
                }
                mine = gs == 4 ? idt << 2 : mine;
                src = gs == 4 ? tq : src;
                sbase = gs == 4 ? 16 + tq : sbase;
            }
            const int got = __shfl_sync(FULL_MASK, mine, src, 4);
            int nxt = got >> 2;
            unsigned slot = (unsigned)(sbase + (got & 3));

            if (slow) {
                bool hit = false;              // some r < E[g]: the straight path's choice stands
#pragma unroll
                for (int g = 0; g < GT; ++g) hit |= r < E[g];
                bool live = false;
#pragma unroll
                for (int g = 0; g < GT; ++g) live |= T[g] > 0.0f;
                const bool need = real & !live;
                unsigned pend = __ballot_sync(FULL_MASK, need & (h == 0));
                if (__any_sync(FULL_MASK, live & !hit)) {   // rounding left no r < prefix: the last live slot
                    int ll = -1, ln = 0;
#pragma unroll
                    for (int j = 0; j < NGL; ++j) {
                        const int s4 = 4 * (4 * j + h);
                        if (w[j][0] > 0.0f) { ll = s4; ln = id[j].x; }
                        if (w[j][1] > 0.0f) { ll = s4 + 1; ln = id[j].y; }
                        if (w[j][2] > 0.0f) { ll = s4 + 2; ln = id[j].z; }
                        if (w[j][3] > 0.0f) { ll = s4 + 3; ln = id[j].w; }
                    }
                    if (TAIL && wt > 0.0f) { ll = 16 + h; ln = idt; }
#pragma unroll
                    for (int o = 1; o < 4; o <<= 1) {
                        const int l2 = __shfl_xor_sync(FULL_MASK, ll, o), n2 = __shfl_xor_sync(FULL_MASK, ln, o);
                        if (l2 > ll) { ll = l2; ln = n2; }
                    }
                    if (live & !hit) { nxt = ln; slot = (unsigned)ll; }
                }
                if (pend) {
                    const bool lists = list.present();
                    const uint16_t *fbl2 = lists ? I.fbl2 : nullptr;
                    int found = -1;
                    if (lists) {
                        int e8[8], first8 = -1;
                        bool ok[8];
                        list8(list, cur, h, n, e8);
#pragma unroll
                        for (int k = 0; k < 8; ++k) ok[k] = q_unvisited(vis, e8[k]);
#pragma unroll
                        for (int k = 7; k >= 0; --k) first8 = ok[k] ? e8[k] : first8;
                        const unsigned lb = (__ballot_sync(FULL_MASK, first8 >= 0) >> qbase) & 15u;
                        const int f = __shfl_sync(FULL_MASK, first8, low_bit(lb | 16u) & 3, 4);
                        found = lb ? f : -1;
                        pend = __ballot_sync(FULL_MASK, need & (found < 0) & (h == 0));
                    }
                    // the second list, then the scan: one ant at a time, whole warp
                    while (pend) {
                        const int sb = low_bit(pend);
                        pend &= pend - 1u;
                        const int scur = __shfl_sync(FULL_MASK, cur, sb);
                        const unsigned *sv = vis_warp + (size_t)(sb >> 2) * stride;
                        int fo = -1;
                        if (fbl2) fo = lookup2(fbl2, scur, lane, n, [&](int u2) { return (sv[u2 >> 5] >> (u2 & 31)) & 1u; });
                        if (fo < 0) fo = scan_nearest(I, sv, scur, xy_scan);
                        if (qbase == sb) found = fo;
                    }
                    if (need) {
                        nxt = found;
                        slot = SLOT_FALLBACK;
                        if (h == 0) fbs[nfb++] = s0 + j1;
                    }
                }
                nxt = (unsigned)nxt >= (unsigned)n ? 0 : nxt;   // unreachable for finite keys; keeps indices in range
                nxt = __shfl_sync(FULL_MASK, nxt, real ? lane : h);   // idle quads follow the first ant
            }

            // next row first, so its latency overlaps the bookkeeping below
            rows.load(nxt, id, ch, idt, ct);
            q_visit(vis, nxt, writer);
            q_store(ra, ((uint32_t)nxt << 8) | slot, writer);
            __syncwarp();
            cur = nxt;
        }
        j0 = 0;
        // the window's records out, the next window's draws in
        const uint4 r4 = *reinterpret_cast<const uint4 *>(ring + 4 * h);
        const uint32_t rec[4] = {r4.x, r4.y, r4.z, r4.w};
        const int o = s0 + 4 * h;
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (real && o + q < n) {
                tour[o + q] = (int)(rec[q] >> 8);
                slots[o + q] = (uint8_t)rec[q];
            }
        __syncwarp();
        fill(s0 + QRING);
        __syncwarp();
    }
    if (writer) I.fbcnt[a] = nfb;
    __syncwarp();
}

}  // namespace hac
