// Tour construction, Algorithm 2, one launch per iteration: every ant of every
// active instance builds one tour, reading candidate rows from global memory
// (128-bit loads of ids and choice values).  The per-ant work is in ant_quad.cuh,
// ant_pair.cuh and ant_lane.cuh; this file maps warps to (instance, ants)
// through the warp table.
#include "ant_lane.cuh"
#include "ant_pair.cuh"
#include "ant_quad.cuh"

namespace hac {

// one ant per lane quad: warp w of the table builds ants a0 .. a0+aw-1 (aw <= 8) of its instance
template <int NGL, bool TAIL>
__global__ void __launch_bounds__(256, 1) k_construct(const DevInst *__restrict__ insts,
                                                   const int4 *__restrict__ warpmap, int nwarps,
                                                   int nwords_max, int aw)
{
    extern __shared__ __align__(16) unsigned char smem_q[];
    const int wib = threadIdx.x >> 5;
    const int gw = blockIdx.x * (blockDim.x >> 5) + wib;
    if (gw >= nwarps) return;                       // warp-uniform
    const int4 wm = warpmap[gw];
    const DevInst &I = insts[wm.x];
    const int t = I.st->t;
    if (t >= I.iters) return;                       // warp-uniform
    uint32_t *ring = reinterpret_cast<uint32_t *>(smem_q) + wib * aw * QRING_W;
    unsigned *vis = reinterpret_cast<unsigned *>(smem_q) + (blockDim.x >> 5) * aw * QRING_W + (size_t)wib * aw * nwords_max;
    const GlobalQuadRows<NGL, TAIL> rows(I, threadIdx.x & 3);
    build_tours_quad<NGL, TAIL>(I, rows, GlobalList{I.fbl}, t, wm.y, min(I.m, wm.y + aw), vis, nwords_max, ring,
                                reinterpret_cast<const float2 *>(I.xy));
}

// one ant per lane: warp w of the table builds ants a0..a0+31 of its instance
template <int NG>
__global__ void __launch_bounds__(256, 1) k_construct_lane(const DevInst *__restrict__ insts,
                                                        const int4 *__restrict__ warpmap, int nwarps,
                                                        int nwords_max)
{
    extern __shared__ unsigned int smem_vis[];
    const int wib = threadIdx.x >> 5;
    const int gw = blockIdx.x * (blockDim.x >> 5) + wib;
    if (gw >= nwarps) return;
    const int4 wm = warpmap[gw];
    const DevInst &I = insts[wm.x];
    const int t = I.st->t;
    if (t >= I.iters) return;
    GlobalRows rows{reinterpret_cast<const int4 *>(I.cand), reinterpret_cast<const float4 *>(I.choice),
                    I.k_pad >> 2, I.n};
    build_tours_lane<NG>(I, rows, GlobalList{I.fbl}, t, wm.y, I.m, smem_vis + (size_t)wib * 32 * nwords_max,
                         reinterpret_cast<const float2 *>(I.xy));
}

// one ant per lane pair: warp w of the table builds ants a0..a0+15 of its instance
template <int NGL>
__global__ void __launch_bounds__(256, 1) k_construct_pair(const DevInst *__restrict__ insts,
                                                        const int4 *__restrict__ warpmap, int nwarps,
                                                        int nwords_max)
{
    extern __shared__ unsigned int smem_vis[];
    const int wib = threadIdx.x >> 5;
    const int gw = blockIdx.x * (blockDim.x >> 5) + wib;
    if (gw >= nwarps) return;
    const int4 wm = warpmap[gw];
    const DevInst &I = insts[wm.x];
    const int t = I.st->t;
    if (t >= I.iters) return;
    GlobalRows rows{reinterpret_cast<const int4 *>(I.cand), reinterpret_cast<const float4 *>(I.choice),
                    I.k_pad >> 2, I.n};
    build_tours_pair<NGL>(I, rows, GlobalList{I.fbl}, t, wm.y, I.m, smem_vis + (size_t)wib * 16 * nwords_max,
                          nwords_max, reinterpret_cast<const float2 *>(I.xy));
}

// every ant's length, a warp per ant: block (instance, ants LEN_ANTS*y ..)
constexpr int LEN_ANTS = 8;
__global__ void k_lengths(const DevInst *insts)
{
    const DevInst &I = insts[blockIdx.x];
    if (I.st->t >= I.iters) return;
    const int a0 = (int)blockIdx.y * LEN_ANTS;
    ant_lengths(I, a0, min(I.m, a0 + LEN_ANTS), I.local_search != 2 && I.local_search != 4);
}

static void launch_lengths(const DevInst *d_inst, int count, int max_m, cudaStream_t s)
{
    k_lengths<<<dim3(count, (max_m + LEN_ANTS - 1) / LEN_ANTS), 32 * LEN_ANTS, 0, s>>>(d_inst);
}

int launch_construct(const DevInst *d_inst, const int4 *d_warpmap, int warpmap_len, int apw,
                     int warps_per_block, int max_n, int max_kp, int max_m, int count, cudaStream_t s)
{
    if (apw == 32) {
        const int nwords = (max_n + 32) / 32;
        const size_t smem = (size_t)warps_per_block * 32 * nwords * sizeof(unsigned);
        const int blocks = (warpmap_len + warps_per_block - 1) / warps_per_block;
        const int G = max_kp / 4;
        auto go = [&](auto kern) {
            if (smem > 48 * 1024)
                cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            kern<<<blocks, warps_per_block * 32, smem, s>>>(d_inst, d_warpmap, warpmap_len, nwords);
        };
        if (G <= 3) go(k_construct_lane<3>);
        else if (G <= 5) go(k_construct_lane<5>);
        else go(k_construct_lane<8>);
        launch_lengths(d_inst, count, max_m, s);
        return 2;
    }
    if (apw == 16) {
        const int nwords = (max_n + 32) / 32;
        const size_t smem = (size_t)warps_per_block * 16 * nwords * sizeof(unsigned);
        const int blocks = (warpmap_len + warps_per_block - 1) / warps_per_block;
        const int G = max_kp / 4;
        auto go = [&](auto kern) {
            if (smem > 48 * 1024)
                cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            kern<<<blocks, warps_per_block * 32, smem, s>>>(d_inst, d_warpmap, warpmap_len, nwords);
        };
        if (G <= 4) go(k_construct_pair<2>);
        else if (G <= 6) go(k_construct_pair<3>);
        else go(k_construct_pair<4>);
        launch_lengths(d_inst, count, max_m, s);
        return 2;
    }
    const int nwords = (max_n + 32) / 32;   // visited bits 0..n (n: padding id)
    const size_t warp_smem = (size_t)apw * (QRING_W + nwords) * sizeof(unsigned);
    while (warps_per_block > 1 && warps_per_block * warp_smem > FUSED_SMEM_LIMIT) warps_per_block /= 2;
    const size_t smem = warps_per_block * warp_smem;
    const int blocks = (warpmap_len + warps_per_block - 1) / warps_per_block;
    auto go = [&](auto kern) {
        if (smem > 48 * 1024)
            cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        kern<<<blocks, warps_per_block * 32, smem, s>>>(d_inst, d_warpmap, warpmap_len, nwords, apw);
    };
    if (max_kp <= 16) go(k_construct<1, false>);
    else if (max_kp <= 20) go(k_construct<1, true>);
    else go(k_construct<2, false>);
    launch_lengths(d_inst, count, max_m, s);
    return 2;
}

}  // namespace hac
