// The fused cluster kernel (fused.cuh): its launch by layout, and the
// one-ant-per-quad form for instances without local search.
#include "fused.cuh"

namespace hac {

cudaError_t launch_fused_quad(const FusedArgs &A, const FusedLaunch &L)
{
    if (A.kp_cap <= 16) return launch_fused_form<8, 4, false>(A, L);
    if (A.kp_cap <= 20) return launch_fused_form<8, 5, false>(A, L);
    return launch_fused_form<8, 8, false>(A, L);
}

// a CTA that leaves room for no other on its SM, for device_shape
__global__ void k_whole_sm() {}

int device_sms()
{
    int d = 0, v = 0;
    if (cudaGetDevice(&d) != cudaSuccess ||
        cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, d) != cudaSuccess || v < 1) {
        cudaGetLastError();
        return DeviceShape().sms;
    }
    return v;
}

DeviceShape device_shape()
{
    DeviceShape S;
    S.sms = S.clusters[0] = device_sms();
    bool ok = cudaFuncSetAttribute(k_whole_sm, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FUSED_SMEM_LIMIT) ==
              cudaSuccess;
    for (int c = 1; c <= 3 && ok; ++c) {
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr;
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = 1u << c;
        attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
        cfg.gridDim = dim3((unsigned)S.sms << c, 1, 1);
        cfg.blockDim = dim3(512, 1, 1);
        cfg.dynamicSmemBytes = FUSED_SMEM_LIMIT;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        int v = 0;
        ok = cudaOccupancyMaxActiveClusters(&v, k_whole_sm, &cfg) == cudaSuccess;
        if (ok && v > 0) S.clusters[c] = v;
    }
    if (!ok) cudaGetLastError();
    return S;
}

size_t fused_smem_bytes(int rows_cap, int kp_cap, int warps, int apw, int stride, int xy_cap,
                        int list_rows)
{
    return fused_table_bytes(rows_cap, kp_cap) + (apw <= 8 ? (size_t)warps * apw * QRING_W * 4 : 0) +
           fused_vis_bytes(warps, apw, stride) + (((size_t)xy_cap * 8 + 15) & ~(size_t)15) + (size_t)list_rows * FBL * 2;
}

cudaError_t launch_fused(const DevInst *d_inst, const int32_t *d_order, const int32_t *d_iters,
                         int clusters, int clog, int apw, bool ls, int warps, int block_warps, int rows_cap, int kp_cap,
                         int stride, int xy_cap, int list_rows, int iters, cudaStream_t s, bool after_resident)
{
    const FusedArgs A{d_inst, d_order, d_iters, iters, rows_cap, kp_cap, stride, warps, apw, xy_cap, list_rows};
    const FusedLaunch L{clog, clusters, block_warps,
                        fused_smem_bytes(rows_cap, kp_cap, warps, apw, stride, xy_cap, list_rows), s, after_resident};
    if (apw > 8) return ls ? launch_fused_lane_ls(A, L) : launch_fused_lane(A, L);
    return ls ? launch_fused_quad_ls(A, L) : launch_fused_quad(A, L);
}

}  // namespace hac
