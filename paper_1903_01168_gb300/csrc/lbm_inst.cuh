// lbm_inst.cuh -- definitions of the step-kernel launchers declared in
// lbm_internal.h.  Included by small translation units that instantiate them
// for one storage type: LBM_INSTANTIATE_FUSED(T, CV) per fused variant, or
// LBM_INSTANTIATE_TWOPASS(T).
#pragma once

#define LBM_DEVICE_HELPERS_ONLY
#include <algorithm>

#include "lbm_internal.h"
#include "lbm_kernels.cuh"

namespace lbm {

template <typename T, int CV>
const void *fused_kernel_cv() {
    return reinterpret_cast<const void *>(&k_step_fused<T, CV, FUSED_W, FUSED_NSLOT, !(CV & CV_OPEN)>);
}

template <typename T, int CV>
int fused_smem_cv() {
    return FusedCfg<T, CV, FUSED_W, FUSED_NSLOT, !(CV & CV_OPEN)>::SMEM;
}

template <typename T, int CV, bool ODD>
cudaError_t fused_launch_odd(const SimDesc *descs, const WorkItem *items, const int *item_off, int n_blocks, int off,
                             int flags, int *err, cudaStream_t st) {
    constexpr int SMEM = FusedCfg<T, CV, FUSED_W, FUSED_NSLOT, ODD>::SMEM;
    static bool attr_done[64] = {false};
    int dev = 0;
    cudaGetDevice(&dev);
    auto kernel = k_step_fused<T, CV, FUSED_W, FUSED_NSLOT, ODD>;
    if (dev < 64 && !attr_done[dev]) {
        cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM);
        if (e != cudaSuccess) return e;
        attr_done[dev] = true;
    }
    // programmatic dependent launch: the launch of step j+1 overlaps the tail of
    // step j; the kernel waits for its prerequisites before its first access
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)n_blocks);
    cfg.blockDim = dim3(FUSED_THREADS);
    cfg.dynamicSmemBytes = SMEM;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = LBM_FUSED_PDL;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, descs, items, item_off, n_blocks, off, flags, err);
}

template <typename T, int CV>
cudaError_t fused_launch_cv(const SimDesc *descs, const WorkItem *items, const int *item_off, int n_blocks, int off,
                            int flags, int *err, cudaStream_t st) {
    constexpr bool PERIODIC = !(CV & CV_OPEN);
    if (PERIODIC && (flags & FUSED_ODD))
        return fused_launch_odd<T, CV, PERIODIC>(descs, items, item_off, n_blocks, off, flags, err, st);
    return fused_launch_odd<T, CV, false>(descs, items, item_off, n_blocks, off, flags, err, st);
}

template <typename T, int CV>
cudaError_t tile_launch_cv(const SimDesc *desc, int nx, int ny, bool walls, int rows, int warps, int off, int *err, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((nx + TILE_W - 1) / TILE_W), (unsigned)((ny + rows - 1) / rows));
    cfg.blockDim = dim3((unsigned)(32 * warps));
    cfg.stream = st;
    cudaLaunchAttribute attr[1];   // programmatic dependent launch, as above
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = LBM_FUSED_PDL;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (walls && nx % FUSED_W == TILE_W + 1) return cudaLaunchKernelEx(&cfg, k_step_tile<T, CV, true>, desc, off, rows, err);
    return cudaLaunchKernelEx(&cfg, k_step_tile<T, CV, false>, desc, off, rows, err);
}

template <typename T, int CV>
cudaError_t twopass_launch_cv(const SimDesc *desc, int off, float *aux, long long nodes, cudaStream_t st) {
    const int g = (int)std::max<long long>(1, std::min<long long>((nodes + 255) / 256, 152LL * 16));
    k_tp_moments<T, CV><<<g, 256, 0, st>>>(desc, off, aux);
    k_tp_collide<T, CV><<<g, 256, 0, st>>>(desc, off, aux);
    return cudaPeekAtLastError();
}

template <typename T>
cudaError_t twopass_launch(int variant, const SimDesc *desc, int off, float *aux, long long nodes, cudaStream_t st) {
    switch (variant & (CV_MRT | CV_HERMITE)) {
    case 0: return twopass_launch_cv<T, 0>(desc, off, aux, nodes, st);
    case CV_MRT: return twopass_launch_cv<T, CV_MRT>(desc, off, aux, nodes, st);
    case CV_HERMITE: return twopass_launch_cv<T, CV_HERMITE>(desc, off, aux, nodes, st);
    default: return twopass_launch_cv<T, CV_MRT | CV_HERMITE>(desc, off, aux, nodes, st);
    }
}

}  // namespace lbm

#define LBM_INSTANTIATE_FUSED(T, CV)                                                                            \
    template cudaError_t lbm::fused_launch_cv<T, CV>(const lbm::SimDesc *, const lbm::WorkItem *, const int *, \
                                                     int, int, int, int *, cudaStream_t);                      \
    template const void *lbm::fused_kernel_cv<T, CV>();                                                        \
    template int lbm::fused_smem_cv<T, CV>();

#define LBM_INSTANTIATE_TILE(T, CV)                                                                                  \
    template cudaError_t lbm::tile_launch_cv<T, CV>(const lbm::SimDesc *, int, int, bool, int, int, int, int *, cudaStream_t);

#define LBM_INSTANTIATE_TWOPASS(T) \
    template cudaError_t lbm::twopass_launch<T>(int, const lbm::SimDesc *, int, float *, long long, cudaStream_t);
