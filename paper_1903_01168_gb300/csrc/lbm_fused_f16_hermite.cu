// lbm_fused_f16_hermite.cu -- the fused step kernel for FP16 split-form deviation storage: BGK
// and MRT with the Hermite equilibrium and no-slip walls, periodic in x.
#include "lbm_inst.cuh"

LBM_INSTANTIATE_FUSED(__half, 2)
LBM_INSTANTIATE_TILE(__half, 2)
LBM_INSTANTIATE_FUSED(__half, 3)
LBM_INSTANTIATE_TILE(__half, 3)
