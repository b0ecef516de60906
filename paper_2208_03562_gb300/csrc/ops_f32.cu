// ops_f32.cu -- kernels and launchers for float storage, float collision.
// Interior-kernel variants (tile w x h, CTA threads, CTAs per SM): PRC_VARIANT(64, 8, 256, 2), PRC_VARIANT(64, 16, 256, 2), PRC_VARIANT(64, 32, 512, 1), PRC_VARIANT(64, 16, 512, 1).
// Fused two-step kernel (tile w x h, CTA threads, CTAs per SM, stages).
#define PRC_S float
#define PRC_T float
#define PRC_OPS ops_f32
#define PRC_NVARIANTS 4
#define PRC_VARIANTS PRC_VARIANT(64, 8, 256, 2), PRC_VARIANT(64, 16, 256, 2), PRC_VARIANT(64, 32, 512, 1), PRC_VARIANT(64, 16, 512, 1)
#define PRC_NFUSED 2
#define PRC_FUSED PRC_FUSED_SHAPE(64, 32, 512, 1, 2), PRC_FUSED_SHAPE(64, 16, 256, 2, 1)
#include "prc_ops_impl.cuh"
