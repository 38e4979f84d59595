// lbmp_fused_t16x8.cu -- the fused D3Q27 FP32 step and its batch form at a
// 16 x 8 tile (a launch shape of the autotuners; kernel source
// lbmp_fused3_body.cuh).
// Four CTAs (16 warps) per SM at 128 registers, ring phi from register loads,
// column and plane offsets in bytes, f' loaded in its own plane.  On the
// 128x128x512 RT workload a step takes 0.753 ms (0.738 at 32 x 4):
// half-warp rows take more L1 and L2 transactions per byte; the smaller
// ring pays on narrow domains only.
#define LBMP_FUSED_MINB 4
#define LBMP_FUSED_BYTEOFF 4
#define LBMP_FUSED_RINGREG 1
#define LBMP_OUT_ORDERED 1
#define LBMP_FUSED_TX 16
#define LBMP_FUSED_TY 8
#define LBMP_TILE_NS tile16x8
#define LBMP_FUSED3_LAUNCH launch_step_fused3_t16x8
#define LBMP_BATCH3_OPS batch3_ops_16x8
#define LBMP_FUSED3_WITH_COMMON 0
#include "lbmp_fused3_body.cuh"
