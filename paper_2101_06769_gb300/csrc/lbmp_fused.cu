// lbmp_fused.cu -- the fused D3Q27 FP32 step and its batch form at the
// default 32 x 4 tile, with the pieces shared by every tile shape (the
// kernel source is lbmp_fused3_body.cuh).
// Two kernels: four CTAs (16 warps) per SM at 128 registers, and three that load
// f' one plane ahead; launch_shape_ahead takes one by size.  Ring phi from
// register loads, column and plane offsets in bytes.  On the 128x128x512 RT
// workload a step takes 0.725 ms with f' loaded ahead (on a slower GPU 0.734,
// and 0.738 without), 0.820 ms with the earlier arithmetic, which issued 2334
// instructions per cell, and two barriers per plane.  While the edges and corners
// of g were summed by Fast2Sum (PairOut), it took 0.715 and without loading ahead
// 0.736; measured then, without loading ahead: 3 or 5 CTAs per SM 0.747 / 0.745
// ms, element indices 0.732, a ring staged by cp.async 0.748, a 32 x 8 tile
// 0.778, and the same access pattern without arithmetic 0.706 ms.
#define LBMP_FUSED_MINB 4
#define LBMP_FUSED_AHEAD 1
#define LBMP_FUSED_BYTEOFF 4
#define LBMP_FUSED_RINGREG 1
#define LBMP_OUT_ORDERED 1
#define LBMP_FUSED3_LAUNCH launch_step_fused3
#define LBMP_BATCH3_OPS batch3_ops_32x4
#define LBMP_FUSED3_WITH_COMMON 1
#define LBMP_FUSED3_OBS 1
#define LBMP_FUSED3_OBS_LAUNCH launch_obs_fused3
#include "lbmp_fused3_body.cuh"
