// lbmp_fused_r.cu -- the fused D3Q27 FP32 step with the phase field on the
// reduced lattice D3Q7 (first-order equilibrium and correction term,
// Sec. 2.2), 32 x 4 tiles (kernel source lbmp_fused3_body.cuh), four CTAs
// (16 warps) per SM.  0.443 ms per step on the 128x128x512 RT workload (0.581
// with the earlier arithmetic; 0.447 with 32 planes per item, and there with
// f' loaded one plane ahead 0.458, element indices 0.457, five CTAs per SM
// 0.456, the ring's g from register loads 0.516).
#define LBMP_PHASE_REDUCED 1
#define LBMP_FUSED_MINB 4
#define LBMP_FUSED_BYTEOFF 4
#define LBMP_TILE_NS tile_red
#define LBMP_FUSED3_LAUNCH launch_step_fused3_red
#define LBMP_BATCH3_OPS batch3_ops_red
#define LBMP_FUSED3_WITH_COMMON 0
#define LBMP_FUSED3_OBS 1
#define LBMP_FUSED3_OBS_LAUNCH launch_obs_fused3_red
#include "lbmp_fused3_body.cuh"
