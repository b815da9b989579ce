// sweep_f32_lean_wide.cu -- the batched sweep kernels: a warp per walker for narrower tiles, FP32, without the paper's geometry.
#define PHAST_SWEEP_KERNELS
#include "sweep_kernels.cuh"

batched_fn pick_f32_lean_wide(int tpw, bool lean) { return pick_batched32_wide<false, false>(tpw, lean); }
