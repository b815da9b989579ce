// sweep_f32_geom_wide.cu -- the batched sweep kernels: a warp per walker for narrower tiles, FP32, with the paper's geometry.
#define PHAST_SWEEP_KERNELS
#include "sweep_kernels.cuh"

batched_fn pick_f32_geom_wide(int tpw, bool lean) { return pick_batched32_wide<true, true>(tpw, lean); }
