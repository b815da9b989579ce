// sweep_f32_exact_wide.cu -- the batched sweep kernels: a warp per walker for narrower tiles, FP32, with the exact path of the torsion terms.
#define PHAST_SWEEP_KERNELS
#include "sweep_kernels.cuh"

batched_fn pick_f32_exact_wide(int tpw, bool lean) { return pick_batched32_wide<false, true>(tpw, lean); }
