// sweep_f32_lean.cu -- the batched sweep kernels: FP32, without the paper's geometry.
#define PHAST_SWEEP_KERNELS
#include "sweep_kernels.cuh"

batched_fn pick_f32_lean(int tpw, bool lean) { return pick_batched32<false, false>(tpw, lean); }
