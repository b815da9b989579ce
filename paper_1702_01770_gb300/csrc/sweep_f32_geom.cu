// sweep_f32_geom.cu -- the batched sweep kernels: FP32, with the paper's geometry.
#define PHAST_SWEEP_KERNELS
#include "sweep_kernels.cuh"

batched_fn pick_f32_geom(int tpw, bool lean) { return pick_batched32<true, true>(tpw, lean); }
