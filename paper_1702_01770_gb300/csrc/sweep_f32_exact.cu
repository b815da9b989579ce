// sweep_f32_exact.cu -- the batched sweep kernels: FP32, without the geometry, with the exact path of the torsion terms.
#define PHAST_SWEEP_KERNELS
#include "sweep_kernels.cuh"

batched_fn pick_f32_exact(int tpw, bool lean) { return pick_batched32<false, true>(tpw, lean); }
