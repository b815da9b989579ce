// sweep_f64.cu -- the batched sweep kernels: FP64.
#define PHAST_SWEEP_KERNELS
#include "sweep_kernels.cuh"

batched_fn pick_f64(int tpw, bool geom) { return geom ? pick_batched64<true>(tpw) : pick_batched64<false>(tpw); }
