// sweep_lane.cu -- the batched sweep kernels: one walker per thread.
#define PHAST_SWEEP_KERNELS
#include "sweep_kernels.cuh"

batched_fn pick_lane(bool fp32, bool geom, bool shared_trials) {
    if (!fp32) return geom ? sweep_lane_kernel<double, true, false> : sweep_lane_kernel<double, false, false>;
    if (shared_trials) return geom ? sweep_lane_kernel<float, true, true> : sweep_lane_kernel<float, false, true>;
    return geom ? sweep_lane_kernel<float, true, false> : sweep_lane_kernel<float, false, false>;
}
