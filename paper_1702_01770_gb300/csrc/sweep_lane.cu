// sweep_lane.cu -- the batched sweep kernels: one walker per thread.
#define PHAST_SWEEP_KERNELS
#include "sweep_kernels.cuh"

batched_fn pick_lane(bool fp32, bool geom) {
    return geom ? (fp32 ? sweep_lane_kernel<float, true> : sweep_lane_kernel<double, true>)
                : (fp32 ? sweep_lane_kernel<float, false> : sweep_lane_kernel<double, false>);
}
