// weights.cu -- Berg's multicanonical weight recursion with accumulated error
// weights (Sec. 2.2): histogram blocks summed, the slope update per adjacent bin
// pair, then lnW re-integrated from lnW_0 = 0 by a scan; plus the flatness
// statistics of Sec. 4.1.
//
// One cluster of kBergCtas CTAs per system type, every type in one launch.  The step is
// bound by latency: the histogram loads and one FP64 logarithm per visited bin (2100
// cycles a warp on this chip), so each CTA takes an eighth of the bins, sums and logs each
// bin once (in shared memory), and the sums and the scan's offsets are exchanged through
// distributed shared memory.  One launch for four system types takes 27 us (four launches of
// one CTA, the blocks summed four times and two logarithms a bin: 41 to 83 us each).
#include <cooperative_groups.h>

#include "common.cuh"

namespace cg = cooperative_groups;

namespace {

constexpr int kThreads = 512;
constexpr int kBergCtas = 8;                                        // a cluster
constexpr int kChunk = (PHAST_MAX_BINS + kBergCtas - 1) / kBergCtas;   // bins of one CTA
constexpr int kPer = kChunk / kThreads;                             // contiguous bins of one thread
static_assert(kPer * kThreads == kChunk, "a CTA's bins are whole per thread");

// Sum of v over the cluster, in rank order (the same value on every thread).
__device__ __forceinline__ double cluster_sum(cg::cluster_group& cl, double* s_part, double v, double* red) {
    v = block_sum(v, red);
    if (threadIdx.x == 0) *s_part = v;
    cl.sync();
    double s = 0.0;
    for (int c = 0; c < kBergCtas; ++c) s += *cl.map_shared_rank(s_part, c);
    return s;
}

__global__ void __launch_bounds__(kThreads) berg_kernel(const BergJobs jobs) {
    __shared__ double H[kChunk + 1], lg[kChunk + 1];   // count and its logarithm of this CTA's bins and the next one
    __shared__ double red[32], s_n, s_sum, s_var, s_max, s_tot, warp_tot[kThreads / 32];
    cg::cluster_group cl = cg::this_cluster();
    const BergJob& J = jobs.job[blockIdx.x / kBergCtas];
    const int K = J.K, rank = (int)cl.block_rank(), tid = threadIdx.x;
    const int chunk = (K + kBergCtas - 1) / kBergCtas;
    const int c0 = min(rank * chunk, K), c1 = min(c0 + chunk, K);   // this CTA's bins

    double n = 0.0, sum = 0.0;
    for (int q = tid; q <= c1 - c0 && c0 + q < K; q += kThreads) {
        unsigned long long s = 0;
        for (int b = 0; b < J.n_blocks; ++b) s += J.hist[(int64_t)b * K + c0 + q];
        const double h = (double)s;
        H[q] = h;
        lg[q] = s ? log(h) : 0.0;
        if (s && c0 + q < c1) { n += 1.0; sum += h; }
    }
    // flatness over visited bins
    n = cluster_sum(cl, &s_n, n, red);
    sum = cluster_sum(cl, &s_sum, sum, red);
    if (J.flat_out) {
        const double mean = n > 0.0 ? sum / n : 0.0;
        double var = 0.0, maxdev = 0.0;
        for (int q = tid; c0 + q < c1; q += kThreads) {
            const double h = H[q];
            if (h > 0.0) {
                var += (h - mean) * (h - mean);
                maxdev = fmax(maxdev, fabs(h - mean) / mean);
            }
        }
        for (int o = 16; o > 0; o >>= 1) maxdev = fmax(maxdev, __shfl_down_sync(0xffffffffu, maxdev, o));
        if ((tid & 31) == 0) warp_tot[tid >> 5] = maxdev;
        __syncthreads();
        if (tid == 0) {
            for (int i = 1; i < kThreads / 32; ++i) maxdev = fmax(maxdev, warp_tot[i]);
            s_max = maxdev;
        }
        var = cluster_sum(cl, &s_var, var, red);
        if (rank == 0 && tid == 0) {
            for (int c = 1; c < kBergCtas; ++c) maxdev = fmax(maxdev, *cl.map_shared_rank(&s_max, c));
            J.flat_out[0] = n;
            J.flat_out[1] = mean;
            J.flat_out[2] = mean > 0.0 ? sqrt(n > 0.0 ? var / n : 0.0) / mean : 0.0;
            J.flat_out[3] = maxdev;
        }
    }
    __syncthreads();

    // slope update: g0 = H_k H_{k+1} / (H_k + H_{k+1}), ghat = g0 / (g_acc + g0); the slope
    // differences lnW_k - lnW_{k+1} of this thread's contiguous bins
    double d[kPer], loc = 0.0;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        const int q = tid * kPer + i, k = c0 + q;
        d[i] = 0.0;
        if (k >= c1 || k + 1 >= K) continue;
        const double h0 = H[q], h1 = H[q + 1];
        const double g0 = (h0 > 0.0 && h1 > 0.0) ? h0 * h1 / (h0 + h1) : 0.0;
        const double den = J.g_acc[k] + g0;
        const double ghat = den > 0.0 ? g0 / den : 0.0;
        J.g_acc[k] = den;
        double dk = J.lnW[k] - J.lnW[k + 1];
        if (g0 > 0.0) dk += ghat * (lg[q + 1] - lg[q]);
        d[i] = dk;
        loc += dk;
        if (J.beta_out) J.beta_out[k] = dk / J.w;
    }
    // lnW_0 = 0, lnW_{k+1} = lnW_k - d_k: scan over the CTA's threads, then over the CTAs
    double incl = loc;
    for (int o = 1; o < 32; o <<= 1) {
        const double v = __shfl_up_sync(0xffffffffu, incl, o);
        if ((tid & 31) >= o) incl += v;
    }
    __syncthreads();   // warp_tot is free
    if ((tid & 31) == 31) warp_tot[tid >> 5] = incl;
    __syncthreads();
    double before = 0.0, total = 0.0;
    for (int i = 0; i < kThreads / 32; ++i) {
        before += i < (tid >> 5) ? warp_tot[i] : 0.0;
        total += warp_tot[i];
    }
    if (tid == 0) s_tot = total;
    cl.sync();   // every lnW of the cluster is read, the totals are there
    double run = before + (incl - loc);
    for (int c = 0; c < rank; ++c) run += *cl.map_shared_rank(&s_tot, c);
    if (rank == 0 && tid == 0) J.lnW[0] = 0.0;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        const int k = c0 + tid * kPer + i;
        if (k >= c1 || k + 1 >= K) break;
        run += d[i];
        J.lnW[k + 1] = -run;
    }
    cl.sync();   // no CTA leaves while another reads its sums
}

}  // namespace

int phast_launch_berg(const BergJobs& jobs, int n_jobs, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)n_jobs * kBergCtas);
    cfg.blockDim = dim3(kThreads);
    cfg.stream = st;
    cudaLaunchAttribute cluster;
    cluster.id = cudaLaunchAttributeClusterDimension;
    cluster.val.clusterDim.x = kBergCtas;
    cluster.val.clusterDim.y = cluster.val.clusterDim.z = 1;
    cfg.attrs = &cluster;
    cfg.numAttrs = 1;
    PHAST_CUDA_TRY(cudaLaunchKernelEx(&cfg, berg_kernel, jobs));
    return PHAST_OK;
}

extern "C" int phast_weight_update(int32_t K, double bin_width, const uint64_t* hist, int32_t n_blocks,
                                   double* lnW, double* g_acc, double* beta_out, double* flat_out, void* stream) {
    if (K < 1 || K > PHAST_MAX_BINS) return phast_set_error(PHAST_EINVAL, "phast_weight_update: K %d outside [1, %d]", K, PHAST_MAX_BINS);
    if (!(bin_width > 0.0)) return phast_set_error(PHAST_EINVAL, "phast_weight_update: bin_width must be > 0");
    if (n_blocks < 1) return phast_set_error(PHAST_EINVAL, "phast_weight_update: n_blocks < 1");
    if (!hist || !lnW || (K > 1 && !g_acc)) return phast_set_error(PHAST_EINVAL, "phast_weight_update: NULL argument");
    BergJobs jobs = {};
    jobs.job[0] = BergJob{K, n_blocks, bin_width, reinterpret_cast<const unsigned long long*>(hist), lnW, g_acc, beta_out, flat_out};
    return phast_launch_berg(jobs, 1, (cudaStream_t)stream);
}
