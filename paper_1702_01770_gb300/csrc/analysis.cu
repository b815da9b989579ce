// analysis.cu -- microcanonical analysis (Eq. 4-6; ANALYST of Sec. 3.3) with
// canonical reweighting, and error bars either by a jackknife over histogram
// blocks (replicate 0 uses every block; replicate r >= 1 leaves block r-1 out)
// or by binning over iterations (replicate i is iteration i, with its own
// weights and histogram; Sec. 4.1).
//   kernels 1, 2, 4 (a CTA per replicate and 256 bins): -lnW + ln H, S_k, beta_k and C_V,k;
//   kernel 3 (a cluster per temperature): <E>_T and c_V(T) of all replicates;
//   kernel 5 (a CTA per 128 bins and quantity, one for the temperatures): c_V peak per
//   replicate, values and errors.
// All of it is FP64 (64 cycles of an SMSP's pipe per instruction and warp), so the work is
// spread over every SM and each exponential is taken once.  K = 8000, 64 temperatures, 16
// blocks: 12, 7, 198, 12 and 14 us for the five (about 5.4 ms for the analysis with one CTA
// per replicate, two exponentials a bin, replicate and temperature, and one CTA for the errors).
#include <cooperative_groups.h>

#include "exp64.cuh"

namespace cg = cooperative_groups;

namespace {

constexpr int kThreads = 512;

struct Work {
    double *S, *beta, *CV, *ET, *cVT, *peak;   // [R][K] x3, [R][n_T] x2, [R][2]
};

__host__ __device__ inline size_t work_doubles(int K, int n_T, int R) {
    return (size_t)R * (3 * (size_t)K + 2 * (size_t)n_T + 2);
}

__host__ __device__ inline Work carve(double* base, int K, int n_T, int R) {
    Work w;
    w.S = base;
    w.beta = w.S + (size_t)R * K;
    w.CV = w.beta + (size_t)R * K;
    w.ET = w.CV + (size_t)R * K;
    w.cVT = w.ET + (size_t)R * n_T;
    w.peak = w.cVT + (size_t)R * n_T;
    return w;
}

__device__ __forceinline__ double block_max(double v, double* red) {
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_down_sync(0xffffffffu, v, o));
    int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = (blockDim.x + 31) >> 5;
    __syncthreads();
    if (l == 0) red[w] = v;
    __syncthreads();
    if (w == 0) {
        v = (l < nw) ? red[l] : -INFINITY;
        for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_down_sync(0xffffffffu, v, o));
        if (l == 0) red[0] = v;
    }
    __syncthreads();
    double r = red[0];
    __syncthreads();
    return r;
}

// H_k of replicate r (block r-1 left out for r >= 1); -1 when no histogram.
__device__ __forceinline__ double rep_hist(const unsigned long long* hist, int n_blocks, int K, int r, int k) {
    if (!hist) return -1.0;
    unsigned long long s = 0;
    for (int b = 0; b < n_blocks; ++b)
        if (b != r - 1) s += hist[(int64_t)b * K + k];
    return (double)s;
}

// E_k = e_min + (k + 1/2) w of bin k, with one fused multiply-add.
__device__ __forceinline__ double bin_energy(double e_min, double w, int k) {
    const double two = count_to_f64(2 * k + 1);   // k + 1/2, halved by its exponent
    return __fma_rn(__hiloint2double(__double2hiint(two) - 0x00100000, 0), w, e_min);
}

constexpr int kEntropyThreads = 256;
__host__ __device__ inline int bin_ctas(int K) { return (K + kEntropyThreads - 1) / kEntropyThreads; }

// -lnW_k + ln H_k of one bin and replicate a thread (NaN: unvisited).
// iters: replicate r is iteration r (weights row r, histogram row r); else the
// jackknife replicates of the histogram blocks with one weight table.
__global__ void __launch_bounds__(kEntropyThreads)
log_kernel(int K, const double* __restrict__ lnW, const unsigned long long* __restrict__ hist, int n_blocks, Work wk,
           int iters) {
    const int r = blockIdx.x / bin_ctas(K), k = (blockIdx.x - r * bin_ctas(K)) * kEntropyThreads + threadIdx.x;
    if (k >= K) return;
    if (iters) lnW += (size_t)r * K;
    const double H = iters ? (hist ? (double)hist[(size_t)r * K + k] : -1.0) : rep_hist(hist, n_blocks, K, r, k);
    double s = __longlong_as_double(0x7ff8000000000000ll);
    if (H < 0.0) s = -lnW[k];
    else if (H > 0.0) s = -lnW[k] + log(H);
    wk.beta[(size_t)r * K + k] = s;   // held in beta's place until entropy_kernel has read it,
    wk.CV[(size_t)r * K + k] = H < 0.0 ? 1.0 : H;   // the counts in C_V's until canonical_kernel has
}

// S_k (shifted to max S = 0) of one bin and replicate a thread, from log_kernel's values;
// every CTA takes the replicate's maximum itself (the bins stay in L2).
__global__ void __launch_bounds__(kEntropyThreads)
entropy_kernel(int K, Work wk) {
    __shared__ long long red[32];
    const int r = blockIdx.x / bin_ctas(K);
    const double* raw = wk.beta + (size_t)r * K;
    long long top = PHAST_KEY_LOWEST;
#pragma unroll 8
    for (int k = threadIdx.x; k < K; k += kEntropyThreads) {
        const double s = raw[k];
        top = is_nan64(s) ? top : max(top, order_key(s));
    }
    const double mx = key_value(block_max_key(top, red));
    const int k = (blockIdx.x - r * bin_ctas(K)) * kEntropyThreads + threadIdx.x;
    if (k < K) wk.S[(size_t)r * K + k] = is_nan64(raw[k]) ? raw[k] : raw[k] - mx;
}

// beta_k and C_V,k of one bin and replicate a thread.
__global__ void __launch_bounds__(kEntropyThreads)
slopes_kernel(int K, double w, int h, Work wk) {
    const int r = blockIdx.x / bin_ctas(K), k = (blockIdx.x - r * bin_ctas(K)) * kEntropyThreads + threadIdx.x;
    if (k >= K) return;
    const double* S = wk.S + (size_t)r * K;
    const double nan = __longlong_as_double(0x7ff8000000000000ll);
    const double he = (double)h * w;
    double b = nan, cv = nan;
    if (k - h >= 0 && k + h < K && !is_nan64(S[k - h]) && !is_nan64(S[k + h])) {
        b = (S[k + h] - S[k - h]) / (2.0 * he);
        if (!is_nan64(S[k])) {
            double s2 = (S[k + h] - 2.0 * S[k] + S[k - h]) / (he * he);
            cv = -(b * b) / s2;
        }
    }
    wk.beta[(size_t)r * K + k] = b;
    wk.CV[(size_t)r * K + k] = cv;
}

// Canonical averages.  A cluster of kCanonicalCtas CTAs takes one temperature and all
// jackknife replicates (or one iteration), each CTA a quarter of the bins.  With S_k = -lnW_k
// + ln H_k the canonical weight of a bin is H_k exp(-lnW_k - E_k / T): the exponential is the
// same for every replicate, which differ in the counts only, so it is taken once per bin and
// temperature and a replicate costs 3 FP64 instructions a bin.  1/T enters as two FP64
// numbers, so the exponent carries only the roundings of its sums.  The moments of the
// replicates are taken about the full histogram's mean; a replicate whose own mean is more than
// half its spread from it (the shift would cost its variance digits: at eight spreads an error of
// 4e-14 of a jackknife error, 7e-16 about its own mean), or whose weights all underflow beside the
// full histogram's largest, is taken again about its own; so is the full histogram itself where one
// bin has all but nothing of the weight and the rounding of its mean would be more than its spread.
constexpr int kCanonicalThreads = kEntropyThreads;
constexpr int kCanonicalCtas = 4;
constexpr int kCanonicalBins = (PHAST_MAX_BINS + kCanonicalCtas - 1) / kCanonicalCtas;
constexpr int kGroup = 6;   // replicates side by side

// Sums v over the cluster's CTAs, in rank order; every thread receives them.  s_part: room
// for M doubles, used again by a later call only after another call's barrier.
template <int M>
__device__ __forceinline__ void cluster_sums(cg::cluster_group& cl, double* s_part, double (&v)[M], double* red) {
    // [warp][M] partials, then one thread a sum
    int first = 0, count = M;
    warp_sums<M>(v, &first, &count);
    __syncthreads();
    if (count == 1) red[(threadIdx.x >> 5) * M + first] = v[0];
    __syncthreads();
    if (threadIdx.x < M) {
        double s = 0.0;
        for (int w = 0; w < kCanonicalThreads / 32; ++w) s += red[w * M + threadIdx.x];
        s_part[threadIdx.x] = s;
    }
    cl.sync();
#pragma unroll
    for (int q = 0; q < M; ++q) {
        double s = 0.0;
        for (int c = 0; c < kCanonicalCtas; ++c) s += cl.map_shared_rank(s_part, c)[q];
        v[q] = s;
    }
}

__global__ void __launch_bounds__(kCanonicalThreads)
canonical_kernel(int K, double e_min, double w, const double* __restrict__ lnW, int R, int iters,
                 const double* __restrict__ T, int n_T, int n_monomers, Work wk) {
    __shared__ double base[kCanonicalBins];   // exp(-lnW_k - E_k / T - max) of this CTA's bins
    __shared__ double red[kCanonicalThreads / 32 * 3 * kGroup], s_part[2][3 * kGroup];
    __shared__ long long s_max;
    cg::cluster_group cl = cg::this_cluster();
    const int job = blockIdx.x / kCanonicalCtas, i = job % n_T, rank = (int)cl.block_rank();
    const int r_first = iters ? job / n_T : 0, n_rep = iters ? 1 : R;
    const double* H = wk.CV + (size_t)r_first * K;   // log_kernel's counts, a row a replicate
    if (iters) lnW += (size_t)r_first * K;
    const int chunk = (K + kCanonicalCtas - 1) / kCanonicalCtas;
    const int k0 = min(rank * chunk, K), k1 = min(k0 + chunk, K);
    const double Ti = T[i];
    const double rT = 1.0 / Ti;
    double rT2 = __fma_rn(-rT, Ti, 1.0) * rT;
    if (!is_finite64(rT2)) rT2 = 0.0;   // T = 0 or infinite
    long long top = PHAST_KEY_LOWEST;
    for (int k = k0 + threadIdx.x; k < k1; k += kCanonicalThreads) {
        double g = __longlong_as_double(0x7ff8000000000000ll);
        if (__double_as_longlong(H[k]) != 0) {
            const double Ek = bin_energy(e_min, w, k);
            g = __fma_rn(-Ek, rT2, __fma_rn(-Ek, rT, -lnW[k]));
            if (!is_nan64(g)) top = max(top, order_key(g));
        }
        base[k - k0] = g;   // read back by the same thread
    }
    top = block_max_key(top, reinterpret_cast<long long*>(red));
    if (threadIdx.x == 0) s_max = top;
    cl.sync();
    for (int c = 0; c < kCanonicalCtas; ++c) top = max(top, *cl.map_shared_rank(&s_max, c));
    const double gmax = key_value(top);
    double first[2] = {0.0, 0.0};   // Z and sum p E of the full histogram
    for (int k = k0 + threadIdx.x; k < k1; k += kCanonicalThreads) {
        double v = base[k - k0];
        v = is_nan64(v) ? 0.0 : exp64_neg(v - gmax);
        base[k - k0] = v;
        if (__double_as_longlong(v) == 0) continue;
        v *= H[k];
        first[0] += v;
        first[1] = __fma_rn(v, bin_energy(e_min, w, k), first[1]);
    }
    cluster_sums<2>(cl, s_part[0], first, red);
    const double m0 = first[1] / first[0];
    int use = 1;
    for (int r0 = 0; r0 < n_rep; r0 += kGroup, use ^= 1) {
        double m[3 * kGroup];   // Z, sum p c, sum p c c with c = E - m0, of kGroup replicates
#pragma unroll
        for (int q = 0; q < 3 * kGroup; ++q) m[q] = 0.0;
        for (int k = k0 + threadIdx.x; k < k1; k += kCanonicalThreads) {
            const double v = base[k - k0];
            if (__double_as_longlong(v) == 0) continue;
            const double c = bin_energy(e_min, w, k) - m0, vc = v * c, vcc = vc * c;
            double n[kGroup];
#pragma unroll
            for (int q = 0; q < kGroup; ++q) n[q] = r0 + q < n_rep ? H[(size_t)(r0 + q) * K + k] : 0.0;
#pragma unroll
            for (int q = 0; q < kGroup; ++q) {
                if (r0 + q >= n_rep) break;
                m[3 * q] = __fma_rn(n[q], v, m[3 * q]);
                m[3 * q + 1] = __fma_rn(n[q], vc, m[3 * q + 1]);
                m[3 * q + 2] = __fma_rn(n[q], vcc, m[3 * q + 2]);
            }
        }
        cluster_sums<3 * kGroup>(cl, s_part[use], m, red);
#pragma unroll
        for (int q = 0; q < kGroup; ++q) {
            const int r = r0 + q;
            if (r >= n_rep) break;
            const double Z = m[3 * q], d = m[3 * q + 1] / Z, raw = m[3 * q + 2] / Z;
            double mean = m0 + d, var = raw - d * d;
            // too far from the full histogram's mean, or every weight (nearly) underflowed: the same on every thread
            if (!(d * d <= 0.25 * var && Z >= 1e-280)) {
                const double* S = wk.S + (size_t)(r_first + r) * K;
                double lmax = -INFINITY, z[2] = {0.0, 0.0};
                auto arg = [&](int k) -> double {
                    const double Ek = bin_energy(e_min, w, k);
                    return __fma_rn(-Ek, rT2, __fma_rn(-Ek, rT, S[k]));
                };
                for (int k = threadIdx.x; k < K; k += kCanonicalThreads)
                    if (!is_nan64(S[k])) lmax = fmax(lmax, arg(k));
                lmax = block_max(lmax, red);
                for (int k = threadIdx.x; k < K; k += kCanonicalThreads) {
                    if (is_nan64(S[k])) continue;
                    const double p = exp64_neg(arg(k) - lmax);
                    z[0] += p;
                    z[1] = __fma_rn(p, bin_energy(e_min, w, k), z[1]);
                }
                const double Zr = block_sum(z[0], red);
                mean = block_sum(z[1], red) / Zr;
                double s = 0.0;
                for (int k = threadIdx.x; k < K; k += kCanonicalThreads) {
                    if (is_nan64(S[k])) continue;
                    const double e = bin_energy(e_min, w, k) - mean;
                    s += exp64_neg(arg(k) - lmax) * e * e;
                }
                var = block_sum(s, red) / Zr;
            }
            if (rank == 0 && threadIdx.x == 0) {
                wk.ET[(size_t)(r_first + r) * n_T + i] = mean;
                wk.cVT[(size_t)(r_first + r) * n_T + i] = var / ((double)n_monomers * Ti * Ti);
            }
        }
    }
    cl.sync();   // no CTA leaves while another reads its sums
}

__device__ __forceinline__ void jackknife(const double* v, size_t stride, int n, double* val, double* err,
                                          size_t idx) {
    // v[0] full estimate, v[r * stride] leave-block-(r-1)-out replicates
    if (val) val[idx] = v[0];
    if (!err) return;
    if (n < 2) { err[idx] = __longlong_as_double(0x7ff8000000000000ll); return; }
    double m = 0.0;
#pragma unroll 8
    for (int r = 1; r <= n; ++r) m += v[r * stride];
    m /= n;
    double s = 0.0;
#pragma unroll 8
    for (int r = 1; r <= n; ++r) {
        const double d = v[r * stride] - m;
        s += d * d;
    }
    err[idx] = sqrt((double)(n - 1) / n * s);
}

// Binning over rows 0 .. n_b * block - 1 of v (stride apart), n_b = R / block:
// the mean of the block means and their standard error (NaN for n_b < 2), with
// the oracle's order of summation.
__device__ __forceinline__ void binning(const double* v, size_t stride, int R, int block, double* val, double* err,
                                        size_t idx) {
    const int n_b = R / block;
    double mean = 0.0;
    for (int b = 0; b < n_b; ++b) {
        double s = 0.0;
        for (int i = b * block; i < (b + 1) * block; ++i) s = s + v[(size_t)i * stride];
        mean = mean + s / (double)block;
    }
    mean = mean / (double)n_b;
    if (val) val[idx] = mean;
    if (!err) return;
    if (n_b < 2) { err[idx] = __longlong_as_double(0x7ff8000000000000ll); return; }
    double q = 0.0;
    for (int b = 0; b < n_b; ++b) {
        double s = 0.0;
        for (int i = b * block; i < (b + 1) * block; ++i) s = s + v[(size_t)i * stride];
        const double d = s / (double)block - mean;
        q = q + d * d;
    }
    err[idx] = sqrt(q / ((double)n_b * (double)(n_b - 1)));
}

// Values and errors: block > 0: binning over iterations in blocks of `block`; else the
// jackknife over the n_jk leave-one-block-out replicates.  CTA (x, y) takes 128 bins of S,
// beta or C_V (y = 0, 1, 2); the last x takes the temperatures and, for y = 2, the c_V peak
// of each replicate (a warp each: grid maximum, refined by a parabola through it and its
// neighbours, a thread each) and its error.
constexpr int kFinishThreads = 128;

__global__ void __launch_bounds__(kFinishThreads)
finish_kernel(int K, const double* __restrict__ T, int n_T, int R, int n_jk, Work wk, phast_micro_out o,
              int block) {
    const int q = blockIdx.y;
    auto both = [&](const double* v, size_t stride, double* val, double* err, size_t idx) {
        if (block > 0) binning(v, stride, R, block, val, err, idx);
        else jackknife(v, stride, n_jk, val, err, idx);
    };
    const int k = blockIdx.x * kFinishThreads + threadIdx.x;
    if (blockIdx.x + 1 < gridDim.x) {
        if (k >= K) return;
        if (q == 0) both(wk.S + k, (size_t)K, o.S, o.S_err, k);
        if (q == 1) both(wk.beta + k, (size_t)K, o.beta, o.beta_err, k);
        if (q == 2) both(wk.CV + k, (size_t)K, o.CV, o.CV_err, k);
        return;
    }
    if (q < 2) {
        for (int i = threadIdx.x; i < n_T; i += kFinishThreads) {
            if (q == 0) both(wk.ET + i, (size_t)n_T, o.E_T, o.E_T_err, i);
            else both(wk.cVT + i, (size_t)n_T, o.cV_T, o.cV_T_err, i);
        }
        return;
    }
    const int lane = threadIdx.x & 31;
    for (int r = threadIdx.x >> 5; r < R && n_T > 0; r += kFinishThreads / 32) {
        // the first of the largest values; NaN never replaces one, and a NaN in front stays
        const double* c = wk.cVT + (size_t)r * n_T;
        long long best = 0;
        int im = INT_MAX;
        for (int i = lane; i < n_T; i += 32) {
            const long long key = order_key(c[i] + 0.0);   // -0 counts as 0
            if (!is_nan64(c[i]) && (im == INT_MAX || key > best)) { best = key; im = i; }
        }
        for (int w = 16; w > 0; w >>= 1) {
            const long long v = __shfl_xor_sync(0xffffffffu, best, w);
            const int iv = __shfl_xor_sync(0xffffffffu, im, w);
            if (iv != INT_MAX && (im == INT_MAX || v > best || (v == best && iv < im))) { best = v; im = iv; }
        }
        if (lane == 0) wk.peak[2 * (size_t)r] = (double)(im == INT_MAX || is_nan64(c[0]) ? 0 : im);
    }
    __syncthreads();
    for (int r = threadIdx.x; r < R; r += kFinishThreads) {
        const double* c = wk.cVT + (size_t)r * n_T;
        double* pk = wk.peak + 2 * (size_t)r;
        if (n_T < 1) {
            pk[0] = pk[1] = __longlong_as_double(0x7ff8000000000000ll);
            continue;
        }
        const int im = (int)pk[0];
        pk[0] = T[im];
        pk[1] = c[im];
        if (im > 0 && im < n_T - 1) {
            double x0 = T[im - 1], x1 = T[im], x2 = T[im + 1], y0 = c[im - 1], y1 = c[im], y2 = c[im + 1];
            double num = (x1 - x0) * (x1 - x0) * (y1 - y2) - (x1 - x2) * (x1 - x2) * (y1 - y0);
            double den = (x1 - x0) * (y1 - y2) - (x1 - x2) * (y1 - y0);
            if (den != 0.0) {
                double xs = x1 - 0.5 * num / den;
                pk[0] = xs;
                pk[1] = y0 * (xs - x1) * (xs - x2) / ((x0 - x1) * (x0 - x2)) +
                        y1 * (xs - x0) * (xs - x2) / ((x1 - x0) * (x1 - x2)) +
                        y2 * (xs - x0) * (xs - x1) / ((x2 - x0) * (x2 - x1));
            }
        }
    }
    __syncthreads();
    if (threadIdx.x < 2) both(wk.peak + threadIdx.x, 2, o.peak, o.peak_err, threadIdx.x);
}

// The analysis of R replicates on stream st (workspace carved into wk).
int launch_micro(int K, double e_min, double w, const double* lnW, const uint64_t* hist, int n_blocks, int h,
                 int n_monomers, int n_T, const double* T, const phast_micro_out& out, const Work& wk, int R, int n_jk,
                 int iters, int block, cudaStream_t st) {
    const unsigned bins = (unsigned)R * (unsigned)bin_ctas(K);
    log_kernel<<<bins, kEntropyThreads, 0, st>>>(K, lnW, reinterpret_cast<const unsigned long long*>(hist), n_blocks, wk,
                                                 iters);
    PHAST_CUDA_TRY(cudaGetLastError());
    entropy_kernel<<<bins, kEntropyThreads, 0, st>>>(K, wk);
    PHAST_CUDA_TRY(cudaGetLastError());
    if (n_T > 0) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)n_T * (iters ? R : 1) * kCanonicalCtas);
        cfg.blockDim = dim3(kCanonicalThreads);
        cfg.stream = st;
        cudaLaunchAttribute cluster;
        cluster.id = cudaLaunchAttributeClusterDimension;
        cluster.val.clusterDim.x = kCanonicalCtas;
        cluster.val.clusterDim.y = cluster.val.clusterDim.z = 1;
        cfg.attrs = &cluster;
        cfg.numAttrs = 1;
        PHAST_CUDA_TRY(cudaLaunchKernelEx(&cfg, canonical_kernel, K, e_min, w, lnW, R, iters, T, n_T, n_monomers, wk));
    }
    slopes_kernel<<<bins, kEntropyThreads, 0, st>>>(K, w, h, wk);
    PHAST_CUDA_TRY(cudaGetLastError());
    finish_kernel<<<dim3((K + kFinishThreads - 1) / kFinishThreads + 1, 3), kFinishThreads, 0, st>>>(
        K, T, n_T, R, n_jk, wk, out, block);
    PHAST_CUDA_TRY(cudaGetLastError());
    return PHAST_OK;
}

// ---------------------------------------------------------------------------
// Free energy (Eq. 7) and the Maxwell construction on the caloric curve
// (ANALYST's Tol_Beta / Tol_L): the equal-area line on beta(E) is the common
// tangent of S(E), an edge of the upper concave hull of (E_k, S_k) over the
// visited bins that spans bins below it.  Among those with a positive slope
// (beta_c = 1/T_c > 0), a latent heat of at least tol_L, and across which
// beta_k = (S_{k+h} - S_{k-h}) / (2 h w) rises by at least tol_beta, the widest
// is taken (the first of equal width).
//
// One cluster of kMaxwellCtas CTAs per replicate, S in the first one's shared memory; the
// logarithms and f are shared by all of them.  The hull's definition is Andrew's monotone
// chain with one FP64 orientation test throughout (chain_drops), so that its vertices are
// those of the sequential definition even for nearly collinear bins.  A serial chain is
// bound by the latency of its FP64 tests (1090 cycles a bin), so the hull is found by all
// threads instead: bins clearly below a chord of two others are removed, round after round
// with chords of several spans, until every remaining bin lies clearly above the chord of
// its neighbours -- those are the hull's vertices, and the sequential test would decide the
// same at each of them, since "clearly" is a change of slope over 1e-9 of the slopes where
// the test's rounding is below 1e-11.  If some triple is not clear, the chain itself runs.
// The edges, the rise of beta along them, the barrier and f run on all threads.
// A cluster's CTAs first thin a stretch of the bins each (a bin below its stretch's hull is
// below the whole one), then one of them the four hulls put together.
// K = 8000, 17 replicates: 132 us (4.6 ms with the chain on one thread; 240 us with all bins
// on one CTA and every span in each round; on clusters of 2 and 8 CTAs 192 and 204 us).
// ---------------------------------------------------------------------------

// E_k = e_min + (k + 1/2) w, each operation rounded separately.
__device__ __forceinline__ double bin_centre(double e_min, double w, int k) {
    return __dadd_rn(e_min, __dmul_rn(__dadd_rn((double)k, 0.5), w));
}

// Monotone-chain test: drop j (i < j < k) when it lies on or below the chord
// from i to k.
__device__ __forceinline__ bool chain_drops(const double* S, double e_min, double w, int i, int j, int k) {
    const double ei = bin_centre(e_min, w, i), ej = bin_centre(e_min, w, j), ek = bin_centre(e_min, w, k);
    return __dmul_rn(__dsub_rn(S[j], S[i]), __dsub_rn(ek, ei)) <= __dmul_rn(__dsub_rn(S[k], S[i]), __dsub_rn(ej, ei));
}

constexpr size_t kMaxwellSmemPerBin = sizeof(double) + sizeof(int) + 1;   // S, hull, precomputed test
constexpr int kMaxwellCtas = 4;                                           // a cluster, one per replicate

// Removes from the list hull[0..nh) of visited bins those clearly below the chord of the
// list's members `span` before and after them, in place; the rest keeps its order.  F64: the
// FP64 test, else an FP32 one with its error bound (it only removes).  *unsure is set where
// the FP64 test is not clear.  Every thread receives the new length.  Members to the left of
// a chunk may have been moved down by an earlier one: any visited bins to the left and to the
// right make a valid chord.
__device__ __forceinline__ bool is_negative64(double x) {   // x < 0, without an FP64 comparison
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    return b > 0x8000000000000000ull && b <= 0xfff0000000000000ull;
}

template <bool F64>
__device__ int thin_hull(const double* S, int* hull, int nh, int span, int* counts, bool* unsure) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int out = 0;
    bool un = false;
    for (int base = 0; base < nh; base += kThreads) {
        const int p = base + threadIdx.x;
        bool keep = p < nh;
        const int j = keep ? hull[p] : 0;
        if (p > 0 && p + 1 < nh) {
            const int i = hull[max(p - span, 0)], k = hull[min(p + span, nh - 1)];
            const int n1 = j - i, n2 = k - j;   // > 0
            if constexpr (F64) {
                const double a1 = (S[j] - S[i]) * count_to_f64(n2), a2 = (S[k] - S[j]) * count_to_f64(n1);
                const double c = a1 - a2, m = 1e-9 * (fabs(a1) + fabs(a2));
                const bool below = is_negative64(c + m), above = is_negative64(m - c);
                keep = !below;
                un |= !below && !above;
            } else {
                const float si = f64_to_f32(S[i]), sj = f64_to_f32(S[j]), sk = f64_to_f32(S[k]);
                const float f1 = (float)n1, f2 = (float)n2;
                const float a1 = (sj - si) * f2, a2 = (sk - sj) * f1;
                const float m = 1e-6f * (fabsf(a1) + fabsf(a2)) + 1.3e-7f * ((fabsf(si) + fabsf(sj)) * f2 + (fabsf(sj) + fabsf(sk)) * f1);
                keep = !(a1 - a2 < -m);
            }
        }
        const unsigned b = __ballot_sync(0xffffffffu, keep);
        if (lane == 0) counts[warp] = __popc(b);
        __syncthreads();   // the chunk is read, its counts are written
        int before = 0, total = 0;
#pragma unroll
        for (int w = 0; w < kThreads / 32; ++w) {
            const int c = counts[w];
            before += w < warp ? c : 0;
            total += c;
        }
        if (keep) hull[out + before + __popc(b & ((1u << lane) - 1u))] = j;
        out += total;
        __syncthreads();
    }
    *unsure = __syncthreads_or(un);
    return out;
}

// The visited bins of [k0, k1) in order; every thread receives their number.
__device__ int visited_bins(const double* S, int k0, int k1, int* hull, int* counts) {
    int nh = 0;
    for (int base = k0; base < k1; base += kThreads) {
        const int k = base + threadIdx.x;
        const bool in = k < k1 && is_finite64(S[k]);
        const unsigned b = __ballot_sync(0xffffffffu, in);
        if ((threadIdx.x & 31) == 0) counts[threadIdx.x >> 5] = __popc(b);
        __syncthreads();
        int before = 0, total = 0;
#pragma unroll
        for (int q = 0; q < kThreads / 32; ++q) {
            before += q < (int)(threadIdx.x >> 5) ? counts[q] : 0;
            total += counts[q];
        }
        if (in) hull[nh + before + __popc(b & ((1u << (threadIdx.x & 31)) - 1u))] = k;
        nh += total;
        __syncthreads();
    }
    return nh;
}

// Thins the list to its hull: FP32 rounds while they still remove a sixteenth of it, then
// FP64 ones until none is removed.  A round takes chords of longer and longer spans while
// they still remove something (8000 noisy bins: 25 passes, 48 with every span in each round).
__device__ int thin_rounds(const double* S, int* hull, int nh, int* counts, bool* unsure) {
    bool f64 = false, u;
    for (;;) {
        const int n0 = nh;
        for (int span = 1; span == 1 || span < nh; span *= 4) {
            const int n = nh;
            nh = f64 ? thin_hull<true>(S, hull, nh, span, counts, &u) : thin_hull<false>(S, hull, nh, span, counts, &u);
            if (span == 1) *unsure = u;
            if (nh == n) break;
        }
        if (f64 && nh == n0) return nh;
        f64 = f64 || nh >= n0 - n0 / 16;
    }
}

// x / b rounded correctly from rb = 1 / b (div_count's correction); plain outside the range
// where the products stay normal.
__device__ __forceinline__ double quot(double x, double b, double rb, bool safe) {
    if (!safe) return x / b;
    const double q = __dmul_rn(x, rb);
    return __fma_rn(__fma_rn(-q, b, x), rb, q);
}
__device__ __forceinline__ bool quot_safe(double b) { return fabs(b) > 1e-100 && fabs(b) < 1e100; }

__global__ void __launch_bounds__(kThreads)
maxwell_kernel(int K, double e_min, double w, const double* __restrict__ lnW,
               const unsigned long long* __restrict__ hist, int n_blocks, int h, int n_monomers, double beta_c_in,
               double tol_beta, double tol_L, double* __restrict__ f_out, double* __restrict__ rep, int fast_hull) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double* S = reinterpret_cast<double*>(smem_raw);                                       // [K]
    int* hull = reinterpret_cast<int*>(smem_raw + sizeof(double) * (size_t)K);             // [K]
    uint8_t* pre = smem_raw + (sizeof(double) + sizeof(int)) * (size_t)K;                  // [K]
    __shared__ double red[32];
    __shared__ int counts[kThreads / 32];
    __shared__ int s_nh, s_best_q;
    __shared__ long long s_top;
    __shared__ double s_bc;
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int r = blockIdx.x / kMaxwellCtas;
    const double nan = __longlong_as_double(0x7ff8000000000000ll);
    const double N = (double)n_monomers;
    double* S0 = cluster.map_shared_rank(S, 0);
    // each CTA has a stretch of the bins (at their own places in its S)
    const int share = (K + kMaxwellCtas - 1) / kMaxwellCtas, k0 = min(rank * share, K), k1 = min(k0 + share, K);
    long long top = PHAST_KEY_LOWEST;
    for (int k = k0 + threadIdx.x; k < k1; k += kThreads) {
        const double H = rep_hist(hist, n_blocks, K, r, k);
        double s = nan;
        if (H < 0.0) s = -lnW[k];
        else if (H > 0.0) s = -lnW[k] + log(H);
        S[k] = s;
        if (!is_nan64(s)) top = max(top, order_key(s));
    }
    top = block_max_key(top, reinterpret_cast<long long*>(red));
    if (threadIdx.x == 0) s_top = top;
    cluster.sync();
    for (int c = 0; c < kMaxwellCtas; ++c) top = max(top, *cluster.map_shared_rank(&s_top, c));
    const double mx = key_value(top);
    for (int k = k0 + threadIdx.x; k < k1; k += kThreads) {   // read back by the same thread
        double s = S[k];
        if (!is_nan64(s)) s -= mx;
        S[k] = s;
        if (rank > 0) S0[k] = s;
    }
    __syncthreads();
    int nh = 0;
    bool unsure = !fast_hull;
    if (beta_c_in <= 0.0 && !unsure) {   // the stretch's own hull: whatever is below it is below the whole one
        nh = visited_bins(S, k0, k1, hull, counts);
        bool u;
        nh = thin_rounds(S, hull, nh, counts, &u);
        if (threadIdx.x == 0) s_nh = nh;
    }
    cluster.sync();
    const bool want_f = r == 0 && f_out;
    if (rank == 0 && beta_c_in <= 0.0 && !unsure) {   // the stretches' hulls one after the other
        for (int c = 1; c < kMaxwellCtas; ++c) {
            const int n = *cluster.map_shared_rank(&s_nh, c);
            const int* other = cluster.map_shared_rank(hull, c);
            for (int q = threadIdx.x; q < n; q += kThreads) hull[nh + q] = other[q];
            nh += n;
        }
    }
    cluster.sync();   // the first CTA has all that it reads of the others
    if (rank > 0 && !want_f) return;
    auto f_share = [&](double bc) {   // this CTA's share of f (Eq. 7)
        const bool ok = bc > 0.0, safe = ok && quot_safe(bc);
        const double rb = 1.0 / bc, rN = 1.0 / N;
        for (int k = rank * kThreads + threadIdx.x; k < K; k += kMaxwellCtas * kThreads) {
            const double s = S0[k];
            f_out[k] = (is_finite64(s) && ok) ? quot(bin_centre(e_min, w, k) - quot(s, bc, rb, safe), N, rN, true) : nan;
        }
    };
    if (rank > 0) {
        cluster.sync();   // beta_c is known
        f_share(*cluster.map_shared_rank(&s_bc, 0));
        cluster.sync();   // the first CTA's shared memory is read
        return;
    }
    if (threadIdx.x == 0) s_best_q = INT_MAX;
    __syncthreads();
    if (beta_c_in <= 0.0 && !unsure) nh = thin_rounds(S, hull, nh, counts, &unsure);
    if (beta_c_in <= 0.0 && unsure) {   // some triple is nearly collinear: the chain itself
        // the chain test of (k-2, k-1, k): 1 drop, 0 keep, 2 not all three visited
        for (int k = threadIdx.x; k < K; k += blockDim.x) {
            uint8_t v = 2;
            if (k >= 2 && isfinite(S[k]) && isfinite(S[k - 1]) && isfinite(S[k - 2]))
                v = chain_drops(S, e_min, w, k - 2, k - 1, k) ? 1 : 0;
            pre[k] = v;
        }
        __syncthreads();
        if (threadIdx.x == 0) {   // upper hull, left to right over the visited bins
            int n = 0;
            for (int k = 0; k < K; ++k) {
                if (!isfinite(S[k])) continue;
                while (n >= 2) {
                    const int i = hull[n - 2], j = hull[n - 1];
                    const bool drop = (i == k - 2 && j == k - 1) ? pre[k] == 1 : chain_drops(S, e_min, w, i, j, k);
                    if (!drop) break;
                    --n;
                }
                hull[n++] = k;
            }
            s_nh = n;
        }
        __syncthreads();
        nh = s_nh;
    }
    // qualifying edges: slope, latent heat and visited bins inside, an edge a thread; the rise
    // max_j (beta_j - min_{k<j} beta_k) over the edge's bins with a defined beta, where it is
    // asked for (it is never negative), a warp an edge
    double my_L = -1.0;
    int my_q = INT_MAX;
    if (beta_c_in <= 0.0) {
        for (int q = threadIdx.x; q + 1 < nh; q += blockDim.x) {
            const int a = hull[q], b = hull[q + 1];
            bool in = false;
            for (int k = a + 1; k < b && !in; ++k) in = is_finite64(S[k]);
            bool ok = false;
            if (in) {
                const double eab = __dsub_rn(bin_centre(e_min, w, b), bin_centre(e_min, w, a));
                if (__ddiv_rn(__dsub_rn(S[b], S[a]), eab) > 0.0) {   // beta_c = 1/T_c > 0
                    const double L = __ddiv_rn(eab, N);
                    ok = L >= tol_L;
                    if (ok && tol_beta <= 0.0 && L > my_L) {   // q rises along this thread's edges
                        my_L = L;
                        my_q = q;
                    }
                }
            }
            pre[q] = ok;
        }
        __syncthreads();
    }
    if (beta_c_in <= 0.0 && !(tol_beta <= 0.0)) {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
        const double den = 2.0 * h * w;
        for (int q = warp; q + 1 < nh; q += n_warps) {
            if (!pre[q]) continue;
            const int a = hull[q], b = hull[q + 1];
            const double L = __ddiv_rn(__dsub_rn(bin_centre(e_min, w, b), bin_centre(e_min, w, a)), N);
            double rise = 0.0, run_min = INFINITY;
            for (int base = a; base <= b; base += 32) {
                const int k = base + lane;
                const bool ok = k <= b && k - h >= 0 && k + h < K && isfinite(S[k - h]) && isfinite(S[k + h]);
                const double bk = ok ? (S[k + h] - S[k - h]) / den : INFINITY;
                double incl = bk;   // inclusive prefix minimum over the lanes
                for (int o = 1; o < 32; o <<= 1) {
                    const double v = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl = fmin(incl, v);
                }
                double excl = __shfl_up_sync(0xffffffffu, incl, 1);
                excl = lane == 0 ? run_min : fmin(run_min, excl);
                if (ok && bk - excl > rise) rise = bk - excl;
                run_min = fmin(run_min, __shfl_sync(0xffffffffu, incl, 31));
            }
            for (int o = 16; o > 0; o >>= 1) rise = fmax(rise, __shfl_xor_sync(0xffffffffu, rise, o));
            if (rise >= tol_beta && L > my_L) {   // q rises along this warp's edges
                my_L = L;
                my_q = q;
            }
        }
    }
    const double best_L = block_max(my_L, red);
    if (best_L >= 0.0 && my_L == best_L) atomicMin(&s_best_q, my_q);
    __syncthreads();
    const int best_q = s_best_q;
    double bc = beta_c_in;
    int best_a = -1, best_b = -1;
    if (best_q != INT_MAX) {
        best_a = hull[best_q];
        best_b = hull[best_q + 1];
        bc = __ddiv_rn(__dsub_rn(S[best_b], S[best_a]),
                       __dsub_rn(bin_centre(e_min, w, best_b), bin_centre(e_min, w, best_a)));
    }
    double gap = 0.0;   // the barrier: the largest drop of S below the common tangent
    if (best_a >= 0) {
        const double ea = bin_centre(e_min, w, best_a);
        for (int k = best_a + 1 + threadIdx.x; k < best_b; k += blockDim.x) {
            if (!isfinite(S[k])) continue;
            const double line = __dadd_rn(S[best_a], __dmul_rn(bc, __dsub_rn(bin_centre(e_min, w, k), ea)));
            if (line - S[k] > gap) gap = line - S[k];
        }
    }
    gap = block_max(gap, red);
    if (threadIdx.x == 0) {
        double out[6] = {nan, nan, nan, nan, nan, 0.0};
        if (best_a >= 0) {
            const double ea = bin_centre(e_min, w, best_a), eb = bin_centre(e_min, w, best_b);
            out[0] = bc;
            out[1] = ea / N;
            out[2] = eb / N;
            out[3] = (eb - ea) / N;
            out[4] = gap / __dmul_rn(bc, N);
            out[5] = 1.0;
        } else if (beta_c_in > 0.0) {
            out[0] = beta_c_in;
        }
        for (int q = 0; q < 6; ++q) rep[(size_t)r * 6 + q] = out[q];
    }
    if (want_f) {
        if (threadIdx.x == 0) s_bc = bc;
        cluster.sync();   // releases the cluster's other CTAs
        f_share(bc);
        cluster.sync();
    }
}

// Jackknife errors of replicate 0's results over the leave-one-block-out rows;
// NaN when a replicate found no transition; err[5] counts the rows that did.
__global__ void maxwell_err_kernel(int R, const double* __restrict__ rep, double* __restrict__ err) {
    const int q = threadIdx.x;
    if (q >= 6) return;
    const double nan = __longlong_as_double(0x7ff8000000000000ll);
    int found = 0;
    double mean = 0.0;
    for (int r = 1; r <= R; ++r) {
        found += rep[(size_t)r * 6 + 5] != 0.0;
        mean += rep[(size_t)r * 6 + q];
    }
    if (q == 5) { err[5] = (double)found; return; }
    if (R < 2 || found < R) { err[q] = nan; return; }
    mean /= R;
    double ss = 0.0;
    for (int r = 1; r <= R; ++r) {
        const double d = rep[(size_t)r * 6 + q] - mean;
        ss += d * d;
    }
    err[q] = sqrt((double)(R - 1) / R * ss);
}

}  // namespace

extern "C" size_t phast_micro_workspace_size(int32_t K, int32_t n_T, int32_t n_blocks) {
    if (K < 1 || n_T < 0 || n_blocks < 0) return 0;
    int R = 1 + (n_blocks >= 2 ? n_blocks : 0);
    return sizeof(double) * work_doubles(K, n_T, R);
}

extern "C" int phast_micro_analysis(int32_t K, double e_min, double bin_width, const double* lnW, const uint64_t* hist,
                                    int32_t n_blocks, int32_t h, int32_t n_monomers, int32_t n_T, const double* T,
                                    const phast_micro_out* out, void* workspace, size_t workspace_bytes,
                                    void* stream) {
    if (K < 1 || K > PHAST_MAX_BINS) return phast_set_error(PHAST_EINVAL, "phast_micro_analysis: K %d outside [1, %d]", K, PHAST_MAX_BINS);
    if (!(bin_width > 0.0) || !isfinite(e_min)) return phast_set_error(PHAST_EINVAL, "phast_micro_analysis: bad bins");
    if (h < 1 || 2 * h >= K) return phast_set_error(PHAST_EINVAL, "phast_micro_analysis: fd_half_width %d outside [1, K/2)", h);
    if (n_monomers < 1) return phast_set_error(PHAST_EINVAL, "phast_micro_analysis: n_monomers < 1");
    if (n_T < 0 || (n_T > 0 && !T)) return phast_set_error(PHAST_EINVAL, "phast_micro_analysis: bad temperature grid");
    if (!lnW || !out) return phast_set_error(PHAST_EINVAL, "phast_micro_analysis: NULL argument");
    if (hist && n_blocks < 1) return phast_set_error(PHAST_EINVAL, "phast_micro_analysis: n_blocks < 1");
    if (!hist) n_blocks = 0;
    const int R = 1 + (n_blocks >= 2 ? n_blocks : 0);
    const size_t need = sizeof(double) * work_doubles(K, n_T, R);
    if (!workspace || workspace_bytes < need)
        return phast_set_error(PHAST_EINVAL, "phast_micro_analysis: workspace of %zu bytes < %zu", workspace_bytes, need);
    cudaStream_t st = (cudaStream_t)stream;
    Work wk = carve((double*)workspace, K, n_T, R);
    return launch_micro(K, e_min, bin_width, lnW, hist, n_blocks, h, n_monomers, n_T, T, *out, wk, R,
                        n_blocks >= 2 ? n_blocks : 0, 0, 0, st);
}

extern "C" size_t phast_micro_binned_workspace_size(int32_t K, int32_t n_T, int32_t n_it) {
    if (K < 1 || n_T < 0 || n_it < 1) return 0;
    return sizeof(double) * work_doubles(K, n_T, n_it);
}

extern "C" int phast_micro_analysis_binned(int32_t K, double e_min, double bin_width, const double* lnW,
                                           const uint64_t* hist, int32_t n_it, int32_t block, int32_t h,
                                           int32_t n_monomers, int32_t n_T, const double* T,
                                           const phast_micro_out* out, void* workspace, size_t workspace_bytes,
                                           void* stream) {
    const char* f = "phast_micro_analysis_binned";
    if (K < 1 || K > PHAST_MAX_BINS) return phast_set_error(PHAST_EINVAL, "%s: K %d outside [1, %d]", f, K, PHAST_MAX_BINS);
    if (!(bin_width > 0.0) || !isfinite(e_min)) return phast_set_error(PHAST_EINVAL, "%s: bad bins", f);
    if (h < 1 || 2 * h >= K) return phast_set_error(PHAST_EINVAL, "%s: fd_half_width %d outside [1, K/2)", f, h);
    if (n_monomers < 1) return phast_set_error(PHAST_EINVAL, "%s: n_monomers < 1", f);
    if (n_T < 0 || (n_T > 0 && !T)) return phast_set_error(PHAST_EINVAL, "%s: bad temperature grid", f);
    if (!lnW || !out) return phast_set_error(PHAST_EINVAL, "%s: NULL argument", f);
    if (n_it < 1 || block < 1 || n_it / block < 1)
        return phast_set_error(PHAST_EINVAL, "%s: %d iterations do not fill one block of %d", f, n_it, block);
    const size_t need = sizeof(double) * work_doubles(K, n_T, n_it);
    if (!workspace || workspace_bytes < need)
        return phast_set_error(PHAST_EINVAL, "%s: workspace of %zu bytes < %zu", f, workspace_bytes, need);
    cudaStream_t st = (cudaStream_t)stream;
    Work wk = carve((double*)workspace, K, n_T, n_it);
    return launch_micro(K, e_min, bin_width, lnW, hist, 0, h, n_monomers, n_T, T, *out, wk, n_it, 0, 1, block, st);
}

// ---------------------------------------------------------------------------
// Allocation-free variant.  Some callers cannot allocate device memory at the
// point where they need the analysis: a plug-in that runs inside another
// program's CUDA context under a fixed memory budget, or code running between
// the steps of a loop that must not change the device's allocations.  For them
// the workspace lives in a file-scope device array that the library reserves
// when its module is loaded on a device (and keeps until the process exits).
// ---------------------------------------------------------------------------
#include <cuda.h>   // CUcontext and CUresult types only; the driver calls are resolved at run time
#include <mutex>

static __device__ __align__(256) double g_micro_scratch[PHAST_MICRO_NOALLOC_DOUBLES];

namespace {
// The array's name is a host-side stand-in: its device address has to be looked
// up, and it differs between CUDA contexts (a module is loaded once per
// context).  The address is cached per context, keyed by the driver's unique
// context ID, so a context created later (after cudaDeviceReset, or a
// non-primary context a host program makes current) gets its own lookup.
typedef CUresult (*ctx_get_current_fn)(CUcontext*);
typedef CUresult (*ctx_get_id_fn)(CUcontext, unsigned long long*);
struct ScratchEntry {
    unsigned long long ctx_id;
    double* addr;
};
constexpr int kScratchCache = 64;
std::mutex g_scratch_mu;
ScratchEntry g_scratch_cache[kScratchCache];
int g_scratch_used = 0, g_scratch_next = 0;
ctx_get_current_fn g_ctx_get_current = nullptr;
ctx_get_id_fn g_ctx_get_id = nullptr;

// ID of the calling thread's current context; 0 when there is none yet.
int current_ctx_id(unsigned long long* id) {
    *id = 0;
    if (!g_ctx_get_current || !g_ctx_get_id) {
        cudaDriverEntryPointQueryResult q1 = cudaDriverEntryPointSymbolNotFound, q2 = q1;
        void *f1 = nullptr, *f2 = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f1, 12000, cudaEnableDefault, &q1) != cudaSuccess ||
            cudaGetDriverEntryPointByVersion("cuCtxGetId", &f2, 12000, cudaEnableDefault, &q2) != cudaSuccess ||
            q1 != cudaDriverEntryPointSuccess || q2 != cudaDriverEntryPointSuccess || !f1 || !f2)
            return phast_set_error(PHAST_ECUDA, "phast_micro_analysis_noalloc: driver context queries unavailable");
        g_ctx_get_current = (ctx_get_current_fn)f1;
        g_ctx_get_id = (ctx_get_id_fn)f2;
    }
    CUcontext ctx = nullptr;
    if (g_ctx_get_current(&ctx) != CUDA_SUCCESS)
        return phast_set_error(PHAST_ECUDA, "phast_micro_analysis_noalloc: cuCtxGetCurrent failed");
    if (ctx && g_ctx_get_id(ctx, id) != CUDA_SUCCESS)
        return phast_set_error(PHAST_ECUDA, "phast_micro_analysis_noalloc: cuCtxGetId failed");
    return PHAST_OK;
}
}  // namespace

extern "C" int phast_micro_analysis_noalloc(int32_t K, double e_min, double bin_width, const double* lnW,
                                            const uint64_t* hist, int32_t n_blocks, int32_t h, int32_t n_monomers,
                                            int32_t n_T, const double* T, const phast_micro_out* out, void* stream) {
    if (K < 1 || K > PHAST_MAX_BINS || n_T < 0 || (hist && n_blocks < 1))
        return phast_micro_analysis(K, e_min, bin_width, lnW, hist, n_blocks, h, n_monomers, n_T, T, out,
                                    nullptr, 0, stream);   // reports the argument error
    const int R = 1 + ((hist && n_blocks >= 2) ? n_blocks : 0);
    const size_t need = work_doubles(K, n_T, R);
    if (need > (size_t)PHAST_MICRO_NOALLOC_DOUBLES)
        return phast_set_error(PHAST_EINVAL,
                               "phast_micro_analysis_noalloc: K=%d, n_T=%d, %d blocks need %zu doubles of scratch, "
                               "more than the %d of the static workspace (use phast_micro_analysis)",
                               K, n_T, n_blocks, need, PHAST_MICRO_NOALLOC_DOUBLES);
    double* scratch = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_scratch_mu);
        unsigned long long id = 0;
        int rc = current_ctx_id(&id);
        if (rc != PHAST_OK) return rc;
        for (int i = 0; i < g_scratch_used && id; ++i)
            if (g_scratch_cache[i].ctx_id == id) scratch = g_scratch_cache[i].addr;
        if (!scratch) {
            // first call in this context: look the address up (this also makes the
            // runtime's context current when none was)
            void* p = nullptr;
            cudaError_t e = cudaGetSymbolAddress(&p, g_micro_scratch);
            if (e != cudaSuccess)
                return phast_set_error(PHAST_ECUDA, "phast_micro_analysis_noalloc: cudaGetSymbolAddress: %s",
                                       cudaGetErrorString(e));
            scratch = (double*)p;
            if (!id && (rc = current_ctx_id(&id)) != PHAST_OK) return rc;
            if (id) {
                const int slot = g_scratch_used < kScratchCache ? g_scratch_used++ : (g_scratch_next++ % kScratchCache);
                g_scratch_cache[slot] = ScratchEntry{id, scratch};
            }
        }
    }
    return phast_micro_analysis(K, e_min, bin_width, lnW, hist, n_blocks, h, n_monomers, n_T, T, out, scratch,
                                sizeof(double) * (size_t)PHAST_MICRO_NOALLOC_DOUBLES, stream);
}

extern "C" int phast_maxwell(int32_t K, double e_min, double bin_width, const double* lnW, const uint64_t* hist,
                             int32_t n_blocks, int32_t fd_half_width, int32_t n_monomers, double beta_c,
                             double tol_beta, double tol_L, double* f_out, double* rep, double* err, void* stream) {
    if (K < 1 || K > PHAST_MAX_BINS) return phast_set_error(PHAST_EINVAL, "phast_maxwell: K %d outside [1, %d]", K, PHAST_MAX_BINS);
    if (!(bin_width > 0.0)) return phast_set_error(PHAST_EINVAL, "phast_maxwell: bin_width must be > 0");
    if (!lnW || !rep) return phast_set_error(PHAST_EINVAL, "phast_maxwell: NULL lnW or rep");
    if (hist && n_blocks < 1) return phast_set_error(PHAST_EINVAL, "phast_maxwell: n_blocks < 1");
    if (fd_half_width < 1) return phast_set_error(PHAST_EINVAL, "phast_maxwell: fd_half_width < 1");
    if (n_monomers < 1) return phast_set_error(PHAST_EINVAL, "phast_maxwell: n_monomers < 1");
    if (!(beta_c >= 0.0) || !(tol_beta >= 0.0) || !(tol_L >= 0.0))
        return phast_set_error(PHAST_EINVAL, "phast_maxwell: beta_c, tol_beta, tol_L must be >= 0");
    const int R = (hist && n_blocks >= 2) ? n_blocks : 0;
    const size_t sm = kMaxwellSmemPerBin * (size_t)K;
    cudaStream_t st = (cudaStream_t)stream;
    PHAST_CUDA_TRY(cudaFuncSetAttribute(maxwell_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)(kMaxwellSmemPerBin * PHAST_MAX_BINS)));
    // the chain test's rounding relative to the slopes is a few ulp of the largest |E_k| over w:
    // far below the 1e-9 of thin_hull for any sensible bins
    const double e_abs = fmax(fabs(e_min), fabs(e_min + K * bin_width));
    const int fast_hull = 16.0 * e_abs * 2.220446049250313e-16 <= 1e-10 * bin_width;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(1 + R) * kMaxwellCtas);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = sm;
    cfg.stream = st;
    cudaLaunchAttribute cluster;
    cluster.id = cudaLaunchAttributeClusterDimension;
    cluster.val.clusterDim.x = kMaxwellCtas;
    cluster.val.clusterDim.y = cluster.val.clusterDim.z = 1;
    cfg.attrs = &cluster;
    cfg.numAttrs = 1;
    PHAST_CUDA_TRY(cudaLaunchKernelEx(&cfg, maxwell_kernel, K, e_min, bin_width, lnW,
                                      reinterpret_cast<const unsigned long long*>(hist), hist ? n_blocks : 0,
                                      fd_half_width, n_monomers, beta_c, tol_beta, tol_L, f_out, rep, fast_hull));
    if (err) {
        maxwell_err_kernel<<<1, 32, 0, st>>>(R, rep, err);
        PHAST_CUDA_TRY(cudaGetLastError());
    }
    return PHAST_OK;
}
