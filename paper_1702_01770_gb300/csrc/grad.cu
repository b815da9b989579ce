// grad.cu -- derivatives of the energy of Eq. 2/3 (with the torsion term) for
// batches of conformations, and multicanonical reweighting of canonical
// averages and their parameter derivatives (Sec. 2.2).
//
// phast_energy_grad and the passes of a training step: one warp per conformation, in FP64 or
// with FP32 pair terms.  No atomics, a deterministic order.  Nothing is stored between the
// forward and the backward pass: the backward pass recomputes (checkpointed recomputation).
#include <cooperative_groups.h>

#include "exp64.cuh"
#include "group.cuh"

namespace cg = cooperative_groups;

namespace {

constexpr int kGradWarps = 4;

template <typename PT>
struct V3 {
    PT x, y, z;
};
template <typename PT>
__device__ __forceinline__ V3<PT> sub3(const P4<PT>& a, const P4<PT>& b) {
    return V3<PT>{a.x - b.x, a.y - b.y, a.z - b.z};
}
template <typename PT>
__device__ __forceinline__ PT dot3(const V3<PT>& a, const V3<PT>& b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
template <typename PT>
__device__ __forceinline__ V3<PT> cross3(const V3<PT>& a, const V3<PT>& b) {
    return V3<PT>{a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x};
}
template <typename PT>
__device__ __forceinline__ V3<PT> axpy3(PT s, const V3<PT>& a, const V3<PT>& b) {   // s a + b
    return V3<PT>{s * a.x + b.x, s * a.y + b.y, s * a.z + b.z};
}

// The force-field parameters the derivatives are taken in, (C_AA, C_BB, C_AB,
// kappa, kappa_C): from the system's force field, or from a device array of five
// doubles in that order (so a caller holding them on the device needs no copy to
// the host).  c(2 s_i + s_j) is C_LJ of Eq. 1 for letters s_i, s_j.
template <typename PT>
struct Coef {
    PT c0, c1, c2, c3, kt, kb;
    __device__ __forceinline__ PT c(int idx) const { return idx == 0 ? c0 : (idx == 1 ? c1 : (idx == 2 ? c2 : c3)); }
};
template <typename PT>
__device__ __forceinline__ Coef<PT> coef(const SysDesc& d, const double* __restrict__ p) {
    if (p) return Coef<PT>{(PT)p[0], (PT)p[2], (PT)p[2], (PT)p[1], (PT)p[3], (PT)p[4]};
    return Coef<PT>{(PT)d.C[0], (PT)d.C[1], (PT)d.C[2], (PT)d.C[3], (PT)d.k_tors, (PT)d.k_bend};
}

// d cos tau_j / dx_{j+which}: n1 = u x v, n2 = v x w from u, v, w the bonds of monomers j..j+3;
// zero for a degenerate dihedral (|n1|^2 |n2|^2 < 1e-20), where the term is 0.
template <typename PT, class Pos>
__device__ V3<PT> torsion_grad(const Pos& pos, int o, int j, int which) {
    const P4<PT> x0 = pos(o + j), x1 = pos(o + j + 1), x2 = pos(o + j + 2), x3 = pos(o + j + 3);
    const V3<PT> u = sub3(x1, x0), v = sub3(x2, x1), w = sub3(x3, x2);
    const V3<PT> n1 = cross3(u, v), n2 = cross3(v, w);
    const PT n11 = dot3(n1, n1), n22 = dot3(n2, n2);
    if (n11 * n22 < (PT)1e-20) return V3<PT>{0, 0, 0};
    const PT l12 = sqrt(n11) * sqrt(n22);
    const PT cs = dot3(n1, n2) / l12;
    const V3<PT> g1 = axpy3(-cs / n11, n1, V3<PT>{n2.x / l12, n2.y / l12, n2.z / l12});
    const V3<PT> g2 = axpy3(-cs / n22, n2, V3<PT>{n1.x / l12, n1.y / l12, n1.z / l12});
    const V3<PT> du = cross3(v, g1);
    const V3<PT> dv = axpy3((PT)1, cross3(g1, u), cross3(w, g2));
    const V3<PT> dw = cross3(g2, v);
    // u = x1 - x0, v = x2 - x1, w = x3 - x2
    if (which == 0) return V3<PT>{-du.x, -du.y, -du.z};
    if (which == 1) return V3<PT>{du.x - dv.x, du.y - dv.y, du.z - dv.z};
    if (which == 2) return V3<PT>{dv.x - dw.x, dv.y - dw.y, dv.z - dw.z};
    return dw;
}

// ---------------------------------------------------------------------------
// FP64 form: one warp per conformation.  An FP64 instruction holds an SMSP's pipe for 64 to 76
// cycles, so their number is what counts: every pair once (a lane's row i against the
// partner s places on, cyclically; the force goes to the row's registers and, with the
// opposite sign, to the partner's sum in shared memory -- the lanes of a step have different
// partners), every bending and torsion term once (added to its monomers in turn), reciprocals
// by one corrected approximation.  23 FP64 instructions a pair.  4096 conformations of a
// 55-mer: 448 us (1200 us with both ends of a pair and the local terms of every monomer).
// ---------------------------------------------------------------------------
struct Grad64Slot {
    double *x, *y, *z;      // [N] positions
    double *gx, *gy, *gz;   // [N] gradient
};
__host__ __device__ inline size_t grad64_slot_bytes(int N) { return sizeof(double) * 6 * (size_t)N; }

__device__ __forceinline__ V3<double> at64(const Grad64Slot& s, int j) { return V3<double>{s.x[j], s.y[j], s.z[j]}; }
__device__ __forceinline__ V3<double> diff64(const V3<double>& a, const V3<double>& b) { return V3<double>{a.x - b.x, a.y - b.y, a.z - b.z}; }
__device__ __forceinline__ void add64(const Grad64Slot& s, int j, double k, const V3<double>& g) {
    s.gx[j] += k * g.x;
    s.gy[j] += k * g.y;
    s.gz[j] += k * g.z;
}

__global__ void __launch_bounds__(32 * kGradWarps)
energy_grad64_kernel(const SysDesc d, int B, const double* __restrict__ xyz, double* __restrict__ E_out,
                     double* __restrict__ grad_xyz, double* __restrict__ grad_ff, const double* __restrict__ pdev) {
    extern __shared__ __align__(16) unsigned char smem[];
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int b = blockIdx.x * kGradWarps + w;
    if (b >= B) return;
    const int N = d.N, nc = d.n_chains;
    double* base = reinterpret_cast<double*>(smem) + (size_t)w * 6 * N;
    const Grad64Slot s{base, base + N, base + 2 * N, base + 3 * N, base + 4 * N, base + 5 * N};
    const double* x64 = xyz + (size_t)b * N * 3;
    bool out = false;   // a monomer beyond the container's wall: infinite energy
    for (int j = lane; j < N; j += 32) {
        const double3 p = ld3(x64 + 3 * j);
        s.x[j] = p.x; s.y[j] = p.y; s.z[j] = p.z;
        s.gx[j] = s.gy[j] = s.gz[j] = 0.0;
        if (d.has_sphere) out |= !inside64(d, p);
    }
    __syncwarp();
    const Coef<double> cf = coef<double>(d, pdev);
    // E, sum 1 - cos theta, -sum cos tau, and minus the sums of k s^3 over AA, BB and AB pairs
    double v[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    for (int c = 0; c < nc; ++c) {
        const int o = d.chain_off[c], n = d.chain_off[c + 1] - o;
        for (int k0 = 1; k0 <= n - 2; k0 += 32) {
            const int k = o + k0 + lane;
            const bool on = k0 + lane <= n - 2;
            V3<double> ga{0, 0, 0}, gb{0, 0, 0};   // d cos / d a, d cos / d b for bonds a, b
            if (on) {
                const V3<double> x1 = at64(s, k), u = diff64(x1, at64(s, k - 1)), t = diff64(at64(s, k + 1), x1);
                const double aa = dot3(u, u), bb = dot3(t, t);
                const double il = rsqrt64(aa * bb), cs = dot3(u, t) * il;
                const double ia = cs * rcp64(aa), ib = cs * rcp64(bb);
                ga = V3<double>{t.x * il - ia * u.x, t.y * il - ia * u.y, t.z * il - ia * u.z};
                gb = V3<double>{u.x * il - ib * t.x, u.y * il - ib * t.y, u.z * il - ib * t.z};
                v[1] += 1.0 - cs;
            }
            if (grad_xyz) {   // 1 - cos: +ga, gb - ga, -gb
                if (on) add64(s, k - 1, cf.kb, ga);
                __syncwarp();
                if (on) add64(s, k, cf.kb, diff64(gb, ga));
                __syncwarp();
                if (on) add64(s, k + 1, -cf.kb, gb);
                __syncwarp();
            }
        }
        for (int j0 = 0; j0 <= n - 4; j0 += 32) {
            const int j = o + j0 + lane;
            const bool on = j0 + lane <= n - 4;
            V3<double> du{0, 0, 0}, dv{0, 0, 0}, dw{0, 0, 0};   // d cos tau by the three bonds
            if (on) {
                const V3<double> x0 = at64(s, j), x1 = at64(s, j + 1), x2 = at64(s, j + 2), x3 = at64(s, j + 3);
                const V3<double> u = diff64(x1, x0), t = diff64(x2, x1), q = diff64(x3, x2);
                const V3<double> n1 = cross3(u, t), n2 = cross3(t, q);
                const double n11 = dot3(n1, n1), n22 = dot3(n2, n2), p = n11 * n22;
                if (!(p < 1e-20)) {   // a degenerate dihedral has no term
                    const double il = rsqrt64(p), cs = dot3(n1, n2) * il;
                    const double c1 = cs * rcp64(n11), c2 = cs * rcp64(n22);
                    const V3<double> g1{n2.x * il - c1 * n1.x, n2.y * il - c1 * n1.y, n2.z * il - c1 * n1.z};
                    const V3<double> g2{n1.x * il - c2 * n2.x, n1.y * il - c2 * n2.y, n1.z * il - c2 * n2.z};
                    du = cross3(t, g1);
                    dv = axpy3(1.0, cross3(g1, u), cross3(q, g2));
                    dw = cross3(g2, t);
                    v[2] -= cs;
                }
            }
            if (grad_xyz) {   // -kappa cos tau: monomers get -du, du - dv, dv - dw, dw
                if (on) add64(s, j, cf.kt, du);
                __syncwarp();
                if (on) add64(s, j + 1, -cf.kt, diff64(du, dv));
                __syncwarp();
                if (on) add64(s, j + 2, -cf.kt, diff64(dv, dw));
                __syncwarp();
                if (on) add64(s, j + 3, -cf.kt, dw);
                __syncwarp();
            }
        }
        if (d.k_fene != 0.0)   // bond l: d/dr [k R^2 C_F ln(1 - x^2)] = -2 k R C_F x / (1 - x^2)
            for (int l0 = 0; l0 <= n - 2; l0 += 32) {
                const int l = o + l0 + lane;
                const bool on = l0 + lane <= n - 2;
                V3<double> u{0, 0, 0};
                double dphi = 0.0;
                if (on) {
                    v[0] += fene_term(d, [&](int j) { return make_double3(s.x[j], s.y[j], s.z[j]); }, l, 0);
                    const V3<double> q = diff64(at64(s, l + 1), at64(s, l));
                    const double r = sqrt(dot3(q, q)), x = (r - d.fene_r0) / d.fene_R;
                    dphi = -2.0 * d.k_fene * d.fene_R * d.C_F[2 * d.seq[l] + d.seq[l + 1]] * x / (1.0 - x * x);
                    u = V3<double>{q.x / r, q.y / r, q.z / r};
                }
                if (grad_xyz) {
                    if (on) add64(s, l, -dphi, u);
                    __syncwarp();
                    if (on) add64(s, l + 1, dphi, u);
                    __syncwarp();
                }
            }
    }
    v[0] += cf.kb * v[1] + cf.kt * v[2];
    for (int i0 = 0; i0 < N; i0 += 32) {
        const int i = i0 + lane;
        const bool row = i < N;
        const V3<double> a = at64(s, row ? i : 0);
        const int ci = row ? d.chain_of[i] : 0, si = row ? d.seq[i] : 0;
        V3<double> g{0, 0, 0};
        for (int m = 1; 2 * m <= N; ++m) {
            int j = i + m;
            if (j >= N) j -= N;
            // every pair once (opposite places from the first half); bonded pairs have no term
            const bool on = row && !(2 * m == N && 2 * i >= N) && !(m == 1 && j == i + 1 && d.chain_of[j] == ci);
            if (on) {
                const bool inter = d.chain_of[j] != ci;
                const int sj = d.seq[j];
                V3<double> q = diff64(a, at64(s, j));
                if (inter) {
                    q.x = mimage64_short(d, q.x);
                    q.y = mimage64_short(d, q.y);
                    q.z = mimage64_short(d, q.z);
                }
                const double k = inter ? d.k_lj_inter : d.k_lj_intra;
                const double C = cf.c(j > i ? 2 * si + sj : 2 * sj + si);   // the earlier monomer's letter first
                const double sv = rcp64(dot3(q, q)), s2 = sv * sv, s3 = s2 * sv, ks3 = k * s3;
                v[0] = __fma_rn(ks3, s3 - C, v[0]);   // k (s^6 - C s^3)
                const int cls = si == sj ? 3 + si : 5;
                const double sum = (cls == 3 ? v[3] : cls == 4 ? v[4] : v[5]) - ks3;
                v[3] = cls == 3 ? sum : v[3];
                v[4] = cls == 4 ? sum : v[4];
                v[5] = cls == 5 ? sum : v[5];
                if (grad_xyz) {
                    const double fr = ks3 * sv * __fma_rn(-12.0, s3, 6.0 * C);   // 2 dphi/d(r^2)
                    g.x = __fma_rn(fr, q.x, g.x);
                    g.y = __fma_rn(fr, q.y, g.y);
                    g.z = __fma_rn(fr, q.z, g.z);
                    s.gx[j] = __fma_rn(-fr, q.x, s.gx[j]);
                    s.gy[j] = __fma_rn(-fr, q.y, s.gy[j]);
                    s.gz[j] = __fma_rn(-fr, q.z, s.gz[j]);
                }
            }
            __syncwarp();
        }
        if (row && grad_xyz) {
            s.gx[i] += g.x;
            s.gy[i] += g.y;
            s.gz[i] += g.z;
        }
        __syncwarp();
    }
    if (grad_xyz)
        for (int e = lane; e < 3 * N; e += 32) {
            const int j = e / 3, q = e - 3 * j;
            grad_xyz[(size_t)b * N * 3 + e] = (q == 0 ? s.gx : q == 1 ? s.gy : s.gz)[j];
        }
    out = __any_sync(full, out);
    int first = 0, count = 6;
    warp_sums<6>(v, &first, &count);
    if (count == 1) {
        if (first == 0 && E_out) E_out[b] = out ? INFINITY : v[0];
        // v[1..5]: kappa_C, kappa, AA, BB, AB -> columns 4, 3, 0, 1, 2
        if (first > 0 && grad_ff) grad_ff[(size_t)b * 5 + (first == 1 ? 4 : first == 2 ? 3 : first - 3)] = v[0];
    }
}

// ---------------------------------------------------------------------------
// FP32 forms: one warp per conformation, two evaluations per paired FP32 instruction
// (f32x2).  The working copy holds FP32 coordinates relative to an origin that is an FP32
// value (a chain's centroid, or one of its monomers), so the subtraction x - o is exact before
// the one rounding, and the minimum-imaged FP32 differences of the origins.  FP64
// instructions hold the pipe of an SMSP for 64 cycles, so sums run in double-float (two FP32
// numbers, TwoSum), conversions by integer instructions, and FP32 coordinates (IN = float: a
// training loop's leaves) are taken as they are.
//   GRAD = false: energies only, each pair once (rows against the partners s places on, s up
//     to half the system).
//   GRAD = true: gradients, each pair from both of its ends (each by its own row): every
//     gradient is a plain sum in a fixed order and needs no atomics; the parameter sums take
//     half of the row sums.  15 paired instructions for a row against two partners: the
//     coupling is applied once per row (and chain), left-out partners by a far distance.
//   VJP = true: the backward pass of a loss with dloss/dE = gE: gradients come out as
//     gE dE/dx in the type of the coordinates, the parameter derivatives summed over the batch
//     (per CTA, then by sum_parts_kernel).
// Bending, torsion and FENE terms are evaluated once each; the terms of a round are added to
// their first, second, ... monomers in turn, so that the lanes of a step touch disjoint ones.
// ---------------------------------------------------------------------------
// Left-out pairs get the squared distance kFar2, rows and partners that do not exist the place
// kFar: 1 / r^6 and the force then underflow to zero exactly, so they add nothing to whatever
// the real pairs give (pairs at r = 1000 contribute 1e-18 each).
constexpr float kFar2 = 1.0e16f, kFar = 1.0e8f;
constexpr int kGrad32Warps = 8;   // warps of a CTA, fewer where their slots exceed the shared memory

struct Grad32Args {
    int B, slot_f4;
    const void* xyz;          // [B][N][3] of IN
    double* E_out;            // [B] or null
    void* grad_xyz;           // [B][N][3] double (VJP: of IN) or null
    double* grad_ff;          // [B][5] or null
    const void* pdev;         // the five parameters or null
    int p32;                  // they are FP32
    const double* gE;         // [B] (VJP)
    double* part;             // [gridDim.x][5] (VJP) or null
};

__device__ __forceinline__ Coef<float> coef32(const SysDesc& d, const Grad32Args& a) {
    const float* p = (const float*)a.pdev;
    if (a.p32 && p) return Coef<float>{p[0], p[2], p[2], p[1], p[3], p[4]};
    return coef<float>(d, (const double*)a.pdev);
}

__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }
__device__ __forceinline__ bool is_inf32(float a) { return (__float_as_int(a) & 0x7fffffff) == 0x7f800000; }

// x - o rounded to FP32, and the FP64 value of a coordinate.
__device__ __forceinline__ float rel32(double x, float o) { return f64_to_f32(x - f32_to_f64(o)); }
__device__ __forceinline__ float rel32(float x, float o) { return __fsub_rn(x, o); }
__device__ __forceinline__ double as64(double x) { return x; }
__device__ __forceinline__ double as64(float x) { return (double)x; }
__device__ __forceinline__ float as32(double x) { return f64_to_f32(x); }
__device__ __forceinline__ float as32(float x) { return x; }

// One component of a gradient: FP64, or scaled by gE in the coordinates' type.
template <bool VJP>
__device__ __forceinline__ void put_grad(double* out, float g, double gE, float, float) {
    *out = VJP ? __dmul_rn(gE, f32_to_f64(g)) : f32_to_f64(g);
}
// FP32: g gE with gE in two FP32 parts, rounded once; the FP64 product where the parts or the
// product leave the range in which they are exact (2^-90 to 2^126: gE of 0, tiny or huge, gradients
// that overflow).
constexpr unsigned kExactLow = 0x12800000u, kExactSpan = 0x7e800000u - kExactLow;
__device__ __forceinline__ bool exact_range(float a) { return ((unsigned)__float_as_int(a) & 0x7fffffffu) - kExactLow < kExactSpan; }
static __device__ __noinline__ float scaled_grad64(float g, double gE) { return (float)((double)g * gE); }
// gE's parts, 0 outside the range (every product then is too).
__device__ __forceinline__ void split_gE(double gE, float* gh, float* gl) {
    const float h = f64_to_f32(gE);
    const bool in = exact_range(h);
    *gh = in ? h : 0.0f;
    *gl = in ? f64_to_f32(gE - f32_to_f64(h)) : 0.0f;
}
template <bool VJP>
__device__ __forceinline__ void put_grad(float* out, float g, double gE, float gh, float gl) {
    const float p = __fmul_rn(g, gh);
    *out = exact_range(p) ? __fadd_rn(p, __fmaf_rn(g, gl, __fmaf_rn(g, gh, -p))) : scaled_grad64(g, gE);
}
template <typename IN, bool VJP> struct GradOut { typedef double T; };
template <> struct GradOut<float, true> { typedef float T; };

// Value and gradient of one bending term 1 - cos theta_k at once (FP32, the
// divisions replaced by one reciprocal square root and products): g[0..2] are
// the derivatives with respect to x_{k-1}, x_k, x_{k+1}.
__device__ __forceinline__ float bend_vg(const float4& x0, const float4& x1, const float4& x2, float3 g[3]) {
    const float ax = x1.x - x0.x, ay = x1.y - x0.y, az = x1.z - x0.z;
    const float bx = x2.x - x1.x, by = x2.y - x1.y, bz = x2.z - x1.z;
    const float aa = ax * ax + ay * ay + az * az, bb = bx * bx + by * by + bz * bz;
    const float ab = ax * bx + ay * by + az * bz;
    const float il = rsqrtf(aa * bb);                 // 1 / (|a| |b|), for bonds up to 4e9
    const float cs = ab * il;
    const float ia = cs / aa, ib = cs / bb;
    // d cos/d a = b il - cs a / aa, d cos/d b = a il - cs b / bb
    const float3 dca = make_float3(bx * il - ia * ax, by * il - ia * ay, bz * il - ia * az);
    const float3 dcb = make_float3(ax * il - ib * bx, ay * il - ib * by, az * il - ib * bz);
    g[0] = dca;                                                         // x_{k-1}: -(-d cos/d a)
    g[1] = make_float3(dcb.x - dca.x, dcb.y - dca.y, dcb.z - dca.z);   // x_k
    g[2] = make_float3(-dcb.x, -dcb.y, -dcb.z);                        // x_{k+1}
    return 1.0f - cs;
}

// Value and gradient of cos tau_j of monomers j..j+3 at once (FP32); zero for a
// degenerate dihedral (|n1|^2 |n2|^2 < 1e-20), whose term is 0.  A dihedral FP32
// cannot resolve (torsion_unresolved32) is taken in FP64 from x64, the coordinates
// of the configuration (monomer j at x64 + 3 j).
template <typename IN>
__device__ __noinline__ float torsion_vg64(const IN* x64, int j, float3 g[4]) {
    auto p = [&](int k) -> P4<double> {
        P4<double> q;
        q.x = as64(x64[3 * k]); q.y = as64(x64[3 * k + 1]); q.z = as64(x64[3 * k + 2]); q.tag = 0; q.pad = 0;
        return q;
    };
    for (int q = 0; q < 4; ++q) {
        const V3<double> t = torsion_grad<double>(p, 0, j, q);
        g[q] = make_float3((float)t.x, (float)t.y, (float)t.z);
    }
    return (float)torsion_term([&](int k) { const P4<double> q = p(k); return make_double3(q.x, q.y, q.z); }, 0, j);
}
template <typename IN>
__device__ __noinline__ float torsion_v64(const IN* x64, int j) {
    return (float)torsion_term([&](int k) { return make_double3(as64(x64[3 * k]), as64(x64[3 * k + 1]), as64(x64[3 * k + 2])); },
                               0, j);
}

// The bonds, normals and squared normals of a dihedral in FP32; false where FP32 cannot resolve it
// (torsion_unresolved32) or hold n11 n22 (the eighth power of a bond length: from 3e4 on).
struct Dihedral32 {
    V3<float> u, v, w, n1, n2;
    float n11, n22;
};
__device__ __forceinline__ bool dihedral32(const float4& x0, const float4& x1, const float4& x2, const float4& x3, Dihedral32* D) {
    const V3<float> u{x1.x - x0.x, x1.y - x0.y, x1.z - x0.z}, v{x2.x - x1.x, x2.y - x1.y, x2.z - x1.z},
        w{x3.x - x2.x, x3.y - x2.y, x3.z - x2.z};
    const V3<float> n1 = cross3(u, v), n2 = cross3(v, w);
    *D = Dihedral32{u, v, w, n1, n2, dot3(n1, n1), dot3(n2, n2)};
    float mx = fmaxf(fmaxf(fabsf(x0.x), fabsf(x0.y)), fabsf(x0.z));
    mx = fmaxf(mx, fmaxf(fmaxf(fabsf(x1.x), fabsf(x1.y)), fabsf(x1.z)));
    mx = fmaxf(mx, fmaxf(fmaxf(fabsf(x2.x), fabsf(x2.y)), fabsf(x2.z)));
    mx = fmaxf(mx, fmaxf(fmaxf(fabsf(x3.x), fabsf(x3.y)), fabsf(x3.z)));
    return !torsion_unresolved32(D->n11, D->n22, mx, true) && fmaxf(D->n11, D->n22) < 1e18f;
}

template <typename IN>
__device__ __forceinline__ float torsion_v(const float4& x0, const float4& x1, const float4& x2, const float4& x3, const IN* x64, int j) {
    Dihedral32 D;
    if (!dihedral32(x0, x1, x2, x3, &D)) return torsion_v64<IN>(x64, j);
    return D.n11 * D.n22 < 1e-20f ? 0.0f : dot3(D.n1, D.n2) * rsqrtf(D.n11 * D.n22);
}

template <typename IN>
__device__ __forceinline__ float torsion_vg(const float4& x0, const float4& x1, const float4& x2, const float4& x3,
                                            float3 g[4], const IN* x64, int j) {
    Dihedral32 D;
    if (!dihedral32(x0, x1, x2, x3, &D)) return torsion_vg64<IN>(x64, j, g);
    const V3<float>&u = D.u, &v = D.v, &w = D.w, &n1 = D.n1, &n2 = D.n2;
    const float n11 = D.n11, n22 = D.n22;
    if (n11 * n22 < 1e-20f) {
        g[0] = g[1] = g[2] = g[3] = make_float3(0.f, 0.f, 0.f);
        return 0.0f;
    }
    const float il = rsqrtf(n11 * n22);
    const float cs = dot3(n1, n2) * il;
    const float c1 = cs / n11, c2 = cs / n22;
    const V3<float> g1{n2.x * il - c1 * n1.x, n2.y * il - c1 * n1.y, n2.z * il - c1 * n1.z};
    const V3<float> g2{n1.x * il - c2 * n2.x, n1.y * il - c2 * n2.y, n1.z * il - c2 * n2.z};
    const V3<float> du = cross3(v, g1);
    const V3<float> dv = axpy3(1.0f, cross3(g1, u), cross3(w, g2));
    const V3<float> dw = cross3(g2, v);
    g[0] = make_float3(-du.x, -du.y, -du.z);
    g[1] = make_float3(du.x - dv.x, du.y - dv.y, du.z - dv.z);
    g[2] = make_float3(dv.x - dw.x, dv.y - dw.y, dv.z - dw.z);
    g[3] = make_float3(dw.x, dw.y, dw.z);
    return cs;
}

__device__ __forceinline__ void acc3(float4* a, int j, float s, float3 g) {
    float4 v = a[j];
    v.x = __fmaf_rn(s, g.x, v.x);
    v.y = __fmaf_rn(s, g.y, v.y);
    v.z = __fmaf_rn(s, g.z, v.z);
    a[j] = v;
}

// Bending, torsion and FENE terms of one chain (n monomers at o in r and lg): energies into
// E, the parameter sums into gp[3] (-sum cos tau) and gp[4] (sum 1 - cos theta), gradients
// into lg (GRAD).
template <bool GRAD, typename IN>
__device__ __forceinline__ void chain_terms32(const SysDesc& d, const float4* r, float4* lg, const IN* x64, int o, int n,
                                              float kb, float kt, int lane, DF& E, DF* gp) {
    auto pos = [&](int j) -> P4<float> {
        const float4 q = r[j];
        P4<float> p;
        p.x = q.x; p.y = q.y; p.z = q.z; p.tag = __float_as_int(q.w);
        return p;
    };
    for (int base = 1; base <= n - 2; base += 32) {
        const int k = o + base + lane;
        const bool on = base + lane <= n - 2;
        float3 g[3];
        if (on) {
            const float t = GRAD ? bend_vg(r[k - 1], r[k], r[k + 1], g) : bend_w<float>(pos, o, base + lane);
            gp[4] = df_add(gp[4], DF{t, 0.0f});
            E = df_add(E, DF{kb * t, 0.0f});
        }
        if constexpr (GRAD)
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                if (on) acc3(lg, k - 1 + q, kb, g[q]);
                __syncwarp();
            }
    }
    for (int base = 0; base <= n - 4; base += 32) {
        const int j = o + base + lane;
        const bool on = base + lane <= n - 4;
        float3 g[4];
        if (on) {
            float t;
            if constexpr (GRAD) t = torsion_vg<IN>(r[j], r[j + 1], r[j + 2], r[j + 3], g, x64, j);
            else t = torsion_v<IN>(r[j], r[j + 1], r[j + 2], r[j + 3], x64, j);
            gp[3] = df_add(gp[3], DF{-t, 0.0f});
            E = df_add(E, DF{-kt * t, 0.0f});
        }
        if constexpr (GRAD)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if (on) acc3(lg, j + q, -kt, g[q]);
                __syncwarp();
            }
    }
    if (d.k_fene != 0.0) {   // bond l: d/dr [k R^2 C_F ln(1 - x^2)] = -2 k R C_F x / (1 - x^2)
        for (int base = 0; base <= n - 2; base += 32) {
            const int l = o + base + lane;
            const bool on = base + lane <= n - 2;
            float3 u = make_float3(0.f, 0.f, 0.f);
            float dphi = 0.0f;
            if (on) {
                E = df_add(E, DF{fene_w<float>(d, pos, l, 0), 0.0f});
                if (GRAD) {
                    const float4 p0 = r[l], p1 = r[l + 1];
                    const float bx = p1.x - p0.x, by = p1.y - p0.y, bz = p1.z - p0.z;
                    const float rb = sqrtf(bx * bx + by * by + bz * bz);
                    const float Rf = (float)d.fene_R;
                    const float xf = (rb - (float)d.fene_r0) / Rf;
                    const float cf = (float)d.C_F[2 * d.seq[l] + d.seq[l + 1]];
                    dphi = (float)(-2.0 * d.k_fene) * Rf * cf * xf / (1.0f - xf * xf);
                    u = make_float3(bx / rb, by / rb, bz / rb);
                }
            }
            if constexpr (GRAD) {
                if (on) acc3(lg, l, -dphi, u);
                __syncwarp();
                if (on) acc3(lg, l + 1, dphi, u);
                __syncwarp();
            }
        }
    }
}

// The warp's totals and their output: E and the parameter derivatives of conformation b, or
// (VJP) this conformation's share of the batch's parameter derivatives, gE dE/dparam, added
// to acc on lanes 0..4.
template <bool VJP>
__device__ __forceinline__ void finish32(const Grad32Args& a, unsigned b, DF E, DF* gp, bool out, double gE, int lane,
                                         double& acc, bool want_ff) {
    const unsigned full = 0xffffffffu;
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) {
        if (!VJP) E = df_add(E, DF{__shfl_xor_sync(full, E.hi, m), __shfl_xor_sync(full, E.lo, m)});
        if (want_ff)
#pragma unroll
            for (int q = 0; q < 5; ++q)
                gp[q] = df_add(gp[q], DF{__shfl_xor_sync(full, gp[q].hi, m), __shfl_xor_sync(full, gp[q].lo, m)});
    }
    // every lane holds the totals: lanes 0..4 convert the parameter derivatives, lane 5 E
    DF mine = E;
#pragma unroll
    for (int q = 0; q < 5; ++q)
        if (lane == q) mine = gp[q];
    // an infinite sum leaves NaN in lo: hi alone
    const double v = f32_to_f64(mine.hi) + (is_inf32(mine.hi) ? 0.0 : f32_to_f64(mine.lo));
    if (VJP) {
        acc = __fma_rn(gE, v, acc);
    } else {
        const bool any_out = __any_sync(full, out);
        if (lane < 5 && a.grad_ff) a.grad_ff[(size_t)b * 5 + lane] = v;
        if (lane == 5 && a.E_out) a.E_out[b] = any_out ? INFINITY : v;
    }
}

// Batch sums of the warps of a CTA (lanes 0..4 of each), in warp order.
__device__ __forceinline__ void finish_part(const Grad32Args& a, double acc, int lane, int w) {
    __shared__ double s_acc[kGrad32Warps][5];
    if (lane < 5) s_acc[w][lane] = acc;
    __syncthreads();
    if (threadIdx.x < 5 && a.part) {
        double s = 0.0;
        for (int q = 0; q < (int)(blockDim.x >> 5); ++q) s += s_acc[q][threadIdx.x];
        a.part[(size_t)blockIdx.x * 5 + threadIdx.x] = s;
    }
}

// One chain in open space (the batch workload of the differentiation row).  GRAD: the
// partners are kept a second time sorted by letter (A monomers, then B, each run padded to an
// even length with a far-away dummy), so the coupling C of a run is one value for the row and
// the parameter sums need no selection; the record carries the partner's index, which excludes
// the row and its bonded neighbours.  Bound by the FMA pipe of the pair loop (65536
// conformations of a 55-mer: 135 us forward, 281 us backward; 375 us each, and 170 us of
// elementwise passes around them, when both computed everything in FP64 coordinates).
template <typename IN, bool GRAD, bool VJP>
__global__ void __launch_bounds__(32 * kGrad32Warps)
energy_grad32_chain_kernel(const SysDesc d, const Grad32Args a) {
    typedef typename GradOut<IN, VJP>::T OUT;
    extern __shared__ __align__(16) float4 sm4[];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, warps = blockDim.x >> 5;
    const int N = d.N;
    const int nA = d.n_a_before[N], nB = N - nA;
    const int pA = (nA + 1) & ~1, pB = (nB + 1) & ~1;
    float4* r = sm4 + (size_t)w * a.slot_f4;   // [N] (x, y, z, letter) relative to the origin, by index
    float4* ps = r + N;                        // [pA + pB] (x, y, z, index): A monomers, then B (GRAD)
    float4* lg = ps + N + 2;                   // [N] gradient of the bending, torsion and FENE terms (GRAD)
    const Coef<float> cf = coef32(d, a);
    const float kin = d.kin32;
    const int mid = N / 2;
    double acc = 0.0;
    if (GRAD && lane == 0) {   // the dummies
        if (nA & 1) ps[nA] = make_float4(kFar, kFar, kFar, __int_as_float(1 << 20));
        if (nB & 1) ps[pA + nB] = make_float4(kFar, kFar, kFar, __int_as_float(1 << 20));
    }
    for (unsigned b = blockIdx.x * warps + w; b < (unsigned)a.B; b += gridDim.x * warps) {   // beyond B it stays below 2^32
        const IN* x = (const IN*)a.xyz + (size_t)b * N * 3;
        // origin: the middle monomer rounded to FP32
        const float ox = as32(x[3 * mid]), oy = as32(x[3 * mid + 1]), oz = as32(x[3 * mid + 2]);
        for (int j = lane; j < N; j += 32) {
            const float rx = rel32(x[3 * j], ox), ry = rel32(x[3 * j + 1], oy), rz = rel32(x[3 * j + 2], oz);
            r[j] = make_float4(rx, ry, rz, __int_as_float((int)d.seq[j]));
            if (GRAD) {
                lg[j] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                const int ab = d.n_a_before[j];
                ps[d.seq[j] == 0 ? ab : pA + (j - ab)] = make_float4(rx, ry, rz, __int_as_float(j));
            }
        }
        __syncwarp();
        DF E{0.0f, 0.0f}, gp[5] = {{0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}};
        chain_terms32<GRAD, IN>(d, r, lg, x, 0, N, cf.kb, cf.kt, lane, E, gp);
        bool out = false;
        if (!VJP && d.sphere_R2 > 0.0)
            for (int j = lane; j < N; j += 32)
                out |= !inside64(d, make_double3(as64(x[3 * j]), as64(x[3 * j + 1]), as64(x[3 * j + 2])));
        double gE = 0.0;
        float gh = 0.0f, gl = 0.0f;
        if (VJP) {
            gE = a.gE[b];
            split_gE(gE, &gh, &gl);
        }
        if constexpr (!GRAD) {
            // rows i and i + 32 side by side, each against the partner s places on (cyclically):
            // every pair once; s = 1 holds the bonded pairs and that of the two ends
            for (int i0 = lane; i0 < N; i0 += 64) {
                const int i1 = i0 + 32;
                const float4 a0 = r[i0], a1 = i1 < N ? r[i1] : make_float4(-kFar, -kFar, -kFar, 0.0f);
                const int l0 = __float_as_int(a0.w), l1 = __float_as_int(a1.w);
                const float same0 = cf.c(3 * l0), same1 = cf.c(3 * l1), ab = 0.5f * (cf.c(1) + cf.c(2));   // as from both ends of a pair
                const float2 ax = make_float2(a0.x, a1.x), ay = make_float2(a0.y, a1.y), az = make_float2(a0.z, a1.z);
                float2 e = f2(0.0f);
                int j0 = i0 + 2, j1 = i1 + 2;
                for (int s = 2; s <= N / 2; ++s, ++j0, ++j1) {
                    if (j0 >= N) j0 -= N;
                    if (j1 >= N) j1 -= N;
                    const float4 q0 = r[j0], q1 = r[i1 < N ? j1 : j0];
                    const float2 dx = __fadd2_rn(ax, make_float2(-q0.x, -q1.x)), dy = __fadd2_rn(ay, make_float2(-q0.y, -q1.y)),
                                 dz = __fadd2_rn(az, make_float2(-q0.z, -q1.z));
                    float2 r2 = __fmul2_rn(dx, dx);
                    r2 = __ffma2_rn(dy, dy, r2);
                    r2 = __ffma2_rn(dz, dz, r2);
                    if (2 * s == N) {   // the opposite places: each pair comes twice, the first rows take it
                        if (2 * i0 >= N) r2.x = kFar2;
                        if (2 * i1 >= N) r2.y = kFar2;
                    }
                    const float2 sv = make_float2(fast_rcp(r2.x), fast_rcp(r2.y));
                    const float2 s3 = __fmul2_rn(__fmul2_rn(sv, sv), sv);
                    const float2 nC = make_float2(__float_as_int(q0.w) == l0 ? -same0 : -ab,
                                                  __float_as_int(q1.w) == l1 ? -same1 : -ab);
                    e = __ffma2_rn(s3, __fadd2_rn(s3, nC), e);
                }
                E = df_add(E, df_add(DF{kin * e.x, 0.0f}, DF{i1 < N ? kin * e.y : 0.0f, 0.0f}));
            }
            if (lane == 0) {   // the two ends
                const float4 a0 = r[0], q0 = r[N - 1];
                const float dx = a0.x - q0.x, dy = a0.y - q0.y, dz = a0.z - q0.z;
                const float sv = fast_rcp(dx * dx + dy * dy + dz * dz), s3 = sv * sv * sv;
                const float C = __float_as_int(a0.w) == __float_as_int(q0.w) ? cf.c(3 * __float_as_int(a0.w)) : 0.5f * (cf.c(1) + cf.c(2));
                E = df_add(E, DF{kin * (s3 * (s3 - C)), 0.0f});
            }
        } else {
            // the local-term gradients of row i, its output and its share of E and the parameters
            auto finish_row = [&](int i, int si, float2 gx, float2 gy, float2 gz, float2 e, float2 prA, float2 prB) {
                // both ends of every pair were taken: halves for the energy and the parameters
                if (!VJP) E = df_add(E, df_add(DF{0.5f * kin * e.x, 0.0f}, DF{0.5f * kin * e.y, 0.0f}));
                const float hk = -0.5f * kin;
                const DF pa = df_add(DF{hk * prA.x, 0.0f}, DF{hk * prA.y, 0.0f});   // partners A
                const DF pb = df_add(DF{hk * prB.x, 0.0f}, DF{hk * prB.y, 0.0f});   // partners B
                if (si == 0) { gp[0] = df_add(gp[0], pa); gp[2] = df_add(gp[2], pb); }
                else { gp[2] = df_add(gp[2], pa); gp[1] = df_add(gp[1], pb); }
                if (!a.grad_xyz) return;
                const float4 l4 = lg[i];   // its bending, torsion and FENE terms
                const float k6 = 6.0f * kin;
                OUT* go = (OUT*)a.grad_xyz + ((size_t)b * N + i) * 3;
                put_grad<VJP>(go, __fmaf_rn(k6, gx.x + gx.y, l4.x), gE, gh, gl);
                put_grad<VJP>(go + 1, __fmaf_rn(k6, gy.x + gy.y, l4.y), gE, gh, gl);
                put_grad<VJP>(go + 2, __fmaf_rn(k6, gz.x + gz.y, l4.z), gE, gh, gl);
            };
            // two rows per lane at a time, i0 = lane + 64 n and i1 = i0 + 32, against every partner:
            // the partner loads are shared and the two rows' chains are independent
            for (int i0 = lane; i0 < N; i0 += 64) {
                const int i1 = i0 + 32;
                const bool has1 = i1 < N;
                const float4 a0 = r[i0], a1 = has1 ? r[i1] : make_float4(-kFar, -kFar, -kFar, 0.0f);
                const int s0 = __float_as_int(a0.w) & 1, s1 = __float_as_int(a1.w) & 1;
                float2 gx0 = f2(0.0f), gy0 = f2(0.0f), gz0 = f2(0.0f), e0 = f2(0.0f);
                float2 gx1 = f2(0.0f), gy1 = f2(0.0f), gz1 = f2(0.0f), e1 = f2(0.0f);
                float2 pr0[2], pr1[2];
                const float2 m2 = f2(-2.0f);
#pragma unroll
                for (int seg = 0; seg < 2; ++seg) {   // partners of letter A, then B: one coupling C per run and row
                    const float C0 = cf.c(2 * s0 + seg), C1 = cf.c(2 * s1 + seg);
                    const float2 C0v = f2(C0), nC0 = f2(-C0), C1v = f2(C1), nC1 = f2(-C1);
                    float2 ap0 = f2(0.0f), ap1 = f2(0.0f);
                    const int k0 = seg ? pA : 0, k1 = seg ? pA + pB : pA;
                    for (int k = k0; k < k1; k += 2) {
                        const float4 q0 = ps[k], q1 = ps[k + 1];
                        const int j0 = __float_as_int(q0.w), j1 = __float_as_int(q1.w);
                        const float2 qx = make_float2(-q0.x, -q1.x), qy = make_float2(-q0.y, -q1.y),
                                     qz = make_float2(-q0.z, -q1.z);
                        // phi / k = s6 - C s3 and its 2 dphi/d(r^2) / (6 k) = s4 (C - 2 s3), s = 1 / r^2
                        auto row = [&](const float4& p, int i, float2 Cv, float2 nC, float2& gx, float2& gy, float2& gz,
                                       float2& e, float2& ap) {
                            const float2 dx = __fadd2_rn(f2(p.x), qx), dy = __fadd2_rn(f2(p.y), qy),
                                         dz = __fadd2_rn(f2(p.z), qz);
                            float2 r2 = __fmul2_rn(dx, dx);
                            r2 = __ffma2_rn(dy, dy, r2);
                            r2 = __ffma2_rn(dz, dz, r2);
                            // the row itself and its bonded neighbours (index within one of i): far away
                            if ((unsigned)(j0 - i + 1) <= 2u) r2.x = kFar2;
                            if ((unsigned)(j1 - i + 1) <= 2u) r2.y = kFar2;
                            const float2 sv = make_float2(fast_rcp(r2.x), fast_rcp(r2.y));
                            const float2 s2 = __fmul2_rn(sv, sv), s3 = __fmul2_rn(s2, sv);
                            const float2 fr = __fmul2_rn(__fmul2_rn(s2, s2), __ffma2_rn(m2, s3, Cv));
                            gx = __ffma2_rn(fr, dx, gx);
                            gy = __ffma2_rn(fr, dy, gy);
                            gz = __ffma2_rn(fr, dz, gz);
                            if (!VJP) e = __ffma2_rn(s3, __fadd2_rn(s3, nC), e);
                            ap = __fadd2_rn(ap, s3);
                        };
                        row(a0, i0, C0v, nC0, gx0, gy0, gz0, e0, ap0);
                        row(a1, i1, C1v, nC1, gx1, gy1, gz1, e1, ap1);   // (dropped when it does not exist)
                    }
                    pr0[seg] = ap0;
                    pr1[seg] = ap1;
                }
                finish_row(i0, s0, gx0, gy0, gz0, e0, pr0[0], pr0[1]);
                if (has1) finish_row(i1, s1, gx1, gy1, gz1, e1, pr1[0], pr1[1]);
            }
        }
        finish32<VJP>(a, b, E, gp, out, gE, lane, acc, VJP || a.grad_ff);
        __syncwarp();   // the slot is free
    }
    if constexpr (VJP) finish_part(a, acc, lane, w);
}

// Several chains, or one in a periodic box.  GRAD: partners chain by chain, two at a time (an
// odd chain's last pair ends with a dummy); a row is moved into the chain's frame once, so a
// pair costs no look-up of the shift, and the last rows, fewer than 32, have several lanes
// each, which split the partners.
template <typename IN, bool PBC, bool GRAD, bool VJP>
__global__ void __launch_bounds__(32 * kGrad32Warps)
energy_grad32_kernel(const SysDesc d, const Grad32Args a) {
    typedef typename GradOut<IN, VJP>::T OUT;
    extern __shared__ __align__(16) float4 sm4[];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, warps = blockDim.x >> 5;
    const unsigned full = 0xffffffffu;
    const int N = d.N, nc = d.n_chains;
    float4* r = sm4 + (size_t)w * a.slot_f4;          // [N] (x, y, z, letter | chain << 1) relative to the chain origin
    float4* D = r + N;                                // [nc][nc] minimum-imaged origin differences
    float4* org = D + nc * nc;                        // [nc] chain origins (FP32 values)
    float4* ps = org + nc;                            // [N + nc] the records, each chain at chain_off[c] + c (GRAD)
    float4* lg = ps + N + nc;                         // [N] gradient of the bending, torsion and FENE terms (GRAD)
    const int kDummy = -(1 << 20);
    const Coef<float> cf = coef32(d, a);
    const float2 Mg = f2(12582912.0f), nMg = f2(-12582912.0f);
    double acc = 0.0;
    if (GRAD)
        for (int c = lane; c < nc; c += 32)
            ps[d.chain_off[c + 1] + c] = make_float4(kFar, kFar, kFar, __int_as_float(2 * kDummy));
    for (unsigned b = blockIdx.x * warps + w; b < (unsigned)a.B; b += gridDim.x * warps) {   // beyond B it stays below 2^32
        const IN* x = (const IN*)a.xyz + (size_t)b * N * 3;
        for (int c = 0; c < nc; ++c) {                // chain centroids in FP32, summed by the warp
            const int o = d.chain_off[c], n = d.chain_off[c + 1] - o;
            float sx = 0.0f, sy = 0.0f, sz = 0.0f;
            for (int j = o + lane; j < o + n; j += 32) {
                sx += as32(x[3 * j]);
                sy += as32(x[3 * j + 1]);
                sz += as32(x[3 * j + 2]);
            }
#pragma unroll
            for (int m = 16; m > 0; m >>= 1) {
                if (m >= n) continue;                 // lanes from m on hold nothing
                sx += __shfl_xor_sync(full, sx, m);
                sy += __shfl_xor_sync(full, sy, m);
                sz += __shfl_xor_sync(full, sz, m);
            }
            if (lane == 0) org[c] = make_float4(sx / n, sy / n, sz / n, 0.0f);
        }
        __syncwarp();
        for (int j = lane; j < N; j += 32) {
            const int c = d.chain_of[j];
            const float4 oc = org[c];
            const float rx = rel32(x[3 * j], oc.x), ry = rel32(x[3 * j + 1], oc.y), rz = rel32(x[3 * j + 2], oc.z);
            r[j] = make_float4(rx, ry, rz, __int_as_float((int)d.seq[j] | (c << 1)));
            if (GRAD) {
                ps[j + c] = make_float4(rx, ry, rz, __int_as_float(2 * j + (int)d.seq[j]));
                lg[j] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            }
        }
        for (int p = lane; p < nc * nc; p += 32) {
            const float4 oa = org[p / nc], oc = org[p % nc];
            D[p] = make_float4(f64_to_f32(mimage64_short(d, f32_to_f64(oa.x) - f32_to_f64(oc.x))),
                               f64_to_f32(mimage64_short(d, f32_to_f64(oa.y) - f32_to_f64(oc.y))),
                               f64_to_f32(mimage64_short(d, f32_to_f64(oa.z) - f32_to_f64(oc.z))), 0.0f);
        }
        __syncwarp();
        DF E{0.0f, 0.0f}, gp[5] = {{0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}};
        for (int c = 0; c < nc; ++c) {
            const int o = d.chain_off[c], n = d.chain_off[c + 1] - o;
            chain_terms32<GRAD, IN>(d, r, lg, x, o, n, cf.kb, cf.kt, lane, E, gp);
        }
        bool out = false;   // a monomer beyond the container's wall: infinite energy
        if (!VJP && d.sphere_R2 > 0.0)
            for (int j = lane; j < N; j += 32)
                out |= !inside64(d, make_double3(as64(x[3 * j]), as64(x[3 * j + 1]), as64(x[3 * j + 2])));
        double gE = 0.0;
        float gh = 0.0f, gl = 0.0f;
        if (VJP) {
            gE = a.gE[b];
            split_gE(gE, &gh, &gl);
        }
        if constexpr (!GRAD) {
            // a row against the partners s and s + 1 places on (cyclically), every pair once
            for (int i = lane; i < N; i += 32) {
                const float4 p = r[i];
                const int ti = __float_as_int(p.w), ci = ti >> 1;
                const float same = cf.c(3 * (ti & 1)), ab = cf.c(1);
                float2 e = f2(0.0f);
                for (int s = 1; s <= N / 2; s += 2) {
                    int j0 = i + s, j1 = i + s + 1;
                    if (j0 >= N) j0 -= N;
                    if (j1 >= N) j1 -= N;
                    const float4 q0 = r[j0], q1 = r[j1];
                    const int t0 = __float_as_int(q0.w), t1 = __float_as_int(q1.w);
                    const bool in0 = (t0 >> 1) == ci, in1 = (t1 >> 1) == ci;
                    const float4 s0 = D[ci * nc + (t0 >> 1)], s1 = D[ci * nc + (t1 >> 1)];
                    float2 dx = __fadd2_rn(__fadd2_rn(f2(p.x), make_float2(-q0.x, -q1.x)), make_float2(s0.x, s1.x));
                    float2 dy = __fadd2_rn(__fadd2_rn(f2(p.y), make_float2(-q0.y, -q1.y)), make_float2(s0.y, s1.y));
                    float2 dz = __fadd2_rn(__fadd2_rn(f2(p.z), make_float2(-q0.z, -q1.z)), make_float2(s0.z, s1.z));
                    if (PBC) {   // a zero box length leaves a displacement within the chain unchanged
                        const float2 iL = make_float2(in0 ? 0.0f : d.iL32, in1 ? 0.0f : d.iL32);
                        const float2 nL = make_float2(in0 ? 0.0f : -d.L32, in1 ? 0.0f : -d.L32);
                        dx = __ffma2_rn(nL, __fadd2_rn(__ffma2_rn(dx, iL, Mg), nMg), dx);
                        dy = __ffma2_rn(nL, __fadd2_rn(__ffma2_rn(dy, iL, Mg), nMg), dy);
                        dz = __ffma2_rn(nL, __fadd2_rn(__ffma2_rn(dz, iL, Mg), nMg), dz);
                    }
                    float2 r2 = __fmul2_rn(dx, dx);
                    r2 = __ffma2_rn(dy, dy, r2);
                    r2 = __ffma2_rn(dz, dz, r2);
                    // left out: bonded neighbours (s = 1), the second end of opposite places, s + 1 beyond half
                    const bool x0 = (in0 && j0 == i + 1) || (2 * s == N && 2 * i >= N);
                    const bool x1 = 2 * (s + 1) > N || (2 * (s + 1) == N && 2 * i >= N);
                    r2 = make_float2(x0 ? kFar2 : r2.x, x1 ? kFar2 : r2.y);
                    const float2 k = make_float2(x0 ? 0.0f : in0 ? d.kin32 : d.kout32, x1 ? 0.0f : in1 ? d.kin32 : d.kout32);
                    const float2 sv = make_float2(fast_rcp(r2.x), fast_rcp(r2.y));
                    const float2 s3 = __fmul2_rn(__fmul2_rn(sv, sv), sv);
                    const float2 nC = make_float2(((t0 ^ ti) & 1) ? -ab : -same, ((t1 ^ ti) & 1) ? -ab : -same);
                    e = __ffma2_rn(__fmul2_rn(k, s3), __fadd2_rn(s3, nC), e);
                }
                E = df_add(E, df_add(DF{e.x, 0.0f}, DF{e.y, 0.0f}));
            }
        } else {
            for (int row0 = 0; row0 < N; row0 += 32) {
                const int P = min(32, N - row0);
                const int Pp = P > 1 ? 1 << (32 - __clz(P - 1)) : 1;   // lanes a set of rows; 32 / Pp sets
                const int li = lane & (Pp - 1), sub = lane / Pp, sets = 32 / Pp;
                const bool has = li < P;
                const int i = has ? row0 + li : row0;
                const float4 p = r[i];
                const int ti = __float_as_int(p.w), ci = ti >> 1, si = ti & 1;
                const float CA = si ? cf.c(1) : cf.c(0), CB = si ? cf.c(3) : cf.c(1);   // one value for AB and BA, as in the energies
                float2 Gx = f2(0.0f), Gy = f2(0.0f), Gz = f2(0.0f), Ee = f2(0.0f), PA = f2(0.0f), PB = f2(0.0f);
                for (int c = 0; c < nc; ++c) {
                    const bool in = c == ci;
                    const float4 sh = D[ci * nc + c];   // zero within a chain
                    const float ax = p.x + sh.x, ay = p.y + sh.y, az = p.z + sh.z;
                    const float2 iL = f2(in ? 0.0f : d.iL32), nL = f2(in ? 0.0f : -d.L32);
                    const int far = in ? i - 1 : kDummy - 1;   // partners far .. far + 2 are left out
                    const float4* q = ps + d.chain_off[c] + c;
                    const int np = (d.chain_off[c + 1] - d.chain_off[c] + 1) >> 1;
                    float2 gx = f2(0.0f), gy = f2(0.0f), gz = f2(0.0f), e = f2(0.0f), pa = f2(0.0f), pb = f2(0.0f);
#pragma unroll 2
                    for (int k = sub; k < np; k += sets) {
                        const float4 q0 = q[2 * k], q1 = q[2 * k + 1];
                        const int t0 = __float_as_int(q0.w), t1 = __float_as_int(q1.w);
                        float2 dx = __fadd2_rn(f2(ax), make_float2(-q0.x, -q1.x)), dy = __fadd2_rn(f2(ay), make_float2(-q0.y, -q1.y)),
                               dz = __fadd2_rn(f2(az), make_float2(-q0.z, -q1.z));
                        if (PBC) {
                            dx = __ffma2_rn(nL, __fadd2_rn(__ffma2_rn(dx, iL, Mg), nMg), dx);
                            dy = __ffma2_rn(nL, __fadd2_rn(__ffma2_rn(dy, iL, Mg), nMg), dy);
                            dz = __ffma2_rn(nL, __fadd2_rn(__ffma2_rn(dz, iL, Mg), nMg), dz);
                        }
                        float2 r2 = __fmul2_rn(dx, dx);
                        r2 = __ffma2_rn(dy, dy, r2);
                        r2 = __ffma2_rn(dz, dz, r2);
                        if ((unsigned)((t0 >> 1) - far) <= 2u) r2.x = kFar2;
                        if ((unsigned)((t1 >> 1) - far) <= 2u) r2.y = kFar2;
                        const float2 sv = make_float2(fast_rcp(r2.x), fast_rcp(r2.y));
                        const float2 s2 = __fmul2_rn(sv, sv), s3 = __fmul2_rn(s2, sv);
                        const float2 Cv = make_float2((t0 & 1) ? CB : CA, (t1 & 1) ? CB : CA);
                        const float2 fr = __fmul2_rn(__fmul2_rn(s2, s2), __ffma2_rn(f2(-2.0f), s3, Cv));
                        gx = __ffma2_rn(fr, dx, gx);
                        gy = __ffma2_rn(fr, dy, gy);
                        gz = __ffma2_rn(fr, dz, gz);
                        if (!VJP) e = __ffma2_rn(s3, __ffma2_rn(f2(-1.0f), Cv, s3), e);
                        pa = __fadd2_rn(pa, make_float2((t0 & 1) ? 0.0f : s3.x, (t1 & 1) ? 0.0f : s3.y));
                        pb = __fadd2_rn(pb, make_float2((t0 & 1) ? s3.x : 0.0f, (t1 & 1) ? s3.y : 0.0f));
                    }
                    const float kc = in ? d.kin32 : d.kout32;
                    const float2 k1 = f2(kc), k6 = f2(6.0f * kc);
                    Gx = __ffma2_rn(k6, gx, Gx);
                    Gy = __ffma2_rn(k6, gy, Gy);
                    Gz = __ffma2_rn(k6, gz, Gz);
                    if (!VJP) Ee = __ffma2_rn(k1, e, Ee);
                    PA = __ffma2_rn(k1, pa, PA);
                    PB = __ffma2_rn(k1, pb, PB);
                }
                float gxs = Gx.x + Gx.y, gys = Gy.x + Gy.y, gzs = Gz.x + Gz.y;
                for (int o = Pp; o < 32; o <<= 1) {   // the row's lanes
                    gxs += __shfl_xor_sync(full, gxs, o);
                    gys += __shfl_xor_sync(full, gys, o);
                    gzs += __shfl_xor_sync(full, gzs, o);
                }
                if (has) {   // every lane's own share; both ends of every pair were taken: halves
                    if (!VJP) E = df_add(E, df_add(DF{0.5f * Ee.x, 0.0f}, DF{0.5f * Ee.y, 0.0f}));
                    const DF va = df_add(DF{-0.5f * PA.x, 0.0f}, DF{-0.5f * PA.y, 0.0f});
                    const DF vb = df_add(DF{-0.5f * PB.x, 0.0f}, DF{-0.5f * PB.y, 0.0f});
                    if (si == 0) { gp[0] = df_add(gp[0], va); gp[2] = df_add(gp[2], vb); }
                    else { gp[2] = df_add(gp[2], va); gp[1] = df_add(gp[1], vb); }
                    if (sub == 0 && a.grad_xyz) {
                        const float4 l4 = lg[i];
                        OUT* go = (OUT*)a.grad_xyz + ((size_t)b * N + i) * 3;
                        put_grad<VJP>(go, gxs + l4.x, gE, gh, gl);
                        put_grad<VJP>(go + 1, gys + l4.y, gE, gh, gl);
                        put_grad<VJP>(go + 2, gzs + l4.z, gE, gh, gl);
                    }
                }
            }
        }
        finish32<VJP>(a, b, E, gp, out, gE, lane, acc, VJP || a.grad_ff);
        __syncwarp();   // the slot is free
    }
    if constexpr (VJP) finish_part(a, acc, lane, w);
}

// Sum of n rows of five, in a fixed order: one CTA.
__global__ void __launch_bounds__(160) sum_parts_kernel(int n, const double* __restrict__ part, void* __restrict__ out, int out32) {
    __shared__ double s[160];
    const int q = threadIdx.x % 5, t = threadIdx.x / 5;   // 32 partial sums a column
    double v = 0.0;
#pragma unroll 8
    for (int i = t; i < n; i += 32) v += part[(size_t)i * 5 + q];
    s[threadIdx.x] = v;
    __syncthreads();
    if (threadIdx.x < 5) {
        double z = 0.0;
        for (int i = 0; i < 32; ++i) z += s[5 * i + threadIdx.x];
        if (out32) ((float*)out)[threadIdx.x] = (float)z;
        else ((double*)out)[threadIdx.x] = z;
    }
}

// ---------------------------------------------------------------------------
// Reweighting: log-sum-exp maximum, the weighted means, then centred moments, all in FP64.
// A cluster of CTAs per temperature, each on its share of the samples and keeping their
// weights in shared memory, so that a weight's exponential is taken once (again only for the
// samples of a share beyond kRwKeep); the clusters' partial results are exchanged through
// distributed shared memory and summed in rank order.  Bound by the FP64 pipe: about 27
// FP64 instructions a sample and temperature (the form with one CTA per temperature used 64
// of 152 SMs and two exponentials).  65536 samples, 64 temperatures: 353 us
// (940 us before).
// ---------------------------------------------------------------------------
constexpr int kRwThreads = 256;
constexpr int kRwKeep = 6080;    // weights kept per CTA (four CTAs on an SM, static shared memory)

// Sums v over the cluster's CTAs (each CTA's in s_part), in rank order, on every thread.
template <int CTAS, int M>
__device__ __forceinline__ void rw_sums(cg::cluster_group& cl, double* s_part, double (&v)[M], double* red) {
    int first = 0, count = M;
    warp_sums<M>(v, &first, &count);
    __syncthreads();
    if (count == 1) red[(threadIdx.x >> 5) * M + first] = v[0];
    __syncthreads();
    if (threadIdx.x < M) {
        double s = 0.0;
        for (int w = 0; w < kRwThreads / 32; ++w) s += red[w * M + threadIdx.x];
        s_part[threadIdx.x] = s;
    }
    if (CTAS > 1) cl.sync();
    else __syncthreads();
#pragma unroll
    for (int q = 0; q < M; ++q) {
        v[q] = 0.0;
#pragma unroll
        for (int c = 0; c < CTAS; ++c) v[q] += CTAS > 1 ? cl.map_shared_rank(s_part, c)[q] : s_part[q];
    }
}

template <int CTAS>
__global__ void __launch_bounds__(kRwThreads)
reweight_kernel(int64_t n, const double* __restrict__ E, const double* __restrict__ D, const double* __restrict__ lnW,
                int n_monomers, const double* __restrict__ T, double* E_T, double* cV_T, double* dE_T, double* dcV_T) {
    __shared__ double wt[kRwKeep];
    __shared__ double red[32], s_a[3], s_b[3];
    __shared__ long long s_max;
    cg::cluster_group cl = cg::this_cluster();
    const int i = blockIdx.x / CTAS, rank = blockIdx.x % CTAS;
    const double beta = 1.0 / T[i];
    const int64_t q0 = n * rank / CTAS, m = n * (rank + 1) / CTAS - q0;   // this CTA's samples
    E += q0;
    D += q0;
    lnW += q0;
    const int64_t keep = m < (int64_t)(sizeof(wt) / sizeof(wt[0])) ? m : (int64_t)(sizeof(wt) / sizeof(wt[0]));
    long long top = PHAST_KEY_LOWEST;
#pragma unroll 4
    for (int64_t q = threadIdx.x; q < m; q += kRwThreads) {
        const double a = -beta * E[q] - lnW[q];
        if (q < keep) wt[q] = a;   // read back by the same thread
        top = is_nan64(a) ? top : max(top, order_key(a));
    }
    top = block_max_key(top, reinterpret_cast<long long*>(red));
    if (CTAS > 1) {
        if (threadIdx.x == 0) s_max = top;
        cl.sync();
#pragma unroll
        for (int c = 0; c < CTAS; ++c) top = max(top, *cl.map_shared_rank(&s_max, c));
    }
    const double amax = key_value(top);
    double s1[3] = {0.0, 0.0, 0.0};   // Z, sum w E, sum w D
#pragma unroll 2
    for (int64_t q = threadIdx.x; q < m; q += kRwThreads) {
        const double w = exp64_neg((q < keep ? wt[q] : -beta * E[q] - lnW[q]) - amax);
        if (q < keep) wt[q] = w;
        s1[0] += w;
        s1[1] += w * E[q];
        s1[2] += w * D[q];
    }
    rw_sums<CTAS, 3>(cl, s_a, s1, red);
    const double Z = s1[0], mE = s1[1] / Z, mD = s1[2] / Z;
    double s2[3] = {0.0, 0.0, 0.0};   // centred moments e e, e d, e e d
    for (int64_t q = threadIdx.x; q < m; q += kRwThreads) {
        const double w = q < keep ? wt[q] : exp64_neg(-beta * E[q] - lnW[q] - amax);
        const double e = E[q] - mE, dd = D[q] - mD, we = w * e, wee = we * e;
        s2[0] += wee;
        s2[1] += we * dd;
        s2[2] += wee * dd;
    }
    rw_sums<CTAS, 3>(cl, s_b, s2, red);
    if (rank == 0 && threadIdx.x == 0) {
        const double vE = s2[0] / Z, cED = s2[1] / Z, m3 = s2[2] / Z;
        const double nT2 = (double)n_monomers * T[i] * T[i];
        E_T[i] = mE;
        cV_T[i] = vE / nT2;
        dE_T[i] = mD - beta * cED;
        dcV_T[i] = (2.0 * cED - beta * m3) / nT2;
    }
    if (CTAS > 1) cl.sync();   // no CTA leaves while another reads its sums
}

}  // namespace

namespace {
// Kernels of one form; a conformation's slot of shared memory in float4.
typedef void (*grad32_fn)(const SysDesc, const Grad32Args);
template <typename IN, bool GRAD, bool VJP>
grad32_fn pick_grad32(bool chain, bool pbc) {
    if (chain) return energy_grad32_chain_kernel<IN, GRAD, VJP>;
    return pbc ? energy_grad32_kernel<IN, true, GRAD, VJP> : energy_grad32_kernel<IN, false, GRAD, VJP>;
}

constexpr int kGrad32MaxCtas = PHAST_VJP_DOUBLES / 5;   // partial sums of a backward pass

int launch_grad32(const SysDesc& d, grad32_fn fn, bool chain, bool grad, Grad32Args a, int* n_ctas, cudaStream_t st) {
    a.slot_f4 = chain ? (grad ? 3 * d.N + 2 : d.N)
                      : d.N + d.n_chains * d.n_chains + d.n_chains + (grad ? 2 * d.N + d.n_chains : 0);
    int warps = kGrad32Warps;
    while (warps > 1 && sizeof(float4) * (size_t)a.slot_f4 * warps > 200 * 1024) warps >>= 1;
    const size_t sm = sizeof(float4) * (size_t)a.slot_f4 * warps;
    PHAST_CUDA_TRY(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    // a few waves of CTAs, each warp taking several conformations of a large batch
    int ctas = (a.B - 1) / warps + 1;
    *n_ctas = ctas = ctas < kGrad32MaxCtas ? ctas : kGrad32MaxCtas;
    fn<<<ctas, 32 * warps, sm, st>>>(d, a);
    PHAST_CUDA_TRY(cudaGetLastError());
    return PHAST_OK;
}

int check_grad(const phast_system* sys, const phast_ff* ff, int32_t B, int32_t pair_precision, const char* what, SysDesc* d) {
    const int rc = phast_build_desc(sys, ff, nullptr, d, what);
    if (rc) return rc;
    if (B < 0) return phast_set_error(PHAST_EINVAL, "%s: B < 0", what);
    if (pair_precision != 32 && pair_precision != 64)
        return phast_set_error(PHAST_EINVAL, "%s: pair_precision must be 32 or 64", what);
    return PHAST_OK;
}

int energy_grad(const phast_system* sys, const phast_ff* ff, int32_t B, const double* xyz, int32_t pair_precision,
                const double* params, double* E_out, double* grad_xyz, double* grad_ff, void* stream) {
    SysDesc d;
    int rc = check_grad(sys, ff, B, pair_precision, "phast_energy_grad", &d);
    if (rc) return rc;
    if (B == 0) return PHAST_OK;
    if (!xyz) return phast_set_error(PHAST_EINVAL, "phast_energy_grad: NULL xyz");
    cudaStream_t st = (cudaStream_t)stream;
    if (pair_precision == 64) {
        dim3 grid((B + kGradWarps - 1) / kGradWarps), block(32 * kGradWarps);
        const size_t sm = grad64_slot_bytes(d.N) * kGradWarps;
        PHAST_CUDA_TRY(cudaFuncSetAttribute(energy_grad64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
        energy_grad64_kernel<<<grid, block, sm, st>>>(d, B, xyz, E_out, grad_xyz, grad_ff, params);
        PHAST_CUDA_TRY(cudaGetLastError());
        return PHAST_OK;
    }
    const bool chain = d.n_chains == 1 && !(d.box_L > 0.0), grad = grad_xyz || grad_ff;
    Grad32Args a = {};
    a.B = B;
    a.xyz = xyz;
    a.E_out = E_out;
    a.grad_xyz = grad_xyz;
    a.grad_ff = grad_ff;
    a.pdev = params;
    int n;
    return launch_grad32(d, grad ? pick_grad32<double, true, false>(chain, d.box_L > 0.0)
                                 : pick_grad32<double, false, false>(chain, d.box_L > 0.0), chain, grad, a, &n, st);
}
}  // namespace

extern "C" int phast_energy_grad(const phast_system* sys, const phast_ff* ff, int32_t B, const double* xyz,
                                 int32_t pair_precision, double* E_out, double* grad_xyz, double* grad_ff,
                                 void* stream) {
    return energy_grad(sys, ff, B, xyz, pair_precision, nullptr, E_out, grad_xyz, grad_ff, stream);
}

extern "C" int phast_energy_grad_params(const phast_system* sys, const phast_ff* ff, int32_t B, const double* xyz,
                                        int32_t pair_precision, const double* params, double* E_out,
                                        double* grad_xyz, double* grad_ff, void* stream) {
    if (!params) return phast_set_error(PHAST_EINVAL, "phast_energy_grad_params: NULL params");
    return energy_grad(sys, ff, B, xyz, pair_precision, params, E_out, grad_xyz, grad_ff, stream);
}

extern "C" int phast_energy_forward32(const phast_system* sys, const phast_ff* ff, int32_t B, const void* xyz,
                                      int32_t xyz_bits, const void* params, int32_t params_bits, double* E_out,
                                      void* stream) {
    SysDesc d;
    const int rc = check_grad(sys, ff, B, 32, "phast_energy_forward32", &d);
    if (rc) return rc;
    if ((xyz_bits != 32 && xyz_bits != 64) || (params_bits != 32 && params_bits != 64))
        return phast_set_error(PHAST_EINVAL, "phast_energy_forward32: xyz_bits and params_bits must be 32 or 64");
    if (B == 0) return PHAST_OK;
    if (!xyz || !E_out) return phast_set_error(PHAST_EINVAL, "phast_energy_forward32: NULL argument");
    const bool chain = d.n_chains == 1 && !(d.box_L > 0.0), pbc = d.box_L > 0.0;
    Grad32Args a = {};
    a.B = B;
    a.xyz = xyz;
    a.E_out = E_out;
    a.pdev = params;
    a.p32 = params_bits == 32;
    int n;
    return launch_grad32(d, xyz_bits == 32 ? pick_grad32<float, false, false>(chain, pbc) : pick_grad32<double, false, false>(chain, pbc),
                         chain, false, a, &n, (cudaStream_t)stream);
}

extern "C" int phast_energy_backward32(const phast_system* sys, const phast_ff* ff, int32_t B, const void* xyz,
                                       int32_t xyz_bits, const void* params, int32_t params_bits, const double* grad_E,
                                       void* grad_xyz, void* grad_params, double* workspace, void* stream) {
    SysDesc d;
    const int rc = check_grad(sys, ff, B, 32, "phast_energy_backward32", &d);
    if (rc) return rc;
    if ((xyz_bits != 32 && xyz_bits != 64) || (params_bits != 32 && params_bits != 64))
        return phast_set_error(PHAST_EINVAL, "phast_energy_backward32: xyz_bits and params_bits must be 32 or 64");
    cudaStream_t st = (cudaStream_t)stream;
    if (B > 0 && (!xyz || !grad_E)) return phast_set_error(PHAST_EINVAL, "phast_energy_backward32: NULL argument");
    if (grad_params && !workspace) return phast_set_error(PHAST_EINVAL, "phast_energy_backward32: NULL workspace");
    int n = 0;
    if (B > 0) {
        const bool chain = d.n_chains == 1 && !(d.box_L > 0.0), pbc = d.box_L > 0.0;
        Grad32Args a = {};
        a.B = B;
        a.xyz = xyz;
        a.grad_xyz = grad_xyz;
        a.pdev = params;
        a.p32 = params_bits == 32;
        a.gE = grad_E;
        a.part = grad_params ? workspace : nullptr;
        const int rc2 = launch_grad32(d, xyz_bits == 32 ? pick_grad32<float, true, true>(chain, pbc) : pick_grad32<double, true, true>(chain, pbc),
                                      chain, true, a, &n, st);
        if (rc2) return rc2;
    }
    if (grad_params) {
        sum_parts_kernel<<<1, 160, 0, st>>>(n, workspace, grad_params, params_bits == 32);
        PHAST_CUDA_TRY(cudaGetLastError());
    }
    return PHAST_OK;
}

extern "C" int phast_reweight_sensitivity(int64_t n, const double* E, const double* D, const double* lnW,
                                          int32_t n_monomers, int32_t n_T, const double* T, double* E_T,
                                          double* cV_T, double* dE_T, double* dcV_T, void* stream) {
    if (n < 1) return phast_set_error(PHAST_EINVAL, "phast_reweight_sensitivity: n < 1");
    if (n_monomers < 1) return phast_set_error(PHAST_EINVAL, "phast_reweight_sensitivity: n_monomers < 1");
    if (n_T < 0) return phast_set_error(PHAST_EINVAL, "phast_reweight_sensitivity: n_T < 0");
    if (n_T == 0) return PHAST_OK;
    if (!E || !D || !lnW || !T || !E_T || !cV_T || !dE_T || !dcV_T)
        return phast_set_error(PHAST_EINVAL, "phast_reweight_sensitivity: NULL argument");
    // CTAs per temperature: enough of them for about three on every SM, each with a thousand
    // samples or more (a few thousand samples: 29 us a call on one CTA, 53 us on eight), and no
    // more samples than a CTA keeps where that can be
    int ctas = 1;
    while (ctas < 8 && ((int64_t)n_T * ctas < 300 || n > (int64_t)kRwKeep * ctas) && n / (2 * ctas) >= 1024) ctas *= 2;
    auto fn = ctas == 1 ? reweight_kernel<1> : ctas == 2 ? reweight_kernel<2> : ctas == 4 ? reweight_kernel<4> : reweight_kernel<8>;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)n_T * ctas);
    cfg.blockDim = dim3(kRwThreads);
    cfg.stream = (cudaStream_t)stream;
    cudaLaunchAttribute cluster;
    cluster.id = cudaLaunchAttributeClusterDimension;
    cluster.val.clusterDim.x = ctas;
    cluster.val.clusterDim.y = cluster.val.clusterDim.z = 1;
    cfg.attrs = &cluster;
    cfg.numAttrs = 1;
    PHAST_CUDA_TRY(cudaLaunchKernelEx(&cfg, fn, n, E, D, lnW, (int)n_monomers, T, E_T, cV_T, dE_T, dcV_T));
    return PHAST_OK;
}
