// energy.cu -- phast_energy (Eq. 2/3 total energy of a batch of
// configurations) and phast_delta_energy (energy change of explicit moves).
// One warp per configuration or move (FP64 energies of larger systems: four), using the
// same group machinery as the sweep.
#include "group.cuh"

namespace {

constexpr int kWarpsPerBlock = 4;
// FP64 energies: systems from here on take far pairs in double-float, four warps each.  It gains from
// 40 monomers on (4096 configurations, double-float against FP64 throughout on one warp each: 36
// monomers 117 and 113 us, 40: 124 and 138, 48: 141 and 198, 64: 176 and 365; of 64 configurations
// 48 monomers take 19 and 46 us); smaller systems keep the plain form.
constexpr int kSplitMinN = 48;
constexpr int kSplitWarps = 4;   // warps of such a configuration
// When a configuration's far pairs may be taken in double-float.  Their errors, over the pairs' sizes v: a
// few 1e-15 of sum |v| (what the products leave out has one sign), and of the root of sum v^2, pair by
// pair, some 1e-14 of the arithmetic and 2e-15 c of the displacements' 48 bits (c: the largest coordinate
// from its chain's origin or difference of origins).  That may come to eight FP64 roundings of the rest of
// the energy (2^-53 of it; every term has a dozen): 4 sum |v| + (12 + 2 c) sqrt(sum v^2) <= the rest.
// Beyond it (nothing near and no bending: conformations blown up, chains that interact from afar;
// unwrapped chains many boxes long) a configuration is taken in FP64 throughout.  Largest errors against
// extended precision in roundings of the sum of the terms' sizes, FP64 throughout -> here: random walks of
// 48 to 512 monomers 2.3 to 7.0 -> 1.5 to 2.8, straight chains (which come nearest to the limit) of 48 to
// 512 2.3 to 7.8 -> 1.3 to 5.3, with bonds of 1.5 8.4 to 22.6 -> 5.8 to 10.8.
constexpr float kSplitCommon = 4.0f, kSplitPair = 12.0f, kSplitCoord = 2.0f;

// FP32 pairs: one warp per configuration.
__global__ void __launch_bounds__(32 * kWarpsPerBlock)
energy32_kernel(const SysDesc d, int B, const double* __restrict__ xyz, double* __restrict__ E_out, SlotLayout L) {
    extern __shared__ __align__(16) unsigned char smem[];
    Group<32> g;
    const int w = threadIdx.x >> 5;
    const int b = blockIdx.x * kWarpsPerBlock + w;
    if (b >= B) return;
    const double* x64 = xyz + (size_t)b * d.N * 3;
    Slot<float> s(smem + (size_t)w * L.bytes, L);
    build_working<32, float>(d, x64, s, g);
    double E = full_energy_working32(d, x64, s, g);
    bool out = false;   // a monomer beyond the container's wall: infinite energy
    if (d.has_sphere)
        for (int j = g.lane; j < d.N; j += 32) out |= !inside64(d, ld3(x64 + 3 * j));
    if (__any_sync(g.mask, out)) E = INFINITY;
    if (g.lane == 0) E_out[b] = E;
}

// ---------------------------------------------------------------------------
// FP64 energies: W warps per configuration.  The pairs are one flat list (index s N + i: the
// pair of monomers i and i + s + 1, cyclically, every pair once), dealt to the lanes.
//
// An FP64 instruction holds an SMSP's pipe for 64 to 76 cycles, 13 to 16 of them make a pair,
// and nearly all pairs of a large system are far apart.  SPLIT: a pair further apart than 4
// (r^-6 below 2.5e-4) is evaluated in double-float arithmetic (two FP32 numbers, about 130
// FP32 instructions) on coordinates relative to a monomer of its chain, to some 1e-14 of it, which
// the near pairs and the bends dwarf (kSplitCommon: else the configuration is taken in FP64);
// nearer pairs, and those whose image count or magnitude FP32 does not settle, are collected and
// take the FP64 instructions, a full warp at a time.
// 1024 configurations of eight 55-mers: 1.05 ms (6.12 ms in FP64 throughout).
// ---------------------------------------------------------------------------
struct NearPair { int i, j; };   // i < j: C_LJ takes the earlier monomer's letter first

__device__ __forceinline__ double pair_energy64(const SysDesc& d, const double* x64, int i, int j) {
    const double3 a = ld3(x64 + 3 * i), b = ld3(x64 + 3 * j);
    double dx = a.x - b.x, dy = a.y - b.y, dz = a.z - b.z;
    const bool inter = d.chain_of[i] != d.chain_of[j];
    if (inter) {
        dx = mimage64_short(d, dx);
        dy = mimage64_short(d, dy);
        dz = mimage64_short(d, dz);
    }
    const double ir2 = rcp64(dx * dx + dy * dy + dz * dz);
    const double ir6 = ir2 * ir2 * ir2;
    return (inter ? d.k_lj_inter : d.k_lj_intra) * (ir6 * (ir6 - d.C[2 * d.seq[i] + d.seq[j]]));
}

// part plus the pairs first, first + stride, ... of the flat list.
__device__ __forceinline__ double add_pairs64(double part, const SysDesc& d, const double* x64, int first, int stride) {
    const int N = d.N, total = N * (N - 1) / 2, dq = stride / N, dt = stride % N;
    int s = first / N, i = first % N;
    for (int idx = first; idx < total; idx += stride) {
        int j = i + s + 1;
        if (j >= N) j -= N;
        if (s > 0 || j != i + 1 || d.chain_of[i] != d.chain_of[j]) part += pair_energy64(d, x64, min(i, j), max(i, j));
        s += dq;
        i += dt;
        if (i >= N) { i -= N; ++s; }
    }
    return part;
}
// A lane's share of a configuration's energy, all of it in FP64.
static __device__ __noinline__ double whole_energy64(const SysDesc& d, const double* x64, int lane, int w, int W) {
    return add_pairs64(local_energy64_warp(d, x64, lane, w, W), d, x64, w * 32 + lane, 32 * W);
}

// a - b and a + b with their rounding errors (TwoSum).
__device__ __forceinline__ float two_diff(float a, float b, float* e) {
    const float s = __fsub_rn(a, b), bb = __fsub_rn(s, a);
    *e = __fsub_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fadd_rn(b, bb));
    return s;
}
__device__ __forceinline__ float two_sum(float a, float b, float* e) {
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    *e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return s;
}

struct SplitBox { float Lh, Ll, iL, edge; };   // box side in two parts, its inverse, L/2 less a margin

// One component of the displacement of far pairs, in double-float: a - b + D, less the box
// length times the nearest count.  *unsure: the count is not settled (|d| within 1e-5 of L/2).
__device__ __forceinline__ float split_diff(float ah, float al, float bh, float bl, float Dh, float Dl, bool inter,
                                            const SplitBox& B, float* lo, bool* unsure) {
    float e;
    float s = two_diff(ah, bh, &e);
    float l = __fadd_rn(__fsub_rn(al, bl), e);
    if (inter) {
        s = two_sum(s, Dh, &e);
        l = __fadd_rn(l, __fadd_rn(Dl, e));
        const float k = image_count(s, B.iL);   // 0 in open space
        if (k != 0.0f) {
            const float p = __fmul_rn(k, B.Lh), pe = __fmaf_rn(k, B.Lh, -p);
            s = two_diff(s, p, &e);
            l = __fadd_rn(l, __fsub_rn(e, __fmaf_rn(k, B.Ll, pe)));
        }
        *unsure |= fabsf(s) > B.edge;
    }
    // the low part may be far above a rounding of the high one (the coordinates are larger than their
    // difference): bring it there, or the products that the square leaves out would count
    const float h = __fadd_rn(s, l);
    *lo = __fsub_rn(l, __fsub_rn(h, s));
    return h;
}

template <int W, bool SPLIT>
__global__ void __launch_bounds__(W > 1 ? 32 * W : 32 * kWarpsPerBlock)
energy64_kernel(const SysDesc d, int B, const double* __restrict__ xyz, double* __restrict__ E_out) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ NearPair s_near[W > 1 ? W : kWarpsPerBlock][64];
    __shared__ double red[32];
    __shared__ float4 s_size[W];   // SPLIT, of each warp: sums of the far pairs' sizes and squares, largest coordinate, size of the rest
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int w = W > 1 ? warp : 0;                                   // the warp's number within the configuration
    const int b = W > 1 ? blockIdx.x : blockIdx.x * kWarpsPerBlock + warp;
    if (b >= B) return;
    const unsigned full = 0xffffffffu;
    const int N = d.N;
    const double* x64 = xyz + (size_t)b * N * 3;
    double part = local_energy64_warp(d, x64, lane, w, W);
    bool out = false;   // a monomer beyond the container's wall: infinite energy
    if (d.has_sphere)
        for (int j = w * 32 + lane; j < N; j += 32 * W) out |= !inside64(d, ld3(x64 + 3 * j));
    if constexpr (SPLIT) {
        const int nc = d.n_chains, total = N * (N - 1) / 2;
        const int dq = 32 * W / N, dt = 32 * W % N;
        int idx = w * 32 + lane;
        int s = idx / N, i = idx % N;
        // records: (x, y, z, letter | chain << 1) and the low parts, relative to the chain's centroid;
        // origin differences in two parts; the chain origins themselves
        float4* hi = reinterpret_cast<float4*>(smem);
        float4* lo = hi + N;
        float4* Dh = lo + N;
        float4* Dl = Dh + nc * nc;
        double* org = reinterpret_cast<double*>(Dl + nc * nc);
        // a monomer of the chain, taken whole: x - origin then loses nothing however far out the chain is
        for (int e = threadIdx.x; e < 3 * nc; e += 32 * W) {
            const int c = e / 3, o = d.chain_off[c], n = d.chain_off[c + 1] - o;
            org[e] = x64[3 * (o + n / 2) + (e - 3 * c)];
        }
        __syncthreads();
        auto split = [](double v, float* h, float* l) {
            *h = f64_to_f32(v);
            *l = f64_to_f32(v - f32_to_f64(*h));
        };
        float extent = 0.0f;   // the largest coordinate that a far pair's displacement is made of
        auto widen = [&](const float4& v) { extent = fmaxf(extent, fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fabsf(v.z))); };
        for (int j = threadIdx.x; j < N; j += 32 * W) {
            const int c = d.chain_of[j];
            float4 h, l;
            split(x64[3 * j] - org[3 * c], &h.x, &l.x);
            split(x64[3 * j + 1] - org[3 * c + 1], &h.y, &l.y);
            split(x64[3 * j + 2] - org[3 * c + 2], &h.z, &l.z);
            h.w = __int_as_float((int)d.seq[j] | (c << 1));
            l.w = 0.0f;
            widen(h);
            hi[j] = h;
            lo[j] = l;
        }
        for (int p = threadIdx.x; p < nc * nc; p += 32 * W) {
            const int a = p / nc, c = p % nc;
            float4 h = make_float4(0.f, 0.f, 0.f, 0.f), l = h;
            split(mimage64_short(d, org[3 * a] - org[3 * c]), &h.x, &l.x);
            split(mimage64_short(d, org[3 * a + 1] - org[3 * c + 1]), &h.y, &l.y);
            split(mimage64_short(d, org[3 * a + 2] - org[3 * c + 2]), &h.z, &l.z);
            widen(h);
            Dh[p] = h;
            Dl[p] = l;
        }
        SplitBox box;
        split(d.box_L, &box.Lh, &box.Ll);
        box.iL = d.iL32;
        box.edge = d.box_L > 0.0 ? 0.5f * box.Lh * (1.0f - 2e-5f) : INFINITY;
        float Ch[4], Cl[4];
        for (int q = 0; q < 4; ++q) split(d.C[q], &Ch[q], &Cl[q]);
        __syncthreads();
        DF in{0.0f, 0.0f}, ex{0.0f, 0.0f};   // far pairs within chains and between them
        float sizes = 0.0f, squares = 0.0f;  // sums of their sizes and squares
        int n_near = 0;
        NearPair* near = s_near[warp];
        auto drain = [&](int n) {   // the first n of the list
            __syncwarp();
            if (lane < n) part += pair_energy64(d, x64, near[lane].i, near[lane].j);
            __syncwarp();
        };
        for (int base = w * 32; base < total; base += 32 * W, idx += 32 * W) {
            bool is_near = false;
            int j = 0;
            if (idx < total) {
                j = i + s + 1;
                if (j >= N) j -= N;
                const float4 ah = hi[i], al = lo[i], bh = hi[j], bl = lo[j];
                const int ta = __float_as_int(ah.w), tb = __float_as_int(bh.w), ca = ta >> 1, cb = tb >> 1;
                const bool inter = ca != cb;
                if (inter || s > 0 || j != i + 1) {   // not a bonded pair
                    const float4 H = Dh[ca * nc + cb], Lo = Dl[ca * nc + cb];
                    bool unsure = false;
                    float lx, ly, lz, e1, e2;
                    const float dx = split_diff(ah.x, al.x, bh.x, bl.x, H.x, Lo.x, inter, box, &lx, &unsure);
                    const float dy = split_diff(ah.y, al.y, bh.y, bl.y, H.y, Lo.y, inter, box, &ly, &unsure);
                    const float dz = split_diff(ah.z, al.z, bh.z, bl.z, H.z, Lo.z, inter, box, &lz, &unsure);
                    const float xx = __fmul_rn(dx, dx), yy = __fmul_rn(dy, dy), zz = __fmul_rn(dz, dz);
                    const float q1 = two_sum(xx, yy, &e1), r2 = two_sum(q1, zz, &e2);
                    is_near = unsure || !(r2 > 16.0f && r2 < 1e24f);
                    if (!is_near) {
                        float l2 = __fadd_rn(e1, e2);
                        l2 = __fadd_rn(l2, __fmaf_rn(dx, dx, -xx));
                        l2 = __fadd_rn(l2, __fmaf_rn(dy, dy, -yy));
                        l2 = __fadd_rn(l2, __fmaf_rn(dz, dz, -zz));
                        l2 = __fmaf_rn(__fadd_rn(dx, dx), lx, l2);
                        l2 = __fmaf_rn(__fadd_rn(dy, dy), ly, l2);
                        l2 = __fmaf_rn(__fadd_rn(dz, dz), lz, l2);
                        // s = 1 / r^2 in two parts, s^3 (with 3 sh sl^2, which all pairs have the same sign of), and s^3 (s^3 - C)
                        const float sh = fast_rcp(r2);
                        const float er = __fmaf_rn(-l2, sh, __fmaf_rn(-r2, sh, 1.0f));
                        const float t = __fmul_rn(sh, er), sl = __fmaf_rn(t, er, t);
                        const float p = __fmul_rn(sh, sh);
                        const float pl = __fmaf_rn(__fmaf_rn(3.0f, sl, __fadd_rn(sh, sh)), sl, __fmaf_rn(sh, sh, -p));
                        const float c3 = __fmul_rn(p, sh);
                        const float c3l = __fmaf_rn(p, sl, __fmaf_rn(pl, sh, __fmaf_rn(p, sh, -c3)));
                        const int cc = j > i ? 2 * (ta & 1) + (tb & 1) : 2 * (tb & 1) + (ta & 1);   // the earlier monomer's letter first
                        const float C0 = cc == 0 ? Ch[0] : cc == 1 ? Ch[1] : cc == 2 ? Ch[2] : Ch[3];
                        const float C1 = cc == 0 ? Cl[0] : cc == 1 ? Cl[1] : cc == 2 ? Cl[2] : Cl[3];
                        float ue;
                        const float u = two_diff(c3, C0, &ue);
                        const float ul = __fadd_rn(ue, __fsub_rn(c3l, C1));
                        const float wh = __fmul_rn(c3, u);
                        const float wl = __fmaf_rn(c3, ul, __fmaf_rn(c3l, u, __fmaf_rn(c3, u, -wh)));
                        const DF v = df_add(inter ? ex : in, DF{wh, wl});
                        sizes += fabsf(wh);
                        squares = __fmaf_rn(wh, wh, squares);
                        if (inter) ex = v;
                        else in = v;
                    }
                }
            }
            const unsigned m = __ballot_sync(full, is_near);
            if (is_near) near[n_near + __popc(m & ((1u << lane) - 1u))] = NearPair{min(i, j), max(i, j)};
            n_near += __popc(m);
            if (n_near >= 32) {
                drain(32);
                n_near -= 32;
                NearPair keep{0, 0};
                if (lane < n_near) keep = near[32 + lane];
                __syncwarp();
                if (lane < n_near) near[lane] = keep;
            }
            s += dq;
            i += dt;
            if (i >= N) { i -= N; ++s; }
        }
        drain(n_near);
        // the far pairs' errors against the roundings of everything else (see kSplitCommon)
        float rest = fabsf(f64_to_f32(part));
#pragma unroll
        for (int m = 16; m > 0; m >>= 1) {
            sizes += __shfl_xor_sync(full, sizes, m);
            squares += __shfl_xor_sync(full, squares, m);
            rest += __shfl_xor_sync(full, rest, m);
            extent = fmaxf(extent, __shfl_xor_sync(full, extent, m));
        }
        if (lane == 0) s_size[warp] = make_float4(sizes, squares, extent, rest);
        __syncthreads();
        float4 size = s_size[0];
#pragma unroll
        for (int q = 1; q < W; ++q) {
            size.x += s_size[q].x;
            size.y += s_size[q].y;
            size.z = fmaxf(size.z, s_size[q].z);
            size.w += s_size[q].w;
        }
        const float k = fmaxf(fabsf(d.kin32), fabsf(d.kout32));
        const float far = k * (kSplitCommon * size.x + (kSplitPair + kSplitCoord * size.z) * sqrtf(size.y));
        if (!(size.w > 1e-12f && far <= size.w)) part = whole_energy64(d, x64, lane, w, W);
        else part += d.k_lj_intra * (f32_to_f64(in.hi) + f32_to_f64(in.lo)) + d.k_lj_inter * (f32_to_f64(ex.hi) + f32_to_f64(ex.lo));
    } else {
        part = add_pairs64(part, d, x64, w * 32 + lane, 32 * W);
    }
    for (int o = 16; o > 0; o >>= 1) part += __shfl_down_sync(full, part, o);
    out = __any_sync(full, out);
    if constexpr (W > 1) {
        if (lane == 0) red[warp] = part;
        out = __syncthreads_or(out);   // whatever the other terms are
        if (threadIdx.x == 0) {
            double E = 0.0;
            for (int q = 0; q < W; ++q) E += red[q];
            E_out[b] = out ? INFINITY : E;
        }
    } else {
        if (lane == 0) E_out[b] = out ? INFINITY : part;
    }
}

template <typename PT>
__global__ void __launch_bounds__(32 * kWarpsPerBlock)
delta_kernel(const SysDesc d, int B, const double* __restrict__ xyz, const phast_move* __restrict__ moves,
             double* __restrict__ dE_out, double* __restrict__ xyz_new, SlotLayout L) {
    extern __shared__ __align__(16) unsigned char smem[];
    Group<32> g;
    const int w = threadIdx.x >> 5;
    const int b = blockIdx.x * kWarpsPerBlock + w;
    if (b >= B) return;
    const double* x64 = xyz + (size_t)b * d.N * 3;
    Slot<PT> s(smem + (size_t)w * L.bytes, L);
    build_working<32, PT>(d, x64, s, g);
    const phast_move mv = moves[b];
    Proposal P;
    P.type = mv.type; P.chain = mv.chain; P.index = mv.index;
    P.angle = mv.angle; P.uz = P.uw = 0u; P.attempt = -1;
    P.axis = make_double3(mv.axis[0], mv.axis[1], mv.axis[2]);
    P.disp = make_double3(mv.disp[0], mv.disp[1], mv.disp[2]);
    P.angle32 = (float)P.angle;
    P.axis32 = make_float3((float)P.axis.x, (float)P.axis.y, (float)P.axis.z);
    P.disp32 = make_float3((float)P.disp.x, (float)P.disp.y, (float)P.disp.z);
    // a move outside the system (type, chain, interior index, amplitude) is
    // reported as NaN instead of being applied
    bool valid = P.type >= 0 && P.type < PHAST_N_MOVES && P.chain >= 0 && P.chain < d.n_chains;
    if (valid) {
        const int n = d.chain_off[P.chain + 1] - d.chain_off[P.chain];
        if (P.type == PHAST_PIVOT || P.type == PHAST_CRANK) valid = P.index >= 1 && P.index <= n - 2;
        if (P.type == PHAST_BOND) valid = P.index >= 0 && P.index <= n - 2 && isfinite(P.angle);
        else if (P.type == PHAST_CAP) valid = P.index >= 0 && P.index <= n - 1;
        if (P.type == PHAST_TRANS) valid = isfinite(P.disp.x) && isfinite(P.disp.y) && isfinite(P.disp.z);
        else if (P.type != PHAST_BOND) valid = valid && fabs(P.angle) <= PHAST_MAX_ANGLE;
        if (P.type == PHAST_PIVOT || P.type == PHAST_ROT || P.type == PHAST_CAP)
            valid = valid && isfinite(P.axis.x) && isfinite(P.axis.y) && isfinite(P.axis.z);
    }
    if (!valid) P.type = PHAST_TRANS, P.chain = 0, P.index = 0;
    const MoveSet M = move_set(d, P.type, P.chain, P.index);
    double dE = __longlong_as_double(0x7ff8000000000000ll);   // NaN for a degenerate or invalid move
    const bool ok = valid && make_new_positions<32, PT>(d, x64, P, M, s, g);
    const bool wall = ok && !container_ok<32, PT>(d, const_cast<double*>(x64), P, M, s, g, true, 0ull, 0ull, nullptr);
    if (wall) dE = INFINITY;   // beyond the container's wall
    if (ok && !wall) {
        double part;
        if constexpr (sizeof(PT) == 4) {
            float fene = 0.0f, tors = 0.0f;
            bool near = false, tnear = false;
            part = (double)local_delta32<32>(d, P, M, s, g, &fene, &near, &tors, &tnear);
            // a FENE bond near its divergence or a dihedral near degenerate: the exact
            // positions give that kind of term's change
            const bool fx = __ballot_sync(g.mask, near), tx = __ballot_sync(g.mask, tnear);
            if (fx || tx) {
                const double dX = local_delta_exact<32, true>(d, const_cast<double*>(x64), P, M, s, g, true, 0ull,
                                                              0ull, nullptr, fx, tx);
                part += g.lane == 0 ? dX : 0.0;
            }
            if (!fx) part += (double)fene;
            if (!tx) part += (double)tors;
            const DF q = d.box_L > 0.0 ? pair_delta32<32, 3, true>(d, M, P.chain, s, g)
                                       : pair_delta32<32, 3, false>(d, M, P.chain, s, g);
            part += (double)q.hi + (double)q.lo;
        } else {
            part = local_delta64<32>(d, P, M, s, g) + pair_delta64<32>(d, M, P.chain, s, g);
            bool inf = false;   // an infinite coordinate gives NaN to every pair it is in, as in FP32 mode
            for (int e = g.lane; M.hi - M.lo + 1 < d.N && e < 3 * d.N; e += 32)
                inf |= ((unsigned)__double2hiint(x64[e]) & 0x7fffffffu) == 0x7ff00000u && __double2loint(x64[e]) == 0;
            if (inf) part = __longlong_as_double(0x7ff8000000000000ll);
        }
        dE = g.sum(part);
    }
    if (g.lane == 0) dE_out[b] = dE;
    if (xyz_new) {
        if (sizeof(PT) == 4 && valid) prepare_exact<32, PT>(d, [&](int j) { return ld3(x64 + 3 * j); }, P, P.axis, s, g);
        double* out = xyz_new + (size_t)b * d.N * 3;
        for (int j = g.lane; j < d.N; j += 32) {
            double3 y = ld3(x64 + 3 * j);
            if (ok && j >= M.lo && j <= M.hi) y = exact_position(P, s.geo, y);
            out[3 * j + 0] = y.x;
            out[3 * j + 1] = y.y;
            out[3 * j + 2] = y.z;
        }
    }
}

}  // namespace

extern "C" int phast_energy(const phast_system* sys, const phast_ff* ff, int32_t B, const double* xyz,
                            int32_t pair_precision, double* E_out, void* stream) {
    SysDesc d;
    int rc = phast_build_desc(sys, ff, nullptr, &d, "phast_energy");
    if (rc) return rc;
    if (B < 0) return phast_set_error(PHAST_EINVAL, "phast_energy: B < 0");
    if (pair_precision != 32 && pair_precision != 64)
        return phast_set_error(PHAST_EINVAL, "phast_energy: pair_precision must be 32 or 64");
    if (B == 0) return PHAST_OK;
    if (!xyz || !E_out) return phast_set_error(PHAST_EINVAL, "phast_energy: NULL xyz or E_out");
    cudaStream_t st = (cudaStream_t)stream;
    dim3 grid((B + kWarpsPerBlock - 1) / kWarpsPerBlock), block(32 * kWarpsPerBlock);
    if (pair_precision == 64) {
        const size_t sm = sizeof(float4) * 2 * (size_t)(d.N + d.n_chains * d.n_chains) + sizeof(double) * 3 * d.n_chains;
        if (d.N >= kSplitMinN) energy64_kernel<kSplitWarps, true><<<B, 32 * kSplitWarps, sm, st>>>(d, B, xyz, E_out);
        else energy64_kernel<1, false><<<grid, block, 0, st>>>(d, B, xyz, E_out);
    } else {
        SlotLayout L = slot_layout<float>(d.N, d.n_chains, d.max_chain);
        size_t sm = (size_t)L.bytes * kWarpsPerBlock;
        PHAST_CUDA_TRY(cudaFuncSetAttribute(energy32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
        energy32_kernel<<<grid, block, sm, st>>>(d, B, xyz, E_out, L);
    }
    PHAST_CUDA_TRY(cudaGetLastError());
    return PHAST_OK;
}

extern "C" int phast_delta_energy(const phast_system* sys, const phast_ff* ff, int32_t B, const double* xyz,
                                  const phast_move* moves, int32_t pair_precision, double* dE_out,
                                  double* xyz_new_out, void* stream) {
    SysDesc d;
    int rc = phast_build_desc(sys, ff, nullptr, &d, "phast_delta_energy");
    if (rc) return rc;
    if (B < 0) return phast_set_error(PHAST_EINVAL, "phast_delta_energy: B < 0");
    if (pair_precision != 32 && pair_precision != 64)
        return phast_set_error(PHAST_EINVAL, "phast_delta_energy: pair_precision must be 32 or 64");
    if (B == 0) return PHAST_OK;
    if (!xyz || !moves || !dE_out) return phast_set_error(PHAST_EINVAL, "phast_delta_energy: NULL argument");
    cudaStream_t st = (cudaStream_t)stream;
    dim3 grid((B + kWarpsPerBlock - 1) / kWarpsPerBlock), block(32 * kWarpsPerBlock);
    if (pair_precision == 64) {
        SlotLayout L = slot_layout<double>(d.N, d.n_chains, d.max_chain);
        size_t sm = (size_t)L.bytes * kWarpsPerBlock;
        PHAST_CUDA_TRY(cudaFuncSetAttribute(delta_kernel<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
        delta_kernel<double><<<grid, block, sm, st>>>(d, B, xyz, moves, dE_out, xyz_new_out, L);
    } else {
        SlotLayout L = slot_layout<float>(d.N, d.n_chains, d.max_chain);
        size_t sm = (size_t)L.bytes * kWarpsPerBlock;
        PHAST_CUDA_TRY(cudaFuncSetAttribute(delta_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
        delta_kernel<float><<<grid, block, sm, st>>>(d, B, xyz, moves, dE_out, xyz_new_out, L);
    }
    PHAST_CUDA_TRY(cudaGetLastError());
    return PHAST_OK;
}
