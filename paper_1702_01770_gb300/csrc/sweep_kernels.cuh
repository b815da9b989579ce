// sweep_kernels.cuh -- the batched sweep kernels (a group of lanes or one lane per walker),
// as templates; the sweep_*.cu files instantiate them, one family each, so that they compile
// side by side.
#pragma once

#include "group.cuh"

// ---------------------------------------------------------------------------
// Launch arguments (by value).
// ---------------------------------------------------------------------------
struct SweepArgs {
    const SysDesc* descs;
    int n_sys, n_jk, wpc, n_tiles;
    int64_t n_sweeps;
    int order[PHAST_MAX_SYSTEMS];
    int tile_start[PHAST_MAX_SYSTEMS + 1];
    int tiles[PHAST_MAX_SYSTEMS];        // tiles of each system, by enumeration position
    int64_t hs_off[PHAST_MAX_SYSTEMS];   // hist_sum offset of each system id
    double* xyz;
    double* E;
    int32_t* bin;
    uint64_t* t;
    const uint64_t* seed;
    phast_walker_stats* stats;
    const double* lnW;
    unsigned long long* hist_sum;
    uint32_t* hist_walker;
    phast_trace* trace;
    int trace_walkers;
    int32_t* tile_counter;
    double* scratch;
    int scratch_stride;                   // doubles per walker in scratch
    SlotLayout L;
    LaneLayout LL;                        // per-warp layout of the one-walker-per-thread form
    int hist_bins;                        // shared histogram capacity (max n_bins)
    uint32_t hist_flush;                  // a shared bin reaching this count moves it into hist_sum
    int hist_flush_on;                    // a tile's counts can reach hist_flush in this launch
};

typedef void (*batched_fn)(const SweepArgs);

// Kernels of a group of tpw lanes per walker (null: no such width); lean: the 64-register
// build of the 16-lane FP32 tiles.
batched_fn pick_f32_lean(int tpw, bool lean);     // FP32, no geometry
batched_fn pick_f32_exact(int tpw, bool lean);    // and the exact path of the torsion terms
batched_fn pick_f32_geom(int tpw, bool lean);     // the paper's geometry
// A warp per walker for tiles of tpw lanes, the sums in those lanes' order (the same results);
// lean: the 64-register build.
batched_fn pick_f32_lean_wide(int tpw, bool lean);
batched_fn pick_f32_exact_wide(int tpw, bool lean);
batched_fn pick_f32_geom_wide(int tpw, bool lean);
batched_fn pick_f64(int tpw, bool geom);
batched_fn pick_lane(bool fp32, bool geom, bool shared_trials);   // one walker per thread

// Moves from move index t to the next multiple of period (0: none), at most 2^30.
__device__ __forceinline__ uint32_t moves_to_period(uint64_t t, uint64_t period) {
    const uint64_t n = period ? period - t % period : 1ull << 30;
    return (uint32_t)(n < (1ull << 30) ? n : 1ull << 30);
}

#ifdef PHAST_SWEEP_KERNELS
#include "lane.cuh"   // the one-walker-per-thread form (uses SweepArgs)
#endif

constexpr int kMaxTileThreads = 512;
constexpr int kLaneMaxThreads = 256;               // one walker per thread
constexpr uint32_t kHistFlushDefault = 1u << 31;   // shared histogram bins stay below 2^31 + wpc

namespace {

__device__ __forceinline__ void copy_desc(SysDesc* dst, const SysDesc* src) {
    const int4* s = reinterpret_cast<const int4*>(src);
    int4* d = reinterpret_cast<int4*>(dst);
    for (int i = threadIdx.x; i < (int)(sizeof(SysDesc) / 16); i += blockDim.x) d[i] = s[i];
}

// Jackknife block of walker w of a type with W walkers split into n blocks
// [b W / n, (b+1) W / n).
__host__ __device__ __forceinline__ int jk_block(int w, int W, int n) {
    return (int)(((int64_t)(w + 1) * n - 1) / W);
}

#ifdef PHAST_SWEEP_KERNELS
// ---------------------------------------------------------------------------
// Batched form.
// ---------------------------------------------------------------------------

// The FP64 full energy replaces the running one (when in range) and the
// working copy is rebuilt.
template <int TPW, typename PT, int ORD = TPW>
__device__ __forceinline__ void recompute_energy(const SysDesc& sd, const double* x64, const double* lnW, Slot<PT>& slot,
                                              const Group<TPW>& g, phast_walker_stats* ls, double& E, int& bin,
                                              double& lnw_here, float& erel) {
    const double Ef = full_energy64<TPW, ORD>(sd, x64, g);
    if (g.lane == 0) {
        ls->drift_max = fmax(ls->drift_max, fabs(E - Ef));
        ls->recomputes++;
    }
    // the running energy always takes the FP64 value (the drift is removed); a
    // value outside the bins (an FP32 rounding let the walker step just past a
    // range edge) counts in the nearest edge bin until a move brings it back
    if (isfinite(Ef)) {
        const int bf = bin_of(sd, Ef);
        E = Ef;
        erel = (float)(E - sd.e_min);
        bin = bf >= 0 ? bf : (Ef < sd.e_min ? 0 : sd.n_bins - 1);
        lnw_here = __ldg(lnW + bin);
        if (bf < 0 && g.lane == 0) ls->recompute_outside++;
    }
    g.sync();
    build_working<TPW, PT>(sd, x64, slot, g);
}
// GEOM: the system types use the paper's own geometry (FENE bonds, container,
// bond-length or cap moves); without it those branches are compiled out, which
// keeps the per-move loop short in the instruction cache.
// EXACT: FP32 local terms near their hard edges are taken in FP64 on the exact positions
// (an out-of-line path); always so with GEOM, and for types that start straight.
// ORD: the lanes per walker whose order of summation every sum takes (the tile's; the group may
// be wider): the walker's results do not depend on how many others share the context.
template <int TPW, typename PT, bool GEOM, bool EXACT, int ORD = TPW>
__device__ void run_walker(const SysDesc& sd, const SweepArgs& a, int s_id, int w_local, Slot<PT>& slot,
                           uint32_t* hist, unsigned long long* const* hist_tile, unsigned long long* hist_g,
                           const Group<TPW>& g) {
    // hist: the tile's shared histogram, whose bins move into *hist_tile (the global
    // sums of the tile's jackknife block, or null; kept in shared memory, read only
    // when a bin reaches a multiple of a.hist_flush); hist_g (non-null): this
    // walker's jackknife block differs from the tile's, so its visits go straight to
    // the global sums
    const int gw = sd.walker_off + w_local;
    double* x64 = a.xyz + sd.xyz_off + (int64_t)w_local * sd.N * 3;
    const double* lnW = a.lnW + sd.lnw_off;
    double E = a.E[gw];
    int bin = a.bin[gw];
    uint64_t t = a.t[gw];
    const uint64_t seed = a.seed[gw];
    phast_walker_stats* ls = slot.st;   // counters of this launch, in shared memory
    if (g.lane == 0) memset(ls, 0, sizeof(*ls));
    uint32_t* hw = a.hist_walker ? a.hist_walker + sd.hw_off + (int64_t)w_local * sd.n_bins : nullptr;
    const bool tracing = a.trace && s_id == 0 && w_local < a.trace_walkers;
    const int64_t n_moves = a.n_sweeps * sd.N;
    const uint64_t period = (uint64_t)sd.recompute_every * (uint64_t)sd.N;

    const uint64_t t_end = t + (uint64_t)n_moves;
    // moves until the next look at the recompute period, in one register (a 64-bit
    // remainder each move costs about a hundred instructions)
    uint32_t left = moves_to_period(t, period);

    build_working<TPW, PT>(sd, x64, slot, g);
    int queued = 0;                                         // accepted moves awaiting their FP64 replay
    const int qcap = ORD < kQueue ? ORD : kQueue;
    // Every lane holds the walker's scalar state and takes the same decision
    // from the same broadcast values; lane 0 alone writes histograms and counters.
    double lnw_here = __ldg(lnW + bin);
    float erel = (float)(E - sd.e_min);                     // FP32 image of E - e_min (FP32 mode)
    constexpr bool OUT = TPW < 32 || EXACT;                 // the Philox rounds out of line
    uint4 blk = stream_block<OUT>(seed, t, (uint32_t)g.lane);   // this lane's block of the current move
    while (t != t_end) {
        const Proposal P = propose_group<TPW, PT, GEOM, EXACT, ORD>(sd, seed, t, blk, g);
        if constexpr (!GEOM) __builtin_assume(P.type >= 0 && P.type < PHAST_BOND);   // no bond or cap moves
        const MoveSet M = move_set(sd, P.type, P.chain, P.index);
        double jac = 1.0;   // Hastings factor (bond-length moves)
        const bool ok = make_new_positions<TPW, PT, GEOM, ORD>(sd, x64, P, M, slot, g, &jac);
        // a trial position beyond the container's wall: infinite energy, not evaluated
        bool wall = false;
        if constexpr (GEOM)
            wall = ok && sd.has_sphere &&
                   !container_ok<TPW, PT>(sd, x64, P, M, slot, g, sizeof(PT) == 8, seed, t, sizeof(PT) == 4 ? &queued : nullptr);
        const bool eval = ok && !wall;
        DF dE32{0.0f, 0.0f};
        double dE64 = 0.0;
        if constexpr (sizeof(PT) == 4) {   // this lane's share in double-float, the group total on every lane
            DF part{0.0f, 0.0f};
            if (eval) {
                part = sd.box_L > 0.0 ? pair_delta32<TPW, 3, true, ORD>(sd, M, P.chain, slot, g)
                                      : pair_delta32<TPW, 3, false, ORD>(sd, M, P.chain, slot, g);
                float fene = 0.0f, tors = 0.0f;
                bool near = false, tnear = false;
                part = df_add(part, DF{local_delta32<TPW, GEOM, EXACT, ORD>(sd, P, M, slot, g, GEOM ? &fene : nullptr,
                                                                       &near, &tors, &tnear), 0.0f});
                if constexpr (EXACT) {
                    // a FENE bond near its divergence or a dihedral near degenerate: the
                    // exact positions give that kind of term's change
                    const bool fx = GEOM && (__ballot_sync(g.mask, near) & g.mask);
                    const bool tx = __ballot_sync(g.mask, tnear) & g.mask;
                    if (fx || tx) {
                        const double dX = local_delta_exact<TPW, GEOM, ORD>(sd, x64, P, M, slot, g, false, seed, t,
                                                                            &queued, fx, tx);
                        if (g.lane == 0) part = df_add(part, df_of(dX));
                    }
                    if (GEOM && !fx) part = df_add(part, DF{fene, 0.0f});
                    if (!tx) part = df_add(part, DF{tors, 0.0f});
                } else {
                    // this build keeps the exact path (an out-of-line call) out of its move
                    // loop: a dihedral whose normals lie below FP32 resolution counts 0, the
                    // FP64 value of collinear bonds (in continuous sampling a dihedral that
                    // is near degenerate without being degenerate has probability ~1e-9, and
                    // the host runs contexts whose chains start straight in the general build)
                    part = df_add(part, DF{tors, 0.0f});
                }
            }
            dE32 = group_sum_df<TPW, ORD>(part, g);
        } else {
            double part = 0.0;
            if (eval) part = local_delta64<TPW, GEOM>(sd, P, M, slot, g) + pair_delta64<TPW>(sd, M, P.chain, slot, g);
            dE64 = g.sum(part);
        }
        const bool finite = eval && (sizeof(PT) == 4 ? (isfinite(dE32.hi) && isfinite(dE32.lo)) : isfinite(dE64));
        int b_new = -1;
        if (finite) b_new = sizeof(PT) == 4 ? bin_after(sd, E, erel, dE32) : bin_of_short(sd, E + dE64);
        const double lnw_new = __ldg(lnW + (b_new >= 0 ? b_new : bin));
        blk = stream_block<OUT>(seed, t + 1, (uint32_t)g.lane);   // next move's block, while the load is in flight
        bool acc = false;
        if (b_new >= 0) {
            const double dl = lnw_new - lnw_here;
            if (GEOM && P.type == PHAST_BOND) acc = accept_stretch(dl, jac, P);
            else acc = accept_weight(dl, P);
        }
        if (acc) {
            E = E + (sizeof(PT) == 4 ? (double)dE32.hi + (double)dE32.lo : dE64);
            bin = b_new;
            lnw_here = lnw_new;
            if constexpr (sizeof(PT) == 4) erel = (float)(E - sd.e_min);
        }
        if (g.lane == 0) {   // histogram and bookkeeping on one lane
            if (hist_g) {
                atomicAdd(hist_g + bin, 1ull);
            } else if (!a.hist_flush_on) {   // the tile cannot count to the flush count in this launch
                atomicAdd(hist + bin, 1u);
            } else if (((atomicAdd(hist + bin, 1u) + 1u) & (a.hist_flush - 1u)) == 0u && *hist_tile) {
                // this increment took the bin to a multiple of the flush count (a power
                // of two): move that many into the 64-bit sums.  Each multiple is crossed
                // by one increment, so the bin stays below the flush count plus the
                // walkers of the tile.
                atomicSub(hist + bin, a.hist_flush);
                atomicAdd(*hist_tile + bin, (unsigned long long)a.hist_flush);
            }
            if (hw) atomicAdd(hw + bin, 1u);
            ls->attempts[P.type]++;
            ls->accepts[P.type] += acc;
            ls->pair_evals += move_pair_evals(sd, P.type, M);
            ls->pair_evals_inter += move_pair_evals_inter(sd, P.type, P.chain, M);
            if (tracing) {
                phast_trace tr;
                // an infinite FP32 term leaves NaN in the double-float's low word: report hi alone
                tr.dE = !ok ? __longlong_as_double(0x7ff8000000000000ll)
                      : wall ? INFINITY
                             : (sizeof(PT) == 4 ? (isinf(dE32.hi) ? (double)dE32.hi : (double)dE32.hi + (double)dE32.lo)
                                                : dE64);
                tr.bin_after = bin;
                tr.accepted = (int32_t)acc;
                a.trace[(int64_t)(w_local + 1) * n_moves - (int64_t)(t_end - t)] = tr;
            }
        }
        if (acc) {
            if constexpr (sizeof(PT) == 4) {
                accept_move32<TPW>(sd, P, t, M, slot, g, queued);
                if (++queued == qcap) {
                    flush_queue<TPW, GEOM>(sd, x64, seed, slot, g, queued);
                    queued = 0;
                }
            } else {
                commit_move64<TPW>(x64, M, slot, g);
            }
        }
        g.sync();
        ++t;
        if (--left == 0) {
            if (period && (t % period) == 0) {   // FP64 full energy kills the drift of the running sum
                if constexpr (sizeof(PT) == 4) {
                    flush_queue<TPW, GEOM>(sd, x64, seed, slot, g, queued);
                    queued = 0;
                }
                recompute_energy<TPW, PT, ORD>(sd, x64, lnW, slot, g, ls, E, bin, lnw_here, erel);
            }
            left = moves_to_period(t, period);
        }
    }
    if constexpr (sizeof(PT) == 4) flush_queue<TPW, GEOM>(sd, x64, seed, slot, g, queued);
    if (g.lane == 0) {
        a.E[gw] = E;
        a.bin[gw] = bin;
        a.t[gw] = t;
        phast_walker_stats* st = a.stats + gw;
        for (int i = 0; i < PHAST_N_MOVES; ++i) { st->attempts[i] += ls->attempts[i]; st->accepts[i] += ls->accepts[i]; }
        st->pair_evals += ls->pair_evals;
        st->pair_evals_inter += ls->pair_evals_inter;
        st->recomputes += ls->recomputes;
        st->recompute_outside += ls->recompute_outside;
        st->drift_max = fmax(st->drift_max, ls->drift_max);
    }
}


// MINB: CTAs of kMaxTileThreads per SM the registers must allow.  Small systems
// run a build held to 64 registers (MINB = 2): their moves are short and
// latency-bound, and twice the warps per SM hide more of it than the spills cost.
template <int TPW, typename PT, bool GEOM, bool EXACT = true, int MINB = 1, int ORD = TPW>
__global__ void __launch_bounds__(kMaxTileThreads, MINB)
sweep_batched_kernel(const SweepArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_tile;
    __shared__ unsigned long long* s_hs_tile;   // the global sums of the tile's jackknife block
    SysDesc& sd = *reinterpret_cast<SysDesc*>(smem);
    uint32_t* hist = reinterpret_cast<uint32_t*>(smem + sizeof(SysDesc));
    unsigned char* slots = smem + sizeof(SysDesc) + align16(4 * a.hist_bins);
    const Group<TPW> g;
    const int slot_id = threadIdx.x / TPW;
    Slot<PT> slot(slots + (size_t)slot_id * a.L.bytes, a.L);

    for (;;) {
        if (threadIdx.x == 0) s_tile = atomicAdd(a.tile_counter, 1);
        __syncthreads();
        const int tile = s_tile;
        if (tile >= a.n_tiles) break;
        int pos = 0;
        while (pos + 1 < a.n_sys && tile >= a.tile_start[pos + 1]) ++pos;
        const int s_id = a.order[pos];
        copy_desc(&sd, a.descs + s_id);
        __syncthreads();
        for (int k = threadIdx.x; k < sd.n_bins; k += blockDim.x) hist[k] = 0u;
        // tile k of this system: walkers [k W / nt, (k + 1) W / nt), at most wpc of them;
        // the shared histogram collects the jackknife block of the first one
        const int k = tile - a.tile_start[pos], nt = a.tiles[pos];
        const int W = sd.n_walkers;
        const int w_a = (int)((int64_t)k * W / nt), w_b = (int)((int64_t)(k + 1) * W / nt);
        const int w_local = w_a + slot_id;
        const int blk = jk_block(w_a, W, a.n_jk);
        __syncthreads();
        if (threadIdx.x == 0) s_hs_tile = a.hist_sum ? a.hist_sum + a.hs_off[s_id] + (int64_t)blk * sd.n_bins : nullptr;
        __syncthreads();
        if (w_local < w_b) {
            const int mine = jk_block(w_local, W, a.n_jk);
            unsigned long long* hg =
                (a.hist_sum && mine != blk) ? a.hist_sum + a.hs_off[s_id] + (int64_t)mine * sd.n_bins : nullptr;
            run_walker<TPW, PT, GEOM, EXACT, ORD>(sd, a, s_id, w_local, slot, hist, &s_hs_tile, hg, g);
        }
        __syncthreads();
        unsigned long long* hs_tile = s_hs_tile;
        if (hs_tile) {
            for (int k = threadIdx.x; k < sd.n_bins; k += blockDim.x)
                if (hist[k]) atomicAdd(hs_tile + k, (unsigned long long)hist[k]);
        }
        __syncthreads();
    }
}

// One walker per thread (small systems): the same persistent tiles, a tile being
// at most the CTA's blockDim.x walkers, spread evenly over its warps, each warp's walkers in
// one lane-interleaved shared-memory slot.

template <typename PT, bool GEOM, bool SH>
__global__ void __launch_bounds__(kLaneMaxThreads)
sweep_lane_kernel(const SweepArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_tile;
    SysDesc& sd = *reinterpret_cast<SysDesc*>(smem);
    uint32_t* hist = reinterpret_cast<uint32_t*>(smem + sizeof(SysDesc));
    unsigned char* warps = smem + sizeof(SysDesc) + align16(4 * a.hist_bins);
    const LaneSlot<PT, SH> slot(warps + (size_t)(threadIdx.x >> 5) * a.LL.bytes, a.LL, threadIdx.x & 31);
    for (;;) {
        if (threadIdx.x == 0) s_tile = atomicAdd(a.tile_counter, 1);
        __syncthreads();
        const int tile = s_tile;
        if (tile >= a.n_tiles) break;
        int pos = 0;
        while (pos + 1 < a.n_sys && tile >= a.tile_start[pos + 1]) ++pos;
        const int s_id = a.order[pos];
        copy_desc(&sd, a.descs + s_id);
        __syncthreads();
        for (int k = threadIdx.x; k < sd.n_bins; k += blockDim.x) hist[k] = 0u;
        const int k = tile - a.tile_start[pos], nt = a.tiles[pos];
        const int W = sd.n_walkers;
        const int w_a = (int)((int64_t)k * W / nt), w_b = (int)((int64_t)(k + 1) * W / nt);
        const int n_warps = blockDim.x >> 5, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        const int per = (w_b - w_a + n_warps - 1) / n_warps;
        const int w_local = lane < per ? w_a + warp * per + lane : w_b;
        const int blk = jk_block(w_a, W, a.n_jk);
        __syncthreads();
        unsigned long long* hs_tile = a.hist_sum ? a.hist_sum + a.hs_off[s_id] + (int64_t)blk * sd.n_bins : nullptr;
        if (w_local < w_b) {
            const int mine = jk_block(w_local, W, a.n_jk);
            unsigned long long* hg =
                (a.hist_sum && mine != blk) ? a.hist_sum + a.hs_off[s_id] + (int64_t)mine * sd.n_bins : nullptr;
            run_walker_lane<PT, GEOM, SH>(sd, a, s_id, w_local, slot, hist, hs_tile, hg);
        }
        __syncthreads();
        if (hs_tile) {
            for (int k = threadIdx.x; k < sd.n_bins; k += blockDim.x)
                if (hist[k]) atomicAdd(hs_tile + k, (unsigned long long)hist[k]);
        }
        __syncthreads();
    }
}


template <bool G, bool X>
batched_fn pick_batched32(int tpw, bool lean) {
    switch (tpw) {
        case 4: return sweep_batched_kernel<4, float, G, X>;
        case 8: return sweep_batched_kernel<8, float, G, X>;
        case 16: return lean ? sweep_batched_kernel<16, float, G, X, 2> : sweep_batched_kernel<16, float, G, X>;
        case 32: return sweep_batched_kernel<32, float, G, X>;
        default: return nullptr;
    }
}

template <bool G, bool X>
batched_fn pick_batched32_wide(int tpw, bool lean) {
    if (tpw == 16) return lean ? sweep_batched_kernel<32, float, G, X, 2, 16> : sweep_batched_kernel<32, float, G, X, 1, 16>;
    return tpw == 8 && !lean ? sweep_batched_kernel<32, float, G, X, 1, 8> : (batched_fn) nullptr;
}

template <bool G>
batched_fn pick_batched64(int tpw) {
    switch (tpw) {
        case 4: return sweep_batched_kernel<4, double, G>;
        case 8: return sweep_batched_kernel<8, double, G>;
        case 16: return sweep_batched_kernel<16, double, G>;
        case 32: return sweep_batched_kernel<32, double, G>;
        default: return nullptr;
    }
}
#endif

}  // namespace
