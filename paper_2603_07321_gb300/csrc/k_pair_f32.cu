// Mixed-precision pair kernels on Verlet lists: Sutton-Chen EAM density and
// forces in FP32.  What a neighbour reads is one 16-byte record, its position
// in fixed point (see the record format), so that r_j - r_i is an exact
// integer difference converted once.
//
// Pass 1 (density): rho_i = sum_j phi_m(r_ij), then B'(rho_i) =
// -eps c / (2 sqrt(rho_i)), stored beside the record scaled by m a^m (the
// force pass's pair terms are arranged around that weight), and the atom's
// pair energy.  Eq. (pe).
// Pass 2 (force):   F_i = sum_j [eps phi_n'(r) + (B'_i + B'_j) phi_m'(r)] (r_j - r_i)/r,
// Eq. (f_int), and the velocity-Verlet update fused behind it
// (atom_update_mixed).  Grip atoms keep v = 0 and F = 0 in the update; their
// internal force still enters the reaction R = -sum_{right grip} F . e of
// Eq. (state_variables).
#include "k_mixed.cuh"

namespace pta {

// f(record) for the entries lane l of atom u reads, in list order: a quad per
// iteration (four gathers in flight), the next quad read ahead, then what is
// left of the last one
template <bool RES, class F>
__device__ __forceinline__ void for_entries(const SpecDev &S, const void *rec, int u, int l, int L,
                                            F f) {
    const uint4 *p = S.plist + nl_col(u, l, L, S.capq);
    const int cnt = chk_count(S, S.pnn[u * L + l], 4 * (S.capq - 1));
    uint4 e = ld_quad<RES>(p);
    for (int t = cnt >> 2; t > 0; --t) {
        p += 32;
        const uint4 nx = ld_quad<RES>(p);
        const int4 x0 = ld_rec<RES>(S, rec, e.x), x1 = ld_rec<RES>(S, rec, e.y);
        const int4 x2 = ld_rec<RES>(S, rec, e.z), x3 = ld_rec<RES>(S, rec, e.w);
        f(x0);
        f(x1);
        f(x2);
        f(x3);
        e = nx;
    }
    const int left = cnt & 3;
    if (left) {
        int4 x0 = ld_rec<RES>(S, rec, e.x), x1 = x0, x2 = x0;
        if (left > 1) x1 = ld_rec<RES>(S, rec, e.y);
        if (left > 2) x2 = ld_rec<RES>(S, rec, e.z);
        f(x0);
        if (left > 1) f(x1);
        if (left > 2) f(x2);
    }
}

// the same in a resident run, from the list in shared memory: twelve gathers
// in flight (a barrier has emptied L1, so they come from L2; at 16 lanes per
// atom that is the whole list in one round)
template <class F>
__device__ __forceinline__ void for_entries(const SpecDev &S, const void *rec, const LaneList &q,
                                            F f) {
    for (int t = 0, left = q.cnt; left > 0; left -= 12, t += 3) {
        int4 x[12];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            if (left <= 4 * k) break;
            const uint4 e = q.quad(t + k);
            x[4 * k] = ld_rec<true>(S, rec, e.x);
            if (left > 4 * k + 1) x[4 * k + 1] = ld_rec<true>(S, rec, e.y);
            if (left > 4 * k + 2) x[4 * k + 2] = ld_rec<true>(S, rec, e.z);
            if (left > 4 * k + 3) x[4 * k + 3] = ld_rec<true>(S, rec, e.w);
        }
#pragma unroll
        for (int k = 0; k < 12; ++k) {
            if (left <= k) break;
            f(x[k]);
        }
    }
}

// the density weight w of atom u from its lanes' sums, stored in its record;
// its energy
template <bool SC76>
__device__ __forceinline__ float density_end(const SpecDev &S, const PotF &P, int L, int u,
                                             bool first, const int4 &ra, RhoSums s, float &w) {
    s.sm = lane_sum(s.sm, L);
    s.sn = lane_sum(s.sn, L);
    s.sr = lane_sum(s.sr, L);
    const float cnt = (float)lane_sum(s.cnt, L);
    const float dr = fmaf(-cnt, P.rc, s.sr);  // sum of r - rc
    const float rho = SC76 ? fmaf(P.am, s.sm, fmaf(P.Bm, dr, __fmul_rn(-cnt, P.Am))) : s.sm;
    const float phn = fmaf(P.an, s.sn, fmaf(P.Bn, dr, __fmul_rn(-cnt, P.An)));
    // w = m a^m B'(rho), B'(rho) = -eps c / (2 sqrt(rho))
    const float rq = rho > 0.f ? rsqrtf(rho) : 0.f;
    w = __fmul_rn(P.fpsc, rq);
    if (first) ((int4 *)S.posfp)[u] = make_int4(ra.x, ra.y, ra.z, __float_as_int(w));
    // the atom's energy 1/2 eps sum_j phi_n + B(rho), B = -eps c sqrt(rho)
    return fmaf(-P.ec, rho > 0.f ? __fmul_rn(rho, rq) : 0.f, __fmul_rn(0.5f * P.eps, phn));
}

// sums of (eV/A^2) x quanta over an atom's lanes, in eV/A
__device__ __forceinline__ void force_end(const SpecDev &S, int L, float f[3]) {
#pragma unroll
    for (int d = 0; d < 3; ++d) f[d] = __fmul_rn(lane_sum(f[d], L), S.f_q);
}

// the passes of one thread (lane l of atom u) with everything in memory
template <bool SC76, bool RES>
__device__ __forceinline__ void density_lane(const SpecDev &S, const PotF &P, int L, int u, int l,
                                             int par) {
    const bool valid = u < S.n;
    RhoSums s;
    int4 ra = make_int4(0, 0, 0, 0);
    if (valid) {
        ra = S.rec[par][u];
        const float q2 = S.f_q2;
        for_entries<RES>(S, S.rec[par], u, l, L,
                         [&](const int4 &x) { rho_pair<SC76>(P, q2, ra, x, s); });
    }
    float w;
    const float pe = density_end<SC76>(S, P, L, u, valid && l == 0, ra, s, w);
    if (valid && l == 0) ((float *)S.pen)[u] = pe;
}

// the force on atom u, in all its lanes
template <bool SC76, bool RES>
__device__ __forceinline__ void force_lane(const SpecDev &S, const PotF &P, int L, int u, int l,
                                           float f[3]) {
    f[0] = f[1] = f[2] = 0.f;
    if (u < S.n) {
        const int4 ra = ((const int4 *)S.posfp)[u];
        const float wa = __int_as_float(ra.w);
        const float q2 = S.f_q2;
        for_entries<RES>(S, S.posfp, u, l, L, [&](const int4 &x) {
            force_pair<SC76>(P, q2, ra, wa, x, f[0], f[1], f[2]);
        });
    }
    force_end(S, L, f);
}
// the update of atom u by one thread, with its state in memory
__device__ __forceinline__ void update_atom(const SpecDev &S, int u, const float f[3], int par,
                                            int mode, int phase, long long done, long long nsteps,
                                            StepVals &v) {
    AtomMixed A;
    A.load(S, par, u);
    atom_update_mixed(S, A, par, u, f, ((const float *)S.pen)[u], mode, phase, done, nsteps, v);
    if (mode != MODE_EVAL) A.store(S, par ^ 1, u);
}

// the launched passes; LT: the lanes per atom of every specimen of the launch,
// or 0
template <int LT, bool SC76>
__global__ void __launch_bounds__(TPB, 8) k_density_f32(const SpecDev *__restrict__ specs,
                                                        const int *__restrict__ b2s, int force,
                                                        const PotF P) {
    const SpecDev &S = specs[b2s[blockIdx.x]];
    if (!force && S.ctl->phase == PH_IDLE) return;
    const int L = LT ? LT : S.L;
    const int u = (blockIdx.x - S.blk_pair0) * (TPB / L) + threadIdx.x / L;
    density_lane<SC76, false>(S, P, L, u, threadIdx.x % L, S.ctl->parity);
}

template <int LT, bool SC76>
__global__ void __launch_bounds__(TPB, 8) k_force_f32(const SpecDev *__restrict__ specs,
                                                      const int *__restrict__ b2s, int mode,
                                                      const PotF P) {
    const SpecDev &S = specs[b2s[blockIdx.x]];
    const SpecCtl *ctl = S.ctl;
    const int phase = ctl->phase;
    if (mode == MODE_STEP && phase == PH_IDLE) return;
    const int par = ctl->parity, lb = blockIdx.x - S.blk_pair0;
    const long long done = ctl->done, nsteps = ctl->nsteps;
    const int L = LT ? LT : S.L, APB = TPB / L;
    float f[3];
    force_lane<SC76, false>(S, P, L, lb * APB + threadIdx.x / L, threadIdx.x % L, f);
    if (L > 1) {
        // the block's atoms to its first threads, so that whole warps update
        // them and not one lane in L of every warp
        __shared__ float sf[3][TPB / (LT ? LT : 2)];
        if (threadIdx.x % L == 0)
#pragma unroll
            for (int d = 0; d < 3; ++d) sf[d][threadIdx.x / L] = f[d];
        __syncthreads();
        if (threadIdx.x < APB)
#pragma unroll
            for (int d = 0; d < 3; ++d) f[d] = sf[d][threadIdx.x];
    }
    const int u = lb * APB + threadIdx.x;
    StepVals v = StepVals{};
    if (threadIdx.x < APB && u < S.n) update_atom(S, u, f, par, mode, phase, done, nsteps, v);
    block_partial<TPB>(S, lb, v, L);
}

// a resident run's warp; LT: the lanes per atom of every specimen, or 0.  Known,
// they leave the sums over lanes without loops: 10.0
// us (loops 10.7) per step of a specimen of 4,000 atoms at 16 lanes
template <bool SC76, int LT>
struct OpsF32 {
    const PotF &P;
    uint4 *cache;
    int quads;
    AtomMixed A;
    LaneList q;
    int4 ra;         // the atom's record (all its lanes)
    float wa, pe;    // its density weight and energy
    int lanes, u, l;
    bool valid;
    __device__ __forceinline__ void load(const SpecDev &S, int tile, int par) {
        const int t = tile * 32 + (threadIdx.x & 31);
        lanes = S.L;
        const int L = LT ? LT : lanes;
        u = t / L;
        l = t % L;
        valid = u < S.n;
        ra = make_int4(0, 0, 0, 0);
        wa = pe = 0.f;
        if (valid) {
            q.fill(S, cache, u, l, L, quads);
            ra = S.rec[par][u];
            if (l == 0) A.load(S, par, u);
        }
    }
    __device__ __forceinline__ void prune(const SpecDev &S, int par) {
        if (!valid) return;
        const int L = LT ? LT : lanes;
        prune_lane<true>(S, u, l, L, par);
        q.fill(S, cache, u, l, L, quads);
        A.pref = ra;
    }
    __device__ __forceinline__ void store(const SpecDev &S, int par) const {
        if (valid && l == 0) A.store(S, par, u);
    }
    __device__ __forceinline__ void density(const SpecDev &S, int par) {
        const int L = LT ? LT : lanes;
        RhoSums s;
        if (valid) {
            const float q2 = S.f_q2;
            for_entries(S, S.rec[par], q,
                        [&](const int4 &x) { rho_pair<SC76>(P, q2, ra, x, s); });
        }
        pe = density_end<SC76>(S, P, L, u, valid && l == 0, ra, s, wa);
    }
    __device__ __forceinline__ StepVals force(const SpecDev &S, int tile, int par, int phase,
                                                  long long done, long long nsteps) {
        const int L = LT ? LT : lanes;
        float f[3] = {0.f, 0.f, 0.f};
        if (valid) {
            const float q2 = S.f_q2;
            for_entries(S, S.posfp, q, [&](const int4 &x) {
                force_pair<SC76>(P, q2, ra, wa, x, f[0], f[1], f[2]);
            });
        }
        force_end(S, L, f);
        StepVals v = StepVals{};
        if (valid && l == 0)
            ra = atom_update_mixed(S, A, par, u, f, pe, MODE_STEP, phase, done, nsteps, v);
        // the new record to the atom's other lanes
        const int src = (threadIdx.x & 31) & ~(L - 1);
        ra.x = __shfl_sync(0xffffffffu, ra.x, src);
        ra.y = __shfl_sync(0xffffffffu, ra.y, src);
        ra.z = __shfl_sync(0xffffffffu, ra.z, src);
        warp_reduce(v, L);
        if ((threadIdx.x & 31) == 0) store_part(part_warp(S, tile), v);
        return v;
    }
};
template <bool SC76, int LT>
__global__ void __launch_bounds__(32 * RUN_WARPS, 1)
    k_run_f32(const SpecDev *specs, int nspec, const int *b2s, int nblk, RunCtl *rc,
              cudaGraphConditionalHandle again, unsigned polls, int quads, const PotF P) {
    extern __shared__ uint4 list_cache[];
    OpsF32<SC76, LT> ops{P, list_cache, quads};
    run_resident(specs, nspec, b2s, nblk, rc, again, polls, ops);
}

// a sweep's warp, on one tile
template <bool SC76>
struct SweepF32 {
    const PotF &P;
    __device__ __forceinline__ void prune(const SpecDev &S, int tile, int par) const {
        const int t = tile * 32 + (threadIdx.x & 31);
        if (t / S.L < S.n) prune_lane<true>(S, t / S.L, t % S.L, S.L, par);
    }
    __device__ __forceinline__ void density(const SpecDev &S, int tile, int par) const {
        const int t = tile * 32 + (threadIdx.x & 31);
        density_lane<SC76, true>(S, P, S.L, t / S.L, t % S.L, par);
    }
    __device__ __forceinline__ StepVals force(const SpecDev &S, int tile, int par, int phase,
                                                  long long done, long long nsteps) const {
        const int t = tile * 32 + (threadIdx.x & 31);
        const int L = S.L, u = t / L;
        float f[3];
        force_lane<SC76, true>(S, P, L, u, t % L, f);
        StepVals v = StepVals{};
        if (u < S.n && t % L == 0) update_atom(S, u, f, par, MODE_STEP, phase, done, nsteps, v);
        warp_reduce(v, L);
        if ((threadIdx.x & 31) == 0) store_part(part_warp(S, tile), v);
        return v;
    }
};
constexpr int SWEEP_WARPS_F32 = 28;  // 72 registers
template <bool SC76>
__global__ void __launch_bounds__(32 * SWEEP_WARPS_F32, 1)
    k_sweep_f32(const SpecDev *specs, int nspec, const int *b2s, int nblk, RunCtl *rc,
                cudaGraphConditionalHandle again, unsigned polls, int, const PotF P) {
    run_sweep(specs, nspec, b2s, nblk, rc, again, polls, SweepF32<SC76>{P});
}

template <int LT>
__global__ void __launch_bounds__(TPB, 8) k_prune(const SpecDev *__restrict__ specs,
                                                  const int *__restrict__ b2s, int force) {
    const SpecDev &S = specs[b2s[blockIdx.x]];
    if (!prune_active(S, force)) return;
    const int L = LT ? LT : S.L;
    const int u = (blockIdx.x - S.blk_pair0) * (TPB / L) + threadIdx.x / L;
    if (u < S.n) prune_lane<false>(S, u, threadIdx.x % L, L, S.ctl->parity);
}

void launch_prune(const Tab &t, int force, cudaStream_t st) {
    for (int i = 0; i < t.ngroups; ++i) {
        const Group &g = t.grp[i];
        if (g.nblk <= 0) continue;
        switch (g.L) {
            case 0: k_prune<0><<<g.nblk, TPB, 0, st>>>(t.specs, g.b2s, force); break;
            case 1: k_prune<1><<<g.nblk, TPB, 0, st>>>(t.specs, g.b2s, force); break;
            case 2: k_prune<2><<<g.nblk, TPB, 0, st>>>(t.specs, g.b2s, force); break;
            case 4: k_prune<4><<<g.nblk, TPB, 0, st>>>(t.specs, g.b2s, force); break;
            case 8: k_prune<8><<<g.nblk, TPB, 0, st>>>(t.specs, g.b2s, force); break;
            default: k_prune<16><<<g.nblk, TPB, 0, st>>>(t.specs, g.b2s, force); break;
        }
    }
}

// After the force pass: a block per specimen adds up its partials and advances
// its control block; with `decide`, the last block also sets what list
// maintenance the next step needs (counters of the specimens done and of those
// that prune or build, in one word).
__global__ void __launch_bounds__(32 * FINISH_WARPS)
    k_finish(const SpecDev *__restrict__ specs, int nspec, int mode, RunCtl *rc, int decide,
             cudaGraphConditionalHandle next) {
    const SpecDev &S = specs[blockIdx.x];
    SpecCtl *ctl = S.ctl;
    const int phase = ctl->phase;
    if (mode == MODE_EVAL || phase != PH_IDLE) {
        const int par = ctl->parity;
        const long long done = ctl->done, nsteps = ctl->nsteps;
        const StepVals t = finish_sums(S);
        if (threadIdx.x == 0)
            advance_ctl(S, t.s[0], t.s[1], t.s[2], t.d2, t.dp2, mode, phase, par, done, nsteps);
    }
    if (!decide || threadIdx.x != 0) return;
    constexpr int BITS = 21;
    constexpr unsigned long long MASK = (1ull << BITS) - 1;
    unsigned long long v = 1ull | (unsigned long long)prune_active(S, 0) << BITS |
                           (unsigned long long)build_active(S, 0) << (2 * BITS);
    v += atomicAdd(&rc->finished, v);
    if ((v & MASK) != (unsigned long long)nspec) return;
    rc->finished = 0;
    cudaGraphSetConditional(next, v >> (2 * BITS)       ? LIST_BUILD
                                  : (v >> BITS) & MASK ? LIST_PRUNE
                                                       : LIST_NONE);
}

void launch_finish(const Tab &t, int mode, RunCtl *rc, const cudaGraphConditionalHandle *next,
                   cudaStream_t st) {
    k_finish<<<t.nspec, 32 * FINISH_WARPS, 0, st>>>(t.specs, t.nspec, mode, rc, next != nullptr,
                                                    next ? *next : cudaGraphConditionalHandle());
}

// ---------------------------------------------------------------------------
// dispatch by (precision, lanes, potential variant)
// ---------------------------------------------------------------------------
void launch_density_f64(const Tab &t, const Group &g, int force, cudaStream_t st);
void launch_force_f64(const Tab &t, const Group &g, int mode, cudaStream_t st);

#define PTA_L_SWITCH(KER, SC)                                                            \
    switch (g.L) {                                                                       \
        case 0: KER<0, SC><<<g.nblk, TPB, 0, st>>>(t.specs, g.b2s, arg, g.pf); break;    \
        case 1: KER<1, SC><<<g.nblk, TPB, 0, st>>>(t.specs, g.b2s, arg, g.pf); break;    \
        case 2: KER<2, SC><<<g.nblk, TPB, 0, st>>>(t.specs, g.b2s, arg, g.pf); break;    \
        case 4: KER<4, SC><<<g.nblk, TPB, 0, st>>>(t.specs, g.b2s, arg, g.pf); break;    \
        case 8: KER<8, SC><<<g.nblk, TPB, 0, st>>>(t.specs, g.b2s, arg, g.pf); break;    \
        default: KER<16, SC><<<g.nblk, TPB, 0, st>>>(t.specs, g.b2s, arg, g.pf); break;  \
    }

void launch_density(const Tab &t, int arg, cudaStream_t st) {
    for (int i = 0; i < t.ngroups; ++i) {
        const Group &g = t.grp[i];
        if (g.nblk <= 0) continue;
        if (g.prec == PTA_PREC_FP64)
            launch_density_f64(t, g, arg, st);
        else if (g.sc76)
            PTA_L_SWITCH(k_density_f32, true)
        else
            PTA_L_SWITCH(k_density_f32, false)
    }
}

void launch_force(const Tab &t, int arg, cudaStream_t st) {
    for (int i = 0; i < t.ngroups; ++i) {
        const Group &g = t.grp[i];
        if (g.nblk <= 0) continue;
        if (g.prec == PTA_PREC_FP64)
            launch_force_f64(t, g, arg, st);
        else if (g.sc76)
            PTA_L_SWITCH(k_force_f32, true)
        else
            PTA_L_SWITCH(k_force_f32, false)
    }
}

// resident runs and sweeps
RunShape run_shape_f64(const Tab &t, bool &fits);
cudaError_t launch_run_f64(const Tab &t, const Group &g, RunCtl *rc,
                           cudaGraphConditionalHandle again, cudaStream_t st);

bool run_possible(const Tab &t, const int *b2s) {
    if (!t.b2s_run || t.nblk_run < 1) return false;
    const Group &g = t.grp[0];
    bool fits = false;
    RunShape r;
    if (g.prec == PTA_PREC_FP64) {
        r = run_shape_f64(t, fits);
    } else {
        r = run_shape(t.nblk_run, t.min_lanes, SWEEP_WARPS_F32, 0.9);
        fits = g.sc76 ? (r.sweep ? run_fits(k_sweep_f32<true>, r) : run_fits(k_run_f32<true, 0>, r) && run_fits(k_run_f32<true, 16>, r))
                      : (r.sweep ? run_fits(k_sweep_f32<false>, r) : run_fits(k_run_f32<false, 0>, r));
    }
    // every block's tiles belong to few specimens
    constexpr int NW = TPB / 32;
    const long long tiles = (long long)t.nblk_run * NW;
    for (int b = 0; b < r.blocks && fits; ++b) {
        const long long t0 = tiles * b / r.blocks, t1 = tiles * (b + 1) / r.blocks;
        fits = b2s[(t1 - 1) / NW] - b2s[t0 / NW] < RESIDENT_SPECS;
    }
    return fits;
}

cudaError_t launch_run(const Tab &t, RunCtl *rc, cudaGraphConditionalHandle again,
                       cudaStream_t st) {
    const Group &g = t.grp[0];
    if (g.prec == PTA_PREC_FP64) return launch_run_f64(t, g, rc, again, st);
    const RunShape r = run_shape(t.nblk_run, t.min_lanes, SWEEP_WARPS_F32, 0.9);
    auto go = [&](auto kernel) {
        return launch_cooperative(kernel, r, st, t.specs, t.nspec, t.b2s_run, t.nblk_run, rc, again,
                                  t.barrier_polls, r.quads, g.pf);
    };
    if (r.sweep) return g.sc76 ? go(k_sweep_f32<true>) : go(k_sweep_f32<false>);
    if (!g.sc76) return go(k_run_f32<false, 0>);
    return t.ngroups == 1 && g.L == 16 ? go(k_run_f32<true, 16>) : go(k_run_f32<true, 0>);
}

}  // namespace pta
