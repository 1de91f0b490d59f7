// FP64 pair kernels: the same two passes as the mixed-precision kernels
// (density, then forces with the fused velocity-Verlet epilogue), with every
// quantity in double.  They serve the plain FP64 form of the method and the
// parity checks against the FP64 oracle.
//
// FP64 runs at 1/75 of the FP32 rate on this GPU (two lanes per clock and
// SM), so the passes are bound by the number of double operations per list
// entry and everything else is nearly free: y = 1/r from one reciprocal square
// root (CUDA's rsqrt on double), no division, no square root; the density pass
// sums y^6, y^7, r and the number of pairs and assembles rho and the pair
// energy once per atom (18 operations per pair within rc, 21 with phi_m formed
// per pair); the force pass takes the weight m a^m B'(rho) from the record as
// the mixed-precision one does (23 operations, 34 before); the cutoff test
// compares the bits as integers.  Sums and products are written as fused
// operations, so that every kernel these passes are compiled into rounds alike.
#include "k_pair_common.cuh"

namespace pta {

__device__ __forceinline__ double ipow(double s, int k) {
    double p = 1.0;
    for (int i = 0; i < k; ++i) p = __dmul_rn(p, s);
    return p;
}

// squared distance and displacement of b from a
__device__ __forceinline__ double pair_r2(const double4_32a &a, const double4_32a &b, double &dx,
                                          double &dy, double &dz) {
    dx = b.x - a.x;
    dy = b.y - a.y;
    dz = b.z - a.z;
    return fma(dz, dz, fma(dy, dy, __dmul_rn(dx, dx)));
}
// r2 < rc2 for non-negative doubles (their bits order as integers): on r2, so
// that coincident atoms (r2 = 0) still give a non-finite result
__device__ __forceinline__ bool within(double r2, double rc2) {
    return __double_as_longlong(r2) < __double_as_longlong(rc2);
}

// density pass, one pair within rc
struct RhoSums64 {
    double sm = 0.0, sn = 0.0, sr = 0.0;
    int cnt = 0;
};
template <bool SC76>
__device__ __forceinline__ void rho_pair64(const PotDev &P, double r2, RhoSums64 &s) {
    const double y = rsqrt(r2);
    if (SC76) {
        const double y3 = __dmul_rn(__dmul_rn(y, y), y), y6 = __dmul_rn(y3, y3);
        s.sm = fma(y3, y3, s.sm);
        s.sn = fma(y6, y, s.sn);
    } else {
        s.sm = __dadd_rn(s.sm, ipow(y, P.m));
        s.sn = __dadd_rn(s.sn, ipow(y, P.n));
    }
    s.sr = fma(r2, y, s.sr);
    s.cnt += 1;
}

// force pass, one pair within rc: [eps phi_n' + (B'_i + B'_j) phi_m'] / r with
// q = w_i + w_j, w = m a^m B'(rho)
template <bool SC76>
__device__ __forceinline__ double force_pair64(const PotDev &P, double r2, double q) {
    const double y = rsqrt(r2), y2 = __dmul_rn(y, y);
    const double c = fma(q, P.bmq, P.ebn);
    double v;
    if (SC76) {
        const double y4 = __dmul_rn(y2, y2);
        v = __dmul_rn(__dmul_rn(y4, y4), fma(P.kn, y, q));
    } else {
        v = __dmul_rn(y2, fma(q, ipow(y, P.m), __dmul_rn(P.kn, ipow(y, P.n))));
    }
    return fma(y, c, -v);
}

template <bool RES>
__device__ __forceinline__ double4_32a ld_pos64(const SpecDev &S, const double4_32a *pos, unsigned e) {
    const double4_32a *p = pos + nl_j(nl_off(S, e));
    if (RES) return *p;
    // the read-only path, two 16-byte loads
    const double2 a = __ldg((const double2 *)p), b = __ldg((const double2 *)p + 1);
    return make_double4_32a(a.x, a.y, b.x, b.y);
}
// f(position) for the entries lane l of atom a reads, in list order (list
// entries are byte offsets of 16-byte records, half of a double4's)
template <bool RES, class F>
__device__ __forceinline__ void for_entries64(const SpecDev &S, const double4_32a *pos, int a,
                                              int l, int L, F f) {
    const uint4 *p = S.plist + nl_col(a, l, L, S.capq);
    const int cnt = chk_count(S, S.pnn[a * L + l], 4 * (S.capq - 1));
    uint4 e = ld_quad<RES>(p);
    for (int t = cnt >> 2; t > 0; --t) {
        p += 32;
        const uint4 nx = ld_quad<RES>(p);
        const double4_32a x0 = ld_pos64<RES>(S, pos, e.x), x1 = ld_pos64<RES>(S, pos, e.y);
        const double4_32a x2 = ld_pos64<RES>(S, pos, e.z), x3 = ld_pos64<RES>(S, pos, e.w);
        f(x0);
        f(x1);
        f(x2);
        f(x3);
        e = nx;
    }
    const int left = cnt & 3;
    if (left > 0) f(ld_pos64<RES>(S, pos, e.x));
    if (left > 1) f(ld_pos64<RES>(S, pos, e.y));
    if (left > 2) f(ld_pos64<RES>(S, pos, e.z));
}

// the same in a resident run, from the list in shared memory
template <class F>
__device__ __forceinline__ void for_entries64(const SpecDev &S, const double4_32a *pos,
                                              const LaneList &q, F f) {
    int t = 0, left = q.cnt;
    for (; left >= 4; left -= 4, ++t) {
        const uint4 e = q.quad(t);
        const double4_32a x0 = ld_pos64<true>(S, pos, e.x), x1 = ld_pos64<true>(S, pos, e.y);
        const double4_32a x2 = ld_pos64<true>(S, pos, e.z), x3 = ld_pos64<true>(S, pos, e.w);
        f(x0);
        f(x1);
        f(x2);
        f(x3);
    }
    if (left > 0) {
        const uint4 e = q.quad(t);
        f(ld_pos64<true>(S, pos, e.x));
        if (left > 1) f(ld_pos64<true>(S, pos, e.y));
        if (left > 2) f(ld_pos64<true>(S, pos, e.z));
    }
}

// An atom's state outside the neighbour records.
struct Atom64 {
    double x[3], v[3];
    int4 ref, pref;
    int flag;
    __device__ __forceinline__ void load(const SpecDev &S, int par, int a) {
        const double4_32a q = ((const double4_32a *)S.pos[par])[a];
        const double4_32a w = ((const double4_32a *)S.vel)[a];
        x[0] = q.x; x[1] = q.y; x[2] = q.z;
        v[0] = w.x; v[1] = w.y; v[2] = w.z;
        ref = S.ref[a];
        pref = S.prune_on ? S.pref[a] : ref;
        flag = S.flags[a];
    }
    // the position goes to buffer par with every step (neighbours read it)
    __device__ __forceinline__ void store_pos(const SpecDev &S, int par, int a) const {
        ((double4_32a *)S.pos[par])[a] = make_double4_32a(x[0], x[1], x[2], 0.0);
    }
    __device__ __forceinline__ void store_vel(const SpecDev &S, int a) const {
        ((double4_32a *)S.vel)[a] = make_double4_32a(v[0], v[1], v[2], 0.0);
    }
};

// After the force pass of atom a (force f, energy pe): as atom_update_mixed,
// in FP64; the new position and record go to the other buffers.
__device__ __forceinline__ void atom_update64(const SpecDev &S, Atom64 &A, int par, int a,
                                              const double f[3], double pe, int mode, int phase,
                                              long long done, long long nsteps,
                                              StepVals &out) {
    chk_force(S, f[0], f[1], f[2]);
    const SpecCtl *ctl = S.ctl;
    out.s[1] = pe;
    if (A.flag == FLAG_RIGHT) out.s[2] = -(S.axis == 0 ? f[0] : (S.axis == 1 ? f[1] : f[2]));
    auto kinetic = [&] {
        out.s[0] = __dmul_rn(
            S.ke_fac, fma(A.v[2], A.v[2], fma(A.v[1], A.v[1], __dmul_rn(A.v[0], A.v[0]))));
    };
    if (mode == MODE_EVAL) {
        kinetic();
        eval_store(S, a, f[0], f[1], f[2], pe);
        return;
    }
    const double kh = S.acc_half;
    // thermal relaxation: the right grip moves along the load axis only
    const bool rfree = A.flag == FLAG_RIGHT && ctl->relax;
    auto kick = [&] {
#pragma unroll
        for (int d = 0; d < 3; ++d)
            if (A.flag == FLAG_MOBILE || (rfree && S.axis == d)) A.v[d] = fma(f[d], kh, A.v[d]);
    };
    if (phase == PH_RUN) {
        kick();
        kinetic();
        if (S.rsum) {
            // Eq. (mean_pos): the sampled state's position
            double *rs = S.rsum + 4LL * S.orig[a];
#pragma unroll
            for (int d = 0; d < 3; ++d) rs[d] = rs[d] + A.x[d];
        }
    }
    const bool start = (phase == PH_REFRESH) || (done + 1 < nsteps);
    if (start && (A.flag == FLAG_MOBILE || rfree)) {
        kick();
#pragma unroll
        for (int d = 0; d < 3; ++d) A.x[d] = fma(A.v[d], S.dt, A.x[d]);
    } else if (start && A.flag == FLAG_RIGHT && ctl->grip_du != 0.0) {
        // continuous loading (fine-dynamics verification)
#pragma unroll
        for (int d = 0; d < 3; ++d)
            A.x[d] = __dadd_rn(A.x[d], S.axis == d ? ctl->grip_du : 0.0);
    }
    A.store_pos(S, par ^ 1, a);
    const int4 r = rec_fp64(S, A.x[0], A.x[1], A.x[2]);
    S.rec[par ^ 1][a] = r;
    out.d2 = moved2(r, A.ref);
    out.dp2 = moved2(r, A.pref);
}

__device__ __forceinline__ double density_end64(const SpecDev &S, int L, int a, bool first,
                                                const double4_32a &pa, RhoSums64 s, double &w) {
    const PotDev &P = S.pot;
    s.sm = lane_sum(s.sm, L);
    s.sn = lane_sum(s.sn, L);
    s.sr = lane_sum(s.sr, L);
    const double cnt = (double)lane_sum(s.cnt, L);
    const double dr = fma(-cnt, P.rc, s.sr);  // sum of r - rc
    const double rho =
        fma(P.am, s.sm, fma(P.am_lo, s.sm, fma(P.Bm, dr, __dmul_rn(-cnt, P.Am))));
    const double phn = fma(P.an, s.sn, fma(P.Bn, dr, __dmul_rn(-cnt, P.An)));
    // w = m a^m B'(rho), B'(rho) = -eps c / (2 sqrt(rho))
    const double sq = rho > 0.0 ? sqrt(rho) : 0.0;
    w = rho > 0.0 ? P.fpsc / sq : 0.0;
    w = fma(w, P.fpsc_rel, w);
    if (first) ((double4_32a *)S.posfp)[a] = make_double4_32a(pa.x, pa.y, pa.z, w);
    // the atom's energy 1/2 eps sum_j phi_n + B(rho), B = -eps c sqrt(rho)
    return fma(-P.ec, sq, __dmul_rn(0.5 * P.eps, phn));
}

template <bool SC76>
__device__ __forceinline__ void force_entry64(const PotDev &P, const double4_32a &pa,
                                              const double4_32a &pj, double f[3]) {
    double dx, dy, dz;
    const double r2 = pair_r2(pa, pj, dx, dy, dz);
    if (within(r2, P.rc2)) {
        const double g = force_pair64<SC76>(P, r2, __dadd_rn(pa.w, pj.w));
        f[0] = fma(g, dx, f[0]);
        f[1] = fma(g, dy, f[1]);
        f[2] = fma(g, dz, f[2]);
    }
}
template <bool SC76>
__device__ __forceinline__ void rho_entry64(const PotDev &P, const double4_32a &pa,
                                            const double4_32a &pj, RhoSums64 &s) {
    double dx, dy, dz;
    const double r2 = pair_r2(pa, pj, dx, dy, dz);
    if (within(r2, P.rc2)) rho_pair64<SC76>(P, r2, s);
}

// the passes of one thread (lane l of atom a) with everything in memory
template <bool SC76, bool RES>
__device__ __forceinline__ void density_lane64(const SpecDev &S, int L, int a, int l, int par) {
    const bool valid = a < S.n;
    const double4_32a *pos = (const double4_32a *)S.pos[par];
    RhoSums64 s;
    double4_32a pa = make_double4_32a(0, 0, 0, 0);
    if (valid) {
        pa = pos[a];
        for_entries64<RES>(S, pos, a, l, L,
                           [&](const double4_32a &pj) { rho_entry64<SC76>(S.pot, pa, pj, s); });
    }
    double w;
    const double pe = density_end64(S, L, a, valid && l == 0, pa, s, w);
    if (valid && l == 0) ((double *)S.pen)[a] = pe;
}

// the force on atom a, in all its lanes
template <bool SC76, bool RES>
__device__ __forceinline__ void force_lane64(const SpecDev &S, int L, int a, int l, double f[3]) {
    f[0] = f[1] = f[2] = 0;
    if (a < S.n) {
        const double4_32a *pf = (const double4_32a *)S.posfp;
        const double4_32a pa = pf[a];
        for_entries64<RES>(S, pf, a, l, L,
                           [&](const double4_32a &pj) { force_entry64<SC76>(S.pot, pa, pj, f); });
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) f[d] = lane_sum(f[d], L);
}
// the update of atom a by one thread, with its state in memory
__device__ __forceinline__ void update_atom64(const SpecDev &S, int a, const double f[3], int par,
                                              int mode, int phase, long long done,
                                              long long nsteps, StepVals &v) {
    Atom64 A;
    A.load(S, par, a);
    atom_update64(S, A, par, a, f, ((const double *)S.pen)[a], mode, phase, done, nsteps, v);
    if (mode != MODE_EVAL) A.store_vel(S, a);
}

template <int LT, bool SC76>
__global__ void __launch_bounds__(TPB) k_density_f64(const SpecDev *__restrict__ specs,
                                                     const int *__restrict__ b2s, int force) {
    const SpecDev &S = specs[b2s[blockIdx.x]];
    if (!force && S.ctl->phase == PH_IDLE) return;
    const int L = LT ? LT : S.L;
    const int a = (blockIdx.x - S.blk_pair0) * (TPB / L) + threadIdx.x / L;
    density_lane64<SC76, false>(S, L, a, threadIdx.x % L, S.ctl->parity);
}

template <int LT, bool SC76>
__global__ void __launch_bounds__(TPB) k_force_f64(const SpecDev *__restrict__ specs,
                                                   const int *__restrict__ b2s, int mode) {
    const SpecDev &S = specs[b2s[blockIdx.x]];
    const SpecCtl *ctl = S.ctl;
    const int phase = ctl->phase;
    if (mode == MODE_STEP && phase == PH_IDLE) return;
    const int par = ctl->parity, lb = blockIdx.x - S.blk_pair0;
    const long long done = ctl->done, nsteps = ctl->nsteps;
    const int L = LT ? LT : S.L, APB = TPB / L;
    double f[3];
    force_lane64<SC76, false>(S, L, lb * APB + threadIdx.x / L, threadIdx.x % L, f);
    if (L > 1) {  // the block's atoms to its first threads, as in mixed precision
        __shared__ double sf[3][TPB / (LT ? LT : 2)];
        if (threadIdx.x % L == 0)
#pragma unroll
            for (int d = 0; d < 3; ++d) sf[d][threadIdx.x / L] = f[d];
        __syncthreads();
        if (threadIdx.x < APB)
#pragma unroll
            for (int d = 0; d < 3; ++d) f[d] = sf[d][threadIdx.x];
    }
    const int a = lb * APB + threadIdx.x;
    StepVals v = StepVals{};
    if (threadIdx.x < APB && a < S.n) update_atom64(S, a, f, par, mode, phase, done, nsteps, v);
    block_partial<TPB>(S, lb, v, L);
}

// a resident run's warp
template <bool SC76>
struct OpsF64 {
    uint4 *cache;
    int quads;
    Atom64 A;
    LaneList q;
    double4_32a pa;  // the atom's position and density weight (all its lanes)
    double pe;
    int L, a, l;
    bool valid;
    __device__ __forceinline__ void load(const SpecDev &S, int tile, int par) {
        const int t = tile * 32 + (threadIdx.x & 31);
        L = S.L;
        a = t / L;
        l = t % L;
        valid = a < S.n;
        pa = make_double4_32a(0, 0, 0, 0);
        pe = 0.0;
        if (valid) {
            q.fill(S, cache, a, l, L, quads);
            pa = ((const double4_32a *)S.pos[par])[a];
            if (l == 0) A.load(S, par, a);
        }
    }
    __device__ __forceinline__ void prune(const SpecDev &S, int par) {
        if (!valid) return;
        prune_lane<true>(S, a, l, L, par);
        q.fill(S, cache, a, l, L, quads);
        A.pref = S.rec[par][a];
    }
    __device__ __forceinline__ void store(const SpecDev &S, int par) const {
        if (valid && l == 0) A.store_vel(S, a);
    }
    __device__ __forceinline__ void density(const SpecDev &S, int par) {
        const double4_32a *pos = (const double4_32a *)S.pos[par];
        RhoSums64 s;
        if (valid)
            for_entries64(S, pos, q,
                          [&](const double4_32a &pj) { rho_entry64<SC76>(S.pot, pa, pj, s); });
        pe = density_end64(S, L, a, valid && l == 0, pa, s, pa.w);
    }
    __device__ __forceinline__ StepVals force(const SpecDev &S, int tile, int par, int phase,
                                                  long long done, long long nsteps) {
        double f[3] = {0, 0, 0};
        if (valid)
            for_entries64(S, (const double4_32a *)S.posfp, q,
                          [&](const double4_32a &pj) { force_entry64<SC76>(S.pot, pa, pj, f); });
#pragma unroll
        for (int d = 0; d < 3; ++d) f[d] = lane_sum(f[d], L);
        StepVals v = StepVals{};
        if (valid && l == 0) {
            atom_update64(S, A, par, a, f, pe, MODE_STEP, phase, done, nsteps, v);
            pa.x = A.x[0];
            pa.y = A.x[1];
            pa.z = A.x[2];
        }
        // the new position to the atom's other lanes
        const int src = (threadIdx.x & 31) & ~(L - 1);
        pa.x = __shfl_sync(0xffffffffu, pa.x, src);
        pa.y = __shfl_sync(0xffffffffu, pa.y, src);
        pa.z = __shfl_sync(0xffffffffu, pa.z, src);
        warp_reduce(v, L);
        if ((threadIdx.x & 31) == 0) store_part(part_warp(S, tile), v);
        return v;
    }
};
template <bool SC76>
__global__ void __launch_bounds__(32 * RUN_WARPS, 1)
    k_run_f64(const SpecDev *specs, int nspec, const int *b2s, int nblk, RunCtl *rc,
              cudaGraphConditionalHandle again, unsigned polls, int quads) {
    extern __shared__ uint4 list_cache[];
    OpsF64<SC76> ops{list_cache, quads};
    run_resident(specs, nspec, b2s, nblk, rc, again, polls, ops);
}

// a sweep's warp, on one tile
template <bool SC76>
struct SweepF64 {
    __device__ __forceinline__ void prune(const SpecDev &S, int tile, int par) const {
        const int t = tile * 32 + (threadIdx.x & 31);
        if (t / S.L < S.n) prune_lane<true>(S, t / S.L, t % S.L, S.L, par);
    }
    __device__ __forceinline__ void density(const SpecDev &S, int tile, int par) const {
        const int t = tile * 32 + (threadIdx.x & 31);
        density_lane64<SC76, true>(S, S.L, t / S.L, t % S.L, par);
    }
    __device__ __forceinline__ StepVals force(const SpecDev &S, int tile, int par, int phase,
                                                      long long done, long long nsteps) const {
        const int t = tile * 32 + (threadIdx.x & 31);
        const int L = S.L, a = t / L;
        double f[3];
        force_lane64<SC76, true>(S, L, a, t % L, f);
        StepVals v = StepVals{};
        if (a < S.n && t % L == 0) update_atom64(S, a, f, par, MODE_STEP, phase, done, nsteps, v);
        warp_reduce(v, L);
        if ((threadIdx.x & 31) == 0) store_part(part_warp(S, tile), v);
        return v;
    }
};
constexpr int SWEEP_WARPS_F64 = 20;
template <bool SC76>
__global__ void __launch_bounds__(32 * SWEEP_WARPS_F64, 1)
    k_sweep_f64(const SpecDev *specs, int nspec, const int *b2s, int nblk, RunCtl *rc,
                cudaGraphConditionalHandle again, unsigned polls, int) {
    run_sweep(specs, nspec, b2s, nblk, rc, again, polls, SweepF64<SC76>{});
}

#define PTA_F64_SWITCH(KER, SC, ARG)                                                   \
    switch (g.L) {                                                                     \
        case 0: KER<0, SC><<<g.nblk, TPB, 0, st>>>(t.specs, g.b2s, ARG); break;        \
        case 1: KER<1, SC><<<g.nblk, TPB, 0, st>>>(t.specs, g.b2s, ARG); break;        \
        case 2: KER<2, SC><<<g.nblk, TPB, 0, st>>>(t.specs, g.b2s, ARG); break;        \
        case 4: KER<4, SC><<<g.nblk, TPB, 0, st>>>(t.specs, g.b2s, ARG); break;        \
        case 8: KER<8, SC><<<g.nblk, TPB, 0, st>>>(t.specs, g.b2s, ARG); break;        \
        default: KER<16, SC><<<g.nblk, TPB, 0, st>>>(t.specs, g.b2s, ARG); break;      \
    }

void launch_density_f64(const Tab &t, const Group &g, int force, cudaStream_t st) {
    if (g.sc76)
        PTA_F64_SWITCH(k_density_f64, true, force)
    else
        PTA_F64_SWITCH(k_density_f64, false, force)
}

void launch_force_f64(const Tab &t, const Group &g, int mode, cudaStream_t st) {
    if (g.sc76)
        PTA_F64_SWITCH(k_force_f64, true, mode)
    else
        PTA_F64_SWITCH(k_force_f64, false, mode)
}

RunShape run_shape_f64(const Tab &t, bool &fits) {
    const RunShape r = run_shape(t.nblk_run, t.min_lanes, SWEEP_WARPS_F64, 0.0);
    fits = t.grp[0].sc76
               ? (r.sweep ? run_fits(k_sweep_f64<true>, r) : run_fits(k_run_f64<true>, r))
               : (r.sweep ? run_fits(k_sweep_f64<false>, r) : run_fits(k_run_f64<false>, r));
    return r;
}

cudaError_t launch_run_f64(const Tab &t, const Group &g, RunCtl *rc,
                           cudaGraphConditionalHandle again, cudaStream_t st) {
    const RunShape r = run_shape(t.nblk_run, t.min_lanes, SWEEP_WARPS_F64, 0.0);
    auto go = [&](auto kernel) {
        return launch_cooperative(kernel, r, st, t.specs, t.nspec, t.b2s_run, t.nblk_run, rc, again,
                                  t.barrier_polls, r.quads);
    };
    if (g.sc76) return r.sweep ? go(k_sweep_f64<true>) : go(k_run_f64<true>);
    return r.sweep ? go(k_sweep_f64<false>) : go(k_run_f64<false>);
}

}  // namespace pta
