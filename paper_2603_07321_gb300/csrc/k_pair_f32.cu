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

// four list entries: read once per pass, so they skip L1 (the neighbour
// records keep the space) and ask L2 to fetch the 256-byte block around them
__device__ __forceinline__ uint4 ld_quad(const uint4 *p) {
    uint4 v;
    asm("ld.global.nc.L1::no_allocate.L2::256B.v4.u32 {%0, %1, %2, %3}, [%4];"
        : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
        : "l"(p));
    return v;
}
__device__ __forceinline__ int4 ld_rec(const SpecDev &S, const void *rec, unsigned e) {
    return __ldg((const int4 *)((const char *)rec + nl_off(S, e)));
}

// f(record) for the entries lane l of atom u reads, in list order: a quad per
// iteration (four gathers in flight), the next quad read ahead, then what is
// left of the last one
template <class F>
__device__ __forceinline__ void for_entries(const SpecDev &S, const void *rec, int u, int l, int L,
                                            F f) {
    const uint4 *p = S.plist + nl_col(u, l, L, S.capq);
    const int cnt = chk_count(S, S.pnn[u * L + l], 4 * (S.capq - 1));
    uint4 e = ld_quad(p);
    for (int t = cnt >> 2; t > 0; --t) {
        p += 32;
        const uint4 nx = ld_quad(p);
        const int4 x0 = ld_rec(S, rec, e.x), x1 = ld_rec(S, rec, e.y);
        const int4 x2 = ld_rec(S, rec, e.z), x3 = ld_rec(S, rec, e.w);
        f(x0);
        f(x1);
        f(x2);
        f(x3);
        e = nx;
    }
    const int left = cnt & 3;
    if (left) {
        int4 x0 = ld_rec(S, rec, e.x), x1 = x0, x2 = x0;
        if (left > 1) x1 = ld_rec(S, rec, e.y);
        if (left > 2) x2 = ld_rec(S, rec, e.z);
        f(x0);
        if (left > 1) f(x1);
        if (left > 2) f(x2);
    }
}

template <int L, bool SC76>
__device__ __forceinline__ void density_block(const SpecDev &S, int lb, int par, const PotF &P) {
    constexpr int UPB = TPB / L;
    const int u = lb * UPB + threadIdx.x / L;
    const int l = threadIdx.x % L;
    const bool valid = u < S.n;
    RhoSums s;
    int4 ra = make_int4(0, 0, 0, 0);
    if (valid) {
        ra = S.rec[par][u];
        const float q2 = S.f_q2;
        for_entries(S, S.rec[par], u, l, L,
                    [&](const int4 &x) { rho_pair<SC76>(P, q2, ra, x, s); });
    }
    s.sm = lane_sum<L>(s.sm);
    s.sn = lane_sum<L>(s.sn);
    s.sr = lane_sum<L>(s.sr);
    const float cnt = (float)lane_sum<L>(s.cnt);
    if (valid && l == 0) {
        const float dr = fmaf(-cnt, P.rc, s.sr);  // sum of r - rc
        const float rho = SC76 ? fmaf(P.am, s.sm, fmaf(P.Bm, dr, -cnt * P.Am)) : s.sm;
        const float phn = fmaf(P.an, s.sn, fmaf(P.Bn, dr, -cnt * P.An));
        // w = m a^m B'(rho), B'(rho) = -eps c / (2 sqrt(rho))
        const float rq = rho > 0.f ? rsqrtf(rho) : 0.f;
        const float w = P.fpsc * rq;
        // the atom's energy 1/2 eps sum_j phi_n + B(rho), B = -eps c sqrt(rho)
        ((float *)S.pen)[u] = fmaf(-P.ec, rho > 0.f ? rho * rq : 0.f, 0.5f * P.eps * phn);
        ((int4 *)S.posfp)[u] = make_int4(ra.x, ra.y, ra.z, __float_as_int(w));
    }
}

template <int L, bool SC76>
__device__ __forceinline__ void force_block(const SpecDev &S, int lb, int par, const PotF &P,
                                            int mode, int phase, long long done,
                                            long long nsteps) {
    constexpr int UPB = TPB / L;
    const int u = lb * UPB + threadIdx.x / L;
    const int l = threadIdx.x % L;
    const bool valid = u < S.n;
    float fx = 0.f, fy = 0.f, fz = 0.f, wa = 0.f;
    if (valid) {
        const int4 ra = ((const int4 *)S.posfp)[u];
        wa = __int_as_float(ra.w);
        const float q2 = S.f_q2;
        for_entries(S, S.posfp, u, l, L,
                    [&](const int4 &x) { force_pair<SC76>(P, q2, ra, wa, x, fx, fy, fz); });
    }
    // sums of (eV/A^2) x quanta
    fx = lane_sum<L>(fx) * S.f_q;
    fy = lane_sum<L>(fy) * S.f_q;
    fz = lane_sum<L>(fz) * S.f_q;
    double ke = 0.0, pe = 0.0, rr = 0.0;
    float d2 = 0.f, dp2 = 0.f;
    if (valid && l == 0)
        atom_update_mixed(S, S.ctl, par, u, S.prune_on != 0, fx, fy, fz, mode, phase, done, nsteps,
                          ke, pe, rr, d2, dp2);
    ke = warp_sum(ke);
    pe = warp_sum(pe);
    rr = warp_sum(rr);
    d2 = warp_max(d2);
    dp2 = warp_max(dp2);
    step_tail<TPB>(S, lb, S.nblk_pair, ke, pe, rr, (double)d2, (double)dp2, mode, phase, done,
                   nsteps);
}

template <int L, bool SC76>
__global__ void __launch_bounds__(TPB, 8) k_density_f32(const SpecDev *__restrict__ specs,
                                                        const int *__restrict__ b2s, int force,
                                                        const PotF P) {
    const SpecDev &S = specs[b2s[blockIdx.x]];
    if (!force && S.ctl->phase == PH_IDLE) return;
    density_block<L, SC76>(S, blockIdx.x - S.blk_pair0, S.ctl->parity, P);
}

template <int L, bool SC76>
__global__ void __launch_bounds__(TPB, 8) k_force_f32(const SpecDev *__restrict__ specs,
                                                      const int *__restrict__ b2s, int mode,
                                                      const PotF P) {
    const SpecDev &S = specs[b2s[blockIdx.x]];
    const SpecCtl *ctl = S.ctl;
    const int phase = ctl->phase;
    if (mode == MODE_STEP && phase == PH_IDLE) return;
    force_block<L, SC76>(S, blockIdx.x - S.blk_pair0, ctl->parity, P, mode, phase, ctl->done,
                         ctl->nsteps);
}

// Pruning (both precisions): every lane appends to the near part of its
// column, in order, the entries of its far part within the pruning radius
// (FP32 distances of the records against (rc + margin)^2 with slack).  Pairs
// within rc are therefore all kept, in the order the lane sums them.
//
// Bound: the gathers of the far part's records (~118 of the ~252 entries of a
// bulk atom at the default 2 A skin).
template <int L>
__global__ void __launch_bounds__(TPB, 8) k_prune(const SpecDev *__restrict__ specs,
                                                  const int *__restrict__ b2s, int force) {
    const SpecDev &S = specs[b2s[blockIdx.x]];
    if (!prune_active(S, force)) return;
    const int par = S.ctl->parity;
    constexpr int UPB = TPB / L;
    const int u = (blockIdx.x - S.blk_pair0) * UPB + threadIdx.x / L;
    const int l = threadIdx.x % L;
    if (u >= S.n) return;
    const int4 *rec = S.rec[par];
    const int4 ra = rec[u];
    const float rp2 = S.f_rp2q;
    const int2 ab = S.nab[u];
    const long long col = nl_col(u, l, L, S.capq);
    const uint4 *p = S.nlist + col;
    unsigned *dst = (unsigned *)(S.plist + col);
    const int nl = chk_count(S, ab.y > l ? (ab.y - l + L - 1) / L : 0, S.cap_use);
    int kept = ab.x / L + (l < ab.x % L);
    auto test = [&](bool have, unsigned e, const int4 &x) {
        const float dx = (float)(x.x - ra.x), dy = (float)(x.y - ra.y), dz = (float)(x.z - ra.z);
        if (fmaf(dz, dz, fmaf(dy, dy, dx * dx)) < rp2 && have) {
            dst[(kept >> 2) * 128 + (kept & 3)] = e;
            ++kept;
        }
    };
    uint4 e = ld_quad(p);
    for (int q = 0; q < nl; q += 4) {
        p += 32;
        const uint4 nx = ld_quad(p);
        const int4 x0 = ld_rec(S, rec, e.x), x1 = ld_rec(S, rec, e.y);
        const int4 x2 = ld_rec(S, rec, e.z), x3 = ld_rec(S, rec, e.w);
        test(true, e.x, x0);
        test(q + 1 < nl, e.y, x1);
        test(q + 2 < nl, e.z, x2);
        test(q + 3 < nl, e.w, x3);
        e = nx;
    }
    S.pnn[u * L + l] = kept;
    if (l == 0) {
        if (S.prec == PTA_PREC_FP64) {
            const double4_32a x = ((const double4_32a *)S.pos[par])[u];
            S.pref[u] = make_float4((float)x.x, (float)x.y, (float)x.z, 0.f);
        } else {
            const float4 hi = ((const float4 *)S.pos[par])[u];
            const float4 lo = S.lo[par][u];
            S.pref[u] = make_float4(hi.x + lo.x, hi.y + lo.y, hi.z + lo.z, 0.f);
        }
    }
}

// after the pruning: clear the flag (a separate kernel, so that every block
// of the pruning kernel reads the same flag)
__global__ void k_prune_done(const SpecDev *__restrict__ specs, int force) {
    const SpecDev &S = specs[blockIdx.x];
    if (!prune_active(S, force)) return;
    if (threadIdx.x == 0) {
        S.ctl->prune = 0;
        S.ctl->prunes += 1;
    }
}

void launch_prune(const Tab &t, int force, cudaStream_t st) {
    for (int i = 0; i < t.ngroups; ++i) {
        const Group &g = t.grp[i];
        if (g.nblk <= 0) continue;
        switch (g.L) {
            case 1: k_prune<1><<<g.nblk, TPB, 0, st>>>(t.specs, g.b2s, force); break;
            case 2: k_prune<2><<<g.nblk, TPB, 0, st>>>(t.specs, g.b2s, force); break;
            case 4: k_prune<4><<<g.nblk, TPB, 0, st>>>(t.specs, g.b2s, force); break;
            case 8: k_prune<8><<<g.nblk, TPB, 0, st>>>(t.specs, g.b2s, force); break;
            default: k_prune<16><<<g.nblk, TPB, 0, st>>>(t.specs, g.b2s, force); break;
        }
    }
    k_prune_done<<<t.nspec, 32, 0, st>>>(t.specs, force);
}

// ---------------------------------------------------------------------------
// dispatch by (precision, lanes, potential variant)
// ---------------------------------------------------------------------------
void launch_density_f64(const Tab &t, const Group &g, int force, cudaStream_t st);
void launch_force_f64(const Tab &t, const Group &g, int mode, cudaStream_t st);

#define PTA_L_SWITCH(KER, SC)                                                            \
    switch (g.L) {                                                                       \
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

}  // namespace pta
