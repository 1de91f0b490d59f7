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
        s.sm = __dadd_rn(s.sm, y6);
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

// f(position) for the entries lane l of atom a reads, in list order (list
// entries are byte offsets of 16-byte records, half of a double4's)
template <class F>
__device__ __forceinline__ void for_entries64(const SpecDev &S, const double4_32a *pos, int a,
                                              int l, int L, F f) {
    const uint4 *p = S.plist + nl_col(a, l, L, S.capq);
    const int cnt = chk_count(S, S.pnn[a * L + l], 4 * (S.capq - 1));
    uint4 e = __ldg(p);
    for (int t = cnt >> 2; t > 0; --t) {
        p += 32;
        const uint4 nx = __ldg(p);
        const double4_32a x0 = pos[nl_j(nl_off(S, e.x))], x1 = pos[nl_j(nl_off(S, e.y))];
        const double4_32a x2 = pos[nl_j(nl_off(S, e.z))], x3 = pos[nl_j(nl_off(S, e.w))];
        f(x0);
        f(x1);
        f(x2);
        f(x3);
        e = nx;
    }
    const int left = cnt & 3;
    if (left > 0) f(pos[nl_j(nl_off(S, e.x))]);
    if (left > 1) f(pos[nl_j(nl_off(S, e.y))]);
    if (left > 2) f(pos[nl_j(nl_off(S, e.z))]);
}

template <int L, bool SC76>
__global__ void __launch_bounds__(TPB) k_density_f64(const SpecDev *__restrict__ specs,
                                                     const int *__restrict__ b2s, int force) {
    const SpecDev &S = specs[b2s[blockIdx.x]];
    const SpecCtl *ctl = S.ctl;
    if (!force && ctl->phase == PH_IDLE) return;
    const int par = ctl->parity;
    constexpr int APB = TPB / L;
    const int a = (blockIdx.x - S.blk_pair0) * APB + threadIdx.x / L;
    const int l = threadIdx.x % L;
    const bool valid = a < S.n;
    const double4_32a *__restrict__ pos = (const double4_32a *)S.pos[par];
    const PotDev &P = S.pot;
    RhoSums64 s;
    double4_32a pa = make_double4_32a(0, 0, 0, 0);
    if (valid) {
        pa = pos[a];
        for_entries64(S, pos, a, l, L, [&](const double4_32a &pj) {
            double dx, dy, dz;
            const double r2 = pair_r2(pa, pj, dx, dy, dz);
            if (within(r2, P.rc2)) rho_pair64<SC76>(P, r2, s);
        });
    }
    s.sm = lane_sum<L>(s.sm);
    s.sn = lane_sum<L>(s.sn);
    s.sr = lane_sum<L>(s.sr);
    const double cnt = (double)lane_sum<L>(s.cnt);
    if (valid && l == 0) {
        const double dr = fma(-cnt, P.rc, s.sr);  // sum of r - rc
        const double rho = fma(P.am, s.sm, fma(P.Bm, dr, __dmul_rn(-cnt, P.Am)));
        const double phn = fma(P.an, s.sn, fma(P.Bn, dr, __dmul_rn(-cnt, P.An)));
        // w = m a^m B'(rho), B'(rho) = -eps c / (2 sqrt(rho))
        const double sq = rho > 0.0 ? sqrt(rho) : 0.0;
        const double w = rho > 0.0 ? P.fpsc / sq : 0.0;
        // the atom's energy 1/2 eps sum_j phi_n + B(rho), B = -eps c sqrt(rho)
        ((double *)S.pen)[a] = fma(-P.ec, sq, __dmul_rn(0.5 * P.eps, phn));
        ((double4_32a *)S.posfp)[a] = make_double4_32a(pa.x, pa.y, pa.z, w);
    }
}

template <int L, bool SC76>
__global__ void __launch_bounds__(TPB) k_force_f64(const SpecDev *__restrict__ specs,
                                                   const int *__restrict__ b2s, int mode) {
    const SpecDev &S = specs[b2s[blockIdx.x]];
    SpecCtl *ctl = S.ctl;
    const int phase = ctl->phase;
    if (mode == MODE_STEP && phase == PH_IDLE) return;
    const int par = ctl->parity;
    const long long done = ctl->done, nsteps = ctl->nsteps;
    constexpr int APB = TPB / L;
    const int lb = blockIdx.x - S.blk_pair0;
    const int a = lb * APB + threadIdx.x / L;
    const int l = threadIdx.x % L;
    const bool valid = a < S.n;
    const double4_32a *__restrict__ pf = (const double4_32a *)S.posfp;
    const PotDev &P = S.pot;
    double fx = 0, fy = 0, fz = 0;
    double4_32a pa = make_double4_32a(0, 0, 0, 0);
    if (valid) {
        pa = pf[a];
        for_entries64(S, pf, a, l, L, [&](const double4_32a &pj) {
            double dx, dy, dz;
            const double r2 = pair_r2(pa, pj, dx, dy, dz);
            if (within(r2, P.rc2)) {
                const double g = force_pair64<SC76>(P, r2, __dadd_rn(pa.w, pj.w));
                fx = fma(g, dx, fx);
                fy = fma(g, dy, fy);
                fz = fma(g, dz, fz);
            }
        });
    }
    fx = lane_sum<L>(fx);
    fy = lane_sum<L>(fy);
    fz = lane_sum<L>(fz);
    double ke = 0, pe = 0, rr = 0, d2 = 0, dp2 = 0;
    if (valid && l == 0) {
        chk_force(S, fx, fy, fz);
        pe = ((const double *)S.pen)[a];
        const uint8_t flag = S.flags[a];
        if (flag == FLAG_RIGHT) rr = -(S.axis == 0 ? fx : (S.axis == 1 ? fy : fz));
        double4_32a v = ((const double4_32a *)S.vel)[a];
        if (mode == MODE_EVAL) {
            ke = __dmul_rn(S.ke_fac, fma(v.z, v.z, fma(v.y, v.y, __dmul_rn(v.x, v.x))));
            ((double4_32a *)S.eval_out)[S.orig[a]] = make_double4_32a(fx, fy, fz, pe);
        } else {
            const double kh = S.acc_half;
            // thermal relaxation: the right grip moves along the load axis only
            const bool rfree = flag == FLAG_RIGHT && S.ctl->relax;
            if (phase == PH_RUN) {
                if (flag == FLAG_MOBILE) {
                    v.x = fma(fx, kh, v.x);
                    v.y = fma(fy, kh, v.y);
                    v.z = fma(fz, kh, v.z);
                } else if (rfree) {
                    if (S.axis == 0) v.x = fma(fx, kh, v.x);
                    else if (S.axis == 1) v.y = fma(fy, kh, v.y);
                    else v.z = fma(fz, kh, v.z);
                }
                ke = __dmul_rn(S.ke_fac, fma(v.z, v.z, fma(v.y, v.y, __dmul_rn(v.x, v.x))));
                if (S.rsum) {
                    // Eq. (mean_pos): the sampled state's position
                    double *rs = S.rsum + 4LL * S.orig[a];
                    rs[0] = rs[0] + pa.x;
                    rs[1] = rs[1] + pa.y;
                    rs[2] = rs[2] + pa.z;
                }
            }
            double x = pa.x, y = pa.y, z = pa.z;
            const bool start = (phase == PH_REFRESH) || (done + 1 < nsteps);
            if (start && (flag == FLAG_MOBILE || rfree)) {
                if (flag == FLAG_MOBILE) {
                    v.x = fma(fx, kh, v.x);
                    v.y = fma(fy, kh, v.y);
                    v.z = fma(fz, kh, v.z);
                } else if (S.axis == 0) {
                    v.x = fma(fx, kh, v.x);
                } else if (S.axis == 1) {
                    v.y = fma(fy, kh, v.y);
                } else {
                    v.z = fma(fz, kh, v.z);
                }
                x = fma(v.x, S.dt, x);
                y = fma(v.y, S.dt, y);
                z = fma(v.z, S.dt, z);
            } else if (start && flag == FLAG_RIGHT && !rfree && S.ctl->grip_du != 0.0) {
                // continuous loading (fine-dynamics verification)
                const double du = S.ctl->grip_du;
                if (S.axis == 0) x = x + du;
                else if (S.axis == 1) y = y + du;
                else z = z + du;
            }
            ((double4_32a *)S.pos[par ^ 1])[a] = make_double4_32a(x, y, z, 0.0);
            S.rec[par ^ 1][a] = rec_fp64(S, x, y, z);
            ((double4_32a *)S.vel)[a] = v;
            const float4 rf = S.ref[a];
            const double ex = x - rf.x, ey = y - rf.y, ez = z - rf.z;
            d2 = fma(ez, ez, fma(ey, ey, __dmul_rn(ex, ex)));
            if (S.prune_on) {
                const float4 pr = S.pref[a];
                const double qx = x - pr.x, qy = y - pr.y, qz = z - pr.z;
                dp2 = fma(qz, qz, fma(qy, qy, __dmul_rn(qx, qx)));
            }
        }
    }
    ke = warp_sum(ke);
    pe = warp_sum(pe);
    rr = warp_sum(rr);
    d2 = (double)warp_max((float)d2);
    dp2 = (double)warp_max((float)dp2);
    step_tail<TPB>(S, lb, S.nblk_pair, ke, pe, rr, d2, dp2, mode, phase, done, nsteps);
}

#define PTA_F64_SWITCH(KER, SC, ARG)                                                   \
    switch (g.L) {                                                                     \
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

}  // namespace pta
