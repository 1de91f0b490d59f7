// Device pieces of the mixed-precision pair kernels: the FP32 pair terms of
// the Sutton-Chen EAM (Eqs. (pe), (f_int)), the exact hi/lo velocity pair,
// and the per-atom velocity-Verlet update of Eqs. (vv_algo_*) fused behind
// the force pass.
//
// Precision: pair terms in FP32 on exact differences of fixed-point records;
// positions are an exact FP32 pair x = hi + lo (hi on a 2^-12 A grid, |lo| <=
// 2^-13 A); velocities an exact FP32 pair v = vh + vl (|vl| <= ulp(vh) / 2) updated by
// error-free addition, so that half-kicks lose nothing to rounding over long
// bursts; K, U and R are converted to FP64 per atom and
// summed in FP64.
#pragma once

#include "k_pair_common.cuh"

namespace pta {

// hardware estimates without the subnormal handling of rsqrtf / division
// (three instructions of each pair's terms): relative errors at most 2^-22.9
// and 2^-23; an infinite argument gives 0
__device__ __forceinline__ float rsq_approx(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float powi(float s, int k) {
    float p = 1.f;
    for (int i = 0; i < k; ++i) p = __fmul_rn(p, s);
    return p;
}

// Squared distance (A^2) of a neighbour's record from the atom's, and the
// displacement in quanta (q2: square of the quantum).
__device__ __forceinline__ float pair_r2(float q2, const int4 &a, const int4 &b, float &dx,
                                         float &dy, float &dz) {
    dx = (float)rec_diff(b.x, a.x);
    dy = (float)rec_diff(b.y, a.y);
    dz = (float)rec_diff(b.z, a.z);
    return __fmul_rn(fmaf(dz, dz, fmaf(dy, dy, __fmul_rn(dx, dx))), q2);
}

// A pair beyond rc gets y = 1/r = 0 (the force pass) or r^2 = infinity, whose
// estimates are 0 (the density pass), which makes every term exactly zero: no
// branch, and no trace of such pairs in the sums.
//
// Bound: instruction dispatch (an FP32 multiply-add of three registers takes
// 1.5 cycles of it; packed FP32 instructions take 2-3 and gave nothing), ~25
// and ~34 instructions per entry.  How the powers of 1/r are formed decides
// the accuracy.  Velocities after 300 steps of the 32,000-atom cube are off by
// 4.6e-7 of their norm in this form; by 6.1e-7 with both passes' powers
// raised from a Newton-refined 1/r (as many instructions in the force pass,
// four more in the density pass), and by 6.9e-7 with plain estimates in the
// force pass as well: an estimate's error changes slowly with r, so it acts
// on a pair in the same direction for many steps.

// density pass, one pair: sums of (1/r)^n, r and the pair count, from which
// phi_n = a^n (1/r)^n - A_n + B_n (r - rc) is assembled once per atom, and of
// (1/r)^m, assembled likewise for the Sutton-Chen exponents (m = 6: the sum is
// far larger than what is taken off it), or of phi_m itself
struct RhoSums {
    float sm = 0.f, sn = 0.f, sr = 0.f;
    int cnt = 0;
};
template <bool SC76>
__device__ __forceinline__ void rho_pair(const PotF &P, float q2, const int4 &a, const int4 &b,
                                         RhoSums &s) {
    float dx, dy, dz;
    const float r2 = pair_r2(q2, a, b, dx, dy, dz);
    const bool in = r2 < P.rc2;
    if (SC76) {
        const float rm = in ? r2 : __int_as_float(0x7f800000);
        const float u = rcp_approx(rm), y = rsq_approx(rm);
        const float u3 = __fmul_rn(__fmul_rn(u, u), u);
        s.sm = __fadd_rn(s.sm, u3);
        s.sn = fmaf(u3, y, s.sn);
        s.sr = fmaf(r2, y, s.sr);
    } else {
        float y = rsq_approx(r2);
        y = in ? y : 0.f;
        y = fmaf(0.5f * y, fmaf(-r2, y * y, 1.f), y);
        const float phi = __fadd_rn(powi(__fmul_rn(P.a, y), P.m), -P.Am);
        s.sm = __fadd_rn(s.sm, in ? fmaf(P.Bm, fmaf(r2, y, -P.rc), phi) : 0.f);
        s.sn = __fadd_rn(s.sn, powi(y, P.n));
        s.sr = fmaf(r2, y, s.sr);
    }
    s.cnt += in;
}

// force pass, one pair: with q = w_i + w_j where each record carries
// w = m a^m B'(rho),
//   [eps phi_n'(r) + (B'_i + B'_j) phi_m'(r)] / r
//       = y (eps Bn + q Bm / (m a^m)) - y^(m+2) (q + eps n a^n y^(n-m))
// (n = 7, m = 6: y^8 = u^4)
template <bool SC76>
__device__ __forceinline__ void force_pair(const PotF &P, float q2, const int4 &a, float wa,
                                           const int4 &b, float &fx, float &fy, float &fz) {
    float dx, dy, dz;
    const float r2 = pair_r2(q2, a, b, dx, dy, dz);
    const float q = wa + __int_as_float(b.w);
    const float c = fmaf(q, P.bmq, P.ebn);
    float y = rsq_approx(r2), v;
    y = r2 < P.rc2 ? y : 0.f;
    // one Newton-Raphson step on both 1/r^2 and 1/r from the same residual
    const float y2 = y * y, e = fmaf(-r2, y2, 1.f);
    y = fmaf(0.5f * y, e, y);
    if (SC76) {
        const float u = fmaf(y2, e, y2), u2 = u * u;
        v = (u2 * u2) * fmaf(P.kn, y, q);
    } else {
        const float ym = powi(y, P.m), yn = powi(y, P.n);
        v = (y * y) * fmaf(q, ym, P.kn * yn);
    }
    const float g = fmaf(y, c, -v);
    fx = fmaf(g, dx, fx);
    fy = fmaf(g, dy, fy);
    fz = fmaf(g, dz, fz);
}

// (h, l) += d exactly up to the final renormalisation: Knuth's two-sum of h
// and d, its error added to l, then h + l renormalised (fast two-sum, valid
// since |l| is far below |h + d| or both are tiny)
__device__ __forceinline__ void hl_add(float &h, float &l, float d) {
    const float s = h + d;
    const float bb = s - h;
    const float e = (h - (s - bb)) + (d - bb);
    const float t = l + e;
    const float hh = s + t;
    l = t - (hh - s);
    h = hh;
}

// An atom's state outside the neighbour records.
struct AtomMixed {
    float vh[3], vl[3], hi[3], lo[3];
    int4 ref, pref;
    int flag;
    __device__ __forceinline__ void load(const SpecDev &S, int par, int a) {
        const VelHL v = ((const VelHL *)S.vel)[a];
        const float4 h = ((const float4 *)S.pos[par])[a], l = S.lo[par][a];
        vh[0] = v.h.x; vh[1] = v.h.y; vh[2] = v.h.z;
        vl[0] = v.l.x; vl[1] = v.l.y; vl[2] = v.l.z;
        hi[0] = h.x; hi[1] = h.y; hi[2] = h.z;
        lo[0] = l.x; lo[1] = l.y; lo[2] = l.z;
        ref = S.ref[a];
        pref = S.prune_on ? S.pref[a] : ref;
        flag = S.flags[a];
    }
    __device__ __forceinline__ void store(const SpecDev &S, int par, int a) const {
        VelHL v;
        v.h = make_float4(vh[0], vh[1], vh[2], 0.f);
        v.l = make_float4(vl[0], vl[1], vl[2], 0.f);
        ((VelHL *)S.vel)[a] = v;
        ((float4 *)S.pos[par])[a] = make_float4(hi[0], hi[1], hi[2], 0.f);
        S.lo[par][a] = make_float4(lo[0], lo[1], lo[2], 0.f);
    }
};

// After the force pass of atom a (force f; its energy pe from the density
// pass): its share of the state functions, and the velocity-Verlet update --
// the half-kick that finishes the step (phase RUN), the sample of K, and
// unless the burst ends the half-kick and drift of the next step; the new
// position (hi + lo, whole grid quanta moved from lo to hi), its neighbour
// record (returned), and the displacements since the last list build and the last
// pruning.  Grip atoms keep v = 0.  MODE_EVAL stores F and the energy
// instead.  Sums and products are written as the operations meant, so that
// every kernel this is compiled into rounds alike.
__device__ __forceinline__ int4 atom_update_mixed(const SpecDev &S, AtomMixed &A, int par, int a,
                                                  const float f[3], float pe, int mode, int phase,
                                                  long long done, long long nsteps,
                                                  StepVals &out) {
    chk_force(S, f[0], f[1], f[2]);
    SpecCtl *ctl = S.ctl;
    out.s[1] = (double)pe;
    if (A.flag == FLAG_RIGHT)
        out.s[2] = (double)-(S.axis == 0 ? f[0] : (S.axis == 1 ? f[1] : f[2]));
    auto kinetic = [&] {
        const float x = A.vh[0] + A.vl[0], y = A.vh[1] + A.vl[1], z = A.vh[2] + A.vl[2];
        out.s[0] = (double)__fmul_rn(S.f_ke_fac, fmaf(z, z, fmaf(y, y, __fmul_rn(x, x))));
    };
    if (mode == MODE_EVAL) {
        kinetic();
        eval_store(S, a, f[0], f[1], f[2], pe);
        return make_int4(0, 0, 0, 0);
    }
    // thermal relaxation: the right grip moves along the load axis only (its
    // other velocity components stay 0, so the drift leaves them in place)
    const bool rfree = A.flag == FLAG_RIGHT && ctl->relax;
    const bool moves = A.flag == FLAG_MOBILE || rfree;
    float k[3];
#pragma unroll
    for (int d = 0; d < 3; ++d)
        k[d] = (A.flag == FLAG_MOBILE || (rfree && S.axis == d)) ? __fmul_rn(f[d], S.f_acc_half)
                                                                 : 0.f;
    if (phase == PH_RUN) {
        if (moves) {
#pragma unroll
            for (int d = 0; d < 3; ++d) hl_add(A.vh[d], A.vl[d], k[d]);
        }
        kinetic();
        if (S.rsum) {
            // Eq. (mean_pos): the sampled state's position, hi + lo exactly
            double *rs = S.rsum + 4LL * S.orig[a];
#pragma unroll
            for (int d = 0; d < 3; ++d) rs[d] = rs[d] + ((double)A.hi[d] + (double)A.lo[d]);
        }
    }
    const bool start = (phase == PH_REFRESH) || (done + 1 < nsteps);
    // continuous loading (fine-dynamics verification): a fixed right grip
    // moves by grip_du along the load axis with every step's drift
    const float gdu =
        (start && A.flag == FLAG_RIGHT && !rfree) ? (float)ctl->grip_du : 0.f;
    if (start && (moves || gdu != 0.f)) {
        if (moves) {
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                hl_add(A.vh[d], A.vl[d], k[d]);
                A.lo[d] = fmaf(A.vh[d] + A.vl[d], S.f_dt, A.lo[d]);
            }
        } else {
#pragma unroll
            for (int d = 0; d < 3; ++d) A.lo[d] += S.axis == d ? gdu : 0.f;
        }
        bool far = false;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            // move whole grid quanta from lo to hi (both steps exact)
            const float sh = __fmul_rn(rintf(A.lo[d] * (float)HI_SCALE), (float)HI_QUANTUM);
            A.hi[d] = __fadd_rn(A.hi[d], sh);
            A.lo[d] = __fsub_rn(A.lo[d], sh);
            far |= fabsf(A.hi[d]) > (float)MIXED_RANGE;
        }
        if (far) atomicOr(&ctl->err, ERR_RANGE);
    }
    const int4 r = rec_mixed(S, A.hi[0], A.hi[1], A.hi[2], A.lo[0], A.lo[1], A.lo[2]);
    S.rec[par ^ 1][a] = r;
    out.d2 = moved2(r, A.ref);
    out.dp2 = moved2(r, A.pref);
    return r;
}

}  // namespace pta
