// Pieces shared by the FP64 and mixed-precision pair kernels: warp
// reductions and the end-of-step reduction that turns per-block partials
// into the state functions K, U, T of Eq. (state_variables) for one step.
#pragma once

#include <algorithm>

#include "pta_dev.cuh"

namespace pta {

// sum over the L lanes that share one atom (lanes are contiguous in the warp)
template <typename T>
__device__ __forceinline__ T lane_sum(T v, int L) {
#pragma unroll
    for (int o = 8; o > 0; o >>= 1)
        if (o < L) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// ---------------------------------------------------------------------------
// The state functions of a step: sums over the atoms of K, U and the reaction
// R, and the largest squared displacements since the list build and since the
// pruning (quanta^2).  Sums are double in both precisions.
//
// FP64 additions run two lanes per clock and SM here (16 cycles per warp), so
// the butterflies below sum K and U in one: its first stage leaves the sums of
// K in one half of the lanes and those of U in the other, five additions for
// both instead of ten; and most warps hold no right-grip atom and skip R.
// ---------------------------------------------------------------------------
// non-negative floats order as their bits
__device__ __forceinline__ float warp_max(float v) {
    return __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(v)));
}

constexpr int PART = 4;         // doubles per partial
constexpr int PART_GROUP = 32;  // blocks per group of partials
struct StepVals {
    double s[3];    // K, U, R
    float d2, dp2;  // displacements
};
__device__ __forceinline__ double add_xor(double v, int o) {
    return __dadd_rn(v, __shfl_xor_sync(0xffffffffu, v, o));
}
// sums over the lanes whose values count, at offsets `first`, first / 2, ...
// `last`: right in lane 0 (of each 2 first lanes)
__device__ __forceinline__ void sum_lanes(double s[3], int first, int last) {
    const bool upper = threadIdx.x & first;
    double r = upper ? s[1] : s[0];
    r = __dadd_rn(r, __shfl_xor_sync(0xffffffffu, upper ? s[0] : s[1], first));
#pragma unroll
    for (int o = 8; o > 0; o >>= 1)
        if (o < first && o >= last) r = add_xor(r, o);
    s[0] = r;
    s[1] = __shfl_xor_sync(0xffffffffu, r, first);
    if (__any_sync(0xffffffffu, s[2] != 0.0)) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            if (o <= first && o >= last) s[2] = add_xor(s[2], o);
    }
}
// over the lanes of a warp whose values count (every mino-th), in lane 0
__device__ __forceinline__ void warp_reduce(StepVals &v, int mino) {
    sum_lanes(v.s, 16, mino);
    v.d2 = warp_max(v.d2);
    v.dp2 = warp_max(v.dp2);
}
// the same sums with the atoms of a tile in 32 / L adjacent lanes
__device__ __forceinline__ void tile_reduce(StepVals &v, int L) {
    sum_lanes(v.s, 16 / L, 1);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        if (o * L >= 32) continue;
        v.d2 = fmaxf(v.d2, __shfl_xor_sync(0xffffffffu, v.d2, o));
        v.dp2 = fmaxf(v.dp2, __shfl_xor_sync(0xffffffffu, v.dp2, o));
    }
}
// a partial in memory: three sums and the two maxima, 32 bytes
__device__ __forceinline__ double pack_maxima(float d2, float dp2) {
    return __hiloint2double(__float_as_int(dp2), __float_as_int(d2));
}
__device__ __forceinline__ double max_pair(double a, double b) {
    return __hiloint2double(max(__double2hiint(a), __double2hiint(b)),
                            max(__double2loint(a), __double2loint(b)));
}
__device__ __forceinline__ void load_part(const double *p, StepVals &v) {
    const double2 a = __ldcg((const double2 *)p), b = __ldcg((const double2 *)p + 1);
    v.s[0] = a.x;
    v.s[1] = a.y;
    v.s[2] = b.x;
    v.d2 = __int_as_float(__double2loint(b.y));
    v.dp2 = __int_as_float(__double2hiint(b.y));
}
__device__ __forceinline__ void store_part(double *p, const StepVals &v) {
    ((double2 *)p)[0] = make_double2(v.s[0], v.s[1]);
    ((double2 *)p)[1] = make_double2(v.s[2], pack_maxima(v.d2, v.dp2));
}
// a += b
__device__ __forceinline__ void merge(StepVals &a, const StepVals &b) {
#pragma unroll
    for (int q = 0; q < 3; ++q) a.s[q] = __dadd_rn(a.s[q], b.s[q]);
    a.d2 = fmaxf(a.d2, b.d2);
    a.dp2 = fmaxf(a.dp2, b.dp2);
}

// squared displacement of a record from an earlier one, quanta^2
__device__ __forceinline__ float moved2(const int4 &a, const int4 &b) {
    const float x = (float)rec_diff(a.x, b.x), y = (float)rec_diff(a.y, b.y),
                z = (float)rec_diff(a.z, b.z);
    return fmaf(z, z, fmaf(y, y, __fmul_rn(x, x)));
}

// The block's partial from its atoms' values, atom t of the block in thread t
// < NT / L: the atoms of each warp tile (32 / L of them) summed as a resident
// run's warp does, then the block's tiles in order.  The kernel behind the
// force pass adds the partials up and takes the step (finish_sums).  When the
// last blocks of the force pass did, every block waited at its end for its
// stores to be visible and for an atomic: a step of 12 specimens of 32,000
// atoms took 235 us instead of 219, of 470,596 atoms 223 instead of 220.
template <int NT>
__device__ __forceinline__ void block_partial(const SpecDev &S, int lb, StepVals v, int L) {
    constexpr int NW = NT / 32;
    __shared__ __align__(16) double sh[NW][PART];
    const int lane = threadIdx.x & 31, q = threadIdx.x;
    if ((threadIdx.x & ~31) < NT / L) {
        tile_reduce(v, L);
        if ((lane & (32 / L - 1)) == 0 && threadIdx.x < NT / L)
            store_part(sh[threadIdx.x / (32 / L)], v);
    }
    __syncthreads();
    if (q >= PART) return;
    // a thread per sum, and one for the maxima
    double a = sh[0][q];
#pragma unroll
    for (int k = 1; k < NW; ++k) a = q < 3 ? __dadd_rn(a, sh[k][q]) : max_pair(a, sh[k][q]);
    S.part[(long long)PART * lb + q] = a;
}

// MODE_EVAL: force and energy of atom a in the arrays of pta_forces
__device__ __forceinline__ void eval_store(const SpecDev &S, int a, double fx, double fy, double fz,
                                           double pe) {
    const int o = S.orig[a];
    double *f = S.eval_out + 3LL * o;
    f[0] = fx;
    f[1] = fy;
    f[2] = fz;
    S.eval_out[3LL * S.n + o] = pe;
}

// One thread: the specimen's control block after a step with these totals.
//   MODE_STEP, phase RUN:     sample (K, U, T) into the series, step count + 1,
//                             burst over after nsteps samples
//   MODE_STEP, phase REFRESH: forces refreshed and the first step started
//   MODE_EVAL:                K, U, T and the error bits stored behind the
//                             atoms' forces and energies
// and in MODE_STEP the position buffers swap, the skin test sets the
// rebuild flag and the pruning margin test the prune flag.
__device__ inline void advance_ctl(const SpecDev &S, double K, double U, double R, float md2,
                                   float mp2, int mode, int phase, int par, long long done,
                                   long long nsteps) {
    SpecCtl *c = S.ctl;
    const double T = R * S.t_fac;
    if (c->prune) {  // this step's passes used the pruned lists
        c->prune = 0;
        c->prunes += 1;
    }
    if (mode == MODE_EVAL) {
        double *o = S.eval_out + 4LL * S.n;
        o[0] = K;
        o[1] = U;
        o[2] = T;
        o[3] = c->err;
        c->rebuild = 0;
        return;
    }
    int now = phase;
    if (phase == PH_RUN) {
        if (!isfinite(K) || !isfinite(U) || !isfinite(T)) {
            c->err |= ERR_NAN;
            now = PH_IDLE;
        } else {
            double *o = S.series + 3 * done;
            o[0] = K;
            o[1] = U;
            o[2] = T;
            if (S.conv_lag > 0) {
                c->sum[0] = c->sum[0] + K;
                c->sum[1] = c->sum[1] + U;
                c->sum[2] = c->sum[2] + T;
            }
            c->done = done + 1;
            if (done + 1 >= nsteps) now = PH_IDLE;
            const long long i = done + 1;
            if (S.conv_lag > 0 && i % S.conv_lag == 0) {
                // appendix, Eq. (R_m_conv): e = |R^(i) - R^(i-k)| / max(|R^(i)|,
                // floor), from i = 2k on; each variable converges on its own
                if (i >= 2LL * S.conv_lag) {
                    for (int q = 0; q < 3; ++q) {
                        if (c->conv_mask & (1 << q)) continue;
                        const double a = c->sum[q] / (double)i;
                        const double b = c->sum_chk[q] / (double)(i - S.conv_lag);
                        const double e = fabs(a - b) / fmax(fabs(a), S.floor_[q]);
                        if (e < S.conv_tol[q]) {
                            c->conv_mask |= 1 << q;
                            c->conv_n[q] = i;
                            c->conv_val[q] = a;
                        }
                    }
                    if (c->conv_mask == 7) now = PH_IDLE;
                }
                for (int q = 0; q < 3; ++q) c->sum_chk[q] = c->sum[q];
            }
        }
    } else if (phase == PH_REFRESH) {
        now = PH_RUN;
    }
    c->phase = now;
    c->rebuild = md2 > S.half_skin2q;
    if (S.prune_on && mp2 > S.half_prune2q) c->prune = 1;
    c->parity = par ^ 1;
}

// Sums over the lanes of a warp of N values each (N a power of two, at most 16),
// along the butterfly of sum_lanes: every stage halves the values that a lane
// holds, until value i is in lanes (32 / N) i and on.
template <int N>
__device__ __forceinline__ double sum_transposed(double *v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 16, n = N / 2; o > 0; o >>= 1, n >>= 1) {
        if (n == 0) {
            v[0] = add_xor(v[0], o);
            continue;
        }
        const bool upper = lane & o;
#pragma unroll
        for (int i = 0; i < n; ++i) {
            const double other = __shfl_xor_sync(0xffffffffu, upper ? v[i] : v[i + n], o);
            v[i] = __dadd_rn(upper ? v[i + n] : v[i], other);
        }
    }
    return v[0];
}

// The totals of a launched step, valid in thread 0 of a block of
// 32 * FINISH_WARPS threads, from the force pass's block partials along a
// fixed tree: groups of 32 consecutive blocks (one per lane, butterfly
// shuffles), 32 groups at a time likewise, then those in order.
//
// Bound: three round trips of latency, and the FP64 additions of one SM.  A
// warp's eight groups are loaded together and summed together, in 16 additions
// of a warp instead of 40: 470,596 atoms 214.5 us per step instead of 217.5.
constexpr int FINISH_WARPS = 16, FINISH_GROUPS = 8;
__device__ __forceinline__ StepVals finish_sums(const SpecDev &S) {
    constexpr int ROUND = FINISH_WARPS * FINISH_GROUPS, G = FINISH_GROUPS;
    __shared__ StepVals sg[ROUND], sc[ROUND / 32];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nblk = S.nblk_pair, ngroups = (nblk + PART_GROUP - 1) / PART_GROUP;
    StepVals t = StepVals{};
    for (int r = 0; r < ngroups; r += ROUND) {
        StepVals a[G];
#pragma unroll
        for (int k = 0; k < G; ++k) {
            const int b = (r + w * G + k) * PART_GROUP + lane;
            a[k] = StepVals{};
            if (b < nblk) load_part(S.part + (long long)PART * b, a[k]);
        }
        if (r + w * G < ngroups) {
            double v[2 * G];
            bool reaction = false;
#pragma unroll
            for (int k = 0; k < G; ++k) {
                v[2 * k] = a[k].s[0];
                v[2 * k + 1] = a[k].s[1];
                reaction |= a[k].s[2] != 0.0;
                const float d2 = warp_max(a[k].d2), dp2 = warp_max(a[k].dp2);
                if (lane == k) {
                    sg[w * G + k].d2 = d2;
                    sg[w * G + k].dp2 = dp2;
                }
            }
            const double ku = sum_transposed<2 * G>(v);
            if ((lane & 1) == 0) sg[w * G + (lane >> 2)].s[(lane >> 1) & 1] = ku;
            double x = 0.0;
            if (__any_sync(0xffffffffu, reaction)) {
#pragma unroll
                for (int k = 0; k < G; ++k) v[k] = a[k].s[2];
                x = sum_transposed<G>(v);
            }
            if ((lane & 3) == 0) sg[w * G + (lane >> 2)].s[2] = x;
        }
        __syncthreads();
        if (w * 32 < min(ROUND, ngroups - r)) {
            StepVals u = r + w * 32 + lane < ngroups ? sg[w * 32 + lane] : StepVals{};
            if (ngroups > 1) warp_reduce(u, 1);
            if (lane == 0) sc[w] = u;
        }
        __syncthreads();
        if (threadIdx.x == 0)
            for (int k = 0; k * 32 < min(ROUND, ngroups - r); ++k) {
                if (r + k == 0) t = sc[0];
                else merge(t, sc[k]);
            }
    }
    return t;
}

// The same tree in a resident run, whose warps store their partials
// (part_warp): one warp sums group g from its blocks' warps, in the order of
// block_partial, and later one warp the groups.
__device__ __forceinline__ double *part_warp(const SpecDev &S, int tile) {
    return S.part + (long long)PART * tile;
}
__device__ __forceinline__ double *part_group(const SpecDev &S, int g) {
    return S.gpart + (long long)PART * g;
}
__device__ inline void reduce_group(const SpecDev &S, int g) {
    constexpr int NW = TPB / 32;
    const int lane = threadIdx.x & 31, blk = g * PART_GROUP + lane;
    StepVals a = StepVals{}, b[NW];
    if (blk < S.nblk_pair) {
#pragma unroll
        for (int k = 0; k < NW; ++k) load_part(part_warp(S, blk * NW + k), b[k]);
        a = b[0];
#pragma unroll
        for (int k = 1; k < NW; ++k) merge(a, b[k]);
    }
    warp_reduce(a, 1);
    if (lane == 0) store_part(part_group(S, g), a);
}
__device__ inline StepVals reduce_groups(const SpecDev &S) {
    const int lane = threadIdx.x & 31;
    const int ngroups = (S.nblk_pair + PART_GROUP - 1) / PART_GROUP;
    StepVals t = StepVals{};
    if (ngroups == 1) {
        if (lane == 0) load_part(part_group(S, 0), t);
        return t;
    }
    for (int b = 0; b < ngroups; b += 32) {
        StepVals u = StepVals{};
        if (b + lane < ngroups) load_part(part_group(S, b + lane), u);
        warp_reduce(u, 1);
        if (b == 0) t = u;
        else merge(t, u);
    }
    return t;
}

// four list entries: read once per pass, so they skip L1 (the neighbour
// records keep the space).  Between kernels (RES false) they come through the
// read-only path and ask L2 to fetch the 256-byte block around them; inside a
// resident run lists and records change between its barriers, so both are
// read with ordinary (coherent after a barrier) loads.
template <bool RES>
__device__ __forceinline__ uint4 ld_quad(const uint4 *p) {
    uint4 v;
    if (RES) {
        asm volatile("ld.global.L1::no_allocate.L2::256B.v4.u32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                     : "l"(p)
                     : "memory");
        return v;
    }
    asm("ld.global.nc.L1::no_allocate.L2::256B.v4.u32 {%0, %1, %2, %3}, [%4];"
        : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
        : "l"(p));
    return v;
}
template <bool RES>
__device__ __forceinline__ int4 ld_rec(const SpecDev &S, const void *rec, unsigned e) {
    const int4 *p = (const int4 *)((const char *)rec + nl_off(S, e));
    return RES ? *p : __ldg(p);
}

// Pruning (both precisions): every lane appends to its near entries, in
// order, the entries of its far part within the pruning radius (FP32
// distances of the records against (rc + margin)^2 with slack).  Pairs
// within rc are therefore all kept, in the order the lane sums them.
//
// Bound: the gathers of the far part's records (~118 of the ~252 entries of a
// bulk atom at the default 2 A skin).
template <bool RES>
__device__ __forceinline__ void prune_lane(const SpecDev &S, int u, int l, int L, int par) {
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
        const float dx = (float)rec_diff(x.x, ra.x), dy = (float)rec_diff(x.y, ra.y),
                    dz = (float)rec_diff(x.z, ra.z);
        if (fmaf(dz, dz, fmaf(dy, dy, dx * dx)) < rp2 && have) {
            dst[(kept >> 2) * 128 + (kept & 3)] = e;
            ++kept;
        }
    };
    uint4 e = ld_quad<RES>(p);
    for (int q = 0; q < nl; q += 4) {
        p += 32;
        const uint4 nx = ld_quad<RES>(p);
        const int4 x0 = ld_rec<RES>(S, rec, e.x), x1 = ld_rec<RES>(S, rec, e.y);
        const int4 x2 = ld_rec<RES>(S, rec, e.z), x3 = ld_rec<RES>(S, rec, e.w);
        test(true, e.x, x0);
        test(q + 1 < nl, e.y, x1);
        test(q + 2 < nl, e.z, x2);
        test(q + 3 < nl, e.w, x3);
        e = nx;
    }
    S.pnn[u * L + l] = kept;
    if (l == 0) S.pref[u] = ra;
}

// ---------------------------------------------------------------------------
// Resident runs.  A table small enough is advanced by one cooperative kernel
// of one block per SM that stays on the GPU from one list build to the next:
// every warp keeps its 32 lanes' atoms, and the passes of a step are separated
// by grid barriers instead of kernel boundaries.  With one launch each for
// the decision, the two passes and a conditional node, a step of a small
// specimen spent ~25 us between kernels.
//
// The latency of a step is that of its chain of L2 round trips (~0.5 us
// each), so whatever can is kept on the SM: the atoms' state, own record and
// density weight in registers (of the 128 a thread, which do not hold all of it
// in mixed precision: ~130 bytes are spilled to local memory), the lists and
// the descriptors in shared memory (a barrier empties L1), the step count by
// every block for itself.  What
// remains is one round of gathers per pass and two barriers.  The sums of a
// step do not hold up the next one: a service warp in every block, beside
// those that hold atoms, sums the groups of partials during the next density
// pass and the groups during the next force pass.  What the next step must
// know at once, whether an atom has moved far enough for a list build or a
// pruning, is counted in the barrier's own word.
//
// Every wait is bounded: a barrier not reached by all blocks within `limit`
// polls (seconds by default) marks the run as stuck and every block returns;
// the host reports PTA_ECUDA and refuses the specimens from then on, whose
// blocks stopped at different points of a step.
// ---------------------------------------------------------------------------
// fields of RunCtl::arrive: arrivals, and how many of them came with a request
// for a list build, a stop (a specimen failed), a pruning.  At most
// RUN_STEPS steps per launch keep every field within its bits.
constexpr int RUN_STEPS = 4000, RUN_BLOCKS = 512;
constexpr int BAR_BUILD = 22, BAR_STOP = 32, BAR_PRUNE = 42;
static_assert((2LL * RUN_STEPS + 8) * RUN_BLOCKS < (1LL << BAR_BUILD) &&
                  RUN_BLOCKS < (1 << (BAR_STOP - BAR_BUILD)) &&
                  RUN_BLOCKS < (1 << (BAR_PRUNE - BAR_STOP)) &&
                  (long long)RUN_STEPS * RUN_BLOCKS < (1LL << (64 - BAR_PRUNE)),
              "fields of the barrier word");

__device__ __forceinline__ unsigned long long ld_relaxed(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void fence_gpu() {
    asm volatile("fence.acq_rel.gpu;" ::: "memory");
}

// The grid barriers of one block of a cooperative launch; RunCtl::arrive is 0
// when the launch begins.
struct GridBarrier {
    RunCtl *rc;
    int *req;                  // shared: requests of this block's warps
    unsigned limit;            // polls before a wait is given up
    unsigned target = 0;       // thread 0
    unsigned long long seen = 0;

    // every block has arrived; returns, at the end of a step, the requests
    // (RunState) that came with it, and RUN_STUCK when the wait ran out
    __device__ __forceinline__ int sync(bool step) {
        __shared__ int sh;
        __syncthreads();
        if (threadIdx.x == 0) {
            const int r = *req;
            *req = 0;
            unsigned long long inc = 1;
            if (r & RUN_BUILD) inc += 1ULL << BAR_BUILD;
            if (r & RUN_STOP) inc += 1ULL << BAR_STOP;
            if (r & RUN_PRUNE) inc += 1ULL << BAR_PRUNE;
            target += gridDim.x;
            fence_gpu();
            atomicAdd(&rc->arrive, inc);
            unsigned polls = 0;
            unsigned long long v;
            do {
                v = ld_relaxed(&rc->arrive);
            } while ((unsigned)(v & ((1u << BAR_BUILD) - 1)) < target && ++polls < limit);
            int got = 0;
            if (polls >= limit) {
                atomicExch(&rc->stuck, 1);
                got = RUN_STUCK;
            }
            // requests come with the end of a step: the fields may grow ahead of
            // this block in the step's first barrier, and stand still here until
            // it has arrived at the next step's
            if (step) {
                const unsigned long long d = (v >> BAR_BUILD) ^ (seen >> BAR_BUILD);
                seen = v;
                if (d & ((1ULL << (BAR_STOP - BAR_BUILD)) - 1)) got |= RUN_BUILD;
                if ((d >> (BAR_STOP - BAR_BUILD)) & ((1ULL << (BAR_PRUNE - BAR_STOP)) - 1))
                    got |= RUN_STOP;
                if (d >> (BAR_PRUNE - BAR_BUILD)) got |= RUN_PRUNE;
            }
            fence_gpu();
            sh = got;
        }
        __syncthreads();
        return sh;
    }
};

constexpr int RESIDENT_SPECS = 8;  // specimens whose tiles one block may hold

__device__ __forceinline__ void load_specs(SpecDev *sh, const SpecDev *specs, int ns) {
    for (int i = threadIdx.x; i < ns * (int)(sizeof(SpecDev) / 4); i += blockDim.x)
        ((int *)sh)[i] = ((const int *)specs)[i];
}
// passes until the last specimen's burst is over (every warp for itself)
__device__ __forceinline__ int run_passes(const SpecDev *specs, int nspec) {
    long long passes = 0;
    for (int s = threadIdx.x & 31; s < nspec; s += 32) {
        const SpecCtl *q = specs[s].ctl;
        const int ph = __ldcg(&q->phase);
        if (ph != PH_IDLE)
            passes = max(passes, __ldcg(&q->nsteps) - __ldcg(&q->done) + (ph == PH_REFRESH));
    }
    return (int)__reduce_max_sync(0xffffffffu, (unsigned)min(passes, (long long)RUN_STEPS));
}
// one warp, at the end of a launch: does any specimen go on?
__device__ __forceinline__ void run_again(const SpecDev *specs, int nspec, int state,
                                          cudaGraphConditionalHandle again) {
    const int lane = threadIdx.x & 31;
    int active = 0;
    for (int s = lane; s < nspec; s += 32) active |= __ldcg(&specs[s].ctl->phase) != PH_IDLE;
    active = __any_sync(0xffffffffu, active);
    if (lane == 0) cudaGraphSetConditional(again, active && !(state & RUN_STUCK) ? 1u : 0u);
}
// one lane: what a warp's displacements after pass `it` ask for
__device__ __forceinline__ void step_requests(const SpecDev &S, const StepVals &v, int it,
                                              int *requests) {
    int r = 0;
    if (v.d2 > S.half_skin2q) {
        r = RUN_BUILD;
        S.ctl->rebuild = 1;
    }
    if (S.prune_on && v.dp2 > S.half_prune2q) {
        r |= RUN_PRUNE;
        S.ctl->prune_at = it;
    }
    if (r) atomicOr(requests, r);
}

// The service warp of a block: the sums of the groups that begin in its tiles,
// and the control blocks of the specimens that do.  The phase and step count
// there are those of the sums, one step behind the atoms.
struct Service {
    const SpecDev *sh;  // the block's specimens
    int ns, t0, t1;
    int *requests;
    template <class F>
    __device__ __forceinline__ void each(F f) const {  // f(specimen, group)
        constexpr int NW = TPB / 32, GT = NW * PART_GROUP;
        for (int k = 0; k < ns; ++k) {
            const int base = sh[k].blk_run0 * NW, end = base + sh[k].nblk_pair * NW;
            const int a = max(t0, base) - base, b = min(t1, end) - base;
            for (int g = (a + GT - 1) / GT; g * GT < b; ++g) f(sh[k], g);
        }
    }
    __device__ __forceinline__ void start() const {
        each([&](const SpecDev &D, int g) {
            if (g == 0 && (threadIdx.x & 31) == 0) {
                D.ctl->rebuild = 0;  // asked for the build before this launch
                D.ctl->prune_at = -1;
            }
        });
    }
    __device__ __forceinline__ void reduce() const {
        each([&](const SpecDev &D, int g) {
            if (__ldcg(&D.ctl->phase) != PH_IDLE) reduce_group(D, g);
        });
    }
    __device__ __forceinline__ void finish() const {
        each([&](const SpecDev &D, int g) {
            SpecCtl *q = D.ctl;
            const int ph = __ldcg(&q->phase);
            if (g != 0 || ph == PH_IDLE) return;
            const StepVals t = reduce_groups(D);
            if ((threadIdx.x & 31) != 0) return;
            if (ph == PH_REFRESH) {
                q->phase = PH_RUN;
                return;
            }
            const double K = t.s[0], U = t.s[1], X = t.s[2] * D.t_fac;
            const long long i = __ldcg(&q->done);
            if (isfinite(K) && isfinite(U) && isfinite(X)) {
                double *o = D.series + 3 * i;
                o[0] = K;
                o[1] = U;
                o[2] = X;
                q->done = i + 1;
                if (i + 1 >= __ldcg(&q->nsteps)) q->phase = PH_IDLE;
            } else {
                atomicOr(&q->err, ERR_NAN);
                q->phase = PH_IDLE;
                atomicOr(requests, RUN_STOP);
            }
        });
        __syncwarp();
    }
};

// A block of a resident run: contiguous warp tiles of the table (tile 4 b + k:
// warp k of pair block b), one per warp, and the service warp behind them.
// OPS (one precision and lane count): a warp's part of the passes.  Its atoms'
// positions and velocities stay in registers from the launch to its end.
template <class OPS>
__device__ __forceinline__ void run_resident(const SpecDev *specs, int nspec, const int *b2s,
                                             int nblk, RunCtl *rc,
                                             cudaGraphConditionalHandle again, unsigned polls,
                                             OPS &ops) {
    constexpr int NW = TPB / 32;
    __shared__ SpecDev sh[RESIDENT_SPECS];
    __shared__ int requests;
    const int ntile = nblk * NW, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int t0 = (int)((long long)ntile * blockIdx.x / gridDim.x);
    const int t1 = (int)((long long)ntile * (blockIdx.x + 1) / gridDim.x);
    const int s0 = b2s[t0 / NW];  // tiles run through the specimens in order
    const int ns = b2s[(t1 - 1) / NW] - s0 + 1;
    load_specs(sh, specs + s0, ns);
    if (threadIdx.x == 0) requests = 0;
    __syncthreads();
    const int tile = t0 + w;
    const bool has = tile < t1;
    const bool service = w == (int)(blockDim.x >> 5) - 1;
    const SpecDev &S = sh[(has ? b2s[tile / NW] : s0) - s0];
    const int local = tile - S.blk_run0 * NW;  // tile of the specimen
    SpecCtl *c = S.ctl;
    // the burst as every warp follows it for its own specimen
    int phase = has ? __ldcg(&c->phase) : (int)PH_IDLE, par = __ldcg(&c->parity);
    bool prune = phase != PH_IDLE && S.prune_on && __ldcg(&c->prune);
    long long done = __ldcg(&c->done);
    const long long nsteps = __ldcg(&c->nsteps);
    const bool mine = phase != PH_IDLE;
    if (mine) ops.load(S, local, par);
    const int limit = run_passes(specs, nspec);
    const Service sums{sh, ns, t0, t1, &requests};
    if (service) sums.start();
    GridBarrier bar{rc, &requests, polls};
    int state = 0, it = 0;
    for (; it < limit && !(state & (RUN_BUILD | RUN_STUCK)); ++it) {
        const bool run = phase != PH_IDLE, pruned = run && prune;
        if (pruned) ops.prune(S, par);
        if (run) ops.density(S, par);
        if (service && it > 0) sums.reduce();
        state = bar.sync(false);
        if (state & RUN_STUCK) break;
        // cleared behind the barrier: by then every block has begun, and each
        // warp has read the flag that it began with
        if (pruned && local == 0 && lane == 0) {
            c->prunes = __ldcg(&c->prunes) + 1;
            c->prune = 0;
        }
        if (run) {
            const StepVals v = ops.force(S, local, par, phase, done, nsteps);
            if (lane == 0) step_requests(S, v, it, &requests);
            par ^= 1;
            done += phase == PH_RUN;
            phase = done < nsteps ? PH_RUN : PH_IDLE;
        }
        if (service && it > 0) sums.finish();
        state = bar.sync(true);
        // of several specimens, which one asked?
        prune = (state & RUN_PRUNE) && S.prune_on && (nspec == 1 || __ldcg(&c->prune_at) == it);
        if (state & RUN_STOP) {
            if (nspec == 1) break;
            if (__ldcg(&c->phase) == PH_IDLE) phase = PH_IDLE;
        }
    }
    // the last step's sums
    if (!(state & RUN_STUCK) && it > 0) {
        if (service) sums.reduce();
        state |= bar.sync(false) & RUN_STUCK;
        if (service) sums.finish();
    }
    if (mine) {
        ops.store(S, par);
        if (local == 0 && lane == 0) {
            c->parity = par;
            if (prune) c->prune = 1;
        }
    }
    state |= bar.sync(false) & RUN_STUCK;
    if (blockIdx.x == 0 && w == 0) run_again(specs, nspec, state, again);
}

// A block of a run over a larger table: contiguous tiles again, handed out one
// at a time, as a block's warps may have more than one each; the atoms' state
// and the lists stay in memory.  Against launched passes it has no launches and
// no conditional node per step (~25 us of it on a specimen of 108,000 atoms).
// Where it stops paying: run_shape.
struct SpecRun {
    int phase, par, prune;
    long long done, nsteps;
};
template <class OPS>
__device__ __forceinline__ void run_sweep(const SpecDev *specs, int nspec, const int *b2s, int nblk,
                                          RunCtl *rc, cudaGraphConditionalHandle again,
                                          unsigned polls, const OPS &ops) {
    constexpr int NW = TPB / 32;
    __shared__ SpecDev sh[RESIDENT_SPECS];
    __shared__ SpecRun run[RESIDENT_SPECS];
    __shared__ int requests, next[2];
    const int ntile = nblk * NW, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int t0 = (int)((long long)ntile * blockIdx.x / gridDim.x);
    const int t1 = (int)((long long)ntile * (blockIdx.x + 1) / gridDim.x);
    const int s0 = b2s[t0 / NW], ns = b2s[(t1 - 1) / NW] - s0 + 1;
    load_specs(sh, specs + s0, ns);
    if (threadIdx.x == 0) requests = next[0] = next[1] = 0;
    __syncthreads();
    // the burst of each specimen of this block, kept by a thread of its own
    const int k = threadIdx.x;
    const bool keeper = k < ns;
    const bool owner = keeper && sh[k].blk_run0 * NW >= t0;  // holds its first tile
    if (keeper) {
        const SpecCtl *c = sh[k].ctl;
        run[k].phase = __ldcg(&c->phase);
        run[k].par = __ldcg(&c->parity);
        run[k].prune = run[k].phase != PH_IDLE && sh[k].prune_on && __ldcg(&c->prune);
        run[k].done = __ldcg(&c->done);
        run[k].nsteps = __ldcg(&c->nsteps);
    }
    const bool active0 = keeper && run[k].phase != PH_IDLE;
    const int limit = run_passes(specs, nspec);
    const Service sums{sh, ns, t0, t1, &requests};
    const bool service = w == 0;
    if (service) sums.start();
    __syncthreads();
    auto each_tile = [&](int *ticket, auto f) {  // f(specimen of the block, its tile)
        for (;;) {
            int i = 0;
            if (lane == 0) i = atomicAdd(ticket, 1);
            i = __shfl_sync(0xffffffffu, i, 0) + t0;
            if (i >= t1) break;
            const int s = ns == 1 ? 0 : b2s[i / NW] - s0;
            if (run[s].phase != PH_IDLE) f(s, i - sh[s].blk_run0 * NW);
            __syncwarp();
        }
    };
    GridBarrier bar{rc, &requests, polls};
    int state = 0, it = 0;
    for (; it < limit && !(state & (RUN_BUILD | RUN_STUCK)); ++it) {
        if (service && it > 0) sums.reduce();
        each_tile(&next[0], [&](int s, int tile) {
            if (run[s].prune) ops.prune(sh[s], tile, run[s].par);
            ops.density(sh[s], tile, run[s].par);
        });
        state = bar.sync(false);
        if (state & RUN_STUCK) break;
        if (threadIdx.x == 0) next[0] = 0;
        if (service && it > 0) sums.finish();
        each_tile(&next[1], [&](int s, int tile) {
            const SpecDev &S = sh[s];
            const StepVals v = ops.force(S, tile, run[s].par, run[s].phase, run[s].done,
                                            run[s].nsteps);
            if (lane == 0) step_requests(S, v, it, &requests);
        });
        state = bar.sync(true);
        if (threadIdx.x == 0) next[1] = 0;
        if (keeper && run[k].phase != PH_IDLE) {
            SpecCtl *c = sh[k].ctl;
            if (run[k].prune && owner) {
                c->prunes = __ldcg(&c->prunes) + 1;
                c->prune = 0;
            }
            run[k].par ^= 1;
            run[k].done += run[k].phase == PH_RUN;
            run[k].phase = run[k].done < run[k].nsteps ? PH_RUN : PH_IDLE;
            run[k].prune = (state & RUN_PRUNE) && sh[k].prune_on &&
                           (nspec == 1 || __ldcg(&c->prune_at) == it);
            if ((state & RUN_STOP) && __ldcg(&c->phase) == PH_IDLE) run[k].phase = PH_IDLE;
        }
        __syncthreads();
        if ((state & RUN_STOP) && nspec == 1) break;
    }
    // the last step's sums
    if (!(state & RUN_STUCK) && it > 0) {
        if (service) sums.reduce();
        state |= bar.sync(false) & RUN_STUCK;
        if (service) sums.finish();
    }
    if (owner && active0) {
        sh[k].ctl->parity = run[k].par;
        if (run[k].prune) sh[k].ctl->prune = 1;
    }
    state |= bar.sync(false) & RUN_STUCK;
    if (blockIdx.x == 0 && w == 0) run_again(specs, nspec, state, again);
}

// f(entry) for the entries of a lane's column whose first `cached` quads lie
// in shared memory
struct LaneList {
    const uint4 *p;    // column in memory
    const uint4 *sh;   // this thread's column in shared memory
    int cnt, cached;
    __device__ __forceinline__ void fill(const SpecDev &S, uint4 *cache, int u, int l, int L,
                                         int quads) {
        p = S.plist + nl_col(u, l, L, S.capq);
        cnt = chk_count(S, __ldcg(S.pnn + u * L + l), 4 * (S.capq - 1));
        cached = min((cnt + 3) >> 2, quads);
        uint4 *own = cache + (threadIdx.x >> 5) * quads * 32 + (threadIdx.x & 31);
        sh = own;
        for (int t = 0; t < cached; ++t) own[t * 32] = __ldcg(p + t * 32);
    }
    __device__ __forceinline__ uint4 quad(int t) const {
        return t < cached ? sh[t * 32] : __ldcg(p + t * 32);
    }
};

// The launch shape of a run over nblk pair blocks, one block per SM.  A warp
// per tile, and a service warp, if that is at most RUN_WARPS warps; as many
// quads of the lists in shared memory as it holds (up to the ~150 entries of a
// bulk atom).  Else, up to SWEEP_TILES tiles per SM, a sweep of at most
// sweep_warps warps: of those counts the one whose last round of tiles is
// fullest.  Larger tables fill the GPU for several waves, and launched passes,
// with 32 warps per SM and the read-only path, are faster; in mixed precision
// so are they where the last of several rounds would leave more than a tenth
// of the warps idle (`full` = 0.9).  Per step, mixed: 27 tiles per SM 71 us
// (launched 82), 30 tiles 106 (90), 36 tiles 112 (101), 39 tiles 114 (116), 53
// tiles 132 (134), 97 tiles 253 (225).  FP64 passes keep the FP64 units busy
// with fewer warps: 36 tiles 1,885 us (1,992), 53 tiles 2,778 (2,886).
constexpr int RUN_WARPS = 16, SWEEP_TILES = 56;
struct RunShape {
    int blocks = 0, threads = 0, quads = 0;
    size_t smem = 0;
    bool sweep = false;
};
inline RunShape run_shape(int nblk, int min_lanes, int sweep_warps, double full) {
    RunShape r;
    int dev = 0, nsm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        cudaGetLastError();
        return r;
    }
    nsm = std::min(nsm, RUN_BLOCKS);
    if (nsm < 1) return r;
    const int tiles = nblk * (TPB / 32);
    r.blocks = std::min(nsm, tiles);
    const int per = (tiles + r.blocks - 1) / r.blocks;
    if (per + 1 <= RUN_WARPS) {
        r.threads = 32 * (per + 1);
        r.quads = std::min(40 / min_lanes + 2, 160 * 1024 / (r.threads * 16));
        r.smem = (size_t)r.quads * r.threads * 16;
        return r;
    }
    if (per > SWEEP_TILES) return RunShape();
    r.sweep = true;
    int best = sweep_warps;
    auto slots = [&](int w) { return (per + w - 1) / w * w; };
    for (int w = sweep_warps; w >= sweep_warps * 3 / 4; --w)
        if (slots(w) < slots(best)) best = w;
    if (per > sweep_warps && per < full * slots(best)) return RunShape();
    r.threads = 32 * best;
    return r;
}
template <class K>
bool run_fits(K kernel, const RunShape &r) {
    int per = 0;
    if (r.blocks < 1) return false;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024) !=
            cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, r.threads, r.smem) !=
            cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return per >= 1;
}
template <class K, class... A>
cudaError_t launch_cooperative(K kernel, const RunShape &r, cudaStream_t st, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.dynamicSmemBytes = r.smem;
    cfg.gridDim = dim3((unsigned)r.blocks);
    cfg.blockDim = dim3((unsigned)r.threads);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

}  // namespace pta
