// Device-side data structures of the fine-burst engine.
//
// One specimen on the device is described by a SpecDev (sizes, constants,
// pointers) and a SpecCtl (the mutable control block the kernels update).
// Kernels take an array of SpecDev plus a block->specimen table, so a single
// launch advances one specimen or a whole batch of them: the block's
// specimen is specs[b2s[blockIdx.x]] and its block index inside that
// specimen is blockIdx.x - first block of that specimen.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "pta.h"

namespace pta {

constexpr int TPB = 128;        // threads per block of the atom and pair kernels
constexpr int CELL_SPLIT = 4;   // cells along x per cell edge along y and z, where divided
constexpr int SCAN_THREADS = 1024;
constexpr int BUILD_WARPS = 4;  // warps per block of the list build
constexpr int NEIGH_CAP_MOST = 4096;  // largest capacity that can be asked for
// The list build's words per warp: candidates, near part in list order, class
// counters.  Up to NEIGH_CAP_MOST entries they lie in shared memory; automatic
// capacities can be larger (a list radius beyond ~22 A in aluminium), and then
// they lie in memory, for at most BUILD_SCRATCH_BLOCKS blocks.
__host__ __device__ constexpr int build_words(int cap) { return 2 * cap + 128 + 16; }
constexpr int BUILD_SMEM_MOST = BUILD_WARPS * 4 * build_words(NEIGH_CAP_MOST);
constexpr int BUILD_SCRATCH_BLOCKS = 608;

// grid quantum of the mixed-precision position split x = hi + lo:
// hi is a multiple of 2^-12 A (exact in FP32 for |x| < 512 A), |lo| <= 2^-13 A
constexpr double HI_SCALE = 4096.0;
constexpr double HI_QUANTUM = 1.0 / 4096.0;
constexpr double MIXED_RANGE = 511.0;

enum Phase : int { PH_IDLE = 0, PH_REFRESH = 1, PH_RUN = 2 };
// ERR_GRID: an atom lay beyond the cell grid's margin at a list build (it is
// binned onto the nearest border cell, which keeps the pair search complete);
// ERR_CHECK: a debug build's index or count test failed
enum ErrBit : int { ERR_OVERFLOW = 1, ERR_NAN = 2, ERR_RANGE = 4, ERR_GRID = 8, ERR_CHECK = 16 };

// Debug builds (compiled with -DPTA_CHECK=1) test every atom, cell-slot and
// list index before the access it feeds, every list count against the
// list's capacity, the cell occupancy against the atom count, and every
// atom's force for finiteness; a failed test sets ERR_CHECK (ERR_NAN for a
// force) and the access goes to index 0 instead, so a debug build never
// reads or writes out of bounds.  Production builds compile the tests away.
#ifndef PTA_CHECK
#define PTA_CHECK 0
#endif
// mixed precision: velocity as an exact FP32 pair v = h + l
struct __align__(32) VelHL {
    float4 h, l;
};
enum Mode : int { MODE_STEP = 0, MODE_EVAL = 1 };
enum AtomFlag : uint8_t { FLAG_MOBILE = 0, FLAG_LEFT = 1, FLAG_RIGHT = 2 };

// Sutton-Chen potential with the shifted-force cut, in both precisions.
//   phi_k(r)  = s^k - A_k + B_k (r - rc),   s = a/r, A_k = (a/rc)^k, B_k = k A_k / rc
//   phi_k'(r) = -k s^k / r + B_k
struct PotDev {
    double eps, c, a, rc, rc2, An, Bn, Am, Bm, ec;
    double an, am, kn, bmq, ebn, fpsc;  // as in PotF, in FP64
    double am_lo, fpsc_rel;  // what rounding took off am; off fpsc, relative to it
    int n, m;
    float f_eps, f_a, f_rc, f_rc2, f_An, f_Bn, f_Am, f_Bm, f_ec;
    int sc76;  // 1 when (n, m) == (7, 6): the fast specialised kernels apply
};

// FP32 constants of the pair terms, passed by value to the mixed-precision
// pair kernels: read from the kernel's constant bank at every use, they cost
// no load and no register inside the pair loops
struct PotF {
    float a, rc, rc2, Am, Bm, An, Bn, eps, ec;
    // force pass (the record's fourth component is w = m a^m B'(rho)):
    float an;    // a^n
    float am;    // a^m (density pass)
    float kn;    // eps n a^n
    float bmq;   // Bm / (m a^m)
    float ebn;   // eps Bn
    float fpsc;  // -eps c m a^m / 2: w = fpsc / sqrt(rho) (density pass)
    int n, m;
};

// slow-variable record of the coarse-step logic (FP64)
struct PtaDev {
    double v[3], R_t[3], R_tmD[3], R_tmh[3];
    double R3[3][3];  // means of the last three bursts, by slot
    double t;
    int has_tmh, init, jump[3], pad;
};

struct SpecCtl {
    int phase;       // Phase
    int parity;      // which position buffer is current
    int rebuild;     // 1: build the neighbour list before the next pair pass
    int err;         // sticky ErrBit mask
    long long nsteps, done;
    int list_L;                // lanes the current list layout was built for
    int rebuilds;              // list builds in the current burst
    int max_nn;                // largest neighbour count at the last build
    int prune;                 // 1: prune the inner list before the next pair pass
    int prunes;                // prunings in the current burst
    int prune_at;              // resident runs: pass after which a pruning was asked for
    double sum[3];             // running sums of K, U, T over the burst (in step order)
    double sum_chk[3];         // adaptive length: running sums at the last check
    double conv_val[3];        // adaptive length: running average at convergence
    long long conv_n[3];       // adaptive length: step of convergence per variable
    int conv_mask;             // adaptive length: bit m set once variable m converged
    int relax;                 // 1: thermal relaxation, right grip free along the load axis
    double grip_du;            // continuous loading: the right grip moves this far (A) along
                               // the load axis with every step (0: held fixed)
    double mb[8];              // scratch of the Maxwell-Boltzmann set-up
    pta_averages last;         // averages of the last finished burst
    PtaDev pta;
};

struct SpecDev {
    // sizes
    int n, L, prec, axis;
    int cap_use;               // list capacity: entries per atom
    int capq;                  // quads per lane column of a list
    int blk_pair0, nblk_pair;  // pair kernels: TPB/L atoms per block (first in its group)
    int blk_run0;              // first pair block in the table (resident runs, sweeps)
    int blk_atom0, nblk_atom;  // one thread per atom
    int blk_bld0, nblk_bld;    // list build: BUILD_WARPS warps of apw atoms
    int apw;
    unsigned *bld_scratch;     // build_words(cap_use) words per warp, or null: in shared memory
    int spec_index;            // index of this specimen in the launch table
    // lattice (creation only)
    int ncl[3];
    double a0, grip_width;
    // cell grid
    double org[3];
    double inv_h, inv_hx;      // cell edges along y and z, along x
    int nc[3];
    int ncell;
    // list radius (rc + skin)^2
    double rl2;
    float f_h, f_hx, f_inv_hx;
    // fixed-point records: quanta per A, A per quantum and its square, shift
    // from the 2^-12 A grid of hi to quanta; grid origin
    float f_rq, f_q, f_q2, f_org[3];
    int rec_shift;
    // squared radii in quanta: bracket of the list radius, near part, pruning
    float f_rl2q_lo, f_rl2q_hi, f_ra2q, f_rp2q;
    float half_skin2q, half_prune2q;  // squared displacements that ask for a build, a pruning
    float f_reach2, f_reach_slack;  // list radius squared (A^2, with slack) and slack (A)
    PotDev pot;
    // integration constants
    double mass, dt, acc_half, ke_fac, t_fac;
    float f_acc_half, f_ke_fac, f_dt;
    int block_steps;
    // coarse-step constants (Table 1)
    double pta_h, pta_Delta, tol_v[3], tol_j[3], floor_[3];
    // adaptive burst length (appendix): test every conv_lag steps (0 = off)
    int conv_lag;
    double conv_tol[3];
    // arrays
    void *pos[2];   // FP64: double4 {x,y,z,0};  MIXED: float4 hi {x,y,z,0}
    float4 *lo[2];  // MIXED only: float4 lo {x,y,z,0}
    int4 *rec[2];   // fixed-point record {x,y,z,0} of every atom
    void *posfp;    // FP64: double4 {x,y,z,w};  MIXED: the record with w (float bits) as
                    // fourth word; w = m a^m B'(rho)
    void *pen;      // energy of each atom, 1/2 eps sum_j phi_n + B(rho) (double; MIXED: float)
    void *vel;      // FP64: double4; MIXED: VelHL
    uint8_t *flags;
    int4 *ref;      // records at the last list build (skin test)
    int *atom_cell, *cell_cnt, *cell_start;
    int2 *cell_tmp;    // atoms by cell, {slot, creation index}
    int *orig;        // original index (creation order) of the atom stored at each slot
    void *perm_tmp;   // scratch of the permutation that sorts atoms by cell
    uint4 *plist;     // what the pair passes read: near part, then the pruned far part
    uint4 *nlist;     // far part of the Verlet list (null without pruning)
    int2 *nab;        // per atom: entries of the near and of the far part
    int *pnn;         // per atom and lane: entries of plist
    int4 *pref;       // records at the last pruning
    int prune_on;
    int prune_first;  // 1: a fresh list is pruned before its first use
    double *part;       // partials of K, U, R and displacements, per block (or warp)
    double *gpart;      // per group of 32 blocks (resident runs)
    double *series;     // series_cap x 3 samples of the current burst
    long long series_cap;
    double *eval_out;   // MODE_EVAL, creation order: n x 3 F, n pe, then K, U, T, error bits
    double *rsum;       // n x 4, creation order: sums of the sampled positions of the
                        // burst (Eq. (mean_pos)); null unless asked for
    double *stage;      // n x 6 doubles: import/export staging
    SpecCtl *ctl;
};

struct Group {
    int prec, L, sc76;  // L: lanes per atom, 0 where the group's specimens differ
    PotF pf;  // the group's potential (specimens of one group share it)
    const int *b2s;
    int nblk;
};

// Control words of a resident run (k_run_*), each on a line of its own: the
// arrivals at its grid barriers (reset before every launch); stuck: a
// barrier's wait ran out.
struct RunCtl {
    unsigned long long arrive, pad0[15];
    unsigned long long finished, pad2[15];  // launched steps: see k_finish
    int stuck, pad1[31];
};
// what a step asks for, or what became of the run
enum RunState : int { RUN_STOP = 1, RUN_BUILD = 2, RUN_PRUNE = 4, RUN_STUCK = 8 };

// one launch table: the specimens and, per kernel kind, block->specimen maps
struct Tab {
    const SpecDev *specs;
    int nspec;
    const int *b2s_atom;
    int nblk_atom;
    const int *b2s_bld;
    int nblk_bld;
    int bld_words;  // shared words per warp of the list build
    bool bld_scratch;  // a specimen's list build works in memory
    // resident runs and sweeps: block->specimen map over all specimens when they
    // share precision and potential (else null), fewest lanes per atom
    const int *b2s_run;
    int nblk_run, min_lanes;
    unsigned barrier_polls;  // polls before a grid barrier's wait is given up
    int ngroups;
    Group grp[8];
};

// Neighbour records and lists.
//
// A record is an atom's position in fixed point: int32 quanta of 2^-k A,
// modulo 2^32.  Only differences of two records are used, and those of atoms
// in neighbouring cells are below 2^31 quanta by the choice of k (2^-26 A at
// the default radii), so they are exact in wrapping int32 arithmetic whatever
// the specimen's extent; a difference is converted once to FP32, and its
// rounding is relative to the distance.  (FP32 records relative to half-cell
// centres with an offset coded in every list entry took 7.5 instructions per
// entry to decode and had the larger error; fixed point that spans the whole
// specimen, 2^-22 A for a 20 nm cube, had the larger error too.)
//
// A list entry is the byte offset of the neighbour's record (slot x 16).
// Lists are stored in quads of four entries: the 32 lanes of a warp read the
// quads of one iteration as 512 contiguous bytes (lane column: tile of 32
// lanes x capq quads).  With L lanes per atom, atom a owns lanes (a L) % 32 +
// 0..L-1 of tile (a L) / 32.
//
// The Verlet list (radius rc + skin) is kept in two parts by the distance at
// the build.  The near part (within rc + NEAR_MARGIN) is read by every pair
// pass as it stands.  The far part is read by the pruning, which appends the
// entries within rc + prune_margin to each lane's near entries.  Pairs beyond
// rc add exactly zero, and the order of a lane's entries does not depend on
// the pruning margin, so results do not either.
//
// In the near part, row r of lane l (counted in the warp) holds a slot with
// slot % 8 == (l + r) % 8 wherever the atom has one: the eight lanes of a
// quarter-warp then gather their 16-byte records from different banks of the
// 128-byte L1 line.  On the 470,596-atom cube that takes the gathers from
// ~10.6 to ~6.5 wavefronts each, and the density pass from 98 to 76 us, the
// force pass from 102 to 84 us (prototype of the pair loops alone).
constexpr int REC_SHIFT = 4;             // log2 of a record's bytes
constexpr double NEAR_MARGIN = 0.3;      // A
constexpr int MAX_ATOMS = 1 << 23;

__host__ __device__ __forceinline__ unsigned nl_entry(int j) { return (unsigned)j << REC_SHIFT; }
__host__ __device__ __forceinline__ int nl_j(unsigned e) { return (int)(e >> REC_SHIFT); }
// first quad of lane l of atom a
__host__ __device__ __forceinline__ long long nl_col(int a, int l, int L, int capq) {
    const long long t = (long long)a * L;
    return (t >> 5) * capq * 32 + (t & 31) + l;
}

// index i of an array of n elements (debug builds: tested, 0 when outside)
__device__ __forceinline__ int chk_index(const SpecDev &S, int i, int n) {
#if PTA_CHECK
    if ((unsigned)i >= (unsigned)n) {
        atomicOr(&S.ctl->err, ERR_CHECK);
        return 0;
    }
#endif
    return i;
}

// the byte offset of the record a list entry names
__device__ __forceinline__ unsigned nl_off(const SpecDev &S, unsigned e) {
#if PTA_CHECK
    return (unsigned)chk_index(S, nl_j(e), S.n) << REC_SHIFT;
#endif
    return e;
}

// a count of list entries read by one lane (debug builds: at most `limit`)
__device__ __forceinline__ int chk_count(const SpecDev &S, int c, int limit) {
#if PTA_CHECK
    if (c < 0 || c > limit) {
        atomicOr(&S.ctl->err, ERR_CHECK);
        return c < 0 ? 0 : limit;
    }
#endif
    return c;
}

// an atom's force (debug builds: finite)
__device__ __forceinline__ void chk_force(const SpecDev &S, double fx, double fy, double fz) {
#if PTA_CHECK
    if (!(isfinite(fx) && isfinite(fy) && isfinite(fz))) atomicOr(&S.ctl->err, ERR_NAN);
#endif
    (void)S; (void)fx; (void)fy; (void)fz;
}

// Cells are numbered along a serpentine path (x reverses on every other row,
// y on every other layer), so that consecutive cells are face neighbours and
// consecutive atoms of the cell-sorted order lie in the same or adjacent
// cells.
__host__ __device__ __forceinline__ int serp_rank(int n0, int n1, int x, int y, int z) {
    const int yr = (z & 1) ? n1 - 1 - y : y;
    const int t = z * n1 + yr;
    const int xr = (t & 1) ? n0 - 1 - x : x;
    return t * n0 + xr;
}
__host__ __device__ __forceinline__ void serp_coords(int n0, int n1, int r, int &x, int &y, int &z) {
    const int t = r / n0, xr = r % n0;
    z = t / n1;
    const int yr = t % n1;
    y = (z & 1) ? n1 - 1 - yr : yr;
    x = (t & 1) ? n0 - 1 - xr : xr;
}
__host__ __device__ __forceinline__ int cell_rank(const int nc[3], int x, int y, int z) {
    return serp_rank(nc[0], nc[1], x, y, z);
}
__host__ __device__ __forceinline__ void cell_coords(const int nc[3], int r, int &x, int &y, int &z) {
    serp_coords(nc[0], nc[1], r, x, y, z);
}

// arithmetic of records, modulo 2^32 (signed arithmetic may not wrap): the
// difference of two coordinates, and a coordinate from quanta of 2^shift and
// of one
__host__ __device__ __forceinline__ int rec_diff(int a, int b) {
    return (int)((unsigned)a - (unsigned)b);
}
__host__ __device__ __forceinline__ int rec_join(int hi, int lo, int shift) {
    return (int)(((unsigned)hi << shift) + (unsigned)lo);
}
// one coordinate of a record: hi is a multiple of 2^-12 A and enters exactly,
// lo is rounded to the nearest quantum (a quantum above 2^-12 A, which takes a
// cutoff of ~0.1 mm, rounds their sum)
__device__ __forceinline__ int rec_coord(const SpecDev &S, float hi, float lo) {
    if (S.rec_shift < 0) return __float2int_rn((hi + lo) * S.f_rq);
    return rec_join(__float2int_rn(hi * (float)HI_SCALE), __float2int_rn(lo * S.f_rq), S.rec_shift);
}
__device__ __forceinline__ int4 rec_mixed(const SpecDev &S, float hx, float hy, float hz, float lx,
                                          float ly, float lz) {
    return make_int4(rec_coord(S, hx, lx), rec_coord(S, hy, ly), rec_coord(S, hz, lz), 0);
}
// FP64 form: rounded once from the double coordinate, low 32 bits
__device__ __forceinline__ int4 rec_fp64(const SpecDev &S, double x, double y, double z) {
    const double rq = (double)S.f_rq;
    return make_int4((int)__double2ll_rn(x * rq), (int)__double2ll_rn(y * rq),
                     (int)__double2ll_rn(z * rq), 0);
}

// segments of the permutation scratch (see perm_layout)
struct PermLayout {
    size_t pos, lo, vel, flags, orig, cell, total;
};
__host__ __device__ inline size_t perm_round(size_t x) { return (x + 255) / 256 * 256; }
__host__ __device__ inline PermLayout perm_layout(size_t n, int prec) {
    const size_t P = prec == PTA_PREC_FP64 ? 32 : 16;
    PermLayout L;
    size_t o = 0;
    L.pos = o;
    o += perm_round(P * n);
    L.lo = o;
    o += prec == PTA_PREC_FP64 ? 0 : perm_round(16 * n);
    L.vel = o;
    o += perm_round(32 * n);  // double4 or VelHL
    L.flags = o;
    o += perm_round(n);
    L.orig = o;
    o += perm_round(4 * n);
    L.cell = o;
    o += perm_round(4 * n);
    L.total = o;
    return L;
}

// one block of SCAN_THREADS threads per specimen: exclusive scan of the cell
// counts into cell_start (cell_start[ncell] = total); the counts are reset to
// 0 for the next build; the specimen's build count + 1.  Each warp scans a
// contiguous part, four cells per lane (cells along each axis are even in
// number), behind a first reading of the parts' sums.
__device__ __forceinline__ void scan_cells(const SpecDev &S) {
    constexpr int NW = SCAN_THREADS / 32;
    __shared__ int wsum[NW];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, n = S.ncell / 4;
    int4 *cnt = (int4 *)S.cell_cnt, *start = (int4 *)S.cell_start;
    const int part = ((n + NW - 1) / NW + 31) & ~31;
    const int c0 = min(w * part, n), c1 = min(c0 + part, n);
    int sum = 0;
#pragma unroll 8
    for (int c = c0 + lane; c < c1; c += 32) {
        const int4 v = cnt[c];
        sum += (v.x + v.y) + (v.z + v.w);
    }
    sum = __reduce_add_sync(0xffffffffu, sum);
    if (lane == 0) wsum[w] = sum;
    __syncthreads();
    if (w == 0) {
        const int v = wsum[lane];
        int s = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        wsum[lane] = s - v;
        if (lane == 31) {
            S.cell_start[S.ncell] = s;
            S.ctl->rebuilds += 1;
#if PTA_CHECK
            if (s != S.n) atomicOr(&S.ctl->err, ERR_CHECK);  // every atom in one cell
#endif
        }
    }
    __syncthreads();
    int carry = wsum[w];
    const int4 zero = make_int4(0, 0, 0, 0);
    int4 nx = c0 + lane < c1 ? cnt[c0 + lane] : zero;
    for (int c = c0 + lane; c - lane < c1; c += 32) {
        const int4 v = nx;
        nx = c + 32 < c1 ? cnt[c + 32] : zero;
        const int own = (v.x + v.y) + (v.z + v.w);
        int x = own;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (c < c1) {
            const int b = carry + x - own;
            start[c] = make_int4(b, b + v.x, b + v.x + v.y, b + v.x + v.y + v.z);
            cnt[c] = zero;
        }
        carry += __shfl_sync(0xffffffffu, x, 31);
    }
}

// ---------------------------------------------------------------------------
// launchers (defined in the .cu files)
// ---------------------------------------------------------------------------
// creation and state exchange, single specimen (d = device SpecDev)
void launch_create(const SpecDev &h, const SpecDev *d, double sigma_v, double kT, uint64_t seed,
                   cudaStream_t st);
void launch_import(const SpecDev &h, const SpecDev *d, cudaStream_t st);
void launch_export(const SpecDev &h, const SpecDev *d, cudaStream_t st);
void launch_fix_right_grip(const SpecDev &h, const SpecDev *d, cudaStream_t st);
// checkpoints: working state <-> permutation scratch in creation order
void launch_ckpt_move(const SpecDev &h, const SpecDev *d, int gather, cudaStream_t st);
// batched
void launch_strain(const Tab &t, const double *du, cudaStream_t st);
void launch_burst_begin(const Tab &t, const long long *nsteps, cudaStream_t st);
void launch_burst_end(const Tab &t, int slot, pta_averages *out, cudaStream_t st);
void launch_any_running(const Tab &t, int *flag, cudaStream_t st);
void launch_pta_update(const Tab &t, const int *ops, pta_coarse_result *out, cudaStream_t st);
void launch_rebuild(const Tab &t, int force, cudaStream_t st);
int build_smem_limit();  // allow k_build its dynamic shared memory; 0 on failure
void launch_prune(const Tab &t, int force, cudaStream_t st);
void launch_decide_rebuild(const Tab &t, RunCtl *rc, cudaGraphConditionalHandle h, cudaStream_t st);
// list maintenance decided on the device: 0 build + prune, 1 prune, 2 nothing
constexpr unsigned LIST_BUILD = 0, LIST_PRUNE = 1, LIST_NONE = 2;

__device__ __forceinline__ bool build_active(const SpecDev &S, int force) {
    const SpecCtl *c = S.ctl;
    if (force) return true;
    if (c->phase == PH_IDLE) return false;
    return c->rebuild != 0 || c->list_L != S.L;
}
__device__ __forceinline__ bool prune_active(const SpecDev &S, int force) {
    if (!S.prune_on) return false;
    if (force) return true;
    return S.ctl->phase != PH_IDLE && S.ctl->prune != 0;
}
void launch_density(const Tab &t, int force, cudaStream_t st);
void launch_force(const Tab &t, int mode, cudaStream_t st);
// the step's end; next: handle of the next step's list maintenance, or null
void launch_finish(const Tab &t, int mode, RunCtl *rc, const cudaGraphConditionalHandle *next,
                   cudaStream_t st);
// resident runs and sweeps (see k_pair_common.cuh): can the table, whose block
// ->specimen map the host passes, be run that way, and the cooperative launch
bool run_possible(const Tab &t, const int *b2s_host);
cudaError_t launch_run(const Tab &t, RunCtl *rc, cudaGraphConditionalHandle again,
                       cudaStream_t st);
void launch_decide_build(const Tab &t, RunCtl *rc, cudaGraphConditionalHandle h, cudaStream_t st);

}  // namespace pta
