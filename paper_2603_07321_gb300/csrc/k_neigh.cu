// Cell binning by counting sort and Verlet-list construction.
//
// The list of atom i holds every j != i with |r_j - r_i|^2 < (rc + skin)^2,
// the squared distance formed as (dx*dx + dy*dy) + dz*dz in FP64 without
// contraction (an FP32 test on the records decides all but a thin band around
// the radius).  Candidates come from the 27 cells around i's cell on a grid
// of edge >= rc + skin; atoms outside the grid are clamped onto its border
// cells, which keeps every pair within reach (clamping is non-expansive), and
// are reported (PTA_ERANGE): the grid's margin is a quarter of the specimen's
// extent, which no atom of a deforming specimen reaches.  Where the atoms fill
// the grid, each cell is cut in CELL_SPLIT along x, to fit a row's candidates to
// the radius.
// After binning, the atoms themselves are permuted into cell order (cells in
// rank order, atoms of a cell in creation order), so that
// the 32 atoms of a warp share a cell and read overlapping neighbours, and a
// cell's atoms are one contiguous range.  The list order (cell order, then
// slot) is therefore a function of positions and grid: builds are
// deterministic.  orig[] keeps each slot's creation-order index.
//
// The list is rebuilt only when the force kernel found an atom that moved
// more than skin/2 since the last build (or on request); every kernel here
// returns at once for a specimen that needs no build.
#include "pta_dev.cuh"

namespace pta {

__device__ __forceinline__ int clampi(int v, int lo, int hi) { return v < lo ? lo : (v > hi ? hi : v); }

// position of atom a in FP64 (exact value of the stored representation)
__device__ __forceinline__ void load_pos64(const SpecDev &S, int par, int a, double &x, double &y,
                                           double &z) {
    if (S.prec == PTA_PREC_FP64) {
        const double4_32a q = ((const double4_32a *)S.pos[par])[a];
        x = q.x;
        y = q.y;
        z = q.z;
    } else {
        const float4 h = ((const float4 *)S.pos[par])[a];
        const float4 l = S.lo[par][a];
        x = (double)h.x + (double)l.x;
        y = (double)h.y + (double)l.y;
        z = (double)h.z + (double)l.z;
    }
}

// the same rounded to FP32
__device__ __forceinline__ float3 load_pos32(const SpecDev &S, int par, int a) {
    if (S.prec == PTA_PREC_FP64) {
        const double4_32a q = ((const double4_32a *)S.pos[par])[a];
        return make_float3((float)q.x, (float)q.y, (float)q.z);
    }
    const float4 h = ((const float4 *)S.pos[par])[a];
    const float4 l = S.lo[par][a];
    return make_float3(h.x + l.x, h.y + l.y, h.z + l.z);
}

// an atom's place among its cell's atoms as they were counted, in the scratch
__device__ __forceinline__ int *place_in_cell(const SpecDev &S) {
    return (int *)((char *)S.perm_tmp + perm_layout(S.n, S.prec).cell);
}

__global__ void k_bin(const SpecDev *__restrict__ specs, const int *__restrict__ b2s, int force) {
    const SpecDev &S = specs[b2s[blockIdx.x]];
    if (!build_active(S, force)) return;
    const int a = (blockIdx.x - S.blk_atom0) * TPB + threadIdx.x;
    if (a >= S.n) return;
    const int par = S.ctl->parity;
    double x[3];
    load_pos64(S, par, a, x[0], x[1], x[2]);
    int ci[3];
    bool out = false;
    for (int d = 0; d < 3; ++d) {
        const double q = floor((x[d] - S.org[d]) * (d == 0 ? S.inv_hx : S.inv_h));
        out |= !(q >= 0.0 && q < (double)S.nc[d]);
        ci[d] = clampi((int)fmax(fmin(q, 1e9), -1e9), 0, S.nc[d] - 1);
    }
    if (out) atomicOr(&S.ctl->err, ERR_GRID);
    const int c = cell_rank(S.nc, ci[0], ci[1], ci[2]);
    S.atom_cell[a] = c;
    place_in_cell(S)[a] = atomicAdd(&S.cell_cnt[c], 1);
}

// one block per specimen: exclusive scan of the cell counts
__global__ void k_scan(const SpecDev *__restrict__ specs, int force) {
    const SpecDev &S = specs[blockIdx.x];
    if (!build_active(S, force)) return;
    if (threadIdx.x == 0) S.ctl->max_nn = 0;  // the build takes the maximum
    scan_cells(S);
}

__global__ void k_scatter(const SpecDev *__restrict__ specs, const int *__restrict__ b2s,
                          int force) {
    const SpecDev &S = specs[b2s[blockIdx.x]];
    if (!build_active(S, force)) return;
    const int a = (blockIdx.x - S.blk_atom0) * TPB + threadIdx.x;
    if (a >= S.n) return;
    const int slot = chk_index(S, S.cell_start[S.atom_cell[a]] + place_in_cell(S)[a], S.n);
    S.cell_tmp[slot] = make_int2(a, S.orig[a]);
}

// orders every cell's atoms by creation index (rank = number of smaller ones),
// so that the order within a cell, and with it every list order, does not
// depend on how cells are numbered or counted; the per-atom state goes to its
// place in the scratch, copied back by the next kernel.
//
// Bound: latency, and from ~100,000 atoms the state's bytes.  A thread per atom
// reads the ~15 indices of its cell: 9 us for 52,700 atoms, 17 for 470,596.  A
// warp per cell of four times the size, eight in turn, whose atoms' state a
// further kernel moved, took 49 and 63 us.
__global__ void k_order(const SpecDev *__restrict__ specs, const int *__restrict__ b2s, int force) {
    const SpecDev &S = specs[b2s[blockIdx.x]];
    if (!build_active(S, force)) return;
    const int p = (blockIdx.x - S.blk_atom0) * TPB + threadIdx.x;
    if (p >= S.n) return;
    const int par = S.ctl->parity;
    const PermLayout Lo = perm_layout(S.n, S.prec);
    char *t = (char *)S.perm_tmp;
    const int2 own = S.cell_tmp[p];
    const int v = chk_index(S, own.x, S.n);
    const int c = S.atom_cell[v];
    const int s = S.cell_start[c], e = S.cell_start[c + 1];
    int r = s;
#pragma unroll 4
    for (int q = s; q < e; ++q) r += S.cell_tmp[chk_index(S, q, S.n)].y < own.y;
    r = chk_index(S, r, S.n);
    // velocities: 32-byte records in both precisions (double4 or VelHL)
    ((double4_32a *)(t + Lo.vel))[r] = ((const double4_32a *)S.vel)[v];
    if (S.prec == PTA_PREC_FP64) {
        ((double4_32a *)(t + Lo.pos))[r] = ((const double4_32a *)S.pos[par])[v];
    } else {
        ((float4 *)(t + Lo.pos))[r] = ((const float4 *)S.pos[par])[v];
        ((float4 *)(t + Lo.lo))[r] = S.lo[par][v];
    }
    ((uint8_t *)(t + Lo.flags))[r] = S.flags[v];
    ((int *)(t + Lo.orig))[r] = own.y;
    ((int *)(t + Lo.cell))[r] = c;
}

__global__ void k_permute_scatter(const SpecDev *__restrict__ specs, const int *__restrict__ b2s,
                                  int force) {
    const SpecDev &S = specs[b2s[blockIdx.x]];
    if (!build_active(S, force)) return;
    const int p = (blockIdx.x - S.blk_atom0) * TPB + threadIdx.x;
    if (p >= S.n) return;
    const int par = S.ctl->parity;
    const PermLayout Lo = perm_layout(S.n, S.prec);
    const char *t = (const char *)S.perm_tmp;
    ((double4_32a *)S.vel)[p] = ((const double4_32a *)(t + Lo.vel))[p];
    // and the records, which the list build and the first density pass read
    if (S.prec == PTA_PREC_FP64) {
        const double4_32a q = ((const double4_32a *)(t + Lo.pos))[p];
        ((double4_32a *)S.pos[par])[p] = q;
        S.rec[par][p] = rec_fp64(S, q.x, q.y, q.z);
    } else {
        const float4 hi = ((const float4 *)(t + Lo.pos))[p], lo = ((const float4 *)(t + Lo.lo))[p];
        ((float4 *)S.pos[par])[p] = hi;
        S.lo[par][p] = lo;
        S.rec[par][p] = rec_mixed(S, hi.x, hi.y, hi.z, lo.x, lo.y, lo.z);
    }
    S.flags[p] = ((const uint8_t *)(t + Lo.flags))[p];
    S.orig[p] = ((const int *)(t + Lo.orig))[p];
    S.atom_cell[p] = ((const int *)(t + Lo.cell))[p];
}

// exact list predicate between atoms a and j, in FP64
__device__ __noinline__ bool in_list_exact(const SpecDev &S, int par, int a, int j) {
    double xa, ya, za, xj, yj, zj;
    load_pos64(S, par, a, xa, ya, za);
    load_pos64(S, par, j, xj, yj, zj);
    const double dx = xj - xa, dy = yj - ya, dz = zj - za;
    const double r2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
    return r2 < S.rl2;
}

// The Verlet list of every atom, one warp per atom: the warp's lanes test 32
// consecutive slots of a row of cells at a time (coalesced record reads) and
// compact the hits in slot order through ballots into shared memory, near
// entries from the front, far ones from the back.  Rows and cells that the
// list radius cannot reach from the atom's place in its cell are skipped.  The near entries are then
// arranged by slot % 8 (see the list format) and both parts written as quads.
//
// Bound: instruction issue (80% of the slots; 2,700 instructions per atom, over
// half of them candidate tests).  470,596 atoms: 1.28 ms (1.69 with undivided
// cells, divisions by the lane count and 72 registers; at 64 registers eight
// blocks share an SM), 52,700 atoms 145 us (187).
//
// MEM: for specimens whose capacity is too large for shared memory.
template <bool MEM>
__global__ void __launch_bounds__(BUILD_WARPS * 32, 8) k_build(const SpecDev *__restrict__ specs,
                                                           const int *__restrict__ b2s,
                                                           int force, int words) {
    extern __shared__ uint4 bsh4[];
    const SpecDev &S = specs[b2s[blockIdx.x]];
    if ((S.bld_scratch != nullptr) != MEM || !build_active(S, force)) return;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const int cap = S.cap_use, L = S.L, n = S.n, par = S.ctl->parity;
    const int sL = 31 - __clz(L);  // L is a power of two
    unsigned *buf = (unsigned *)bsh4 + (size_t)w * words;  // cap entries
    if constexpr (MEM)
        buf = S.bld_scratch + (size_t)((blockIdx.x - S.blk_bld0) * BUILD_WARPS + w) * build_words(cap);
    unsigned *out = buf + cap;                             // near part in list order
    int *cls = (int *)(out + cap + 128);                   // 8 counters
    const int4 *__restrict__ rec = S.rec[par];
    const float h = S.f_h, hi2 = S.f_rl2q_hi, ra2 = S.f_ra2q;
    float lo2 = S.f_rl2q_lo;
    constexpr unsigned EMPTY = 0xffffffffu;
    // an atom beyond the cell grid may be farther from a candidate than the
    // records' period allows: then every hit is confirmed in FP64
    if (S.ctl->err & ERR_GRID) lo2 = 0.f;
    int most = 0;
    for (int i = 0; i < S.apw; ++i) {
        const int a = ((blockIdx.x - S.blk_bld0) * BUILD_WARPS + w) * S.apw + i;
        if (a >= n) break;
        const int4 ra = rec[a];
        // lanes 0..8: the slot range of row (dy, dz) of cells
        int rs = 0, re = 0;
        if (lane < 9) {
            int cx, cy, cz;
            cell_coords(S.nc, S.atom_cell[a], cx, cy, cz);
            const int dy = lane % 3 - 1, dz = lane / 3 - 1;
            const int yy = cy + dy, zz = cz + dz;
            const float sl = S.f_reach_slack;
            const float3 x = load_pos32(S, par, a);
            const float px = x.x - S.f_org[0] - (float)cx * S.f_hx;
            const float py = x.y - S.f_org[1] - (float)cy * h;
            const float pz = x.z - S.f_org[2] - (float)cz * h;
            const float ey = dy == 0 ? 0.f : fmaxf((dy < 0 ? py : h - py) - sl, 0.f);
            const float ez = dz == 0 ? 0.f : fmaxf((dz < 0 ? pz : h - pz) - sl, 0.f);
            const float rem = S.f_reach2 - ey * ey - ez * ez;
            if (rem > 0.f && yy >= 0 && zz >= 0 && yy < S.nc[1] && zz < S.nc[2]) {
                const float reach = sqrtf(rem) + sl;
                // (the atom's own cell in any case: one beyond the grid is
                // counted in the cell at its edge)
                const int x0 = min(max(cx + (int)floorf((px - reach) * S.f_inv_hx), 0), cx);
                const int x1 = max(min(cx + (int)floorf((px + reach) * S.f_inv_hx), S.nc[0] - 1), cx);
                const int r0 = cell_rank(S.nc, x0, yy, zz), r1 = cell_rank(S.nc, x1, yy, zz);
                rs = chk_count(S, S.cell_start[min(r0, r1)], n);
                re = chk_count(S, S.cell_start[max(r0, r1) + 1], n);
            }
        }
        int na = 0, stored = 0, tot = 0;  // near and all entries stored; all found
        for (int r = 0; r < 9; ++r) {
            const int s = __shfl_sync(0xffffffffu, rs, r), e = __shfl_sync(0xffffffffu, re, r);
            if (s >= e) continue;
            int j = s + lane;
            int4 nx = rec[min(j, e - 1)];
            for (int b = s; b < e; b += 32, j += 32) {
                const int4 rj = nx;
                if (b + 32 < e) nx = rec[min(j + 32, e - 1)];
                const float fx = (float)rec_diff(rj.x, ra.x), fy = (float)rec_diff(rj.y, ra.y),
                            fz = (float)rec_diff(rj.z, ra.z);
                const float r2 = fmaf(fz, fz, fmaf(fy, fy, fx * fx));
                bool in = r2 < hi2 && j < e && j != a;
                if (in && r2 >= lo2) in = in_list_exact(S, par, a, j);
                const unsigned ml = __ballot_sync(0xffffffffu, in);
                if (!ml) continue;
                const bool near = r2 < ra2;
                const unsigned ma = __ballot_sync(0xffffffffu, in && near);
                const int nb = stored - na;
                tot += __popc(ml);
                if (tot > cap) continue;  // reported below
                stored = tot;
                const int k = __popc((near ? ma : ml ^ ma) & lt);
                if (in) buf[near ? na + k : cap - 1 - nb - k] = nl_entry(j);
                na += __popc(ma);
            }
        }
        const int nb = stored - na;
        most = max(most, tot);
        // near part: lane l gets rows [0, na / L + (l < na % L))
        const int rows = na >> sL, rest = na & (L - 1);
        const int lane0 = (int)(((long long)a * L) & 31);
        const int cells = ((rows + 4) >> 2) * 4 * L;
        for (int m = lane; m < cells / 4; m += 32)
            ((uint4 *)out)[m] = make_uint4(EMPTY, EMPTY, EMPTY, EMPTY);
        if (lane < 8) cls[lane] = 0;
        __syncwarp();
        int nov = 0;  // entries whose class has no row left
        for (int k0 = 0; k0 < na; k0 += 32) {
            const int k = k0 + lane;
            const bool act = k < na;
            const unsigned e = act ? buf[k] : 0u;
            const int c = act ? (int)(e >> REC_SHIFT) & 7 : 8;
            const unsigned peers = __match_any_sync(0xffffffffu, c);
            const int rank = __popc(peers & lt);
            const int base = act ? cls[c] : 0;
            __syncwarp();
            if (act && rank == 0) cls[c] = base + __popc(peers);
            const int t = base + rank, li = t & (L - 1);
            const int row = 8 * (t >> sL) + ((c - lane0 - li) & 7);
            const bool ok = act && row < rows + (li < rest);
            if (ok) out[((row >> 2) * L + li) * 4 + (row & 3)] = e;
            const unsigned mo = __ballot_sync(0xffffffffu, act && !ok);
            if (act && !ok) buf[nov + __popc(mo & lt)] = e;  // never past what has been read
            nov += __popc(mo);
            __syncwarp();
        }
        // the rows left empty take them, in order
        for (int m0 = 0, got = 0; got < nov && m0 < cells; m0 += 32) {
            const int m = m0 + lane;
            const int li = (m >> 2) & (L - 1), row = (m >> (sL + 2)) * 4 + (m & 3);
            const bool hole = m < cells && row < rows + (li < rest) && out[m] == EMPTY;
            const unsigned mh = __ballot_sync(0xffffffffu, hole);
            const int q = got + __popc(mh & lt);
            if (hole && q < nov) out[m] = buf[q];
            got += __popc(mh);
        }
        __syncwarp();
        uint4 *dst = S.plist + nl_col(a, 0, L, S.capq);
        for (int m = lane; m < cells / 4; m += 32) dst[(m >> sL) * 32 + (m & (L - 1))] = ((uint4 *)out)[m];
        // far part, entry k in lane k % L
        if (S.prune_on) {
            uint4 *far = S.nlist + nl_col(a, 0, L, S.capq);
            const int qb = (((nb + L - 1) >> sL) + 3) >> 2;
            for (int m = lane; m < qb * L; m += 32) {
                unsigned v[4];
#pragma unroll
                for (int s = 0; s < 4; ++s) {
                    const int k = (((m >> sL) * 4 + s) << sL) + (m & (L - 1));
                    v[s] = k < nb ? buf[cap - 1 - k] : 0u;  // slot 0 where there is none
                }
                far[(m >> sL) * 32 + (m & (L - 1))] = make_uint4(v[0], v[1], v[2], v[3]);
            }
            if (lane < L) S.pnn[a * L + lane] = rows + (lane < rest);
        } else {
            __syncwarp();
            for (int k = lane; k < nb; k += 32) {
                const int l = k & (L - 1), row = rows + (l < rest) + (k >> sL);
                ((unsigned *)(dst + (row >> 2) * 32 + l))[row & 3] = buf[cap - 1 - k];
            }
            if (lane < L)
                S.pnn[a * L + lane] = rows + (lane < rest) + (nb > lane ? (nb - lane + L - 1) >> sL : 0);
        }
        if (lane == 0) {
            S.nab[a] = make_int2(na, nb);
            S.ref[a] = ra;
            if (S.prune_on) S.pref[a] = ra;
        }
        __syncwarp();
    }
    if (lane == 0 && most > 0) {
        atomicMax(&S.ctl->max_nn, most);
        if (most > cap) atomicOr(&S.ctl->err, ERR_OVERFLOW);
    }
}

// after the build: record the layout the list was built for (a separate
// kernel, so that the gate above reads the same value in every block)
__global__ void k_build_done(const SpecDev *__restrict__ specs, int force) {
    const SpecDev &S = specs[blockIdx.x];
    if (!build_active(S, force)) return;
    if (threadIdx.x == 0) {
        S.ctl->list_L = S.L;
        // the near part alone serves until an atom has moved half the pruning
        // margin, unless that margin is wider than the near part
        S.ctl->prune = S.prune_first;
    }
}

// one block: does any specimen of the table need a list build, or only a
// pruning of its inner list, before its next pair pass?  Sets the condition
// of the graph node that holds that work (LIST_BUILD, LIST_PRUNE, LIST_NONE).
__global__ void k_decide_rebuild(const SpecDev *__restrict__ specs, int nspec, RunCtl *rc,
                                 cudaGraphConditionalHandle handle) {
    int build = 0, prune = 0;
    for (int s = threadIdx.x; s < nspec; s += blockDim.x) {
        build |= build_active(specs[s], 0);
        prune |= prune_active(specs[s], 0);
    }
    build = __syncthreads_or(build);
    prune = __syncthreads_or(prune);
    if (threadIdx.x == 0) {
        rc->finished = 0;
        cudaGraphSetConditional(handle, build ? LIST_BUILD : (prune ? LIST_PRUNE : LIST_NONE));
    }
}

// the same for resident runs, which prune by themselves: 1 when any specimen
// needs a list build; and the run's barrier word starts at 0
__global__ void k_decide_build(const SpecDev *__restrict__ specs, int nspec, RunCtl *rc,
                               cudaGraphConditionalHandle handle) {
    int build = 0;
    for (int s = threadIdx.x; s < nspec; s += blockDim.x) build |= build_active(specs[s], 0);
    build = __syncthreads_or(build);
    if (threadIdx.x == 0) {
        rc->arrive = 0;
        cudaGraphSetConditional(handle, build ? 1u : 0u);
    }
}

void launch_decide_build(const Tab &t, RunCtl *rc, cudaGraphConditionalHandle h, cudaStream_t st) {
    k_decide_build<<<1, 128, 0, st>>>(t.specs, t.nspec, rc, h);
}

void launch_decide_rebuild(const Tab &t, RunCtl *rc, cudaGraphConditionalHandle h,
                           cudaStream_t st) {
    k_decide_rebuild<<<1, 128, 0, st>>>(t.specs, t.nspec, rc, h);
}

// the limit belongs to the function and so to every context of the process:
// always the same value, that of the largest capacity
int build_smem_limit() {
    return cudaFuncSetAttribute(k_build<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                BUILD_SMEM_MOST) == cudaSuccess;
}

void launch_rebuild(const Tab &t, int force, cudaStream_t st) {
    k_bin<<<t.nblk_atom, TPB, 0, st>>>(t.specs, t.b2s_atom, force);
    k_scan<<<t.nspec, SCAN_THREADS, 0, st>>>(t.specs, force);
    k_scatter<<<t.nblk_atom, TPB, 0, st>>>(t.specs, t.b2s_atom, force);
    k_order<<<t.nblk_atom, TPB, 0, st>>>(t.specs, t.b2s_atom, force);
    k_permute_scatter<<<t.nblk_atom, TPB, 0, st>>>(t.specs, t.b2s_atom, force);
    k_build<false><<<t.nblk_bld, BUILD_WARPS * 32, BUILD_WARPS * t.bld_words * 4, st>>>(
        t.specs, t.b2s_bld, force, t.bld_words);
    if (t.bld_scratch)
        k_build<true><<<t.nblk_bld, BUILD_WARPS * 32, 0, st>>>(t.specs, t.b2s_bld, force, 0);
    k_build_done<<<t.nspec, 32, 0, st>>>(t.specs, force);
}

}  // namespace pta
