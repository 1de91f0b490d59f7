// Cell binning by counting sort and Verlet-list construction.
//
// The list of atom i holds every j != i with |r_j - r_i|^2 < (rc + skin)^2,
// the squared distance formed as (dx*dx + dy*dy) + dz*dz in FP64 without
// contraction (an FP32 test on the records decides all but a thin band around
// the radius).  Candidates come from the 27 cells around i's cell on a grid
// of edge >= rc + skin; atoms outside the grid are clamped onto its border
// cells, which keeps every pair within reach (clamping is non-expansive), and
// are reported (PTA_ERANGE): the grid's margin is a quarter of the specimen's
// extent, which no atom of a deforming specimen reaches.
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
        const double q = floor((x[d] - S.org[d]) * S.inv_h);
        out |= !(q >= 0.0 && q < (double)S.nc[d]);
        ci[d] = clampi((int)fmax(fmin(q, 1e9), -1e9), 0, S.nc[d] - 1);
    }
    if (out) atomicOr(&S.ctl->err, ERR_GRID);
    const int c = cell_rank(S.nc, ci[0], ci[1], ci[2]);
    S.atom_cell[a] = c;
    atomicAdd(&S.cell_cnt[c], 1);
}

// one block per specimen: exclusive scan of the cell counts; counts reset to
// 0 for use as fill counters by the scatter
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
    const int c = S.atom_cell[a];
    const int slot = chk_index(S, S.cell_start[c] + atomicAdd(&S.cell_cnt[c], 1), S.n);
    S.cell_tmp[slot] = a;
}

// each warp orders CELLS_PER_WARP cells in turn (most cells of the grid's
// margin are empty): a cell's atoms by creation index (rank = number of
// smaller ones), so that the order within a cell, and with it every list
// order, does not depend on how cells are numbered; then the cell's counter
// is cleared for the next build
__global__ void k_cell_sort(const SpecDev *__restrict__ specs, const int *__restrict__ b2s,
                            int force) {
    const SpecDev &S = specs[b2s[blockIdx.x]];
    if (!build_active(S, force)) return;
    const int lane = threadIdx.x & 31;
    const int c0 = (blockIdx.x - S.blk_cell0) * CELL_WARPS * CELLS_PER_WARP + (threadIdx.x >> 5);
    for (int i = 0; i < CELLS_PER_WARP; ++i) {
        const int c = c0 + i * CELL_WARPS;
        if (c >= S.ncell) return;
        const int s = S.cell_start[c], e = S.cell_start[c + 1];
        for (int p = s + lane; p < e; p += 32) {
            const int v = chk_index(S, S.cell_tmp[chk_index(S, p, S.n)], S.n);
            const int ov = S.orig[v];
            int r = 0;
            for (int q = s; q < e; ++q) r += (S.orig[chk_index(S, S.cell_tmp[chk_index(S, q, S.n)], S.n)] < ov);
            S.cell_atoms[chk_index(S, s + r, S.n)] = v;
        }
        if (lane == 0) S.cell_cnt[c] = 0;
    }
}

// sort the per-atom state into cell order: gather into scratch, then copy back
__global__ void k_permute_gather(const SpecDev *__restrict__ specs, const int *__restrict__ b2s,
                                 int force) {
    const SpecDev &S = specs[b2s[blockIdx.x]];
    if (!build_active(S, force)) return;
    const int p = (blockIdx.x - S.blk_atom0) * TPB + threadIdx.x;
    if (p >= S.n) return;
    const int src = chk_index(S, S.cell_atoms[p], S.n);
    const int par = S.ctl->parity;
    const PermLayout Lo = perm_layout(S.n, S.prec);
    char *t = (char *)S.perm_tmp;
    // velocities: 32-byte records in both precisions (double4 or VelHL)
    ((double4_32a *)(t + Lo.vel))[p] = ((const double4_32a *)S.vel)[src];
    if (S.prec == PTA_PREC_FP64) {
        ((double4_32a *)(t + Lo.pos))[p] = ((const double4_32a *)S.pos[par])[src];
    } else {
        ((float4 *)(t + Lo.pos))[p] = ((const float4 *)S.pos[par])[src];
        ((float4 *)(t + Lo.lo))[p] = S.lo[par][src];
    }
    ((uint8_t *)(t + Lo.flags))[p] = S.flags[src];
    ((int *)(t + Lo.orig))[p] = S.orig[src];
    ((int *)(t + Lo.cell))[p] = S.atom_cell[src];
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
// list radius cannot reach from the atom's place in its cell are skipped
// (about a quarter of the 27 cells' candidates).  The near entries are then
// arranged by slot % 8 (see the list format) and both parts written as quads.
//
// Bound: instruction issue (candidate tests).  One thread per atom over the
// same 27 cells, which this replaces, ran 1,674 tests in sequence: ~1.33 ms
// for 470,596 atoms and a latency of ~0.1 ms for small specimens.
__global__ void __launch_bounds__(BUILD_WARPS * 32) k_build(const SpecDev *__restrict__ specs,
                                                           const int *__restrict__ b2s,
                                                           int force, int words) {
    extern __shared__ uint4 bsh4[];
    const SpecDev &S = specs[b2s[blockIdx.x]];
    if (!build_active(S, force)) return;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const int cap = S.cap_use, L = S.L, n = S.n, par = S.ctl->parity;
    unsigned *buf = (unsigned *)bsh4 + (size_t)w * words;  // cap entries
    unsigned *out = buf + cap;                             // near part in list order
    int *cls = (int *)(out + cap + 128);                   // 8 counters
    const int4 *__restrict__ rec = S.rec[par];
    const float h = S.f_h, lo2 = S.f_rl2q_lo, hi2 = S.f_rl2q_hi, ra2 = S.f_ra2q;
    constexpr unsigned EMPTY = 0xffffffffu;
    // an atom beyond the cell grid may be farther from a candidate than the
    // records' period allows: then every hit is confirmed in FP64
    const bool sure = !(S.ctl->err & ERR_GRID);
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
            const float px = x.x - S.f_org[0] - (float)cx * h;
            const float py = x.y - S.f_org[1] - (float)cy * h;
            const float pz = x.z - S.f_org[2] - (float)cz * h;
            const float ey = dy == 0 ? 0.f : fmaxf((dy < 0 ? py : h - py) - sl, 0.f);
            const float ez = dz == 0 ? 0.f : fmaxf((dz < 0 ? pz : h - pz) - sl, 0.f);
            const float rem = S.f_reach2 - ey * ey - ez * ez;
            if (rem > 0.f && yy >= 0 && zz >= 0 && yy < S.nc[1] && zz < S.nc[2]) {
                const float reach = sqrtf(rem) + sl;
                const int x0 = (cx > 0 && px < reach) ? cx - 1 : cx;
                const int x1 = (cx + 1 < S.nc[0] && h - px < reach) ? cx + 1 : cx;
                const int r0 = cell_rank(S.nc, x0, yy, zz), r1 = cell_rank(S.nc, x1, yy, zz);
                rs = chk_count(S, S.cell_start[min(r0, r1)], n);
                re = chk_count(S, S.cell_start[max(r0, r1) + 1], n);
            }
        }
        int na = 0, nb = 0, tot = 0;  // stored near and far entries; all found
        for (int r = 0; r < 9; ++r) {
            const int s = __shfl_sync(0xffffffffu, rs, r), e = __shfl_sync(0xffffffffu, re, r);
            if (s >= e) continue;
            int4 nx = rec[min(s + lane, e - 1)];
            for (int b = s; b < e; b += 32) {
                const int4 rj = nx;
                const int j = b + lane;
                if (b + 32 < e) nx = rec[min(j + 32, e - 1)];
                const float fx = (float)(rj.x - ra.x), fy = (float)(rj.y - ra.y),
                            fz = (float)(rj.z - ra.z);
                const float r2 = fmaf(fz, fz, fmaf(fy, fy, fx * fx));
                bool in = r2 < hi2 && j < e && j != a;
                if (in && (r2 >= lo2 || !sure)) in = in_list_exact(S, par, a, j);
                const unsigned ml = __ballot_sync(0xffffffffu, in);
                if (!ml) continue;
                const unsigned ma = __ballot_sync(0xffffffffu, in && r2 < ra2);
                const int k = __popc(ml);
                tot += k;
                if (na + nb + k > cap) continue;  // reported below
                if (in) {
                    if (r2 < ra2) buf[na + __popc(ma & lt)] = nl_entry(j);
                    else buf[cap - 1 - nb - __popc(ml & ~ma & lt)] = nl_entry(j);
                }
                na += __popc(ma);
                nb += k - __popc(ma);
            }
        }
        most = max(most, tot);
        // near part: lane l gets rows [0, na / L + (l < na % L))
        const int rows = na / L, rest = na % L;
        const int lane0 = (int)(((long long)a * L) & 31);
        const int cells = ((rows + 4) >> 2) * 4 * L;
        for (int m = lane; m < cells; m += 32) out[m] = EMPTY;
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
            const int row = 8 * (t / L) + ((c - lane0 - li) & 7);
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
            const int li = (m >> 2) & (L - 1), row = (m / (4 * L)) * 4 + (m & 3);
            const bool hole = m < cells && row < rows + (li < rest) && out[m] == EMPTY;
            const unsigned mh = __ballot_sync(0xffffffffu, hole);
            const int q = got + __popc(mh & lt);
            if (hole && q < nov) out[m] = buf[q];
            got += __popc(mh);
        }
        __syncwarp();
        uint4 *dst = S.plist + nl_col(a, 0, L, S.capq);
        for (int m = lane; m < cells / 4; m += 32) dst[(m / L) * 32 + (m & (L - 1))] = ((uint4 *)out)[m];
        // far part, entry k in lane k % L
        if (S.prune_on) {
            uint4 *far = S.nlist + nl_col(a, 0, L, S.capq);
            const int qb = ((nb + L - 1) / L + 3) >> 2;
            for (int m = lane; m < qb * L; m += 32) {
                unsigned v[4];
#pragma unroll
                for (int s = 0; s < 4; ++s) {
                    const int k = ((m / L) * 4 + s) * L + (m & (L - 1));
                    v[s] = k < nb ? buf[cap - 1 - k] : 0u;  // slot 0 where there is none
                }
                far[(m / L) * 32 + (m & (L - 1))] = make_uint4(v[0], v[1], v[2], v[3]);
            }
            if (lane < L) S.pnn[a * L + lane] = rows + (lane < rest);
        } else {
            __syncwarp();
            for (int k = lane; k < nb; k += 32) {
                const int l = k & (L - 1), row = rows + (l < rest) + k / L;
                ((unsigned *)(dst + (row >> 2) * 32 + l))[row & 3] = buf[cap - 1 - k];
            }
            if (lane < L)
                S.pnn[a * L + lane] = rows + (lane < rest) + (nb > lane ? (nb - lane + L - 1) / L : 0);
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

int build_smem_limit(int bytes) {
    return cudaFuncSetAttribute(k_build, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) ==
           cudaSuccess;
}

void launch_rebuild(const Tab &t, int force, cudaStream_t st) {
    k_bin<<<t.nblk_atom, TPB, 0, st>>>(t.specs, t.b2s_atom, force);
    k_scan<<<t.nspec, SCAN_THREADS, 0, st>>>(t.specs, force);
    k_scatter<<<t.nblk_atom, TPB, 0, st>>>(t.specs, t.b2s_atom, force);
    k_cell_sort<<<t.nblk_cell, CELL_WARPS * 32, 0, st>>>(t.specs, t.b2s_cell, force);
    k_permute_gather<<<t.nblk_atom, TPB, 0, st>>>(t.specs, t.b2s_atom, force);
    k_permute_scatter<<<t.nblk_atom, TPB, 0, st>>>(t.specs, t.b2s_atom, force);
    k_build<<<t.nblk_bld, BUILD_WARPS * 32, BUILD_WARPS * t.bld_words * 4, st>>>(
        t.specs, t.b2s_bld, force, t.bld_words);
    k_build_done<<<t.nspec, 32, 0, st>>>(t.specs, force);
}

}  // namespace pta
