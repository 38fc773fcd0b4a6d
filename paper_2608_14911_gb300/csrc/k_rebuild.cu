// Rebuild pipeline: linked-cell binning, the periodic Hilbert resort of every
// particle array into cell order, and the full Verlet list with skin.  Paper
// "Software design" ("Parallelization": CellGrid linked cells;
// "Performance optimizations": cell decomposition and data sorting) and
// "Example usage" (VerletList(system, cutoff) with system.skin).
//
// Every rebuild (inside the step graphs, when a replica asked for it):
//   prep      latch the per-replica requests, clear those replicas' cell counts
//   bin       cell of every particle and its arrival index (atomic histogram)
//   scan x3   exclusive scan of the counts in cell-index order: first entry of
//             every cell in one compact entry array (no per-cell capacity)
//   place     every particle's entry (position, storage slot) into its cell
//   cellsort  entries of each cell in ascending storage slot, so the list does
//             not depend on the order of the atomics
//   verlet    (k_verlet.cu) stencil search from the cell entries, streamed as
//             contiguous row ranges; full list (both directions) as groups of
//             four indices, nbr4[g * stride + i]; records the build positions
// A resort (launched between step graphs every `resort_every` steps, and on
// every explicit build) additionally runs, between cellsort and verlet:
//   scan x3   exclusive scan of the cell counts in Hilbert-rank order
//   scatter   new slot of every entry (its cell's first slot + its rank in the
//             cell); the entries switch to the new slots
//   gather    permuted copies of positions, velocities, forces, images
//   copyback  copies back and maps bond partners to their new slots
// Replicas whose request flag is clear skip every per-particle and per-cell
// step after `prep`; their counts and entries stay those of their last build,
// so the global scan keeps every replica's entries in its own slot range.
#include "kernels.cuh"
#include "scan.cuh"

namespace espp {


template <class T>
__device__ __forceinline__ int cell_of(const RepGeom<T>& g, const V4<T>& p) {
    const int cx = cell_coord(p.x, g.cells_per_len[0], g.nc[0]);
    const int cy = cell_coord(p.y, g.cells_per_len[1], g.nc[1]);
    const int cz = cell_coord(p.z, g.cells_per_len[2], g.nc[2]);
    return g.cell_off + (cz * g.nc[1] + cy) * g.nc[0] + cx;
}

template <class T>
__global__ void __launch_bounds__(256) k_prep(DevSys<T> s) {
    if (s.ctrl->abort) return;
    for (int h = blockIdx.x * blockDim.x + threadIdx.x; h < s.ncells; h += gridDim.x * blockDim.x)
        if (s.req[s.cell_rep[h]]) s.cell_cnt[h] = 0;
    if (blockIdx.x == 0) {
        // Lees-Edwards: the offset at this build, for the rebuild criterion
        // and the sheared rows of the search (kept as stored after a
        // checkpoint load)
        const long long pstep = s.ctrl->step + (long long)s.ctrl->pos_ahead;
        const bool keep = s.ctrl->le_keep != 0;
        for (int r = threadIdx.x; r < s.R; r += blockDim.x) {
            s.now[r] = s.req[r];
            if (s.le_on && s.req[r] && !keep) s.le_db[r] = le_offset(s, s.reps[r], pstep);
        }
        __syncthreads();
        if (threadIdx.x == 0) s.ctrl->le_keep = 0;
        if (threadIdx.x == 0 && s.ctrl->any_req) {
            s.ctrl->n_rebuilds += 1;
            s.ctrl->max_count = 0;
        }
    }
}

// Cell of every particle of a flagged replica and its arrival index in that
// cell (counting-sort histogram); positions are wrapped into the box here,
// at list builds only.
template <class T>
__global__ void __launch_bounds__(TILE) k_bin(DevSys<T> s, int cur) {
    // the first tile's record is requested together with the abort flag
    Tile tl0 = {0, 0, 0, 0};
    if ((int)blockIdx.x < s.ntiles) tl0 = ld_tile_early(s.tiles + blockIdx.x);
    if (s.ctrl->abort) return;
    if (blockIdx.x == 0) {
        for (int r = threadIdx.x; r < s.R; r += blockDim.x) s.req[r] = 0;
        if (threadIdx.x == 0) s.ctrl->any_req = 0;
    }
    V4<T>* __restrict__ P = s.pos[buffer_of(s, cur)];
    for (int t = blockIdx.x; t < s.ntiles; t += gridDim.x) {
        const Tile tl = t == (int)blockIdx.x ? tl0 : s.tiles[t];
        if (!s.now[tl.rep] || (int)threadIdx.x >= tl.count) continue;
        const int i = tl.start + threadIdx.x;
        V4<T> p = P[i];
        const RepGeom<T>& g = s.reps[tl.rep];
        int wx, wy, wz;
        if (s.le_on && !(p.z >= T(0) && p.z < g.L[2])) {
            // across a sheared face: the image entered is displaced and moving
            const double L[3] = {(double)g.L[0], (double)g.L[1], (double)g.L[2]};
            double q[3] = {(double)p.x, (double)p.y, (double)p.z};
            V4<T> v = s.vel[i];
            double vx = (double)v.x;
            int k[3];
            le_wrap(q, vx, k, L, s.le_db[tl.rep], s.le_shear);
            p.x = (T)q[0];
            p.y = (T)q[1];
            p.z = (T)q[2];
            // a coordinate rounded up to L in the conversion stays in its
            // image, just below L
            if (!(p.x < g.L[0])) p.x = below(g.L[0]);
            if (!(p.y < g.L[1])) p.y = below(g.L[1]);
            if (!(p.z < g.L[2])) p.z = below(g.L[2]);
            v.x = (T)vx;
            s.vel[i] = v;
            wx = k[0];
            wy = k[1];
            wz = k[2];
        } else {
            wx = wrap_coord(p.x, g.L[0]);
            wy = wrap_coord(p.y, g.L[1]);
            wz = wrap_coord(p.z, g.L[2]);
        }
        if (wx | wy | wz) {
            P[i] = p;
            int4 im = s.img[i];
            im.x += wx;
            im.y += wy;
            im.z += wz;
            s.img[i] = im;
        }
        const int h = cell_of(g, p);
        s.cellh[i] = h;
        s.in_cell[i] = atomicAdd(&s.cell_cnt[h], 1);
    }
}

// Entry (wrapped position, storage slot in the w lane) of every particle of a
// flagged replica at its cell's first entry + its arrival index.
template <class T>
__global__ void __launch_bounds__(TILE) k_place(DevSys<T> s, int cur) {
    // the first tile's record is requested together with the abort flag
    Tile tl0 = {0, 0, 0, 0};
    if ((int)blockIdx.x < s.ntiles) tl0 = ld_tile_early(s.tiles + blockIdx.x);
    if (s.ctrl->abort) return;
    const V4<T>* __restrict__ P = s.pos[buffer_of(s, cur)];
    for (int t = blockIdx.x; t < s.ntiles; t += gridDim.x) {
        const Tile tl = t == (int)blockIdx.x ? tl0 : s.tiles[t];
        if (!s.now[tl.rep] || (int)threadIdx.x >= tl.count) continue;
        const int i = tl.start + threadIdx.x;
        V4<T> p = ld4<T>(P + i);
        p.w = int_bits_as(T(0), i);
        s.cell_ent[s.cell_beg[s.cellh[i]] + s.in_cell[i]] = p;
    }
}

// Entries of each cell in ascending storage slot (a handful per cell), so the
// list does not depend on the order of the atomics.
template <class T>
__global__ void __launch_bounds__(256) k_cellsort(DevSys<T> s) {
    if (s.ctrl->abort) return;
    for (int h = blockIdx.x * blockDim.x + threadIdx.x; h < s.ncells; h += gridDim.x * blockDim.x) {
        if (!s.now[s.cell_rep[h]]) continue;
        V4<T>* p = s.cell_ent + s.cell_beg[h];
        const int e = s.cell_beg[h + 1] - s.cell_beg[h];
        for (int k = 1; k < e; ++k) {
            const V4<T> key = p[k];
            const int kk = bits_as_int(key.w);
            int q = k - 1;
            while (q >= 0 && bits_as_int(p[q].w) > kk) {
                p[q + 1] = p[q];
                --q;
            }
            p[q + 1] = key;
        }
        // FP64 handles: the float copies that the list search tests first
        if constexpr (sizeof(T) == 8)
            for (int k = 0; k < e; ++k) {
                const V4<T> q = p[k];
                s.cell_ent32[s.cell_beg[h] + k] = make_float4((float)q.x, (float)q.y, (float)q.z, __int_as_float(bits_as_int(q.w)));
            }
        // list-free mode with DPD: the velocities in entry order as well
        if (s.cells_mode && s.dpd)
            for (int k = 0; k < e; ++k) s.cell_vel[s.cell_beg[h] + k] = s.vel[bits_as_int(p[k].w)];
    }
}

// ---- exclusive scan of the cell counts (three phases, no inter-block waits) --
// RANK = false: cells in index order -> cell_beg (every rebuild);
// RANK = true: cells in Hilbert-rank order -> rank_start (resort only).
template <class T, bool RANK>
__device__ __forceinline__ int scan_count(const DevSys<T>& s, int k) {
    return k < s.ncells ? s.cell_cnt[RANK ? s.cell_by_rank[k] : k] : 0;
}

template <class T, bool RANK>
__global__ void __launch_bounds__(SCAN_THREADS) k_scan_reduce(DevSys<T> s) {
    if (s.ctrl->abort) return;
    const int base = blockIdx.x * SCAN_TILE + threadIdx.x * SCAN_ITEMS;
    int sum = 0;
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) sum += scan_count<T, RANK>(s, base + k);
    int excl;
    const int total = block_excl_scan(sum, &excl);
    if (threadIdx.x == 0) s.scan_part[blockIdx.x] = total;
}

template <class T>
__global__ void __launch_bounds__(SCAN_THREADS) k_scan_top(DevSys<T> s) {
    if (s.ctrl->abort) return;
    int carry = 0;
    for (int b0 = 0; b0 < s.nscan_blocks; b0 += SCAN_THREADS) {
        const int b = b0 + threadIdx.x;
        const int v = b < s.nscan_blocks ? s.scan_part[b] : 0;
        int excl;
        const int total = block_excl_scan(v, &excl);
        if (b < s.nscan_blocks) s.scan_part[b] = carry + excl;
        carry += total;
    }
}

template <class T, bool RANK>
__global__ void __launch_bounds__(SCAN_THREADS) k_scan_down(DevSys<T> s) {
    if (s.ctrl->abort) return;
    const int base = blockIdx.x * SCAN_TILE + threadIdx.x * SCAN_ITEMS;
    int v[SCAN_ITEMS];
    int sum = 0;
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) {
        v[k] = scan_count<T, RANK>(s, base + k);
        sum += v[k];
    }
    int excl;
    block_excl_scan(sum, &excl);
    int run = s.scan_part[blockIdx.x] + excl;
    int* out = RANK ? s.rank_start : s.cell_beg;
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) {
        if (base + k < s.ncells) out[base + k] = run;
        run += v[k];
    }
}

// ---- resort ------------------------------------------------------------------
// Entry k of the cell of rank h moves to slot rank_start[h] + k; the entry
// follows.
template <class T>
__global__ void __launch_bounds__(256) k_resort_scatter(DevSys<T> s) {
    if (s.ctrl->abort) return;
    for (int h = blockIdx.x * blockDim.x + threadIdx.x; h < s.ncells; h += gridDim.x * blockDim.x) {
        const int c = s.cell_by_rank[h];
        if (!s.now[s.cell_rep[c]]) continue;
        V4<T>* p = s.cell_ent + s.cell_beg[c];
        const int b = s.rank_start[h], e = s.cell_beg[c + 1] - s.cell_beg[c];
        for (int k = 0; k < e; ++k) {
            s.perm[b + k] = bits_as_int(p[k].w);
            p[k].w = int_bits_as(T(0), b + k);
            if constexpr (sizeof(T) == 8) s.cell_ent32[s.cell_beg[c] + k].w = __int_as_float(b + k);
        }
    }
}

template <class T>
__global__ void __launch_bounds__(TILE) k_gather(DevSys<T> s, int cur, int permute_force) {
    if (s.ctrl->abort) return;
    const V4<T>* __restrict__ P = s.pos[cur];
    V4<T>* __restrict__ Q = s.pos[cur ^ 1];
    for (int t = blockIdx.x; t < s.ntiles; t += gridDim.x) {
        const Tile tl = s.tiles[t];
        if (!s.now[tl.rep] || (int)threadIdx.x >= tl.count) continue;
        const int n = tl.start + threadIdx.x;
        const int o = s.perm[n];
        Q[n] = ld4<T>(P + o);
        const V4<T> v = s.vel[o];
        s.vel_alt[n] = v;
        s.img_alt[n] = s.img[o];
        if (permute_force) s.frc_alt[n] = s.frc[o];
        s.slot_of_id[s.reps[tl.rep].p_off + bits_as_int(v.w)] = n;
    }
}

template <class T>
__global__ void __launch_bounds__(TILE) k_copyback(DevSys<T> s, int cur, int permute_force) {
    if (s.ctrl->abort) return;
    V4<T>* __restrict__ P = s.pos[cur];
    const V4<T>* __restrict__ Q = s.pos[cur ^ 1];
    for (int t = blockIdx.x; t < s.ntiles; t += gridDim.x) {
        const Tile tl = s.tiles[t];
        if (!s.now[tl.rep] || (int)threadIdx.x >= tl.count) continue;
        const int n = tl.start + threadIdx.x;
        P[n] = Q[n];
        const V4<T> v = s.vel_alt[n];
        s.vel[n] = v;
        s.img[n] = s.img_alt[n];
        if (permute_force) s.frc[n] = s.frc_alt[n];
        const int2 pg = s.bond_gid[s.reps[tl.rep].p_off + bits_as_int(v.w)];
        s.bond_slot[n] = make_int2(pg.x >= 0 ? s.slot_of_id[pg.x] : -1,
                                   pg.y >= 0 ? s.slot_of_id[pg.y] : -1);
    }
}

template <class T>
__global__ void k_request_all(DevSys<T> s) {
    for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < s.R; r += gridDim.x * blockDim.x)
        s.req[r] = 1;
    if (blockIdx.x == 0 && threadIdx.x == 0) s.ctrl->any_req = 1;
}

// ---- launchers -------------------------------------------------------------------
static inline int grid_for(int n, int block) { return (n + block - 1) / block; }

template <class T>
int Launch<T>::rebuild(const DevSys<T>& s, int cur, bool resort, bool permute_force, cudaStream_t st) {
    const int gt = s.ntiles;
    const int gc = grid_for(s.ncells, 256);
    k_prep<T><<<gc, 256, 0, st>>>(s);
    k_bin<T><<<gt, TILE, 0, st>>>(s, cur);
    k_scan_reduce<T, false><<<s.nscan_blocks, SCAN_THREADS, 0, st>>>(s);
    k_scan_top<T><<<1, SCAN_THREADS, 0, st>>>(s);
    k_scan_down<T, false><<<s.nscan_blocks, SCAN_THREADS, 0, st>>>(s);
    k_place<T><<<gt, TILE, 0, st>>>(s, cur);
    k_cellsort<T><<<gc, 256, 0, st>>>(s);
    int launched = 7;
    if (resort) {
        k_scan_reduce<T, true><<<s.nscan_blocks, SCAN_THREADS, 0, st>>>(s);
        k_scan_top<T><<<1, SCAN_THREADS, 0, st>>>(s);
        k_scan_down<T, true><<<s.nscan_blocks, SCAN_THREADS, 0, st>>>(s);
        k_resort_scatter<T><<<gc, 256, 0, st>>>(s);
        k_gather<T><<<gt, TILE, 0, st>>>(s, cur, permute_force ? 1 : 0);
        k_copyback<T><<<gt, TILE, 0, st>>>(s, cur, permute_force ? 1 : 0);
        launched += 6;
    }
    // list-free mode: the binning is all that is needed
    if (s.cells_mode) return launched;
    Launch<T>::verlet(s, cur, st);
    launched += 1;
    // mirrored entries for the learned potential's pair-once evaluation
    if (s.mlp_on && s.mlp_rev) launched += Launch<T>::mlp_rev(s, st);
    return launched;
}

template <class T>
void Launch<T>::request_all(const DevSys<T>& s, cudaStream_t st) {
    k_request_all<T><<<grid_for(s.R, 256), 256, 0, st>>>(s);
}

template int Launch<float>::rebuild(const DevSys<float>&, int, bool, bool, cudaStream_t);
template int Launch<double>::rebuild(const DevSys<double>&, int, bool, bool, cudaStream_t);
template void Launch<float>::request_all(const DevSys<float>&, cudaStream_t);
template void Launch<double>::request_all(const DevSys<double>&, cudaStream_t);

int scan_blocks_for(int ncells) { return (ncells + SCAN_TILE - 1) / SCAN_TILE; }

}  // namespace espp
