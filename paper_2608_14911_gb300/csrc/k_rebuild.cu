// Rebuild pipeline: linked-cell binning, the periodic Hilbert resort of every
// particle array into cell order, and the full Verlet list with skin.  Paper
// "Software design" ("Parallelization": CellGrid linked cells;
// "Performance optimizations": cell decomposition and data sorting) and
// "Example usage" (VerletList(system, cutoff) with system.skin).
//
// Every rebuild (inside the step graphs, when a replica asked for it):
//   latch     the per-replica requests
//   bin       cell of every particle and its arrival index (atomic histogram)
//   scan      exclusive scan of the counts in cell-index order: first entry of
//             every cell in one compact entry array (no per-cell capacity); the
//             counts are cleared for the next build
//   place     every particle's storage slot at its arrival place in its cell
//   rank      a particle's rank among its cell's slots gives its entry (position,
//             storage slot) its place: entries of a cell in ascending slot, so the
//             list does not depend on the order of the atomics
//   verlet    (k_verlet.cu) stencil search from the cell entries, streamed as
//             contiguous row ranges; full list (both directions) as groups of
//             four indices, nbr4[g * stride + i]; records the build positions
// The phases up to rank are one cooperative kernel (k_binning) on handles small
// enough for launches to count, and kernels of their own beyond.
// A resort (launched between step graphs every `resort_every` steps, and on
// every explicit build) additionally runs, between rank and verlet:
//   scan      exclusive scan of the cell counts in Hilbert-rank order
//   scatter   new slot of every entry (its cell's first slot + its rank in the
//             cell); the entries switch to the new slots
//   gather    permuted copies of positions, velocities, forces, images
//   copyback  copies back and maps bond partners to their new slots
// Replicas whose request flag is clear skip every per-particle step after the
// latch; their entries stay those of their last build, in their own slot range.
#include <algorithm>

#include "grid_barrier.cuh"
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

// The requests of this rebuild, by one block.  Lees-Edwards: the offset at this
// build as well, for the rebuild criterion and the sheared rows of the search
// (kept as stored after a checkpoint load).
template <class T>
__device__ __forceinline__ void latch_requests(const DevSys<T>& s) {
    const long long pstep = s.ctrl->step + (long long)s.ctrl->pos_ahead;
    const bool keep = s.ctrl->le_keep != 0;
    for (int r = threadIdx.x; r < s.R; r += blockDim.x) {
        s.now[r] = s.req[r];
        if (s.le_on && s.req[r] && !keep) s.le_db[r] = le_offset(s, s.reps[r], pstep);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        s.ctrl->le_keep = 0;
        if (s.ctrl->any_req) {
            s.ctrl->n_rebuilds += 1;
            s.ctrl->max_count = 0;
        }
    }
}

template <class T>
__device__ __forceinline__ void clear_requests(const DevSys<T>& s) {
    for (int r = threadIdx.x; r < s.R; r += blockDim.x) s.req[r] = 0;
    if (threadIdx.x == 0) s.ctrl->any_req = 0;
}

// Cell of particle i and its arrival index in that cell (counting-sort
// histogram); positions are wrapped into the box here, at list builds only.
template <class T>
__device__ __forceinline__ void bin_particle(const DevSys<T>& s, V4<T>* P, const RepGeom<T>& g, int rep, int i) {
    V4<T> p = P[i];
    int wx, wy, wz;
    if (s.le_on && !(p.z >= T(0) && p.z < g.L[2])) {
        // across a sheared face: the image entered is displaced and moving
        const double L[3] = {(double)g.L[0], (double)g.L[1], (double)g.L[2]};
        double q[3] = {(double)p.x, (double)p.y, (double)p.z};
        V4<T> v = s.vel[i];
        double vx = (double)v.x;
        int k[3];
        le_wrap(q, vx, k, L, s.le_db[rep], s.le_shear);
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

// Entry of particle i: its rank among the slots of its cell (a few to a few dozen,
// contiguous; all of them read by every thread of the cell, so mostly from L1).
template <class T>
__device__ __forceinline__ void rank_particle(const DevSys<T>& s, const V4<T>* P, int i) {
    const int h = s.cellh[i];
    const int b = s.cell_beg[h], e = s.cell_beg[h + 1];
    V4<T> p = P[i];
    int rank = 0;
    for (int k = b; k < e; ++k) rank += s.cell_slot[k] < i ? 1 : 0;
    s.in_cell[i] = rank;
    p.w = int_bits_as(T(0), i);
    s.cell_ent[b + rank] = p;
    // FP64 handles: the float copies that the list search tests
    if constexpr (sizeof(T) == 8)
        s.cell_ent32[b + rank] = make_float4((float)p.x, (float)p.y, (float)p.z, __int_as_float(i));
    // list-free mode with DPD: the velocities in entry order as well
    if (s.cells_mode && s.dpd) s.cell_vel[b + rank] = s.vel[i];
}

// One block: the requests and, for batches, the list of the tiles to rebuild (in
// a batch some replica asks at nearly every step, a tenth of them at a time).
template <class T>
__global__ void __launch_bounds__(SCAN_THREADS) k_latch(DevSys<T> s) {
    if (s.ctrl->abort) return;
    latch_requests(s);
    if (s.R == 1) return;
    int carry = 0;
    for (int r0 = 0; r0 < s.R; r0 += SCAN_THREADS) {
        const int r = r0 + threadIdx.x;
        const bool on = r < s.R && s.now[r] != 0;
        const int a = on ? s.rep_tile_off[r] : 0, n = on ? s.rep_tile_off[r + 1] - a : 0;
        int excl;
        const int total = block_excl_scan(n, &excl);
        // a thread writes its replica's tiles; a warp with a large replica among its
        // 32 writes them together, one replica after the other
        if (__any_sync(0xffffffffu, n > 128)) {
            for (unsigned int left = __ballot_sync(0xffffffffu, n > 0); left; left &= left - 1) {
                const int q = __ffs(left) - 1;
                const int to = carry + __shfl_sync(0xffffffffu, excl, q), from = __shfl_sync(0xffffffffu, a, q),
                          m = __shfl_sync(0xffffffffu, n, q);
                for (int k = threadIdx.x & 31; k < m; k += 32) s.act[to + k] = from + k;
            }
        } else {
            for (int k = 0; k < n; ++k) s.act[carry + excl + k] = a + k;
        }
        carry += total;
    }
    if (threadIdx.x == 0) s.ctrl->nact = carry;
}

template <class T>
__global__ void __launch_bounds__(TILE) k_bin(DevSys<T> s, int cur) {
    ActiveTiles<T> at(s);
    if (s.ctrl->abort) return;
    if (blockIdx.x == 0) clear_requests(s);
    V4<T>* P = s.pos[buffer_of(s, cur)];
    Tile tl;
    while (at.next(tl))
        if ((int)threadIdx.x < tl.count) bin_particle(s, P, s.reps[tl.rep], tl.rep, tl.start + threadIdx.x);
}

template <class T>
__global__ void __launch_bounds__(TILE) k_place(DevSys<T> s) {
    ActiveTiles<T> at(s);
    if (s.ctrl->abort) return;
    Tile tl;
    while (at.next(tl)) {
        const int i = tl.start + threadIdx.x;
        if ((int)threadIdx.x < tl.count) s.cell_slot[s.cell_beg[s.cellh[i]] + s.in_cell[i]] = i;
    }
}

template <class T>
__global__ void __launch_bounds__(TILE) k_rank(DevSys<T> s, int cur) {
    ActiveTiles<T> at(s);
    if (s.ctrl->abort) return;
    const V4<T>* P = s.pos[buffer_of(s, cur)];
    Tile tl;
    while (at.next(tl))
        if ((int)threadIdx.x < tl.count) rank_particle(s, P, tl.start + threadIdx.x);
}

// Batches of small replicas: one block per replica scans the cells of its replica
// alone, whose entries start at its first slot (a scan over every replica's cells
// ran at nearly every step of a batch for the tenth of them that had asked).
template <class T>
__global__ void __launch_bounds__(SCAN_THREADS) k_scan_replica(DevSys<T> s) {
    if (s.ctrl->abort || !s.now[blockIdx.x]) return;
    const RepGeom<T>& g = s.reps[blockIdx.x];
    const int n = g.nc[0] * g.nc[1] * g.nc[2];
    int* cnt = s.cell_cnt + g.cell_off;
    int* beg = s.cell_beg + g.cell_off;
    int carry = g.p_off;
    for (int k0 = 0; k0 < n; k0 += SCAN_TILE) {
        const int k = k0 + threadIdx.x * SCAN_ITEMS;
        int v[SCAN_ITEMS], sum = 0, excl;
#pragma unroll
        for (int q = 0; q < SCAN_ITEMS; ++q) {
            v[q] = k + q < n ? cnt[k + q] : 0;
            sum += v[q];
        }
        const int total = block_excl_scan(sum, &excl);
        int run = carry + excl;
#pragma unroll
        for (int q = 0; q < SCAN_ITEMS; ++q) {
            if (k + q < n) {
                beg[k + q] = run;
                cnt[k + q] = 0;
            }
            run += v[q];
        }
        carry += total;
    }
}

// ---- exclusive scan of the cell counts (three phases, no inter-block waits) --
// RANK = false: cells in index order -> cell_beg (every rebuild);
// RANK = true: cells in Hilbert-rank order -> rank_start, by cell (resort only).
// The counts of this build are in cell_cnt, which is zero between builds.  A
// replica that is not rebuilt counts all its particles in its last cell: what comes
// after starts where it did, and its own cells are neither read nor written.
template <class T, bool RANK>
__device__ __forceinline__ int scan_count(const DevSys<T>& s, int k, bool& build) {
    build = false;
    if (k >= s.ncells) return 0;
    if (RANK) {
        const int c = s.cell_by_rank[k];
        return s.cell_beg[c + 1] - s.cell_beg[c];
    }
    const int r = s.R == 1 ? 0 : s.cell_rep[k];
    build = s.now[r] != 0;
    if (build) return s.cell_cnt[k];
    if (s.R == 1 || (k + 1 < s.ncells && s.cell_rep[k + 1] == r)) return 0;
    return (r + 1 < s.R ? s.reps[r + 1].p_off : s.N) - s.reps[r].p_off;
}

template <class T, bool RANK>
__global__ void __launch_bounds__(SCAN_THREADS) k_scan_reduce(DevSys<T> s) {
    if (s.ctrl->abort) return;
    const int base = blockIdx.x * SCAN_TILE + threadIdx.x * SCAN_ITEMS;
    int sum = 0;
    bool build;
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) sum += scan_count<T, RANK>(s, base + k, build);
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
    bool build[SCAN_ITEMS];
    int sum = 0;
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) {
        v[k] = scan_count<T, RANK>(s, base + k, build[k]);
        sum += v[k];
    }
    int excl;
    block_excl_scan(sum, &excl);
    int run = s.scan_part[blockIdx.x] + excl;
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) {
        if (base + k < s.ncells) {
            if (RANK) {
                s.rank_start[s.cell_by_rank[base + k]] = run;
            } else if (build[k]) {
                s.cell_beg[base + k] = run;
                s.cell_cnt[base + k] = 0;
            }
        }
        run += v[k];
    }
}

// ---- the phases up to rank in one launch -----------------------------------------
// Every phase is a few microseconds of dependent memory accesses on a small
// handle, a kernel of its own each time costs as much again: five kernel
// boundaries become grid barriers.
template <class T>
__global__ void __launch_bounds__(SCAN_THREADS, 4) k_binning(DevSys<T> s, int cur) {
    static_assert(SCAN_THREADS % TILE == 0, "whole tiles per block");
    constexpr int TB = SCAN_THREADS / TILE;
    Ctrl* c = s.ctrl;
    // no block changes any_req before every block has read it; abort is set by a
    // block whose wait ran out, and one that starts after that is counted as left
    if (c->abort) {
        grid_leave(c, [] {});
        return;
    }
    if (!c->any_req) {
        // nothing is built: the kernels after this one read the latched flag
        if (blockIdx.x == 0 && threadIdx.x == 0) s.now[0] = 0;
        return;
    }
    V4<T>* P = s.pos[buffer_of(s, cur)];
    const int lt = threadIdx.x % TILE, t0 = blockIdx.x * TB + threadIdx.x / TILE;
    unsigned int phase = 1;
    bool ok = true;
    if (blockIdx.x == 0) latch_requests(s);
    if (s.le_on) ok = grid_barrier(c, phase++, s.bin_fault, [] {});  // (bin reads the build's offset)
    if (ok)
        for (int t = t0; t < s.ntiles; t += gridDim.x * TB) {
            const Tile tl = s.tiles[t];
            if (s.req[tl.rep] && lt < tl.count) bin_particle(s, P, s.reps[tl.rep], tl.rep, tl.start + lt);
        }
    ok = ok && grid_barrier(c, phase++, s.bin_fault, [] {});
    // the scan: every block one stretch of cells
    const int per = (s.ncells + gridDim.x - 1) / gridDim.x;
    const int c0 = min((int)blockIdx.x * per, s.ncells), c1 = min(c0 + per, s.ncells);
    int excl;
    if (ok) {
        if (blockIdx.x == 0) clear_requests(s);
        int sum = 0;
        for (int k = c0 + threadIdx.x; k < c1; k += SCAN_THREADS) sum += s.cell_cnt[k];
        const int total = block_excl_scan(sum, &excl);
        if (threadIdx.x == 0) s.scan_part[blockIdx.x] = total;
    }
    ok = ok && grid_barrier(c, phase++, s.bin_fault, [] {});
    if (ok) {
        int before = 0;
        for (int b = threadIdx.x; b < (int)blockIdx.x; b += SCAN_THREADS) before += s.scan_part[b];
        int carry = block_excl_scan(before, &excl);
        for (int k0 = c0; k0 < c1; k0 += SCAN_THREADS) {
            const int k = k0 + threadIdx.x;
            const int v = k < c1 ? s.cell_cnt[k] : 0;
            const int total = block_excl_scan(v, &excl);
            if (k < c1) {
                s.cell_beg[k] = carry + excl;
                s.cell_cnt[k] = 0;
            }
            carry += total;
        }
    }
    ok = ok && grid_barrier(c, phase++, s.bin_fault, [] {});
    if (ok)
        for (int t = t0; t < s.ntiles; t += gridDim.x * TB) {
            const Tile tl = s.tiles[t];
            const int i = tl.start + lt;
            if (s.now[tl.rep] && lt < tl.count) s.cell_slot[s.cell_beg[s.cellh[i]] + s.in_cell[i]] = i;
        }
    ok = ok && grid_barrier(c, phase++, s.bin_fault, [] {});
    if (ok)
        for (int t = t0; t < s.ntiles; t += gridDim.x * TB) {
            const Tile tl = s.tiles[t];
            if (s.now[tl.rep] && lt < tl.count) rank_particle(s, P, tl.start + lt);
        }
    grid_leave(c, [] {});
}

// ---- resort ------------------------------------------------------------------
// Particle i moves to its cell's first new slot plus its rank in the cell; its
// entry follows.
template <class T>
__global__ void __launch_bounds__(TILE) k_resort_scatter(DevSys<T> s) {
    if (s.ctrl->abort) return;
    for (int t = blockIdx.x; t < s.ntiles; t += gridDim.x) {
        const Tile tl = s.tiles[t];
        if (!s.now[tl.rep] || (int)threadIdx.x >= tl.count) continue;
        const int i = tl.start + threadIdx.x;
        const int h = s.cellh[i], rank = s.in_cell[i], n = s.rank_start[h] + rank;
        s.perm[n] = i;
        s.cell_ent[s.cell_beg[h] + rank].w = int_bits_as(T(0), n);
        if constexpr (sizeof(T) == 8) s.cell_ent32[s.cell_beg[h] + rank].w = __int_as_float(n);
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

// Blocks of the fused binning: four an SM are resident at once (its launch bounds).
int binning_blocks(int sms) { return 4 * sms; }

// The fused binning has a block for every SCAN_THREADS particles, and for every
// BIN_CELLS cells: in a dilute system the scan is most of its work.  us per step,
// blocks by particles alone / by both / kernels of their own (list; cells): gas of
// 1,000 in 287,000 cells 34.8 / 14.5 / 14.8, 577 / 32.0 / 41.3 (in 730,000); of 20,000
// 17.7 / 16.7 / 16.6, 62.6 / 41.6 / 47.7; of 90,000 in 2.3 million 20.6 / 19.8 / 20.8, 93
// / 73.5 / 110.  BIN_CELLS of 256 and 4096 instead of 1024: 5,000 in 62,000 (cells)
// 32.0 and 39.2 against 30.4, dense systems the same.
constexpr int BIN_CELLS = 4 * SCAN_THREADS;

// us per step, kernels of their own / fused: DPD fluid in cells (binned every
// step) 24,000 63.4 / 60.1, 98,304 91.2 / 90.0, 192,000 135 / 139; KG melt of 5,000
// 9.42 / 9.18, of 200,000 29.2 / 29.5: beyond some 100,000 particles a kernel's own
// blocks hide more latency than a barrier saves.
template <class T>
static bool binning_fused(const DevSys<T>& s) { return s.N < 100000 && s.R == 1; }

// A batch's cells: a block per replica, or all cells by the three phases where a
// cell's replica has many of them (the mean over cells, so that one large replica
// does not decide for hundreds of small ones).  us per step, by replica / three
// phases, KG melts on whole cells: 64 x 10,000 beads (2,700 cells) 94.4 / 97.3, 64 x
// 20,000 (5,800) 137.7 / 139.8, 64 uneven ones (10,600) 171 / 161, 64 x 50,000
// (15,600) 275 / 265, 4 x 100,000 (32,000) 65 / 51, 2 x 1,000,000 276 / 159.  The line lies
// above where the times cross: two more kernels in every captured step make a new
// handle's first call longer (the uneven batch's 10.0 -> 11.3 ms).
constexpr int SCAN_REP_CELLS = 16384;
template <class T>
static bool scan_by_replica(const DevSys<T>& s) { return s.R > 1 && s.rep_cells <= SCAN_REP_CELLS; }

template <class T>
int Launch<T>::binning_launches(const DevSys<T>& s) { return binning_fused(s) ? 1 : scan_by_replica(s) ? 5 : 7; }

template <class T>
int Launch<T>::rebuild(const DevSys<T>& s, int cur, bool resort, bool permute_force, cudaStream_t st) {
    const int gt = s.ntiles;
    int launched;
    if (binning_fused(s)) {
        DevSys<T> a = s;
        void* args[] = {&a, &cur};
        const int blocks = std::min(std::max(grid_for(s.N, SCAN_THREADS), grid_for(s.ncells, BIN_CELLS)), binning_blocks(s.sms));
        cudaLaunchCooperativeKernel((const void*)k_binning<T>, dim3(blocks), dim3(SCAN_THREADS), args, 0, st);
        launched = 1;
    } else {
        const int ga = active_grid(s);
        k_latch<T><<<1, SCAN_THREADS, 0, st>>>(s);
        k_bin<T><<<ga, TILE, 0, st>>>(s, cur);
        if (scan_by_replica(s)) {
            k_scan_replica<T><<<s.R, SCAN_THREADS, 0, st>>>(s);
        } else {
            k_scan_reduce<T, false><<<s.nscan_blocks, SCAN_THREADS, 0, st>>>(s);
            k_scan_top<T><<<1, SCAN_THREADS, 0, st>>>(s);
            k_scan_down<T, false><<<s.nscan_blocks, SCAN_THREADS, 0, st>>>(s);
        }
        k_place<T><<<ga, TILE, 0, st>>>(s);
        k_rank<T><<<ga, TILE, 0, st>>>(s, cur);
        launched = binning_launches(s);
    }
    if (resort) {
        k_scan_reduce<T, true><<<s.nscan_blocks, SCAN_THREADS, 0, st>>>(s);
        k_scan_top<T><<<1, SCAN_THREADS, 0, st>>>(s);
        k_scan_down<T, true><<<s.nscan_blocks, SCAN_THREADS, 0, st>>>(s);
        k_resort_scatter<T><<<gt, TILE, 0, st>>>(s);
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
template int Launch<float>::binning_launches(const DevSys<float>&);
template int Launch<double>::binning_launches(const DevSys<double>&);
template void Launch<float>::request_all(const DevSys<float>&, cudaStream_t);
template void Launch<double>::request_all(const DevSys<double>&, cudaStream_t);

int scan_blocks_for(int ncells) { return (ncells + SCAN_TILE - 1) / SCAN_TILE; }

}  // namespace espp
