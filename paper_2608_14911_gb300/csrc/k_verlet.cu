// The Verlet list search (paper "Example usage": VerletList(system, cutoff)
// with system.skin; "Performance optimizations": cells of the list radius / W,
// W = 1, 2 or 3).
//
// A particle's stencil is (2W+1)^2 rows of up to 2W+1 cells; the cells of a row
// are consecutive in index order, so a row is one contiguous range of the entry
// array, and one more where it crosses a face of the box.
//
// What bounds it is instruction issue: about six (whole cells) candidates are
// tested per hit, and a warp that branches on every hit runs that branch for
// nearly every candidate (1 - (5/6)^32) with a few lanes in it.  So the search
// has no hit branch: a hit is one predicated store of the entry into the lane's
// column of shared memory (conflict-free: the column is the bank), and the
// columns are written out as whole int4 groups, all lanes together, when they
// fill and at the end.  KG melt, 1M beads, FP32, whole cells: 138 us a build under
// ncu, 95.0 M warp instructions, 23 of 32 lanes active (with the hit branch 226 us,
// 172.6 M, 14); LJ fluid, 4.2M, half cells: 1.8 ms (3.1 ms).  What is left is
// half issue (54%) and half the L1 data pipe (64%: each candidate is a 16-byte
// gather of its own).
//
// FP64 handles test the candidates in FP32, on float copies of the entries; a
// candidate nearer to the list radius than those coordinates' error is marked
// and gets the exact FP64 test when its column is written out: the same list,
// with the FP64 unit idle but for a few pairs in a hundred thousand.
#include "kernels.cuh"

namespace espp {

// entries a lane's column holds, and candidates in flight per lane (LJ fluid of
// 4.2M, rebuild node per step: 2 336 us, 4 301, 6 305, 8 320)
constexpr int VB = 32;
constexpr int VU = 4;
// lanes that share one particle in the team form, entries of a team's buffer
constexpr int VTEAM = 8;
constexpr int VTB = 64;
static_assert(VTEAM >= 4, "a team carries a partial group of up to three entries");
// Handles below these particle counts take the team form: with one thread per
// particle they leave most of the chip idle, and a thread's search is one long
// chain.  Time of the rebuild node, thread / team, us per step: LJ fluid of
// 4,000, FP32 17.5 / 14.9 (27,436: 19.4 / 21.0); FP64 (whose exact tests add to
// the chain) KG melt of 1,000 13.5 / 12.4, LJ fluid of 27,436 90 / 47, KG melt of
// 40,000 15.3 / 16.9.
template <class T> constexpr int verlet_team_below() { return sizeof(T) == 4 ? 8192 : 32768; }

// x cells of the particle's chord in a row, clipped to the stencil
struct RowSpan {
    int lo, hi;
};

// The search of one particle by TS lanes (1, or VTEAM neighbouring lanes).
// TS = 1: `col` is the lane's column (stride 32); TS > 1: the team's buffer
// (stride 1), filled in candidate order by ballots.
template <class T, int W, bool EXCL, bool LE, int TS>
struct VerletSearch {
    const DevSys<T>& s;
    const RepGeom<T>& g;
    const float4* __restrict__ EF;  // entries in FP32 (x, y, z, slot bits)
    int* col;
    int idx;        // the particle's own entry
    int i;          // its storage slot
    V4<T> xi;
    float fx, fy, fz;
    int2 ex;
    int sub;        // lane inside the team
    unsigned int tmask;  // the team's lanes
    int cnt = 0;    // entries waiting in the column
    int done = 0;   // whole groups written
    float rl2f;     // list radius^2 of the FP32 test
    float rl2in;    // FP64 handles: below it the FP32 test is certain
    const V4<T>* __restrict__ P;
    T le_d = T(0), inv_L0 = T(0);
    int4* __restrict__ out4;

    static constexpr bool EXACT = sizeof(T) == 4;  // the FP32 test is the handle's own
    static constexpr int CS = TS == 1 ? 32 : 1;    // column stride
    static constexpr int CAPB = TS == 1 ? VB : VTB;
    static constexpr int STEP = TS * (TS == 1 ? VU : 2);

    __device__ __forceinline__ VerletSearch(const DevSys<T>& s_, const RepGeom<T>& g_) : s(s_), g(g_) {}

    // ---- candidates [p, e) of one row ---------------------------------------
    // SHIFT: the range lies across a face (coordinates shifted as the image
    // codes say); without it the difference is the plain one, which equals the
    // shifted form with zero shifts.  LEX: a row across a sheared face: x is the
    // nearest image of x_i - nz delta - x_j (xL holds nz delta).  Reads up to
    // STEP - 1 entries past e (the array is padded).
    template <bool SHIFT, bool LEX>
    __device__ __forceinline__ void range(int p, int e, float xo, float yo, float zo, float xL, float yL, float zL,
                                          int tag) {
        constexpr int U = STEP / TS;
        const float Lx = LEX ? (float)g.L[0] : 0.f, inv = LEX ? (float)inv_L0 : 0.f;
        for (; p < e; p += STEP) {
            float4 x[U];
#pragma unroll
            for (int k = 0; k < U; ++k) x[k] = __ldg(EF + p + k * TS + sub);
#pragma unroll
            for (int k = 0; k < U; ++k) {
                const int q = p + k * TS + sub;
                float dx;
                if (LEX) {
                    dx = (xo - x[k].x) - xL;
                    dx -= Lx * rintf(dx * inv);
                } else {
                    dx = SHIFT ? xo - (x[k].x - xL) : xo - x[k].x;
                }
                const float dy = SHIFT ? yo - (x[k].y - yL) : yo - x[k].y;
                const float dz = SHIFT ? zo - (x[k].z - zL) : zo - x[k].z;
                const int j = __float_as_int(x[k].w);
                const float r2 = dx * dx + dy * dy + dz * dz;
                bool hit = r2 < rl2f && q != idx && (q < e || (TS == 1 && k == 0));
                if (EXCL) hit = hit && j != ex.x && j != ex.y;
                int val = j | tag;
                if (!EXACT && !(r2 < rl2in)) val |= (int)0x80000000;  // too near the list radius to tell
                if constexpr (TS == 1) {
                    if (hit) {
                        col[cnt * CS] = val;
                        ++cnt;
                    }
                } else {
                    const unsigned int m = __ballot_sync(tmask, hit) & tmask;
                    if (hit) col[cnt + __popc(m & ((1u << (threadIdx.x & 31)) - 1u))] = val;
                    cnt += __popc(m);
                }
            }
            if (cnt > CAPB - STEP) flush();
        }
    }

    // FP64 handles: the exact test of a waiting entry too near the list radius
    // for the FP32 one
    __device__ __forceinline__ bool exact_hit(int v) const {
        const int code = (v & 0x7fffffff) >> NBR_INDEX_BITS;
        const V4<T> xj = ld4<T>(P + nbr_slot(v));
        T dx;
        if (LE && (code & 3) == 3) {
            const T nd = (code >> 4) == 1 ? le_d : -le_d;
            dx = (xi.x - xj.x) - nd;
            dx -= g.L[0] * rint(dx * inv_L0);
        } else {
            dx = shifted_diff(xi.x, xi.x - g.L[0], xj.x, g.L[0], code & 3);
        }
        const T dy = shifted_diff(xi.y, xi.y - g.L[1], xj.y, g.L[1], (code >> 2) & 3);
        const T dz = shifted_diff(xi.z, xi.z - g.L[2], xj.z, g.L[2], code >> 4);
        return dx * dx + dy * dy + dz * dz < s.rlist2;
    }

    // the waiting entries that belong to the list, in place
    __device__ __forceinline__ void settle() {
        if constexpr (!EXACT) {
            if constexpr (TS == 1) {
                int w = 0;
                for (int k = 0; k < cnt; ++k) {
                    const int v = col[k * CS];
                    if (v < 0 && !exact_hit(v)) continue;
                    col[w * CS] = v & 0x7fffffff;
                    ++w;
                }
                cnt = w;
            } else {
                __syncwarp(tmask);
                int w = 0;
                for (int k = 0; k < cnt; k += TS) {
                    const int v = k + sub < cnt ? col[k + sub] : 0;
                    const bool keep = k + sub < cnt && (v >= 0 || exact_hit(v));
                    const unsigned int m = __ballot_sync(tmask, keep) & tmask;
                    if (keep) col[w + __popc(m & ((1u << (threadIdx.x & 31)) - 1u))] = v & 0x7fffffff;
                    w += __popc(m);
                    __syncwarp(tmask);
                }
                cnt = w;
            }
        }
    }

    // the whole groups of the column, then the rest to its start
    __device__ __forceinline__ void flush() {
        settle();
        const int ng = cnt >> 2;
        const int gcap = s.cap >> 2;
        const size_t stride = (size_t)s.stride;
        if constexpr (TS == 1) {
            for (int q = 0; q < ng; ++q) {
                const int4 v = make_int4(col[(4 * q) * CS], col[(4 * q + 1) * CS], col[(4 * q + 2) * CS],
                                         col[(4 * q + 3) * CS]);
                if (done + q < gcap) out4[(size_t)(done + q) * stride] = v;
            }
            const int r = cnt & 3;
            for (int k = 0; k < r; ++k) col[k * CS] = col[(4 * ng + k) * CS];
            cnt = r;
        } else {
            __syncwarp(tmask);
            for (int q = sub; q < ng; q += TS)
                if (done + q < gcap) out4[(size_t)(done + q) * stride] = reinterpret_cast<const int4*>(col)[q];
            const int r = cnt & 3;
            const int keep = sub < r ? col[4 * ng + sub] : 0;
            __syncwarp(tmask);
            if (sub < r) col[sub] = keep;
            __syncwarp(tmask);
            cnt = r;
        }
        done += ng;
    }

    // ---- the stencil -----------------------------------------------------------
    // With W >= 2 a row is searched only over the x cells that the list
    // sphere's chord at the row's nearest point reaches, and rows the sphere
    // misses are skipped: the row lies dmin_y, dmin_z away (the particle's
    // offset inside its own cell to the row's slab), the chord's half-width is
    // sqrt(rl^2 - dmin^2).  Margins of 1e-4 cell (more where the grid is so long
    // that FP32 cell units round coarser) widen every range against rounding;
    // the distance test itself is unchanged.  A third of the candidates go.
    // On whole cells the trimming costs more per row than the quarter of the
    // candidates it saves.
    float ux, fcy, fcz, ey, ez, cpl0, margin;
    int cx, cy, cz;
    bool live;

    __device__ __forceinline__ float slab(int d, float f, float edge) const {
        const float m = d > 0 ? (float)d - f : (d < 0 ? f + (float)(-d - 1) : 0.f);
        return m > margin ? (m - margin) * edge : 0.f;
    }
    __device__ __forceinline__ RowSpan span(int dy, float dz2) const {
        if (W == 1) return {cx - W, cx + W};
        const float dmy = slab(dy, fcy, ey);
        const float d2 = dmy * dmy + dz2;
        if (!(d2 < rl2f)) return {0, -1};
        const float wc = sqrtf(rl2f - d2) * cpl0 + margin;
        return {max(cx - W, (int)floorf(ux - wc)), min(cx + W, (int)floorf(ux + wc))};
    }

    // rows in ascending (z, y), each in ascending x, unwrapped: the list's
    // order, whichever form walks it
    __device__ __forceinline__ void stencil() {
        const int nc0 = g.nc[0], nc1 = g.nc[1], nc2 = g.nc[2];
        const bool near = live && (cx < W || cx + W >= nc0 || cy < W || cy + W >= nc1 || cz < W || cz + W >= nc2);
        // lanes whose stencil crosses a face: their warp takes the general form
        if (TS == 1 ? __any_sync(0xffffffffu, near) : near) faces();
        else inside();
    }

    // every row inside the box
    __device__ __forceinline__ void inside() {
        const int nc0 = g.nc[0], nc1 = g.nc[1];
        const int* __restrict__ B = s.cell_beg;
        // (one copy of the row's code: with the rows of a plane unrolled and their
        // ranges loaded together the loop left the instruction cache, LJ fluid of
        // 4.2M, half cells, 350 us per step instead of 301)
#pragma unroll 1
        for (int dz = -W; dz <= W; ++dz) {
            const float dmz = W > 1 ? slab(dz, fcz, ez) : 0.f;
#pragma unroll 1
            for (int dy = -W; dy <= W; ++dy) {
                const RowSpan c = span(dy, dmz * dmz);
                int pb = 0, pe = 0;
                if (live && c.lo <= c.hi) {
                    const int base = g.cell_off + ((cz + dz) * nc1 + cy + dy) * nc0;
                    pb = __ldg(B + base + c.lo);
                    pe = __ldg(B + base + c.hi + 1);
                }
                range<false, false>(pb, pe, fx, fy, fz, 0.f, 0.f, 0.f, 0);
            }
            // the warp's columns are written together once some lane has many
            if (TS == 1 && __any_sync(0xffffffffu, cnt > VB / 2)) flush();
        }
    }

    // the same rows where some lane's stencil crosses a face: a row is the
    // piece below the box (image code 2), the one inside and the one above
    // (code 1), those across a face with shifted coordinates
    __device__ __forceinline__ void faces() {
        const int nc0 = g.nc[0], nc1 = g.nc[1], nc2 = g.nc[2];
        const int* __restrict__ B = s.cell_beg;
        const float L0 = (float)g.L[0], L1 = (float)g.L[1], L2 = (float)g.L[2];
#pragma unroll 1
        for (int dz = -W; dz <= W; ++dz) {
            int az = cz + dz, czc = 0;
            if (az < 0) { az += nc2; czc = 2; }
            else if (az >= nc2) { az -= nc2; czc = 1; }
            const float dmz = W > 1 ? slab(dz, fcz, ez) : 0.f;
            const float zo = (czc & 1) ? (float)(xi.z - g.L[2]) : fz, zL = (czc & 2) ? L2 : 0.f;
            const bool sheared = LE && czc != 0;
            int cxs = 0;
            T nd = T(0);
            if (sheared) {
                // the partners' image is displaced by nz delta along x; its x
                // cells are found around x_i - nz delta, cyclic in the row
                nd = czc == 1 ? le_d : -le_d;
                T xs = xi.x - nd;
                if (xs < T(0)) xs += g.L[0];
                if (xs >= g.L[0]) xs -= g.L[0];
                cxs = cell_coord(xs, g.cells_per_len[0], nc0);
            }
#pragma unroll 1
            for (int dy = -W; dy <= W; ++dy) {
                int ay = cy + dy, cyc = 0;
                if (ay < 0) { ay += nc1; cyc = 2; }
                else if (ay >= nc1) { ay -= nc1; cyc = 1; }
                const float yo = (cyc & 1) ? (float)(xi.y - g.L[1]) : fy, yL = (cyc & 2) ? L1 : 0.f;
                const int base = g.cell_off + (az * nc1 + ay) * nc0;
                RowSpan c = sheared ? RowSpan{cxs - W, cxs + W} : span(dy, dmz * dmz);
                if (!live) c.hi = c.lo - 1;
                const int rest = (cyc << 2) | (czc << 4);
#pragma unroll 1
                for (int part = 0; part < 3; ++part) {
                    const int lo = part == 0 ? c.lo + nc0 : part == 1 ? max(c.lo, 0) : max(c.lo, nc0) - nc0;
                    const int hi = part == 0 ? min(c.hi, -1) + nc0 : part == 1 ? min(c.hi, nc0 - 1) : c.hi - nc0;
                    const bool some = lo <= hi;
                    const int p = some ? __ldg(B + base + lo) : 0, e = some ? __ldg(B + base + hi + 1) : 0;
                    const int cxc = part == 0 ? 2 : part == 2 ? 1 : 0;
                    if (LE && sheared)
                        range<true, true>(p, e, fx, yo, zo, (float)nd, yL, zL, (3 | rest) << NBR_INDEX_BITS);
                    else if ((cxc | rest) == 0)
                        range<false, false>(p, e, fx, fy, fz, 0.f, 0.f, 0.f, 0);
                    else
                        range<true, false>(p, e, (cxc & 1) ? (float)(xi.x - g.L[0]) : fx, yo, zo,
                                           (cxc & 2) ? L0 : 0.f, yL, zL, (cxc | rest) << NBR_INDEX_BITS);
                }
            }
            if (TS == 1 && __any_sync(0xffffffffu, cnt > VB / 2)) flush();
        }
    }

    __device__ __forceinline__ void setup(int idx_, bool live_) {
        idx = idx_;
        live = live_;
        xi = ld4<T>(s.cell_ent + idx);
        i = bits_as_int(xi.w);
        fx = (float)xi.x;
        fy = (float)xi.y;
        fz = (float)xi.z;
        ex = EXCL ? s.bond_slot[i] : make_int2(-1, -1);
        out4 = reinterpret_cast<int4*>(s.nbr) + i;
        if (LE) {
            // delta of this build reduced into [0, Lx)
            le_d = (T)le_reduce(s.le_db[(int)(&g - s.reps)], (double)g.L[0]);
            inv_L0 = T(1) / g.L[0];
        }
        cx = cell_coord(xi.x, g.cells_per_len[0], g.nc[0]);
        cy = cell_coord(xi.y, g.cells_per_len[1], g.nc[1]);
        cz = cell_coord(xi.z, g.cells_per_len[2], g.nc[2]);
        if constexpr (EXACT) {
            rl2f = (float)s.rlist2;
        } else {
            // rl^2 widened by the rounding of the float coordinates: every
            // component of a difference is off by at most 2^-23 Lmax (both
            // operands rounded to nearest) plus its own rounding, and by that
            // again where a sheared image is taken
            const float Lm = (float)fmax((double)g.L[0], fmax((double)g.L[1], (double)g.L[2]));
            const float r2 = (float)s.rlist2, r = sqrtf(r2), e = 6e-7f * (Lm + r);
            const float m = 2.f * 1.7320509f * r * e + 3.f * e * e;
            rl2f = (r2 + m) * 1.000001f;
            rl2in = (r2 - m) * 0.999999f;
        }
        if (W > 1) {
            cpl0 = (float)g.cells_per_len[0];
            ux = (float)(xi.x * g.cells_per_len[0]);
            fcy = (float)(xi.y * g.cells_per_len[1] - (T)cy);
            fcz = (float)(xi.z * g.cells_per_len[2] - (T)cz);
            ey = (float)g.L[1] / (float)g.nc[1];
            ez = (float)g.L[2] / (float)g.nc[2];
            margin = fmaxf(1e-4f, 5e-7f * (float)max(g.nc[0], max(g.nc[1], g.nc[2])));
        }
    }

    // the last, partial group and the particle's count; returns the count
    __device__ __forceinline__ int finish() {
        flush();
        const int total = 4 * done + cnt;
        const int cap = s.cap, pad = s.nbr_pad;
        if (live && (TS == 1 || sub == 0)) {
            if (cnt != 0 && done < (cap >> 2)) {
                const int a = col[0], b = cnt > 1 ? col[CS] : pad, c = cnt > 2 ? col[2 * CS] : pad;
                out4[(size_t)done * s.stride] = make_int4(a, b, c, pad);
            }
            s.nbr_cnt[i] = total < cap ? total : cap;
            s.xb[i] = xi;
            if (total > cap) {
                atomicMax(&s.ctrl->need_cap, (unsigned int)total);
                atomicOr(&s.ctrl->err, ERRBIT_OVERFLOW);
                s.ctrl->abort = 1;
            }
        }
        return total;
    }
};

// One thread per particle, threads in entry (cell) order: a warp walks a run of
// cells along x, whose stencils share their rows.
template <class T, int W, bool EXCL, bool LE>
__global__ void __launch_bounds__(TILE, sizeof(T) == 4 ? 8 : 6) k_verlet(DevSys<T> s, int cur) {
    __shared__ int buf[TILE / 32][VB * 32];
    ActiveTiles<T> at(s);
    if (s.ctrl->abort) return;
    Tile tl;
    while (at.next(tl)) {  // (uniform over the block)
        VerletSearch<T, W, EXCL, LE, 1> v(s, s.reps[tl.rep]);
        v.EF = entries_f(s);
        v.P = sizeof(T) == 8 ? s.pos[buffer_of(s, cur)] : nullptr;  // (FP32 handles have no second test)
        v.col = buf[threadIdx.x >> 5] + (threadIdx.x & 31);
        v.sub = 0;
        v.tmask = 0;
        // a replica's entries fill the same index range as its slots; idle
        // threads of the last tile walk along with empty ranges
        const bool live = (int)threadIdx.x < tl.count;
        v.setup(tl.start + (live ? (int)threadIdx.x : 0), live);
        v.stencil();
        int cnt = v.finish();
        if (!live) cnt = 0;
        // largest count: one atomic per warp, no block barrier
        cnt = __reduce_max_sync(0xffffffffu, cnt);
        if ((threadIdx.x & 31) == 0 && cnt > 0) atomicMax(&s.ctrl->max_count, (unsigned int)cnt);
    }
}

// VTEAM lanes per particle (TILE / VTEAM particles per block), for systems that
// do not fill the chip with one thread per particle.
template <class T, int W, bool EXCL, bool LE>
__global__ void __launch_bounds__(TILE, 6) k_verlet_team(DevSys<T> s, int cur) {
    __shared__ __align__(16) int buf[TILE / VTEAM][VTB];
    if (s.ctrl->abort) return;
    const int t = blockIdx.x / VTEAM;
    if (t >= s.ntiles) return;
    const Tile tl = s.tiles[t];
    if (!s.now[tl.rep]) return;  // uniform over the block
    const int lane = threadIdx.x & 31, team = threadIdx.x / VTEAM;
    const int q = (blockIdx.x % VTEAM) * (TILE / VTEAM) + team;
    if (q >= tl.count) return;   // whole teams
    VerletSearch<T, W, EXCL, LE, VTEAM> v(s, s.reps[tl.rep]);
    v.EF = entries_f(s);
    v.P = sizeof(T) == 8 ? s.pos[buffer_of(s, cur)] : nullptr;  // (FP32 handles have no second test)
    v.col = buf[team];
    v.sub = lane % VTEAM;
    v.tmask = ((1u << VTEAM) - 1u) << (lane / VTEAM * VTEAM);
    v.setup(tl.start + q, true);
    v.stencil();
    const int cnt = v.finish();
    if (v.sub == 0 && cnt > 0) atomicMax(&s.ctrl->max_count, (unsigned int)cnt);
}

template <class T>
void Launch<T>::verlet(const DevSys<T>& s, int cur, cudaStream_t st) {
    const bool team = s.N < verlet_team_below<T>();
#define ESPP_VERLET(W, E)                                                                                  \
    do {                                                                                                   \
        if (team) {                                                                                        \
            if (s.le_on) k_verlet_team<T, W, E, true><<<s.ntiles * VTEAM, TILE, 0, st>>>(s, cur);               \
            else k_verlet_team<T, W, E, false><<<s.ntiles * VTEAM, TILE, 0, st>>>(s, cur);                      \
        } else {                                                                                           \
            if (s.le_on) k_verlet<T, W, E, true><<<active_grid(s), TILE, 0, st>>>(s, cur);                            \
            else k_verlet<T, W, E, false><<<active_grid(s), TILE, 0, st>>>(s, cur);                                   \
        }                                                                                                  \
    } while (0)
#define ESPP_VERLET_W(E)                    \
    do {                                    \
        if (s.cell_w == 1) ESPP_VERLET(1, E);      \
        else if (s.cell_w == 2) ESPP_VERLET(2, E); \
        else ESPP_VERLET(3, E);                    \
    } while (0)
    if (s.excl_bonded) ESPP_VERLET_W(true);
    else ESPP_VERLET_W(false);
#undef ESPP_VERLET_W
#undef ESPP_VERLET
}

#if !defined(ESPP_STEP_PRECISION) || ESPP_STEP_PRECISION == 32
template void Launch<float>::verlet(const DevSys<float>&, int, cudaStream_t);
#endif
#if !defined(ESPP_STEP_PRECISION) || ESPP_STEP_PRECISION == 64
template void Launch<double>::verlet(const DevSys<double>&, int, cudaStream_t);
#endif

}  // namespace espp
