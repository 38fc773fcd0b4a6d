// List-free pair forces from the cell stencil (paper "Performance
// optimizations": linked cells and the sub-cell decomposition of Yao et al.,
// cells of edge rc / W).  In this mode the particles are binned every step
// (the rebuild pipeline without the Verlet search) and one thread per cell
// entry streams the (2W+1)^3 neighbouring cells' entries, which the binning
// left contiguous by rows, testing each against the cutoff.  No list is built
// or read, so nothing depends on a skin: the mode pays for the binning and a
// wider candidate set every step, and wins where a Verlet list would be
// rebuilt every step or two anyway (fast particles, large time steps).
//
// The search tests the candidates in FP32 without branching on a hit and hands
// those inside to the warp's pair queue (pair_queue.cuh): one in six candidates
// lies inside the cutoff, so a kernel that evaluates a pair where it finds it
// runs the pair term (a Philox block with DPD) for nearly every candidate with a
// few lanes in it.
//
// The kernel writes per storage slot the pair force and pair energy (and, in
// the energy pass, the virial and its xz part), which the step kernel adds
// in place of its list loop; the DPD thermostat's pair term (velocities from
// the cell-ordered copy written at binning) and the Lees-Edwards planes are
// evaluated here too.
#include "kernels.cuh"
#include "pair_queue.cuh"
#include "pair_terms.cuh"

// minimum resident blocks per SM the FP32 register budget is fitted to
#ifndef ESPP_CF_MINB32
#define ESPP_CF_MINB32 8
#endif

namespace espp {

// Terms held at a time, and the lanes that share a particle where one thread per
// particle would not fill the chip.  Force kernels of a step of the DPD fluid
// (event-timed), one thread / eight lanes a particle: 3,000 45.4 / 22.9 us,
// 24,000 45.6 / 36.9, 98,304 63.7 / 90.6, 786,432 313 / 608 (evaluating every pair
// where it was found: 24,000 118, 786,432 653).
constexpr int CFR = 128;
constexpr int CFT = 8;
template <class T, bool DPD, int TS>
struct CellQueue {
    static constexpr int CFC = TS == 1 ? 16 : 32;
    int col[CFC * (32 / TS)];
    T fr[CFR], dx[CFR], dy[CFR], dz[CFR];
    T th[DPD ? CFR : 1];
};

// TS lanes per particle (1, or CFT).  Threads follow the entry array (cell
// order); a replica's entries fill the same index range as its slots.
template <class T, int W, bool ENERGY, bool MULTI, bool DPD, bool LE, int TS>
__global__ void __launch_bounds__(TILE, sizeof(T) == 4 ? ESPP_CF_MINB32 : 4) k_cellforce(DevSys<T> s, int cur) {
    __shared__ CellQueue<T, DPD, TS> queues[TILE / 32];
    if (s.ctrl->abort) return;
    constexpr int PPW = 32 / TS, CFC = CellQueue<T, DPD, TS>::CFC;
    constexpr int U = TS == 1 ? 4 : 2;       // candidates in flight per lane
    constexpr int STEP = TS * U;
    static_assert(STEP <= CFC, "a step's hits fit an empty column");
    const V4<T>* __restrict__ P = s.pos[cur];  // type bits of the partners (several types)
    const V4<T>* __restrict__ E = s.cell_ent;
    const float4* __restrict__ EF = entries_f(s);
    const V4<T>* __restrict__ VE = s.cell_vel;
    const int* __restrict__ B = s.cell_beg;
    const long long step = s.ctrl->step + (long long)s.ctrl->pos_ahead;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sub = lane % TS, pw = lane / TS;
    const unsigned int tmask = TS == 1 ? 0u : ((1u << TS) - 1u) << (pw * TS);
    CellQueue<T, DPD, TS>& Q = queues[warp];
    int* __restrict__ col = Q.col + pw;
    const int t = blockIdx.x / TS;
    if (t >= s.ntiles) return;
    const Tile tl = s.tiles[t];
    const int first = (blockIdx.x % TS) * (TILE / TS) + warp * PPW;  // the warp's first entry in the tile
    if (first >= tl.count) return;
    const bool live = first + pw < tl.count;
    const RepGeom<T>& g = s.reps[tl.rep];
    const int ibase = tl.start + first, idx = ibase + (live ? pw : 0);
    const V4<T> xi = ld4<T>(E + idx);
    const int i = bits_as_int(xi.w);
    PairRec<T> prl;
    if (!MULTI) prl = s.pair[0];
    const PairRec<T>* pr1 = MULTI ? nullptr : &prl;
    const int2 ex = s.excl_bonded ? s.bond_slot[i] : make_int2(-1, -1);
    const bool excl = s.excl_bonded != 0;
    T rcmax2 = s.rc_max2;
    if (DPD) rcmax2 = max(rcmax2, s.ip->dpd_rc2);
    float rc2 = (float)rcmax2;
    const float L0 = (float)g.L[0], L1 = (float)g.L[1], L2 = (float)g.L[2];
    if constexpr (sizeof(T) == 8) {
        // widened by the rounding of the float copies of the entries
        const float r = sqrtf(rc2), e = 6e-7f * (fmaxf(L0, fmaxf(L1, L2)) + r);
        rc2 = (rc2 + 3.47f * r * e + 3.f * e * e) * 1.000001f;
    }
    const T inv_L0 = LE ? T(1) / g.L[0] : T(0);
    // Lees-Edwards: delta of this step (binned with it) reduced into [0, Lx)
    const T le_d = LE ? (T)le_reduce(s.le_db[tl.rep], (double)g.L[0]) : T(0);
    const float linv = (float)inv_L0;
    const int nc0 = g.nc[0], nc1 = g.nc[1], nc2 = g.nc[2];
    const int cx = cell_coord(xi.x, g.cells_per_len[0], nc0);
    const int cy = cell_coord(xi.y, g.cells_per_len[1], nc1);
    const int cz = cell_coord(xi.z, g.cells_per_len[2], nc2);
    const float x = (float)xi.x, y = (float)xi.y, z = (float)xi.z;
    T fx = 0, fy = 0, fz = 0, pe = 0, vir = 0, vxz = 0;
    int cnt = 0;  // entries in the particle's column

    // the warp's queue evaluated and added; every lane takes part
    auto evaluate = [&]() {
        int total;
        const int off = queue_offsets(sub == 0 ? cnt : 0, total);
        const int from = TS == 1 ? off : __shfl_sync(0xffffffffu, off, pw * TS), to = from + cnt;
        for (int r0 = 0; r0 < total; r0 += CFR) {
            const int nr = min(CFR, total - r0);
            __syncwarp();
            for (int b = 0; b < nr; b += 32) {
                const int q = min(b + lane, nr - 1) + r0;
                int k;
                const int p = queue_owner(off, q, k) / TS;
                if (b + lane < nr) {
                    const int v = Q.col[k * PPW + p], ej = v & NBR_INDEX_MASK, code = v >> NBR_INDEX_BITS;
                    const V4<T> a = ld4<T>(E + ibase + p), xj = ld4<T>(E + ej);
                    int nz = 0;
                    T dx;
                    if (LE && (code & 3) == 3) {
                        nz = (code >> 4) == 1 ? 1 : -1;
                        dx = (a.x - xj.x) - (T)nz * le_d;
                        dx -= g.L[0] * rint(dx * inv_L0);
                    } else {
                        dx = shifted_diff(a.x, a.x - g.L[0], xj.x, g.L[0], code & 3);
                    }
                    const T dy = shifted_diff(a.y, a.y - g.L[1], xj.y, g.L[1], (code >> 2) & 3);
                    const T dz = shifted_diff(a.z, a.z - g.L[2], xj.z, g.L[2], code >> 4);
                    const T r2 = dx * dx + dy * dy + dz * dz;
                    int ti = 0, tj = 0;
                    if (MULTI) {
                        ti = bits_as_int(P[bits_as_int(a.w)].w);
                        tj = bits_as_int(P[bits_as_int(xj.w)].w);
                    }
                    Q.fr[b + lane] = pair_scalar<T, ENERGY, MULTI, false>(s, ti, pr1, dx, dz, r2, tj, pe, vir, vxz);
                    Q.dx[b + lane] = dx;
                    Q.dy[b + lane] = dy;
                    Q.dz[b + lane] = dz;
                    if (DPD) {
                        T th = T(0);
                        if (less_nonneg(r2, s.ip->dpd_rc2)) {
                            DpdCtx<T> dc;
                            dc.vi = ld4<T>(VE + ibase + p);
                            dc.seed = g.seed;
                            dc.step = step;
                            dc.le_vs = LE ? (T)(s.le_shear * (double)g.L[2]) : T(0);
                            th = dpd_value<T, LE>(s.ip, dc, dx, dy, dz, r2, ld4<T>(VE + ej), nz);
                        }
                        Q.th[b + lane] = th;
                    }
                }
            }
            __syncwarp();
            queue_add<T, DPD, TS>(Q, max(from, r0) - r0, min(to, r0 + nr) - r0, sub, fx, fy, fz);
        }
        __syncwarp();
        cnt = 0;
    };

#pragma unroll 1
    for (int dzc = -W; dzc <= W; ++dzc) {
        int az = cz + dzc, czc = 0;
        if (az < 0) { az += nc2; czc = 2; }
        else if (az >= nc2) { az -= nc2; czc = 1; }
        const float zo = (czc & 1) ? (float)(xi.z - g.L[2]) : z, zL = (czc & 2) ? L2 : 0.f;
        const bool sheared = LE && czc != 0;
        float xL = 0.f;
        int cxr = cx;
        if (sheared) {
            // the partners' image is displaced by nz delta along x: its cells
            // are found around x_i - nz delta
            const T nd = czc == 1 ? le_d : -le_d;
            xL = (float)nd;
            T xs = xi.x - nd;
            if (xs < T(0)) xs += g.L[0];
            if (xs >= g.L[0]) xs -= g.L[0];
            cxr = cell_coord(xs, g.cells_per_len[0], nc0);
        }
        const int lo = cxr - W, hi = cxr + W;
#pragma unroll 1
        for (int dyc = -W; dyc <= W; ++dyc) {
            int ay = cy + dyc, cyc = 0;
            if (ay < 0) { ay += nc1; cyc = 2; }
            else if (ay >= nc1) { ay -= nc1; cyc = 1; }
            const float yo = (cyc & 1) ? (float)(xi.y - g.L[1]) : y, yL = (cyc & 2) ? L1 : 0.f;
            const int base = g.cell_off + (az * nc1 + ay) * nc0;
            // the row's cyclic x range: two pieces where it wraps
            const bool wraps = lo < 0 || hi >= nc0;
#pragma unroll 1
            for (int part = 0; part < 2; ++part) {
                int p = 0, e = 0, cxc = 0;
                if (live && (part == 0 || wraps)) {
                    const int a0 = part == 1 ? 0 : lo < 0 ? lo + nc0 : lo;
                    const int a1 = part == 1 ? (lo < 0 ? hi : hi - nc0) : wraps ? nc0 - 1 : hi;
                    p = __ldg(B + base + a0);
                    e = __ldg(B + base + a1 + 1);
                    cxc = part == 0 ? (lo < 0 ? 2 : 0) : (hi >= nc0 ? 1 : 0);
                }
                const float xo = (!sheared && (cxc & 1)) ? (float)(xi.x - g.L[0]) : x;
                const float xS = sheared ? xL : (cxc & 2) ? L0 : 0.f;
                const int tag = ((sheared ? 3 : cxc) | (cyc << 2) | (czc << 4)) << NBR_INDEX_BITS;
                const int longest = __reduce_max_sync(0xffffffffu, e - p);
                if (part == 1 && longest <= 0) break;
                for (int k0 = 0; k0 < longest; k0 += STEP) {
                    float4 xj[U];
#pragma unroll
                    for (int k = 0; k < U; ++k) {
                        const int q = p + k0 + k * TS + sub;
                        xj[k] = __ldg(EF + (q < e ? q : idx));
                    }
#pragma unroll
                    for (int k = 0; k < U; ++k) {
                        const int q = p + k0 + k * TS + sub;
                        float dx;
                        if (LE && sheared) {
                            dx = (xo - xj[k].x) - xS;
                            dx -= L0 * rintf(dx * linv);
                        } else {
                            dx = xo - (xj[k].x - xS);
                        }
                        const float dy = yo - (xj[k].y - yL);
                        const float dz = zo - (xj[k].z - zL);
                        bool in = dx * dx + dy * dy + dz * dz < rc2 && q < e && q != idx;
                        if (excl) {
                            const int j = __float_as_int(xj[k].w);
                            in = in && j != ex.x && j != ex.y;
                        }
                        if constexpr (TS == 1) {
                            if (in) {
                                col[cnt * PPW] = q | tag;
                                ++cnt;
                            }
                        } else {
                            const unsigned int m = __ballot_sync(0xffffffffu, in) & tmask;
                            if (in) col[(cnt + __popc(m & ((1u << lane) - 1u))) * PPW] = q | tag;
                            cnt += __popc(m);
                        }
                    }
                    // the next step's hits must fit every column
                    if (__any_sync(0xffffffffu, cnt > CFC - STEP)) evaluate();
                }
            }
        }
    }
    evaluate();
    if constexpr (TS > 1) {
        const T f = fx;
        fx = __shfl_sync(0xffffffffu, f, pw * TS);
        fy = __shfl_sync(0xffffffffu, f, pw * TS + 1);
        fz = __shfl_sync(0xffffffffu, f, pw * TS + 2);
    }
    if (ENERGY) {
        // a lane holds the sums of the pairs it evaluated, whosever they are:
        // a particle takes its lanes' sums, and those of the places of the warp
        // that hold no particle
#pragma unroll
        for (int o = TS / 2; o > 0; o >>= 1) {
            pe += __shfl_xor_sync(0xffffffffu, pe, o);
            vir += __shfl_xor_sync(0xffffffffu, vir, o);
            vxz += __shfl_xor_sync(0xffffffffu, vxz, o);
        }
        const int nlive = min(PPW, tl.count - first);
        for (int o = nlive; o < PPW; o += nlive) {
            const int from = pw + o < PPW ? (pw + o) * TS : 0;
            const T a = __shfl_sync(0xffffffffu, pe, from), b = __shfl_sync(0xffffffffu, vir, from),
                    d = __shfl_sync(0xffffffffu, vxz, from);
            if (live && pw + o < PPW) {
                pe += a;
                vir += b;
                vxz += d;
            }
        }
    }
    if (live && sub == 0) {
        s.cpf[i] = mk4<T>(fx, fy, fz, pe);
        if (ENERGY) s.cpv[i] = mk4<T>(vir, vxz, T(0), T(0));
    }
}

template <class T>
int Launch<T>::cellforce(const DevSys<T>& s, int cur, bool energy, bool dpd, cudaStream_t st) {
    const int gt = s.ntiles;
    const bool multi = s.ntypes > 1;
    const bool spread = s.N < 40960;  // see CFT
#define ESPP_CF(W, E, M, D, L)                                                                          \
    do {                                                                                               \
        if (spread) k_cellforce<T, W, E, M, D, L, CFT><<<gt * CFT, TILE, 0, st>>>(s, cur);             \
        else k_cellforce<T, W, E, M, D, L, 1><<<gt, TILE, 0, st>>>(s, cur);                            \
    } while (0)
#define ESPP_CF_L(W, E, M, D)                    \
    do {                                         \
        if (s.le_on) ESPP_CF(W, E, M, D, true);  \
        else ESPP_CF(W, E, M, D, false);         \
    } while (0)
#define ESPP_CF_D(W, E, M)                       \
    do {                                         \
        if (dpd) ESPP_CF_L(W, E, M, true);       \
        else ESPP_CF_L(W, E, M, false);          \
    } while (0)
#define ESPP_CF_M(W, E)                          \
    do {                                         \
        if (multi) ESPP_CF_D(W, E, true);        \
        else ESPP_CF_D(W, E, false);             \
    } while (0)
    if (s.cell_w == 1) {
        if (energy) ESPP_CF_M(1, true);
        else ESPP_CF_M(1, false);
    } else {
        if (energy) ESPP_CF_M(2, true);
        else ESPP_CF_M(2, false);
    }
#undef ESPP_CF_M
#undef ESPP_CF_D
#undef ESPP_CF_L
#undef ESPP_CF
    return 1;
}

template int Launch<float>::cellforce(const DevSys<float>&, int, bool, bool, cudaStream_t);
template int Launch<double>::cellforce(const DevSys<double>&, int, bool, bool, cudaStream_t);

}  // namespace espp
