// The per-step kernel: pair forces over the Verlet list (Lennard-Jones / WCA /
// capped LJ, paper "Software design": VerletListInteractionTemplate<Potential>
// with computeForce/computeEnergy; "Example usage": LennardJones(..., shift=
// 'auto'), LennardJonesCapped), FENE bonds, the Langevin thermostat
// ("Example usage": LangevinThermostat(gamma, temperature) attached through
// addExtension) and velocity Verlet ("Example usage": VelocityVerlet), fused
// into one pass per particle.
//
// One thread per particle, particles in cell (Hilbert) order, 128 per block.
// Each thread sums the forces on its own particle from both directions of the
// full list, so no force atomics are needed.  In MODE_STEP the thread then
// completes the step and starts the next one:
//   F_s  = F_pair + F_bond - gamma m v_{s-1/2} + sqrt(24 gamma m kT/dt) r_s
//   v_s  = v_{s-1/2} + dt/2 F_s/m           (the full-step velocity)
//   v_{s+1/2} = v_s + dt/2 F_s/m
//   x_{s+1}   = x_s + dt v_{s+1/2}           (wrapped; written to the other buffer)
// and checks the displacement since the last list build against skin/2.
#include "kernels.cuh"
#include "pair_walk.cuh"

// Launch shapes of the FP32 step kernel on the plain list path, chosen at run
// time by the autotuner (espp_tune_step_shape): int4 neighbour groups read per
// batch, the minimum resident blocks per SM the register budget is fitted to,
// and the tiles one block takes.  A block of several consecutive tiles holds
// a larger compact piece of the Hilbert order, so more of its neighbours'
// positions are shared in the SM's L1 (the halo of a piece shrinks relative
// to its volume).  Shape 0 is the default.
struct StepShape {
    int groups;  // list groups per batch
    int minb;    // minimum resident blocks per SM
    int tpb;     // tiles (of TILE particles) per block
};
constexpr StepShape STEP_SHAPES[ESPP_STEP_SHAPES] = {{1, 8, 1}, {2, 8, 1}, {1, 12, 1}, {1, 10, 1},
                                                     {1, 5, 2}, {1, 3, 3}, {1, 2, 4},  {1, 2, 5}};
#ifndef ESPP_STEP_MINB32
#define ESPP_STEP_MINB32 8  // KG 1M FP32: 0.1027 ms per step (8), 0.1123 (10)
#endif
#ifndef ESPP_STEP_MINB32_DPD  // the same for the DPD variants
#define ESPP_STEP_MINB32_DPD 7
#endif
#ifndef ESPP_STEP_LATE  // loads issued after the pair loop: 1 bond partners, 2 velocity and build position
#define ESPP_STEP_LATE 3  // KG 1M FP32 at 8 blocks per SM: 58.7 us (3), 61.5 (1); fewer values live across the loop
#endif

namespace espp {

// DPD thermostat forces on particle i as a pass of their own over the list,
// for the learned potential, whose pair forces come from k_mlp.
template <class T, bool LE>
__device__ __forceinline__ void dpd_loop(const DevSys<T>& s, const V4<T>* __restrict__ P, int i, int n,
                                         const V4<T>& xi, const DpdCtx<T>& c, const LeCtx<T>& le, T L0, T L1,
                                         T L2, T& fx, T& fy, T& fz) {
    const IntParams<T>* __restrict__ ip = s.ip;
    const T rc2 = ip->dpd_rc2;
    const T xim = xi.x - L0, yim = xi.y - L1, zim = xi.z - L2;
    const int4* __restrict__ nb = reinterpret_cast<const int4*>(s.nbr) + i;
    const V4<T>* __restrict__ VS = s.vsnap;
    const size_t stride = (size_t)s.stride;
    for (int g = 0; 4 * g < n; ++g) {
        const int4 a = __ldg(nb + g * stride);
        const int jj[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (4 * g + q >= n) continue;
            const int j = nbr_slot(jj[q]), code = nbr_code(jj[q]);
            const V4<T> xj = ld4<T>(P + j);
            int nz = 0;
            T dx;
            if (LE && (code & 3) == 3) {
                nz = (code >> 4) == 1 ? 1 : -1;
                dx = le_dx(xi.x, xj.x, nz, le.d, L0, le.inv_Lx);
            } else {
                dx = shifted_diff(xi.x, xim, xj.x, L0, code & 3);
            }
            const T dy = shifted_diff(xi.y, yim, xj.y, L1, (code >> 2) & 3);
            const T dz = shifted_diff(xi.z, zim, xj.z, L2, code >> 4);
            const T r2 = dx * dx + dy * dy + dz * dz;
            if (!(r2 < rc2)) continue;
            dpd_term<T, LE>(ip, c, dx, dy, dz, r2, ld4<T>(VS + j), fx, fy, fz, nz);
        }
    }
}

// velocities at the force evaluation, read by the DPD pass for the neighbours
template <class T>
__global__ void __launch_bounds__(TILE) k_vsnap(DevSys<T> s) {
    if (s.ctrl->abort) return;
    for (int t = blockIdx.x; t < s.ntiles; t += gridDim.x) {
        const Tile tl = s.tiles[t];
        if ((int)threadIdx.x < tl.count) s.vsnap[tl.start + threadIdx.x] = s.vel[tl.start + threadIdx.x];
    }
}

// SH: launch shape (STEP_SHAPES) of the plain FP32 list path.  PPW: particles
// per warp of the queue path (32, or 8 with four lanes per particle).  WALK: FP32
// DPD walks the lists instead (see step_walks).
template <class T, int MODE, bool ENERGY, bool FAST, bool DPD, bool LE, int SH = 0, int PPW = 32, bool WALK = false>
__global__ void __launch_bounds__(TILE * STEP_SHAPES[SH].tpb,
                                  sizeof(T) == 4 ? (DPD ? ESPP_STEP_MINB32_DPD
                                                        : (SH == 0 ? ESPP_STEP_MINB32 : STEP_SHAPES[SH].minb))
                                                 : 4)
    k_step(DevSys<T> s, int cur, double* __restrict__ f_out, unsigned long long next_cond) {
    // TPB consecutive tiles per block; the block-wide energy reduction below
    // is written for one
    constexpr int TPB = STEP_SHAPES[SH].tpb;
    static_assert(TPB == 1 || !ENERGY, "energy reductions take one tile per block");
    static_assert(PPW == 32 || (TPB == 1 && !ENERGY), "four lanes per particle: single tiles, no reductions");
    constexpr bool QUEUE = (sizeof(T) == 8 || DPD) && !WALK;
    constexpr int TPP = 32 / PPW;  // lanes per particle, blocks per tile
    // index inside the tile
    const int lt = TPP > 1 ? (int)(blockIdx.x % TPP) * (TILE / TPP) + (int)threadIdx.x / TPP
                 : TPB > 1 ? (int)threadIdx.x % TILE : (int)threadIdx.x;
    Ctrl* c = s.ctrl;
    const int t0 = TPP > 1 ? blockIdx.x / TPP : blockIdx.x * TPB + (TPB > 1 ? (int)threadIdx.x / TILE : 0);
    // the first tile's record is requested together with the abort flag
    Tile tl0 = {0, 0, 0, 0};
    if (t0 < s.ntiles) tl0 = ld_tile_early(s.tiles + t0);
    if (MODE != MODE_FORCES && c->abort) return;
    const long long step = c->step + (MODE >= MODE_STEP ? 1 : 0);
    const V4<T>* __restrict__ P = s.pos[cur];
    V4<T>* __restrict__ Pn = s.pos[cur ^ 1];
    const IntParams<T>* __restrict__ ip = s.ip;
    static_assert(8 * NPART % 32 == 0 && 8 * NPART <= TILE, "whole warps reduce");
    // the warps' queues; after the forces the energy sums
    constexpr size_t QUEUE_BYTES = QUEUE ? sizeof(PairQueue<T, DPD, PPW>) * (TILE / 32) : 16;
    constexpr size_t RED_BYTES = ENERGY ? NPART * (TILE + 4) * sizeof(double) : 16;
    constexpr size_t SMEM_BYTES = QUEUE_BYTES > RED_BYTES ? QUEUE_BYTES : RED_BYTES;
    static_assert(SMEM_BYTES <= 48 * 1024, "static shared memory");
    __shared__ __align__(16) unsigned char smem[SMEM_BYTES];
    double (*red)[TILE + 4] = reinterpret_cast<double (*)[TILE + 4]>(smem);

    for (int t = t0; t < s.ntiles; t += TPP > 1 ? s.ntiles : gridDim.x * TPB) {
        const Tile tl = t == t0 ? tl0 : s.tiles[t];
        const bool active = lt < tl.count;
        const RepGeom<T>& g = s.reps[tl.rep];
        double acc[NPART];
        if (ENERGY) {
#pragma unroll
            for (int k = 0; k < NPART; ++k) acc[k] = 0.0;
        }
        // Lees-Edwards: the tile's offset now and, after the drift, the
        // displacement bound that keeps the list valid: pairs across a sheared
        // face also move apart by the change of delta since the build
        LeCtx<T> le;
        T skin_thr2 = s.half_skin2;
        if (LE) {
            double q[2] = {0.0, 0.0};
            if ((threadIdx.x & 31) == 0) {
                const double dnow = le_offset(s, g, step);
                q[0] = le_reduce(dnow, (double)g.L[0]);
                if (MODE == MODE_STEP) {
                    const double h = 0.5 * ((double)s.skin - fabs(le_offset(s, g, step + 1) - s.le_db[tl.rep]));
                    q[1] = h > 0.0 ? h * h : 0.0;
                }
            }
            q[0] = __shfl_sync(0xffffffffu, q[0], 0);
            q[1] = __shfl_sync(0xffffffffu, q[1], 0);
            le.d = (T)q[0];
            le.inv_Lx = T(1) / g.L[0];
            le.shear = (T)s.le_shear;
            le.vs = (T)(s.le_shear * (double)g.L[2]);
            if (MODE == MODE_STEP) skin_thr2 = (T)q[1];
        } else {
            le.d = le.inv_Lx = le.vs = le.shear = T(0);
        }
        // a warp's queue takes all of its lanes: those without a particle
        // stand at the tile's first one with an empty list
        const int i = tl.start + (active ? lt : 0);
        const T L0 = g.L[0], L1 = g.L[1], L2 = g.L[2];
        T fx = 0, fy = 0, fz = 0, pe = 0, pb = 0, vir = 0, vxz = 0;
        double blen = 0.0, bcnt = 0.0;
        if constexpr (QUEUE) {
            if (!s.mlp_on && (FAST || !s.cells_mode)) {
                const V4<T> xi = ld4<T>(P + i);
                const int n = active ? s.nbr_cnt[i] : 0;
                PairQueue<T, DPD, PPW>& q = reinterpret_cast<PairQueue<T, DPD, PPW>*>(smem)[threadIdx.x >> 5];
                const int ibase = tl.start + lt / PPW * PPW;
                T rcmax2 = s.rc_max2;
                if (DPD) rcmax2 = max(rcmax2, s.ip->dpd_rc2);
                if (FAST || s.ntypes == 1) {
                    const PairRec<T> pr = s.pair[0];
                    queue_loop<T, ENERGY, false, FAST, DPD, LE, PPW>(s, P, q, ibase, i, n, g, xi, &pr, rcmax2, le, step,
                                                                    fx, fy, fz, pe, vir, vxz);
                } else {
                    queue_loop<T, ENERGY, true, false, DPD, LE, PPW>(s, P, q, ibase, i, n, g, xi, nullptr, rcmax2, le,
                                                                    step, fx, fy, fz, pe, vir, vxz);
                }
            }
        }
        if (active && (TPP == 1 || threadIdx.x % TPP == 0)) {
            const T H2 = g.halfL[2];
            // independent loads first: own position, list count, bond slots,
            // velocity and build position, then the bond partners' positions
            const V4<T> xi = ld4<T>(P + i);
            const int ti = bits_as_int(xi.w);
            const int n = s.nbr_cnt[i];
            const bool bonded = s.bond.kind != 0;
            const int2 b = bonded ? s.bond_slot[i] : make_int2(-1, -1);
            // loads the pair loop does not need, issued before it (latency
            // hidden behind the loop) or after it (fewer registers held)
            constexpr bool LATE_BOND = (ESPP_STEP_LATE & 1) != 0;
            constexpr bool LATE_VEL = (ESPP_STEP_LATE & 2) != 0;
            V4<T> v, xbi, xp0, xp1;
            if (!LATE_VEL) {
                v = s.vel[i];
                if (MODE == MODE_STEP && (FAST || !s.cells_mode)) xbi = s.xb[i];
            }
            if (!LATE_BOND) {
                xp0 = b.x >= 0 ? ld4<T>(P + b.x) : xi;
                xp1 = b.y >= 0 ? ld4<T>(P + b.y) : xi;
            }
            if (s.mlp_on) {
                // pair forces of the learned potential, computed by k_mlp
                if constexpr (sizeof(T) == 8) {
                    // FP64 handle: the network evaluated in double (k_mlp_f64)
                    const V4<T> fm = s.mlp_fT[i];
                    fx = fm.x;
                    fy = fm.y;
                    fz = fm.z;
                    if (ENERGY) {
                        pe = fm.w;
                        vir = s.mlp_wT[i];
                    }
                } else {
                    const float4 fm = s.mlp_f[i];
                    fx = (T)fm.x;
                    fy = (T)fm.y;
                    fz = (T)fm.z;
                    if (ENERGY) {
                        pe = (T)fm.w;
                        vir = (T)s.mlp_w[i];
                    }
                }
                if (DPD) {
                    DpdCtx<T> dc;
                    dc.vi = s.vel[i];
                    dc.seed = g.seed;
                    dc.step = step;
                    dc.le_vs = le.vs;
                    dpd_loop<T, LE>(s, P, i, n, xi, dc, le, L0, L1, L2, fx, fy, fz);
                }
            } else if (!FAST && s.cells_mode) {
                // list-free mode: pair forces (with the DPD pair term) from
                // the cell-stencil kernel
                const V4<T> f = s.cpf[i];
                fx = f.x;
                fy = f.y;
                fz = f.z;
                if (ENERGY) {
                    pe = f.w;
                    const V4<T> w = s.cpv[i];
                    vir = w.x;
                    vxz = w.y;
                }
            } else if constexpr (!QUEUE) {
                DpdCtx<T> dc;
                if constexpr (DPD) {
                    dc.vi = s.vel[i];
                    dc.seed = g.seed;
                    dc.step = step;
                    dc.le_vs = le.vs;
                }
                if (FAST) {
                    PairRec<T> pr;
                    pr.rc2 = s.pair[0].rc2;
                    pr.sig2 = s.pair[0].sig2;
                    pr.eps24 = s.pair[0].eps24;
                    if (ENERGY) {
                        pr.eps4 = s.pair[0].eps4;
                        pr.shift = s.pair[0].shift;
                    }
                    pair_loop<T, ENERGY, false, true, LE, STEP_SHAPES[SH].groups, false, DPD>(
                        s, P, i, n, xi, ti, &pr, L0, L1, L2, fx, fy, fz, pe, vir, vxz, &le, &dc);
                } else if (s.ntypes == 1) {
                    const PairRec<T> pr = s.pair[0];
                    if (DPD || pr.kind != 0)
                        pair_loop<T, ENERGY, false, false, LE, 1, false, DPD>(s, P, i, n, xi, ti, &pr, L0, L1, L2, fx, fy,
                                                                              fz, pe, vir, vxz, &le, &dc);
                } else {
                    pair_loop<T, ENERGY, true, false, LE, 1, false, DPD>(s, P, i, n, xi, ti, nullptr, L0, L1, L2, fx, fy,
                                                                         fz, pe, vir, vxz, &le, &dc);
                }
            }
            if (LATE_VEL) {
                v = s.vel[i];
                if (MODE == MODE_STEP && (FAST || !s.cells_mode)) xbi = s.xb[i];
            }
            if (LATE_BOND) {
                xp0 = b.x >= 0 ? ld4<T>(P + b.x) : xi;
                xp1 = b.y >= 0 ? ld4<T>(P + b.y) : xi;
            }
            if (bonded && bond_forces<T, ENERGY, LE>(s, g, xi, b, xp0, xp1, le, fx, fy, fz, pb, vir, vxz, blen, bcnt)) {
                atomicOr(&c->err, ERRBIT_BOND);
                c->abort = 1;
                __threadfence();
            }
            if (MODE == MODE_FORCES) {
                if (f_out) {
                    const size_t gid = (size_t)g.p_off + bits_as_int(v.w);
                    f_out[3 * gid + 0] = (double)fx;
                    f_out[3 * gid + 1] = (double)fy;
                    f_out[3 * gid + 2] = (double)fz;
                }
                if (ENERGY) {
                    const double m = (double)ip->mass[ti];
                    // kinetic terms relative to the shear profile (Lees-Edwards)
                    const double vxp = LE ? (double)v.x - (double)le.shear * ((double)xi.z - (double)H2) : (double)v.x;
                    acc[P_KE] = 0.5 * m * (vxp * vxp + (double)v.y * v.y + (double)v.z * v.z);
                    acc[P_KIN_XZ] = m * vxp * (double)v.z;
                    acc[P_PX] = m * v.x;
                    acc[P_PY] = m * v.y;
                    acc[P_PZ] = m * v.z;
                }
            } else {
                const T inv_m = ip->inv_mass[ti];
                if (!DPD) langevin_forces<T, LE>(ip, g, ti, xi, v, step, le, fx, fy, fz);
                if (MODE == MODE_INIT) {
                    s.frc[i] = mk4<T>(fx, fy, fz, T(0));
                } else {
                    const T hdt = ip->half_dt;
                    v.x = half_kick(v.x, fx, hdt, inv_m);
                    v.y = half_kick(v.y, fy, hdt, inv_m);
                    v.z = half_kick(v.z, fz, hdt, inv_m);
                    if (MODE == MODE_FINAL) {
                        s.vel[i] = v;
                        s.frc[i] = mk4<T>(fx, fy, fz, T(0));
                    } else {
                        v.x = half_kick(v.x, fx, hdt, inv_m);
                        v.y = half_kick(v.y, fy, hdt, inv_m);
                        v.z = half_kick(v.z, fz, hdt, inv_m);
                        const T dt = ip->dt;
                        T x = drift(xi.x, v.x, dt), y = drift(xi.y, v.y, dt), z = drift(xi.z, v.z, dt);
                        // no wrap here: positions stay in the image frame of the
                        // last list build until the next build wraps them
                        if (!(abs_less(x, T(1e30)) && abs_less(y, T(1e30)) && abs_less(z, T(1e30)))) {
                            atomicOr(&c->err, ERRBIT_NONFINITE);
                            c->abort = 1;
                            __threadfence();
                            x = xi.x; y = xi.y; z = xi.z;
                        }
                        if (!FAST && s.cells_mode) {
                            // list-free mode: every step is binned again
                            if (lt == 0) {
                                s.req[tl.rep] = 1;
                                c->any_req = 1;
                                __threadfence();
                            }
                        } else {
                            const T ex = x - xbi.x, ey = y - xbi.y, ez = z - xbi.z;
                            if (less_nonneg(skin_thr2, ex * ex + ey * ey + ez * ez)) {
                                s.req[tl.rep] = 1;
                                c->any_req = 1;
                                __threadfence();
                            }
                        }
                        Pn[i] = mk4<T>(x, y, z, xi.w);
                        s.vel[i] = v;
                    }
                }
            }
        }
        if (ENERGY) {
            // the queue's lanes hold the pairs they evaluated, whosever they are
            acc[P_PE_PAIR] = 0.5 * (double)pe;
            acc[P_PE_BOND] = 0.5 * (double)pb;
            acc[P_VIRIAL] = 0.5 * (double)vir;
            acc[P_BOND_LEN] = 0.5 * blen;
            acc[P_BOND_CNT] = 0.5 * bcnt;
            acc[P_VIR_XZ] = 0.5 * (double)vxz;
            if (QUEUE) __syncthreads();  // every warp is done with its queue
            // eight threads per quantity add 16 particles each, then each other's
            // sums: a fifth of the FP64 additions of a tree over every warp
#pragma unroll
            for (int k = 0; k < NPART; ++k) red[k][threadIdx.x] = acc[k];
            __syncthreads();
            if (threadIdx.x < 8 * NPART) {
                const int k = threadIdx.x >> 3, q = threadIdx.x & 7;
                double sum = 0.0;
                for (int j = 0; j < TILE / 8; ++j) sum += red[k][8 * j + q];
#pragma unroll
                for (int o = 4; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
                if (q == 0) s.partials[(size_t)t * NPART + k] = sum;
            }
            __syncthreads();
        }
    }

    if (MODE == MODE_STEP || MODE == MODE_FINAL) {
        // the last block to finish advances the step counter and arms the
        // conditional rebuild node of the next step
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            const unsigned int done = atomicAdd(&c->blocks_done, 1u);
            if (done == gridDim.x - 1) {
                __threadfence();
                c->step = step;
                if (MODE == MODE_FINAL) c->pos_ahead = 0;
                c->blocks_done = 0;
                if (next_cond) {
                    const unsigned int want = *(volatile unsigned int*)&c->any_req;
                    const unsigned int ab = *(volatile unsigned int*)&c->abort;
                    cudaGraphSetConditional(next_cond, (want && !ab) ? 1u : 0u);
                }
            }
        }
    }
}

// First half-kick and drift of an integrate call: v_{n+1/2}, x_{n+1}.
template <class T>
__global__ void __launch_bounds__(TILE) k_prologue(DevSys<T> s, int cur) {
    Ctrl* c = s.ctrl;
    if (c->abort) return;
    const V4<T>* __restrict__ P = s.pos[cur];
    V4<T>* __restrict__ Pn = s.pos[cur ^ 1];
    const IntParams<T>* __restrict__ ip = s.ip;
    // the stored positions become those of step + 1 (read by the rebuilds)
    if (blockIdx.x == 0 && threadIdx.x == 0) c->pos_ahead = 1;
    const long long step = c->step;
    for (int t = blockIdx.x; t < s.ntiles; t += gridDim.x) {
        const Tile tl = s.tiles[t];
        if ((int)threadIdx.x >= tl.count) continue;
        const int i = tl.start + threadIdx.x;
        T skin_thr2 = s.half_skin2;
        if (s.le_on) {
            // Lees-Edwards: the change of delta since the build uses up skin
            const double h = 0.5 * ((double)s.skin - fabs(le_offset(s, s.reps[tl.rep], step + 1) - s.le_db[tl.rep]));
            skin_thr2 = h > 0.0 ? (T)(h * h) : T(0);
        }
        const V4<T> xi = P[i];
        const int ti = bits_as_int(xi.w);
        const V4<T> f = s.frc[i];
        V4<T> v = s.vel[i];
        const T hdt = ip->half_dt, inv_m = ip->inv_mass[ti];
        v.x = half_kick(v.x, f.x, hdt, inv_m);
        v.y = half_kick(v.y, f.y, hdt, inv_m);
        v.z = half_kick(v.z, f.z, hdt, inv_m);
        const T dt = ip->dt;
        T x = drift(xi.x, v.x, dt), y = drift(xi.y, v.y, dt), z = drift(xi.z, v.z, dt);
        if (!(abs_less(x, T(1e30)) && abs_less(y, T(1e30)) && abs_less(z, T(1e30)))) {
            atomicOr(&c->err, ERRBIT_NONFINITE);
            c->abort = 1;
            x = xi.x; y = xi.y; z = xi.z;
        }
        if (s.cells_mode) {
            // list-free mode: every step is binned again
            s.req[tl.rep] = 1;
            c->any_req = 1;
        } else {
            const V4<T> b = s.xb[i];
            const T ex = x - b.x, ey = y - b.y, ez = z - b.z;
            if (less_nonneg(skin_thr2, ex * ex + ey * ey + ez * ez)) {
                s.req[tl.rep] = 1;
                c->any_req = 1;
            }
        }
        Pn[i] = mk4<T>(x, y, z, xi.w);
        s.vel[i] = v;
    }
}

template <class T>
__global__ void k_set_cond(DevSys<T> s, unsigned long long h) {
    const unsigned int want = *(volatile unsigned int*)&s.ctrl->any_req;
    const unsigned int ab = *(volatile unsigned int*)&s.ctrl->abort;
    cudaGraphSetConditional(h, (want && !ab) ? 1u : 0u);
}

// Four lanes per particle on the queue path while one lane per particle leaves
// SMs idle, and on long lists, whose eight-particle queues are full anyway.
// Step kernel (event-timed), one lane / four: KG melt FP64 1,000 25.4 / 16.6 us,
// 5,000 27.8 / 20.9, 10,000 28.8 / 27.0, 20,000 29.6 / 40, 40,000 39 / 58; LJ
// fluid FP64 (76 entries) 27,436 194 / 137, 256,000 1186 / 822; DPD fluid FP32
// 24,000 47 / 27, 98,304 56 / 62.
template <class T>
static bool queue_spread(const DevSys<T>& s) {
    if (sizeof(T) == 8) return s.N < 12288 || s.cap >= 64;
    return s.N < 49152;
}

// FP32 handles with the DPD thermostat and one lane per particle walk their lists
// (pair_loop, the thermostat's term where it is met) instead of taking the queue
// where the queue has little to save: few entries inside the thermostat's cutoff
// (its term then runs rarely, and every other entry would pass through shared memory
// for a Lennard-Jones term), or most entries inside some cutoff.  The fractions are
// those of a uniform density outside the potentials' cores (0.9 sigma).  Step kernel
// (event-timed), queue / walk, thermostat inside x, any cutoff inside y of the list:
//   LJ 2.5, skin 0.3, DPD 1.0 (0.01, 0.70): 55,000 54.5 / 33.5 us, 256,000 172 / 74, 780,000
//     469 / 180; two types 256,000 184 / 115; under shear 187 / 93
//   LJ 2.5, skin 1.0, DPD 1.0 (0.01, 0.35): 256,000 214 / 126
//   LJ 2.5, skin 0.3, DPD 1.5 (0.12, 0.70): 55,000 72.7 / 67.9, 256,000 218 / 167
//   the same, DPD 2.5 (0.70, 0.70): 55,000 75.7 / 81.6, 256,000 226 / 206
//   table 1.5, skin 0.05, DPD 1.5 (0.90, 0.90): 256,000 69 / 64
//   table 1.5, skin 0.4, DPD 1.0 (0.15, 0.49): 256,000 73 / 75
//   LJ 2.5, skin 1.0, DPD 2.0 (0.17, 0.35): 256,000 267 / 313
//   WCA, skin 0.4, DPD 1.1 (0.21, 0.25): 256,000 35.5 / 46.9
//   table 1.0, skin 0.6, DPD 1.0 (0.24, 0.24): 256,000 95 / 163
template <class T>
static bool step_walks(const DevSys<T>& s) {
    if (sizeof(T) == 8) return false;
    const double core = s.pair_core3, list = pow((double)s.rlist2, 1.5) - core;
    const double dpd = pow((double)s.dpd_rc2, 1.5) - core;
    const double any = pow((double)(s.dpd_rc2 > s.rc_max2 ? s.dpd_rc2 : s.rc_max2), 1.5) - core;
    return dpd < 0.1 * list || (any > 0.65 * list && s.N >= 131072);
}

template <class T>
int Launch<T>::step(const DevSys<T>& s, int mode, bool energy, int cur, double* f_out,
                    unsigned long long next_cond, int grid, cudaStream_t st) {
    const int gr = grid > 0 ? grid : s.ntiles;
    int extra = s.mlp_on ? Launch<T>::mlp(s, cur, energy, st) : 0;
    const bool dpd = s.dpd && mode != MODE_FORCES;
    if (s.cells_mode) {
        // list-free: pair forces (and the DPD pair term) from the cell stencil
        extra += Launch<T>::cellforce(s, cur, energy, dpd, st);
    } else if (dpd) {
        k_vsnap<T><<<s.ntiles, TILE, 0, st>>>(s);
        extra += 1;
    }
    // the plain FP32 list path of a step takes the tuned launch shape
    const int sh = (sizeof(T) == 4 && s.lj_fast && !s.le_on && !s.cells_mode && !s.mlp_on &&
                    (mode == MODE_STEP || mode == MODE_FINAL) && !dpd) ? s.step_shape : 0;
    // queue path of a small handle: four lanes per particle (see the rule above)
    const bool spread = (sizeof(T) == 8 || dpd) && !s.mlp_on && !s.cells_mode && queue_spread(s);
    const bool walk = dpd && !spread && !s.mlp_on && !s.cells_mode && step_walks(s);
#define ESPP_STEP_Q(M, E, F, D, LE)                                                                        \
    do {                                                                                                   \
        if constexpr ((sizeof(T) == 8 || (D)) && !(E)) {                                                   \
            if (spread) {                                                                                  \
                k_step<T, M, E, F, D, LE, 0, 8><<<4 * s.ntiles, TILE, 0, st>>>(s, cur, f_out, next_cond);  \
                break;                                                                                     \
            }                                                                                              \
        }                                                                                                  \
        if constexpr (sizeof(T) == 4 && (D)) {                                                             \
            if (walk) {                                                                                    \
                k_step<T, M, E, F, D, LE, 0, 32, true><<<gr, TILE, 0, st>>>(s, cur, f_out, next_cond);     \
                break;                                                                                     \
            }                                                                                              \
        }                                                                                                  \
        k_step<T, M, E, F, D, LE><<<gr, TILE, 0, st>>>(s, cur, f_out, next_cond);                          \
    } while (0)
#define ESPP_STEP_SHAPED(M, E, D, LE, K)                                                                   \
    k_step<T, M, E, true, D, LE, K>                                                                        \
        <<<(gr + STEP_SHAPES[K].tpb - 1) / STEP_SHAPES[K].tpb, TILE * STEP_SHAPES[K].tpb, 0, st>>>(s, cur, f_out, next_cond)
#define ESPP_STEP_SH(M, E, D, LE)                                                                          \
    do {                                                                                                   \
        if constexpr (sizeof(T) == 4 && !(D) && !(LE) && ((M) == MODE_STEP || (M) == MODE_FINAL)) {        \
            switch (sh) {                                                                                  \
                case 1: ESPP_STEP_SHAPED(M, E, D, LE, 1); break;                                           \
                case 2: ESPP_STEP_SHAPED(M, E, D, LE, 2); break;                                           \
                case 3: ESPP_STEP_SHAPED(M, E, D, LE, 3); break;                                           \
                case 4: ESPP_STEP_SHAPED(M, E, D, LE, 4); break;                                           \
                case 5: ESPP_STEP_SHAPED(M, E, D, LE, 5); break;                                           \
                case 6: ESPP_STEP_SHAPED(M, E, D, LE, 6); break;                                           \
                case 7: ESPP_STEP_SHAPED(M, E, D, LE, 7); break;                                           \
                default: break;                                                                            \
            }                                                                                              \
            if (sh != 0) break;                                                                            \
        }                                                                                                  \
        ESPP_STEP_Q(M, E, true, D, LE);                                                                    \
    } while (0)
#define ESPP_STEP_LE(M, E, D, LE)                                                                \
    do {                                                                                         \
        if (s.lj_fast) ESPP_STEP_SH(M, E, D, LE);                                                \
        else ESPP_STEP_Q(M, E, false, D, LE);                                                    \
    } while (0)
#define ESPP_STEP(M, E, D)                            \
    do {                                              \
        if (s.le_on) ESPP_STEP_LE(M, E, D, true);     \
        else ESPP_STEP_LE(M, E, D, false);            \
    } while (0)
    switch (mode) {
        case MODE_FORCES:
            if (energy) ESPP_STEP(MODE_FORCES, true, false); else ESPP_STEP(MODE_FORCES, false, false);
            break;
        case MODE_INIT:
            if (dpd) ESPP_STEP(MODE_INIT, false, true); else ESPP_STEP(MODE_INIT, false, false);
            break;
        case MODE_STEP:
            if (dpd) ESPP_STEP(MODE_STEP, false, true); else ESPP_STEP(MODE_STEP, false, false);
            break;
        default:
            if (dpd) ESPP_STEP(MODE_FINAL, false, true); else ESPP_STEP(MODE_FINAL, false, false);
            break;
    }
#undef ESPP_STEP
#undef ESPP_STEP_Q
#undef ESPP_STEP_LE
#undef ESPP_STEP_SH
#undef ESPP_STEP_SHAPED
    return 1 + extra;
}

template <class T>
void Launch<T>::prologue(const DevSys<T>& s, int cur, int grid, cudaStream_t st) {
    k_prologue<T><<<grid > 0 ? grid : s.ntiles, TILE, 0, st>>>(s, cur);
}

template <class T>
void Launch<T>::set_cond(const DevSys<T>& s, unsigned long long cond, cudaStream_t st) {
    k_set_cond<T><<<1, 1, 0, st>>>(s, cond);
}

// The two precisions compile as separate units (k_step_f32.cu, k_step_f64.cu)
// that include this file with ESPP_STEP_PRECISION set, so they build in
// parallel; compiled alone, this file instantiates both.
#if !defined(ESPP_STEP_PRECISION) || ESPP_STEP_PRECISION == 32
template int Launch<float>::step(const DevSys<float>&, int, bool, int, double*, unsigned long long, int, cudaStream_t);
template void Launch<float>::prologue(const DevSys<float>&, int, int, cudaStream_t);
template void Launch<float>::set_cond(const DevSys<float>&, unsigned long long, cudaStream_t);
#endif
#if !defined(ESPP_STEP_PRECISION) || ESPP_STEP_PRECISION == 64
template int Launch<double>::step(const DevSys<double>&, int, bool, int, double*, unsigned long long, int, cudaStream_t);
template void Launch<double>::prologue(const DevSys<double>&, int, int, cudaStream_t);
template void Launch<double>::set_cond(const DevSys<double>&, unsigned long long, cudaStream_t);
#endif

}  // namespace espp
