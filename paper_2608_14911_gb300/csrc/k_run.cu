// The resident run kernel: many steps of a small system in one launch.
//
// A step of a few thousand particles is a few microseconds of dependent loads; as
// a graph node behind a conditional rebuild node it costs three times that (KG
// melt of 5,000, FP32: 16.7 us a step without a rebuild).  Here every thread
// keeps its particle (position, velocity, build position, bonds) in registers,
// and the blocks, all resident (a cooperative launch), meet at a grid barrier
// after every step.  The kernel returns when a rebuild is requested, an error was
// found or the segment's last step is done; the graph around it loops: rebuild,
// run.  Positions go through the two buffers in memory with coherent loads, for
// other SMs rewrite them while the kernel runs.
//
// It serves the list path of one particle type with a Lennard-Jones / WCA
// potential, bonds and the Langevin thermostat, as long as one round of blocks
// holds every particle (see run_fits); the arithmetic is the step kernel's, so the
// trajectories are the same bits.
#include "grid_barrier.cuh"
#include "pair_walk.cuh"

namespace espp {

// PPW: particles per warp (FP64 handles: the pair queue; FP32: one lane each);
// GB: list groups per batch (FP32); MINB: resident blocks per SM.
template <class T, int PPW, int GB, int MINB>
__global__ void __launch_bounds__(TILE, MINB) k_run(DevSys<T> s, unsigned long long cond) {
    constexpr bool QUEUE = sizeof(T) == 8;
    constexpr int TPP = 32 / PPW;  // lanes per particle, blocks per tile
    extern __shared__ __align__(16) unsigned char queue_mem[];  // FP64: the warps' queues, up to 48 KB
    __shared__ long long stopped;
    Ctrl* c = s.ctrl;
    // what every block sees before any block can change it
    const long long step0 = *(volatile long long*)&c->step, target = c->target;
    const int fin = c->final_step;
    int buf = c->buf;
    const bool go = *(volatile unsigned int*)&c->abort == 0 && *(volatile unsigned int*)&c->any_req == 0 &&
                    step0 < target;
    unsigned int phase = 1;
    bool ok = grid_barrier(c, phase++, s.run_fault, [] {});
    long long step = step0;
    if (ok && go) {
        const int lt = TPP > 1 ? (int)(blockIdx.x % TPP) * (TILE / TPP) + (int)threadIdx.x / TPP : (int)threadIdx.x;
        const Tile tl = s.tiles[blockIdx.x / TPP];
        const bool active = lt < tl.count, lead = active && (TPP == 1 || threadIdx.x % TPP == 0);
        const RepGeom<T>& g = s.reps[tl.rep];
        const IntParams<T>* __restrict__ ip = s.ip;
        const int i = tl.start + (active ? lt : 0);
        const T L0 = g.L[0], L1 = g.L[1], L2 = g.L[2];
        const int n = active ? s.nbr_cnt[i] : 0;
        V4<T> xi = s.pos[buf][i], v = s.vel[i];
        const V4<T> xbi = s.xb[i];
        const int ti = bits_as_int(xi.w);
        const bool bonded = s.bond.kind != 0;
        const int2 b = bonded ? s.bond_slot[i] : make_int2(-1, -1);
        const PairRec<T> pr = s.pair[0];
        const T inv_m = ip->inv_mass[ti], hdt = ip->half_dt, dt = ip->dt;
        LeCtx<T> le;
        le.d = le.inv_Lx = le.vs = le.shear = T(0);
        for (;;) {
            ++step;
            const bool last = fin && step == target;
            const V4<T>* P = s.pos[buf];
            T fx = 0, fy = 0, fz = 0, pe = 0, pb = 0, vir = 0, vxz = 0;
            double blen = 0, bcnt = 0;
            const V4<T> xp0 = b.x >= 0 ? ldp<T, true>(P + b.x) : xi;
            const V4<T> xp1 = b.y >= 0 ? ldp<T, true>(P + b.y) : xi;
            if constexpr (QUEUE) {
                PairQueue<T, false, PPW>& q =
                    reinterpret_cast<PairQueue<T, false, PPW>*>(queue_mem)[threadIdx.x >> 5];
                queue_loop<T, false, false, true, false, false, PPW, true>(s, P, q, tl.start + lt / PPW * PPW, i, n, g, xi,
                                                                           &pr, s.rc_max2, le, step, fx, fy, fz, pe, vir,
                                                                           vxz);
            } else if (active) {
                // GB groups in flight: the gathers' latency is the step's time
                pair_loop<T, false, false, true, false, GB, true>(s, P, i, n, xi, ti, &pr, L0, L1, L2, fx, fy, fz, pe,
                                                                 vir, vxz, &le);
            }
            if (lead) {
                unsigned int bad = 0;
                bool request = false;
                if (bonded && bond_forces<T, false, false>(s, g, xi, b, xp0, xp1, le, fx, fy, fz, pb, vir, vxz, blen,
                                                           bcnt))
                    bad = ERRBIT_BOND;
                langevin_forces<T, false>(ip, g, ti, xi, v, step, le, fx, fy, fz);
                v.x = half_kick(v.x, fx, hdt, inv_m);
                v.y = half_kick(v.y, fy, hdt, inv_m);
                v.z = half_kick(v.z, fz, hdt, inv_m);
                if (last) {
                    s.frc[i] = mk4<T>(fx, fy, fz, T(0));
                } else {
                    v.x = half_kick(v.x, fx, hdt, inv_m);
                    v.y = half_kick(v.y, fy, hdt, inv_m);
                    v.z = half_kick(v.z, fz, hdt, inv_m);
                    T x = drift(xi.x, v.x, dt), y = drift(xi.y, v.y, dt), z = drift(xi.z, v.z, dt);
                    if (!(abs_less(x, T(1e30)) && abs_less(y, T(1e30)) && abs_less(z, T(1e30)))) {
                        bad |= ERRBIT_NONFINITE;
                        x = xi.x;
                        y = xi.y;
                        z = xi.z;
                    }
                    const T ex = x - xbi.x, ey = y - xbi.y, ez = z - xbi.z;
                    request = less_nonneg(s.half_skin2, ex * ex + ey * ey + ez * ez);
                    xi.x = x;
                    xi.y = y;
                    xi.z = z;
                    s.pos[buf ^ 1][i] = xi;
                }
                if (bad != 0 || request) {
                    if (bad) {
                        atomicOr(&c->err, bad);
                        c->abort = 1;
                    }
                    if (request) {
                        s.req[tl.rep] = 1;
                        c->any_req = 1;
                    }
                    // the step's own number: a block that is still reading it after
                    // this step's barrier does not take the next step's for it
                    *(volatile long long*)&c->stop = step;
                }
            }
            if (!last) buf ^= 1;
            if constexpr (TPP > 1) {
                // the particle's four lanes test its entries at one position
                xi.x = __shfl_sync(0xffffffffu, xi.x, threadIdx.x & 28);
                xi.y = __shfl_sync(0xffffffffu, xi.y, threadIdx.x & 28);
                xi.z = __shfl_sync(0xffffffffu, xi.z, threadIdx.x & 28);
            }
            ok = grid_barrier(c, phase++, s.run_fault, [&] { stopped = *(volatile long long*)&c->stop; });
            if (!ok || step == target || stopped == step) break;
        }
        if (lead) s.vel[i] = v;
    }
    // the last block to leave hands over to the graph
    grid_leave(c, [&] {
        c->step = step;
        c->buf = buf;
        if (fin && step == target) c->pos_ahead = 0;
        c->stop = -1;
        __threadfence();
        const bool more = step < target && *(volatile unsigned int*)&c->abort == 0;
        if (cond) cudaGraphSetConditional(cond, more ? 1u : 0u);
    });
}

template <class T>
__global__ void k_run_begin(DevSys<T> s, long long target, int final_step, int buf) {
    s.ctrl->target = target;
    s.ctrl->final_step = final_step;
    s.ctrl->buf = buf;
    s.ctrl->stop = -1;
}

// The forms of the kernel, the first whose blocks are resident at once beside
// nothing else being taken: FP32 16 entries in flight at two blocks an SM, then 8
// at six; FP64 four lanes per particle, then one (whose queues of long lists are
// slower than the step kernel with four: not taken there).  us per step as step
// graphs / resident, rebuilds included: KG melt FP32 1,000 17.2 / 8.4, 5,000 17.9 /
// 9.7, 40,000 18.7 / 11.5, 110,000 23 / 16.6; LJ fluid FP32 4,000 26.9 / 17.1, 27,436
// 34.3 / 25.0, 108,000 44.6 / 39.7; KG melt FP64 1,000 24.0 / 15.8, 10,000 33.9 / 25.5,
// 40,000 47.6 / 39.6.  Batches take them by the same rule, though some replica of a
// large one ends the kernel at nearly every step: FP32 2 x 1,000 beads 18.5 / 9.9, 64 x
// 1,000 50.9 / 49.1, 16 x 5,000 45.6 / 44.5; FP64 2 x 1,000 26.1 / 17.8, 64 x 1,000 94.2 /
// 93.4, 16 x 5,000 99.0 / 99.0.
enum : int { RUN_NONE = 0, RUN_A, RUN_B };
template <class T>
static int run_form(const DevSys<T>& s) {
    if (!s.lj_fast || s.dpd || s.le_on || s.mlp_on || s.cells_mode) return RUN_NONE;
    const int sms = s.sms;
    if (sizeof(T) == 4) return s.ntiles <= 2 * sms ? RUN_A : s.ntiles <= 6 * sms ? RUN_B : RUN_NONE;
    if (4 * s.ntiles <= 3 * sms) return RUN_A;
    return s.ntiles <= 3 * sms && s.cap < 64 ? RUN_B : RUN_NONE;
}

template <class T>
bool Launch<T>::run_fits(const DevSys<T>& s) { return run_form(s) != RUN_NONE; }

template <class T>
void Launch<T>::run_begin(const DevSys<T>& s, long long target, int final_step, int buf, cudaStream_t st) {
    k_run_begin<T><<<1, 1, 0, st>>>(s, target, final_step, buf);
}

template <class T>
cudaError_t Launch<T>::run(const DevSys<T>& s, unsigned long long cond, cudaStream_t st) {
    DevSys<T> a = s;
    void* args[] = {&a, &cond};
    const bool first = run_form(s) == RUN_A;
    const void* f;
    int blocks = s.ntiles;
    size_t smem = 0;
    if constexpr (sizeof(T) == 4) {
        f = first ? (const void*)k_run<T, 32, 4, 2> : (const void*)k_run<T, 32, 2, 6>;
    } else {
        f = first ? (const void*)k_run<T, 8, 1, 3> : (const void*)k_run<T, 32, 1, 3>;
        if (first) blocks *= 4;
        smem = (TILE / 32) * (first ? sizeof(PairQueue<T, false, 8>) : sizeof(PairQueue<T, false, 32>));
        const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    return cudaLaunchCooperativeKernel(f, dim3(blocks), dim3(TILE), args, smem, st);
}

template bool Launch<float>::run_fits(const DevSys<float>&);
template bool Launch<double>::run_fits(const DevSys<double>&);
template void Launch<float>::run_begin(const DevSys<float>&, long long, int, int, cudaStream_t);
template void Launch<double>::run_begin(const DevSys<double>&, long long, int, int, cudaStream_t);
template cudaError_t Launch<float>::run(const DevSys<float>&, unsigned long long, cudaStream_t);
template cudaError_t Launch<double>::run(const DevSys<double>&, unsigned long long, cudaStream_t);

}  // namespace espp
