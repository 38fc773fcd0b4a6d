// The per-particle force walks shared by the step kernel and the resident run
// kernel: the Verlet list (thread per particle, or through the warp's pair
// queue), the bonds and the Langevin thermostat.
#pragma once
#include <type_traits>

#include "kernels.cuh"
#include "packed.cuh"
#include "pair_queue.cuh"
#include "pair_terms.cuh"
#include "philox.cuh"

#ifndef ESPP_STEP_PREFETCH
#define ESPP_STEP_PREFETCH 2  // request the next batch's list groups early (see pair_loop)
#endif

namespace espp {

// A position: read-only for the whole kernel, or (COH) rewritten by other SMs
// between the grid barriers of a running kernel.  Then it is a plain load (never
// the non-coherent path, which the compiler may choose for a const restrict
// pointer): the barrier's acquire makes the others' writes visible to it, L1
// included.
template <class T, bool COH>
__device__ __forceinline__ V4<T> ldp(const V4<T>* p) {
    if constexpr (!COH) {
        return ld4<T>(p);
    } else if constexpr (sizeof(T) == 4) {
        V4<T> r;
        asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];"
                     : "=f"(r.x), "=f"(r.y), "=f"(r.z), "=f"(r.w)
                     : "l"(p));
        return r;
    } else {
        V4<T> r;
        asm volatile("ld.global.v2.f64 {%0, %1}, [%4];\n ld.global.v2.f64 {%2, %3}, [%4+16];"
                     : "=d"(r.x), "=d"(r.y), "=d"(r.z), "=d"(r.w)
                     : "l"(p));
        return r;
    }
}

// Sum of the pair forces on particle i over its Verlet list.  The list is
// read in batches of int4 groups: all indices of a batch first, then all
// neighbour positions, then the arithmetic, so that each thread keeps several
// independent loads in flight; the next batch's indices are prefetched.
// (FP64 handles, and the DPD thermostat but where step_walks says so, take
// queue_loop; the thermostat's terms follow each pair's force here as there.)
// Entries with x code 3 cross a sheared face (Lees-Edwards): their x
// difference is taken from the current offset in *le.
template <class T, bool ENERGY, bool MULTI, bool FAST, bool LE, int GB32 = 1, bool COH = false, bool DPD = false>
__device__ __forceinline__ void pair_loop(const DevSys<T>& s, const V4<T>* __restrict__ P, int i, int n,
                                          const V4<T>& xi, int ti, const PairRec<T>* pr1,
                                          T L0, T L1, T L2, T& fx, T& fy, T& fz, T& pe, T& vir, T& vxz,
                                          const LeCtx<T>* le, const DpdCtx<T>* dc = nullptr) {
    const T xim = xi.x - L0, yim = xi.y - L1, zim = xi.z - L2;
    constexpr int GB = GB32;  // int4 groups per batch
    const int ng = (n + 3) >> 2;
    const int4* __restrict__ nb = reinterpret_cast<const int4*>(s.nbr) + i;
    const size_t stride = (size_t)s.stride;
    const int gcap = s.cap >> 2;  // groups allocated per particle (>= 2)
    // the groups of the next batch are requested before the positions of the
    // current one, so their latency overlaps the current batch; the first
    // batch is read without waiting for the count (groups past the count are
    // allocated, and dropped whole)
    // padding entries (the rest of the last group, and whole groups past the
    // count) name the padding slot, whose position is far outside the box:
    // every entry is loaded and evaluated without a test of its own
    const int pad = s.nbr_pad;
    const int4 pad4 = make_int4(pad, pad, pad, pad);
    // FP32 single-type Lennard-Jones without energies (the step's hot path):
    // two entries per packed FP32x2 instruction, forces summed in two lanes
    constexpr bool PACK = FAST && !ENERGY && !DPD;
    f32x2 px = 0ull, py = 0ull, pz = 0ull;
    f32x2 xi2 = 0ull, yi2 = 0ull, zi2 = 0ull, sg2 = 0ull, e24 = 0ull;
    if constexpr (PACK) {
        xi2 = f2(xi.x, xi.x);
        yi2 = f2(xi.y, xi.y);
        zi2 = f2(xi.z, xi.z);
        sg2 = f2(pr1->sig2, pr1->sig2);
        e24 = f2(pr1->eps24, pr1->eps24);
    }
    int4 nxt[GB];
#pragma unroll
    for (int q = 0; q < GB; ++q) nxt[q] = q < gcap ? __ldg(nb + q * stride) : pad4;
    for (int g0 = 0; g0 < ng || g0 == 0; g0 += GB) {
        int jj[4 * GB];
#pragma unroll
        for (int q = 0; q < GB; ++q) {
            if (!ESPP_STEP_PREFETCH && g0 > 0) nxt[q] = __ldg(nb + (g0 + q) * stride);
            int4 a = nxt[q];
            if (g0 + q >= ng) a = pad4;
            jj[4 * q + 0] = a.x;
            jj[4 * q + 1] = a.y;
            jj[4 * q + 2] = a.z;
            jj[4 * q + 3] = a.w;
        }
#pragma unroll
        for (int q = 0; q < GB; ++q) {
            const int gn = g0 + GB + q;
            // ESPP_STEP_PREFETCH 1: request while the count may be in flight
            // (reads one group past the list); 2: only groups inside the list
            if ((ESPP_STEP_PREFETCH == 1 && gn < gcap) || (ESPP_STEP_PREFETCH == 2 && gn < ng))
                nxt[q] = __ldg(nb + gn * stride);
        }
        int codes = 0;
#pragma unroll
        for (int q = 0; q < 4 * GB; ++q) codes |= jj[q];
        V4<T> xj[4 * GB];
#pragma unroll
        for (int q = 0; q < 4 * GB; ++q) xj[q] = ldp<T, COH>(P + nbr_slot(jj[q]));
        if constexpr (PACK) {
            // entries two at a time; every entry goes through the same
            // arithmetic whichever batch it falls in, so the sums do not
            // depend on the batch shape
            const T rc2 = pr1->rc2;
            const f32x2 two = f2(2.f, 2.f), mone = f2(-1.f, -1.f);
            const bool plain = (codes & ~NBR_INDEX_MASK) == 0;  // no pair of the batch crosses a face
#pragma unroll
            for (int q = 0; q < 4 * GB; q += 2) {
                f32x2 dx, dy, dz;
                if (plain) {
                    dx = f2sub(xi2, f2(xj[q].x, xj[q + 1].x));
                    dy = f2sub(yi2, f2(xj[q].y, xj[q + 1].y));
                    dz = f2sub(zi2, f2(xj[q].z, xj[q + 1].z));
                } else {
                    T d[2][3];
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int code = nbr_code(jj[q + h]);
                        if (LE && (code & 3) == 3)
                            d[h][0] = le_dx(xi.x, xj[q + h].x, (code >> 4) == 1 ? 1 : -1, le->d, L0, le->inv_Lx);
                        else
                            d[h][0] = shifted_diff(xi.x, xim, xj[q + h].x, L0, code & 3);
                        d[h][1] = shifted_diff(xi.y, yim, xj[q + h].y, L1, (code >> 2) & 3);
                        d[h][2] = shifted_diff(xi.z, zim, xj[q + h].z, L2, code >> 4);
                    }
                    dx = f2(d[0][0], d[1][0]);
                    dy = f2(d[0][1], d[1][1]);
                    dz = f2(d[0][2], d[1][2]);
                }
                float ra, rb;
                f2split(f2fma(dz, dz, f2fma(dy, dy, f2mul(dx, dx))), ra, rb);
                const f32x2 inv = f2(recip(ra), recip(rb));
                const f32x2 s2 = f2mul(sg2, inv);
                const f32x2 s6 = f2mul(f2mul(s2, s2), s2);
                float fa, fb;
                f2split(f2mul(f2mul(f2mul(e24, s6), f2fma(s6, two, mone)), inv), fa, fb);
                const f32x2 fr = f2(ra < rc2 ? fa : 0.f, rb < rc2 ? fb : 0.f);
                px = f2fma(fr, dx, px);
                py = f2fma(fr, dy, py);
                pz = f2fma(fr, dz, pz);
            }
        } else if ((codes & ~NBR_INDEX_MASK) == 0) {
            // no pair of this batch crosses a face (the common case)
#pragma unroll
            for (int q = 0; q < 4 * GB; ++q) {
                const T dx = xi.x - xj[q].x, dy = xi.y - xj[q].y, dz = xi.z - xj[q].z;
                pair_term<T, ENERGY, MULTI, FAST>(s, ti, pr1, dx, dy, dz, bits_as_int(xj[q].w), fx, fy, fz, pe,
                                                  vir, vxz);
                if constexpr (DPD) {
                    const T r2 = dx * dx + dy * dy + dz * dz;
                    if (r2 < s.ip->dpd_rc2)
                        dpd_term<T, LE>(s.ip, *dc, dx, dy, dz, r2, ld4<T>(s.vsnap + nbr_slot(jj[q])), fx, fy, fz);
                }
            }
        } else {
#pragma unroll
            for (int q = 0; q < 4 * GB; ++q) {
                const int code = nbr_code(jj[q]);
                int nz = 0;
                T dx;
                if (LE && (code & 3) == 3) {
                    nz = (code >> 4) == 1 ? 1 : -1;
                    dx = le_dx(xi.x, xj[q].x, nz, le->d, L0, le->inv_Lx);
                } else {
                    dx = shifted_diff(xi.x, xim, xj[q].x, L0, code & 3);
                }
                const T dy = shifted_diff(xi.y, yim, xj[q].y, L1, (code >> 2) & 3);
                const T dz = shifted_diff(xi.z, zim, xj[q].z, L2, code >> 4);
                pair_term<T, ENERGY, MULTI, FAST>(s, ti, pr1, dx, dy, dz, bits_as_int(xj[q].w), fx, fy, fz,
                                                  pe, vir, vxz);
                if constexpr (DPD) {
                    const T r2 = dx * dx + dy * dy + dz * dz;
                    if (r2 < s.ip->dpd_rc2)
                        dpd_term<T, LE>(s.ip, *dc, dx, dy, dz, r2, ld4<T>(s.vsnap + nbr_slot(jj[q])), fx, fy, fz, nz);
                }
            }
        }
    }
    if constexpr (PACK) {
        float a, b;
        f2split(px, a, b);
        fx += a + b;
        f2split(py, a, b);
        fy += a + b;
        f2split(pz, a, b);
        fz += a + b;
    }
}

// ---- the warp's pair queue ---------------------------------------------------
// FP64 handles and the DPD thermostat: a pair's term is expensive (FP64
// instructions at a small fraction of the FP32 rate; a Philox block) and a
// quarter to two thirds of the list entries lie beyond the cutoff, so a thread
// that walks its own list runs the term for nearly every entry, with the lanes
// whose entry is inside.  Here a warp first tests QG groups of every list in
// FP32 (FP64 handles: on coordinates cut to FP32, against a widened cutoff) and
// keeps the entries inside, then evaluates the warp's entries 32 at a time, one
// per lane whoever owns them, the exact test included, into shared memory; every
// particle then adds its own terms in list order, as a walk of the list would.
// Step kernel, walking its own list / queue: KG melt of 1M FP64 876 / 458 us, LJ
// fluid of 256,000 FP64 1241 / 822 us, DPD fluid of 786,432 FP32 446 / 301 us (215 M
// warp instructions instead of 284 M, 26 of 32 lanes active instead of 11).
template <class T, bool DPD, int PPW>
struct PairQueueTerms {
    // list groups per block of the queue, terms held at a time.  FP32: small,
    // for the shared memory they take is L1 that the gathers lose (DPD fluid of
    // 786,432, step kernel: 4 / 128 301 us, 8 / 256 377 us, 4 / 64 303 us); FP64:
    // large, for every stretch of terms costs its particles' additions once
    // more (KG melt of 1M: 8 / 256 458 us, 4 / 128 493 us, 4 / 64 527 us)
    static constexpr int QG = sizeof(T) == 8 ? 8 : 4;
    static constexpr int QR = sizeof(T) == 8 && !DPD ? 256 : 128;
    int col[QG * 4 * PPW];  // entries inside: row k of the particle's column
    T fr[QR], dx[QR], dy[QR], dz[QR];
};
// with the thermostat's term (FP64 without it: four warps' queues are 48 KB)
template <class T, int PPW>
struct PairQueueTh : PairQueueTerms<T, true, PPW> {
    T th[PairQueueTerms<T, true, PPW>::QR];
};
template <class T, bool DPD, int PPW>
using PairQueue = std::conditional_t<DPD, PairQueueTh<T, PPW>, PairQueueTerms<T, false, PPW>>;

// PPW: particles per warp, 32 (one lane each) or 8 (four lanes share a
// particle: lane t takes entry t of every group).  Returns the pair force on the
// lane's particle (PPW 8: on each of its four lanes); pe, vir, vxz: sums over the
// pairs this lane evaluated.
template <class T, bool ENERGY, bool MULTI, bool FAST, bool DPD, bool LE, int PPW, bool COH = false>
__device__ __forceinline__ void queue_loop(const DevSys<T>& s, const V4<T>* __restrict__ P,
                                           PairQueue<T, DPD, PPW>& Q, int ibase, int i, int n, const RepGeom<T>& g,
                                           const V4<T>& xi, const PairRec<T>* pr1, T rcmax2, const LeCtx<T>& le,
                                           long long step, T& fx, T& fy, T& fz, T& pe, T& vir, T& vxz) {
    constexpr int TPP = 32 / PPW;         // lanes per particle
    constexpr int QG = PairQueue<T, DPD, PPW>::QG, QR = PairQueue<T, DPD, PPW>::QR;
    constexpr int C = TPP == 1 ? 4 : 1;   // entries of a group per lane
    static_assert(TPP == 1 || TPP == 4, "one or four lanes per particle");
    const int lane = threadIdx.x & 31, t0 = TPP == 1 ? 0 : lane & 3;
    int* __restrict__ col = Q.col + (TPP == 1 ? lane : lane >> 2);
    const float L0 = (float)g.L[0], L1 = (float)g.L[1], L2 = (float)g.L[2];
    const float x = cut(xi.x), y = cut(xi.y), z = cut(xi.z);
    float rc2;
    if constexpr (sizeof(T) == 4) {
        rc2 = rcmax2;
    } else {
        // every component is off by at most 2^-20 of a coordinate on either
        // side (and by its image shift's rounding)
        const float r2 = (float)rcmax2, r = sqrtf(r2), e = 3e-6f * (fmaxf(L0, fmaxf(L1, L2)) + 2.f * (float)s.skin);
        rc2 = (r2 + 3.47f * r * e + 3.f * e * e) * 1.00001f;
    }
    const float led = (float)le.d, linv = (float)le.inv_Lx;
    const int ng = (n + 3) >> 2;
    const int ngw = __reduce_max_sync(0xffffffffu, ng);
    const size_t stride = (size_t)s.stride;
    const int pad = s.nbr_pad;
    const int4* __restrict__ nb4 = reinterpret_cast<const int4*>(s.nbr) + i;
    const int* __restrict__ nb1 = s.nbr + 4 * (size_t)i + t0;
    for (int g0 = 0; g0 < ngw; g0 += QG) {
        int cnt = 0;  // entries in the particle's column
        const int g1 = min(g0 + QG, ngw);
        // ---- the entries inside the (widened) cutoff
#pragma unroll 2
        for (int q = g0; q < g1; ++q) {
            int e[C];
            if constexpr (C == 4) {
                const int4 a = q < ng ? __ldg(nb4 + q * stride) : make_int4(pad, pad, pad, pad);
                e[0] = a.x;
                e[1 % C] = a.y;
                e[2 % C] = a.z;
                e[3 % C] = a.w;
            } else {
                e[0] = q < ng ? __ldg(nb1 + 4 * (size_t)q * stride) : pad;
            }
            V4<T> xj[C];
#pragma unroll
            for (int t = 0; t < C; ++t) xj[t] = ldp<T, COH>(P + nbr_slot(e[t]));
#pragma unroll
            for (int t = 0; t < C; ++t) {
                const int code = nbr_code(e[t]);
                const float xq = cut(xj[t].x), yq = cut(xj[t].y), zq = cut(xj[t].z);
                float dx = x - xq, dy = y - yq, dz = z - zq;
                if (code != 0) {
                    dx = shifted_diff(x, x - L0, xq, L0, code & 3);
                    dy = shifted_diff(y, y - L1, yq, L1, (code >> 2) & 3);
                    dz = shifted_diff(z, z - L2, zq, L2, code >> 4);
                    if (LE && (code & 3) == 3) dx = le_dx(x, xq, (code >> 4) == 1 ? 1 : -1, led, L0, linv);
                }
                const bool in = dx * dx + dy * dy + dz * dz < rc2;
                if constexpr (TPP == 1) {
                    if (in) {
                        col[cnt * PPW] = e[t];
                        ++cnt;
                    }
                } else {
                    const unsigned int m = (__ballot_sync(0xffffffffu, in) >> (lane & 28)) & 15u;
                    if (in) col[(cnt + __popc(m & ((1u << t0) - 1u))) * PPW] = e[t];
                    cnt += __popc(m);
                }
            }
        }
        // where each particle's terms start in the warp's queue
        int total;
        const int off = queue_offsets(t0 == 0 ? cnt : 0, total);
        const int from = TPP == 1 ? off : __shfl_sync(0xffffffffu, off, lane & 28), to = from + cnt;
        for (int r0 = 0; r0 < total; r0 += QR) {
            const int nr = min(QR, total - r0);
            __syncwarp();
            for (int b = 0; b < nr; b += 32) {
                const int q = min(b + lane, nr - 1) + r0;
                int k;
                const int own = queue_owner(off, q, k);
                if (b + lane < nr) {
                    const int p = TPP == 1 ? own : own >> 2;
                    const int e = Q.col[k * PPW + p];
                    const int ii = ibase + p, j = nbr_slot(e), code = nbr_code(e);
                    const V4<T> a = ldp<T, COH>(P + ii), xj = ldp<T, COH>(P + j);
                    int nz = 0;
                    T dx, dy, dz;
                    if (code == 0) {
                        dx = a.x - xj.x;
                        dy = a.y - xj.y;
                        dz = a.z - xj.z;
                    } else {
                        if (LE && (code & 3) == 3) {
                            nz = (code >> 4) == 1 ? 1 : -1;
                            dx = le_dx(a.x, xj.x, nz, le.d, g.L[0], le.inv_Lx);
                        } else {
                            dx = shifted_diff(a.x, a.x - g.L[0], xj.x, g.L[0], code & 3);
                        }
                        dy = shifted_diff(a.y, a.y - g.L[1], xj.y, g.L[1], (code >> 2) & 3);
                        dz = shifted_diff(a.z, a.z - g.L[2], xj.z, g.L[2], code >> 4);
                    }
                    const T r2 = dx * dx + dy * dy + dz * dz;
                    Q.fr[b + lane] = pair_scalar<T, ENERGY, MULTI, FAST>(s, MULTI ? bits_as_int(a.w) : 0, pr1, dx, dz, r2,
                                                                         bits_as_int(xj.w), pe, vir, vxz);
                    Q.dx[b + lane] = dx;
                    Q.dy[b + lane] = dy;
                    Q.dz[b + lane] = dz;
                    if constexpr (DPD) {
                        T th = T(0);
                        if (less_nonneg(r2, s.ip->dpd_rc2)) {
                            DpdCtx<T> dc;
                            dc.vi = ld4<T>(s.vsnap + ii);
                            dc.seed = g.seed;
                            dc.step = step;
                            dc.le_vs = le.vs;
                            th = dpd_value<T, LE>(s.ip, dc, dx, dy, dz, r2, ld4<T>(s.vsnap + j), nz);
                        }
                        Q.th[b + lane] = th;
                    }
                }
            }
            __syncwarp();
            queue_add<T, DPD, TPP>(Q, max(from, r0) - r0, min(to, r0 + nr) - r0, t0, fx, fy, fz);
        }
        __syncwarp();
    }
    if constexpr (TPP == 4) {
        const T f = fx;
        fx = __shfl_sync(0xffffffffu, f, lane & 28);
        fy = __shfl_sync(0xffffffffu, f, (lane & 28) + 1);
        fz = __shfl_sync(0xffffffffu, f, (lane & 28) + 2);
    }
}

// Bond forces (paper "Functionality": bonded interactions; FENE or tabulated) of
// a particle with partners b at xp0, xp1; returns whether a bond is broken.
template <class T, bool ENERGY, bool LE>
__device__ __forceinline__ bool bond_forces(const DevSys<T>& s, const RepGeom<T>& g, const V4<T>& xi, int2 b,
                                            const V4<T>& xp0, const V4<T>& xp1, const LeCtx<T>& le, T& fx, T& fy,
                                            T& fz, T& pb, T& vir, T& vxz, double& blen, double& bcnt) {
    const T L0 = g.L[0], L1 = g.L[1], L2 = g.L[2];
    const T H0 = g.halfL[0], H1 = g.halfL[1], H2 = g.halfL[2];
    bool broken = false;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int p = q == 0 ? b.x : b.y;
        if (p < 0) continue;
        const V4<T> xp = q == 0 ? xp0 : xp1;
        const T dz = min_image(xi.z, xp.z, L2, H2);
        const T dy = min_image(xi.y, xp.y, L1, H1);
        T dx;
        if (LE && (xi.z - xp.z > H2 || xi.z - xp.z < -H2)) {
            // bond across a sheared face
            dx = le_dx(xi.x, xp.x, xi.z - xp.z > H2 ? 1 : -1, le.d, L0, le.inv_Lx);
        } else {
            dx = min_image(xi.x, xp.x, L0, H0);
        }
        const T r2 = dx * dx + dy * dy + dz * dz;
        T fr, ub = T(0);
        if (s.bond.kind == ESPP_FENE) {
            T one_m = T(1) - r2 * s.bond.inv_R02;
            if (!positive(one_m)) {
                broken = true;
                one_m = T(1e-6);
            }
            fr = -s.bond.K * recip(one_m);
            if (ENERGY) ub = -s.bond.halfKR02 * log(one_m);
        } else {
            T r = sqrt(r2), F;
            if (!(r < s.bond.rmax)) {
                broken = true;
                r = T(0);
            }
            table_lookup(s.tab + s.bond.tab_off, s.bond.tab_n, s.bond.inv_dr, r, ub, F);
            fr = r > T(0) ? F / r : T(0);
        }
        fx += fr * dx;
        fy += fr * dy;
        fz += fr * dz;
        if (ENERGY) {
            pb += ub;
            vir += fr * r2;
            vxz += fr * dx * dz;
            blen += sqrt((double)r2);
            bcnt += 1.0;
        }
    }
    return broken;
}

// Langevin friction and noise of the step, added to the force.
template <class T, bool LE>
__device__ __forceinline__ void langevin_forces(const IntParams<T>* __restrict__ ip, const RepGeom<T>& g, int ti,
                                                const V4<T>& xi, const V4<T>& v, long long step, const LeCtx<T>& le,
                                                T& fx, T& fy, T& fz) {
    if (ip->gamma == T(0)) return;
    T rx, ry, rz;
    langevin_noise<T>(g.seed, bits_as_int(v.w), step, rx, ry, rz);
    const T amp = ip->noise_amp[ti];
    const T gm = ip->gamma * ip->mass[ti];
    // friction relative to the shear profile (Lees-Edwards)
    const T vxp = LE ? v.x - le.shear * (xi.z - g.halfL[2]) : v.x;
    fx += -gm * vxp + amp * rx;
    fy += -gm * v.y + amp * ry;
    fz += -gm * v.z + amp * rz;
}

}  // namespace espp
