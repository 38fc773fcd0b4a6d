// The warp's pair queue: entries found inside the cutoff by the lanes of a warp,
// evaluated 32 at a time whoever owns them, their terms added by their owners in
// order.  Used by the step kernel (Verlet lists) and the list-free cell forces.
#pragma once
#include "common.cuh"

namespace espp {

// a coordinate in FP32: FP64 ones are cut to 20 mantissa bits (|x| < 2^-126 to 0)
__device__ __forceinline__ float cut(float x) { return x; }
__device__ __forceinline__ float cut(double x) {
    const int hi = __double2hiint(x);
    const unsigned int a = max(hi & 0x7fffffff, 0x38000000) - 0x38000000;
    return __uint_as_float((a << 3) | (hi & 0x80000000u));
}

// Exclusive offsets of the lanes' counts in the warp's queue, and the total.
__device__ __forceinline__ int queue_offsets(int cnt, int& total) {
    const int lane = threadIdx.x & 31;
    int off = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, off, o);
        if (lane >= o) off += u;
    }
    total = __shfl_sync(0xffffffffu, off, 31);
    return off - cnt;
}

// The lane that owns entry q of the queue (the last one whose entries start at or
// before q) and the entry's place k among that lane's.
__device__ __forceinline__ int queue_owner(int off, int q, int& k) {
    int own = 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        if (__shfl_sync(0xffffffffu, off, own + o) <= q) own += o;
    k = q - __shfl_sync(0xffffffffu, off, own);
    return own;
}

// The terms [k0, k1) of Q added to the lane's particle in order, as a walk of its
// list adds them (conservative force, then the thermostat's).  TPP > 1: the
// particle's lane `sub` adds component `sub`, held in fx.
template <class T, bool DPD, int TPP, class Q>
__device__ __forceinline__ void queue_add(const Q& q, int k0, int k1, int sub, T& fx, T& fy, T& fz) {
    if constexpr (TPP == 1) {
        for (int k = k0; k < k1; ++k) {
            const T fr = q.fr[k], dx = q.dx[k], dy = q.dy[k], dz = q.dz[k];
            fx = fma_rn(fr, dx, fx);
            fy = fma_rn(fr, dy, fy);
            fz = fma_rn(fr, dz, fz);
            if constexpr (DPD) {
                const T th = q.th[k];
                fx = fma_rn(th, dx, fx);
                fy = fma_rn(th, dy, fy);
                fz = fma_rn(th, dz, fz);
            }
        }
    } else if (sub < 3) {
        const T* d = sub == 0 ? q.dx : sub == 1 ? q.dy : q.dz;
        for (int k = k0; k < k1; ++k) {
            const T dd = d[k];
            fx = fma_rn(q.fr[k], dd, fx);
            if constexpr (DPD) fx = fma_rn(q.th[k], dd, fx);
        }
    }
}

}  // namespace espp
