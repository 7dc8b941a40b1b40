// frame.cuh -- device side of the frame schedules (frame.h): a thread's slots
// and parities in a stage, <Z> and O psi on the last stage's blocks.
#pragma once

#include "frame.h"
#include "sweep.cuh"

namespace vqc {

// XOR of v[0 .. 16) over the set bits of t (v 16-byte aligned, entries past nb
// zero): all loads independent, four entries each.
__device__ __forceinline__ uint32_t xor_bits(const void* v, int nb, int t) {
    const uint4* p = reinterpret_cast<const uint4*>(v);
    uint32_t b = 0;
    auto four = [&](int i) {
        const uint4 x = p[i];
        b ^= ((t >> (4 * i)) & 1) ? x.x : 0u;
        b ^= ((t >> (4 * i + 1)) & 1) ? x.y : 0u;
        b ^= ((t >> (4 * i + 2)) & 1) ? x.z : 0u;
        b ^= ((t >> (4 * i + 3)) & 1) ? x.w : 0u;
    };
    four(0);
    four(1);
    if (nb > 8) {
        four(2);
        four(3);
    }
    return b;
}

// Slot base (and, when the stage needs them, outside parities) of thread t; fl is
// the tile's flip of the stage.
template <int K>
__device__ __forceinline__ StageView frame_view(const FStage* sp, int t, uint32_t fl_slot, uint32_t fl_mask,
                                                int h, int32_t (&sg)[K]) {
#pragma unroll
    for (int j = 0; j < K; ++j) sg[j] = sp->sigma[j];
    const int nb = sp->nthreadbits;
    StageView v;
    v.swb = (uint32_t)h ^ fl_slot ^ xor_bits(sp->tau, nb, t);
    v.pb = 0;
    if (sp->nsel) v.pb = fl_mask ^ xor_bits(sp->tmask, nb, t);
    return v;
}

// In place: v[c] becomes the sum over r of (-1)^parity(c & r) v[r].
template <typename R, int K>
__device__ __forceinline__ void walsh(R (&v)[1 << K]) {
#pragma unroll
    for (int b = 0; b < K; ++b)
#pragma unroll
        for (int r = 0; r < (1 << K); ++r)
            if (!((r >> b) & 1)) {
                const R x = v[r], y = v[r | (1 << b)];
                v[r] = x + y;
                v[r | (1 << b)] = x - y;
            }
}

// Per-warp sums of E_j = sum (-1)^{bit j} |a|^2 over the group's blocks, to
// red[warp_in_group * n + j].  One Walsh transform of the block's |a|^2 holds the
// signed sum of every local mask; qubit j takes its own, signed by its outside
// parity (bit j of pbf).  Full-warp groups sum 16 qubits at a time by a
// reduce-scatter butterfly.
template <typename R, int K, bool FULL>
__device__ __forceinline__ void expz_frame(const uint8_t* lmask, uint32_t pbf, const C2<R> (&a)[1 << K], int n,
                                           R* red, const Geo& q, int lane, int warp_in_group) {
    R W[1 << K];
#pragma unroll
    for (int r = 0; r < (1 << K); ++r) W[r] = fma(a[r].x, a[r].x, a[r].y * a[r].y);
    walsh<R, K>(W);
    if constexpr (FULL) {
        for (int j0 = 0; j0 < n; j0 += 16) {
            R ez[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                ez[j] = 0;
                if (j0 + j < n) {
                    const R s = W[lmask[j0 + j]];
                    ez[j] = ((pbf >> (j0 + j)) & 1u) ? -s : s;
                }
            }
            const int j = j0 + warp_reduce_scatter<R, 16>(ez, lane);
            if ((lane & 1) == 0 && j < n) red[warp_in_group * n + j] = ez[0];
        }
    } else {
        for (int j = 0; j < n; ++j) {
            const R s = W[lmask[j]];
            const R val = reduce1<R>(((pbf >> j) & 1u) ? -s : s, q.lanes, q.mask);
            if ((q.t & (q.lanes - 1)) == 0) red[warp_in_group * n + j] = val;
        }
    }
}

// lam = O psi on the block, O = sum_j gE_j Z_j: the coefficients of each local
// mask, one Walsh transform.
template <typename R, int K, typename GI>
__device__ __forceinline__ void lambda_frame(const uint8_t* lmask, uint32_t pbf, const GI* gb, int n,
                                             const C2<R> (&a)[1 << K], C2<R> (&l)[1 << K]) {
    R g[1 << K];
#pragma unroll
    for (int r = 0; r < (1 << K); ++r) g[r] = 0;
    for (int j = 0; j < n; ++j) {
        const R v = as_r<R>(gb[j]);
        g[lmask[j]] += ((pbf >> j) & 1u) ? -v : v;
    }
    walsh<R, K>(g);
#pragma unroll
    for (int r = 0; r < (1 << K); ++r) l[r] = cm<R>(g[r] * a[r].x, g[r] * a[r].y);
}

}  // namespace vqc
