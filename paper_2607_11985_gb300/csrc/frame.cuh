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

// XOR of cols[i] over the set bits of v.
template <typename T, int N>
__device__ __forceinline__ uint32_t xor_cols(const T (&cols)[N], uint32_t v) {
    uint32_t r = 0;
    for (int i = 0; v; ++i, v >>= 1)
        if (v & 1u) r ^= (uint32_t)cols[i];
    return r;
}

// A thread's block in a stage: the byte offset of its base in the group's tiles and
// (when the stage needs them) its outside parities; sb the local bits' byte offsets.
// base: the offset in the tile that does not depend on the tile (frame_base); fl:
// the tile's flip of the stage, as a byte offset, and its parities.
struct FrameView {
    uint32_t off, pb;
};
template <typename R>
__device__ __forceinline__ uint32_t frame_base(const FStage* sp, int t, uint32_t g0) {
    return (g0 ^ xor_bits(sp->tau, sp->nthreadbits, t)) * (uint32_t)sizeof(C2<R>);
}
template <typename R, int K>
__device__ __forceinline__ FrameView frame_view(const FStage* sp, int t, uint32_t base, uint2 fl,
                                                uint32_t (&sb)[K]) {
#pragma unroll
    for (int j = 0; j < K; ++j) sb[j] = (uint32_t)sp->sigma[j] * (uint32_t)sizeof(C2<R>);
    FrameView v;
    v.off = base ^ fl.x;
    v.pb = 0;
    if (sp->nsel) v.pb = fl.y ^ xor_bits(sp->tmask, sp->nthreadbits, t);
    return v;
}

// The block's amplitudes between registers and shared memory, in Gray-code order:
// one XOR per access on a running byte offset (two of them, for the two halves of
// the block).  tiles: start of the CTA's tiles.
template <typename R, int K>
__device__ __forceinline__ void frame_load(C2<R> (&a)[1 << K], const unsigned char* tiles, uint32_t off,
                                           const uint32_t (&sb)[K]) {
    constexpr int H = 1 << (K - 1);
    uint32_t o0 = off, o1 = off ^ sb[K - 1];
#pragma unroll
    for (int i = 0; i < H; ++i) {
        const int r = i ^ (i >> 1);
        a[r] = *reinterpret_cast<const C2<R>*>(tiles + o0);
        a[r | H] = *reinterpret_cast<const C2<R>*>(tiles + o1);
        if (i + 1 < H) {
            const int b = (i & 1) == 0 ? 0 : (i & 2) == 0 ? 1 : (i & 4) == 0 ? 2 : 3;   // the bit that changes
            o0 ^= sb[b];
            o1 ^= sb[b];
        }
    }
}
// (An empty asm hides off's value from the compiler, so that it does not keep the
// load's offsets live in registers across the stage's ops.)
template <typename R, int K>
__device__ __forceinline__ void frame_store(const C2<R> (&a)[1 << K], unsigned char* tiles, uint32_t off,
                                            const uint32_t (&sb)[K]) {
    constexpr int H = 1 << (K - 1);
    asm volatile("" : "+r"(off));
    uint32_t o0 = off, o1 = off ^ sb[K - 1];
#pragma unroll
    for (int i = 0; i < H; ++i) {
        const int r = i ^ (i >> 1);
        *reinterpret_cast<C2<R>*>(tiles + o0) = a[r];
        *reinterpret_cast<C2<R>*>(tiles + o1) = a[r | H];
        if (i + 1 < H) {
            const int b = (i & 1) == 0 ? 0 : (i & 2) == 0 ? 1 : (i & 4) == 0 ? 2 : 3;
            o0 ^= sb[b];
            o1 ^= sb[b];
        }
    }
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

// Per-warp sums of E_j = sum (-1)^{bit j} |a|^2 over the group's blocks: put(j, sum)
// in one lane per qubit.  One Walsh transform of the block's |a|^2 holds the signed
// sum of every local mask; qubit j takes its own, signed by its outside parity (bit
// j of pbf).  Full-warp groups sum 16 (or 8) qubits at a time by a reduce-scatter
// butterfly.
template <typename R, int K, int NV, typename Put>
__device__ __forceinline__ void expz_group(const uint8_t* lmask, uint32_t pbf, const R (&W)[1 << K], int n, int j0,
                                           int lane, Put put) {
    R ez[NV];
#pragma unroll
    for (int j = 0; j < NV; ++j) {
        ez[j] = 0;
        if (j0 + j < n) {
            const R s = W[lmask[j0 + j]];
            ez[j] = ((pbf >> (j0 + j)) & 1u) ? -s : s;
        }
    }
    const int j = j0 + warp_reduce_scatter<R, NV>(ez, lane);
    if ((lane & (32 / NV - 1)) == 0 && j < n) put(j, ez[0]);
}
template <typename R, int K, bool FULL, typename Put>
__device__ __forceinline__ void expz_frame(const uint8_t* lmask, uint32_t pbf, const C2<R> (&a)[1 << K], int n,
                                           const Geo& q, int lane, Put put) {
    R W[1 << K];
#pragma unroll
    for (int r = 0; r < (1 << K); ++r) W[r] = fma(a[r].x, a[r].x, a[r].y * a[r].y);
    walsh<R, K>(W);
    if constexpr (FULL) {
        if (n <= 8) {
            expz_group<R, K, 8>(lmask, pbf, W, n, 0, lane, put);
        } else {
            for (int j0 = 0; j0 < n; j0 += 16) expz_group<R, K, 16>(lmask, pbf, W, n, j0, lane, put);
        }
    } else {
        for (int j = 0; j < n; ++j) {
            const R s = W[lmask[j]];
            const R val = reduce1<R>(((pbf >> j) & 1u) ? -s : s, q.lanes, q.mask);
            if ((q.t & (q.lanes - 1)) == 0) put(j, val);
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

// ---------------------------------------------------------------- pure stages
// A stage of 2x2 updates only, at most one per local position: straight-line code
// over the positions, each under one uniform branch, instead of a descriptor load
// and a jump per op.
template <typename R, int EW = EntryWords<R>::value>
__device__ __forceinline__ const R* op_table(uint2 raw, const R* sh_tab, const R* ps_tab) {
    return (((raw.x >> 24) & OPF_PER_SAMPLE) ? ps_tab : sh_tab) + EW * (raw.y & 0xffff);
}

template <typename R, int K, int EW = EntryWords<R>::value>
__device__ __forceinline__ void pure_forward(const uint2* ops, unsigned pm, C2<R> (&a)[1 << K], const R* sh_tab,
                                             const R* ps_tab) {
    const R* tp[K];
    {
        int o = 0;
#pragma unroll
        for (int j = 0; j < K; ++j) {
            tp[j] = op_table<R, EW>(ops[o], sh_tab, ps_tab);
            o += (pm >> j) & 1;
        }
    }
#define VQC_PURE(T_) \
    if constexpr (T_ < K) if ((pm >> T_) & 1) m1_entry<R, K, T_, false>(a, tp[T_]);
    VQC_PURE(0) VQC_PURE(1) VQC_PURE(2) VQC_PURE(3) VQC_PURE(4)
#undef VQC_PURE
}

// Sum the three components of K <= 4 ops over a warp by one reduce-scatter
// butterfly (13 shuffles for 4 ops).  Returns 4 op + component for the lanes
// that end up with a sum (in v[0][0]), -1 for the others.
template <typename R, int K>
__device__ __forceinline__ int reduce_runs(R (&v)[K][3], int lane) {
    static_assert(K >= 1 && K <= 4, "K");
    const unsigned full = 0xffffffffu;
    const int u0 = (lane >> 4) & 1, u1 = (lane >> 3) & 1, u2 = (lane >> 2) & 1, u3 = (lane >> 1) & 1;
#pragma unroll
    for (int i = 0; i < (K > 1 ? 2 : 1); ++i)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            if (i + 2 < K) {
                const R send = u0 ? v[i][c] : v[i + 2 < K ? i + 2 : 0][c];
                const R keep = u0 ? v[i + 2 < K ? i + 2 : 0][c] : v[i][c];
                v[i][c] = keep + shx<R>(send, 16, full);
            } else {
                v[i][c] += shx<R>(v[i][c], 16, full);
            }
        }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        if (K > 1) {
            const R send = u1 ? v[0][c] : v[K > 1 ? 1 : 0][c];
            const R keep = u1 ? v[K > 1 ? 1 : 0][c] : v[0][c];
            v[0][c] = keep + shx<R>(send, 8, full);
        } else {
            v[0][c] += shx<R>(v[0][c], 8, full);
        }
    }
    const R p = shx<R>(u2 ? v[0][0] : v[0][2], 4, full), r = shx<R>(v[0][1], 4, full);
    R x = (u2 ? v[0][2] : v[0][0]) + p, y = v[0][1] + r;
    const R send = u2 ? x : (u3 ? x : y), keep = u2 ? x : (u3 ? y : x);
    x = keep + shx<R>(send, 2, full);
    x += shx<R>(x, 1, full);
    v[0][0] = x;
    const int op = 2 * u0 + u1;
    return (lane & 1) || (u2 && u3) || op >= K ? -1 : 4 * op + (u2 ? 2 : u3);
}

// The adjoint of a pure stage.  Its runs act on different local bits, so every
// run's (tx, ty, tz) can be taken at the stage's output, and one butterfly sums all
// of them over the warp before the updates, whose registers it would otherwise
// hold (16-qubit step 6.90 -> 6.74 ms).  Packed forms of the sums (two components
// per FFMA2, the tz of all runs from one product per amplitude) execute fewer
// instructions but measured 2-3% slower.
template <int K>
__device__ __forceinline__ void pure_backward(const uint2* ops, unsigned pm, float2 (&a)[1 << K],
                                              float2 (&l)[1 << K], const float* sh_tab, const float* ps_tab,
                                              float* acc, int wg, int lane, int warp_in_group) {
    uint2 raw[K];
    unsigned am = 0;   // positions that accumulate
    {
        int o = 0;
#pragma unroll
        for (int j = 0; j < K; ++j) {
            raw[j] = ops[o];
            const unsigned on = (pm >> j) & 1;
            o += on;
            am |= (on && ((raw[j].x >> 24) & OPF_HAS_ACC)) ? 1u << j : 0u;
        }
    }
    if (am) {
        float v[K][3];
#pragma unroll
        for (int j = 0; j < K; ++j) v[j][0] = v[j][1] = v[j][2] = 0;
#define VQC_PURE(T_)                                     \
        if constexpr (T_ < K)                            \
            if ((am >> T_) & 1) {                        \
                float t[4] = {0, 0, 0, 0};               \
                m1_t3<float, K, T_>(a, l, t);            \
                v[T_][0] = t[0];                         \
                v[T_][1] = t[1];                         \
                v[T_][2] = t[2];                         \
            }
        VQC_PURE(0) VQC_PURE(1) VQC_PURE(2) VQC_PURE(3)
#undef VQC_PURE
        const int idx = reduce_runs<float, K>(v, lane);
        const int j = idx >> 2;
        if (idx >= 0 && ((am >> j) & 1)) {
            const unsigned aux = ops[__popc(pm & ((1u << j) - 1u))].y >> 16;
            acc[((size_t)aux * wg + warp_in_group) * 8 + (idx & 3)] = v[0][0];
        }
    }
#define VQC_PURE(T_)                                                                 \
    if constexpr (T_ < K)                                                            \
        if ((pm >> T_) & 1) {                                                        \
            const float* tp = op_table<float>(raw[T_], sh_tab, ps_tab);              \
            m1_entry<float, K, T_, true>(a, tp);                                     \
            m1_entry<float, K, T_, true>(l, tp);                                     \
        }
    VQC_PURE(0) VQC_PURE(1) VQC_PURE(2) VQC_PURE(3)
#undef VQC_PURE
}

// ---------------------------------------------------------------- factored stages
// double-float stages of runs: with every run as diag(p) rotation diag(q), a stage is
// one diagonal over the block's 2^K amplitudes (the product of its runs' q), K real
// rotations, one more diagonal (their p).  A rotation is 4 two-term dot products a
// pair (76 operations) where a 2x2 update is 4 four-term ones (172), and double-float
// is bound by the FP32 pipe: 16 qubits x 77 step 9.64 -> 7.82 ms (with the running rho
// sums of ddsum).  The diagonals are tabulated in shared memory, [stage][q, p][2^K].
template <typename R, int K>
__device__ __forceinline__ void build_diagonals(const FStage* stages, int nst, const uint2* ops, int op_base,
                                                const R* sh_tab, const R* ps_tab, bool per_sample, int t, int T,
                                                C2<R>* dg) {
    for (int i = t; i < (nst << (K + 1)); i += T) {
        const FStage* sp = stages + (i >> (K + 1));
        const int which = (i >> K) & 1, r = i & ((1 << K) - 1);
        if (!(sp->pure & (which ? kStageP : kStageQ)) || ((sp->pure & kStagePs) != 0) != per_sample) continue;
        const uint2* op = ops + (sp->op_begin - op_base);
        double2 f = make_double2(1, 0);
        for (int j = 0; j < K; ++j)
            if ((sp->pmask >> j) & 1) {
                const R* e = op_table<R>(*op++, sh_tab, ps_tab) + 10;
                const double2 ph = reinterpret_cast<const double2*>(e)[(which ? 0 : 2) + ((r >> j) & 1)];
                f = make_double2(fma(f.x, ph.x, -f.y * ph.y), fma(f.x, ph.y, f.y * ph.x));
            }
        dg[i] = cm<R>(R(f.x), R(f.y));
    }
}

template <typename R, int K, bool ADJ>
__device__ __forceinline__ void apply_diagonal(C2<R> (&a)[1 << K], const C2<R>* f) {
#pragma unroll
    for (int r = 0; r < (1 << K); ++r) a[r] = cmul<R>(a[r], ADJ ? cconj<R>(f[r]) : f[r]);
}

// [[C, -S], [S, C]] on local bit T (ADJ: its transpose).
template <typename R, int K, int T, bool ADJ>
__device__ __forceinline__ void rotate(C2<R> (&a)[1 << K], const R* e) {
    const R C = e[0], S = ADJ ? -e[1] : e[1], M = -S;
#pragma unroll
    for (int p = 0; p < (1 << (K - 1)); ++p) {
        const int i0 = pair_lo<T>(p), i1 = i0 | (1 << T);
        const C2<R> u = a[i0], v = a[i1];
        if constexpr (std::is_same<R, dd>::value) {
            a[i0] = cm<R>(dot2(C, u.x, M, v.x), dot2(C, u.y, M, v.y));
            a[i1] = cm<R>(dot2(S, u.x, C, v.x), dot2(S, u.y, C, v.y));
        } else {
            a[i0] = cm<R>(fma(C, u.x, M * v.x), fma(C, u.y, M * v.y));
            a[i1] = cm<R>(fma(S, u.x, C * v.x), fma(S, u.y, C * v.y));
        }
    }
}

template <typename R, int K>
__device__ __forceinline__ void factored_forward(const FStage* sp, const uint2* ops, C2<R> (&a)[1 << K],
                                                 const R* sh_tab, const R* ps_tab, const C2<R>* dg) {
    if (sp->pure & kStageQ) apply_diagonal<R, K, false>(a, dg);
    const unsigned pm = sp->pmask;
#define VQC_PURE(T_) \
    if constexpr (T_ < K) if ((pm >> T_) & 1) rotate<R, K, T_, false>(a, op_table<R>(*ops++, sh_tab, ps_tab) + 8);
    VQC_PURE(0) VQC_PURE(1) VQC_PURE(2) VQC_PURE(3) VQC_PURE(4)
#undef VQC_PURE
    if (sp->pure & kStageP) apply_diagonal<R, K, false>(a, dg + (1 << K));
}

// The adjoint, the runs' rho first as in pure_backward.
template <typename R, int K>
__device__ __forceinline__ void factored_backward(const FStage* sp, const uint2* ops, C2<R> (&a)[1 << K],
                                                  C2<R> (&l)[1 << K], const R* sh_tab, const R* ps_tab,
                                                  const C2<R>* dg, R* acc, int wg, int lane, int warp_in_group) {
    const unsigned pm = sp->pmask;
    unsigned am = 0;
    {
        const uint2* o = ops;
#pragma unroll
        for (int j = 0; j < K; ++j)
            if ((pm >> j) & 1) {
                if (((o->x) >> 24) & OPF_HAS_ACC) am |= 1u << j;
                ++o;
            }
    }
    if (am) {
        R v[K][3];
#pragma unroll
        for (int j = 0; j < K; ++j) v[j][0] = v[j][1] = v[j][2] = 0;
#define VQC_PURE(T_)                                     \
        if constexpr (T_ < K)                            \
            if ((am >> T_) & 1) {                        \
                R t[4] = {0, 0, 0, 0};                   \
                m1_t3<R, K, T_>(a, l, t);                \
                v[T_][0] = t[0];                         \
                v[T_][1] = t[1];                         \
                v[T_][2] = t[2];                         \
            }
        VQC_PURE(0) VQC_PURE(1) VQC_PURE(2) VQC_PURE(3)
#undef VQC_PURE
        const int idx = reduce_runs<R, K>(v, lane);
        const int j = idx >> 2;
        if (idx >= 0 && ((am >> j) & 1)) {
            const unsigned aux = ops[__popc(pm & ((1u << j) - 1u))].y >> 16;
            acc[((size_t)aux * wg + warp_in_group) * 8 + (idx & 3)] = v[0][0];
        }
    }
    if (sp->pure & kStageP) {
        apply_diagonal<R, K, true>(a, dg + (1 << K));
        apply_diagonal<R, K, true>(l, dg + (1 << K));
    }
#define VQC_PURE(T_)                                                             \
    if constexpr (T_ < K)                                                        \
        if ((pm >> T_) & 1) {                                                    \
            const R* e = op_table<R>(*ops++, sh_tab, ps_tab) + 8;                \
            rotate<R, K, T_, true>(a, e);                                        \
            rotate<R, K, T_, true>(l, e);                                        \
        }
    VQC_PURE(0) VQC_PURE(1) VQC_PURE(2) VQC_PURE(3)
#undef VQC_PURE
    if (sp->pure & kStageQ) {
        apply_diagonal<R, K, true>(a, dg);
        apply_diagonal<R, K, true>(l, dg);
    }
}

}  // namespace vqc
