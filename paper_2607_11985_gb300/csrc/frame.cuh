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

// ---------------------------------------------------------------- stages
// A stage is rounds of a group of diagonal ops and runs on distinct local positions
// (FSeg).  The runs are straight-line code over the positions, each under one uniform
// branch (against a descriptor load and a jump per op: complex64 16-qubit workload 7.61
// -> 7.24 ms).  complex128 kernels collect a group of diagonal ops per thread into one
// factor for the block and one pair of factors per local position that it touches;
// phases of two local positions, the same for every thread, go through a table in
// shared memory: a ring of RZZ then costs a few multiplications of the block instead of
// one per gate (16-qubit RZZ rings in native complex128 7.05 -> 6.52 ms, 16-qubit CZ
// rings in double-float 1.60 -> 1.44).  Two kinds of stages take the op switch instead:
// double-float ones with phases, whose collected factors round alike for a whole block
// (error of <Z> of a 15-qubit random circuit 4.4e-14 -> 6.3e-14; 2.07 -> 1.49 ms on
// 18-qubit RZZ rings, not kept; resident kernels of such circuits take 2x2 updates in
// every stage), and complex64 ones with diagonal ops, where a
// multiplication is cheap beside the walk over the group (scalar phases: 13-qubit random circuit 216
// us, 247 in rounds; 15-qubit RZZ rings 797 us against 835).  Native complex128 resident
// launches of circuits with few phases a round take it throughout (rounds_pay).
template <typename R, bool PH2>
__device__ __forceinline__ bool op_switch(unsigned kind) {
    return std::is_same<R, float>::value ? !(kind & kStagePure)
                                         : std::is_same<R, dd>::value && PH2 && (kind & kStagePhases);
}
template <typename R, int EW = EntryWords<R>::value>
__device__ __forceinline__ const R* op_table(uint2 raw, const R* sh_tab, const R* ps_tab) {
    return (((raw.x >> 24) & OPF_PER_SAMPLE) ? ps_tab : sh_tab) + EW * (raw.y & 0xffff);
}
__device__ __forceinline__ bool is_cz(unsigned code) { return code < DC_PH2_LL; }
// The diagonal op's class (frame.h): 0 both qubits outside, 1 + position, 10 both local.
__device__ __forceinline__ int diag_class(unsigned code) {
    if (code == DC_CZ_PP || code == DC_PH2_PP) return 0;
    if (code >= DC_CZ_PL && code < DC_CZ_PP) return 1 + (int)code - DC_CZ_PL;
    if (code >= DC_PH2_PL) return 1 + (int)code - DC_PH2_PL;
    return 10;
}

// The tables of a pass's rounds (dg: [table][2^K]): the product of a group's phases of
// two local positions (native), of the runs' own diagonals (double-float).  Products
// are taken in double: their rounding is the same for every amplitude.
template <typename R, int K, int EW = EntryWords<R>::value>
__device__ __forceinline__ void build_diagonals(const FSeg* segs, int nseg, const uint2* ops, int op_base,
                                                const R* sh_tab, const R* ps_tab, bool per_sample, int t, int T,
                                                C2<R>* dg) {
    constexpr bool DF = std::is_same<R, dd>::value;
    for (int i = t; i < (nseg << (K + 1)); i += T) {
        const FSeg* sp = segs + (i >> (K + 1));
        const int which = (i >> K) & 1, r = i & ((1 << K) - 1);
        const unsigned fl = sp->flags;
        const bool ll = !DF && which == 0 && (fl & kSegL), own = DF && (fl & (which ? kSegP : kSegQ));
        if (!(ll || own) || ((fl & kSegPs) != 0) != per_sample) continue;
        double fx = 1, fy = 0;
        auto times = [&](double x, double y) {
            const double nx = fma(fx, x, -fy * y), ny = fma(fx, y, fy * x);
            fx = nx;
            fy = ny;
        };
        const uint2* run = ops + (sp->run_begin - op_base);
        if constexpr (DF) {
            const uint2* op = run;
            for (int j = 0; own && j < K; ++j)
                if ((sp->pmask >> j) & 1) {
                    const R* e = op_table<R, EW>(*op++, sh_tab, ps_tab) + 10;
                    const double2 ph = reinterpret_cast<const double2*>(e)[(which ? 0 : 2) + ((r >> j) & 1)];
                    times(ph.x, ph.y);
                }
        }
        if (ll)   // the last ops of the group
            for (const uint2* o = run - 1; o >= ops + (sp->op_begin - op_base); --o) {
                const unsigned code = o->x & 0xff;
                if (code < DC_PH2_LL || code >= DC_PH2_PL) break;
                const int s = ((r >> ((o->x >> 8) & 0xff)) & 1) + 2 * ((r >> ((o->x >> 16) & 0xff)) & 1);
                const R* tp = op_table<R, EW>(*o, sh_tab, ps_tab) + 2 * s;
                if constexpr (!DF) times(tp[0], tp[1]);
            }
        dg[((size_t)sp->dg[which] << K) + r] = cm<R>(R(fx), R(fy));
    }
}

template <typename R, int K, bool ADJ>
__device__ __forceinline__ void apply_table(C2<R> (&a)[1 << K], const C2<R>* f) {
#pragma unroll
    for (int r = 0; r < (1 << K); ++r) a[r] = cmul<R>(a[r], ADJ ? cconj<R>(f[r]) : f[r]);
}
// Amplitudes with local bit L clear times f0, set times f1.
template <typename R, int K, int L>
__device__ __forceinline__ void apply_pair(C2<R> (&a)[1 << K], C2<R> f0, C2<R> f1) {
#pragma unroll
    for (int r = 0; r < (1 << K); ++r) a[r] = cmul<R>(a[r], ((r >> L) & 1) ? f1 : f0);
}
template <typename R, int K>
__device__ __forceinline__ void apply_pair_at(int L, C2<R> (&a)[1 << K], C2<R> f0, C2<R> f1) {
    switch (L) {
    case 0: apply_pair<R, K, 0>(a, f0, f1); break;
    case 1: if constexpr (K > 1) apply_pair<R, K, 1>(a, f0, f1); break;
    case 2: if constexpr (K > 2) apply_pair<R, K, 2>(a, f0, f1); break;
    case 3: if constexpr (K > 3) apply_pair<R, K, 3>(a, f0, f1); break;
    case 4: if constexpr (K > 4) apply_pair<R, K, 4>(a, f0, f1); break;
    default: break;
    }
}
template <typename R, int K>
__device__ __forceinline__ void flip_at(int L, C2<R> (&a)[1 << K], bool p) {   // z1_pred at a runtime position
    switch (L) {
    case 0: z1_pred<R, K, 0>(a, p); break;
    case 1: if constexpr (K > 1) z1_pred<R, K, 1>(a, p); break;
    case 2: if constexpr (K > 2) z1_pred<R, K, 2>(a, p); break;
    case 3: if constexpr (K > 3) z1_pred<R, K, 3>(a, p); break;
    case 4: if constexpr (K > 4) z1_pred<R, K, 4>(a, p); break;
    default: break;
    }
}
template <typename R, int K>
__device__ __forceinline__ void cz_local(unsigned code, C2<R> (&a)[1 << K]) {
    switch (code) {
#define VQC_CZLL(A_, B_) \
    case DC_CZ_LL + cz_pair_index(A_, B_): if constexpr (A_ < K && B_ < K) z2_ll<R, K, A_, B_>(a); break;
        VQC_CZLL(0, 1) VQC_CZLL(0, 2) VQC_CZLL(0, 3) VQC_CZLL(0, 4)
        VQC_CZLL(1, 2) VQC_CZLL(1, 3) VQC_CZLL(1, 4)
        VQC_CZLL(2, 3) VQC_CZLL(2, 4) VQC_CZLL(3, 4)
#undef VQC_CZLL
    default: break;
    }
}

// Apply the diagonal group ops [b, e) (ADJ: its inverse) to a and, with TWO, to l.
// table: the group's table, nullptr when it has none.
template <typename R, int K, bool ADJ, bool TWO, bool PH2, int EW>
__device__ __forceinline__ void apply_group(const uint2* b, const uint2* e, uint32_t pb, C2<R> (&a)[1 << K],
                                            C2<R> (&l)[1 << K], const R* sh_tab, const R* ps_tab,
                                            const C2<R>* table) {
    C2<R> g = cm<R>(1, 0);
    bool neg = false, ph = false;   // sign of the whole block, and whether g is more than 1
    auto phase = [&](uint2 raw, int s) {
        const R* tp = op_table<R, EW>(raw, sh_tab, ps_tab) + 2 * s;
        return cm<R>(tp[0], ADJ ? -tp[1] : tp[1]);
    };
    for (; b < e; ++b) {   // both qubits outside
        const uint2 raw = *b;
        const unsigned code = raw.x & 0xff;
        if (diag_class(code) != 0) break;
        const bool ba = physbit(pb, (raw.x >> 8) & 0xff), bb = physbit(pb, (raw.x >> 16) & 0xff);
        if (is_cz(code)) {
            neg ^= ba && bb;
        } else if constexpr (PH2) {
            g = cmul<R>(g, phase(raw, (int)ba + 2 * (int)bb));
            ph = true;
        }
    }
    while (b < e) {   // one local position at a time
        const int cls = diag_class(b->x & 0xff);
        if (cls == 10) break;
        C2<R> f0 = g, f1 = g;
        bool flip = false, any = ph;
        for (; b < e; ++b) {
            const uint2 raw = *b;
            const unsigned code = raw.x & 0xff;
            if (diag_class(code) != cls) break;
            const int ra = (raw.x >> 8) & 0xff, rb = (raw.x >> 16) & 0xff;
            const bool la = ra < kRefPhys, p = physbit(pb, la ? rb : ra);
            if (is_cz(code)) {
                flip ^= p;
            } else if constexpr (PH2) {
                f0 = cmul<R>(f0, phase(raw, la ? 2 * (int)p : (int)p));
                f1 = cmul<R>(f1, phase(raw, la ? 1 + 2 * (int)p : 2 + (int)p));
                any = true;
            }
        }
        if (PH2 && any) {
            if (neg) f0 = cm<R>(-f0.x, -f0.y);
            if (neg != flip) f1 = cm<R>(-f1.x, -f1.y);
            apply_pair_at<R, K>(cls - 1, a, f0, f1);
            if (TWO) apply_pair_at<R, K>(cls - 1, l, f0, f1);
            g = cm<R>(1, 0);
            ph = neg = false;
        } else {
            flip_at<R, K>(cls - 1, a, flip);
            if (TWO) flip_at<R, K>(cls - 1, l, flip);
        }
    }
    if (PH2 && ph) {
        if (neg) g = cm<R>(-g.x, -g.y);
#pragma unroll
        for (int r = 0; r < (1 << K); ++r) {
            a[r] = cmul<R>(a[r], g);
            if (TWO) l[r] = cmul<R>(l[r], g);
        }
    } else if (__any_sync(0xffffffffu, neg)) {
#pragma unroll
        for (int r = 0; r < (1 << K); ++r) {
            a[r] = negated<R>(a[r], neg);
            if (TWO) l[r] = negated<R>(l[r], neg);
        }
    }
    for (; b < e; ++b) {   // both local: CZ here, phases in the table
        const unsigned code = b->x & 0xff;
        if (!is_cz(code)) break;
        cz_local<R, K>(code, a);
        if (TWO) cz_local<R, K>(code, l);
    }
    if (table) {
        apply_table<R, K, ADJ>(a, table);
        if (TWO) apply_table<R, K, ADJ>(l, table);
    }
}

// Gradient terms Im <lam| G |psi> of a diagonal group's phases, G their generators,
// all from one Walsh transform of the block's Im(conj(lam) psi), which no diagonal op
// changes; eight ops at a time summed over the warp.
template <typename R, int K>
__device__ __forceinline__ void group_terms(const uint2* b, const uint2* e, uint32_t pb, const C2<R> (&a)[1 << K],
                                            const C2<R> (&l)[1 << K], R* acc, int wg, int lane, int warp_in_group) {
    R W[1 << K];
#pragma unroll
    for (int r = 0; r < (1 << K); ++r) W[r] = im_conj_mul<R>(l[r], a[r]);
    walsh<R, K>(W);
    for (; b < e; b += 8) {
        R v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            v[u] = 0;
            if (b + u < e) {
                const uint2 raw = b[u];
                const unsigned fl = raw.x >> 24;
                if (fl & OPF_HAS_ACC) {
                    const int ra = (raw.x >> 8) & 0xff, rb = (raw.x >> 16) & 0xff;
                    const unsigned ma = ra < kRefPhys ? 1u << ra : 0u, mb = rb < kRefPhys ? 1u << rb : 0u;
                    const bool na = ra >= kRefPhys && physbit(pb, ra), nb = rb >= kRefPhys && physbit(pb, rb);
                    const R ab = na != nb ? -W[ma ^ mb] : W[ma ^ mb];   // Z_a Z_b
                    if (fl & OPF_GEN_CRZ) v[u] = R(0.5f) * ((nb ? -W[mb] : W[mb]) - ab);   // |1><1|_a Z_b
                    else v[u] = ab;
                }
            }
        }
        const int u = warp_reduce_scatter<R, 8>(v, lane);
        if ((lane & 3) == 0 && b + u < e && ((b[u].x >> 24) & OPF_HAS_ACC))
            acc[((size_t)(b[u].y >> 16) * wg + warp_in_group) * 8] = v[0];
    }
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

// [[C, -S], [S, C]] of a double-float run (store_factors): 4 two-term dot products a
// pair (76 operations) where a 2x2 update is 4 four-term ones (172).  With its runs as
// diag(p) rotation diag(q), a stage is the product of the q, the rotations, the product
// of the p; double-float is bound by the FP32 pipe: 16 qubits x 77 step 9.64 -> 7.81 ms
// (with the running rho sums of ddsum).
template <typename R, int K, int T, bool ADJ>
__device__ __forceinline__ void rotate(C2<R> (&a)[1 << K], const R* e) {
    const R C = e[0], S = ADJ ? -e[1] : e[1], M = -S;
#pragma unroll
    for (int p = 0; p < (1 << (K - 1)); ++p) {
        const int i0 = pair_lo<T>(p), i1 = i0 | (1 << T);
        const C2<R> u = a[i0], v = a[i1];
        a[i0] = cm<R>(dot2(C, u.x, M, v.x), dot2(C, u.y, M, v.y));
        a[i1] = cm<R>(dot2(S, u.x, C, v.x), dot2(S, u.y, C, v.y));
    }
}

// The runs of a stage, forward.
template <typename R, int K, int EW>
__device__ __forceinline__ void forward_runs(const uint2* ops, unsigned pm, C2<R> (&a)[1 << K], const R* sh_tab,
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
#define VQC_RUN(T_)                                                                                 \
    if constexpr (T_ < K)                                                                           \
        if ((pm >> T_) & 1) {                                                                       \
            if constexpr (std::is_same<R, dd>::value) rotate<R, K, T_, false>(a, tp[T_] + 8);       \
            else m1_entry<R, K, T_, false>(a, tp[T_]);                                              \
        }
    VQC_RUN(0) VQC_RUN(1) VQC_RUN(2) VQC_RUN(3) VQC_RUN(4)
#undef VQC_RUN
}

// rho of a stage's runs.  They act on different local bits, so every run's (tx, ty, tz)
// can be taken where its last one's output is, and one butterfly sums all of them over
// the warp before the updates, whose registers it would otherwise hold (16-qubit
// step 6.90 -> 6.74 ms).  Packed forms of the sums (two components per FFMA2, the tz of
// all runs from one product per amplitude) execute fewer instructions but measured 2-3%
// slower.
template <typename R, int K>
__device__ __forceinline__ void run_terms(const uint2* ops, unsigned pm, const C2<R> (&a)[1 << K],
                                          const C2<R> (&l)[1 << K], R* acc, int wg, int lane, int warp_in_group) {
    unsigned am = 0;   // positions that accumulate
    {
        int o = 0;
#pragma unroll
        for (int j = 0; j < K; ++j) {
            const unsigned on = (pm >> j) & 1;
            am |= (on && ((ops[o].x >> 24) & OPF_HAS_ACC)) ? 1u << j : 0u;
            o += on;
        }
    }
    if (!am) return;
    R v[K][3];
#pragma unroll
    for (int j = 0; j < K; ++j) v[j][0] = v[j][1] = v[j][2] = 0;
#define VQC_RUN(T_)                              \
    if constexpr (T_ < K)                        \
        if ((am >> T_) & 1) {                    \
            R t[4] = {0, 0, 0, 0};               \
            m1_t3<R, K, T_>(a, l, t);            \
            v[T_][0] = t[0];                     \
            v[T_][1] = t[1];                     \
            v[T_][2] = t[2];                     \
        }
    VQC_RUN(0) VQC_RUN(1) VQC_RUN(2) VQC_RUN(3)
#undef VQC_RUN
    const int idx = reduce_runs<R, K>(v, lane);
    const int j = idx >> 2;
    if (idx >= 0 && ((am >> j) & 1)) {
        const unsigned aux = ops[__popc(pm & ((1u << j) - 1u))].y >> 16;
        acc[((size_t)aux * wg + warp_in_group) * 8 + (idx & 3)] = v[0][0];
    }
}

// The runs of a stage taken back on psi and lam.
template <typename R, int K>
__device__ __forceinline__ void backward_runs(const uint2* ops, unsigned pm, C2<R> (&a)[1 << K],
                                              C2<R> (&l)[1 << K], const R* sh_tab, const R* ps_tab) {
    const R* tp[K];
    {
        int o = 0;
#pragma unroll
        for (int j = 0; j < K; ++j) {
            tp[j] = op_table<R>(ops[o], sh_tab, ps_tab);
            o += (pm >> j) & 1;
        }
    }
#define VQC_RUN(T_)                                                     \
    if constexpr (T_ < K)                                               \
        if ((pm >> T_) & 1) {                                           \
            if constexpr (std::is_same<R, dd>::value) {                 \
                rotate<R, K, T_, true>(a, tp[T_] + 8);                  \
                rotate<R, K, T_, true>(l, tp[T_] + 8);                  \
            } else {                                                    \
                m1_back<R, K, T_>(a, l, tp[T_]);                        \
            }                                                           \
        }
    VQC_RUN(0) VQC_RUN(1) VQC_RUN(2) VQC_RUN(3)
#undef VQC_RUN
}

// Table k of a round (FSeg::dg), nullptr when the kernel's type has none.
template <typename R, int K>
__device__ __forceinline__ const C2<R>* seg_table(const FSeg* sp, int k, const C2<R>* dg) {
    constexpr bool df = std::is_same<R, dd>::value;
    return (sp->flags & (df ? (k ? kSegP : kSegQ) : k ? 0 : kSegL)) ? dg + ((size_t)sp->dg[k] << K) : nullptr;
}

// A stage's rounds on its block; ops: the schedule's op op_base and seg: its round
// seg_base, in shared memory.
template <typename R, int K, bool PH2, int EW>
__device__ __forceinline__ void stage_forward(const FStage* st, const FSeg* segs, int seg_base, const uint2* ops,
                                              int op_base, uint32_t pb, C2<R> (&a)[1 << K], const R* sh_tab,
                                              const R* ps_tab, const C2<R>* dg, const Geo& q, int lane,
                                              int warp_in_group) {
    constexpr bool PHASES = PH2 && std::is_same<R, double>::value;
    constexpr bool DG = sizeof(R) == 8;
    if (op_switch<R, PH2>(st->kind)) {
        run_ops<R, K, 0, true, PH2, EW>(reinterpret_cast<const DOp*>(ops), st->op_begin - op_base,
                                               st->op_end - op_base, pb, a, a, sh_tab, ps_tab, nullptr, q, lane,
                                               warp_in_group);
        return;
    }
    if constexpr (std::is_same<R, float>::value) {
        forward_runs<R, K, EW>(ops + (st->op_begin - op_base), st->pmask, a, sh_tab, ps_tab);
        return;
    }
    for (int i = st->seg_begin; i < st->seg_end; ++i) {
        const FSeg* sp = segs + (i - seg_base);
        const uint2 *b = ops + (sp->op_begin - op_base), *r = ops + (sp->run_begin - op_base);
        const C2<R>* t = DG ? seg_table<R, K>(sp, 0, dg) : nullptr;
        if (b < r || t) apply_group<R, K, false, false, PHASES, EW>(b, r, pb, a, a, sh_tab, ps_tab, t);
        forward_runs<R, K, EW>(r, sp->pmask, a, sh_tab, ps_tab);
        if constexpr (std::is_same<R, dd>::value)
            if (const C2<R>* t1 = seg_table<R, K>(sp, 1, dg)) apply_table<R, K, false>(a, t1);
    }
}

template <typename R, int K, bool PH2>
__device__ __forceinline__ void stage_backward(const FStage* st, const FSeg* segs, int seg_base, const uint2* ops,
                                               int op_base, uint32_t pb, C2<R> (&a)[1 << K], C2<R> (&l)[1 << K],
                                               const R* sh_tab, const R* ps_tab, const C2<R>* dg, R* acc,
                                               const Geo& q, int lane, int warp_in_group) {
    constexpr int EW = EntryWords<R>::value;
    constexpr bool PHASES = PH2 && std::is_same<R, double>::value;
    constexpr bool DG = sizeof(R) == 8;
    const int wg = q.wg;
    if (op_switch<R, PH2>(st->kind)) {
        run_ops<R, K, 1, true, PH2, EW>(reinterpret_cast<const DOp*>(ops), st->op_begin - op_base,
                                               st->op_end - op_base, pb, a, l, sh_tab, ps_tab, acc, q, lane,
                                               warp_in_group);
        return;
    }
    if constexpr (std::is_same<R, float>::value) {
        const uint2* r = ops + (st->op_begin - op_base);
        run_terms<R, K>(r, st->pmask, a, l, acc, wg, lane, warp_in_group);
        backward_runs<R, K>(r, st->pmask, a, l, sh_tab, ps_tab);
        return;
    }
    for (int i = st->seg_end - 1; i >= st->seg_begin; --i) {
        const FSeg* sp = segs + (i - seg_base);
        const uint2 *b = ops + (sp->op_begin - op_base), *r = ops + (sp->run_begin - op_base);
        if (sp->pmask) {
            run_terms<R, K>(r, sp->pmask, a, l, acc, wg, lane, warp_in_group);
            if constexpr (std::is_same<R, dd>::value)
                if (const C2<R>* t1 = seg_table<R, K>(sp, 1, dg)) {
                    apply_table<R, K, true>(a, t1);
                    apply_table<R, K, true>(l, t1);
                }
            backward_runs<R, K>(r, sp->pmask, a, l, sh_tab, ps_tab);
        }
        if (PHASES && (sp->flags & kSegA)) group_terms<R, K>(b, r, pb, a, l, acc, wg, lane, warp_in_group);
        const C2<R>* t = DG ? seg_table<R, K>(sp, 0, dg) : nullptr;
        if (b < r || t) apply_group<R, K, true, true, PHASES, EW>(b, r, pb, a, l, sh_tab, ps_tab, t);
    }
}

}  // namespace vqc
