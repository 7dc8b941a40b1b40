// pass.cuh -- HBM-tiled path for states that do not fit one SM's shared memory
// (paper, Sec. 3 "Complexity and Tradeoffs": the state, O(B 2^n), is the
// memory wall; here it lives in HBM between passes).
//
// One launch per pass of a frame schedule (frame.h): each CTA gathers S tiles of
// 2^m amplitudes, in whole 128-byte lines, into shared memory, runs the pass's
// register-block stages there and writes the tiles back, in the order that gives
// the next pass whole lines again.  The forward's last pass emits per-tile <Z>
// partials; the backward emits per-tile rho sums of the pass's accumulators,
// which reduce_terms adds up per sample and turns into gradient terms.  reduce_*
// kernels sum partials in a fixed order (deterministic).
#pragma once

#include "frame.cuh"

namespace vqc {

// R here is the storage real type (pass kernels take PArgs<St<R>>).
template <typename R>
struct PArgs {
    const DOp* ops;               // the pass's ops and stages
    const FStage* stages;
    const FSeg* segs;
    const FFlip* flips;           // [stages][nout]
    const FFinal* fin;            // last pass only (forward: <Z>; backward: lam = O psi)
    const int32_t* pass_entries;  // table slots of the pass's entries
    const int32_t* pass_accs;
    int n, m, tbits, G, S, nout, nstages, nops, op_begin, nsegs, seg_begin;
    int ps_begin, ps_count, sh_begin, sh_count, acc_begin, acc_count, n_accs;
    const void* ps_g;       // per-sample table entries [B][n_ps][entry words], kernel real type
    const void* sh_g;       // shared table entries [n_sh][entry words] (both from run_tables)
    int n_ps;
    int B;
    int nunits;
    uint32_t ga[kMaxTileBits], sa[kMaxTileBits];   // tile bit -> address, read and written order
    int32_t gs[kMaxTileBits], ss[kMaxTileBits];    // tile bit -> slot, read and written order
    uint32_t go[kMaxOuterBits], so[kMaxOuterBits]; // tile index bit -> address
    int32_t sosl[kMaxOuterBits];                   // tile index bit -> slot, written order
    const R* gE;
    const C2<R>* src_psi;   // tiles are read from here (nullptr: start from |0...0>)
    C2<R>* dst_psi;         // and written here (nullptr: not written)
    const C2<R>* src_lam;   // backward: lam tiles (nullptr: lam = O psi in the first stage)
    C2<R>* dst_lam;
    R* E_part;              // forward, last pass: [B * ntiles, n]
    R* rho;                 // backward: per-tile rho sums [B * ntiles][n_accs][4] (3 used)
    int sm_sh, sm_ps, sm_lam, sm_acc, sm_red;
    int sm_plan;            // copies of the pass's stages, ops, flips, rounds and fin
    int sm_tfl;             // per tile: each stage's flip (uint2), then the logical parities
    int sm_dg, ndg;         // the stages' diagonal tables (build_diagonals), per tile of the CTA
    int sm_tbase;           // each thread's block base in every stage: [nstages][threads]
    int sm_toff;            // tile-copy offsets of each thread: uint4
    int sm_koff;            // tile-copy offsets per vector round, read order then written order: uint2
    unsigned* err;          // the plan's error word (launch self-check)
    // double-float kernels only: src_psi / src_lam / dst_psi and dst_lam hold
    // raw (hi, lo) float pairs (workspace state passed between passes) rather
    // than complex128 values (caller buffers); ignored by other kernels
    int src_raw, lam_raw, dst_raw;
};

// 16-byte vectors of amplitudes, moved without taking register addresses.
template <typename R> struct Vec16;
template <> struct Vec16<float> {
    float2 a[2];
    __device__ __forceinline__ void ld(const float2* p) {
        const float4 v = __ldcs(reinterpret_cast<const float4*>(p));
        a[0] = make_float2(v.x, v.y);
        a[1] = make_float2(v.z, v.w);
    }
    __device__ __forceinline__ void st(float2* p) const {
        __stcs(reinterpret_cast<float4*>(p), make_float4(a[0].x, a[0].y, a[1].x, a[1].y));
    }
};
template <> struct Vec16<double> {
    double2 a[1];
    __device__ __forceinline__ void ld(const double2* p) { a[0] = __ldcs(p); }
    __device__ __forceinline__ void st(double2* p) const { __stcs(p, a[0]); }
};
// double-float kernels: complex128 in HBM, split on the way in, rejoined on the way out
template <> struct Vec16<dd> {
    dd2 a[1];
    __device__ __forceinline__ void ld(const double2* p) { a[0] = c2_in<dd>(__ldcs(p)); }
    __device__ __forceinline__ void st(double2* p) const { __stcs(p, c2_out<dd>(a[0])); }
};
// raw (hi, lo) pairs in a workspace buffer between double-float passes: no
// conversion (the conversions run on the FP64 units, a pass's slowest work)
struct Vec16Raw {
    dd2 a[1];
    __device__ __forceinline__ void ld(const double2* p) {
        const float4 v = __ldcs(reinterpret_cast<const float4*>(p));
        a[0].x = dd(v.x, v.y);
        a[0].y = dd(v.z, v.w);
    }
    __device__ __forceinline__ void st(double2* p) const {
        __stcs(reinterpret_cast<float4*>(p), make_float4(a[0].x.hi, a[0].x.lo, a[0].y.hi, a[0].y.lo));
    }
};
template <typename R, bool RAW> struct VecSel { using t = Vec16<R>; };
template <> struct VecSel<dd, true> { using t = Vec16Raw; };

// Tile copies between HBM and shared memory.  A CTA-thread t moves vectors
// v = t + k*T; address and slot of an amplitude are XOR-linear in its tile index,
// so each is a per-thread part XOR a per-k part (tabulated once per pass in
// shared memory: koff[k] = (address, slot)).  s1 is the slot offset of a
// vector's second amplitude.
template <typename R, bool RAW = false, int U = 8>
__device__ __forceinline__ void tile_gather(C2<R>* sm, const SC2<R>* gs, uint32_t gt, uint32_t st, uint32_t s1,
                                            const uint2* koff, int nk) {
    using V = typename VecSel<R, RAW>::t;
    constexpr int APV = 16 / sizeof(C2<R>);
    int k = 0;
    for (; k + U <= nk; k += U) {
        V v[U];
#pragma unroll
        for (int j = 0; j < U; ++j) v[j].ld(gs + (gt ^ koff[k + j].x));
#pragma unroll
        for (int j = 0; j < U; ++j) {
            const uint32_t sl = st ^ koff[k + j].y;
            sm[sl] = v[j].a[0];
            if constexpr (APV == 2) sm[sl ^ s1] = v[j].a[1];
        }
    }
    for (; k < nk; ++k) {
        V v;
        v.ld(gs + (gt ^ koff[k].x));
        const uint32_t sl = st ^ koff[k].y;
        sm[sl] = v.a[0];
        if constexpr (APV == 2) sm[sl ^ s1] = v.a[1];
    }
}

template <typename R, bool RAW = false>
__device__ __forceinline__ void tile_scatter(const C2<R>* sm, SC2<R>* gs, uint32_t gt, uint32_t st, uint32_t s1,
                                             const uint2* koff, int nk) {
    using V = typename VecSel<R, RAW>::t;
    constexpr int APV = 16 / sizeof(C2<R>);
    for (int k = 0; k < nk; ++k) {
        V v;
        const uint32_t sl = st ^ koff[k].y;
        v.a[0] = sm[sl];
        if constexpr (APV == 2) v.a[1] = sm[sl ^ s1];
        v.st(gs + (gt ^ koff[k].x));
    }
}

// Bring a tile's 128-byte lines into L2 ahead of its gather (a hint: no result,
// no wait).  With T >= 8 (every production tile) vectors t .. t+7 of one k
// share a line, so every eighth thread takes the lines; smaller groups touch
// some lines more than once.
template <typename R>
__device__ __forceinline__ void tile_prefetch(const SC2<R>* gs, uint32_t gt, const uint2* koff, int nk,
                                              int t) {
    if (t & 7) return;
    for (int k = 0; k < nk; ++k)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(gs + (gt ^ koff[k].x)));
}

// FULL: tile groups span whole warps (2^(m-K) >= 32 threads; every production
// tile), see sweep_kernel.
template <typename R, int K, int MODE, bool FULL, bool PH2 = true>
__global__ void __launch_bounds__(256, 2) pass_kernel(const __grid_constant__ PArgs<St<R>> A) {
    if (geometry_bad(blockDim.x != (unsigned)(A.S << A.tbits) || A.tbits != A.m - K || A.nstages < 1 ||
                         A.m > kMaxTileBits || A.nout > kMaxOuterBits,
                     A.err, kErrPassGeometry))
        return;
    extern __shared__ __align__(16) unsigned char smem[];
    R* sh_tab = reinterpret_cast<R*>(smem + A.sm_sh);
    R* ps_all = reinterpret_cast<R*>(smem + A.sm_ps);
    unsigned char* psi_t = smem;                // the CTA's S tiles first, so that a slot's byte
    unsigned char* lam_t = smem + A.sm_lam;     // offset is its address up to a constant
    R* acc_all = reinterpret_cast<R*>(smem + A.sm_acc);
    R* red_all = reinterpret_cast<R*>(smem + A.sm_red);
    const int nthr = blockDim.x, nst = A.nstages;

    // the pass's program (no kernel writes the plan, so this may precede the wait)
    FStage* stages = reinterpret_cast<FStage*>(smem + A.sm_plan);
    FFinal* fin = reinterpret_cast<FFinal*>(stages + nst);
    uint2* ops = reinterpret_cast<uint2*>(fin + 1);
    FFlip* flips = reinterpret_cast<FFlip*>(ops + A.nops);
    FSeg* segs = reinterpret_cast<FSeg*>(flips + nst * A.nout);
    async_region(reinterpret_cast<unsigned char*>(stages), reinterpret_cast<const unsigned char*>(A.stages),
                 nst * (int)sizeof(FStage));
    if (A.fin)
        async_region(reinterpret_cast<unsigned char*>(fin), reinterpret_cast<const unsigned char*>(A.fin),
                     sizeof(FFinal));
    for (int i = threadIdx.x; i < A.nops; i += nthr) async_elem<uint2>(ops + i, reinterpret_cast<const uint2*>(A.ops) + i);
    for (int i = threadIdx.x; i < A.nsegs * (int)(sizeof(FSeg) / 4); i += nthr)
        async_elem<int>(reinterpret_cast<int*>(segs) + i, reinterpret_cast<const int*>(A.segs) + i);
    for (int i = threadIdx.x; i < nst * A.nout; i += nthr)
        async_elem<uint2>(reinterpret_cast<uint2*>(flips) + i, reinterpret_cast<const uint2*>(A.flips) + i);

    const int n = A.n, G = A.G, tdim = 1 << A.m;
    const int total_tiles = A.B << A.nout;   // (at most states in memory over 64 amplitudes)
    const uint32_t tmask = (1u << A.nout) - 1u;
    constexpr bool DDK = !std::is_same<St<R>, R>::value;   // double-float kernel
    constexpr bool DG = sizeof(R) == 8;   // the stages may have diagonal tables
    Geo q;
    q.T = 1 << A.tbits;
    q.lanes = q.T < 32 ? q.T : 32;
    q.wg = q.T > 32 ? q.T / 32 : 1;
    q.g = threadIdx.x / q.T;
    q.t = threadIdx.x % q.T;
    q.h = 0;
    if (A.tbits < G) q.h = ((q.g & ((1 << (G - A.tbits)) - 1)) << A.tbits) & (tdim - 1);
    q.mask = blockDim.x >= 32 ? 0xffffffffu : ((1u << blockDim.x) - 1u);
    const int lane = q.t & 31;
    const int warp_in_group = q.t >> 5;

    // Tile copy geometry: vectors v = t + k*T of APV amplitudes.
    constexpr int APV = 16 / sizeof(C2<R>);
    const int nvec = tdim / APV;
    const int nk = (nvec + q.T - 1) / q.T;
    uint2* koff_g = reinterpret_cast<uint2*>(smem + A.sm_koff);
    uint2* koff_s = koff_g + nk;
    for (int k = threadIdx.x; k < nk; k += nthr) {
        const uint32_t u = (uint32_t)k * q.T * APV;
        koff_g[k] = make_uint2(xor_cols(A.ga, u), xor_cols(A.gs, u));
        koff_s[k] = make_uint2(xor_cols(A.sa, u), xor_cols(A.ss, u));
    }
    // each thread's own part, kept in shared memory: four registers across the stages
    uint4* toff = reinterpret_cast<uint4*>(smem + A.sm_toff) + threadIdx.x;
    {
        const uint32_t u = (uint32_t)q.t * APV;
        *toff = make_uint4(xor_cols(A.ga, u), xor_cols(A.gs, u) ^ (uint32_t)q.h, xor_cols(A.sa, u),
                           xor_cols(A.ss, u) ^ (uint32_t)q.h);
    }
    const uint32_t g_one = (uint32_t)A.gs[0], s_one = (uint32_t)A.ss[0];

    grid_dep_wait();
    grid_dep_launch();
    {   // the pass's shared entries
        constexpr int V = EntryWords<R>::value * (int)sizeof(R) / 16;   // 16-byte vectors per entry
        const unsigned char* gtab = static_cast<const unsigned char*>(A.sh_g);
        for (int i = threadIdx.x; i < A.sh_count * V; i += nthr) {
            const int k = i / V, v = i - k * V;
            async_copy<16>(reinterpret_cast<unsigned char*>(sh_tab) + 16 * i,
                           gtab + 16 * ((size_t)vqc_ld(&A.pass_entries[A.sh_begin + k]) * V + v));
        }
    }
    async_wait();
    __syncthreads();

    C2<R>* psi = reinterpret_cast<C2<R>*>(psi_t) + (size_t)q.g * tdim;
    C2<R>* lam = reinterpret_cast<C2<R>*>(lam_t) + (size_t)q.g * tdim;
    const uint32_t g0 = (uint32_t)(q.g * tdim) ^ (uint32_t)q.h;
    R* ps_tab = ps_all + (size_t)q.g * A.ps_count * EntryWords<R>::value;
    R* acc = acc_all + (size_t)q.g * A.acc_count * q.wg * 8;
    C2<R>* dg = reinterpret_cast<C2<R>*>(smem + A.sm_dg) + (((size_t)q.g * A.ndg) << K);
    if constexpr (FULL && DG) if (A.ndg)
        build_diagonals<R, K>(segs, A.nsegs, ops, A.op_begin, sh_tab, ps_tab, false, q.t, q.T, dg);
    uint2* tfl_all = reinterpret_cast<uint2*>(smem + A.sm_tfl);
    const uint2* tfl = tfl_all + q.g * (nst + 1);
    // each thread's block base in every stage (read by itself only)
    uint32_t* tbase = reinterpret_cast<uint32_t*>(smem + A.sm_tbase) + threadIdx.x;
    for (int s = 0; s < nst; ++s) tbase[s * nthr] = frame_base<R>(stages + s, q.t, g0);

    for (int unit = blockIdx.x; unit < A.nunits; unit += gridDim.x) {
        const int tid_raw = unit * A.S + q.g;
        const bool valid = tid_raw < total_tiles;
        const int tile_id = valid ? tid_raw : total_tiles - 1;
        const int b = tile_id >> A.nout;
        const uint32_t tau = (uint32_t)tile_id & tmask;

        // the tile's flip of each stage, and its logical parities
        for (int i = threadIdx.x; i < A.S * (nst + 1); i += nthr) {
            const int gg = i / (nst + 1), s = i - gg * (nst + 1);
            const uint32_t tt = (uint32_t)min(unit * A.S + gg, total_tiles - 1) & tmask;
            uint2 f = make_uint2(0, 0);
            if (s < nst) {
                for (int o = 0; o < A.nout; ++o)
                    if ((tt >> o) & 1) {
                        f.x ^= (uint32_t)flips[s * A.nout + o].slot * (uint32_t)sizeof(C2<R>);
                        f.y ^= flips[s * A.nout + o].mask;
                    }
            } else if (A.fin) {
                f.x = xor_cols(fin->omask, tt);
            }
            tfl_all[i] = f;
        }
        if (A.ps_count) {   // the pass's per-sample entries
            constexpr int V = EntryWords<R>::value * (int)sizeof(R) / 16;
            const int4* gtab = static_cast<const int4*>(A.ps_g);
            int4* stab = reinterpret_cast<int4*>(ps_all);
            const int per = A.ps_count * V;
            for (int i = threadIdx.x; i < A.S * per; i += nthr) {
                const int gg = i / per, r = i - gg * per, k = r / V, v = r - k * V;
                const int bb = min(unit * A.S + gg, total_tiles - 1) >> A.nout;
                stab[i] = gtab[((size_t)bb * A.n_ps + vqc_ld(&A.pass_entries[A.ps_begin + k])) * V + v];
            }
        }
        const size_t sbase = (size_t)b << n;
        const uint2 gto = *reinterpret_cast<const uint2*>(toff);
        const uint32_t ga = gto.x ^ xor_cols(A.go, tau), g_slot = gto.y;
        if (A.src_psi) {
            if (DDK && A.src_raw) tile_gather<R, DDK>(psi, A.src_psi + sbase, ga, g_slot, g_one, koff_g, nk);
            else   // 16 loads in flight where one state is gathered, 8 beside lam's registers
                tile_gather<R, false, MODE == 0 ? 16 : 8>(psi, A.src_psi + sbase, ga, g_slot, g_one, koff_g, nk);
        }
        if (MODE == 1 && A.src_lam) {
            if (DDK && A.lam_raw) tile_gather<R, DDK>(lam, A.src_lam + sbase, ga, g_slot, g_one, koff_g, nk);
            else tile_gather<R>(lam, A.src_lam + sbase, ga, g_slot, g_one, koff_g, nk);
        }
        if (unit + (int)gridDim.x < A.nunits) {   // the CTA's next tile into L2 during this one's stages
            const int nt = min((int)(unit + gridDim.x) * A.S + q.g, total_tiles - 1);
            const uint32_t nga = gto.x ^ xor_cols(A.go, (uint32_t)nt & tmask);
            const size_t nsb = (size_t)(nt >> A.nout) << n;
            if (A.src_psi) tile_prefetch<R>(A.src_psi + nsb, nga, koff_g, nk, q.t);
            if (MODE == 1 && A.src_lam) tile_prefetch<R>(A.src_lam + nsb, nga, koff_g, nk, q.t);
        }
        __syncthreads();
        if constexpr (FULL && DG) if (A.ndg && A.ps_count) {
            build_diagonals<R, K>(segs, A.nsegs, ops, A.op_begin, sh_tab, ps_tab, true, q.t, q.T, dg);
            __syncthreads();
        }

        C2<R> a[1 << K];
        uint32_t sb[K];
        FrameView v{0, 0};
        if constexpr (MODE == 0) {
            for (int s = 0; s < nst; ++s) {
                const FStage* sp = stages + s;
                const uint2 fl = tfl[s];
                v = frame_view<R, K>(sp, q.t, tbase[s * nthr], fl, sb);
                if (s == 0 && !A.src_psi) {
#pragma unroll
                    for (int r = 0; r < (1 << K); ++r) a[r] = cm<R>(0, 0);
                    if ((q.t | tau) == 0) a[0] = cm<R>(1, 0);
                } else {
                    frame_load<R, K>(a, psi_t, v.off, sb);
                }
                if constexpr (FULL)
                    stage_forward<R, K, PH2, EntryWords<R>::value>(sp, segs, A.seg_begin, ops, A.op_begin, v.pb, a,
                                                                        sh_tab, ps_tab, dg, q, lane, warp_in_group);
                else
                    run_ops<R, K, 0, FULL, PH2>(reinterpret_cast<const DOp*>(ops), sp->op_begin - A.op_begin,
                                                       sp->op_end - A.op_begin, v.pb, a, a, sh_tab, ps_tab, nullptr,
                                                       q, lane, warp_in_group);
                if (s + 1 < nst || A.dst_psi) {
                    frame_store<R, K>(a, psi_t, v.off, sb);
                    group_sync<R>(q);
                }
            }
            if (A.E_part) {
                R* red = red_all + (size_t)q.g * q.wg * n;
                const uint32_t pbf = tfl[nst].x ^ xor_bits(fin->tmask, A.tbits, q.t);
                expz_frame<R, K, FULL>(fin->lmask, pbf, a, n, q, lane,
                                       [&](int j, R e) { red[warp_in_group * n + j] = e; });
                __syncthreads();
                if (valid)
                    for (int j = q.t; j < n; j += q.T) {
                        R e = 0;
                        for (int k = 0; k < q.wg; ++k) e += red[k * n + j];
                        A.E_part[(size_t)tile_id * n + j] = as_out<St<R>>(e);
                    }
            }
            __syncthreads();
            if (A.dst_psi && valid) {
                const uint2 sto = *(reinterpret_cast<const uint2*>(toff) + 1);
                const uint32_t da = sto.x ^ xor_cols(A.so, tau), ds = sto.y ^ xor_cols(A.sosl, tau);
                if (DDK && A.dst_raw) tile_scatter<R, DDK>(psi, A.dst_psi + sbase, da, ds, s_one, koff_s, nk);
                else tile_scatter<R>(psi, A.dst_psi + sbase, da, ds, s_one, koff_s, nk);
            }
            __syncthreads();
        } else {
            // backward: stages of the pass in reverse
            for (int s = nst - 1; s >= 0; --s) {
                const FStage* sp = stages + s;
                const uint2 fl = tfl[s];
                C2<R> l[1 << K];
                v = frame_view<R, K>(sp, q.t, tbase[s * nthr], fl, sb);
                frame_load<R, K>(a, psi_t, v.off, sb);
                if (s == nst - 1 && !A.src_lam) {
                    const uint32_t pbf = tfl[nst].x ^ xor_bits(fin->tmask, A.tbits, q.t);
                    lambda_frame<R, K>(fin->lmask, pbf, A.gE + (size_t)b * n, n, a, l);
                } else {
                    frame_load<R, K>(l, lam_t, v.off, sb);
                }
                if constexpr (FULL)
                    stage_backward<R, K, PH2>(sp, segs, A.seg_begin, ops, A.op_begin, v.pb, a, l, sh_tab, ps_tab, dg,
                                              acc, q, lane, warp_in_group);
                else
                    run_ops<R, K, 1, FULL, PH2>(reinterpret_cast<const DOp*>(ops), sp->op_begin - A.op_begin,
                                                       sp->op_end - A.op_begin, v.pb, a, l, sh_tab, ps_tab, acc, q,
                                                       lane, warp_in_group);
                if (s > 0 || A.dst_psi) {
                    frame_store<R, K>(a, psi_t, v.off, sb);
                    frame_store<R, K>(l, lam_t, v.off, sb);
                }
                group_sync<R>(q);
            }
            __syncthreads();
            if (valid && A.dst_psi) {
                const uint2 sto = *(reinterpret_cast<const uint2*>(toff) + 1);
                const uint32_t da = sto.x ^ xor_cols(A.so, tau), s_slot = sto.y;
                if (DDK && A.dst_raw) {
                    tile_scatter<R, DDK>(psi, A.dst_psi + sbase, da, s_slot, s_one, koff_s, nk);
                    tile_scatter<R, DDK>(lam, A.dst_lam + sbase, da, s_slot, s_one, koff_s, nk);
                } else {
                    tile_scatter<R>(psi, A.dst_psi + sbase, da, s_slot, s_one, koff_s, nk);
                    tile_scatter<R>(lam, A.dst_lam + sbase, da, s_slot, s_one, koff_s, nk);
                }
            }
            // the tile's rho sums (warps in order), in parallel over accumulators and
            // components; the per-sample turn into terms is reduce_terms' work
            for (int i = threadIdx.x; i < A.S * A.acc_count * 3; i += nthr) {
                const int gg = i / (A.acc_count * 3), r = i % (A.acc_count * 3), k = r / 3, c = r % 3;
                const int tt = unit * A.S + gg;
                if (tt >= total_tiles) continue;
                const R* ap = acc_all + ((size_t)gg * A.acc_count + k) * q.wg * 8 + c;
                R sum = 0;
                for (int wi = 0; wi < q.wg; ++wi) sum += ap[wi * 8];
                A.rho[((size_t)tt * A.n_accs + vqc_ld(&A.pass_accs[A.acc_begin + k])) * 4 + c] = as_out<St<R>>(sum);
            }
            __syncthreads();
        }
    }
}

// E[b, j] = sum over tiles of E_part[b * ntiles + tau, j]  (fixed order).
template <typename R>
__global__ void reduce_expz(const R* E_part, int B, int ntiles, int n, R* E) {
    grid_dep_wait();
    grid_dep_launch();
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < (long long)B * n;
         i += (long long)gridDim.x * blockDim.x) {
        const long long b = i / n, j = i % n;
        R s = 0;
        for (int t = 0; t < ntiles; ++t) s += E_part[(b * ntiles + t) * n + j];
        E[i] = s;
    }
}

// Table entries, evaluated once per call for all passes, in the kernels' real
// type R: the shared ones to out_sh [n_sh][entry words], every sample's
// x-dependent ones to out_ps [B][n_ps][entry words] (slot order = list order).
template <typename R>
__global__ void __launch_bounds__(256) run_tables(const DEntry* entries, const int32_t* ps_list,
                                                  const int32_t* sh_list, const DConst* consts, const R* cang,
                                                  const R* cmat, const St<R>* x, int Px, const St<R>* w, int B,
                                                  int n_ps, int n_sh, const int32_t* ps_sel, const int32_t* sh_sel,
                                                  R* out_ps, R* out_sh) {
    grid_dep_wait();
    grid_dep_launch();
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < (long long)B * n_ps + n_sh;
         i += (long long)gridDim.x * blockDim.x) {
        if (i < n_sh) {
            const DEntry e = entries[vqc_ld(&sh_list[sh_sel ? vqc_ld(&sh_sel[i]) : i])];
            eval_entry<R>(e, consts, static_cast<const St<R>*>(nullptr), w, cang, cmat,
                          out_sh + (size_t)(sh_sel ? (int)i : e.slot) * EntryWords<R>::value);
            continue;
        }
        const long long j = i - n_sh, b = j / n_ps;
        const int k = (int)(j % n_ps);
        const DEntry e = entries[vqc_ld(&ps_list[ps_sel ? vqc_ld(&ps_sel[k]) : k])];
        eval_entry<R>(e, consts, x + b * Px, w, cang, cmat,
                      out_ps + ((size_t)b * n_ps + (ps_sel ? k : e.slot)) * EntryWords<R>::value);
    }
}

// Gradient terms of every accumulator of every sample: the sample's per-tile
// rho sums added in tile order, then the constituent walk of acc_terms (one
// partial), in the kernels' arithmetic R (the plan's constants are stored as R:
// (hi, lo) float pairs for double-float plans).  sel: the accumulators that rho holds
// (nullptr: all of them).  terms: [B, n_terms].
template <typename R>
__global__ void __launch_bounds__(256) reduce_terms(const St<R>* rho, int B, int ntiles, int n_accs,
                                                    const int32_t* sel, const DAcc* accs, const DEntry* entries,
                                                    const DConst* consts, const R* cang, const R* cmat,
                                                    const St<R>* x, int Px, const St<R>* w, int n_terms,
                                                    St<R>* terms) {
    grid_dep_wait();
    grid_dep_launch();
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < (long long)B * n_accs;
         i += (long long)gridDim.x * blockDim.x) {
        const long long b = i / n_accs;
        const int k = (int)(i % n_accs);
        R t[4] = {0, 0, 0, 0};
        for (int tau = 0; tau < ntiles; ++tau) {
            const St<R>* r = rho + ((b * ntiles + tau) * n_accs + k) * 4;
            t[0] += as_r<R>(r[0]);
            t[1] += as_r<R>(r[1]);
            t[2] += as_r<R>(r[2]);
        }
        const DAcc ac = accs[sel ? vqc_ld(&sel[k]) : k];
        acc_terms<R>(ac, entries[ac.entry], t, 1, consts,
                     x ? x + b * Px : static_cast<const St<R>*>(nullptr), w, cang, cmat, terms + b * n_terms);
    }
}

// dx[b, p] = sum over the terms of x column p, in order: the element i of dx.
template <typename R>
__device__ __forceinline__ void dx_element(const R* terms, long long i, int nt, const int32_t* ptr,
                                           const int32_t* occ, int Px, R* dx) {
    const R* row = terms + (i / Px) * nt;
    const int p = (int)(i % Px);
    R s = 0;
    for (int k = vqc_ld(&ptr[p]); k < vqc_ld(&ptr[p + 1]); ++k) s += row[vqc_ld(&occ[k])];
    dx[i] = s;
}

// dw[p] = sum over every row of the terms of w index p: one block per p, fixed
// strided partial sums then a fixed-shape tree.
template <typename R>
__device__ __forceinline__ void dw_column(const R* terms, long long rows, int nt, const int32_t* ptr,
                                          const int32_t* occ, int p, R* dw) {
    __shared__ R part[256];
    const int k0 = vqc_ld(&ptr[p]), k1 = vqc_ld(&ptr[p + 1]);
    R s = 0;
    for (long long r = threadIdx.x; r < rows; r += 256) {
        const R* row = terms + r * nt;
        for (int k = k0; k < k1; ++k) s += row[vqc_ld(&occ[k])];
    }
    part[threadIdx.x] = s;
    __syncthreads();
    for (int w = 128; w >= 1; w >>= 1) {
        if (threadIdx.x < w) part[threadIdx.x] += part[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) dw[p] = part[0];
}

template <typename R>
__global__ void reduce_dx(const R* terms, int B, int nt, const int32_t* ptr, const int32_t* occ, int Px, R* dx) {
    grid_dep_wait();
    grid_dep_launch();
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < (long long)B * Px;
         i += (long long)gridDim.x * blockDim.x)
        dx_element<R>(terms, i, nt, ptr, occ, Px, dx);
}

template <typename R>
__global__ void __launch_bounds__(256) reduce_dw(const R* terms, long long rows, int nt,
                                                 const int32_t* ptr, const int32_t* occ, R* dw) {
    grid_dep_wait();
    grid_dep_launch();
    dw_column<R>(terms, rows, nt, ptr, occ, blockIdx.x, dw);
}

// Both in one launch (complex64): the first Pw blocks take dw, the others dx.
template <typename R>
__global__ void __launch_bounds__(256) reduce_grads(const R* terms, int B, int nt, const int32_t* xptr,
                                                    const int32_t* xocc, int Px, R* dx, const int32_t* wptr,
                                                    const int32_t* wocc, int Pw, R* dw) {
    grid_dep_wait();
    grid_dep_launch();
    if ((int)blockIdx.x < Pw) {
        dw_column<R>(terms, B, nt, wptr, wocc, blockIdx.x, dw);
        return;
    }
    for (long long i = (blockIdx.x - Pw) * (long long)blockDim.x + threadIdx.x; i < (long long)B * Px;
         i += (long long)(gridDim.x - Pw) * blockDim.x)
        dx_element<R>(terms, i, nt, xptr, xocc, Px, dx);
}

// probs[i] = |psi[i]|^2 over count amplitudes (the probabilities output).
template <typename R>
__global__ void __launch_bounds__(256) abs2_kernel(const C2<R>* psi, long long count, R* probs) {
    grid_dep_wait();
    grid_dep_launch();
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < count;
         i += (long long)gridDim.x * blockDim.x) {
        const C2<R> v = psi[i];
        probs[i] = fma(v.x, v.x, v.y * v.y);
    }
}

}  // namespace vqc
