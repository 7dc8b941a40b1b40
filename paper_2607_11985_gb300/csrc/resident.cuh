// resident.cuh -- the resident sweep kernel: whole samples in shared memory, the
// stages of a frame schedule (frame.h) one after the other.
#pragma once

#include "frame.cuh"

namespace vqc {

// MODE 0: forward, MODE 1: backward.
// FULL: every sample group spans whole warps (2^(n-K) >= 32 threads), so warp
// reductions are fixed full-warp butterflies; the launch picks the variant.
// FUSED (MODE 1 only): the backward that recomputes the states also writes E
// (vqc_forward_backward); a separate instantiation keeps that code out of the
// plain backward kernel.
// PH2: the schedule may hold CRZ / RZZ.  Double-float: 2x2 updates throughout (else
// factored stages, in groups of whole warps).
// RND: stages in rounds, where the type has them, else the op switch throughout (the
// launch of a complex128 circuit with few phases a round or no room for their tables).
template <typename R, int K, int MODE, bool FULL, bool FUSED, bool PH2 = true, bool RND = true>
__global__ void __launch_bounds__(512) sweep_kernel(const __grid_constant__ KArgs<St<R>> A) {
    if (geometry_bad(blockDim.x != (unsigned)(A.S * A.tpg) || A.tpg != (1 << A.tbits) ||
                         A.tbits != A.n - K || A.n > kMaxTileBits || A.nstages < 1,
                     A.err, kErrSweepGeometry))
        return;
    extern __shared__ __align__(16) unsigned char smem[];
    R* sh_tab = reinterpret_cast<R*>(smem + A.sm_sh);
    R* ps_all = reinterpret_cast<R*>(smem + A.sm_ps);
    unsigned char* psi_t = smem;              // the CTA's S states first (see pass_kernel)
    unsigned char* lam_t = smem + A.sm_lam;
    R* acc_all = reinterpret_cast<R*>(smem + A.sm_acc);
    R* terms_all = reinterpret_cast<R*>(smem + A.sm_terms);
    R* dw_cta = reinterpret_cast<R*>(smem + A.sm_dw);
    R* red_all = reinterpret_cast<R*>(smem + A.sm_red);

    constexpr bool DF = std::is_same<R, dd>::value;
    constexpr bool ROUNDS = RND && FULL && (!DF || Factored<R, FULL, PH2>::value);
    constexpr bool DG = sizeof(R) == 8 && ROUNDS;   // the stages may have diagonal tables
    constexpr int EW = ResidentWords<R, MODE, FULL, PH2>::value;
    const int n = A.n, G = A.G;
    const int dim = 1 << n;
    Geo q;
    q.T = A.tpg;
    q.lanes = q.T < 32 ? q.T : 32;
    q.wg = q.T > 32 ? q.T / 32 : 1;
    q.g = threadIdx.x / q.T;
    q.t = threadIdx.x % q.T;
    q.h = 0;
    if (A.tbits < G) q.h = ((q.g & ((1 << (G - A.tbits)) - 1)) << A.tbits) & (dim - 1);
    q.mask = blockDim.x >= 32 ? 0xffffffffu : ((1u << blockDim.x) - 1u);
    const int lane = q.t & 31;
    const int warp_in_group = q.t >> 5;
    const int nthr = blockDim.x;

    R* w_sm = reinterpret_cast<R*>(smem + A.sm_w);
    R* xg_all = reinterpret_cast<R*>(smem + A.sm_xg);
    const int xgw = A.Px + n;   // row width of the x / gE staging area
    const uint32_t g0 = (uint32_t)(q.g * dim) ^ (uint32_t)q.h;   // first slot of the group's state, bank-spread
    C2<R>* psi = reinterpret_cast<C2<R>*>(psi_t);

    // initial (forward) or final (backward) state source; null: |0...0>
    const SC2<R>* src = MODE == 1 ? A.psi_final : A.psi0;
    if (MODE == 1 && !src) src = A.psi0;
    const bool from_global = src != nullptr;
    const bool final_order = MODE == 1 && A.psi_final != nullptr;   // amplitude order of src
    // slot of amplitude t + i T of a given state: a per-thread part XOR a per-i
    // part; the latter for the given and (forward) the returned states' order, 2^K each
    uint32_t* ioff = reinterpret_cast<uint32_t*>(smem + A.sm_io);
    for (int i = threadIdx.x; i < ((MODE == 0 ? 2 : 1) << K); i += blockDim.x) {
        const uint32_t u = (uint32_t)(i & ((1 << K) - 1)) << A.tbits;
        ioff[i] = (i >> K) || final_order ? xor_cols(A.sout, u) : xor_cols(A.sin, u);
    }
    auto state_slot0 = [&](bool fin_order) {
        return g0 ^ (fin_order ? xor_cols(A.sout, (uint32_t)q.t) : xor_cols(A.sin, (uint32_t)q.t));
    };

    // One unit's inputs to shared memory, asynchronously: x (and, backward,
    // gE) rows of its samples and each sample's initial / final state
    // (coalesced reads, swizzled slots).
    // (Double-float kernels copy the stored doubles as they are and split them
    // in place afterwards, unit_to_dd: both types are 8 bytes.)
    St<R>* xg_st = reinterpret_cast<St<R>*>(xg_all);
    SC2<R>* psi_st = reinterpret_cast<SC2<R>*>(psi);
    auto stage_unit = [&](int unit) {
        for (int i = threadIdx.x; i < A.S * xgw; i += nthr) {
            const int gg = i / xgw, c = i % xgw;
            const int bb = min(unit * A.S + gg, A.B - 1);
            if (c < A.Px) async_elem<St<R>>(xg_st + i, A.x + (size_t)bb * A.Px + c);
            else if (MODE == 1) async_elem<St<R>>(xg_st + i, A.gE + (size_t)bb * n + (c - A.Px));
        }
        if (from_global) {
            const int b = min(unit * A.S + q.g, A.B - 1);
            const SC2<R>* gs = src + (size_t)b * dim;
            const uint32_t s0 = state_slot0(final_order);
            for (int i = 0; i < (1 << K); ++i) async_elem<SC2<R>>(psi_st + (s0 ^ ioff[i]), gs + q.t + i * q.T);
        }
    };
    // after async_wait(): stored doubles -> dd in place, each by the thread that
    // issued its copy (its own copies are visible to it); a barrier follows
    auto unit_to_dd = [&]() {
        if constexpr (!std::is_same<St<R>, R>::value) {
            for (int i = threadIdx.x; i < A.S * xgw; i += nthr) {
                const int c = i % xgw;
                if (c < A.Px || MODE == 1) xg_all[i] = R(xg_st[i]);
            }
            if (from_global) {
                const uint32_t s0 = state_slot0(final_order);
                for (int i = 0; i < (1 << K); ++i) psi[s0 ^ ioff[i]] = c2_in<R>(psi_st[s0 ^ ioff[i]]);
            }
        }
    };

    // Prologue: the plan regions, w and the first unit's inputs all in flight
    // at once, one wait.
    const unsigned char* smt = nullptr;
    const unsigned char* sms = nullptr;
    if (A.plan_smem) {
        unsigned char* t = smem + A.sm_plan;
        unsigned char* u = t + (A.tab_smem ? (A.tab_bytes + 15) & ~15 : 0);
        if (A.tab_smem) async_region(t, A.plan + A.tab_off, A.tab_bytes);
        async_region(u, A.plan + A.sched_off, A.sched_bytes);
        smt = A.tab_smem ? t : nullptr;
        sms = u;
    }
    if (from_global) __syncthreads();   // ioff
    grid_dep_wait();
    grid_dep_launch();
    for (int i = threadIdx.x; i < A.Pw; i += nthr)
        async_elem<St<R>>(reinterpret_cast<St<R>*>(w_sm) + i, A.w + i);
    if ((int)blockIdx.x < A.nunits) stage_unit(blockIdx.x);
    if (MODE == 1)
        for (int i = threadIdx.x; i < A.Pw; i += nthr) dw_cta[i] = 0;
    PlanPtrs P;
    P.ops = rebase(A.ops, A.plan, A.sched_off, sms);
    const FStage* stages = rebase(A.fstages, A.plan, A.sched_off, sms);
    const FSeg* segs = rebase(A.segs, A.plan, A.sched_off, sms);
    const FFinal* fin = rebase(A.fin, A.plan, A.sched_off, sms);
    P.entries = rebase(A.entries, A.plan, A.tab_off, smt);
    P.ps_list = rebase(A.ps_list, A.plan, A.tab_off, smt);
    P.sh_list = rebase(A.sh_list, A.plan, A.tab_off, smt);
    P.consts = rebase(A.consts, A.plan, A.tab_off, smt);
    P.cmat = rebase(reinterpret_cast<const unsigned char*>(A.cmat), A.plan, A.tab_off, smt);
    P.cang = rebase(reinterpret_cast<const unsigned char*>(A.cang), A.plan, A.tab_off, smt);
    P.accs = rebase(A.accs, A.plan, A.tab_off, smt);
    P.xocc_ptr = rebase(A.xocc_ptr, A.plan, A.tab_off, smt);
    P.xocc = rebase(A.xocc, A.plan, A.tab_off, smt);
    P.wocc_ptr = rebase(A.wocc_ptr, A.plan, A.tab_off, smt);
    P.wocc = rebase(A.wocc, A.plan, A.tab_off, smt);
    const R* Pcmat = reinterpret_cast<const R*>(P.cmat);
    const R* Pcang = reinterpret_cast<const R*>(P.cang);
    async_wait();
    if constexpr (!std::is_same<St<R>, R>::value) {
        for (int i = threadIdx.x; i < A.Pw; i += nthr) w_sm[i] = R(reinterpret_cast<const St<R>*>(w_sm)[i]);
        if ((int)blockIdx.x < A.nunits) unit_to_dd();
    }
    __syncthreads();

    // shared table (w and constants) once per CTA, on the CTA's last threads
    // so that it runs beside the first unit's per-sample table
    for (int i = nthr - 1 - threadIdx.x; i < A.n_sh; i += nthr) {
        const int id = vqc_ld(&P.sh_list[i]);
        const DEntry e = P.entries[id];
        eval_entry<R, EW>(e, P.consts, static_cast<const R*>(nullptr), w_sm, Pcang, Pcmat,
                      sh_tab + EW * e.slot);
    }

    const uint2* ops = reinterpret_cast<const uint2*>(P.ops);
    R* ps_tab = ps_all + (size_t)q.g * A.n_ps * EW;
    R* acc = acc_all + (size_t)q.g * A.n_accs * q.wg * 8;
    R* terms = terms_all + (size_t)q.g * A.n_terms;

    for (int unit = blockIdx.x; unit < A.nunits; unit += gridDim.x) {
        const int b_raw = unit * A.S + q.g;
        const bool valid = b_raw < A.B;
        const int b = valid ? b_raw : A.B - 1;
        if (unit != (int)blockIdx.x) {
            stage_unit(unit);
            async_wait();
            if constexpr (!std::is_same<St<R>, R>::value) unit_to_dd();
            __syncthreads();
        }
        const R* xrow = xg_all + (size_t)q.g * xgw;

        // per-sample table (x-dependent runs): threads of the CTA over (sample, entry)
        for (int i = threadIdx.x; i < A.S * A.n_ps; i += nthr) {
            const int gg = i / A.n_ps, k = i % A.n_ps;
            const int id = vqc_ld(&P.ps_list[k]);
            const DEntry e = P.entries[id];
            eval_entry<R, EW>(e, P.consts, xg_all + (size_t)gg * xgw, w_sm, Pcang, Pcmat,
                          ps_all + ((size_t)gg * A.n_ps + e.slot) * EW);
        }
        __syncthreads();
        C2<R>* dg = reinterpret_cast<C2<R>*>(smem + A.sm_dg) + (((size_t)q.g * A.ndg) << K);
        if constexpr (DG) if (A.ndg) {
            if (unit == (int)blockIdx.x)
                build_diagonals<R, K, EW>(segs, A.nsegs, ops, 0, sh_tab, ps_tab, false, q.t, q.T, dg);
            build_diagonals<R, K, EW>(segs, A.nsegs, ops, 0, sh_tab, ps_tab, true, q.t, q.T, dg);
            __syncthreads();
        }

        C2<R> a[1 << K];
        uint32_t sb[K];
        const bool recompute = MODE == 1 && A.psi_final == nullptr;
        const int ns = A.nstages;

        // -------- forward sweep (forward mode, or backward recompute; the
        // recompute also writes E when the caller asks for it)
        R* red = red_all + (size_t)q.g * q.wg * n;
        const bool want_E = MODE == 0 || (FUSED && recompute && A.E != nullptr);
        if (MODE == 0 || recompute) {
            for (int s = 0; s < ns; ++s) {
                const FStage* sp = stages + s;
                const FrameView v = frame_view<R, K>(sp, q.t, frame_base<R>(sp, q.t, g0), make_uint2(0, 0), sb);
                if (s == 0 && !from_global) {
#pragma unroll
                    for (int r = 0; r < (1 << K); ++r) a[r] = cm<R>(0, 0);
                    if (q.t == 0) a[0] = cm<R>(1, 0);
                } else {
                    frame_load<R, K>(a, psi_t, v.off, sb);
                }
                if constexpr (ROUNDS)
                    stage_forward<R, K, PH2, EW>(sp, segs, 0, ops, 0, v.pb, a, sh_tab, ps_tab, dg, q, lane, warp_in_group);
                else
                    run_ops<R, K, 0, FULL, PH2, EW>(P.ops, sp->op_begin, sp->op_end, v.pb, a, a, sh_tab,
                                                           ps_tab, nullptr, q, lane, warp_in_group);
                if (s + 1 < ns || (MODE == 0 && A.state_out)) {
                    frame_store<R, K>(a, psi_t, v.off, sb);
                    group_sync<R>(q);
                }
            }
            if (want_E) {   // <Z_j> from the final blocks; a single-warp group writes E itself
                const uint32_t pbf = xor_bits(fin->tmask, A.tbits, q.t);
                expz_frame<R, K, FULL>(fin->lmask, pbf, a, n, q, lane, [&](int j, R e) {
                    if (FULL && q.wg == 1) {
                        if (valid) A.E[(size_t)b * n + j] = as_out<St<R>>(e);
                    } else {
                        red[warp_in_group * n + j] = e;
                    }
                });
            }
        }

        if (MODE == 0) {
            const bool direct = FULL && q.wg == 1;   // E already written
            if (!direct || A.state_out) {
                __syncthreads();
                if (valid) {
                    if (!direct) {
                        for (int j = q.t; j < n; j += q.T) {
                            R e = 0;
                            for (int k = 0; k < q.wg; ++k) e += red[k * n + j];
                            A.E[(size_t)b * n + j] = as_out<St<R>>(e);
                        }
                    }
                    if (A.state_out) {
                        SC2<R>* go = A.state_out + (size_t)b * dim;
                        const uint32_t s0 = state_slot0(true);
                        for (int i = 0; i < (1 << K); ++i)
                            go[q.t + i * q.T] = c2_out<R>(psi[s0 ^ ioff[i + (1 << K)]]);
                    }
                }
            }
            if (unit + (int)gridDim.x < A.nunits) __syncthreads();
            continue;
        }

        if (MODE == 1 && want_E && !(FULL && q.wg == 1)) {   // E of the recomputed states
            __syncthreads();
            if (valid)
                for (int j = q.t; j < n; j += q.T) {
                    R e = 0;
                    for (int k = 0; k < q.wg; ++k) e += red[k * n + j];
                    A.E[(size_t)b * n + j] = as_out<St<R>>(e);
                }
        }

        // -------- backward: reverse sweep with psi and lam
        if constexpr (MODE == 1) {
            for (int s = ns - 1; s >= 0; --s) {
                const FStage* sp = stages + s;
                const FrameView v = frame_view<R, K>(sp, q.t, frame_base<R>(sp, q.t, g0), make_uint2(0, 0), sb);
                C2<R> l[1 << K];
                if (s < ns - 1 || !recompute) frame_load<R, K>(a, psi_t, v.off, sb);
                if (s == ns - 1)
                    lambda_frame<R, K>(fin->lmask, xor_bits(fin->tmask, A.tbits, q.t), xrow + A.Px, n, a, l);
                else
                    frame_load<R, K>(l, lam_t, v.off, sb);
                if constexpr (ROUNDS)
                    stage_backward<R, K, PH2>(sp, segs, 0, ops, 0, v.pb, a, l, sh_tab, ps_tab, dg, acc, q, lane, warp_in_group);
                else
                    run_ops<R, K, 1, FULL, PH2, EW>(P.ops, sp->op_begin, sp->op_end, v.pb, a, l, sh_tab,
                                                           ps_tab, acc, q, lane, warp_in_group);
                if (s > 0) {
                    frame_store<R, K>(a, psi_t, v.off, sb);
                    frame_store<R, K>(l, lam_t, v.off, sb);
                }
                group_sync<R>(q);
            }
        }
        __syncthreads();

        // -------- gradient terms from the accumulated rho / scalars
        for (int i = threadIdx.x; i < A.S * A.n_accs; i += nthr) {
            const int gg = i / A.n_accs, k = i % A.n_accs;
            const DAcc ac = P.accs[k];
            acc_terms<R>(ac, P.entries[ac.entry], acc_all + ((size_t)gg * A.n_accs + k) * q.wg * 8,
                         q.wg, P.consts, xg_all + (size_t)gg * xgw, w_sm, Pcang, Pcmat,
                         terms_all + (size_t)gg * A.n_terms);
        }
        __syncthreads();
        // dx rows of this CTA's samples; dw partial of this CTA (fixed order)
        if (A.dx) {
            for (int i = threadIdx.x; i < A.S * A.Px; i += nthr) {
                const int gg = i / A.Px, p = i % A.Px;
                const int bb = unit * A.S + gg;
                if (bb >= A.B) continue;
                const R* tm = terms_all + (size_t)gg * A.n_terms;
                const int k0 = vqc_ld(&P.xocc_ptr[p]), k1 = vqc_ld(&P.xocc_ptr[p + 1]);
                R sum = 0;
                for (int k = k0; k < k1; ++k) sum += tm[vqc_ld(&P.xocc[k])];
                A.dx[(size_t)bb * A.Px + p] = as_out<St<R>>(sum);
            }
        }
        const int nvalid = min(A.S, A.B - unit * A.S);
        for (int p = threadIdx.x; p < A.Pw; p += nthr) {
            // samples in order, each sample's occurrences in order
            const int k0 = vqc_ld(&P.wocc_ptr[p]), k1 = vqc_ld(&P.wocc_ptr[p + 1]);
            R sum = dw_cta[p];
            if (k1 - k0 == 1) {   // the common case: independent loads
                const int j = vqc_ld(&P.wocc[k0]);
                for (int gg = 0; gg < nvalid; ++gg) sum += terms_all[(size_t)gg * A.n_terms + j];
            } else {
                for (int gg = 0; gg < nvalid; ++gg) {
                    const R* tm = terms_all + (size_t)gg * A.n_terms;
                    for (int k = k0; k < k1; ++k) sum += tm[vqc_ld(&P.wocc[k])];
                }
            }
            dw_cta[p] = sum;
        }
        __syncthreads();
    }

    if (MODE == 1 && A.Pw > 0 && A.dw) {
        // per-CTA partial of dw; reduce_cols sums the partials in CTA order
        for (int p = threadIdx.x; p < A.Pw; p += nthr)
            A.dw_part[(size_t)blockIdx.x * A.Pw + p] = as_out<St<R>>(dw_cta[p]);
    }
}

}  // namespace vqc
