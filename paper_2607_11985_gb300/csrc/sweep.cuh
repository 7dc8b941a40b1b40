// sweep.cuh -- sm_103a kernels of the batched statevector engine.
//
// Forward (paper, Alg. 1 execute phase): per sample, psi = U_G ... U_1 psi0
// and E[b, j] = sum_k (-1)^{k_j} |psi[k]|^2 (Alg. 1, return statement).
// Backward (paper, Sec. 3, gradients w.r.t. trainable parameters), adjoint
// method: lam = O psi with O = sum_j gE[b, j] Z_j; the plan is swept in
// reverse, un-applying every op on psi and lam, and for every parametrised
// angle t of a gate exp(-i t P / 2) the term dL/dt = Im <lam|P|psi> is taken
// at the gate's output.  For a fused single-qubit run V the kernel
// accumulates rho = sum_pairs psi_pair lam_pair^dag (a 2x2 matrix) once at
// the run's output; each constituent j of the run then gives
// dL/dt_j = Im Tr(W_j P_j W_j^dag rho) with W_j the constituents after j.
//
// Execution model ("resident" path).  A sample's state lives in shared
// memory.  A group of T = 2^(n-K) threads owns one sample; in each stage a
// thread loads the 2^K amplitudes spanned by the stage's K directions (frame.h)
// into registers (its block; the other n-K index bits come from the thread index),
// applies all of the stage's ops there, and stores the block back.  Blocks of
// different threads are disjoint, so one group barrier per stage suffices.
// Gate matrices are evaluated once per sample (sincos once per angle) into a
// shared-memory table before the sweep.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "dd.cuh"
#include "frame.h"
#include "plan.h"

namespace vqc {

template <typename R> struct V2;
template <> struct V2<float> { using t = float2; };
template <> struct V2<double> { using t = double2; };
template <> struct V2<dd> { using t = dd2; };
template <typename R> using C2 = typename V2<R>::t;

// The real type arrays have outside a kernel (caller memory, workspaces,
// partials) for the kernel's arithmetic type R: R itself, except double for
// double-float kernels, which split values on reading and rejoin them on
// writing.  For float and double every conversion below is the identity.
template <typename R> struct StoreOf { using t = R; };
template <> struct StoreOf<dd> { using t = double; };
template <typename R> using St = typename StoreOf<R>::t;
template <typename R> using SC2 = C2<St<R>>;

template <typename R, typename T>
__device__ __forceinline__ R as_r(T v) {
    if constexpr (std::is_same<T, R>::value) return v;
    else return R(v);
}
template <typename O, typename R>
__device__ __forceinline__ O as_out(R v) {
    if constexpr (std::is_same<O, R>::value) return v;
    else return v.to_double();
}
template <typename R>
__device__ __forceinline__ C2<R> c2_in(SC2<R> v) {
    if constexpr (std::is_same<St<R>, R>::value) return v;
    else { C2<R> r; r.x = R(v.x); r.y = R(v.y); return r; }
}
template <typename R>
__device__ __forceinline__ SC2<R> c2_out(C2<R> v) {
    if constexpr (std::is_same<St<R>, R>::value) return v;
    else { SC2<R> r; r.x = v.x.to_double(); r.y = v.y.to_double(); return r; }
}

template <typename R>
__device__ __forceinline__ C2<R> cm(R x, R y) { C2<R> r; r.x = x; r.y = y; return r; }

template <typename R>
__device__ __forceinline__ C2<R> cmul(C2<R> a, C2<R> b) {
    if constexpr (std::is_same<R, dd>::value)
        return cm<R>(dot2(a.x, b.x, -a.y, b.y), dot2(a.x, b.y, a.y, b.x));
    else
        return cm<R>(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}
// m0 * u + m1 * v
template <typename R>
__device__ __forceinline__ C2<R> cmv2(C2<R> m0, C2<R> u, C2<R> m1, C2<R> v) {
    if constexpr (std::is_same<R, dd>::value) {   // each component one compensated dot product
        C2<R> r;
        r.x = dot4(m0.x, u.x, -m0.y, u.y, m1.x, v.x, -m1.y, v.y);
        r.y = dot4(m0.x, u.y, m0.y, u.x, m1.x, v.y, m1.y, v.x);
        return r;
    }
    R x = fma(m0.x, u.x, fma(-m0.y, u.y, fma(m1.x, v.x, -m1.y * v.y)));
    R y = fma(m0.x, u.y, fma(m0.y, u.x, fma(m1.x, v.y, m1.y * v.x)));
    return cm<R>(x, y);
}
template <typename R>
__device__ __forceinline__ C2<R> cconj(C2<R> a) { return cm<R>(a.x, -a.y); }

template <typename R> struct M2 { C2<R> a, b, c, d; };   // [[a, b], [c, d]]

template <typename R>
__device__ __forceinline__ M2<R> mmul(const M2<R>& p, const M2<R>& q) {   // p * q
    M2<R> r;
    r.a = cmv2<R>(p.a, q.a, p.b, q.c);
    r.b = cmv2<R>(p.a, q.b, p.b, q.d);
    r.c = cmv2<R>(p.c, q.a, p.d, q.c);
    r.d = cmv2<R>(p.c, q.b, p.d, q.d);
    return r;
}
template <typename R>
__device__ __forceinline__ M2<R> mdag(const M2<R>& p) {
    M2<R> r;
    r.a = cconj<R>(p.a); r.b = cconj<R>(p.c); r.c = cconj<R>(p.b); r.d = cconj<R>(p.d);
    return r;
}
template <typename R>
__device__ __forceinline__ M2<R> mident() {
    M2<R> r;
    r.a = cm<R>(1, 0); r.b = cm<R>(0, 0); r.c = cm<R>(0, 0); r.d = cm<R>(1, 0);
    return r;
}

// Plain load: plan arrays may live in shared memory (copied at kernel start)
// or, when too large, in global memory.
template <typename T>
__device__ __forceinline__ T vqc_ld(const T* p) { return *p; }

// Asynchronous global -> shared copies (cp.async, 4/8/16 bytes, both addresses
// aligned to the size).  They hold no registers while in flight, so a thread
// can issue all of a CTA's staging loads before the first wait; async_wait()
// then blocks until this thread's copies have landed (a __syncthreads must
// follow before other threads read them).
template <int BYTES>
__device__ __forceinline__ void async_copy(void* sdst, const void* gsrc) {
    const unsigned sa = static_cast<unsigned>(__cvta_generic_to_shared(sdst));
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(sa), "l"(gsrc), "n"(BYTES)
                 : "memory");
}
__device__ __forceinline__ void async_wait() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

__device__ __forceinline__ void async_region(unsigned char* dst, const unsigned char* src, int bytes) {
    for (int i = threadIdx.x; i < bytes / 16; i += blockDim.x) async_copy<16>(dst + 16 * i, src + 16 * i);
}
template <typename T>
__device__ __forceinline__ void async_elem(T* sdst, const T* gsrc) {
    async_copy<sizeof(T)>(sdst, gsrc);
}

// Programmatic dependent launch.  Every kernel of the library is launched so
// that it may start while the previous kernel in the stream is finishing; it
// reads and writes no caller memory (inputs, outputs, workspace) before
// grid_dep_wait(), which returns once that kernel has completed and its writes
// are visible (immediately when the launch had no such predecessor).  Only the
// plan, which no kernel writes, is read before it.  grid_dep_launch() then lets
// the next kernel in the stream begin its own prologue.
__device__ __forceinline__ void grid_dep_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
__device__ __forceinline__ void grid_dep_launch() {
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
}

// Pointer into the shared copy of a plan region (or the global one).
template <typename T>
__device__ __forceinline__ const T* rebase(const T* g, const unsigned char* plan, int region_off,
                                           const unsigned char* sm_region) {
    if (!sm_region) return g;
    return reinterpret_cast<const T*>(sm_region +
                                      (reinterpret_cast<const unsigned char*>(g) - plan - region_off));
}

// sin and cos for complex64 table entries, written out so that the half-angle
// evaluation is a short chain of FMAs: Cody-Waite reduction t = k pi/2 + r
// with pi/2 split in three parts (the head has 8 significant bits, so k *
// head is exact for |k| < 2^16), |r| <= pi/4, then the Taylor polynomials of
// sin (through r^9) and cos (through r^10), whose truncation errors on
// [-pi/4, pi/4] are below 2e-9, and the quadrant of k.  The reduction is exact
// only while |k| < 2^16; arguments beyond |t| = 65536 (|k| <= 41722), and NaN,
// go to the library sincosf instead.  complex128 uses the library routine.
__device__ __forceinline__ void sc(float t, float* s, float* c) {
    if (!(fabsf(t) <= 65536.0f)) {
        sincosf(t, s, c);
        return;
    }
    const float k = rintf(t * 0.636619772367581343f);   // t / (pi/2)
    float r = fmaf(-k, 1.5703125f, t);
    r = fmaf(-k, 4.838267923332751e-4f, r);
    r = fmaf(-k, 2.5633440682570896e-12f, r);
    const float r2 = r * r;
    float ps = fmaf(r2, 2.75573192239858907e-6f, -1.98412698412698413e-4f);   // 1/9!, -1/7!
    ps = fmaf(r2, ps, 8.33333333333333333e-3f);                               // 1/5!
    ps = fmaf(r2, ps, -1.66666666666666667e-1f);                              // -1/3!
    const float sr = fmaf(r * r2, ps, r);
    float pc = fmaf(r2, -2.75573192239858907e-7f, 2.48015873015873016e-5f);   // -1/10!, 1/8!
    pc = fmaf(r2, pc, -1.38888888888888889e-3f);                              // -1/6!
    pc = fmaf(r2, pc, 4.16666666666666667e-2f);                               // 1/4!
    pc = fmaf(r2, pc, -0.5f);                                                 // -1/2!
    const float cr = fmaf(r2, pc, 1.0f);
    const int q = (int)k & 3;
    const float sv = (q & 1) ? cr : sr, cv = (q & 1) ? sr : cr;
    *s = (q & 2) ? -sv : sv;
    *c = ((q + 1) & 2) ? -cv : cv;
}
__device__ __forceinline__ void sc(double t, double* s, double* c) { sincos(t, s, c); }
// double-float: the library routine in double (once per angle), then split
__device__ __forceinline__ void sc(dd t, dd* s, dd* c) {
    double sd, cd;
    sincos(t.to_double(), &sd, &cd);
    *s = dd(sd);
    *c = dd(cd);
}

// ---------------------------------------------------------------- kernel args
// R here is the storage real type (kernels take KArgs<St<R>>).
template <typename R>
struct KArgs {
    // plan
    const DOp* ops;
    const DStage* stages;
    int nstages;
    const DEntry* entries;
    const int32_t* ps_list;   // per-sample entry ids
    const int32_t* sh_list;   // shared entry ids
    const DConst* consts;
    const R* cmat;
    const R* cang;
    const DAcc* accs;
    const int32_t* xocc_ptr;
    const int32_t* xocc;
    const int32_t* wocc_ptr;
    const int32_t* wocc;
    unsigned* err;
    int n, K, tbits, G, S;     // S = samples per CTA
    int tpg;                   // threads per sample group (2^tbits)
    int n_ps, n_sh, n_accs, n_terms, Px, Pw;
    // batch
    int B, nunits;
    const R* x;
    const R* w;
    const C2<R>* psi0;
    const C2<R>* psi_final;
    const R* gE;
    R* E;
    C2<R>* state_out;
    R* dx;
    R* dw;
    R* dw_part;          // [gridDim.x, Pw]
    // shared-memory carve-up (byte offsets)
    int sm_sh, sm_ps, sm_psi, sm_lam, sm_acc, sm_terms, sm_dw, sm_red;
    int sm_w, sm_xg;   // shared copies of w [Pw] and of the unit's x / gE rows [S][Px + n]
    // plan regions copied to shared memory at sm_plan when plan_smem is set:
    // table data [tab_off, tab_off + tab_bytes) and this schedule's
    // [sched_off, sched_off + sched_bytes) of the plan's device blob.
    const unsigned char* plan;
    // (tab_smem 0: the table data is read where it lies, which leaves room for more CTAs)
    int tab_off, tab_bytes, sched_off, sched_bytes, sm_plan, plan_smem, tab_smem;
    // resident path (resident.cuh): the frame schedule, and the slots of the state's
    // bits in the order of a given state (sin) and of the final one (sout)
    const FStage* fstages;
    const FSeg* segs;
    const FFinal* fin;
    int32_t sin[kMaxTileBits], sout[kMaxTileBits];
    int sm_io, sm_dg, ndg, nsegs;
    // cluster path only (cluster.cuh): log2 CTAs per sample, rank 0's <Z> gather area
    int cl, sm_ecl;
};

struct PlanPtrs {
    const DOp* ops;
    const DStage* stages;
    const DEntry* entries;
    const int32_t* ps_list;
    const int32_t* sh_list;
    const DConst* consts;
    const void* cmat;
    const void* cang;
    const DAcc* accs;
    const int32_t* xocc_ptr;
    const int32_t* xocc;
    const int32_t* wocc_ptr;
    const int32_t* wocc;
};

// ---------------------------------------------------------------- tables
// Reals per table entry.  complex64 stores each 2x2 run matrix U twice in the
// operand form of the packed-FP32 update (see m1_apply_f2w): U at [0, 16) and
// U^dag at [16, 32), each as the pairs (m, i m) = (Re m, Im m), (-Im m, Re m) of
// its four entries m.
// complex128 stores U (8 reals), double-float also its factors (store_factors).  Phase
// entries use the first 8 reals.
template <typename R> struct EntryWords {
    static constexpr int value = entry_reals(sizeof(R) == 8, std::is_same<R, dd>::value);
};

// A double-float run's factors at offset 8 of its entry: C, S, then p0, p1, q0, q1 as
// doubles, with U = diag(p0, p1) [[C, -S], [S, C]] diag(q0, q1).  Stages of runs apply
// the real rotations one by one and the diagonals of all of them at once (frame.cuh).
// Each phase comes from the larger of two entries, so a vanishing one costs no
// accuracy; the phases stay doubles until the stage's products of them are split, so
// that their roundings, the same for every amplitude, are not double-float's.
// (Native complex128 keeps the 2x2 updates: factors rounded to double doubled its
// gradients' error against 64 bits, 3.2e-15 -> 6.4e-15 at 16 qubits.)
constexpr double kTiny = 1e-36;   // squared moduli below this count as 0: their phase is never seen

// 1 / sqrt(x) for x in [kTiny, 4]: a float start and two Newton steps, y (3 - x y^2) / 2
// (relative error 2^-22 -> 2^-43 -> double); the FP64 pipe is slow and the library's
// square root and divisions took longer than the rest of an entry.
__device__ __forceinline__ double inv_sqrt(double x) {
    if (!(x > kTiny)) return x != x ? x : 0.0;
    double y = (double)rsqrtf((float)x);
    const double h = 0.5 * x;
    y = fma(y, fma(-h * y, y, 0.5), y);
    return fma(y, fma(-h * y, y, 0.5), y);
}

template <typename R>
__device__ __forceinline__ void store_factors(const M2<R>& m, int form, R* o) {
    if constexpr (std::is_same<R, dd>::value) {
        auto d2 = [](C2<R> v) { const SC2<R> w = c2_out<R>(v); return make_double2(w.x, w.y); };
        auto scale = [](double2 v, double f) { return make_double2(v.x * f, v.y * f); };
        auto mulc = [](double2 x, double2 y) {   // x conj(y)
            return make_double2(fma(x.x, y.x, x.y * y.y), fma(x.y, y.x, -x.x * y.y));
        };
        const double2 a = d2(m.a), b = d2(m.b), c = d2(m.c), d = d2(m.d), one = make_double2(1, 0);
        double2 p0 = one, p1 = one, q0 = one, q1 = one;
        double C = a.x, S = c.x;
        if (form != 0) {
            const double a2 = fma(a.x, a.x, a.y * a.y), c2 = fma(c.x, c.x, c.y * c.y);
            const double ra = inv_sqrt(a2), rc = inv_sqrt(c2);   // 1 / |a|, 1 / |c|
            const bool big = a2 >= c2;
            C = a2 * ra;
            S = c2 * rc;
            if (form == 3) {   // q0 = 1
                if (a2 > kTiny || !(c2 > kTiny)) p0 = scale(a, ra);
                if (c2 > kTiny || !(a2 > kTiny)) p1 = scale(c, rc);
                q1 = big ? scale(mulc(d, p1), ra) : scale(mulc(b, p0), -rc);
            } else if (form == 2) {
                if (big) {
                    p0 = scale(a, ra);
                    p1 = scale(d, ra);
                    S = mulc(c, p1).x;
                } else {
                    p1 = scale(c, rc);
                    p0 = scale(b, -rc);
                    C = mulc(a, p0).x;
                }
            } else {
                if (big) {
                    q0 = scale(a, ra);
                    q1 = scale(d, ra);
                    S = mulc(c, q0).x;
                } else {
                    q0 = scale(c, rc);
                    q1 = scale(b, -rc);
                    C = mulc(a, q0).x;
                }
            }
        }
        o[0] = R(C); o[1] = R(S);
        double2* ph = reinterpret_cast<double2*>(o + 2);
        ph[0] = p0; ph[1] = p1; ph[2] = q0; ph[3] = q1;
        o[10] = R(0); o[11] = R(0);
    }
}

// Tables of the resident path: complex64 forward ones without U^dag (a 13-qubit random
// circuit's tables 36 -> 18 KB per sample), double-float ones of the kernels without
// factored stages (Factored) without the factors.
template <typename R, bool FULL, bool PH2> struct Factored {
    static constexpr bool value = std::is_same<R, dd>::value && FULL && !PH2;
};
template <typename R, int MODE, bool FULL, bool PH2> struct ResidentWords {
    static constexpr bool dbf = std::is_same<R, dd>::value;
    static constexpr int value = dbf && !Factored<R, FULL, PH2>::value ? entry_reals(true, false)
                                              : EntryWords<R>::value / (!dbf && sizeof(R) == 4 && MODE == 0 ? 2 : 1);
};

template <typename R, int EW = EntryWords<R>::value>
__device__ __forceinline__ void store_matrix(const M2<R>& m, R* out) {
    if constexpr (sizeof(R) == 4) {   // 16-byte stores (entries are 128-byte aligned)
        const C2<R> e[4] = {m.a, m.b, m.c, m.d};
        const C2<R> d[4] = {cconj<R>(m.a), cconj<R>(m.c), cconj<R>(m.b), cconj<R>(m.d)};
        float4* o4 = reinterpret_cast<float4*>(out);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            o4[k] = make_float4(e[k].x, e[k].y, -e[k].y, e[k].x);        // (m, i m)
            if (EW == EntryWords<R>::value) o4[4 + k] = make_float4(d[k].x, d[k].y, -d[k].y, d[k].x);
        }
    } else {
        out[0] = m.a.x; out[1] = m.a.y; out[2] = m.b.x; out[3] = m.b.y;
        out[4] = m.c.x; out[5] = m.c.y; out[6] = m.d.x; out[7] = m.d.y;
    }
}
template <typename R, typename XI, typename WI>
__device__ __forceinline__ R angle_of(uint8_t src, int32_t idx, const XI* xb, const WI* w,
                                      const R* cang) {
    if (src == SRC_X) return as_r<R>(xb[idx]);
    if (src == SRC_W) return as_r<R>(w[idx]);
    return cang[idx];
}

// Matrix of one constituent of a run.
template <typename R, typename XI, typename WI>
__device__ __forceinline__ M2<R> constituent(const DConst& c, const XI* xb, const WI* w, const R* cang,
                             const R* cmat) {
    M2<R> u;
    if (c.kind == CK_CONST) {
        const R* m = cmat + 8 * c.idx0;
        u.a = cm<R>(m[0], m[1]); u.b = cm<R>(m[2], m[3]);
        u.c = cm<R>(m[4], m[5]); u.d = cm<R>(m[6], m[7]);
        return u;
    }
    R t = angle_of<R>(c.src0, c.idx0, xb, w, cang);
    if (c.kind == CK_GPHASE) t += angle_of<R>(c.src1, c.idx1, xb, w, cang);
    R s, co;
    sc(t * R(0.5), &s, &co);
    const C2<R> z = cm<R>(0, 0);
    switch (c.kind) {
    case CK_RX: u.a = cm<R>(co, 0); u.b = cm<R>(0, -s); u.c = cm<R>(0, -s); u.d = cm<R>(co, 0); break;
    case CK_RY: u.a = cm<R>(co, 0); u.b = cm<R>(-s, 0); u.c = cm<R>(s, 0); u.d = cm<R>(co, 0); break;
    case CK_RZ: u.a = cm<R>(co, -s); u.b = z; u.c = z; u.d = cm<R>(co, s); break;
    default:    u.a = cm<R>(co, s); u.b = z; u.c = z; u.d = cm<R>(co, s); break;   // CK_GPHASE
    }
    return u;
}

// Evaluate one table entry (8 reals) for sample row xb.
template <typename R, int EW = EntryWords<R>::value, typename XI, typename WI>
__device__ __forceinline__ void eval_entry(const DEntry& e, const DConst* consts, const XI* xb, const WI* w,
                           const R* cang, const R* cmat, R* out) {
    if (e.phase) {
        const DConst c = consts[e.cfirst];
        R t = angle_of<R>(c.src0, c.idx0, xb, w, cang);
        R s, co;
        sc(t * R(0.5), &s, &co);
        if (c.kind == CK_CRZ) {
            out[0] = 1; out[1] = 0; out[2] = co; out[3] = -s;
            out[4] = 1; out[5] = 0; out[6] = co; out[7] = s;
        } else {   // CK_RZZ: parity 0 -> e^{-it/2}, parity 1 -> e^{it/2}
            out[0] = co; out[1] = -s; out[2] = co; out[3] = s;
            out[4] = co; out[5] = s; out[6] = co; out[7] = -s;
        }
        return;
    }
    M2<R> m = mident<R>();
    for (int k = 0; k < e.ccount; ++k) {
        const DConst c = consts[e.cfirst + k];
        m = mmul<R>(constituent<R>(c, xb, w, cang, cmat), m);
    }
    store_matrix<R, EW>(m, out);
    if constexpr (std::is_same<R, dd>::value && EW == EntryWords<R>::value)
        store_factors<R>(m, run_form(consts + e.cfirst, e.ccount), out + 8);
}

template <typename R>
__device__ __forceinline__ M2<R> load_m2(const R* p) {
    M2<R> m;
    m.a = cm<R>(p[0], p[1]); m.b = cm<R>(p[2], p[3]);
    m.c = cm<R>(p[4], p[5]); m.d = cm<R>(p[6], p[7]);
    return m;
}

// ---------------------------------------------------------------- block ops
// Pair (i0, i1) = (r with bit T clear, r with bit T set), p enumerates pairs.
template <int T>
__host__ __device__ constexpr int pair_lo(int p) { return ((p >> T) << (T + 1)) | (p & ((1 << T) - 1)); }

template <typename R, int K, int T>
__device__ __forceinline__ void m1_apply(C2<R> (&a)[1 << K], const M2<R>& m) {
#pragma unroll
    for (int p = 0; p < (1 << (K - 1)); ++p) {
        const int i0 = pair_lo<T>(p), i1 = i0 | (1 << T);
        C2<R> u = a[i0], v = a[i1];
        a[i0] = cmv2<R>(m.a, u, m.b, v);
        a[i1] = cmv2<R>(m.c, u, m.d, v);
    }
}

// Gradient accumulator of a fused run.  With rho = sum_pairs psi conj(lam)^T
// (2x2, rho[a][b] = psi_a conj(lam_b)), every term the run needs is
// Im Tr(P rho') for a Pauli P and rho' = W^dag rho W, i.e. it depends only on
// the traceless anti-Hermitian part of rho, (i/2)(tx X + ty Y + tz Z), and that
// part stays traceless anti-Hermitian under W^dag . W.  So three reals per
// thread are summed instead of rho's eight:
//   tx = Im(rho01 + rho10), ty = Re(rho01 - rho10), tz = Im(rho00 - rho11).
// One running sum per component: two partial sums (shorter FMA chains) held
// more registers and measured 2-4% slower in the backward kernels.
template <typename R, int K, int T>
__device__ __forceinline__ void m1_t3(const C2<R> (&ps)[1 << K], const C2<R> (&la)[1 << K],
                                      R (&v)[4]) {
    if constexpr (std::is_same<R, dd>::value) {   // each component one long compensated dot product
        ddsum sx, sy, sz;
#pragma unroll
        for (int p = 0; p < (1 << (K - 1)); ++p) {
            const int i0 = pair_lo<T>(p), i1 = i0 | (1 << T);
            const dd2 u = ps[i0], w = ps[i1], q0 = la[i0], q1 = la[i1];
            sx.add(u.y, q1.x); sx.add(-u.x, q1.y); sx.add(w.y, q0.x); sx.add(-w.x, q0.y);
            sy.add(u.x, q1.x); sy.add(u.y, q1.y); sy.add(-w.x, q0.x); sy.add(-w.y, q0.y);
            sz.add(u.y, q0.x); sz.add(-u.x, q0.y); sz.add(-w.y, q1.x); sz.add(w.x, q1.y);
        }
        v[0] += sx.value();
        v[1] += sy.value();
        v[2] += sz.value();
        return;
    }
    R xa = 0, ya = 0, za = 0;
#pragma unroll
    for (int p = 0; p < (1 << (K - 1)); ++p) {
        const int i0 = pair_lo<T>(p), i1 = i0 | (1 << T);
        const C2<R> u = ps[i0], w = ps[i1], q0 = la[i0], q1 = la[i1];
        // Im(u conj q1) + Im(w conj q0)
        xa = fma(u.y, q1.x, fma(-u.x, q1.y, fma(w.y, q0.x, fma(-w.x, q0.y, xa))));
        // Re(u conj q1) - Re(w conj q0)
        ya = fma(u.x, q1.x, fma(u.y, q1.y, fma(-w.x, q0.x, fma(-w.y, q0.y, ya))));
        // Im(u conj q0) - Im(w conj q1)
        za = fma(u.y, q0.x, fma(-u.x, q0.y, fma(-w.y, q1.x, fma(w.x, q1.y, za))));
    }
    v[0] += xa;
    v[1] += ya;
    v[2] += za;
}

// complex64 2x2 update with Blackwell's packed FP32 instructions (FFMA2 on
// (re, im) pairs), the operand pairs read directly from a table entry (w: 8
// float2 = a, i a, b, i b, c, i c, d, i d).  With each state component
// broadcast to both lanes,
//   m u = (u.re, u.re) * m + (u.im, u.im) * (i m)
// so a complex multiply-add is two FFMA2 and a pair update eight.  (The form
// with the table's (Re m, Re m), (-Im m, Im m) pairs needs the swapped state
// pair (u.im, u.re) instead and measured 2-8% slower.)
//
// Four pairs of a state at a time: the first product of all of them, then the second,
// and so on, since each waits for the one before it.  (Pair by pair the compiler kept
// most chains whole: 16-qubit step, B = 512, 6.41 ms against 6.24; BOTH
// states of a backward stage together, eight pairs at a time, take another 1% off the
// 12-qubit resident step, 1.69 -> 1.68 ms at B = 4096.)
template <int K, int T, bool BOTH>
__device__ __forceinline__ void m1_apply_f2w(float2 (&a)[1 << K], float2 (&l)[1 << K], const float* wp) {
    const float4 w0 = *reinterpret_cast<const float4*>(wp);
    const float4 w1 = *reinterpret_cast<const float4*>(wp + 4);
    const float4 w2 = *reinterpret_cast<const float4*>(wp + 8);
    const float4 w3 = *reinterpret_cast<const float4*>(wp + 12);
    const float2 ar = make_float2(w0.x, w0.y), ai = make_float2(w0.z, w0.w);
    const float2 br = make_float2(w1.x, w1.y), bi = make_float2(w1.z, w1.w);
    const float2 cr = make_float2(w2.x, w2.y), ci = make_float2(w2.z, w2.w);
    const float2 dr = make_float2(w3.x, w3.y), di = make_float2(w3.z, w3.w);
    constexpr int N = 1 << (K - 1), H = N < 4 ? N : 4, GR = BOTH ? 2 * H : H;
#pragma unroll
    for (int p0 = 0; p0 < N; p0 += H) {
        float2 u[GR], v[GR], nu[GR], nv[GR];
#pragma unroll
        for (int g = 0; g < GR; ++g) {
            const int i0 = pair_lo<T>(p0 + g % H), i1 = i0 | (1 << T);
            u[g] = g < H ? a[i0] : l[i0];
            v[g] = g < H ? a[i1] : l[i1];
        }
        // entries hold (m, i m): m u = u.re (m) + u.im (i m)
#pragma unroll
        for (int g = 0; g < GR; ++g) {
            nu[g] = __fmul2_rn(ar, make_float2(u[g].x, u[g].x));
            nv[g] = __fmul2_rn(cr, make_float2(u[g].x, u[g].x));
        }
#pragma unroll
        for (int g = 0; g < GR; ++g) {
            nu[g] = __ffma2_rn(ai, make_float2(u[g].y, u[g].y), nu[g]);
            nv[g] = __ffma2_rn(ci, make_float2(u[g].y, u[g].y), nv[g]);
        }
#pragma unroll
        for (int g = 0; g < GR; ++g) {
            nu[g] = __ffma2_rn(br, make_float2(v[g].x, v[g].x), nu[g]);
            nv[g] = __ffma2_rn(dr, make_float2(v[g].x, v[g].x), nv[g]);
        }
#pragma unroll
        for (int g = 0; g < GR; ++g) {
            const int i0 = pair_lo<T>(p0 + g % H), i1 = i0 | (1 << T);
            nu[g] = __ffma2_rn(bi, make_float2(v[g].y, v[g].y), nu[g]);
            nv[g] = __ffma2_rn(di, make_float2(v[g].y, v[g].y), nv[g]);
            (g < H ? a : l)[i0] = nu[g];
            (g < H ? a : l)[i1] = nv[g];
        }
    }
}

// Apply the table entry at tp (forward: U; adjoint: U^dag).
template <typename R, int K, int T, bool ADJ>
__device__ __forceinline__ void m1_entry(C2<R> (&a)[1 << K], const R* tp) {
    if constexpr (sizeof(R) == 4) {
        m1_apply_f2w<K, T, false>(a, a, tp + (ADJ ? 16 : 0));
    } else {
        M2<R> m = load_m2<R>(tp);
        if (ADJ) m = mdag<R>(m);
        m1_apply<R, K, T>(a, m);
    }
}

// U^dag of the entry at tp on psi and lam.
template <typename R, int K, int T>
__device__ __forceinline__ void m1_back(C2<R> (&a)[1 << K], C2<R> (&l)[1 << K], const R* tp) {
    if constexpr (sizeof(R) == 4) {
        m1_apply_f2w<K, T, true>(a, l, tp + 16);
    } else {
        m1_entry<R, K, T, true>(a, tp);
        m1_entry<R, K, T, true>(l, tp);
    }
}

// v, negated when p.  double: its sign bit, beside the FP64 pipe, which a product with -1
// would take 16 cycles a warp of.
template <typename R>
__device__ __forceinline__ C2<R> negated(C2<R> v, bool p) {
    if constexpr (std::is_same<R, double>::value) {
        const int m = p ? (int)0x80000000 : 0;
        return cm<R>(__hiloint2double(__double2hiint(v.x) ^ m, __double2loint(v.x)),
                     __hiloint2double(__double2hiint(v.y) ^ m, __double2loint(v.y)));
    } else {
        const R s = p ? R(-1) : R(1);
        return cm<R>(s * v.x, s * v.y);
    }
}
// Negate amplitudes with local bits A and Bq set (when p) -- CZ inside the block.
template <typename R, int K, int A, int Bq>
__device__ __forceinline__ void z2_ll(C2<R> (&a)[1 << K]) {
#pragma unroll
    for (int r = 0; r < (1 << K); ++r)
        if (((r >> A) & 1) && ((r >> Bq) & 1)) a[r] = cm<R>(-a[r].x, -a[r].y);
}
template <typename R, int K, int A>
__device__ __forceinline__ void z1_pred(C2<R> (&a)[1 << K], bool p) {
#pragma unroll
    for (int r = 0; r < (1 << K); ++r)
        if ((r >> A) & 1) a[r] = negated<R>(a[r], p);
}

// ---------------------------------------------------------------- reductions
// Butterfly exchange with lane ^ m (double-float: both parts).
template <typename R>
__device__ __forceinline__ R shx(R v, int m, unsigned mask) {
    if constexpr (std::is_same<R, dd>::value)
        return dd(__shfl_xor_sync(mask, v.hi, m), __shfl_xor_sync(mask, v.lo, m));
    else
        return __shfl_xor_sync(mask, v, m);
}

// Reduce 4 values over a group of `lanes` lanes (power of two <= 32) and write
// the 4 sums to dst[0..3] (reduce-scatter: 2 + 1 exchanges, then plain steps).
template <typename R>
__device__ __forceinline__ void reduce4_store(R (&v)[4], int lanes, int lane, R* dst,
                                              unsigned mask, bool add) {
    int u0 = 0, u1 = 0;
    if (lanes >= 2) {
        const int m = lanes >> 1;
        u0 = (lane & m) ? 1 : 0;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            R send = u0 ? v[i] : v[i + 2];
            R keep = u0 ? v[i + 2] : v[i];
            v[i] = keep + shx<R>(send, m, mask);
        }
    }
    if (lanes >= 4) {
        const int m = lanes >> 2;
        u1 = (lane & m) ? 1 : 0;
        R send = u1 ? v[0] : v[1];
        R keep = u1 ? v[1] : v[0];
        v[0] = keep + shx<R>(send, m, mask);
        for (int mm = lanes >> 3; mm >= 1; mm >>= 1) v[0] += shx<R>(v[0], mm, mask);
        if ((lane & ((lanes >> 2) - 1)) == 0) {
            R* d = dst + 2 * u0 + u1;
            *d = add ? *d + v[0] : v[0];
        }
    } else if (lanes == 2) {
        for (int i = 0; i < 2; ++i) dst[2 * u0 + i] = add ? dst[2 * u0 + i] + v[i] : v[i];
    } else {
        for (int i = 0; i < 4; ++i) dst[i] = add ? dst[i] + v[i] : v[i];
    }
}

// reduce4_store for a full warp, branch-free: 2 + 1 scatter shuffles and 3
// plain ones; lanes with (lane & 7) == 0 write their sum.
template <typename R>
__device__ __forceinline__ void reduce4_full(R (&v)[4], int lane, R* dst, bool add) {
    const unsigned full = 0xffffffffu;
    const int u0 = (lane >> 4) & 1, u1 = (lane >> 3) & 1;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const R send = u0 ? v[i] : v[i + 2];
        const R keep = u0 ? v[i + 2] : v[i];
        v[i] = keep + shx<R>(send, 16, full);
    }
    {
        const R send = u1 ? v[0] : v[1];
        const R keep = u1 ? v[1] : v[0];
        v[0] = keep + shx<R>(send, 8, full);
    }
    v[0] += shx<R>(v[0], 4, full);
    v[0] += shx<R>(v[0], 2, full);
    v[0] += shx<R>(v[0], 1, full);
    if ((lane & 7) == 0) {
        R* d = dst + 2 * u0 + u1;
        *d = add ? *d + v[0] : v[0];
    }
}

template <typename R>
__device__ __forceinline__ R reduce1(R v, int lanes, unsigned mask) {
    for (int m = lanes >> 1; m >= 1; m >>= 1) v += shx<R>(v, m, mask);
    return v;
}

// ---------------------------------------------------------------- addressing
struct Geo {
    int T;        // threads per sample group
    int lanes;    // min(T, 32)
    int wg;       // warps per group (>= 1)
    int g;        // group (sample slot) index in the CTA
    int t;        // thread index in the group
    int h;        // per-sample XOR on the slot index (bank spreading of small groups)
    unsigned mask;   // lanes of this warp that exist (a CTA smaller than a warp)
};

__device__ __forceinline__ uint32_t swz(uint32_t u, int G) {
    uint32_t v = u >> G, f = 0;
    while (v) { f ^= v; v >>= G; }
    return u ^ (f & ((1u << G) - 1));
}

template <typename R>
__device__ __forceinline__ void group_sync(const Geo& q) {
    if (q.T > 32) __syncthreads(); else __syncwarp(q.mask);
}

template <int K>
__device__ __forceinline__ uint32_t block_off(int r, const int32_t (&sg)[K]) {
    uint32_t o = 0;
#pragma unroll
    for (int j = 0; j < K; ++j)
        if ((r >> j) & 1) o ^= (uint32_t)sg[j];
    return o;
}

struct StageView {
    uint32_t swb, pb;
};

// XOR of the entries of v[0 .. 16) selected by the set bits of t, with all
// loads independent (no loop-carried branch): a thread's slot base.  Entries
// past the stage's thread bits are zero in the record, and t has no bits there.
__device__ __forceinline__ uint32_t xor_select(const int32_t* v, int nb, int t) {
    uint32_t b = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) b ^= ((t >> i) & 1) ? (uint32_t)vqc_ld(&v[i]) : 0u;
    if (nb > 8) {
#pragma unroll
        for (int i = 8; i < kMaxThreadBits; ++i) b ^= ((t >> i) & 1) ? (uint32_t)vqc_ld(&v[i]) : 0u;
    }
    return b;
}

template <int K>
__device__ __forceinline__ StageView stage_view(const DStage* sp, int t, int h, int32_t (&sg)[K]) {
#pragma unroll
    for (int j = 0; j < K; ++j) sg[j] = vqc_ld(&sp->sigma[j]);
    const int nb = vqc_ld(&sp->nthreadbits);   // uint8 load
    StageView v;
    v.swb = (uint32_t)h ^ xor_select(sp->tau, nb, t);
    v.pb = xor_select(reinterpret_cast<const int32_t*>(sp->tmask), nb, t);   // disjoint bits
    return v;
}

// Slot base of thread t and the local offsets of a stage's load map (ST false)
// or store map (ST true), read from the stage record.
template <int K, bool ST>
__device__ __forceinline__ uint32_t map_base(const DStage* sp, int t, int h, int32_t (&sg)[K]) {
    const int32_t* sig = ST ? sp->sigma_st : sp->sigma;
#pragma unroll
    for (int j = 0; j < K; ++j) sg[j] = vqc_ld(&sig[j]);
    const int nb = vqc_ld(&sp->nthreadbits);
    return (uint32_t)h ^ xor_select(ST ? sp->tau_st : sp->tau, nb, t);
}

template <typename R, int K>
__device__ __forceinline__ void block_load(C2<R> (&a)[1 << K], const C2<R>* st, uint32_t swb,
                                           const int32_t (&sg)[K]) {
#pragma unroll
    for (int r = 0; r < (1 << K); ++r) a[r] = st[swb ^ block_off<K>(r, sg)];
}
// The store recomputes the 2^K slot offsets (an empty asm hides swb's value
// from the compiler) instead of keeping the load's offsets live in registers
// across the stage's ops.
template <typename R, int K>
__device__ __forceinline__ void block_store(const C2<R> (&a)[1 << K], C2<R>* st, uint32_t swb,
                                            const int32_t (&sg)[K]) {
    asm volatile("" : "+r"(swb));
    int32_t s2[K];
#pragma unroll
    for (int j = 0; j < K; ++j) {
        s2[j] = sg[j];
        asm volatile("" : "+r"(s2[j]));
    }
#pragma unroll
    for (int r = 0; r < (1 << K); ++r) st[swb ^ block_off<K>(r, s2)] = a[r];
}

// Diagonal two-qubit phase (CRZ, RZZ): amplitude r is multiplied by ph[s],
// s = bit a + 2 bit b (a, b = the gate's first and second qubit), conjugated in
// the backward, where the gradient term Im <lam|P|psi> = sum_r g[s] Im(conj(lam_r)
// psi_r) is taken first (g = the generator's diagonal: CRZ (0, 1, 0, -1), RZZ
// (1, -1, -1, 1)).  Three forms by where a and b live; each resolves s per
// amplitude at compile time except for one per-op selection.
template <typename R>
__device__ __forceinline__ void ph2_gen(uint8_t flags, R (&g)[4]) {
    if (flags & OPF_GEN_CRZ) { g[0] = 0; g[1] = 1; g[2] = 0; g[3] = -1; }
    else { g[0] = 1; g[1] = -1; g[2] = -1; g[3] = 1; }
}
template <typename R>
__device__ __forceinline__ R gen_at(uint8_t flags, int s) {   // g[s] for a runtime s
    if (flags & OPF_GEN_CRZ) return s == 1 ? R(1) : s == 3 ? R(-1) : R(0);
    return (s == 0 || s == 3) ? R(1) : R(-1);
}
template <typename R>
__device__ __forceinline__ R im_conj_mul(const C2<R>& la, const C2<R>& ps) {
    return la.x * ps.y - la.y * ps.x;
}
// s + Im(conj(la) ps).
template <typename R>
__device__ __forceinline__ R im_conj_add(const C2<R>& la, const C2<R>& ps, R s) {
    if constexpr (std::is_same<R, float>::value) return fma(la.x, ps.y, fma(-la.y, ps.x, s));
    else return s + im_conj_mul<R>(la, ps);
}
// v f; complex64 in packed instructions, each component's roundings those of cmul: half
// the instructions of a phase op, and with the gradient term's sums per phase instead of
// a product with the generator's sign each, no spills in the kernels with phase cases
// (backward pass kernel 68/252 bytes before).  15-qubit QAOA step, B = 96, 787 -> 712 us;
// 13-qubit random forward, B = 256, 219 -> 199 us.
template <typename R>
__device__ __forceinline__ C2<R> phase_mul(C2<R> v, C2<R> f) {
    if constexpr (std::is_same<R, float>::value)
        return __ffma2_rn(make_float2(v.x, v.x), f, __fmul2_rn(make_float2(v.y, v.y), make_float2(-f.y, f.x)));
    else
        return cmul<R>(v, f);
}
template <typename R, bool FULL>
__device__ __forceinline__ void ph2_term_store(R tv, const Geo& q, R* accp, bool acc_add) {
    if (FULL) {
#pragma unroll
        for (int m = 16; m >= 1; m >>= 1) tv += shx<R>(tv, m, 0xffffffffu);
    } else {
        tv = reduce1<R>(tv, q.lanes, q.mask);
    }
    if ((q.t & (q.lanes - 1)) == 0) accp[0] = acc_add ? accp[0] + tv : tv;
}
template <typename R, int K, int MODE, bool FULL, int LO, int HI>
__device__ __forceinline__ void ph2_ll(bool swapped, const R* tp, uint8_t flags,
                                       C2<R> (&a)[1 << K], C2<R> (&l)[1 << K], const Geo& q,
                                       R* accp, bool acc_add) {
    // index by (bit LO) + 2 (bit HI): swap entries 1 and 2 when a is the higher position
    C2<R> ph[4] = {cm<R>(tp[0], tp[1]), cm<R>(tp[2], tp[3]), cm<R>(tp[4], tp[5]), cm<R>(tp[6], tp[7])};
    R g[4];
    ph2_gen<R>(flags, g);
    if (swapped) {
        const C2<R> t = ph[1]; ph[1] = ph[2]; ph[2] = t;
        const R u = g[1]; g[1] = g[2]; g[2] = u;
    }
    if (MODE == 1) {
#pragma unroll
        for (int s = 0; s < 4; ++s) ph[s].y = -ph[s].y;
        if (flags & OPF_HAS_ACC) {
            R tv = 0;
            if constexpr (std::is_same<R, float>::value) {
                R t[4] = {0, 0, 0, 0};
#pragma unroll
                for (int r = 0; r < (1 << K); ++r) {
                    const int s = ((r >> LO) & 1) + 2 * ((r >> HI) & 1);
                    t[s] = im_conj_add<R>(l[r], a[r], t[s]);
                }
                tv = fma(g[0], t[0], g[1] * t[1]) + fma(g[2], t[2], g[3] * t[3]);
            } else {
#pragma unroll
                for (int r = 0; r < (1 << K); ++r)
                    tv = fma(g[((r >> LO) & 1) + 2 * ((r >> HI) & 1)], im_conj_mul<R>(l[r], a[r]), tv);
            }
            ph2_term_store<R, FULL>(tv, q, accp, acc_add);
        }
    }
#pragma unroll
    for (int r = 0; r < (1 << K); ++r) {
        const int s = ((r >> LO) & 1) + 2 * ((r >> HI) & 1);
        a[r] = phase_mul<R>(a[r], ph[s]);
        if (MODE == 1) l[r] = phase_mul<R>(l[r], ph[s]);
    }
}
template <typename R, int K, int MODE, bool FULL, int L>
__device__ __forceinline__ void ph2_pl(bool a_local, bool p, const R* tp, uint8_t flags,
                                       C2<R> (&a)[1 << K], C2<R> (&l)[1 << K], const Geo& q,
                                       R* accp, bool acc_add) {
    // s = bit L + 2 p (a local) or p + 2 bit L (b local)
    const int s0 = a_local ? 2 * (int)p : (int)p, s1 = a_local ? 1 + 2 * (int)p : (int)p + 2;
    C2<R> f0 = cm<R>(tp[2 * s0], tp[2 * s0 + 1]), f1 = cm<R>(tp[2 * s1], tp[2 * s1 + 1]);
    const R g0 = gen_at<R>(flags, s0), g1 = gen_at<R>(flags, s1);
    if (MODE == 1) {
        f0.y = -f0.y;
        f1.y = -f1.y;
        if (flags & OPF_HAS_ACC) {
            R tv = 0;
            if constexpr (std::is_same<R, float>::value) {
                R t[2] = {0, 0};
#pragma unroll
                for (int r = 0; r < (1 << K); ++r) t[(r >> L) & 1] = im_conj_add<R>(l[r], a[r], t[(r >> L) & 1]);
                tv = fma(g0, t[0], g1 * t[1]);
            } else {
#pragma unroll
                for (int r = 0; r < (1 << K); ++r)
                    tv = fma(((r >> L) & 1) ? g1 : g0, im_conj_mul<R>(l[r], a[r]), tv);
            }
            ph2_term_store<R, FULL>(tv, q, accp, acc_add);
        }
    }
#pragma unroll
    for (int r = 0; r < (1 << K); ++r) {
        const C2<R> f = ((r >> L) & 1) ? f1 : f0;
        a[r] = phase_mul<R>(a[r], f);
        if (MODE == 1) l[r] = phase_mul<R>(l[r], f);
    }
}
template <typename R, int K, int MODE, bool FULL>
__device__ __forceinline__ void ph2_pp(int s, const R* tp, uint8_t flags, C2<R> (&a)[1 << K],
                                       C2<R> (&l)[1 << K], const Geo& q, R* accp, bool acc_add) {
    C2<R> f = cm<R>(tp[2 * s], tp[2 * s + 1]);
    if (MODE == 1) {
        f.y = -f.y;
        if (flags & OPF_HAS_ACC) {
            constexpr int NT = std::is_same<R, float>::value ? 4 : 1;
            R t[4] = {0, 0, 0, 0};
#pragma unroll
            for (int r = 0; r < (1 << K); ++r) t[r % NT] = im_conj_add<R>(l[r], a[r], t[r % NT]);
            const R tv = NT == 1 ? t[0] : (t[0] + t[1]) + (t[2] + t[3]);
            ph2_term_store<R, FULL>(gen_at<R>(flags, s) * tv, q, accp, acc_add);
        }
    }
#pragma unroll
    for (int r = 0; r < (1 << K); ++r) {
        a[r] = phase_mul<R>(a[r], f);
        if (MODE == 1) l[r] = phase_mul<R>(l[r], f);
    }
}

// The same for every place of a and b, their positions and the phase of an amplitude
// taken at run time: double-float, whose products (about 40 instructions an amplitude)
// hide that, and whose code for each place, 5 to 10 KB, does not fit the instruction
// cache with the others' (QAOA circuits of 8 to 12 qubits, forward and backward, 1.18
// times as fast in the mean).  Blocks of 16 amplitudes spill more with it (0.88 to 0.97
// times at batch 1600) and keep the cases.
template <typename R, int K, int MODE, bool FULL>
__device__ __forceinline__ void ph2_any(int ra, int rb, uint32_t pb, const R* tp, uint8_t flags, C2<R> (&a)[1 << K],
                                        C2<R> (&l)[1 << K], const Geo& q, R* accp, bool acc_add) {
    const int pa = ra >= kRefPhys ? (int)((pb >> (ra - kRefPhys)) & 1u) : 0;
    const int pc = rb >= kRefPhys ? (int)((pb >> (rb - kRefPhys)) & 1u) : 0;
    const int ma = ra >= kRefPhys ? 0 : 1 << ra, mb = rb >= kRefPhys ? 0 : 1 << rb;
    const C2<R>* ph = reinterpret_cast<const C2<R>*>(tp);
    const bool acc = MODE == 1 && (flags & OPF_HAS_ACC);
    R tv = 0;
#pragma unroll
    for (int r = 0; r < (1 << K); ++r) {
        const int s = (pa | ((r & ma) ? 1 : 0)) + 2 * (pc | ((r & mb) ? 1 : 0));
        C2<R> f = ph[s];
        if (MODE == 1) {
            f.y = -f.y;
            if (acc) tv = fma(gen_at<R>(flags, s), im_conj_mul<R>(l[r], a[r]), tv);
            l[r] = cmul<R>(l[r], f);
        }
        a[r] = cmul<R>(a[r], f);
    }
    if (acc) ph2_term_store<R, FULL>(tv, q, accp, acc_add);
}

// ---------------------------------------------------------------- op dispatch
__device__ __forceinline__ bool physbit(uint32_t pb, int ref) {
    return ((pb >> (ref - kRefPhys)) & 1u) != 0;
}

// Apply op `raw` to the block(s).  MODE 0: forward on a.  MODE 1: backward --
// accumulate the op's gradient slot, then un-apply on a (psi) and l (lam).
// One switch over the dispatch code; every case has fixed local positions.
// WITH_PH2: the schedule may hold diagonal two-qubit phase ops (CRZ, RZZ).
// Kernels for plans without them are instantiated with the cases left out:
// their register allocation then needs fewer spills (measured 8-11% faster on
// the 12-qubit resident sweeps and the 16-qubit forward passes); the launch
// code picks the instantiation from the plan.
template <typename R, int K, int MODE, bool FULL, bool WITH_PH2 = true, int EW = EntryWords<R>::value>
__device__ __forceinline__ void apply_op(uint2 raw, uint32_t pb, C2<R> (&a)[1 << K],
                                         C2<R> (&l)[1 << K], const R* sh_tab, const R* ps_tab,
                                         R* acc, const Geo& q, int lane, int warp_in_group,
                                         bool acc_add) {
    const int code = raw.x & 0xff, ra = (raw.x >> 8) & 0xff, rb = (raw.x >> 16) & 0xff;
    const int flags = raw.x >> 24, slot = raw.y & 0xffff, aux = raw.y >> 16;
    const R* tp = ((flags & OPF_PER_SAMPLE) ? ps_tab : sh_tab) + EW * slot;
    R* accp = acc + ((size_t)aux * q.wg + warp_in_group) * 8;
    const int rlane = FULL ? lane : q.t;
    constexpr bool ANY = std::is_same<R, dd>::value && K < 4;   // ph2_any
    if constexpr (WITH_PH2 && ANY)
        if (code >= DC_PH2_LL) {
            ph2_any<R, K, MODE, FULL>(ra, rb, pb, tp, flags, a, l, q, accp, acc_add);
            return;
        }
    switch (code) {
#define VQC_M1(T_)                                                                   \
    case DC_M1 + T_:                                                                 \
        if constexpr (T_ < K) {                                                      \
            if (MODE == 0) {                                                         \
                m1_entry<R, K, T_, false>(a, tp);                                    \
            } else {                                                                 \
                if constexpr (FULL) {                                                \
                    /* one basic block; the butterfly is issued before the    */     \
                    /* adjoint updates so that the accumulator registers are */     \
                    /* free while both blocks are updated (fewer spills under */     \
                    /* the pass kernels' 128-register cap)                    */     \
                    if (flags & OPF_HAS_ACC) {                                       \
                        R rh[4] = {0, 0, 0, 0};                                      \
                        m1_t3<R, K, T_>(a, l, rh);                                   \
                        reduce4_full<R>(rh, lane, accp, acc_add);                    \
                        m1_entry<R, K, T_, true>(a, tp);                             \
                        m1_entry<R, K, T_, true>(l, tp);                             \
                    } else {                                                         \
                        m1_entry<R, K, T_, true>(a, tp);                             \
                        m1_entry<R, K, T_, true>(l, tp);                             \
                    }                                                                \
                } else {                                                             \
                    if (flags & OPF_HAS_ACC) {                                       \
                        R rh[4] = {0, 0, 0, 0};                                      \
                        m1_t3<R, K, T_>(a, l, rh);                                   \
                        reduce4_store<R>(rh, q.lanes, rlane, accp, q.mask, acc_add); \
                    }                                                                \
                    m1_entry<R, K, T_, true>(a, tp);                                 \
                    m1_entry<R, K, T_, true>(l, tp);                                 \
                }                                                                    \
            }                                                                        \
        }                                                                            \
        break;
        VQC_M1(0) VQC_M1(1) VQC_M1(2) VQC_M1(3) VQC_M1(4)
#undef VQC_M1
#define VQC_CZLL(A_, B_)                                                             \
    case DC_CZ_LL + cz_pair_index(A_, B_):                                           \
        if constexpr (A_ < K && B_ < K) {                                            \
            z2_ll<R, K, A_, B_>(a);                                                  \
            if (MODE == 1) z2_ll<R, K, A_, B_>(l);                                   \
        }                                                                            \
        break;
        VQC_CZLL(0, 1) VQC_CZLL(0, 2) VQC_CZLL(0, 3) VQC_CZLL(0, 4)
        VQC_CZLL(1, 2) VQC_CZLL(1, 3) VQC_CZLL(1, 4)
        VQC_CZLL(2, 3) VQC_CZLL(2, 4) VQC_CZLL(3, 4)
#undef VQC_CZLL
#define VQC_CZPL(L_)                                                                 \
    case DC_CZ_PL + L_:                                                              \
        if constexpr (L_ < K) {                                                      \
            const bool p_ = physbit(pb, rb);                                         \
            z1_pred<R, K, L_>(a, p_);                                                \
            if (MODE == 1) z1_pred<R, K, L_>(l, p_);                                 \
        }                                                                            \
        break;
        VQC_CZPL(0) VQC_CZPL(1) VQC_CZPL(2) VQC_CZPL(3) VQC_CZPL(4)
#undef VQC_CZPL
    case DC_CZ_PP: {
        const bool neg = physbit(pb, ra) && physbit(pb, rb);
#pragma unroll
        for (int r = 0; r < (1 << K); ++r) {
            a[r] = negated<R>(a[r], neg);
            if (MODE == 1) l[r] = negated<R>(l[r], neg);
        }
        break;
    }
#define VQC_PH2LL(LO_, HI_)                                                          \
    case DC_PH2_LL + cz_pair_index(LO_, HI_):                                        \
        if constexpr (WITH_PH2 && !ANY && LO_ < K && HI_ < K) ph2_ll<R, K, MODE, FULL, LO_, HI_>(ra > rb, tp, flags, a, l, q, accp, acc_add); \
        break;
        VQC_PH2LL(0, 1) VQC_PH2LL(0, 2) VQC_PH2LL(0, 3) VQC_PH2LL(0, 4)
        VQC_PH2LL(1, 2) VQC_PH2LL(1, 3) VQC_PH2LL(1, 4)
        VQC_PH2LL(2, 3) VQC_PH2LL(2, 4) VQC_PH2LL(3, 4)
#undef VQC_PH2LL
#define VQC_PH2PL(L_)                                                                \
    case DC_PH2_PL + L_:                                                             \
        if constexpr (WITH_PH2 && !ANY && L_ < K) ph2_pl<R, K, MODE, FULL, L_>(ra < kRefPhys, physbit(pb, ra < kRefPhys ? rb : ra), tp, flags, a, l, q, accp, acc_add); \
        break;
        VQC_PH2PL(0) VQC_PH2PL(1) VQC_PH2PL(2) VQC_PH2PL(3) VQC_PH2PL(4)
#undef VQC_PH2PL
    case DC_PH2_PP:
        if constexpr (WITH_PH2 && !ANY)
            ph2_pp<R, K, MODE, FULL>((int)physbit(pb, ra) + 2 * (int)physbit(pb, rb), tp, flags, a, l, q,
                                     accp, acc_add);
        break;
    default:
        break;
    }
}

// Run ops [ob, oe) of a stage (forward: in order; backward: reversed).  The
// descriptor is read when the op starts: keeping a prefetched one live across
// the dispatch switch costs more registers than the load latency it hides.
template <typename R, int K, int MODE, bool FULL, bool WITH_PH2 = true, int EW = EntryWords<R>::value>
__device__ __forceinline__ void run_ops(const DOp* ops, int ob, int oe, uint32_t pb,
                                        C2<R> (&a)[1 << K], C2<R> (&l)[1 << K], const R* sh_tab,
                                        const R* ps_tab, R* acc, const Geo& q, int lane,
                                        int warp_in_group, bool acc_add = false) {
    const uint2* op2 = reinterpret_cast<const uint2*>(ops);
    if (MODE == 0) {
        for (int o = ob; o < oe; ++o)
            apply_op<R, K, MODE, FULL, WITH_PH2, EW>(vqc_ld(op2 + o), pb, a, l, sh_tab, ps_tab, acc, q, lane,
                                          warp_in_group, acc_add);
    } else {
        for (int o = oe - 1; o >= ob; --o)
            apply_op<R, K, MODE, FULL, WITH_PH2, EW>(vqc_ld(op2 + o), pb, a, l, sh_tab, ps_tab, acc, q, lane,
                                          warp_in_group, acc_add);
    }
}

// lam = O psi on the block, O = sum_j gE_j Z_j (diagonal): the sign of Z_j comes
// from local bit j of r for active qubits and from the block base pb otherwise.
template <typename R, int K, typename GI>
__device__ __forceinline__ void lambda_init(const DStage* sp, uint32_t pb, const GI* gb, int n,
                                            const C2<R> (&a)[1 << K], C2<R> (&l)[1 << K]) {
    R ge_loc[K];
    R cst = 0;
    uint32_t actmask = 0;
#pragma unroll
    for (int j = 0; j < K; ++j) {
        const int aq = vqc_ld(&sp->active[j]);
        actmask |= 1u << aq;
        ge_loc[j] = as_r<R>(gb[aq]);
    }
    for (int j = 0; j < n; ++j)
        if (!((actmask >> j) & 1)) cst += ((pb >> j) & 1u) ? -as_r<R>(gb[j]) : as_r<R>(gb[j]);
#pragma unroll
    for (int r = 0; r < (1 << K); ++r) {
        R o = cst;
#pragma unroll
        for (int j = 0; j < K; ++j) o += ((r >> j) & 1) ? -ge_loc[j] : ge_loc[j];
        l[r] = cm<R>(o * a[r].x, o * a[r].y);
    }
}

// Adds this block's contributions to E_j = sum (-1)^{bit j} |a|^2 for qubits
// j < NV into ez[j] (a qubit outside the block contributes +-(block norm) by
// its bit in pb; entries j >= n stay untouched and are never read).
template <typename R, int K, int NV>
__device__ __forceinline__ void expz_accum(const DStage* sp, uint32_t pb, const C2<R> (&a)[1 << K],
                                           R (&ez)[NV]) {
    R ptot = 0;
    R dloc[K];
#pragma unroll
    for (int j = 0; j < K; ++j) dloc[j] = 0;
#pragma unroll
    for (int r = 0; r < (1 << K); ++r) {
        const R pr = fma(a[r].x, a[r].x, a[r].y * a[r].y);
        ptot += pr;
#pragma unroll
        for (int j = 0; j < K; ++j) dloc[j] += ((r >> j) & 1) ? -pr : pr;
    }
    uint32_t actmask = 0;
    int aq[K];
#pragma unroll
    for (int j = 0; j < K; ++j) {
        aq[j] = vqc_ld(&sp->active[j]);
        actmask |= 1u << aq[j];
    }
#pragma unroll
    for (int j = 0; j < NV; ++j) {
        R val = ((pb >> j) & 1u) ? -ptot : ptot;
#pragma unroll
        for (int k = 0; k < K; ++k) val = aq[k] == j ? dloc[k] : val;
        ez[j] += val;
    }
}

// Sum NV values over the 32 lanes of a warp (reduce-scatter butterfly, NV - 1
// + log2(32 / NV) shuffles).  Returns the value index this lane ends up with;
// v[0] then holds that value's warp sum in every lane whose bits below the
// scatter bits are zero (and in their partners).
template <typename R, int NV>
__device__ __forceinline__ int warp_reduce_scatter(R (&v)[NV], int lane) {
    int idx = 0;
    int m = 16;
#pragma unroll
    for (int w = NV; w > 1; w >>= 1, m >>= 1) {
        const int u = (lane & m) ? 1 : 0;
        const int h = w >> 1;
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const R send = u ? v[i] : v[i + h];
            const R keep = u ? v[i + h] : v[i];
            v[i] = keep + shx<R>(send, m, 0xffffffffu);
        }
        idx = 2 * idx + u;
    }
#pragma unroll
    for (; m >= 1; m >>= 1) v[0] += shx<R>(v[0], m, 0xffffffffu);
    return idx;
}

// Gradient terms of one accumulator slot (summed over the wg per-warp
// partials at ap): a phase op's scalar, or Im Tr(W_j P_j W_j^dag rho) for each
// parametrised constituent j of a run.  Writes out[term].
template <typename R, typename XI, typename WI, typename O>
__device__ void acc_terms(const DAcc& ac, const DEntry& e, const R* ap, int wg,
                          const DConst* consts, const XI* xg, const WI* w, const R* cang,
                          const R* cmat, O* out) {
    if (ac.kind == 1) {
        R sum = 0;
        for (int k2 = 0; k2 < wg; ++k2) sum += ap[k2 * 8];
        out[consts[e.cfirst].term] = as_out<O>(sum);
        return;
    }
    R vx = 0, vy = 0, vz = 0;
    for (int k2 = 0; k2 < wg; ++k2) {
        vx += ap[k2 * 8 + 0];
        vy += ap[k2 * 8 + 1];
        vz += ap[k2 * 8 + 2];
    }
    // The accumulator holds (tx, ty, tz) of rho's traceless anti-Hermitian part
    // rho' = (i/2)(tx X + ty Y + tz Z).  term_j = Im Tr(W_j P_j W_j^dag rho) =
    // Im Tr(P_j rho_j) = the P_j component of rho_j = W_j^dag rho' W_j, carried
    // from the last constituent backwards: rho' <- U^dag rho' U after each one.
    // For U = exp(-i t P / 2) that turns (tx, ty, tz) by the full angle t about
    // P's axis; a scalar phase leaves it; a constant 2x2 goes through its matrix.
    for (int c = e.ccount - 1; c >= 0; --c) {
        const DConst cn = consts[e.cfirst + c];
        if (cn.term >= 0) out[cn.term] = as_out<O>(cn.kind == CK_RX ? vx : cn.kind == CK_RY ? vy : vz);
        if (c == 0) break;
        if (cn.kind == CK_RX || cn.kind == CK_RY || cn.kind == CK_RZ) {
            R sn, co;
            sc(angle_of<R>(cn.src0, cn.idx0, xg, w, cang), &sn, &co);
            if (cn.kind == CK_RX) {
                const R y2 = vy * co + vz * sn, z2 = vz * co - vy * sn;
                vy = y2; vz = z2;
            } else if (cn.kind == CK_RY) {
                const R x2 = vx * co - vz * sn, z2 = vz * co + vx * sn;
                vx = x2; vz = z2;
            } else {
                const R x2 = vx * co + vy * sn, y2 = vy * co - vx * sn;
                vx = x2; vy = y2;
            }
        } else if (cn.kind == CK_CONST) {
            const R h = R(0.5);
            M2<R> rho;
            rho.a = cm<R>(0, h * vz); rho.b = cm<R>(h * vy, h * vx);
            rho.c = cm<R>(-h * vy, h * vx); rho.d = cm<R>(0, -h * vz);
            const M2<R> u = constituent<R>(cn, xg, w, cang, cmat);
            rho = mmul<R>(mdag<R>(u), mmul<R>(rho, u));
            // Im Tr(X rho) = Im r01 + Im r10, Im Tr(Y rho) = Re r01 - Re r10,
            // Im Tr(Z rho) = Im r00 - Im r11
            vx = rho.b.y + rho.c.y;
            vy = rho.b.x - rho.c.x;
            vz = rho.a.y - rho.d.y;
        }
    }
}


// Launch-geometry self-check (kernel side): the host derives the block size,
// the sample groups and the register blocks from one plan; a launch whose
// numbers disagree records `code` in the plan's error word (read back by
// vqc_sync_check) and does no work.  Uniform over the grid: every thread takes
// the same branch.
__device__ __forceinline__ bool geometry_bad(bool bad, unsigned* err, unsigned code) {
    if (bad && threadIdx.x == 0 && err) atomicOr(err, code);
    return bad;
}
enum : unsigned { kErrSweepGeometry = 1u, kErrPassGeometry = 2u, kErrClusterGeometry = 4u };

// out[c] = sum over rows r of part[r * cols + c]: one block per column,
// fixed strided partial sums, then a fixed-shape tree (deterministic).
template <typename R>
__global__ void __launch_bounds__(256) reduce_cols(const R* part, int rows, int cols, R* out) {
    __shared__ R buf[256];
    const int c = blockIdx.x;
    grid_dep_wait();
    grid_dep_launch();
    R s = 0;
    for (int r = threadIdx.x; r < rows; r += 256) s += part[(size_t)r * cols + c];
    buf[threadIdx.x] = s;
    __syncthreads();
    for (int w = 128; w >= 1; w >>= 1) {
        if (threadIdx.x < w) buf[threadIdx.x] += buf[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[c] = buf[0];
}

}  // namespace vqc
