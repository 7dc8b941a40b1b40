// capi.cu -- the C ABI declared in include/vqc.h: plan lifetime, launch
// geometry, workspace layout and kernel launches.  No exception crosses the
// ABI; every entry point returns a vqc_status and records a thread-local
// message on failure.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <initializer_list>
#include <map>
#include <memory>
#include <mutex>
#include <new>
#include <set>
#include <string>
#include <vector>

#include "engine.h"
#include "kernels.h"
#include "pass.cuh"
#include "sweep.cuh"

namespace vqc {
namespace {
// Launch geometry depends only on (plan, mode, batch, device): cache it so a
// call does not repeat the attribute and occupancy queries.
struct GeoKey {
    const void* plan;
    int mode, batch, dev, hbm, arith;
    bool operator<(const GeoKey& o) const {
        if (arith != o.arith) return arith < o.arith;
        if (plan != o.plan) return plan < o.plan;
        if (mode != o.mode) return mode < o.mode;
        if (batch != o.batch) return batch < o.batch;
        if (dev != o.dev) return dev < o.dev;
        return hbm < o.hbm;
    }
};
}  // namespace
}  // namespace vqc

namespace vqc {
namespace {

thread_local std::string g_err;

vqc_status fail(vqc_status s, const std::string& msg) {
    g_err = msg;
    return s;
}

vqc_status cuda_fail(cudaError_t e, const char* what) {
    return fail(VQC_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

#define VQC_CUDA(call)                                          \
    do {                                                        \
        cudaError_t e_ = (call);                                \
        if (e_ != cudaSuccess) return cuda_fail(e_, #call);     \
    } while (0)

struct DevInfo {
    int sms = 0, smem_optin = 0, smem_sm = 0, smem_reserved = 0;
    bool ok = false;
};

std::mutex g_mu;
std::vector<DevInfo> g_dev;

vqc_status device_info(int dev, DevInfo& out) {
    std::lock_guard<std::mutex> lk(g_mu);
    if ((int)g_dev.size() <= dev) g_dev.resize(dev + 1);
    if (!g_dev[dev].ok) {
        VQC_CUDA(cudaDeviceGetAttribute(&g_dev[dev].sms, cudaDevAttrMultiProcessorCount, dev));
        VQC_CUDA(cudaDeviceGetAttribute(&g_dev[dev].smem_optin,
                                        cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
        VQC_CUDA(cudaDeviceGetAttribute(&g_dev[dev].smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev));
        VQC_CUDA(cudaDeviceGetAttribute(&g_dev[dev].smem_reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev));
        g_dev[dev].ok = true;
    }
    out = g_dev[dev];
    return VQC_OK;
}

// Let `fn` take up to the device's opt-in shared memory per CTA, once per
// (kernel, device).  The attribute is per kernel, not per launch geometry:
// setting it to each geometry's own need would let a later, smaller geometry of
// the same kernel (another plan, batch or environment setting) lower it below a
// cached larger geometry's need, whose launch would then fail.
std::mutex g_smem_attr_mu;
std::set<std::pair<const void*, int>> g_smem_attr_done;

vqc_status allow_max_smem(const void* fn, int dev, int smem_optin) {
    std::lock_guard<std::mutex> lk(g_smem_attr_mu);
    if (g_smem_attr_done.count({fn, dev})) return VQC_OK;
    VQC_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_optin));
    g_smem_attr_done.insert({fn, dev});
    return VQC_OK;
}

// mode 2: the backward with the forward sweep and E inside (vqc_forward_backward)
// factored: double-float stages of factored runs; rounds: native complex128 ones in rounds
const void* kernel_ptr(int dtype, bool dfloat, int mode, int K, bool full, bool ph2,
                       bool factored, bool rounds) {
    // complex64 sweeps of plans without CRZ / RZZ: the instantiations without
    // the phase cases (fewer spills)
    if (!dfloat && dtype == VQC_C64 && !ph2)
        return mode == 0 ? sweep_ptr_f32_fwd_nph(K, full)
             : mode == 1 ? sweep_ptr_f32_bwd_nph(K, full) : sweep_ptr_f32_fused_nph(K, full);
    if (dfloat)
        return mode == 2 ? sweep_ptr_dd_fused(K, full, factored)
             : mode == 0 ? sweep_ptr_dd_fwd(K, full, factored) : sweep_ptr_dd_bwd(K, full, factored);
    if (mode == 2) return dtype == VQC_C64 ? sweep_ptr_f32_fused(K, full)
                                           : sweep_ptr_f64_fused(K, full, rounds);
    if (full) {
        if (dtype == VQC_C64) return mode == 0 ? sweep_ptr_f32_fwd(K) : sweep_ptr_f32_bwd(K);
        return mode == 0 ? sweep_ptr_f64_fwd(K, rounds) : sweep_ptr_f64_bwd(K, rounds);
    }
    if (dtype == VQC_C64) return mode == 0 ? sweep_ptr_f32_fwd_small(K) : sweep_ptr_f32_bwd_small(K);
    return mode == 0 ? sweep_ptr_f64_fwd_small(K) : sweep_ptr_f64_bwd_small(K);
}

size_t align16(size_t v) { return (v + 15) & ~size_t(15); }
size_t align256(size_t v) { return (v + 255) & ~size_t(255); }

// Launch geometry of one call.
struct Launch {
    const Schedule* s = nullptr;        // cluster path
    const FrameSchedule* f = nullptr;   // resident path
    int K = 0, T = 0, S = 0, block = 0, grid = 0, nunits = 0, wg = 1;
    size_t smem = 0;
    size_t smem_states = 0;   // resident: the same of a launch that writes final states
    int sm_sh = 0, sm_ps = 0, sm_psi = 0, sm_lam = 0, sm_acc = 0, sm_terms = 0, sm_dw = 0,
        sm_red = 0, sm_plan = 0, sm_w = 0, sm_xg = 0, sm_io = 0, sm_dg = 0, ndg = 0;
    int cl = 0, sm_ecl = 0;   // cluster path: log2 CTAs per sample, <Z> gather area
    bool factored = false;    // double-float: stages of factored runs
    bool plan_smem = false, tab_smem = true;   // resident: the plan's schedule / table data in shared memory
    const void* fn = nullptr;
};

int env_int(const char* name, int dflt) {
    const char* v = std::getenv(name);
    return v && *v ? std::atoi(v) : dflt;
}

int cta_threads() {
    const int t = env_int("VQC_CTA_THREADS", 128);
    return t >= 32 && t <= 512 ? t : 128;
}

// Shared memory to ask for so that a grid of one wave spreads over the SMs.  A kernel that
// is scheduled while the one before it still runs (launch) finds free shared memory
// unevenly, and SMs then take more CTAs than their share while others stay idle: 12 qubits
// x 100, RY x 8 layers, backward after forward 171 us, 110 spread; native complex128, 16
// qubits x 3, step, 980 / 745 us, 11 qubits x 100, 1.8 times.  So no SM can hold more than
// ceil(grid / SMs), as far as that asks for at most twice the memory -- for several CTAs
// an SM at most 1.3 times, since more keeps the next kernel's CTAs out (9 qubits x 1600,
// complex128 step 0.8 times), and not where a forward writes states, whose backward
// comes next (10 qubits x 1600, re-uploading x 4, saved, 145 us spread, 120 not).  Grids of half the SMs find as many free ones, and the larger
// request itself took time (double-float, 9 qubits x 3, step 316 -> 339 us).
size_t spread_smem(size_t smem, int grid, int per_sm, const DevInfo& di) {
    const int share = (grid + di.sms - 1) / di.sms;
    if (share >= per_sm || 2 * grid <= di.sms || di.smem_sm <= 0) return smem;
    const size_t pad = align16((size_t)di.smem_sm / (share + 1) - di.smem_reserved + 1);
    const double most = (share == 1 ? 2.0 : 1.3) * (double)smem;
    return pad > smem && (double)pad <= most && pad <= (size_t)di.smem_optin ? pad : smem;
}

// The environment switches, read once per call from outside (a call asks for some of
// them dozens of times, and each getenv walks the environment).
struct Env {
    int k_fwd = 0, k_bwd = 0, cta = 128;
    bool plan_smem = true, force = false, hbm = false, cluster = false;
};
thread_local Env t_env;

// The arithmetic that launch geometry is worked out for: the plan's own (-1), or native
// (0) or double-float (1) for a complex128 plan.  A workspace holds either of them, so
// that plans of the two types can share one (vqc_workspace_bytes).
thread_local int t_arith = -1;
struct ArithScope {
    const int saved = t_arith;
    explicit ArithScope(int a) { t_arith = a; }
    ~ArithScope() { t_arith = saved; }
};
bool dfloat_of(const HostPlan& p) { return t_arith < 0 ? p.dfloat : p.dtype == VQC_C128 && t_arith == 1; }

thread_local int t_env_depth = 0;
struct EnvScope {
    EnvScope() {
        if (t_env_depth++) return;
        Env e;
        e.k_fwd = env_int("VQC_FORCE_K_FWD", 0);
        e.k_bwd = env_int("VQC_FORCE_K_BWD", 0);
        e.cta = cta_threads();
        e.plan_smem = env_int("VQC_PLAN_IN_SMEM", 1) != 0;
        if (const char* f = std::getenv("VQC_FORCE_PATH")) {
            e.force = true;
            e.hbm = !std::strcmp(f, "hbm");
            e.cluster = !std::strcmp(f, "cluster");
        }
        t_env = e;
    }
    ~EnvScope() { --t_env_depth; }
};

// Launch with programmatic stream serialisation: the kernel may be scheduled
// while the previous kernel in the stream finishes, and waits for it (every
// kernel calls grid_dep_wait() before touching caller memory), which hides most
// of the launch gap between the back-to-back kernels of one call and between
// consecutive calls.  VQC_PDL=0 turns it off (plain stream order).
bool use_pdl() {
    static const bool pdl = env_int("VQC_PDL", 1) != 0;
    return pdl;
}
cudaError_t launch(const void* fn, dim3 grid, dim3 block, void** args, size_t smem,
                   cudaStream_t stream) {
    if (!use_pdl()) return cudaLaunchKernel(fn, grid, block, args, smem, stream);
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelExC(&cfg, fn, args);
}

// Pick the register-block size: the largest K that still gives the batch
// enough threads to cover every SM's schedulers (SMs x 4 warps), but not below
// 3 (a block of 8 amplitudes) where the circuit allows it.  Of the forced sizes
// (VQC_FORCE_K_*: RX RY RZ layers, CX ring, complex64; 8 qubits x 100, 1024 and 8192,
// 10 x 251, 12 x 100 and 4096; forward, one call, saved) this choice was the fastest
// everywhere but in the 8-qubit x 8192 one-call step (156 us, 136 with 3 / 3): smaller
// blocks add stages (shared-memory round trips and barriers) faster than the extra warps
// hide latency (12 x 4096 step 1.67 ms with 5 / 4, 1.73 with 4 / 4, 2.36 with 3 / 3).
int choose_k(const HostPlan& p, int mode, int B, int sms, bool any_size = false) {
    const int forced = mode == 0 ? t_env.k_fwd : t_env.k_bwd;
    if (forced > 0 && find_frame(p, mode, VQC_PATH_RESIDENT, forced)) return forced;
    int kmax = 0;
    for (const auto& s : p.frames)
        if (s.mode == mode && s.path == VQC_PATH_RESIDENT) kmax = std::max(kmax, s.K);
    if (kmax == 0) return 0;
    // Double-float circuits with CRZ / RZZ: blocks of 8 where threads allow (ph2_any; 11-qubit
    // QAOA x 1600, 8 layers, forward 1.57 ms, 2.40 with blocks of 16).
    // any_size: without that rule, where such a launch does not fit.
    if (!any_size && dfloat_of(p) && p.has_ph2 && kmax > 3 && find_frame(p, mode, VQC_PATH_RESIDENT, 3)) kmax = 3;
    const int kmin = std::min(kmax, 3);
    const double want = (double)sms * 4 * 32;
    int K = kmax;
    while (K > kmin && (double)B * std::ldexp(1.0, p.n - K) < want && find_frame(p, mode, VQC_PATH_RESIDENT, K - 1))
        --K;
    return K;
}

// Double-float resident sweeps with factored stages: circuits without CRZ / RZZ (whose
// stages take 2x2 updates; 9-qubit QAOA x 1600, 8 layers, forward 1036 us with the
// factors beside them, 442 without), except small forwards of few stages, where the
// factors and diagonals of a call, a chain of FP64 operations, take longer than they
// save (RX RY RZ layers, CX ring, forward, factored / not: 8 qubits x 100, 1 layer 26 /
// 20 us, 8 layers 74 / 67; 9 x 100, 8 layers 61 / 62; 11 x 100, 1 layer 45 / 36; 11 x 1600,
// 1 layer 180 / 211; 12 x 100, 1 layer 46 / 53).
bool factors_pay(const HostPlan& p, int mode, int B, const FrameSchedule& f, int sms) {
    if (p.has_ph2) return false;
    const bool small = p.n <= 11 && (double)B * std::ldexp(1.0, p.n) <= sms * 8192.0;
    return mode == 1 || f.passes[0].ndg == 0 || !small || (p.n > 8 && f.stages.size() >= 12);
}

// Diagonal tables of a pass: of two-local phases, and double-float's own (complex128
// schedules hold both).
int diagonal_tables(const HostPlan& p, const FrameSchedule& s, size_t pass) {
    return dfloat_of(p) ? s.passes[pass].ndg : s.phase_tables[pass];
}

// The resident launch with blocks of 2^K amplitudes; lean: without diagonal tables, native
// complex128 by the op switch, double-float without the runs' factors.
vqc_status plan_launch_as(const HostPlan& p, int launch_mode, int B, int K, bool lean, int dev, const DevInfo& di,
                          Launch& L) {
    // mode 2 (fused) has the backward's schedule and layout, its own kernel
    const int mode = launch_mode == 2 ? 1 : launch_mode;
    vqc_status st;
    L = Launch();
    L.K = K;
    L.f = L.K ? find_frame(p, mode, VQC_PATH_RESIDENT, L.K) : nullptr;
    if (!L.f)
        return fail(VQC_ERR_UNSUPPORTED, "no resident schedule for this circuit (n = " +
                                             std::to_string(p.n) + ")");
    const bool dbl = p.dtype == VQC_C128;
    const size_t rs = dbl ? 8 : 4, cs = 2 * rs;
    L.T = 1 << (p.n - L.K);   // one register block per thread (n - K <= 9)
    L.wg = L.T > 32 ? L.T / 32 : 1;
    // Shared memory: a fixed part per CTA and a part per resident sample.
    const size_t dim = (size_t)1 << p.n;
    const size_t io = (size_t)(mode == 0 ? 8 : 4) << L.K;   // slot offsets of the state copies
    const bool factored = L.factored = dfloat_of(p) && !lean && L.T >= 32 && factors_pay(p, mode, B, *L.f, di.sms);
    const size_t ew = entry_reals(dbl, factored) / (mode == 0 && !dbl ? 2 : 1);   // ResidentWords
    const size_t fixed = align16((size_t)p.n_sh * ew * rs) + align16(mode == 1 ? (size_t)p.num_w * rs : 0) +
                         align16((size_t)p.num_w * rs) + io +
                         (mode == 0 ? 2 : 3) * 16;   // rounding up: red, xg, the backward's terms
    L.ndg = L.T >= 32 && dbl && !lean && (dfloat_of(p) ? factored : p.has_ph2) ? diagonal_tables(p, *L.f, 0) : 0;
    const size_t dgb = ((size_t)L.ndg << L.K) * cs;
    const size_t per_sample = dgb + (size_t)p.n_ps * ew * rs + dim * cs * (mode == 1 ? 2 : 1) +
                              (size_t)(p.num_x + p.n) * rs +
                              (mode == 1 ? p.accs.size() * L.wg * 8 * rs + p.term_src.size() * rs : 0) +
                              (size_t)L.wg * p.n * rs;
    // samples per CTA: groups up to VQC_CTA_THREADS (default 128) threads
    int S = std::max(1, t_env.cta / L.T);
    if ((size_t)di.smem_optin > fixed) {
        size_t fit = ((size_t)di.smem_optin - fixed) / per_sample;
        S = (int)std::min<size_t>((size_t)S, fit);
    } else {
        S = 0;
    }
    if (S < 1)
        return fail(VQC_ERR_UNSUPPORTED,
                    "state does not fit in shared memory on the resident path (" +
                        std::to_string(fixed + per_sample) + " > " +
                        std::to_string(di.smem_optin) + " bytes)");
    // Groups smaller than a warp fill whole warps when the CTA spans more than one.
    if (L.T < 32 && S * L.T > 32) S -= S % (32 / L.T);
    L.S = S;
    L.block = L.S * L.T;
    if (L.block > kSweepMaxThreads)
        return fail(VQC_ERR_UNSUPPORTED, "thread group too large for this kernel");
    size_t off = 0;
    auto take = [&](size_t bytes) {
        size_t o = off;
        off = align16(off + bytes);
        return (int)o;
    };
    take((size_t)L.S * dim * cs);   // psi at offset 0
    L.sm_lam = take(mode == 1 ? (size_t)L.S * dim * cs : 0);
    L.sm_sh = take((size_t)p.n_sh * ew * rs);
    L.sm_ps = take((size_t)L.S * p.n_ps * ew * rs);
    L.sm_io = take(io);
    L.sm_dg = take(L.S * dgb);
    L.sm_acc = take(mode == 1 ? (size_t)L.S * p.accs.size() * L.wg * 8 * rs : 0);
    L.sm_terms = take(mode == 1 ? (size_t)L.S * p.term_src.size() * rs : 0);
    L.sm_dw = take(mode == 1 ? (size_t)p.num_w * rs : 0);
    L.sm_red = take((size_t)L.S * L.wg * p.n * rs);   // <Z> partials (forward, or recompute with E)
    L.sm_w = take((size_t)p.num_w * rs);
    L.sm_xg = take((size_t)L.S * (p.num_x + p.n) * rs);
    L.fn = kernel_ptr(p.dtype, dfloat_of(p), launch_mode, L.K, L.T >= 32, p.has_ph2, factored, !lean);
    if (!L.fn) return fail(VQC_ERR_UNSUPPORTED, "kernel not instantiated for this K");
    st = allow_max_smem(L.fn, dev, di.smem_optin);
    if (st != VQC_OK) return st;
    L.nunits = (B + L.S - 1) / L.S;
    // The plan's table data and this schedule go to shared memory when they fit; the
    // table data, which only the table evaluation reads, stays out when that lets more
    // CTAs onto an SM and the batch has units for them (13-qubit random circuit x 256,
    // 18 KB of table data: one wave of two CTAs an SM instead of two of one).
    const size_t tab = align16(p.dev_tab_end - p.dev_tab_begin), sched = L.f->dev_region_end - L.f->dev_region_begin;
    auto per_sm_with = [&](size_t extra, int& per_sm) -> vqc_status {
        per_sm = 0;
        if (off + extra > (size_t)di.smem_optin) return VQC_OK;
        VQC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, L.fn, L.block, off + extra));
        return VQC_OK;
    };
    int per_sm = 0, with_sched = 0;
    if (t_env.plan_smem) {
        st = per_sm_with(tab + sched, per_sm);
        if (st != VQC_OK) return st;
        L.plan_smem = L.tab_smem = per_sm > 0;
        if (L.nunits > per_sm * di.sms) {
            st = per_sm_with(sched, with_sched);
            if (st != VQC_OK) return st;
            if (with_sched > per_sm) {
                per_sm = with_sched;
                L.plan_smem = true;
                L.tab_smem = false;
            }
        }
    }
    L.sm_plan = L.plan_smem ? take((L.tab_smem ? tab : 0) + sched) : 0;
    L.smem = off;
    if (L.smem > (size_t)di.smem_optin)
        return fail(VQC_ERR_UNSUPPORTED, "shared-memory layout exceeds the per-CTA limit");
    if (!L.plan_smem) {
        st = per_sm_with(0, per_sm);
        if (st != VQC_OK) return st;
    }
    if (per_sm < 1) return fail(VQC_ERR_UNSUPPORTED, "kernel cannot be resident with this geometry");
    L.grid = std::max(1, std::min(L.nunits, per_sm * di.sms));
    L.smem_states = L.smem;
    L.smem = spread_smem(L.smem, L.grid, per_sm, di);
    if (L.grid <= di.sms) L.smem_states = L.smem;
    return VQC_OK;
}

// Native complex128 resident sweeps: whether stages in rounds are the faster ones.  They
// are for circuits without diagonal ops, and where a round that has phases has two or
// more of them to collect (RZZ rings, 2.5 to 4: 9 qubits x 1600, one layer, forward 0.75 of
// the op switch's time, 8 to 13 qubits 0.9 to 1.0).  With fewer (random circuits, 1.3 to
// 1.8; step, 9 qubits x 100, 500 gates: 1.92 ms, 1.76 by the switch) or signs only (CZ
// rings, forward 1.02 to 1.08 of the switch's time) the walk over the groups costs more.
bool rounds_pay(const FrameSchedule& f) {
    int phases = 0, groups = 0, signs = 0;
    for (const FSeg& s : f.segs) {
        int here = 0;
        for (int i = s.op_begin; i < s.run_begin; ++i) ++(f.ops[i].code >= DC_PH2_LL ? here : signs);
        phases += here;
        groups += here > 0;
    }
    return phases ? phases >= 2 * groups : signs == 0;
}

// Of a factored launch f that fits and its lean form l, whether l is the faster one.  At 8
// and 9 qubits a sample's updates are few beside its factors and diagonals, FP64 work of
// every per-sample run, and its larger tables.  So l where these cost f a wave of CTAs
// (9 qubits x 1600, re-uploading, 8 layers, forward: 544 us factored, 338 lean; weights
// only, 303 / 347: kept but at 8 qubits), and backward, few stages, beyond a CTA per SM,
// where most runs depend on the sample (8 qubits x 1600, 2 layers 227 / 184, 4 layers 306 /
// 388; 9 qubits, re-uploading, 2 layers 393 / 345; one layer 209 / 215, but 232 behind a
// lean forward).  From 10 qubits on f was faster everywhere (1.06 to 1.6 times).
bool lean_pays(const HostPlan& p, int mode, const Launch& f, const Launch& l, int sms) {
    if (p.n > 9 || f.ndg == 0) return false;
    auto waves = [](const Launch& x) { return (x.nunits + x.grid - 1) / x.grid; };
    const bool sample = 2 * p.n_ps >= p.n_runs;
    if (waves(l) < waves(f) && (sample || (p.n == 8 && waves(f) >= 2 * waves(l)))) return true;
    return mode == 1 && f.nunits > sms && f.f->stages.size() < 8 && (p.n_ps == p.n_runs || (sample && f.S * p.n_ps >= 32));
}

// The launch of the chosen block size; where a complex128 layout does not fit a CTA, the
// lean one (double-float, 12 qubits x 7 layers of RX RY RZ, backward: 245 KB factored, 230
// with 2x2 updates), then double-float's blocks of 16, with fewer warps to keep partials for.
vqc_status plan_launch_uncached(const HostPlan& p, int launch_mode, int B, Launch& L) {
    const int mode = launch_mode == 2 ? 1 : launch_mode;
    int dev = 0;
    VQC_CUDA(cudaGetDevice(&dev));
    DevInfo di;
    vqc_status st = device_info(dev, di);
    if (st != VQC_OK) return st;
    const int K = choose_k(p, mode, B, di.sms);
    const FrameSchedule* f = K ? find_frame(p, mode, VQC_PATH_RESIDENT, K) : nullptr;
    const bool by_switch = f && p.dtype == VQC_C128 && !dfloat_of(p) && !rounds_pay(*f);
    st = plan_launch_as(p, launch_mode, B, K, by_switch, dev, di, L);
    if (st == VQC_OK && L.factored) {
        Launch l;
        if (plan_launch_as(p, launch_mode, B, K, true, dev, di, l) == VQC_OK && lean_pays(p, mode, L, l, di.sms)) L = l;
    }
    if (st == VQC_OK || p.dtype != VQC_C128 || K == 0 || by_switch) return st;
    const std::string why = g_err;   // of the layout that the choice asked for
    for (int k : {K, choose_k(p, mode, B, di.sms, true)})
        if (plan_launch_as(p, launch_mode, B, k, true, dev, di, L) == VQC_OK) return VQC_OK;
    return fail(st, why);
}

std::mutex g_geo_mu;
std::map<GeoKey, Launch> g_launch_cache;
std::map<GeoKey, Launch> g_cluster_cache;   // cluster-path geometry (forget_plan clears it too)
std::map<GeoKey, size_t> g_workspace_cache;  // complex128: of both arithmetics

GeoKey geo_key(const HostPlan& p, int mode, int B, int hbm) {
    int dev = -1;
    cudaGetDevice(&dev);
    // environment switches that change the geometry are part of the key
    const int env = t_env.k_fwd * 1000 + t_env.k_bwd * 10 + (t_env.plan_smem ? 1 : 0) + t_env.cta * 1000000;
    return GeoKey{&p, mode, B, dev, hbm * 100000 + env, t_arith};
}

vqc_status plan_launch(const HostPlan& p, int mode, int B, Launch& L) {
    const GeoKey k = geo_key(p, mode, B, 0);
    {
        std::lock_guard<std::mutex> lk(g_geo_mu);
        auto it = g_launch_cache.find(k);
        if (it != g_launch_cache.end()) {
            L = it->second;
            return VQC_OK;
        }
    }
    vqc_status st = plan_launch_uncached(p, mode, B, L);
    if (st == VQC_OK && p.dbuf) {   // (without a device copy its layout is not known)
        std::lock_guard<std::mutex> lk(g_geo_mu);
        g_launch_cache[k] = L;
    }
    return st;
}

template <typename R>
void fill_plan_args(const HostPlan& p, const Launch& L, KArgs<R>& a) {
    const char* base = static_cast<const char*>(p.dbuf);
    if (L.f) {
        a.ops = reinterpret_cast<const DOp*>(base + L.f->dev_ops);
        a.fstages = reinterpret_cast<const FStage*>(base + L.f->dev_stages);
        a.segs = reinterpret_cast<const FSeg*>(base + L.f->dev_segs);
        a.nsegs = (int)L.f->segs.size();
        a.fin = reinterpret_cast<const FFinal*>(base + L.f->dev_fin);
        a.nstages = (int)L.f->stages.size();
        for (int i = 0; i < p.n; ++i) {
            a.sin[i] = L.f->passes[0].sin[i];
            a.sout[i] = L.f->passes[0].sout[i];
        }
        a.sched_off = (int)L.f->dev_region_begin;
        a.sched_bytes = (int)(L.f->dev_region_end - L.f->dev_region_begin);
    } else {
        a.ops = reinterpret_cast<const DOp*>(base + L.s->dev_ops);
        a.stages = reinterpret_cast<const DStage*>(base + L.s->dev_stages);
        a.nstages = (int)L.s->stages.size();
        a.sched_off = (int)L.s->dev_region_begin;
        a.sched_bytes = (int)(L.s->dev_region_end - L.s->dev_region_begin);
    }
    a.entries = reinterpret_cast<const DEntry*>(base + p.dev_entries);
    a.ps_list = reinterpret_cast<const int32_t*>(base + p.dev_ps_list);
    a.sh_list = reinterpret_cast<const int32_t*>(base + p.dev_sh_list);
    a.consts = reinterpret_cast<const DConst*>(base + p.dev_consts);
    a.cmat = reinterpret_cast<const R*>(base + p.dev_cmat);
    a.cang = reinterpret_cast<const R*>(base + p.dev_cang);
    a.accs = reinterpret_cast<const DAcc*>(base + p.dev_accs);
    a.xocc_ptr = reinterpret_cast<const int32_t*>(base + p.dev_xocc_ptr);
    a.xocc = reinterpret_cast<const int32_t*>(base + p.dev_xocc);
    a.wocc_ptr = reinterpret_cast<const int32_t*>(base + p.dev_wocc_ptr);
    a.wocc = reinterpret_cast<const int32_t*>(base + p.dev_wocc);
    a.err = p.dev_error;
    a.n = p.n;
    a.K = L.K;
    a.tbits = p.n - L.K;
    a.G = p.G_swz;
    a.S = L.S;
    a.tpg = L.T;
    a.n_ps = p.n_ps;
    a.n_sh = p.n_sh;
    a.n_accs = (int)p.accs.size();
    a.n_ps = p.n_ps;
    a.n_terms = (int)p.term_src.size();
    a.Px = p.num_x;
    a.Pw = p.num_w;
    a.sm_sh = L.sm_sh; a.sm_ps = L.sm_ps; a.sm_psi = L.sm_psi; a.sm_lam = L.sm_lam;
    a.sm_acc = L.sm_acc; a.sm_terms = L.sm_terms; a.sm_dw = L.sm_dw; a.sm_red = L.sm_red;
    a.sm_w = L.sm_w; a.sm_xg = L.sm_xg; a.sm_io = L.sm_io; a.sm_dg = L.sm_dg; a.ndg = L.ndg;
    a.plan = static_cast<const unsigned char*>(p.dbuf);
    a.tab_off = (int)p.dev_tab_begin;
    a.tab_bytes = (int)(p.dev_tab_end - p.dev_tab_begin);
    a.sm_plan = L.sm_plan;
    a.plan_smem = L.plan_smem ? 1 : 0;
    a.tab_smem = L.tab_smem ? 1 : 0;
    a.cl = L.cl;
    a.sm_ecl = L.sm_ecl;
}

// Device buffer layout of a plan (all sections 16-byte aligned).
// Uploaded plans (their device error words are read by vqc_sync_check).
std::mutex g_plans_mu;
std::set<const HostPlan*> g_plans;

vqc_status upload(HostPlan& p) {
    const bool dbl = p.dtype == VQC_C128;
    std::vector<uint8_t> blob;
    auto put = [&](const void* src, size_t bytes) {
        size_t off = blob.size();
        blob.resize(align16(off + bytes), 0);
        if (bytes && src) std::memcpy(blob.data() + off, src, bytes);
        return off;
    };
    std::vector<int32_t> ps_list, sh_list;
    for (size_t i = 0; i < p.entries.size(); ++i)
        (p.entries[i].per_sample ? ps_list : sh_list).push_back((int32_t)i);
    // the kernels index lists by slot order, which is entry order within each list
    std::vector<double> cm_d = p.cmat, ca_d = p.cang;
    std::vector<float> cm_f(cm_d.begin(), cm_d.end()), ca_f(ca_d.begin(), ca_d.end());
    if (p.dfloat) {
        // double-float kernels read constants as (hi, lo) float pairs in the 8
        // bytes a double takes: hi = the double rounded to float, lo = the rest
        auto split = [](std::vector<double>& v) {
            for (double& d : v) {
                const float hi = (float)d, lo = (float)(d - (double)hi);
                std::memcpy(reinterpret_cast<char*>(&d), &hi, 4);
                std::memcpy(reinterpret_cast<char*>(&d) + 4, &lo, 4);
            }
        };
        split(cm_d);
        split(ca_d);
    }
    p.dev_entries = put(p.entries.data(), p.entries.size() * sizeof(DEntry));
    p.dev_ps_list = put(ps_list.data(), ps_list.size() * 4);
    p.dev_sh_list = put(sh_list.data(), sh_list.size() * 4);
    p.dev_consts = put(p.consts.data(), p.consts.size() * sizeof(DConst));
    p.dev_cmat = dbl ? put(cm_d.data(), cm_d.size() * 8) : put(cm_f.data(), cm_f.size() * 4);
    p.dev_cang = dbl ? put(ca_d.data(), ca_d.size() * 8) : put(ca_f.data(), ca_f.size() * 4);
    p.dev_accs = put(p.accs.data(), p.accs.size() * sizeof(DAcc));
    p.dev_xocc_ptr = put(p.xocc_ptr.data(), p.xocc_ptr.size() * 4);
    p.dev_xocc = put(p.xocc.data(), p.xocc.size() * 4);
    p.dev_wocc_ptr = put(p.wocc_ptr.data(), p.wocc_ptr.size() * 4);
    p.dev_wocc = put(p.wocc.data(), p.wocc.size() * 4);
    p.dev_tab_begin = p.dev_entries;
    p.dev_tab_end = blob.size();
    for (auto& s : p.scheds) {
        s.dev_region_begin = blob.size();
        s.dev_ops = put(s.ops.data(), s.ops.size() * sizeof(DOp));
        s.dev_stages = put(s.stages.data(), s.stages.size() * sizeof(DStage));
        s.dev_region_end = blob.size();
    }
    std::vector<int32_t> iota;   // 0, 1, ...: the indices of a pass's own tables (own_tables)
    for (const auto& s : p.frames)
        if (s.path == VQC_PATH_HBM)
            for (const auto& f : s.passes)
                while ((int)iota.size() < std::max({f.ps_count, f.sh_count, f.acc_count}))
                    iota.push_back((int32_t)iota.size());
    p.dev_iota = put(iota.data(), iota.size() * 4);
    for (auto& s : p.frames) {
        s.dev_region_begin = blob.size();
        s.dev_ops = put(s.ops.data(), s.ops.size() * sizeof(DOp));
        s.dev_stages = put(s.stages.data(), s.stages.size() * sizeof(FStage));
        s.dev_segs = put(s.segs.data(), s.segs.size() * sizeof(FSeg));
        s.dev_fin = put(&s.fin, sizeof(FFinal));
        s.dev_region_end = blob.size();
        s.dev_flips = put(s.flips.data(), s.flips.size() * sizeof(FFlip));
        // the passes copy their entries from the tables by slot
        std::vector<int32_t> slots;
        for (int32_t e : s.pass_entries) slots.push_back(p.entries[e].slot);
        s.dev_pass_entries = put(slots.data(), slots.size() * 4);
        s.dev_pass_accs = put(s.pass_accs.data(), s.pass_accs.size() * 4);
    }
    size_t err_off = put(nullptr, 16);
    blob.resize(align256(blob.size()), 0);
    VQC_CUDA(cudaGetDevice(&p.device));
    // (a call uploads the plan of every schedule, and its stream may be in capture: a copy
    // beside it, which the relaxed mode allows)
    cudaStreamCaptureMode mode = p.every ? cudaStreamCaptureModeRelaxed : cudaStreamCaptureModeGlobal;
    if (p.every) VQC_CUDA(cudaThreadExchangeStreamCaptureMode(&mode));
    void* d = nullptr;
    cudaStream_t s = nullptr;
    cudaError_t e = cudaMalloc(&d, blob.size());
    const bool room = e == cudaSuccess;
    if (!p.every) {
        if (room) e = cudaMemcpy(d, blob.data(), blob.size(), cudaMemcpyHostToDevice);
    } else {
        if (room) e = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
        if (e == cudaSuccess) e = cudaMemcpyAsync(d, blob.data(), blob.size(), cudaMemcpyHostToDevice, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (s) cudaStreamDestroy(s);
        VQC_CUDA(cudaThreadExchangeStreamCaptureMode(&mode));
    }
    if (!room) {
        (void)cudaGetLastError();
        return fail(VQC_ERR_OUT_OF_MEMORY, "cudaMalloc of the plan failed");
    }
    if (e != cudaSuccess) {
        cudaFree(d);
        return cuda_fail(e, "cudaMemcpy(plan)");
    }
    p.dbuf = d;
    p.dbytes = blob.size();
    p.dev_error = reinterpret_cast<unsigned*>(static_cast<char*>(d) + err_off);
    std::lock_guard<std::mutex> lk(g_plans_mu);
    g_plans.insert(&p);
    return VQC_OK;
}

// Workspace of a backward call: [0, 256) control block (reserved), then the
// per-CTA dw partials [grid, num_w].
size_t bwd_workspace(const HostPlan& p, const Launch& L) {
    const size_t rs = p.dtype == VQC_C128 ? 8 : 4;
    return 256 + align256((size_t)L.grid * std::max(p.num_w, 1) * rs);
}

// For a scratch of given size (a multiple of 256): a grid of fewer CTAs than the SMs
// hold, down to half, where its dw partials fit (any grid covers the batch).
void fit_grid(const HostPlan& p, size_t bytes, Launch& L) {
    const size_t row = (size_t)std::max(p.num_w, 1) * (p.dtype == VQC_C128 ? 8 : 4);
    const size_t rows = (bytes - 256) / row;
    if (rows < (size_t)L.grid && 2 * rows >= (size_t)L.grid) L.grid = (int)rows;
}

bool misaligned(const void* ptr, size_t a) {
    return (reinterpret_cast<uintptr_t>(ptr) & (a - 1)) != 0;
}

template <typename R>
vqc_status run(const HostPlan& p, int mode, int B, const void* x, const void* w, const void* psi0,
               const void* psi_final, const void* gE, void* E, void* state_out, void* dx, void* dw,
               void* ws, size_t ws_bytes, cudaStream_t stream, bool fit = false) {
    using C = C2<R>;
    Launch L;
    vqc_status st = plan_launch(p, mode, B, L);
    if (st != VQC_OK) return st;
    if (fit) fit_grid(p, ws_bytes, L);
    KArgs<R> a{};
    fill_plan_args<R>(p, L, a);
    a.B = B;
    a.nunits = L.nunits;
    a.x = static_cast<const R*>(x);
    a.w = static_cast<const R*>(w);
    a.psi0 = static_cast<const C*>(psi0);
    a.psi_final = static_cast<const C*>(psi_final);
    a.gE = static_cast<const R*>(gE);
    a.E = static_cast<R*>(E);
    a.state_out = static_cast<C*>(state_out);
    a.dx = static_cast<R*>(dx);
    a.dw = static_cast<R*>(dw);
    if (mode >= 1) {
        size_t need = bwd_workspace(p, L);
        if (!ws || ws_bytes < need || misaligned(ws, 256))
            return fail(VQC_ERR_WORKSPACE, "backward workspace must be >= " + std::to_string(need) +
                                               " bytes and 256-byte aligned");
        a.dw_part = reinterpret_cast<R*>(static_cast<char*>(ws) + 256);
    }
    void* args[] = {&a};
    VQC_CUDA(launch(L.fn, dim3(L.grid), dim3(L.block), args, state_out ? L.smem_states : L.smem, stream));
    if (mode >= 1 && dw && p.num_w > 0) {
        const R* part = a.dw_part;
        int rows = L.grid, cols = p.num_w;
        R* out = static_cast<R*>(dw);
        void* rargs[] = {&part, &rows, &cols, &out};
        VQC_CUDA(launch(reduce_cols_ptr(p.dtype == VQC_C128), dim3(cols), dim3(256), rargs,
                                  0, stream));
    }
    return VQC_OK;
}

// ---------------------------------------------------------------- cluster path

// One state per sample of a batch, as the passes keep it in HBM.
size_t hbm_state_bytes(const HostPlan& p, int B) {
    return align256((size_t)B * ((size_t)1 << p.n) * (p.dtype == VQC_C128 ? 16 : 8));
}

vqc_status plan_cluster(const HostPlan& p, int mode, int B, Launch& L) {
    const GeoKey k = geo_key(p, mode, B, 2);
    {
        std::lock_guard<std::mutex> lk(g_geo_mu);
        auto it = g_cluster_cache.find(k);
        if (it != g_cluster_cache.end()) {
            L = it->second;
            return VQC_OK;
        }
    }
    L = Launch();
    L.s = find_cluster_schedule(p, mode);
    if (!L.s) return fail(VQC_ERR_UNSUPPORTED, "no cluster schedule for this circuit");
    int dev = 0;
    VQC_CUDA(cudaGetDevice(&dev));
    DevInfo di;
    vqc_status st = device_info(dev, di);
    if (st != VQC_OK) return st;
    const bool dbl = p.dtype == VQC_C128;
    const size_t rs = dbl ? 8 : 4, cs = 2 * rs, ew = entry_reals(dbl, false);   // ClusterWords
    L.K = L.s->K;
    L.cl = p.n - L.K - L.s->cta_bits;
    L.T = 1 << (p.n - L.K);           // threads of a sample group, over the whole cluster
    L.block = L.T >> L.cl;            // 2^cta_bits: 256 or 512
    L.S = 1;
    L.wg = L.block / 32;
    size_t off = 0;
    auto take = [&](size_t bytes) {
        size_t o = off;
        off = align16(off + bytes);
        return (int)o;
    };
    const size_t slice = ((size_t)1 << (p.n - L.cl)) * cs;
    L.sm_sh = take((size_t)p.n_sh * ew * rs);
    L.sm_ps = take((size_t)p.n_ps * ew * rs);
    L.sm_psi = take(slice);
    if (mode == 0) {
        L.sm_red = take((size_t)L.wg * p.n * rs);
        L.sm_ecl = take(((size_t)1 << L.cl) * p.n * rs);
        L.sm_w = take((size_t)p.num_w * rs);
        L.sm_xg = take((size_t)p.num_x * rs);
    } else {   // lam, rho partials [accs][warps][4], terms, dw partial, x and gE rows
        L.sm_lam = take(slice);
        L.sm_acc = take(std::max<size_t>(p.accs.size(), 1) * L.wg * 4 * rs);
        L.sm_terms = take(std::max<size_t>(p.term_src.size(), 1) * rs);
        L.sm_dw = take((size_t)std::max(p.num_w, 1) * rs);
        L.sm_w = take((size_t)std::max(p.num_w, 1) * rs);
        L.sm_xg = take((size_t)(p.num_x + p.n) * rs);
    }
    const size_t plan_bytes = align16(p.dev_tab_end - p.dev_tab_begin) +
                              (L.s->dev_region_end - L.s->dev_region_begin);
    L.plan_smem = off + plan_bytes <= (size_t)di.smem_optin && t_env.plan_smem;
    L.sm_plan = L.plan_smem ? take(plan_bytes) : 0;
    L.smem = off;
    if (L.smem > (size_t)di.smem_optin)
        return fail(VQC_ERR_UNSUPPORTED, "cluster slice does not fit in shared memory");
    L.fn = mode == 0 ? (dfloat_of(p) ? cluster_ptr_dd() : cluster_ptr(dbl)) : cluster_bwd_ptr(dbl, dfloat_of(p));
    st = allow_max_smem(L.fn, dev, di.smem_optin);
    if (st != VQC_OK) return st;
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1u << L.cl;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(1u << L.cl);
    cfg.blockDim = dim3(L.block);
    cfg.dynamicSmemBytes = L.smem;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int nclusters = 0;
    VQC_CUDA(cudaOccupancyMaxActiveClusters(&nclusters, L.fn, &cfg));
    if (nclusters < 1) return fail(VQC_ERR_UNSUPPORTED, "cluster kernel cannot be resident");
    L.nunits = B;
    L.grid = std::min(B, nclusters) << L.cl;
    if (p.dbuf) {
        std::lock_guard<std::mutex> lk(g_geo_mu);
        g_cluster_cache[k] = L;
    }
    return VQC_OK;
}

// Whether a 2-CTA cluster schedule exists and (backward) its shared-memory layout --
// two slices, the per-warp rho partials, the tables -- fits one CTA.
bool cluster_fits(const HostPlan& p, int mode) {
    const Schedule* s = find_cluster_schedule(p, mode);
    if (!s) return false;
    if (mode == 0) return true;
    Launch L;
    const std::string saved = g_err;
    const bool ok = plan_cluster(p, 1, 1, L) == VQC_OK;
    g_err = saved;
    return ok;
}

// By default 2-CTA clusters (complex64 15 qubits forward, 14 backward; complex128 one
// less) take batches of at most one wave, a cluster per sample, which need no state
// in HBM; beyond that the HBM passes run, which then measured faster on every
// circuit: complex64 14 qubits, batch 100, backward 257 / 358 / 469 us by clusters
// (layered / RZZ rings / random) and 159 / 269 / 327 us by passes; 15 qubits forward
// 191 / 232 / 312 and 118 / 172 / 200 us; complex128 1.0 to 1.3 times.  (Within a wave
// the passes are 1.0 to 2.2 times faster too; that choice is kept for its workspace,
// which holds no states.)  The double-float backward stays on clusters: 762 / 1319 /
// 1555 us at batch 152 against 770 / 2203 / 1558 by passes.  Batches whose states between
// passes exceed kPassStates (65536 samples of a 14-qubit backward) take clusters too,
// which need none.  Larger clusters run only
// when VQC_FORCE_PATH=cluster asks; VQC_FORCE_PATH=hbm turns them off.
constexpr size_t kPassStates = (size_t)16 << 30;
bool use_cluster(const HostPlan& p, int mode, int B) {
    const Schedule* s = find_cluster_schedule(p, mode);
    if (!s) return false;
    if (t_env.cluster) return cluster_fits(p, mode);
    if (t_env.hbm) return false;
    if (p.n - s->K - s->cta_bits != 1) return false;
    if (!(dfloat_of(p) && mode == 1) && find_frame(p, mode, VQC_PATH_HBM)) {
        int dev = 0, sms = 152;   // without a device: GB300's SM count
        DevInfo di;
        if (cudaGetDevice(&dev) == cudaSuccess && device_info(dev, di) == VQC_OK) sms = di.sms;
        else (void)cudaGetLastError();
        if (B > sms / 2 && (mode == 0 ? 1 : 2) * hbm_state_bytes(p, B) <= kPassStates) return false;
    }
    return cluster_fits(p, mode);
}

template <typename R>
vqc_status run_cluster_forward(const HostPlan& p, int B, const void* x, const void* w,
                               const void* psi0, void* E, void* state_out, cudaStream_t stream) {
    using C = C2<R>;
    Launch L;
    vqc_status st = plan_cluster(p, 0, B, L);
    if (st != VQC_OK) return st;
    KArgs<R> a{};
    fill_plan_args<R>(p, L, a);
    a.B = B;
    a.nunits = B;
    a.x = static_cast<const R*>(x);
    a.w = static_cast<const R*>(w);
    a.psi0 = static_cast<const C*>(psi0);
    a.E = static_cast<R*>(E);
    a.state_out = static_cast<C*>(state_out);
    void* args[] = {&a};
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1u << L.cl;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(L.grid);
    cfg.blockDim = dim3(L.block);
    cfg.dynamicSmemBytes = L.smem;
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = use_pdl() ? 2 : 1;
    VQC_CUDA(cudaLaunchKernelExC(&cfg, L.fn, args));
    return VQC_OK;
}

// Workspace of a cluster backward: [0, 256) control block, then the per-cluster
// dw partials [clusters, num_w].
size_t cluster_bwd_workspace(const HostPlan& p, const Launch& L) {
    const size_t rs = p.dtype == VQC_C128 ? 8 : 4;
    return 256 + align256((size_t)(L.grid >> L.cl) * std::max(p.num_w, 1) * rs);
}

template <typename R>
vqc_status run_cluster_backward(const HostPlan& p, int B, const void* x, const void* w,
                                const void* psi0, const void* psi_final, const void* gE, void* dx,
                                void* dw, void* ws, size_t ws_bytes, cudaStream_t stream) {
    using C = C2<R>;
    Launch L;
    vqc_status st = plan_cluster(p, 1, B, L);
    if (st != VQC_OK) return st;
    const size_t need = cluster_bwd_workspace(p, L);
    if (!ws || ws_bytes < need || misaligned(ws, 256))
        return fail(VQC_ERR_WORKSPACE, "backward workspace must be >= " + std::to_string(need) +
                                           " bytes and 256-byte aligned");
    KArgs<R> a{};
    fill_plan_args<R>(p, L, a);
    a.B = B;
    a.nunits = B;
    a.x = static_cast<const R*>(x);
    a.w = static_cast<const R*>(w);
    a.psi0 = static_cast<const C*>(psi0);
    a.psi_final = static_cast<const C*>(psi_final);
    a.gE = static_cast<const R*>(gE);
    a.dx = static_cast<R*>(dx);
    a.dw = static_cast<R*>(dw);
    a.dw_part = reinterpret_cast<R*>(static_cast<char*>(ws) + 256);
    void* args[] = {&a};
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1u << L.cl;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(L.grid);
    cfg.blockDim = dim3(L.block);
    cfg.dynamicSmemBytes = L.smem;
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = use_pdl() ? 2 : 1;
    VQC_CUDA(cudaLaunchKernelExC(&cfg, L.fn, args));
    if (dw && p.num_w > 0) {
        const R* part = a.dw_part;
        int rows = L.grid >> L.cl, cols = p.num_w;
        R* out = static_cast<R*>(dw);
        void* rargs[] = {&part, &rows, &cols, &out};
        VQC_CUDA(launch(reduce_cols_ptr(p.dtype == VQC_C128), dim3(cols), dim3(256), rargs, 0, stream));
    }
    return VQC_OK;
}

// ---------------------------------------------------------------- HBM path
struct PassGeo {
    const FrameSchedule* s = nullptr;
    int K = 0, T = 0, S = 0, block = 0, grid = 0, wg = 1, ntiles = 1;
    int nunits = 0;
    size_t smem = 0;
    int sm_sh = 0, sm_ps = 0, sm_lam = 0, sm_acc = 0, sm_red = 0, sm_plan = 0, sm_tfl = 0, sm_koff = 0, sm_toff = 0, sm_tbase = 0, sm_dg = 0;
    bool tables = false;   // the stages' diagonal tables are used
    const void* fn = nullptr;
};

vqc_status plan_hbm_uncached(const HostPlan& p, int mode, int B, PassGeo& L) {
    L.s = find_frame(p, mode, VQC_PATH_HBM);
    if (!L.s) return fail(VQC_ERR_UNSUPPORTED, "no HBM-tiled schedule for this circuit");
    int dev = 0;
    VQC_CUDA(cudaGetDevice(&dev));
    DevInfo di;
    vqc_status st = device_info(dev, di);
    if (st != VQC_OK) return st;
    const bool dbl = p.dtype == VQC_C128;
    const size_t rs = dbl ? 8 : 4, cs = 2 * rs;
    const int m = L.s->m;
    L.K = L.s->K;
    L.T = 1 << (m - L.K);
    L.wg = L.T > 32 ? L.T / 32 : 1;
    L.ntiles = 1 << (p.n - m);
    PassNeeds c;
    for (size_t i = 0; i < L.s->passes.size(); ++i) c.cover(L.s->passes[i], diagonal_tables(p, *L.s, i));
    const size_t tdim = (size_t)1 << m;
    const size_t ew = entry_reals(dbl, dfloat_of(p));
    const size_t apv = 16 / cs, nk = (tdim / apv + L.T - 1) / L.T;
    L.tables = L.T >= 32 && dbl && (dfloat_of(p) || p.has_ph2);   // as on the resident path
    const PassBytes pb = pass_bytes(c, p.n, mode, p.dtype, dfloat_of(p), L.tables, m, L.K);
    const size_t fixed = pb.fixed, per_tile = pb.tile;
    int S = std::max(1, 128 / L.T);
    if ((size_t)di.smem_optin <= fixed + per_tile)
        S = (size_t)di.smem_optin >= fixed + per_tile ? 1 : 0;
    else
        S = (int)std::min<size_t>((size_t)S, ((size_t)di.smem_optin - fixed) / per_tile);
    if (S < 1) return fail(VQC_ERR_UNSUPPORTED, "HBM tile does not fit in shared memory");
    if (L.T < 32 && S * L.T > 32) S -= S % (32 / L.T);
    L.S = S;
    L.block = S * L.T;
    if (L.block > 512) return fail(VQC_ERR_UNSUPPORTED, "HBM tile group too large");
    size_t off = 0;
    auto take = [&](size_t bytes) {
        size_t o = off;
        off = align16(off + bytes);
        return (int)o;
    };
    take((size_t)S * tdim * cs);   // psi tiles at offset 0
    L.sm_lam = take(mode == 1 ? (size_t)S * tdim * cs : 0);
    L.sm_sh = take((size_t)c.sh * ew * rs);
    L.sm_ps = take((size_t)S * c.ps * ew * rs);
    L.sm_acc = take(mode == 1 ? (size_t)S * c.acc * L.wg * 8 * rs : 0);
    L.sm_red = take(mode == 0 ? (size_t)S * L.wg * p.n * rs : 0);
    L.sm_koff = take(2 * nk * 8);   // tile-copy offsets: one uint2 per vector round, read and written
    L.sm_toff = take((size_t)L.block * 16);   // and each thread's own part
    L.sm_dg = take(S * pb.diagonals);
    L.sm_tbase = take((size_t)c.stages * L.block * 4);
    L.sm_plan = take(c.program(L.s->nout));
    L.sm_tfl = take((size_t)S * (c.stages + 1) * 8);
    L.smem = off;
    L.fn = dfloat_of(p) ? pass_ptr_dd(mode, L.K, L.T >= 32)
           : (!dbl && !p.has_ph2) ? pass_ptr_f32_nph(mode, L.K, L.T >= 32)   // no phase cases
                                  : pass_ptr(dbl, mode, L.K, L.T >= 32);
    if (!L.fn) return fail(VQC_ERR_UNSUPPORTED, "pass kernel not instantiated for this K");
    st = allow_max_smem(L.fn, dev, di.smem_optin);
    if (st != VQC_OK) return st;
    int per_sm = 0;
    VQC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, L.fn, L.block, L.smem));
    if (per_sm < 1) return fail(VQC_ERR_UNSUPPORTED, "pass kernel cannot be resident");
    const long long nunits = ((long long)B * L.ntiles + S - 1) / S;
    if ((long long)B * L.ntiles > 0x3fffffffLL) return fail(VQC_ERR_UNSUPPORTED, "too many tiles");
    L.nunits = (int)nunits;
    L.grid = std::max(1, std::min(L.nunits, per_sm * di.sms));
    L.smem = spread_smem(L.smem, L.grid, per_sm, di);
    return VQC_OK;
}

std::map<GeoKey, PassGeo> g_pass_cache;

vqc_status plan_hbm(const HostPlan& p, int mode, int B, PassGeo& L) {
    const GeoKey k = geo_key(p, mode, B, 1);
    {
        std::lock_guard<std::mutex> lk(g_geo_mu);
        auto it = g_pass_cache.find(k);
        if (it != g_pass_cache.end()) {
            L = it->second;
            return VQC_OK;
        }
    }
    vqc_status st = plan_hbm_uncached(p, mode, B, L);
    if (st == VQC_OK && p.dbuf) {
        std::lock_guard<std::mutex> lk(g_geo_mu);
        g_pass_cache[k] = L;
    }
    return st;
}

void forget_plan(const HostPlan* p) {
    std::lock_guard<std::mutex> lk(g_geo_mu);
    for (auto it = g_launch_cache.begin(); it != g_launch_cache.end();)
        it = it->first.plan == p ? g_launch_cache.erase(it) : std::next(it);
    for (auto it = g_pass_cache.begin(); it != g_pass_cache.end();)
        it = it->first.plan == p ? g_pass_cache.erase(it) : std::next(it);
    for (auto it = g_cluster_cache.begin(); it != g_cluster_cache.end();)
        it = it->first.plan == p ? g_cluster_cache.erase(it) : std::next(it);
    for (auto it = g_workspace_cache.begin(); it != g_workspace_cache.end();)
        it = it->first.plan == p ? g_workspace_cache.erase(it) : std::next(it);
}

// Workspace of the HBM path.  Forward: [control | working state | <Z> partials |
// tables].  Backward: [control | psi | lam | rho sums | gradient terms | tables].
struct HbmWs {
    size_t state = 0, lam = 0, part = 0, terms = 0, ps = 0, sh = 0, total = 0;
    bool by_pass = false;   // the rho sums and the table entries of one pass at a time
};

HbmWs hbm_layout(const HostPlan& p, int mode, int B, int ntiles) {
    const size_t rs = p.dtype == VQC_C128 ? 8 : 4;
    const size_t sbytes = hbm_state_bytes(p, B);
    const size_t entry = entry_reals(p.dtype == VQC_C128, dfloat_of(p)) * rs;
    HbmWs w;
    w.state = 256;
    if (mode == 0) {
        w.part = w.state + sbytes;
        w.ps = w.part + align256((size_t)B * ntiles * p.n * rs);
    } else {   // per-tile rho sums [B * ntiles][accs][4], then the per-sample terms [B][terms]
        w.lam = w.state + sbytes;
        w.part = w.lam + sbytes;
        w.terms = w.part + align256((size_t)B * ntiles * std::max<size_t>(p.accs.size(), 1) * 4 * rs);
        w.ps = w.terms + align256((size_t)B * std::max<size_t>(p.term_src.size(), 1) * rs);
    }
    // table entries: every sample's [B][n_ps], the shared ones [n_sh]
    w.sh = w.ps + align256((size_t)B * p.n_ps * entry);
    w.total = w.sh + align256((size_t)p.n_sh * entry);
    return w;
}

// The backward's layout with room for one pass's rho sums and table entries, where a
// call's whole ones would exceed the built-in scratch of vqc_backward_noalloc.
HbmWs hbm_layout_by_pass(const HostPlan& p, int B, int ntiles) {
    const size_t rs = p.dtype == VQC_C128 ? 8 : 4, sbytes = hbm_state_bytes(p, B);
    const size_t entry = entry_reals(p.dtype == VQC_C128, dfloat_of(p)) * rs;
    size_t accs = 1, ps = 0, sh = 0;
    for (int mode = 0; mode < 2; ++mode)
        for (const auto& f : find_frame(p, mode, VQC_PATH_HBM)->passes) {
            if (mode == 1) accs = std::max(accs, (size_t)f.acc_count);
            ps = std::max(ps, (size_t)f.ps_count);
            sh = std::max(sh, (size_t)f.sh_count);
        }
    HbmWs w;
    w.by_pass = true;
    w.state = 256;
    w.lam = w.state + sbytes;
    w.part = w.lam + sbytes;
    w.terms = w.part + align256((size_t)B * ntiles * accs * 4 * rs);
    w.ps = w.terms + align256((size_t)B * std::max<size_t>(p.term_src.size(), 1) * rs);
    w.sh = w.ps + align256((size_t)B * ps * entry);
    w.total = w.sh + align256(sh * entry);
    return w;
}

// Scratch that the limit of vqc_backward_noalloc counts: states, the rho sums of tiles
// of hbm_tile_qubits bits, terms and the per-sample 2x2 matrices.
size_t hbm_counted_scratch(const HostPlan& p, int B) {
    const bool dbl = p.dtype == VQC_C128;
    const size_t rs = dbl ? 8 : 4;
    const int k = hbm_k(1, p.dtype);
    const int m = p.env_tile ? std::min(std::max(p.env_tile, k + 1), k + 8)
                             : std::min(hbm_tile_qubits(1, p.dtype, p.G_swz), p.n - 1);
    return 256 + 2 * hbm_state_bytes(p, B) +
           align256(((size_t)B << (p.n - m)) * std::max<size_t>(p.accs.size(), 1) * 4 * rs) +
           align256((size_t)B * std::max<size_t>(p.term_src.size(), 1) * rs) +
           align256((size_t)B * p.n_ps * entry_reals(dbl, false) * rs);
}

// The call's table entries (run_tables), read by every pass; with `only`, that pass's
// ones, in its own order.
template <typename R>
vqc_status launch_tables(const HostPlan& p, int B, const void* x, const void* w, void* out_ps, void* out_sh,
                         cudaStream_t stream, const FrameSchedule* s = nullptr, const FPass* only = nullptr) {
    int nps = only ? only->ps_count : p.n_ps, nsh = only ? only->sh_count : p.n_sh;
    if (nps + nsh == 0) return VQC_OK;
    const char* base = static_cast<const char*>(p.dbuf);
    const DEntry* entries = reinterpret_cast<const DEntry*>(base + p.dev_entries);
    const int32_t* ps_list = reinterpret_cast<const int32_t*>(base + p.dev_ps_list);
    const int32_t* sh_list = reinterpret_cast<const int32_t*>(base + p.dev_sh_list);
    const DConst* consts = reinterpret_cast<const DConst*>(base + p.dev_consts);
    const R* cang = reinterpret_cast<const R*>(base + p.dev_cang);
    const R* cmat = reinterpret_cast<const R*>(base + p.dev_cmat);
    const R* xr = static_cast<const R*>(x);
    const R* wr = static_cast<const R*>(w);
    const int32_t* slots = only ? reinterpret_cast<const int32_t*>(base + s->dev_pass_entries) : nullptr;
    const int32_t *ps_sel = only ? slots + only->ps_begin : nullptr, *sh_sel = only ? slots + only->sh_begin : nullptr;
    int Px = p.num_x, Bi = B;
    void* args[] = {&entries, &ps_list, &sh_list, &consts, &cang, &cmat, &xr, &Px, &wr, &Bi, &nps, &nsh,
                    &ps_sel, &sh_sel, &out_ps, &out_sh};
    const int blocks = (int)std::min<long long>(4096, ((long long)B * nps + nsh + 255) / 256);
    VQC_CUDA(launch(p.dfloat ? run_tables_ptr_dd() : run_tables_ptr(p.dtype == VQC_C128), dim3(blocks), dim3(256),
                    args, 0, stream));
    return VQC_OK;
}

template <typename R>
void fill_pass_args(const HostPlan& p, const PassGeo& L, const FPass& ps, const void* ps_g, const void* sh_g,
                    PArgs<R>& a) {
    const char* base = static_cast<const char*>(p.dbuf);
    const FrameSchedule& s = *L.s;
    const bool back = s.mode == 1;   // reads what the forward order writes
    a.ops = reinterpret_cast<const DOp*>(base + s.dev_ops) + ps.op_begin;
    a.stages = reinterpret_cast<const FStage*>(base + s.dev_stages) + ps.stage_begin;
    a.flips = reinterpret_cast<const FFlip*>(base + s.dev_flips) + (size_t)ps.stage_begin * s.nout;
    a.fin = &ps == &s.passes.back() ? reinterpret_cast<const FFinal*>(base + s.dev_fin) : nullptr;
    a.err = p.dev_error;
    a.pass_entries = reinterpret_cast<const int32_t*>(base + s.dev_pass_entries);
    a.pass_accs = reinterpret_cast<const int32_t*>(base + s.dev_pass_accs);
    a.n = p.n;
    a.m = s.m;
    a.tbits = s.m - L.K;
    a.G = p.G_swz;
    a.S = L.S;
    a.nout = s.nout;
    a.nstages = ps.stage_end - ps.stage_begin;
    a.nops = ps.op_end - ps.op_begin;
    a.segs = reinterpret_cast<const FSeg*>(base + s.dev_segs) + ps.seg_begin;
    a.nsegs = ps.seg_end - ps.seg_begin;
    a.seg_begin = ps.seg_begin;
    a.op_begin = ps.op_begin;
    a.ps_begin = ps.ps_begin;
    a.ps_count = ps.ps_count;
    a.sh_begin = ps.sh_begin;
    a.sh_count = ps.sh_count;
    a.acc_begin = ps.acc_begin;
    a.acc_count = ps.acc_count;
    a.n_accs = (int)p.accs.size();
    a.n_ps = p.n_ps;
    a.ps_g = ps_g;
    a.sh_g = sh_g;
    a.nunits = L.nunits;
    for (int i = 0; i < kMaxTileBits; ++i) {
        a.ga[i] = back ? ps.gout[i] : ps.gin[i];
        a.sa[i] = back ? ps.gin[i] : ps.gout[i];
        a.gs[i] = back ? ps.sout[i] : ps.sin[i];
        a.ss[i] = back ? ps.sin[i] : ps.sout[i];
    }
    for (int i = 0; i < kMaxOuterBits; ++i) {
        a.go[i] = back ? ps.oout[i] : ps.oin[i];
        a.so[i] = back ? ps.oin[i] : ps.oout[i];
        a.sosl[i] = back ? 0 : ps.oslot[i];
    }
    a.sm_sh = L.sm_sh; a.sm_ps = L.sm_ps; a.sm_lam = L.sm_lam;
    a.sm_acc = L.sm_acc; a.sm_red = L.sm_red; a.sm_koff = L.sm_koff;
    a.sm_plan = L.sm_plan; a.sm_tfl = L.sm_tfl; a.sm_toff = L.sm_toff;
    a.sm_tbase = L.sm_tbase;
    a.sm_dg = L.sm_dg;
    a.ndg = L.tables ? diagonal_tables(p, s, &ps - s.passes.data()) : 0;
}

// Makes a pass read tables of its own entries and write rho sums of its own accumulators.
template <typename R>
void own_tables(const HostPlan& p, PArgs<R>& a) {
    a.pass_entries = a.pass_accs = reinterpret_cast<const int32_t*>(static_cast<const char*>(p.dbuf) + p.dev_iota);
    a.ps_begin = a.sh_begin = a.acc_begin = 0;
    a.n_ps = a.ps_count;
    a.n_accs = a.acc_count;
}

// The forward passes: psi0 (nullptr: |0...0>) -> out in logical order (nullptr:
// not written), the state between passes in W (not out: the last pass writes
// other addresses than it reads).  out_raw: double-float passes follow.
template <typename R>
vqc_status forward_passes(const HostPlan& p, const PassGeo& L, int B, const void* x, const void* w,
                          const void* psi0, void* W, void* out, bool out_raw, R* E_part, void* ps_g, void* sh_g,
                          bool by_pass, cudaStream_t stream) {
    using C = C2<R>;
    const int np = (int)L.s->passes.size();
    if (np == 1 && psi0 && out) {   // one pass from a caller's state into itself: through W
        const size_t bytes = ((size_t)B << p.n) * sizeof(C);
        const char *i = static_cast<const char*>(psi0), *o = static_cast<const char*>(out);
        if (i < o + bytes && o < i + bytes) {
            VQC_CUDA(cudaMemcpyAsync(W, psi0, bytes, cudaMemcpyDeviceToDevice, stream));
            psi0 = W;
        }
    }
    for (int i = 0; i < np; ++i) {
        PArgs<R> a{};
        fill_pass_args<R>(p, L, L.s->passes[i], ps_g, sh_g, a);
        if (by_pass) {
            vqc_status st = launch_tables<R>(p, B, x, w, ps_g, sh_g, stream, L.s, &L.s->passes[i]);
            if (st != VQC_OK) return st;
            own_tables<R>(p, a);
        }
        const bool last = i == np - 1;
        a.B = B;
        a.src_psi = static_cast<const C*>(i == 0 ? psi0 : W);
        a.dst_psi = static_cast<C*>(last ? out : W);
        a.E_part = last ? E_part : nullptr;
        // double-float: raw pairs between passes, complex128 in and out
        a.src_raw = i > 0;
        a.dst_raw = !last || out_raw;
        void* args[] = {&a};
        VQC_CUDA(launch(L.fn, dim3(L.grid), dim3(L.block), args, L.smem, stream));
    }
    return VQC_OK;
}

template <typename R>
vqc_status run_hbm_forward(const HostPlan& p, int B, const void* x, const void* w,
                           const void* psi0, void* E, void* state_out, void* ws, size_t ws_bytes,
                           cudaStream_t stream) {
    PassGeo L;
    vqc_status st = plan_hbm(p, 0, B, L);
    if (st != VQC_OK) return st;
    const HbmWs lay = hbm_layout(p, 0, B, L.ntiles);
    if (!ws || ws_bytes < lay.total || misaligned(ws, 256))
        return fail(VQC_ERR_WORKSPACE, "forward workspace must be >= " + std::to_string(lay.total) +
                                           " bytes and 256-byte aligned");
    char* wsc = static_cast<char*>(ws);
    R* E_part = reinterpret_cast<R*>(wsc + lay.part);
    st = launch_tables<R>(p, B, x, w, wsc + lay.ps, wsc + lay.sh, stream);
    if (st != VQC_OK) return st;
    st = forward_passes<R>(p, L, B, x, w, psi0, wsc + lay.state, state_out, false, E_part, wsc + lay.ps,
                           wsc + lay.sh, false, stream);
    if (st != VQC_OK) return st;
    const R* Ep = E_part;
    R* Eo = static_cast<R*>(E);
    int Bi = B, nt = L.ntiles, n = p.n;
    void* args[] = {&Ep, &Bi, &nt, &n, &Eo};
    const int blocks = (int)std::min<long long>(4096, ((long long)B * n + 255) / 256);
    VQC_CUDA(launch(reduce_expz_ptr(p.dtype == VQC_C128), dim3(std::max(blocks, 1)), dim3(256), args, 0, stream));
    return VQC_OK;
}

template <typename R>
vqc_status run_hbm_backward(const HostPlan& p, int B, const void* x, const void* w,
                            const void* psi0, const void* psi_final, const void* gE, void* dx,
                            void* dw, void* ws, size_t ws_bytes, cudaStream_t stream, bool by_pass = false) {
    using C = C2<R>;
    PassGeo L;
    vqc_status st = plan_hbm(p, 1, B, L);
    if (st != VQC_OK) return st;
    HbmWs lay = hbm_layout(p, 1, B, L.ntiles);
    if (by_pass && lay.total > ws_bytes) lay = hbm_layout_by_pass(p, B, L.ntiles);
    size_t need = lay.total;
    if (!ws || ws_bytes < need || misaligned(ws, 256))
        return fail(VQC_ERR_WORKSPACE, "backward workspace must be >= " + std::to_string(need) +
                                           " bytes and 256-byte aligned");
    char* wsc = static_cast<char*>(ws);
    C* Psi = reinterpret_cast<C*>(wsc + lay.state);
    C* Lam = reinterpret_cast<C*>(wsc + lay.lam);
    R* rho = reinterpret_cast<R*>(wsc + lay.part);
    R* terms = reinterpret_cast<R*>(wsc + lay.terms);
    void *ps_g = wsc + lay.ps, *sh_g = wsc + lay.sh;
    if (!lay.by_pass) st = launch_tables<R>(p, B, x, w, ps_g, sh_g, stream);
    if (st != VQC_OK) return st;
    const C* src0 = static_cast<const C*>(psi_final);
    if (!src0) {
        // recompute the final state into Psi (no <Z>); lam's region holds the
        // state between these passes
        PassGeo Lf;
        st = plan_hbm(p, 0, B, Lf);
        if (st != VQC_OK) return st;
        st = forward_passes<R>(p, Lf, B, x, w, psi0, Lam, Psi, true, static_cast<R*>(nullptr), ps_g, sh_g,
                               lay.by_pass, stream);
        if (st != VQC_OK) return st;
        src0 = Psi;
    }
    const char* base = static_cast<const char*>(p.dbuf);
    const bool dbl = p.dtype == VQC_C128;
    int nt = (int)p.term_src.size();
    const int32_t* pass_accs = reinterpret_cast<const int32_t*>(base + L.s->dev_pass_accs);
    // per-sample gradient terms from the per-tile rho sums of na accumulators
    auto sum_terms = [&](int na, const int32_t* sel) -> vqc_status {
        if (!((dx && p.num_x > 0) || (dw && p.num_w > 0)) || na == 0) return VQC_OK;
        const R* r = rho;
        int Bi = B, ntl = L.ntiles, Px = p.num_x;
        const DAcc* accs = reinterpret_cast<const DAcc*>(base + p.dev_accs);
        const DEntry* entries = reinterpret_cast<const DEntry*>(base + p.dev_entries);
        const DConst* consts = reinterpret_cast<const DConst*>(base + p.dev_consts);
        const R* cang = reinterpret_cast<const R*>(base + p.dev_cang);
        const R* cmat = reinterpret_cast<const R*>(base + p.dev_cmat);
        const R* xr = static_cast<const R*>(x);
        const R* wr = static_cast<const R*>(w);
        R* o = terms;
        void* args[] = {&r, &Bi, &ntl, &na, &sel, &accs, &entries, &consts, &cang, &cmat, &xr, &Px, &wr, &nt, &o};
        const int blocks = (int)std::min<long long>(4096, ((long long)B * na + 255) / 256);
        VQC_CUDA(launch(p.dfloat ? reduce_terms_ptr_dd() : reduce_terms_ptr(dbl), dim3(std::max(blocks, 1)),
                        dim3(256), args, 0, stream));
        return VQC_OK;
    };
    const int np = (int)L.s->passes.size();
    for (int i = np - 1; i >= 0; --i) {
        PArgs<R> a{};
        fill_pass_args<R>(p, L, L.s->passes[i], ps_g, sh_g, a);
        a.B = B;
        a.gE = static_cast<const R*>(gE);
        const bool first = i == np - 1, last = i == 0;
        a.src_psi = first ? src0 : Psi;
        a.src_lam = first ? nullptr : Lam;
        a.dst_psi = last ? nullptr : Psi;
        a.dst_lam = last ? nullptr : Lam;
        a.src_raw = first ? psi_final == nullptr : 1;   // recomputed states are raw
        a.lam_raw = 1;
        a.dst_raw = 1;
        a.rho = rho;
        if (lay.by_pass) {
            st = launch_tables<R>(p, B, x, w, ps_g, sh_g, stream, L.s, &L.s->passes[i]);
            if (st != VQC_OK) return st;
            own_tables<R>(p, a);
        }
        void* args[] = {&a};
        VQC_CUDA(launch(L.fn, dim3(L.grid), dim3(L.block), args, L.smem, stream));
        if (lay.by_pass) {
            st = sum_terms(a.acc_count, pass_accs + L.s->passes[i].acc_begin);
            if (st != VQC_OK) return st;
        }
    }
    if (!lay.by_pass) st = sum_terms((int)p.accs.size(), nullptr);
    if (st != VQC_OK) return st;
    const R* t = terms;
    const int32_t* xptr = reinterpret_cast<const int32_t*>(base + p.dev_xocc_ptr);
    const int32_t* xocc = reinterpret_cast<const int32_t*>(base + p.dev_xocc);
    const int32_t* wptr = reinterpret_cast<const int32_t*>(base + p.dev_wocc_ptr);
    const int32_t* wocc = reinterpret_cast<const int32_t*>(base + p.dev_wocc);
    R *ox = static_cast<R*>(dx), *ow = static_cast<R*>(dw);
    int Bi = B, Px = p.num_x, Pw = p.num_w;
    const bool want_x = dx && Px > 0, want_w = dw && Pw > 0;
    const int xblocks = (int)std::max<long long>(1, std::min<long long>(4096, ((long long)B * Px + 255) / 256));
    if (!dbl && want_x && want_w) {
        void* args[] = {&t, &Bi, &nt, &xptr, &xocc, &Px, &ox, &wptr, &wocc, &Pw, &ow};
        VQC_CUDA(launch(reduce_grads_ptr(), dim3(Pw + xblocks), dim3(256), args, 0, stream));
        return VQC_OK;
    }
    if (want_x) {
        void* args[] = {&t, &Bi, &nt, &xptr, &xocc, &Px, &ox};
        VQC_CUDA(launch(reduce_dx_ptr(dbl), dim3(xblocks), dim3(256), args, 0, stream));
    }
    if (want_w) {
        long long rows = B;
        void* args[] = {&t, &rows, &nt, &wptr, &wocc, &ow};
        VQC_CUDA(launch(reduce_dw_ptr(dbl), dim3(Pw), dim3(256), args, 0, stream));
    }
    return VQC_OK;
}

// The resident path when it can take the batch (and VQC_FORCE_PATH does not
// ask for the HBM path), else the HBM path.
bool use_hbm(const HostPlan& p, int mode, int B) {
    if (t_env.hbm && find_frame(p, mode, VQC_PATH_HBM)) return true;
    Launch L;
    std::string saved = g_err;
    if (plan_launch(p, mode, B, L) == VQC_OK) return false;
    g_err = saved;
    return find_frame(p, mode, VQC_PATH_HBM) != nullptr;
}

// vqc_forward_backward on the resident path: one launch of the fused kernel,
// unless the forward takes a larger register block than the backward.  The
// fused kernel sweeps forward with the backward's schedule, so then the
// forward call (its own, larger blocks) followed by the backward from the saved
// states is faster (12-qubit workload, batch 4096: 1.68 ms against 1.75 ms).  The same where
// a double-float forward could have taken larger blocks but for its phases (choose_k), up
// to 11 qubits, beyond three CTAs an SM, or two where there are stages enough (rings of
// RZZ, two calls / fused, us: 9 qubits x 4 layers, batch 700 489 / 503, 1000 758 / 1027; 10
// x 1, 320 217 / 197, 500 292 / 310; 10 x 4, 1000 1480 / 2029; 11 x 1, 800 775 / 741; 12 x 1,
// 600 1106 / 1023; random circuits, 11 qubits, 800 1488 / 1642): the fused kernel holds the
// code of both sweeps, two calls a second launch and the states' way through HBM.
bool resident_two_calls(const HostPlan& p, int B) {
    Launch Lf, Lb;
    const std::string saved = g_err;
    const bool ok = plan_launch(p, 0, B, Lf) == VQC_OK && plan_launch(p, 1, B, Lb) == VQC_OK;
    g_err = saved;
    if (!ok || Lf.K > Lb.K) return ok;
    if (!dfloat_of(p) || !p.has_ph2 || p.n > 11) return false;
    int dev = 0;
    DevInfo di;
    if (cudaGetDevice(&dev) != cudaSuccess || device_info(dev, di) != VQC_OK) return false;
    const bool deep = Lb.f->stages.size() >= 8;
    return choose_k(p, 0, B, di.sms, true) > Lb.K && Lb.nunits > (deep && p.n < 11 ? 2 : 3) * di.sms &&
           (p.n < 11 || deep);
}

// Workspace of the two-call form: [backward workspace | final states].
size_t two_call_state_offset(const HostPlan& p, int B) {
    Launch Lb;
    const std::string saved = g_err;
    const vqc_status st = plan_launch(p, 1, B, Lb);
    g_err = saved;
    return st == VQC_OK ? align256(bwd_workspace(p, Lb)) : 0;
}

std::mutex g_upload_mu;

// The plan that a call runs: the compiled one, or the one with every schedule where the
// environment asks for a path or block size that the first has none for.
const HostPlan& plan_for(const vqc_plan* plan) {
    const HostPlan& p = plan->hp;
    auto lacks = [&](int mode, int K) { return K > 0 && !find_frame(p, mode, VQC_PATH_RESIDENT, K); };
    if (!(t_env.hbm && !find_frame(p, 0, VQC_PATH_HBM)) && !lacks(0, t_env.k_fwd) && !lacks(1, t_env.k_bwd)) return p;
    std::lock_guard<std::mutex> lk(g_upload_mu);
    if (!plan->every) {
        std::unique_ptr<HostPlan> e(new HostPlan());
        e->every = true;
        e->env_tile = p.env_tile;
        std::string err;
        if (compile_host(plan->gates.data(), (int32_t)plan->gates.size(), p.n, p.num_x, p.num_w, p.dtype, *e, err) !=
            VQC_OK)
            return p;
        e->dfloat = p.dfloat;
        if (p.dbuf) {   // (launch geometry is worked out from the device copy's layout)
            const std::string saved = g_err;
            int cur = -1;
            if (cudaGetDevice(&cur) != cudaSuccess) return p;
            if (cur != p.device) cudaSetDevice(p.device);
            const vqc_status st = upload(*e);
            if (cur != p.device) cudaSetDevice(cur);
            g_err = saved;
            if (st != VQC_OK) return p;
        }
        plan->every = std::move(e);
    }
    return *plan->every;
}

// p: the plan that the call runs.
vqc_status check_common(const vqc_plan* plan, int32_t batch, const HostPlan*& p) {
    if (!plan) return fail(VQC_ERR_INVALID_ARG, "plan is NULL");
    if (batch < 0) return fail(VQC_ERR_INVALID_ARG, "batch must be >= 0");
    int dev = -1;
    VQC_CUDA(cudaGetDevice(&dev));
    auto ready = [](const HostPlan& h) -> vqc_status {
        std::lock_guard<std::mutex> lk(g_upload_mu);
        return h.dbuf ? VQC_OK : upload(const_cast<HostPlan&>(h));
    };
    vqc_status st = ready(plan->hp);
    if (st != VQC_OK) return st;
    if (dev != plan->hp.device)
        return fail(VQC_ERR_INVALID_ARG, "plan was compiled for device " +
                                             std::to_string(plan->hp.device) +
                                             " but the current device is " + std::to_string(dev));
    p = &plan_for(plan);
    return p == &plan->hp ? VQC_OK : ready(*p);
}

// Real arrays (E, gE, dx, dw, probabilities) must be aligned to the real type,
// state arrays to the complex type; NULL passes (each call checks presence).
vqc_status check_out_ptrs(const HostPlan& p, std::initializer_list<const void*> reals,
                          std::initializer_list<const void*> states) {
    const size_t rs = p.dtype == VQC_C128 ? 8 : 4;
    for (const void* q : reals)
        if (q && misaligned(q, rs)) return fail(VQC_ERR_INVALID_ARG, "real arrays must be aligned to the real type");
    for (const void* q : states)
        if (q && misaligned(q, 2 * rs))
            return fail(VQC_ERR_INVALID_ARG, "state arrays must be aligned to the complex type");
    return VQC_OK;
}

vqc_status check_ptrs(const HostPlan& p, const void* x, const void* w, const void* psi0,
                      const void* psi_final) {
    const size_t rs = p.dtype == VQC_C128 ? 8 : 4;
    if (p.num_x > 0 && !x) return fail(VQC_ERR_INVALID_ARG, "x is NULL but the circuit uses x");
    if (p.num_w > 0 && !w) return fail(VQC_ERR_INVALID_ARG, "w is NULL but the circuit uses w");
    if ((x && misaligned(x, rs)) || (w && misaligned(w, rs)))
        return fail(VQC_ERR_INVALID_ARG, "x / w must be aligned to the real type");
    if ((psi0 && misaligned(psi0, 2 * rs)) || (psi_final && misaligned(psi_final, 2 * rs)))
        return fail(VQC_ERR_INVALID_ARG, "state arrays must be aligned to the complex type");
    return VQC_OK;
}

}  // namespace

vqc_status set_error(vqc_status s, const std::string& msg) { return fail(s, msg); }

// tc_stage.cu: the error word of vqc_stage_apply's kernels (read and cleared).
vqc_status stage_error_check();

// host_eval.cu: the per-plan arena of vqc_evaluate_host.
void release_host_arena(const vqc_plan* plan);

// The backward with an explicit scratch buffer, for vqc_backward_noalloc: the
// scratch must hold the same layout as a vqc_backward workspace; with
// clear_control the control block is zeroed on `stream` before the launch.
vqc_status backward_with_scratch(const vqc_plan* plan, int32_t batch, const void* x,
                                 const void* w, const void* psi0, const void* psi_final,
                                 const void* grad_expz, void* grad_x, void* grad_w, void* scratch,
                                 size_t scratch_bytes, void* stream, bool clear_control) {
    const EnvScope env;
    const HostPlan* hp = nullptr;
    vqc_status st = check_common(plan, batch, hp);
    if (st != VQC_OK) return st;
    const HostPlan& p = *hp;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (batch == 0) {
        if (grad_w && p.num_w > 0)
            VQC_CUDA(cudaMemsetAsync(grad_w, 0, (size_t)p.num_w * (p.dtype == VQC_C128 ? 8 : 4), s));
        return VQC_OK;
    }
    st = check_ptrs(p, x, w, psi0, psi_final);
    if (st != VQC_OK) return st;
    if (!grad_expz) return fail(VQC_ERR_INVALID_ARG, "grad_expz is NULL");
    st = check_out_ptrs(p, {grad_expz, grad_x, grad_w}, {});
    if (st != VQC_OK) return st;
    // the same path choice as vqc_backward: the cluster backward when the
    // environment asks for it, resident when the batch fits a resident launch,
    // else the HBM-tiled passes (each with its own workspace layout)
    bool clu = use_cluster(p, 1, batch);
    bool hbm = !clu && use_hbm(p, 1, batch);
    if (hbm && !t_env.force) {   // states that do not fit the scratch may fit a cluster
        const Schedule* s = find_cluster_schedule(p, 1);
        PassGeo L;
        st = plan_hbm(p, 1, batch, L);
        if (st != VQC_OK) return st;
        if (s && p.n - s->K - s->cta_bits == 1 && hbm_layout(p, 1, batch, L.ntiles).total > scratch_bytes &&
            cluster_fits(p, 1)) {
            clu = true;
            hbm = false;
        }
    }
    size_t need = 0;
    if (clu) {
        Launch L;
        st = plan_cluster(p, 1, batch, L);
        if (st != VQC_OK) return st;
        need = cluster_bwd_workspace(p, L);
    } else if (hbm) {
        PassGeo L;
        st = plan_hbm(p, 1, batch, L);
        if (st != VQC_OK) return st;
        need = hbm_layout(p, 1, batch, L.ntiles).total;
        if (need > scratch_bytes && hbm_counted_scratch(p, batch) <= scratch_bytes)
            need = hbm_layout_by_pass(p, batch, L.ntiles).total;
    } else {
        Launch L;
        st = plan_launch(p, 1, batch, L);
        if (st != VQC_OK) return st;
        fit_grid(p, scratch_bytes, L);
        need = bwd_workspace(p, L);
    }
    if (need > scratch_bytes)
        return fail(VQC_ERR_WORKSPACE, "this batch needs " + std::to_string(need) +
                                           " bytes of scratch; the built-in scratch holds " +
                                           std::to_string(scratch_bytes));
    if (clear_control) VQC_CUDA(cudaMemsetAsync(scratch, 0, 256, s));
    if (clu) {
        if (p.dtype == VQC_C64)
            return run_cluster_backward<float>(p, batch, x, w, psi0, psi_final, grad_expz, grad_x,
                                               grad_w, scratch, scratch_bytes, s);
        return run_cluster_backward<double>(p, batch, x, w, psi0, psi_final, grad_expz, grad_x,
                                            grad_w, scratch, scratch_bytes, s);
    }
    if (hbm) {
        if (p.dtype == VQC_C64)
            return run_hbm_backward<float>(p, batch, x, w, psi0, psi_final, grad_expz, grad_x,
                                           grad_w, scratch, scratch_bytes, s, true);
        return run_hbm_backward<double>(p, batch, x, w, psi0, psi_final, grad_expz, grad_x,
                                        grad_w, scratch, scratch_bytes, s, true);
    }
    if (p.dtype == VQC_C64)
        return run<float>(p, 1, batch, x, w, psi0, psi_final, grad_expz, nullptr, nullptr, grad_x,
                          grad_w, scratch, scratch_bytes, s, true);
    return run<double>(p, 1, batch, x, w, psi0, psi_final, grad_expz, nullptr, nullptr, grad_x,
                       grad_w, scratch, scratch_bytes, s, true);
}

namespace {

// Workspace bytes of a call in the arithmetic of t_arith.
size_t workspace_need(const vqc_plan* plan, int batch, int mode) {
    if (mode == 3) {   // vqc_forward_backward: its one-launch form, or either call's workspace
        size_t need = std::max(workspace_need(plan, batch, 0), workspace_need(plan, batch, 1));
        const HostPlan& p = plan_for(plan);
        Launch L;
        const std::string saved = g_err;
        if (batch > 0 && !use_cluster(p, 0, batch) && !use_hbm(p, 0, batch) && !use_hbm(p, 1, batch)) {
            if (resident_two_calls(p, batch)) {
                const size_t cs = p.dtype == VQC_C128 ? 16 : 8;
                need = std::max(need, two_call_state_offset(p, batch) + align256(((size_t)batch << p.n) * cs));
            } else if (plan_launch(p, 2, batch, L) == VQC_OK) {
                need = std::max(need, bwd_workspace(p, L));
            }
        }
        if (batch > 0 && !use_cluster(p, 1, batch) && use_hbm(p, 1, batch)) {
            // the final states in the backward's psi region, the forward's workspace behind them
            need = std::max(need, hbm_state_bytes(p, batch) + workspace_need(plan, batch, 0));
        }
        if (batch > 0 && use_cluster(p, 1, batch)) {   // [either call's workspace | final states]
            const size_t cs = p.dtype == VQC_C128 ? 16 : 8;
            need = align256(need) + align256(((size_t)batch << p.n) * cs);
        }
        g_err = saved;
        return need;
    }
    if (mode == 2 && batch > 0) {   // vqc_probabilities: forward workspace + state + E
        const HostPlan& p = plan_for(plan);
        const size_t rs = p.dtype == VQC_C128 ? 8 : 4;
        return align256(workspace_need(plan, batch, 0)) +
               align256(((size_t)batch << p.n) * 2 * rs) + align256((size_t)batch * p.n * rs);
    }
    if ((mode != 0 && mode != 1) || batch <= 0) return 0;
    const HostPlan& p = plan_for(plan);
    if (use_cluster(p, mode, batch)) {
        if (mode == 0) return 0;
        Launch L;
        if (plan_cluster(p, 1, batch, L) != VQC_OK) return 0;
        return cluster_bwd_workspace(p, L);
    }
    if (use_hbm(p, mode, batch)) {
        PassGeo L;
        if (plan_hbm(p, mode, batch, L) != VQC_OK) return 0;
        return hbm_layout(p, mode, batch, L.ntiles).total;
    }
    if (mode == 0) return 0;
    Launch L;
    if (plan_launch(p, 1, batch, L) != VQC_OK) return 0;
    return bwd_workspace(p, L);
}

}  // namespace

}  // namespace vqc

using namespace vqc;

extern "C" {

vqc_status vqc_compile(const vqc_gate* gates, int32_t num_gates, int32_t num_qubits,
                       int32_t num_x, int32_t num_w, vqc_dtype dtype, vqc_plan** out_plan) {
    try {
        if (!out_plan) return fail(VQC_ERR_INVALID_ARG, "out_plan is NULL");
        *out_plan = nullptr;
        if (num_gates < 0 || num_x < 0 || num_w < 0 || (num_gates > 0 && !gates))
            return fail(VQC_ERR_INVALID_ARG, "negative count or NULL gate list");
        if (dtype != VQC_C64 && dtype != VQC_C128 && dtype != VQC_C128_DF)
            return fail(VQC_ERR_INVALID_ARG, "bad dtype");
        if (num_qubits < 1 || num_qubits > VQC_MAX_QUBITS)
            return fail(VQC_ERR_TOO_MANY_QUBITS, "num_qubits must be in 1.." +
                                                     std::to_string(VQC_MAX_QUBITS));
        std::unique_ptr<vqc_plan> p(new vqc_plan());
        std::string err;
        // VQC_C128_DF plans are complex128 plans (same layouts and schedules)
        // whose kernels compute in double-float
        const vqc_dtype store = dtype == VQC_C128_DF ? VQC_C128 : dtype;
        vqc_status st = compile_host(gates, num_gates, num_qubits, num_x, num_w, store, p->hp, err);
        if (st != VQC_OK) return fail(st, err);
        p->hp.dfloat = dtype == VQC_C128_DF;
        p->gates.assign(gates, gates + num_gates);
        // Upload now when a CUDA device is present; a host-only plan (no device
        // in this process) still serves vqc_plan_export and vqc_plan_info, and
        // is uploaded by the first launching call.
        int ndev = 0;
        if (cudaGetDeviceCount(&ndev) != cudaSuccess) {
            (void)cudaGetLastError();
            ndev = 0;
        }
        if (ndev > 0) {
            st = upload(p->hp);
            if (st != VQC_OK) return st;
        }
        *out_plan = p.release();
        return VQC_OK;
    } catch (const std::bad_alloc&) {
        return fail(VQC_ERR_OUT_OF_MEMORY, "host allocation failed");
    } catch (...) {
        return fail(VQC_ERR_INVALID_ARG, "internal error in vqc_compile");
    }
}

void vqc_free(vqc_plan* plan) {
    if (!plan) return;
    {
        std::lock_guard<std::mutex> lk(g_plans_mu);
        g_plans.erase(&plan->hp);
        g_plans.erase(plan->every.get());
    }
    release_host_arena(plan);
    for (const HostPlan* p : std::initializer_list<const HostPlan*>{&plan->hp, plan->every.get()}) {
        if (!p) continue;
        forget_plan(p);
        if (!p->dbuf) continue;
        int cur = -1;
        cudaGetDevice(&cur);
        if (cur != p->device) cudaSetDevice(p->device);
        cudaFree(p->dbuf);
        if (cur != p->device && cur >= 0) cudaSetDevice(cur);
    }
    delete plan;
}

size_t vqc_workspace_bytes(const vqc_plan* plan, int32_t batch, int32_t mode) {
    if (!plan) return (size_t)-1;
    try {
        const EnvScope env;
        const HostPlan& p = plan_for(plan);
        if (p.dtype != VQC_C128) return workspace_need(plan, batch, mode);
        // either arithmetic's (t_arith), kept: the launches of both are worked out once
        const GeoKey k = geo_key(p, mode, batch, 3 + (t_env.hbm ? 1 : 0) + (t_env.cluster ? 2 : 0));
        {
            std::lock_guard<std::mutex> lk(g_geo_mu);
            auto it = g_workspace_cache.find(k);
            if (it != g_workspace_cache.end()) return it->second;
        }
        size_t need = 0;
        for (int a : {0, 1}) {
            const ArithScope as(a);
            need = std::max(need, workspace_need(plan, batch, mode));
        }
        if (p.dbuf) {
            std::lock_guard<std::mutex> lk(g_geo_mu);
            g_workspace_cache[k] = need;
        }
        return need;
    } catch (...) {
        return (size_t)-1;
    }
}

vqc_status vqc_probabilities(const vqc_plan* plan, int32_t batch, const void* x, const void* w,
                             const void* psi0, void* probs_out, void* workspace,
                             size_t workspace_bytes, void* stream) {
    try {
        const EnvScope env;
        const HostPlan* hp = nullptr;
        vqc_status st = check_common(plan, batch, hp);
        if (st != VQC_OK) return st;
        if (batch == 0) return VQC_OK;
        const HostPlan& p = *hp;
        if (!probs_out) return fail(VQC_ERR_INVALID_ARG, "probs_out is NULL");
        st = check_out_ptrs(p, {probs_out}, {});
        if (st != VQC_OK) return st;
        const bool dbl = p.dtype == VQC_C128;
        const size_t rs = dbl ? 8 : 4;
        const size_t fws = vqc_workspace_bytes(plan, batch, 0);
        const size_t need = vqc_workspace_bytes(plan, batch, 2);
        if (!workspace || workspace_bytes < need || misaligned(workspace, 256))
            return fail(VQC_ERR_WORKSPACE, "probabilities workspace must be >= " + std::to_string(need) +
                                               " bytes and 256-byte aligned");
        char* base = static_cast<char*>(workspace);
        void* state = base + align256(fws);
        void* E = base + align256(fws) + align256(((size_t)batch << p.n) * 2 * rs);
        st = vqc_forward(plan, batch, x, w, psi0, E, state, fws ? workspace : nullptr, fws, stream);
        if (st != VQC_OK) return st;
        cudaStream_t s = static_cast<cudaStream_t>(stream);
        long long count = (long long)batch << p.n;
        int blocks = (int)std::min<long long>((count + 255) / 256, 152LL * 16);
        const void* src = state;
        void* dst = probs_out;
        void* args[] = {&src, &count, &dst};
        VQC_CUDA(launch(abs2_ptr(dbl), dim3(std::max(blocks, 1)), dim3(256), args, 0, s));
        return VQC_OK;
    } catch (...) {
        return fail(VQC_ERR_INVALID_ARG, "internal error in vqc_probabilities");
    }
}

vqc_status vqc_workspace_init(void* workspace, size_t workspace_bytes, void* stream) {
    if (!workspace || workspace_bytes < 256) return fail(VQC_ERR_WORKSPACE, "workspace too small");
    VQC_CUDA(cudaMemsetAsync(workspace, 0, 256, static_cast<cudaStream_t>(stream)));
    return VQC_OK;
}

vqc_status vqc_forward(const vqc_plan* plan, int32_t batch, const void* x, const void* w,
                       const void* psi0, void* expz_out, void* state_out, void* workspace,
                       size_t workspace_bytes, void* stream) {
    try {
        const EnvScope env;
        const HostPlan* hp = nullptr;
        vqc_status st = check_common(plan, batch, hp);
        if (st != VQC_OK) return st;
        if (batch == 0) return VQC_OK;
        const HostPlan& p = *hp;
        st = check_ptrs(p, x, w, psi0, nullptr);
        if (st != VQC_OK) return st;
        if (!expz_out) return fail(VQC_ERR_INVALID_ARG, "expz_out is NULL");
        st = check_out_ptrs(p, {expz_out}, {state_out});
        if (st != VQC_OK) return st;
        cudaStream_t s = static_cast<cudaStream_t>(stream);
        if (use_cluster(p, 0, batch)) {
            if (p.dtype == VQC_C64)
                return run_cluster_forward<float>(p, batch, x, w, psi0, expz_out, state_out, s);
            return run_cluster_forward<double>(p, batch, x, w, psi0, expz_out, state_out, s);
        }
        if (use_hbm(p, 0, batch)) {
            if (p.dtype == VQC_C64)
                return run_hbm_forward<float>(p, batch, x, w, psi0, expz_out, state_out, workspace,
                                              workspace_bytes, s);
            return run_hbm_forward<double>(p, batch, x, w, psi0, expz_out, state_out, workspace,
                                           workspace_bytes, s);
        }
        if (p.dtype == VQC_C64)
            return run<float>(p, 0, batch, x, w, psi0, nullptr, nullptr, expz_out, state_out,
                              nullptr, nullptr, nullptr, 0, s);
        return run<double>(p, 0, batch, x, w, psi0, nullptr, nullptr, expz_out, state_out, nullptr,
                           nullptr, nullptr, 0, s);
    } catch (...) {
        return fail(VQC_ERR_INVALID_ARG, "internal error in vqc_forward");
    }
}

vqc_status vqc_backward(const vqc_plan* plan, int32_t batch, const void* x, const void* w,
                        const void* psi0, const void* psi_final, const void* grad_expz,
                        void* grad_x, void* grad_w, void* workspace, size_t workspace_bytes,
                        void* stream) {
    try {
        const EnvScope env;
        const HostPlan* hp = nullptr;
        vqc_status st = check_common(plan, batch, hp);
        if (st != VQC_OK) return st;
        const HostPlan& p = *hp;
        cudaStream_t s = static_cast<cudaStream_t>(stream);
        if (batch == 0) {
            if (grad_w && p.num_w > 0)
                VQC_CUDA(cudaMemsetAsync(grad_w, 0, (size_t)p.num_w * (p.dtype == VQC_C128 ? 8 : 4), s));
            return VQC_OK;
        }
        st = check_ptrs(p, x, w, psi0, psi_final);
        if (st != VQC_OK) return st;
        if (!grad_expz) return fail(VQC_ERR_INVALID_ARG, "grad_expz is NULL");
        st = check_out_ptrs(p, {grad_expz, grad_x, grad_w}, {});
        if (st != VQC_OK) return st;
        if (use_cluster(p, 1, batch)) {
            if (p.dtype == VQC_C64)
                return run_cluster_backward<float>(p, batch, x, w, psi0, psi_final, grad_expz, grad_x,
                                                   grad_w, workspace, workspace_bytes, s);
            return run_cluster_backward<double>(p, batch, x, w, psi0, psi_final, grad_expz, grad_x,
                                                grad_w, workspace, workspace_bytes, s);
        }
        if (use_hbm(p, 1, batch)) {
            if (p.dtype == VQC_C64)
                return run_hbm_backward<float>(p, batch, x, w, psi0, psi_final, grad_expz, grad_x,
                                               grad_w, workspace, workspace_bytes, s);
            return run_hbm_backward<double>(p, batch, x, w, psi0, psi_final, grad_expz, grad_x,
                                            grad_w, workspace, workspace_bytes, s);
        }
        if (p.dtype == VQC_C64)
            return run<float>(p, 1, batch, x, w, psi0, psi_final, grad_expz, nullptr, nullptr,
                              grad_x, grad_w, workspace, workspace_bytes, s);
        return run<double>(p, 1, batch, x, w, psi0, psi_final, grad_expz, nullptr, nullptr, grad_x,
                           grad_w, workspace, workspace_bytes, s);
    } catch (...) {
        return fail(VQC_ERR_INVALID_ARG, "internal error in vqc_backward");
    }
}

vqc_status vqc_forward_backward(const vqc_plan* plan, int32_t batch, const void* x, const void* w,
                                const void* psi0, const void* grad_expz, void* expz_out, void* grad_x,
                                void* grad_w, void* workspace, size_t workspace_bytes, void* stream) {
    try {
        const EnvScope env;
        const HostPlan* hp = nullptr;
        vqc_status st = check_common(plan, batch, hp);
        if (st != VQC_OK) return st;
        const HostPlan& p = *hp;
        cudaStream_t s = static_cast<cudaStream_t>(stream);
        if (batch == 0) {
            if (grad_w && p.num_w > 0)
                VQC_CUDA(cudaMemsetAsync(grad_w, 0, (size_t)p.num_w * (p.dtype == VQC_C128 ? 8 : 4), s));
            return VQC_OK;
        }
        st = check_ptrs(p, x, w, psi0, nullptr);
        if (st != VQC_OK) return st;
        if (!grad_expz) return fail(VQC_ERR_INVALID_ARG, "grad_expz is NULL");
        if (!expz_out) return fail(VQC_ERR_INVALID_ARG, "expz_out is NULL");
        st = check_out_ptrs(p, {expz_out, grad_expz, grad_x, grad_w}, {});
        if (st != VQC_OK) return st;
        if (!use_cluster(p, 0, batch) && !use_hbm(p, 0, batch) && !use_hbm(p, 1, batch) &&
            resident_two_calls(p, batch)) {
            // the forward (larger register blocks) saves the final states after the
            // backward's workspace; the backward starts from them
            const size_t need = vqc_workspace_bytes(plan, batch, 3);
            if (!workspace || workspace_bytes < need || misaligned(workspace, 256))
                return fail(VQC_ERR_WORKSPACE, "workspace must be >= " + std::to_string(need) +
                                                   " bytes and 256-byte aligned");
            void* psi_final = static_cast<char*>(workspace) + two_call_state_offset(p, batch);
            st = vqc_forward(plan, batch, x, w, psi0, expz_out, psi_final, nullptr, 0, stream);
            if (st != VQC_OK) return st;
            return vqc_backward(plan, batch, x, w, psi0, psi_final, grad_expz, grad_x, grad_w, workspace,
                                workspace_bytes, stream);
        }
        if (!use_cluster(p, 0, batch) && !use_hbm(p, 0, batch) && !use_hbm(p, 1, batch)) {
            // one launch: the backward kernel sweeps forward itself (the state stays in
            // shared memory), writes E, then sweeps back
            if (p.dtype == VQC_C64)
                return run<float>(p, 2, batch, x, w, psi0, nullptr, grad_expz, expz_out, nullptr, grad_x,
                                  grad_w, workspace, workspace_bytes, s);
            return run<double>(p, 2, batch, x, w, psi0, nullptr, grad_expz, expz_out, nullptr, grad_x,
                               grad_w, workspace, workspace_bytes, s);
        }
        if (use_cluster(p, 1, batch)) {
            // the forward leaves the final states after the larger of the two calls'
            // workspaces; the cluster backward starts from them
            const size_t need = vqc_workspace_bytes(plan, batch, 3);
            if (!workspace || workspace_bytes < need || misaligned(workspace, 256))
                return fail(VQC_ERR_WORKSPACE, "workspace must be >= " + std::to_string(need) +
                                                   " bytes and 256-byte aligned");
            const size_t cs = p.dtype == VQC_C128 ? 16 : 8;
            const size_t soff = need - align256(((size_t)batch << p.n) * cs);
            void* psi_final = static_cast<char*>(workspace) + soff;
            st = vqc_forward(plan, batch, x, w, psi0, expz_out, psi_final, workspace, soff, stream);
            if (st != VQC_OK) return st;
            return vqc_backward(plan, batch, x, w, psi0, psi_final, grad_expz, grad_x, grad_w, workspace,
                                soff, stream);
        }
        // states beyond one SM: the forward (passes or cluster) leaves the final
        // states in the psi region of the backward's HBM layout, in this
        // workspace, and the backward passes start from them; the forward's own
        // workspace follows them, where the backward's lam goes later
        if (use_hbm(p, 1, batch)) {
            PassGeo Lb;
            st = plan_hbm(p, 1, batch, Lb);
            if (st != VQC_OK) return st;
            const HbmWs lay = hbm_layout(p, 1, batch, Lb.ntiles);
            const size_t need = vqc_workspace_bytes(plan, batch, 3);
            if (!workspace || workspace_bytes < need || misaligned(workspace, 256))
                return fail(VQC_ERR_WORKSPACE, "workspace must be >= " + std::to_string(need) +
                                                   " bytes and 256-byte aligned");
            char* base = static_cast<char*>(workspace);
            const size_t sbytes = hbm_state_bytes(p, batch);
            void* psi_final = base + lay.state;
            st = vqc_forward(plan, batch, x, w, psi0, expz_out, psi_final, base + sbytes,
                             workspace_bytes - sbytes, stream);
            if (st != VQC_OK) return st;
            return vqc_backward(plan, batch, x, w, psi0, psi_final, grad_expz, grad_x, grad_w,
                                workspace, workspace_bytes, stream);
        }
        st = vqc_forward(plan, batch, x, w, psi0, expz_out, nullptr, workspace, workspace_bytes, stream);
        if (st != VQC_OK) return st;
        return vqc_backward(plan, batch, x, w, psi0, nullptr, grad_expz, grad_x, grad_w, workspace,
                            workspace_bytes, stream);
    } catch (...) {
        return fail(VQC_ERR_INVALID_ARG, "internal error in vqc_forward_backward");
    }
}

vqc_status vqc_plan_info(const vqc_plan* plan, int32_t batch, vqc_plan_stats* out) try {
    const EnvScope env;
    if (!plan || !out) return fail(VQC_ERR_INVALID_ARG, "NULL argument");
    const HostPlan& p = plan_for(plan);
    std::memset(out, 0, sizeof(*out));
    out->num_qubits = p.n;
    out->num_x = p.num_x;
    out->num_w = p.num_w;
    out->dtype = p.dfloat ? VQC_C128_DF : p.dtype;
    out->num_gates_in = p.num_gates_in;
    out->num_ops = (int32_t)p.ops.size();
    out->num_runs = p.n_runs;
    out->num_terms = (int32_t)p.term_src.size();
    out->fwd_flops_per_eval = p.fwd_flops;
    out->bwd_flops_per_eval = p.bwd_flops;
    out->recompute_flops_per_eval = p.recompute_flops;
    const int B = std::max(batch, 1);
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess) {
        (void)cudaGetLastError();
        ndev = 0;
    }
    const std::string saved = g_err;
    int sms = 152;   // without a device: GB300's SM count
    if (ndev > 0) {
        int dev = 0;
        DevInfo di;
        if (cudaGetDevice(&dev) == cudaSuccess && device_info(dev, di) == VQC_OK) sms = di.sms;
        else (void)cudaGetLastError();
    }
    const double sbytes = std::ldexp(1.0, p.n) * (p.dtype == VQC_C128 ? 16.0 : 8.0);
    for (int mode = 0; mode < 2; ++mode) {
        int* path = mode == 0 ? &out->fwd_path : &out->bwd_path;
        int* kk = mode == 0 ? &out->fwd_k : &out->bwd_k;
        int* ns = mode == 0 ? &out->fwd_stages : &out->bwd_stages;
        int* np = mode == 0 ? &out->fwd_passes : &out->bwd_passes;
        int* tps = mode == 0 ? &out->fwd_threads_per_sample : &out->bwd_threads_per_sample;
        int* tq = mode == 0 ? &out->fwd_tile_qubits : &out->bwd_tile_qubits;
        double* hb = mode == 0 ? &out->fwd_hbm_bytes_per_eval : &out->bwd_hbm_bytes_per_eval;
        int K = choose_k(p, mode, B, sms);
        const bool clu = use_cluster(p, mode, B);
        const bool hbm = !clu && (ndev > 0 ? use_hbm(p, mode, B)
                                           : (K == 0 && find_frame(p, mode, VQC_PATH_HBM) != nullptr));
        if (clu) {
            const Schedule* s = find_cluster_schedule(p, mode);
            *path = s->path;
            *kk = s->K;
            *ns = (int)s->stages.size();
            *tq = s->m;
            *np = 1;
            *tps = 1 << (p.n - s->K);
            continue;
        }
        Launch L;
        if (!clu && !hbm && ndev > 0 && plan_launch(p, mode, B, L) == VQC_OK) K = L.K;
        const FrameSchedule* s = hbm ? find_frame(p, mode, VQC_PATH_HBM)
                                     : K ? find_frame(p, mode, VQC_PATH_RESIDENT, K) : nullptr;
        if (!s) {
            *path = -1;
            continue;
        }
        const int P = (int)s->passes.size();
        *path = s->path;
        *kk = s->K;
        *ns = (int)s->stages.size();
        *tq = s->m;
        *np = P;
        *tps = (1 << (s->m - s->K)) << s->nout;
        // state traffic of the HBM passes: forward reads and writes the state once
        // per pass; the backward reads psi (and lam after the first pass) and writes
        // both (except after the last pass)
        if (hbm) *hb = mode == 0 ? 2.0 * P * sbytes : (4.0 * P - 3.0) * sbytes;
    }
    g_err = saved;
    return VQC_OK;
} catch (...) {
    return fail(VQC_ERR_OUT_OF_MEMORY, "vqc_plan_info failed");
}

vqc_status vqc_plan_export(const vqc_plan* plan, void* buf, size_t* inout_bytes) {
    if (!plan || !inout_bytes) return fail(VQC_ERR_INVALID_ARG, "NULL argument");
    try {
        std::vector<uint8_t> b = export_plan(plan->hp);
        size_t cap = *inout_bytes;
        *inout_bytes = b.size();
        if (!buf) return VQC_OK;
        if (cap < b.size()) return fail(VQC_ERR_INVALID_ARG, "buffer too small");
        std::memcpy(buf, b.data(), b.size());
        return VQC_OK;
    } catch (...) {
        return fail(VQC_ERR_OUT_OF_MEMORY, "export failed");
    }
}

vqc_status vqc_sync_check(void* stream) {
    cudaError_t e = cudaStreamSynchronize(static_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) return cuda_fail(e, "cudaStreamSynchronize");
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetLastError");
    // the kernels' launch self-checks: each plan's error word on this device
    int dev = -1;
    VQC_CUDA(cudaGetDevice(&dev));
    std::vector<const HostPlan*> plans;
    {
        std::lock_guard<std::mutex> lk(g_plans_mu);
        plans.assign(g_plans.begin(), g_plans.end());
    }
    unsigned tripped = 0;
    for (const HostPlan* p : plans) {
        if (p->device != dev || !p->dev_error) continue;
        unsigned w = 0;
        VQC_CUDA(cudaMemcpy(&w, p->dev_error, sizeof(w), cudaMemcpyDeviceToHost));
        if (w) {
            tripped |= w;
            VQC_CUDA(cudaMemset(p->dev_error, 0, sizeof(w)));
        }
    }
    if (tripped)
        return fail(VQC_ERR_DEVICE_CHECK,
                    std::string("a kernel's launch self-check tripped:") +
                        ((tripped & 1u) ? " resident sweep geometry" : "") +
                        ((tripped & 2u) ? " HBM pass geometry" : "") +
                        ((tripped & 4u) ? " cluster geometry" : "") + " (the work was skipped)");
    return stage_error_check();   // vqc_stage_apply's tensor-core waits
}

vqc_status vqc_frames_export(const vqc_plan* plan, void* buf, size_t* inout_bytes) {
    if (!plan || !inout_bytes) return fail(VQC_ERR_INVALID_ARG, "NULL argument");
    try {
        std::vector<uint8_t> b = export_frames(plan->hp);
        size_t cap = *inout_bytes;
        *inout_bytes = b.size();
        if (!buf) return VQC_OK;
        if (cap < b.size()) return fail(VQC_ERR_INVALID_ARG, "buffer too small");
        std::memcpy(buf, b.data(), b.size());
        return VQC_OK;
    } catch (...) {
        return fail(VQC_ERR_OUT_OF_MEMORY, "export failed");
    }
}

const char* vqc_last_error(void) { return g_err.c_str(); }

int32_t vqc_abi_version(void) { return VQC_ABI_VERSION; }

}  // extern "C"
