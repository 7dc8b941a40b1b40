// engine.h -- host-side plan object shared by the compiler (compiler.cpp) and
// the C ABI / launch code (capi.cu).  Not part of the public ABI.
#pragma once

#include <cstddef>
#include <cstdint>
#include <memory>
#include <string>
#include <vector>

#include "frame.h"
#include "plan.h"
#include "../../include/vqc.h"

static_assert(sizeof(vqc_gate) == 48, "vqc_gate layout");

namespace vqc {

// A fused op of the lowered circuit (time-valid order).
struct HOp {
    uint8_t type;      // OpType
    int q0, q1;        // M1: q0 target; CX: q0 control, q1 target; CZ/PH2: q0, q1
    int entry;         // table entry id for M1 / PH2, else -1
    uint8_t gen;       // OPF_GEN_* for PH2
};

// One register-block stage schedule for a (mode, K, tile) choice: the cluster path's, and
// the axis-aligned ones that vqc_plan_export builds for itself.
struct Schedule {
    int mode = 0;          // 0 forward, 1 backward
    int K = 0;             // register-block qubits
    int m = 0;             // qubits per shared-memory tile (== n on the resident path)
    int path = VQC_PATH_RESIDENT;
    int thread_bits = 0;   // m - K
    int group_lanes_log2 = 0;   // log2(threads per sample group) when < 2^G
    int cta_bits = 0;           // cluster path: log2(threads per CTA); 2^(m-K-cta_bits) CTAs
    std::vector<DOp> ops;
    std::vector<DStage> stages;
    // exported HBM schedules only: one record per pass, its table entries (per sample, then
    // shared) and its accumulators
    std::vector<DPass> passes;
    std::vector<int32_t> pass_entries, pass_accs;
    // Per stage, kMaxK + kMaxThreadBits physical-index masks: the image under
    // the stage's absorbed permutation of each local bit, then of each thread
    // bit (exported for tests; the kernels use the swizzled store map).
    std::vector<uint32_t> store_masks;
    size_t dev_ops = 0, dev_stages = 0;   // byte offsets inside the device buffer
    size_t dev_region_begin = 0, dev_region_end = 0;   // [ops, stages] in the blob
};

struct HostPlan {
    int n = 0, num_x = 0, num_w = 0, dtype = 0, num_gates_in = 0;
    int G_swz = 4;                         // swizzle chunk bits (4: c64, 3: c128)
    bool dfloat = false;                   // VQC_C128_DF: complex128 storage, double-float kernels
    bool has_ph2 = false;                  // the op list holds diagonal two-qubit phases (CRZ / RZZ)
    std::vector<HOp> ops;
    std::vector<DEntry> entries;
    std::vector<DConst> consts;
    std::vector<double> cmat;              // 8 doubles per constant 2x2 matrix
    std::vector<double> cang;              // constant angles
    std::vector<int32_t> term_src, term_idx;   // per term: SRC_X / SRC_W, column
    std::vector<DAcc> accs;
    std::vector<int32_t> xocc_ptr, xocc, wocc_ptr, wocc;   // terms of each x column / w index
    int n_ps = 0, n_sh = 0;                // per-sample / shared table sizes
    int n_runs = 0;
    int env_tile = 0;                      // VQC_HBM_TILE_QUBITS at compile time, 0: none
    bool every = false;                    // all schedules: HBM passes and block sizes below 3 as well
    std::vector<Schedule> scheds;          // of the cluster path
    std::vector<FrameSchedule> frames;     // of the resident and HBM-tiled kernels
    double fwd_flops = 0, bwd_flops = 0, recompute_flops = 0;

    // device copy
    int device = -1;
    void* dbuf = nullptr;
    size_t dbytes = 0;
    size_t dev_entries = 0, dev_ps_list = 0, dev_sh_list = 0, dev_consts = 0, dev_cmat = 0, dev_cang = 0;
    size_t dev_xocc_ptr = 0, dev_xocc = 0, dev_wocc_ptr = 0, dev_wocc = 0, dev_accs = 0, dev_iota = 0;
    unsigned* dev_error = nullptr;        // device error word (kernel self-checks)
    size_t dev_tab_begin = 0, dev_tab_end = 0;   // [entries .. wocc] in the blob
};

// Largest n whose state(s) fit one CTA's shared memory on the resident path.
inline int resident_max_qubits(int mode, int dtype) {
    if (dtype == VQC_C64) return mode == 0 ? 14 : 13;
    return mode == 0 ? 13 : 12;
}
// Tile qubits of an HBM pass: 64 KiB of tile state per CTA (two states for the backward).
inline int hbm_tile_qubits(int mode, int dtype, int G) {
    (void)G;
    if (dtype == VQC_C64) return mode == 0 ? 13 : 12;
    return mode == 0 ? 12 : 11;
}
inline int hbm_k(int mode, int dtype) {
    if (dtype == VQC_C64) return mode == 0 ? 5 : 4;
    return mode == 0 ? 4 : 3;
}

// Tile bits offered to the frame schedules of the HBM passes.  complex64: 32 KiB of
// forward tile (18-qubit / batch-48 forward 451 us, 485 with 13 bits, 488 with 11),
// or one bit less where that costs no pass and no stage (16-qubit / batch-512 step
// 6.21 ms against 6.50): a pass is bound by the latency of its stages, and smaller
// tiles mean more CTAs per SM, each waiting for fewer warps.  complex128: 64 KiB
// (16-qubit / batch-77 double-float step 7.79 ms, 8.03 with 11 bits both ways, 9.74 with 10).
inline std::vector<int> frame_tile_qubits(int mode, int dtype, int n) {
    auto fit = [n](int m) { return m < n - 1 ? m : n - 1; };
    if (dtype == VQC_C64) return {fit(12), fit(11)};
    return {fit(mode == 0 ? 12 : 11)};
}

// Shared memory that a CTA can have on sm_103a (227 KB), and each of two on one SM.
constexpr size_t kCtaSharedMemory = 232448;
constexpr size_t kHalfSharedMemory = 115712;

// The largest of each count that sizes a launch of a pass: of one, or over all passes
// of a schedule (whose launches share one layout).
struct PassNeeds {
    int ps = 0, sh = 0, acc = 0, stages = 0, ops = 0, segs = 0, ndg = 0;
    void cover(const FPass& p, int tables) {
        auto most = [](int& a, int b) { a = b > a ? b : a; };
        most(ps, p.ps_count);
        most(sh, p.sh_count);
        most(acc, p.acc_count);
        most(stages, p.stage_end - p.stage_begin);
        most(ops, p.op_end - p.op_begin);
        most(segs, p.seg_end - p.seg_begin);
        most(ndg, tables);
    }
    // the pass's program: copies of its stages, ops, flips, rounds and FFinal
    size_t program(int nout) const {
        return (size_t)stages * sizeof(FStage) + sizeof(FFinal) + (size_t)ops * sizeof(DOp) +
               (size_t)stages * nout * sizeof(FFlip) + (size_t)segs * sizeof(FSeg);
    }
};

// Shared memory of a pass launch (plan_hbm places the parts): bytes per CTA, and per
// tile of the CTA.
struct PassBytes {
    size_t fixed, tile;
    size_t diagonals;   // of the tile's: the stages' diagonal tables
};
inline PassBytes pass_bytes(const PassNeeds& c, int n, int mode, int dtype, bool dfloat, bool tables, int m, int K) {
    const size_t rs = dtype == VQC_C128 ? 8 : 4, cs = 2 * rs, ew = entry_reals(dtype == VQC_C128, dfloat);
    const size_t T = (size_t)1 << (m - K), wg = T > 32 ? T / 32 : 1, dim = (size_t)1 << m;
    const size_t nk = (dim / (16 / cs) + T - 1) / T;
    auto align16 = [](size_t v) { return (v + 15) & ~size_t(15); };
    PassBytes b;
    b.fixed = align16((size_t)c.sh * ew * rs) + align16(c.program(n - m)) + align16(2 * nk * 8) + 8 * 16;
    b.diagonals = tables ? ((size_t)c.ndg << K) * cs : 0;
    b.tile = b.diagonals + (size_t)c.ps * ew * rs + dim * cs * (mode == 1 ? 2 : 1) + (size_t)(c.stages + 1) * 8 +
             T * (16 + 4 * (size_t)c.stages) + (mode == 1 ? (size_t)c.acc * wg * 8 * rs : wg * n * rs);
    return b;
}

// Maximum K per (mode, dtype) for register-resident blocks.
inline int max_k(int mode, int dtype) {
    if (dtype == VQC_C64) return mode == 0 ? 5 : 4;
    return mode == 0 ? 4 : 3;
}

// compiler.cpp
vqc_status compile_host(const vqc_gate* gates, int32_t G, int32_t n, int32_t nx, int32_t nw,
                        int dtype, HostPlan& out, std::string& err);
const Schedule* find_cluster_schedule(const HostPlan& p, int mode);
const FrameSchedule* find_frame(const HostPlan& p, int mode, int path, int K = 0);
std::vector<uint8_t> export_plan(const HostPlan& p);

}  // namespace vqc

// The opaque handle of the C ABI: a compiled host plan (and its device copy).
struct vqc_plan {
    vqc::HostPlan hp;
    // The same circuit with the schedules that only environment switches ask for, compiled
    // by the first call that finds one set (plan_for).
    std::vector<vqc_gate> gates;
    mutable std::unique_ptr<vqc::HostPlan> every;
};
