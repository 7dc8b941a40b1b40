// frame.h -- frame schedules: the stage and pass programs of the resident and
// HBM-tiled kernels, host form and the POD records the kernels read.
//
// CX gates (and SWAPs) cost nothing here: they are never applied.  The state
// stays in a storage index s and the compiler tracks which GF(2)-linear
// functions of s the logical qubits are.  Logical qubit q has a selector r_q
// (its bit is the parity of r_q & s) and a direction d_q (flipping it, all
// other qubits fixed, is s ^ d_q), with r_p . d_q = [p = q].  CX(c, t) is
// r_t ^= r_c, d_c ^= d_t.  A single-qubit run is a 2x2 update on the pairs
// (s, s ^ d) with the parity r . s telling which of the two is |0>; CZ, CRZ and
// RZZ are diagonal in two parities.  Two ops commute when the one's directions
// meet the other's selectors evenly, so ops of different layers, whose CX rings
// would otherwise order them, can share a pass and a stage.
//
// A pass works on the cosets ("tiles") of an m-dimensional subspace V of the
// storage index, a stage on the cosets of a K-dimensional subspace D of V held
// in registers, one coset per thread: every run of the stage has its direction
// among D's basis vectors and its selector zero on the others and on the thread
// vectors, so it is a 2x2 update on one local bit.  A selector that is odd on a
// tile's representative is met by moving the representative along that
// direction (FFlip).
//
// Between passes the state lies in HBM at the address M s, M an invertible
// matrix per pass.  A tile's addresses always contain the 2^G amplitudes of
// whole 128-byte lines: after a pass M is changed inside the tile (P, below), so
// that the low address bits become G directions that the next pass's V also
// holds; the set of addresses of a tile stays the same, so a pass can work in
// place.
#pragma once

#include <cstdint>
#include <memory>
#include <string>
#include <vector>

#include "plan.h"

namespace vqc {

constexpr int kMaxTileBits = 14;    // m: bits of a tile (resident: the whole state)
constexpr int kMaxOuterBits = 20;   // n - m
constexpr int kMaxSelectors = 32;   // parities of one stage outside its registers

// One stage.  Thread t of a tile holds the amplitudes at the slots
// XOR(tau of t's bits) ^ flip(tile) ^ XOR(sigma of r's bits), r < 2^K, loads and
// stores alike.  pb, the word of the stage's outside parities, is the XOR of
// tmask over t's bits and of the tile's flips' masks.  An op's qubit ref is a
// local position or kRefPhys + a bit of pb.
struct FStage {
    int32_t tau[kMaxThreadBits];
    uint32_t tmask[kMaxThreadBits];
    int32_t sigma[kMaxK];
    int32_t seg_begin, seg_end;
    int32_t op_begin, op_end;
    uint8_t nthreadbits, nsel;   // nsel: parities in pb (0: pb is not needed)
    uint8_t kind;                // kStagePure: one round of runs and no diagonal op (or no op at all);
                                 // kStagePhases: it has CRZ or RZZ
    uint8_t pmask;               // its positions
    int32_t pad1[2];
};
static_assert(sizeof(FStage) == 176, "FStage layout");
enum : uint8_t { kStagePure = 1, kStagePhases = 2 };

// A stage's ops in rounds: diagonal ones [op_begin, run_begin), then runs [run_begin,
// op_end) in the order of their local positions, at most one each.  The diagonal group
// is ordered by where its qubits live: both outside the block, one local (by position),
// both local (CZ, then phases).
struct FSeg {
    int32_t op_begin, run_begin, op_end;
    uint8_t flags;
    uint8_t pmask;               // positions that have a run
    // diagonal tables of the pass (kNoDiagonal: none): the group's two-local phases and
    // (double-float's, counted for complex128) the runs' q, the runs' p
    uint16_t dg[2];
    uint16_t pad;
};
static_assert(sizeof(FSeg) == 20, "FSeg layout");
enum : uint8_t {
    kSegPs = 1,             // a table depends on the sample
    kSegQ = 2, kSegP = 4,   // some run needs its diagonal before / after the rotation (run_form);
                            // not in stages with phases, whose runs double-float does not factor
    kSegA = 8,              // the group has gradient terms
    kSegL = 16              // it has phases of two local positions
};
constexpr uint16_t kNoDiagonal = 0xffff;

// What tile bit o (of the n - m outer bits) adds to a stage: the slot offset of
// the register block's base and its parities.
struct FFlip {
    int32_t slot;
    uint32_t mask;
};

// The logical qubits on the last stage's register blocks: qubit j's bit of local
// amplitude r is parity(lmask[j] & r) ^ bit j of (XOR of tmask over t's bits ^
// XOR of omask over the tile's bits).
struct FFinal {
    uint32_t tmask[kMaxThreadBits];
    uint32_t omask[kMaxOuterBits];
    uint8_t lmask[32];
};
static_assert(sizeof(FFinal) == 176, "FFinal layout");

// One pass, passes in circuit order.  Amplitude u of a tile before the pass:
// address XOR(gin of u's bits) ^ XOR(oin of the tile's bits), slot XOR(sin); after
// it: gout, oout, sout, the slot also moved by oslot of the tile's bits.  The backward reads what lies after a pass and writes what
// lies before it, every pass in place; the forward's last pass writes logical
// order, at other addresses than its tiles were read from.
struct FPass {
    int32_t stage_begin, stage_end;
    int32_t op_begin, op_end, seg_begin, seg_end;
    uint32_t gin[kMaxTileBits], gout[kMaxTileBits];
    int32_t sin[kMaxTileBits], sout[kMaxTileBits];
    uint32_t oin[kMaxOuterBits], oout[kMaxOuterBits];
    int32_t oslot[kMaxOuterBits];  // zero but in the forward's last pass
    int32_t ps_begin, ps_count;    // per-sample table entries of the pass (into pass_entries)
    int32_t sh_begin, sh_count;    // shared table entries of the pass
    int32_t acc_begin, acc_count;  // accumulators of the pass (into pass_accs)
    int32_t ndg;                   // diagonal tables of its stages
};

struct FrameSchedule {
    int mode = 0, K = 0, m = 0, path = 0;
    int nout = 0;
    std::vector<DOp> ops;
    std::vector<FStage> stages;
    std::vector<FSeg> segs;
    std::vector<FFlip> flips;              // [stages][nout]
    std::vector<FPass> passes;             // one on the resident path
    std::vector<int32_t> phase_tables;     // per pass: its tables of two-local phases, numbered first
                                           // (all that a native complex128 launch needs)
    std::vector<int32_t> pass_entries, pass_accs;
    FFinal fin{};
    size_t dev_ops = 0, dev_stages = 0, dev_segs = 0, dev_flips = 0, dev_fin = 0, dev_pass_entries = 0, dev_pass_accs = 0;
    size_t dev_region_begin = 0, dev_region_end = 0;   // ops, stages, segs, fin in the plan's device blob
};

struct HostPlan;

// frames.cpp: builds a plan's frame schedules.
struct FrameOps;
class FrameBuilder {
  public:
    explicit FrameBuilder(const HostPlan& p);
    ~FrameBuilder();
    // tiles: the tile sizes to choose from (the resident path: the qubit count)
    FrameSchedule build(int mode, int path, const std::vector<int>& tiles, int K) const;

  private:
    const HostPlan& p;
    std::unique_ptr<FrameOps> ops;
};
std::vector<uint8_t> export_frames(const HostPlan& p);

}  // namespace vqc
