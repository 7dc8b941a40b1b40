// frames.cpp -- builds the frame schedules of frame.h from a plan's op list.
#include <algorithm>
#include <cstring>

#include "engine.h"

namespace vqc {
namespace {

// A short list of vectors of the index space (or selectors), held in place: a plan
// builds thousands of them.
struct Vecs {
    uint32_t v[32];
    int n = 0;
    Vecs() = default;
    explicit Vecs(size_t count) : n((int)count) { std::memset(v, 0, sizeof(v)); }
    Vecs(const Vecs& o) : n(o.n) { std::memcpy(v, o.v, sizeof(uint32_t) * n); }
    Vecs& operator=(const Vecs& o) {
        n = o.n;
        std::memmove(v, o.v, sizeof(uint32_t) * n);
        return *this;
    }
    size_t size() const { return (size_t)n; }
    bool empty() const { return n == 0; }
    void clear() { n = 0; }
    void push_back(uint32_t x) { v[n++] = x; }
    uint32_t& operator[](size_t i) { return v[i]; }
    uint32_t operator[](size_t i) const { return v[i]; }
    uint32_t* begin() { return v; }
    uint32_t* end() { return v + n; }
    const uint32_t* begin() const { return v; }
    const uint32_t* end() const { return v + n; }
    void append(const Vecs& o) {
        for (uint32_t x : o) push_back(x);
    }
    void erase(int i) {
        for (--n; i < n; ++i) v[i] = v[i + 1];
    }
    Vecs first(int count) const {
        Vecs r;
        for (int i = 0; i < count; ++i) r.push_back(v[i]);
        return r;
    }
};

inline bool odd(uint32_t v) { return __builtin_parity(v) != 0; }

// An op in the storage frame: a run (direction d, selector r), or a diagonal op
// on the parities r and r2.
struct FOp {
    bool run = false;
    uint32_t d = 0, r = 0, r2 = 0;
    int hop = -1;
};

// The subspace spanned by the vectors added so far.
struct Span {
    uint32_t piv[24] = {0};   // by highest set bit (at most 24 qubits)
    int dim = 0;
    uint32_t reduce(uint32_t v) const {
        while (v) {
            const int h = 31 - __builtin_clz(v);
            if (!piv[h]) return v;
            v ^= piv[h];
        }
        return 0;
    }
    bool add(uint32_t v) {
        v = reduce(v);
        if (!v) return false;
        piv[31 - __builtin_clz(v)] = v;
        ++dim;
        return true;
    }
    Vecs basis() const {
        Vecs b;
        for (uint32_t v : piv)
            if (v) b.push_back(v);
        return b;
    }
};

// The ops that a scan in time order leaves behind.  An op commutes with all of them
// when its selectors are even on their directions and its direction on their
// selectors: both are tests against a basis.  Once the directions fill the space
// nothing later can pass.
struct Waiting {
    Span d, s;
    uint32_t dv[24], sv[24];   // the bases, dense
    int nd = 0, ns = 0;
    bool passes(const FOp& o) const {
        if (o.run) {
            for (int i = 0; i < nd; ++i)
                if (odd(o.r & dv[i])) return false;
            for (int i = 0; i < ns; ++i)
                if (odd(o.d & sv[i])) return false;
        } else {
            for (int i = 0; i < nd; ++i)
                if (odd(o.r & dv[i]) || odd(o.r2 & dv[i])) return false;
        }
        return true;
    }
    void add(const FOp& o) {
        if (o.run && d.add(o.d)) dv[nd++] = o.d;
        if (s.add(o.r)) sv[ns++] = o.r;
        if (!o.run && s.add(o.r2)) sv[ns++] = o.r2;
    }
};

// Coordinates in a basis: coord(v) has bit i set when basis vector i is in v.
struct Coords {
    uint32_t piv[32] = {0}, comb[32] = {0};
    explicit Coords(const Vecs& b) {
        for (size_t i = 0; i < b.size(); ++i) {
            uint32_t v = b[i], c = 1u << i;
            while (v) {
                const int h = 31 - __builtin_clz(v);
                if (!piv[h]) {
                    piv[h] = v;
                    comb[h] = c;
                    break;
                }
                v ^= piv[h];
                c ^= comb[h];
            }
        }
    }
    uint32_t operator()(uint32_t v) const {
        uint32_t c = 0;
        while (v) {
            const int h = 31 - __builtin_clz(v);
            c ^= comb[h];
            v ^= piv[h];
        }
        return c;
    }
};

// The vectors of span(vs) on which every functional of `sel` is even (a basis).
Vecs annihilated(Vecs vs, const Vecs& sel) {
    for (uint32_t s : sel) {
        int k = -1;
        for (size_t i = 0; i < vs.size(); ++i)
            if (odd(vs[i] & s)) {
                if (k < 0) k = (int)i;
                else vs[i] ^= vs[k];
            }
        if (k >= 0) vs.erase(k);
    }
    return vs;
}

uint32_t image(const Vecs& cols, uint32_t v) {   // XOR of cols[i] over v's bits
    uint32_t r = 0;
    for (size_t i = 0; i < cols.size(); ++i)
        if ((v >> i) & 1) r ^= cols[i];
    return r;
}

Vecs inverse(Vecs cols) {   // of an invertible matrix, as columns
    const size_t n = cols.size();
    Vecs inv(n);
    for (size_t i = 0; i < n; ++i) inv[i] = 1u << i;
    for (size_t b = 0; b < n; ++b) {
        size_t k = b;
        while (!((cols[k] >> b) & 1)) ++k;
        std::swap(cols[k], cols[b]);
        std::swap(inv[k], inv[b]);
        for (size_t j = 0; j < n; ++j)
            if (j != b && ((cols[j] >> b) & 1)) {
                cols[j] ^= cols[b];
                inv[j] ^= inv[b];
            }
    }
    return inv;
}

// Table entries and accumulators of one pass, and ops of one stage: what of a pass's
// shared memory is not bounded by giving its later stages a pass of their own (split).
constexpr int kMaxPassEntries = 96;
constexpr size_t kMaxStageOps = 2048;

struct StagePlan {
    std::vector<int> ops;              // indices into the FOp list, time order
    Vecs D, R;        // directions and selectors of its runs, by local position
    Vecs sels;        // distinct selectors of its diagonal ops
};

// Cut a pass's ops into stages of at most K directions.
std::vector<StagePlan> cut(const std::vector<FOp>& f, const std::vector<int>& ops, int n, int K) {
    std::vector<StagePlan> out;
    std::vector<int> rem = ops;
    do {   // an empty op list still gets one (empty) stage
        StagePlan s;
        std::vector<int> defer;
        Waiting w;
        Span sp;   // of D
        size_t i = 0;
        for (; i < rem.size() && w.d.dim < n; ++i) {
            const FOp& o = f[rem[i]];
            bool ok = w.passes(o) && s.ops.size() < kMaxStageOps;
            if (ok && o.run) {
                size_t j = 0;
                while (j < s.D.size() && !(s.D[j] == o.d && s.R[j] == o.r)) ++j;
                if (j == s.D.size()) {   // a new direction: dual to the others and to the parities
                    ok = (int)s.D.size() < K;
                    ok = ok && sp.reduce(o.d) != 0;
                    for (size_t k = 0; ok && k < s.D.size(); ++k)
                        ok = !odd(s.R[k] & o.d) && !odd(o.r & s.D[k]);
                    for (size_t k = 0; ok && k < s.sels.size(); ++k)
                        ok = !odd(s.sels[k] & o.d) || s.sels[k] == o.r;
                    if (ok) {
                        sp.add(o.d);
                        s.D.push_back(o.d);
                        s.R.push_back(o.r);
                    }
                }
            } else if (ok) {
                Vecs add;
                for (uint32_t r : {o.r, o.r2}) {   // a parity that a run changes is that run's own
                    for (size_t k = 0; k < s.D.size(); ++k) ok = ok && (!odd(r & s.D[k]) || r == s.R[k]);
                    if (std::find(s.sels.begin(), s.sels.end(), r) == s.sels.end()) add.push_back(r);
                }
                ok = ok && s.sels.size() + add.size() <= (size_t)kMaxSelectors;
                if (ok) s.sels.append(add);
            }
            (ok ? s.ops : defer).push_back(rem[i]);
            if (!ok) w.add(o);
        }
        defer.insert(defer.end(), rem.begin() + i, rem.end());
        out.push_back(std::move(s));
        rem.swap(defer);
    } while (!rem.empty());
    return out;
}

// Complete a stage's D to K vectors of the tile: every pad is even on the runs'
// selectors, meets at most one diagonal selector, and no selector meets two of D.
// False when the diagonal ops leave no such pads.
bool pad(StagePlan& s, const Vecs& V, int K) {
    Vecs A = annihilated(V, s.R);
    Vecs free = annihilated(A, s.sels);
    // A's vectors dual to the diagonal selectors that D does not meet yet, then the free ones
    Vecs cand = free;
    Vecs rest = A;
    for (size_t i = 0; i < s.sels.size(); ++i) {
        int k = -1;
        for (size_t j = 0; j < rest.size(); ++j)
            if (odd(rest[j] & s.sels[i])) {
                if (k < 0) k = (int)j;
                else rest[j] ^= rest[k];
            }
        if (k < 0) continue;
        uint32_t v = rest[k];
        rest.erase(k);
        for (size_t l = i + 1; l < s.sels.size(); ++l)   // even on the later selectors if the rest allows it
            if (odd(v & s.sels[l]))
                for (uint32_t t : rest) {
                    bool only = odd(t & s.sels[l]);
                    for (size_t q = i + 1; only && q < l; ++q) only = !odd(t & s.sels[q]);
                    if (only) { v ^= t; break; }
                }
        cand.push_back(v);
    }
    Span sp;
    for (uint32_t d : s.D) sp.add(d);
    for (uint32_t v : cand) {
        if ((int)s.D.size() == K) break;
        if (!sp.reduce(v)) continue;
        bool ok = true;
        int hits = 0;
        for (uint32_t r : s.sels) {
            if (!odd(r & v)) continue;
            ++hits;
            for (uint32_t d : s.D) ok = ok && !odd(r & d);
        }
        ok = ok && hits <= 1;
        if (!ok) continue;
        sp.add(v);
        s.D.push_back(v);
    }
    return (int)s.D.size() == K;
}

struct PassPlan {
    std::vector<int> ops;
    Vecs V;           // basis of the tile's subspace
    std::vector<StagePlan> stages;
};

// A base vector of the stage moved along D so that every selector with a local
// bit is even on it: the local bit alone is then the parity.
uint32_t settle(const StagePlan& s, uint32_t v) {
    const size_t nr = s.R.size();
    for (size_t k = 0; k < nr; ++k)
        if (odd(s.R[k] & v)) v ^= s.D[k];
    for (uint32_t r : s.sels)
        for (size_t k = nr; k < s.D.size(); ++k)
            if (odd(r & s.D[k]) && odd(r & v)) v ^= s.D[k];
    return v;
}

int rank_of(const Vecs& v) {
    Span s;
    for (uint32_t x : v) s.add(x);
    return s.dim;
}

struct Rng {   // small deterministic generator (xorshift32) for the swizzle search
    uint32_t s = 2463534242u;
    uint32_t next() {
        s ^= s << 13;
        s ^= s >> 17;
        s ^= s << 5;
        return s;
    }
};

}  // namespace

// The op list in the storage frame, and the frame at its end.
struct FrameOps {
    Vecs dir, sel;
    std::vector<FOp> f;
};

namespace {

FrameOps lower(const HostPlan& p) {
    const int n = p.n;
    FrameOps L;
    Vecs &dir = L.dir, &sel = L.sel;
    for (int q = 0; q < n; ++q) {
        dir.push_back(1u << q);
        sel.push_back(1u << q);
    }
    for (size_t i = 0; i < p.ops.size(); ++i) {
        const HOp& o = p.ops[i];
        if (o.type == OP_CX) {
            sel[o.q1] ^= sel[o.q0];
            dir[o.q0] ^= dir[o.q1];
            continue;
        }
        FOp g;
        g.hop = (int)i;
        g.run = o.type == OP_M1;
        g.r = sel[o.q0];
        if (g.run) g.d = dir[o.q0];
        else g.r2 = sel[o.q1];
        L.f.push_back(g);
    }
    return L;
}

// The passes over tiles of m bits (the resident path: one pass, m = n) and their
// stages of K directions.
std::vector<PassPlan> plan_passes(const HostPlan& p, const FrameOps& L, int mode, bool tiled, int m, int K,
                                  int max_entries = kMaxPassEntries) {
    const int n = p.n, G = std::min(p.G_swz, m);
    const std::vector<FOp>& f = L.f;
    const Vecs& dir = L.dir;

    // ---- passes: each takes, in time order, every op that commutes with the ops
    // it leaves behind while the tile has room for its direction.  At most m - G
    // directions lie outside the previous tile (G shared ones carry the 128-byte
    // lines); the last tile also holds the directions of the G lowest logical
    // qubits, in whose order the final state is written.
    std::vector<PassPlan> passes;
    std::vector<int> rem(f.size());
    for (size_t i = 0; i < f.size(); ++i) rem[i] = (int)i;
    if (!tiled) {
        PassPlan ps;
        ps.ops = rem;
        for (int q = 0; q < n; ++q) ps.V.push_back(1u << q);
        passes.push_back(std::move(ps));
    } else {
        Vecs prev, last_dirs = dir.first(G);
        // the forward's first tile holds the lines of the given state; the
        // backward's first is its last to run and writes nothing
        for (int i = 0; i < G; ++i) prev.push_back(1u << i);
        bool shares = mode == 0;
        for (;;) {
            const int room = shares ? m - G : m;   // directions outside the previous tile
            struct Try {
                Span v, mod;                 // the tile; the previous tile plus the tile
                std::vector<int> taken, left;
                int fresh = 0;               // directions outside the previous tile
                bool add(uint32_t d, int m, int room) {
                    if (!v.reduce(d)) return true;
                    const bool f = mod.reduce(d) != 0;
                    if (v.dim >= m || (f && fresh >= room)) return false;
                    v.add(d);
                    if (f) { mod.add(d); ++fresh; }
                    return true;
                }
            };
            auto attempt = [&](const Vecs& pre, Try& t) {
                for (uint32_t d : prev) t.mod.add(d);
                for (uint32_t d : pre)
                    if (!t.add(d, m, room)) return false;
                int entries = 0;
                std::vector<char> have(p.entries.size(), 0);
                Waiting w;
                size_t i = 0;
                for (; i < rem.size() && w.d.dim < n; ++i) {
                    const FOp& o = f[rem[i]];
                    bool ok = w.passes(o);
                    const int e = p.ops[o.hop].entry;
                    const bool newe = e >= 0 && !have[e];
                    if (ok && newe) ok = entries < max_entries;
                    if (ok && o.run) ok = t.add(o.d, m, room);
                    if (ok && newe) {
                        have[e] = 1;
                        ++entries;
                    }
                    (ok ? t.taken : t.left).push_back(rem[i]);
                    if (!ok) w.add(o);
                }
                t.left.insert(t.left.end(), rem.begin() + i, rem.end());
                return true;
            };
            Try t;
            bool end = false;
            attempt(Vecs(), t);
            if (t.left.empty()) {
                Try fin;
                if (attempt(last_dirs, fin)) {   // the last tile, or all of it but what it has no room for
                    end = fin.left.empty();
                    t = fin;
                } else {   // move towards the last tile
                    for (uint32_t d : last_dirs) t.add(d, m, room);
                }
            }
            // fill up: G directions shared with the previous tile (its last-tile
            // directions first), then unit vectors
            {
                Vecs shared;
                Span pv;
                for (uint32_t d : prev) pv.add(d);
                for (uint32_t d : last_dirs)
                    if (!pv.reduce(d)) shared.push_back(d);
                shared.append(prev);
                for (uint32_t d : shared)
                    if (t.v.dim - t.fresh < G) t.add(d, m, room);
                for (int q = 0; q < n; ++q) t.add(1u << q, m, room);
                for (uint32_t d : shared) t.add(d, m, room);
            }
            PassPlan ps;
            ps.ops = t.taken;
            ps.V = t.v.basis();
            prev = ps.V;
            shares = true;
            passes.push_back(std::move(ps));
            rem.swap(t.left);
            if (end) break;
        }
    }
    // ---- stages of each pass; a stage whose diagonal ops leave no room for its
    // pads gives its later diagonal ops to a stage of their own
    for (PassPlan& ps : passes) {
        std::vector<StagePlan> st = cut(f, ps.ops, n, K), out;
        for (StagePlan& s : st) {
            std::vector<StagePlan> work{s};
            while (!work.empty()) {
                StagePlan w = work.back();
                work.pop_back();
                StagePlan w0 = w;
                if (pad(w, ps.V, K)) {
                    out.push_back(std::move(w));
                    continue;
                }
                // split in time order: the first half's ops, then the second's
                std::vector<int> a(w0.ops.begin(), w0.ops.begin() + (w0.ops.size() + 1) / 2),
                    b(w0.ops.begin() + (w0.ops.size() + 1) / 2, w0.ops.end());
                std::vector<StagePlan> sb = cut(f, b, n, K), sa = cut(f, a, n, K);
                for (size_t i = sb.size(); i-- > 0;) work.push_back(sb[i]);
                for (size_t i = sa.size(); i-- > 0;) work.push_back(sa[i]);
            }
        }
        ps.stages = std::move(out);
    }
    return passes;
}

// Gives the later half of a pass's stages, on the same tile, to a pass of its own:
// every pass that exceeds a CTA's shared memory by itself, or else the one that needs
// most (the launches share the layout of the schedule's largest counts).  False when
// no pass has two stages.
bool split(std::vector<PassPlan>& passes, const FrameSchedule& S, const HostPlan& p) {
    std::vector<size_t> bytes;
    size_t most = 0;
    for (size_t i = 0; i < passes.size(); ++i) {
        PassNeeds c;
        c.cover(S.passes[i], S.passes[i].ndg);
        const bool dbl = p.dtype == VQC_C128;   // (double-float plans run the same schedules)
        const PassBytes b = pass_bytes(c, p.n, S.mode, p.dtype, dbl, dbl, S.m, S.K);
        bytes.push_back(passes[i].stages.size() > 1 ? b.fixed + b.tile : 0);
        most = std::max(most, bytes.back());
    }
    if (most == 0) return false;
    std::vector<PassPlan> out;
    for (size_t i = 0; i < passes.size(); ++i) {
        PassPlan& ps = passes[i];
        if (bytes[i] < std::min(most, kCtaSharedMemory + 1)) {
            out.push_back(std::move(ps));
            continue;
        }
        const size_t half = (ps.stages.size() + 1) / 2;
        for (size_t from : {(size_t)0, half}) {
            PassPlan q;
            q.V = ps.V;
            q.stages.assign(ps.stages.begin() + from, from ? ps.stages.end() : ps.stages.begin() + half);
            for (const StagePlan& s : q.stages) q.ops.insert(q.ops.end(), s.ops.begin(), s.ops.end());
            out.push_back(std::move(q));
        }
    }
    passes.swap(out);
    return true;
}

FrameSchedule lay_out(const HostPlan& p, const FrameOps& L, int mode, int path, int m, int K,
                      const std::vector<PassPlan>& passes);

}  // namespace

FrameBuilder::FrameBuilder(const HostPlan& plan) : p(plan), ops(new FrameOps(lower(plan))) {}
FrameBuilder::~FrameBuilder() = default;

FrameSchedule FrameBuilder::build(int mode, int path, const std::vector<int>& tiles, int K) const {
    const int n = p.n;
    const bool tiled = path == VQC_PATH_HBM;
    const FrameOps& L = *ops;

    // of the tile sizes offered, the first unless a later one takes no more passes and stages
    int m = 0;
    size_t nst = 0;
    std::vector<PassPlan> passes;
    for (size_t i = 0; i < tiles.size(); ++i) {
        const int t = tiles[i];
        if (i && t == tiles[i - 1]) continue;
        std::vector<PassPlan> q = plan_passes(p, L, mode, tiled, t, K);
        size_t c = 0;
        for (const PassPlan& ps : q) c += ps.stages.size();
        if (m && (q.size() > passes.size() || c > nst)) continue;
        m = t;
        nst = c;
        passes = std::move(q);
    }
    FrameSchedule S = lay_out(p, L, mode, path, m, K, passes);
    if (!tiled) return S;
    const bool dbl = p.dtype == VQC_C128;
    auto bytes = [&](const FrameSchedule& s) {
        PassNeeds c;
        for (const FPass& ps : s.passes) c.cover(ps, ps.ndg);
        const PassBytes b = pass_bytes(c, n, mode, p.dtype, dbl, dbl, m, K);
        return b.fixed + b.tile;
    };
    // complex128: two CTAs an SM, where passes of fewer table entries, at most twice as many,
    // give them (double-float rings of RZZ, 15 qubits x 57, 5 layers, step: 4.58 ms with one CTA
    // an SM, 3.81 with two)
    if (dbl && bytes(S) > kHalfSharedMemory)
        for (int entries : {72, 56, 40}) {
            std::vector<PassPlan> q = plan_passes(p, L, mode, tiled, m, K, entries);
            if (q.size() > 2 * passes.size()) break;
            FrameSchedule T = lay_out(p, L, mode, path, m, K, q);
            if (bytes(T) <= kHalfSharedMemory) return T;
        }
    while (bytes(S) > kCtaSharedMemory && split(passes, S, p)) S = lay_out(p, L, mode, path, m, K, passes);
    return S;
}

namespace {

// The schedule's records from its passes and stages.
FrameSchedule lay_out(const HostPlan& p, const FrameOps& L, int mode, int path, int m, int K,
                      const std::vector<PassPlan>& passes) {
    const int n = p.n;
    const bool tiled = path == VQC_PATH_HBM;
    const std::vector<FOp>& f = L.f;
    const Vecs &dir = L.dir, &sel = L.sel;
    const int G = std::min(p.G_swz, m), np = (int)passes.size(), nout = n - m;
    FrameSchedule S;
    S.mode = mode;
    S.K = K;
    S.m = m;
    S.path = path;
    S.nout = nout;

    // ---- addresses, slots and records, in the order the passes run (the backward
    // from the last).  A pass reads the state at the addresses M s; the forward
    // starts at M = 1 (a state in logical order before the first gate) and writes
    // logical order at its end, the backward starts there.
    Vecs M(n), Minv(n);   // columns: address of e_i; index vector of address bit i
    for (int i = 0; i < n; ++i) {
        M[i] = Minv[i] = 1u << i;
        if (mode == 1) {
            Minv[i] = dir[i];
            M[i] = 0;
            for (int j = 0; j < n; ++j) M[i] |= ((sel[j] >> i) & 1u) << j;
        }
    }
    S.passes.resize(np);
    S.phase_tables.resize(np);
    S.fin = FFinal{};
    Rng rng;
    for (int step = 0; step < np; ++step) {
        const int pi = mode == 0 ? step : np - 1 - step;
        const PassPlan& ps = passes[pi];
        const bool last = pi == np - 1, end = step == np - 1;
        FPass fp{};
        // the tile's addresses as read: a reduced echelon basis with the G low units first
        Vecs gin, vin, opos, ovec;
        auto echelon = [&](const Vecs& addr, Vecs& g) {
            uint32_t lowm = (1u << G) - 1;
            g.clear();
            for (int i = 0; i < G; ++i) g.push_back(1u << i);
            Vecs r;
            for (uint32_t a : addr) r.push_back(a & ~lowm);
            Span sp;
            for (uint32_t a : r) sp.add(a);
            Vecs b = sp.basis();   // ascending highest bit
            for (size_t i = 0; i < b.size(); ++i)   // fully reduce
                for (size_t j = 0; j < i; ++j) {
                    const int h = 31 - __builtin_clz(b[j]);
                    if ((b[i] >> h) & 1) b[i] ^= b[j];
                }
            g.append(b);
        };
        if (tiled) {
            Vecs addr;
            for (uint32_t v : ps.V) addr.push_back(image(M, v));
            echelon(addr, gin);
        } else {
            for (int i = 0; i < n; ++i) gin.push_back(1u << i);
        }
        uint32_t pivots = 0;
        for (uint32_t g : gin) pivots |= 1u << (31 - __builtin_clz(g));
        for (uint32_t g : gin) vin.push_back(image(Minv, g));
        for (int b = 0; b < n; ++b)
            if (!((pivots >> b) & 1)) {
                opos.push_back(1u << b);
                ovec.push_back(Minv[b]);
            }
        const Coords coord(vin);

        // directions that the written lines will hold: ones that the next tile has
        // too, at the forward's end the last logical ones
        Vecs line;
        if (end) {
            if (mode == 0) line = dir.first(G);
        } else {
            // V intersect V': vectors of V whose sum with V' vectors vanishes
            const Vecs &a = ps.V, &b = passes[pi + (mode == 0 ? 1 : -1)].V;
            uint32_t piv[32] = {0}, ca[32] = {0};
            auto ins = [&](uint32_t v, uint32_t c, bool fromb) {
                while (v) {
                    const int h = 31 - __builtin_clz(v);
                    if (!piv[h]) {
                        piv[h] = v;
                        ca[h] = c;
                        return;
                    }
                    v ^= piv[h];
                    c ^= ca[h];
                }
                if (fromb && (int)line.size() < G) line.push_back(c);
            };
            // c: the part of the combination that comes from V
            for (uint32_t v : a) ins(v, v, false);
            for (uint32_t v : b) ins(v, 0, true);
        }

        // swizzle: slot bits 0..G-1 of tile bit i >= G also get column F[i], chosen so
        // that lanes hit distinct banks in every stage and both copies
        Vecs F(m);
        const int tb = m - K, gl = std::min(G, tb);   // lanes that must differ in the low gl slot bits
        auto slot_of = [&](uint32_t c) {
            uint32_t s = c;
            for (uint32_t hi = c >> G; hi; hi &= hi - 1) s ^= F[G + __builtin_ctz(hi)];
            return s;
        };
        auto bank = [&](uint32_t v) { return slot_of(coord(v)) & ((1u << G) - 1); };
        // the stages' thread spaces: V's vectors even on the runs' selectors, without the pads
        struct Threads {
            Vecs basis;
        };
        std::vector<Threads> th(ps.stages.size());
        for (size_t si = 0; si < ps.stages.size(); ++si) {
            const StagePlan& s = ps.stages[si];
            Span sp;
            for (uint32_t d : s.D) sp.add(d);
            for (uint32_t v : annihilated(vin, s.R))
                if (sp.add(v)) th[si].basis.push_back(settle(s, v));
        }
        const int vbits = p.dtype == VQC_C64 ? 1 : 0;   // bits inside a 16-byte vector of amplitudes
        {
            // sets of tile coordinates whose banks should be independent, and how many
            struct Want {
                int rank, weight;
                uint32_t mask;
                Vecs c, b;   // tile coordinates, their banks under F
            };
            std::vector<Want> want;
            want.reserve(th.size() + 2);
            for (const Threads& t : th) {
                want.push_back(Want{gl, 1, (1u << gl) - 1, {}, {}});
                for (uint32_t v : t.basis) want.back().c.push_back(coord(v));
            }
            want.push_back(Want{0, 1, (1u << G) - 1, {}, {}});
            for (int i = vbits; i < std::min(m, G + vbits); ++i) want.back().c.push_back(1u << i);
            want.back().rank = (int)want.back().c.size();
            if (!line.empty()) {
                want.push_back(Want{G - vbits, 2, (1u << G) - 1, {}, {}});
                for (uint32_t v : line) want.back().c.push_back(coord(v));
            }
            auto score = [&](int limit) {
                int bad = 0;
                for (const Want& w : want) {
                    uint32_t piv[4] = {0, 0, 0, 0};
                    int rank = 0;
                    for (size_t i = 0; i < w.b.size() && rank < w.rank; ++i) {
                        uint32_t v = w.b[i] & w.mask;
                        while (v) {
                            const int h = 31 - __builtin_clz(v);
                            if (!piv[h]) {
                                piv[h] = v;
                                ++rank;
                                break;
                            }
                            v ^= piv[h];
                        }
                    }
                    bad += w.weight * (w.rank - rank);
                    if (bad > limit) break;
                }
                return bad;
            };
            auto turn = [&](int i, uint32_t delta) {   // F[i] ^= delta
                F[i] ^= delta;
                for (Want& w : want)
                    for (size_t k = 0; k < w.c.size(); ++k)
                        if ((w.c[k] >> i) & 1) w.b[k] ^= delta;
            };
            // from the plain fold of the high bits, one random column at a time
            for (int i = G; i < m; ++i) F[i] = 1u << (i % G);
            for (Want& w : want)
                for (uint32_t c : w.c) w.b.push_back(slot_of(c) & ((1u << G) - 1));
            int best = score(1 << 20);
            for (int trial = 0; trial < 64 && best > 0 && m > G; ++trial) {
                const int i = G + (int)((rng.next() >> 4) % (uint32_t)(m - G));
                const uint32_t delta = (rng.next() >> 8) & ((1u << G) - 1);
                if (!delta) continue;
                turn(i, delta);
                const int bad = score(best);
                if (bad <= best) best = bad;
                else turn(i, delta);
            }
        }

        // written order: the line's directions lowest, chosen so that the lanes that
        // read the tile back differ in their banks
        Vecs gout, vout;
        if (end && mode == 0 && tiled) {
            Vecs addr;
            for (uint32_t v : ps.V) {
                uint32_t a = 0;
                for (int j = 0; j < n; ++j) a |= (uint32_t)odd(sel[j] & v) << j;
                addr.push_back(a);
            }
            echelon(addr, gout);
            for (uint32_t g : gout) vout.push_back(image(dir, g));
        } else if (!tiled) {   // given and final order of whole states
            gout = gin;
            vout = dir;
            if (mode == 1)
                for (int i = 0; i < n; ++i) vout[i] = 1u << i;
        } else if (end) {   // the backward's end: nothing is written
            gout = gin;
            vout = vin;
        } else {
            gout = gin;
            Vecs l = line;
            Span bs;
            if (vbits) {   // the vector's own bit: the one whose bank the others can spare
                for (size_t i = 0; i < l.size(); ++i) {
                    Vecs b;
                    for (size_t j = 0; j < l.size(); ++j)
                        if (j != i) b.push_back(bank(l[j]));
                    if (rank_of(b) == (int)l.size() - 1 || i + 1 == l.size()) {
                        std::swap(l[0], l[i]);
                        break;
                    }
                }
            }
            vout = l;
            Span sp;
            for (uint32_t v : vout) sp.add(v);
            for (size_t i = vbits; i < vout.size(); ++i) bs.add(bank(vout[i]));
            Vecs others;
            for (uint32_t v : vin)
                if (sp.add(v)) others.push_back(v);
            for (size_t i = 0; i < others.size(); ++i)
                if (bs.reduce(bank(others[i]))) {
                    std::swap(others[0], others[i]);
                    break;
                }
            vout.append(others);
        }
        if (end && mode == 0 && tiled && vbits) {   // the same for the final order's fifth bit
            Span bs;
            for (int i = 1; i < G; ++i) bs.add(bank(vout[i]));
            for (int i = G; i < m; ++i)
                if (bs.reduce(bank(vout[i]))) {
                    std::swap(vout[G], vout[i]);
                    std::swap(gout[G], gout[i]);
                    break;
                }
        }
        for (int i = 0; i < m; ++i) {   // in / out: before and after the pass in circuit order
            (mode == 0 ? fp.gin : fp.gout)[i] = gin[i];
            (mode == 0 ? fp.gout : fp.gin)[i] = gout[i];
            (mode == 0 ? fp.sin : fp.sout)[i] = (int32_t)slot_of(coord(vin[i]));
            (mode == 0 ? fp.sout : fp.sin)[i] = (int32_t)slot_of(coord(vout[i]));
        }
        for (int o = 0; o < nout; ++o) {
            fp.oin[o] = fp.oout[o] = opos[o];
            if (!(end && mode == 0)) continue;
            // logical order: the tile's address with the line's bits (and its other
            // pivots) zero, and the slot that amplitude is in
            uint32_t a = 0;
            for (int j = 0; j < n; ++j) a |= (uint32_t)odd(sel[j] & ovec[o]) << j;
            for (int i = m - 1; i >= 0; --i)
                if ((a >> (31 - __builtin_clz(gout[i]))) & 1) {
                    a ^= gout[i];
                    fp.oslot[o] ^= fp.sout[i];
                }
            fp.oout[o] = a;
        }

        // tables of the pass (the resident path keeps the plan's own slots)
        std::vector<int> slot_id(p.entries.size(), -1), acc_id(p.accs.size(), -1);
        if (tiled) {
            fp.ps_begin = (int32_t)S.pass_entries.size();
            for (int want = 1; want >= 0; --want) {
                if (!want) fp.sh_begin = (int32_t)S.pass_entries.size();
                for (int x : ps.ops) {
                    const int e = p.ops[f[x].hop].entry;
                    if (e < 0 || slot_id[e] >= 0 || p.entries[e].per_sample != want) continue;
                    slot_id[e] = want ? fp.ps_count++ : fp.sh_count++;
                    S.pass_entries.push_back(e);
                }
            }
            fp.acc_begin = (int32_t)S.pass_accs.size();
            for (int x : ps.ops) {
                const int e = p.ops[f[x].hop].entry;
                if (e < 0 || p.entries[e].acc == 0xffff || acc_id[p.entries[e].acc] >= 0) continue;
                acc_id[p.entries[e].acc] = fp.acc_count++;
                S.pass_accs.push_back(p.entries[e].acc);
            }
        } else {
            for (size_t i = 0; i < p.entries.size(); ++i) slot_id[i] = p.entries[i].slot;
            for (size_t i = 0; i < p.accs.size(); ++i) acc_id[i] = (int)i;
        }

        // stage records
        fp.stage_begin = (int32_t)S.stages.size();
        fp.op_begin = (int32_t)S.ops.size();
        fp.seg_begin = (int32_t)S.segs.size();
        for (size_t si = 0; si < ps.stages.size(); ++si) {
            const StagePlan& s = ps.stages[si];
            FStage st{};
            for (int k = 0; k < K; ++k) st.sigma[k] = (int32_t)slot_of(coord(s.D[k]));
            // thread vectors: the first gl with independent banks
            Vecs tv, others;
            Span bs;
            for (uint32_t v : th[si].basis) {
                if ((int)tv.size() < gl && bs.add(bank(v) & ((1u << gl) - 1))) tv.push_back(v);
                else others.push_back(v);
            }
            tv.append(others);
            st.nthreadbits = (uint8_t)tv.size();
            // parities outside the registers
            Vecs outside;
            auto ref = [&](uint32_t r) -> uint8_t {
                for (int k = 0; k < K; ++k)
                    if (odd(r & s.D[k])) return (uint8_t)k;
                size_t i = 0;
                while (i < outside.size() && outside[i] != r) ++i;
                if (i == outside.size()) outside.push_back(r);
                return (uint8_t)(kRefPhys + i);
            };
            auto record = [&](int x) {
                const FOp& o = f[x];
                const HOp& h = p.ops[o.hop];
                DOp d{};
                if (h.entry >= 0) {
                    const DEntry& e = p.entries[h.entry];
                    d.slot = (uint16_t)slot_id[h.entry];
                    d.flags = (uint8_t)((e.per_sample ? OPF_PER_SAMPLE : 0) |
                                        (e.acc != 0xffff ? OPF_HAS_ACC : 0) | h.gen);
                    d.aux = e.acc != 0xffff ? (uint16_t)acc_id[e.acc] : (uint16_t)0xffff;
                }
                if (o.run) {
                    int k = 0;
                    while (s.D[k] != o.d || s.R[k] != o.r) ++k;
                    d.a = (uint8_t)k;
                    d.code = (uint8_t)(DC_M1 + k);
                    return d;
                }
                uint8_t ra = ref(o.r), rb = ref(o.r2);
                const bool la = ra < kRefPhys, lb = rb < kRefPhys;
                if (h.type == OP_CZ) {
                    if (la && lb) {
                        if (ra > rb) std::swap(ra, rb);
                        d.code = (uint8_t)(DC_CZ_LL + cz_pair_index(ra, rb));
                    } else if (la || lb) {
                        if (!la) std::swap(ra, rb);
                        d.code = (uint8_t)(DC_CZ_PL + ra);
                    } else {
                        d.code = DC_CZ_PP;
                    }
                } else if (la && lb) {
                    d.code = (uint8_t)(DC_PH2_LL + cz_pair_index(std::min(ra, rb), std::max(ra, rb)));
                } else if (la || lb) {
                    d.code = (uint8_t)(DC_PH2_PL + (la ? ra : rb));
                } else {
                    d.code = DC_PH2_PP;
                }
                d.a = ra;
                d.b = rb;
                return d;
            };
            // order of a diagonal group: PP, PL by position, LL CZ, LL phases
            auto key = [](const DOp& d) {
                if (d.code == DC_CZ_PP || d.code == DC_PH2_PP) return 0;
                if (d.code >= DC_CZ_PL && d.code < DC_CZ_PP) return 1 + d.code - DC_CZ_PL;
                if (d.code >= DC_PH2_PL && d.code < DC_PH2_PP) return 1 + d.code - DC_PH2_PL;
                return d.code < DC_CZ_PL ? 10 : 11;
            };
            // each op's round: a run follows the diagonal ops it does not commute with in
            // the same round or an earlier one, and the run before it on its position; a
            // diagonal op follows such runs by a round
            std::vector<std::vector<int>> round(1);
            int after_run[kMaxK] = {0}, after_diag[kMaxK] = {0};   // earliest rounds, by position
            for (int x : s.ops) {
                const FOp& o = f[x];
                int rd = 0;
                for (int k = 0; k < K; ++k) {
                    const bool meets = o.run ? s.D[k] == o.d : odd(o.r & s.D[k]) || odd(o.r2 & s.D[k]);
                    if (meets) rd = std::max({rd, after_run[k], o.run ? after_diag[k] : 0});
                }
                for (int k = 0; k < K; ++k) {
                    if (o.run && s.D[k] == o.d) after_run[k] = rd + 1;
                    if (!o.run && (odd(o.r & s.D[k]) || odd(o.r2 & s.D[k]))) after_diag[k] = std::max(after_diag[k], rd);
                }
                if ((int)round.size() <= rd) round.resize(rd + 1);
                round[rd].push_back(x);
            }
            st.op_begin = (int32_t)S.ops.size();
            st.seg_begin = (int32_t)S.segs.size();
            bool phases = false;
            for (int x : s.ops) phases = phases || p.ops[f[x].hop].type == OP_PH2;
            for (size_t rd = 0; rd < round.size() && !s.ops.empty(); ++rd) {
                FSeg sg{};
                std::vector<DOp> diag, runs;
                for (int x : round[rd]) {
                    const DOp d = record(x);
                    if (f[x].run) {
                        sg.pmask |= (uint8_t)(1u << d.a);
                        if (d.flags & OPF_PER_SAMPLE) sg.flags |= kSegPs;
                        const DEntry& e = p.entries[p.ops[f[x].hop].entry];
                        const int form = phases ? 0 : run_form(&p.consts[e.cfirst], e.ccount);
                        sg.flags |= (uint8_t)((form & 1 ? kSegQ : 0) | (form & 2 ? kSegP : 0));
                        runs.push_back(d);
                    } else {
                        if (d.flags & OPF_HAS_ACC) sg.flags |= kSegA;
                        if (key(d) == 11) sg.flags |= (uint8_t)(kSegL | (d.flags & OPF_PER_SAMPLE ? kSegPs : 0));
                        diag.push_back(d);
                    }
                }
                std::stable_sort(diag.begin(), diag.end(), [&](const DOp& a, const DOp& b) { return key(a) < key(b); });
                std::sort(runs.begin(), runs.end(), [](const DOp& a, const DOp& b) { return a.a < b.a; });
                sg.op_begin = (int32_t)S.ops.size();
                S.ops.insert(S.ops.end(), diag.begin(), diag.end());
                sg.run_begin = (int32_t)S.ops.size();
                S.ops.insert(S.ops.end(), runs.begin(), runs.end());
                sg.op_end = (int32_t)S.ops.size();
                // tables: two-local phases, and (double-float) the runs' own diagonals
                const bool factors = p.dtype == VQC_C128;
                const bool has[2] = {(sg.flags & kSegL) || (factors && (sg.flags & kSegQ)),
                                     factors && (sg.flags & kSegP)};
                for (int k = 0; k < 2; ++k) sg.dg[k] = has[k] ? 0 : kNoDiagonal;   // numbered below
                S.segs.push_back(sg);
            }
            st.seg_end = (int32_t)S.segs.size();
            if (st.seg_begin == st.seg_end ||
                (st.seg_begin + 1 == st.seg_end && S.segs.back().op_begin == S.segs.back().run_begin)) {
                st.kind = kStagePure;
                st.pmask = st.seg_begin < st.seg_end ? S.segs.back().pmask : 0;
            }
            if (phases) st.kind |= kStagePhases;
            st.op_end = (int32_t)S.ops.size();
            st.nsel = (uint8_t)outside.size();
            auto word = [&](uint32_t v) {
                uint32_t w = 0;
                for (size_t i = 0; i < outside.size(); ++i) w |= (uint32_t)odd(outside[i] & v) << i;
                return w;
            };
            for (size_t i = 0; i < tv.size(); ++i) {
                st.tau[i] = (int32_t)slot_of(coord(tv[i]));
                st.tmask[i] = word(tv[i]);
            }
            for (int o = 0; o < nout; ++o) {
                const uint32_t v = settle(s, ovec[o]);
                S.flips.push_back(FFlip{(int32_t)slot_of(coord(v ^ ovec[o])), word(v)});
            }
            S.stages.push_back(st);
            if (last && si + 1 == ps.stages.size()) {
                for (size_t i = 0; i < tv.size(); ++i)
                    for (int j = 0; j < n; ++j)
                        S.fin.tmask[i] |= (uint32_t)odd(sel[j] & tv[i]) << j;
                for (int o = 0; o < nout; ++o)
                    for (int j = 0; j < n; ++j)
                        S.fin.omask[o] |= (uint32_t)odd(sel[j] & settle(s, ovec[o])) << j;
                for (int j = 0; j < n; ++j)
                    for (int k = 0; k < K; ++k) S.fin.lmask[j] |= (uint8_t)(odd(sel[j] & s.D[k]) << k);
            }
        }
        fp.stage_end = (int32_t)S.stages.size();
        fp.op_end = (int32_t)S.ops.size();
        fp.seg_end = (int32_t)S.segs.size();
        // the tables: those of two-local phases, then double-float's alone
        for (int own = 0; own < 2; ++own) {
            for (int i = fp.seg_begin; i < fp.seg_end; ++i)
                for (int k = 0; k < 2; ++k) {
                    FSeg& sg = S.segs[i];
                    if (sg.dg[k] != kNoDiagonal && (k == 0 && (sg.flags & kSegL)) == !own) sg.dg[k] = (uint16_t)fp.ndg++;
                }
            if (!own) S.phase_tables[pi] = fp.ndg;
        }
        S.passes[pi] = fp;

        // the frame after the pass: M' vout[i] = gin[i], M' = M on the outer vectors
        if (!end) {
            Vecs Mi(n);
            for (int o = 0; o < nout; ++o) Mi[31 - __builtin_clz(opos[o])] = ovec[o];
            for (int i = 0; i < m; ++i) {
                const int h = 31 - __builtin_clz(gin[i]);
                uint32_t v = vout[i];
                for (int o = 0; o < nout; ++o)
                    if (gin[i] & opos[o]) v ^= ovec[o];
                Mi[h] = v;
            }
            Minv = Mi;
            M = inverse(Minv);
        }
    }
    return S;
}

}  // namespace

std::vector<uint8_t> export_frames(const HostPlan& p) {
    std::vector<uint8_t> out = {'V', 'Q', 'C', 'F'};
    auto put = [&](const void* d, size_t bytes) {
        const uint8_t* b = static_cast<const uint8_t*>(d);
        out.insert(out.end(), b, b + bytes);
    };
    auto num = [&](int32_t v) { put(&v, 4); };
    num((int32_t)p.frames.size());
    for (const FrameSchedule& s : p.frames) {
        for (int v : {s.mode, s.K, s.m, s.path, s.nout, (int)s.ops.size(), (int)s.stages.size(),
                      (int)s.passes.size(), (int)s.pass_entries.size(), (int)s.pass_accs.size(), (int)s.segs.size()})
            num(v);
        put(s.ops.data(), s.ops.size() * sizeof(DOp));
        put(s.stages.data(), s.stages.size() * sizeof(FStage));
        put(s.segs.data(), s.segs.size() * sizeof(FSeg));
        put(s.flips.data(), s.flips.size() * sizeof(FFlip));
        put(s.passes.data(), s.passes.size() * sizeof(FPass));
        put(s.pass_entries.data(), s.pass_entries.size() * 4);
        put(s.pass_accs.data(), s.pass_accs.size() * 4);
        put(&s.fin, sizeof(FFinal));
    }
    return out;
}

}  // namespace vqc
