"""CPU tests of the frame schedules (csrc/frame.h): the exported records, run on
the CPU with the kernels' addressing, against the oracle.

Every schedule of every circuit is executed tile by tile and stage by stage
from the records alone: gather, register blocks, ops, scatter, <Z> and the
adjoint gradients.  Each copy and each stage must touch every slot of a tile
exactly once.
"""
import ctypes
import struct

import numpy as np
import pytest

from oracle import oracle as orc
from paper_2607_11985_gb300 import binding as B
from paper_2607_11985_gb300 import workloads as wl
from tests import plan_emulator as pe

DOP = pe.DOP
FSTAGE = np.dtype([("tau", "<i4", 16), ("tmask", "<u4", 16), ("sigma", "<i4", 5), ("seg_begin", "<i4"),
                   ("seg_end", "<i4"), ("op_begin", "<i4"), ("op_end", "<i4"), ("nthreadbits", "u1"),
                   ("nsel", "u1"), ("kind", "u1"), ("pmask", "u1"), ("pad1", "<i4", 2)])
FSEG = np.dtype([("op_begin", "<i4"), ("run_begin", "<i4"), ("op_end", "<i4"), ("flags", "u1"), ("pmask", "u1"),
                 ("dg", "<u2", 2), ("pad", "<u2")])
PS, Q, P_, ACC, LL = (1 << i for i in range(5))
NO_DIAGONAL = 0xffff
FFLIP = np.dtype([("slot", "<i4"), ("mask", "<u4")])
FPASS = np.dtype([("stage_begin", "<i4"), ("stage_end", "<i4"), ("op_begin", "<i4"), ("op_end", "<i4"),
                  ("seg_begin", "<i4"), ("seg_end", "<i4"), ("gin", "<u4", 14), ("gout", "<u4", 14), ("sin", "<i4", 14), ("sout", "<i4", 14),
                  ("oin", "<u4", 20), ("oout", "<u4", 20), ("oslot", "<i4", 20), ("ps_begin", "<i4"), ("ps_count", "<i4"),
                  ("sh_begin", "<i4"), ("sh_count", "<i4"), ("acc_begin", "<i4"), ("acc_count", "<i4"), ("ndg", "<i4")])
FFINAL = np.dtype([("tmask", "<u4", 16), ("omask", "<u4", 20), ("lmask", "u1", 32)])
MAX_PASS_ENTRIES = 96


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2607_11985_gb300 import build
    build.build()


def compile_spec(spec, dtype):
    arr = B.gates_array(spec)
    return B.vqc_compile(arr, len(spec.gates), spec.n, spec.num_x, spec.num_w, dtype)


def frames(plan):
    fn = B.lib().vqc_frames_export
    n = ctypes.c_size_t(0)
    assert fn(plan, None, ctypes.byref(n)) == 0
    buf = ctypes.create_string_buffer(n.value)
    assert fn(plan, buf, ctypes.byref(n)) == 0
    blob, off = buf.raw, 4
    assert blob[:4] == b"VQCF"
    (count,) = struct.unpack_from("<i", blob, off)
    off += 4
    out = []
    for _ in range(count):
        mode, K, m, path, nout, nops, nst, nps, npe, npa, nsg = struct.unpack_from("<11i", blob, off)
        off += 44
        s = dict(mode=mode, K=K, m=m, path=path, nout=nout)
        for name, dt, k in (("ops", DOP, nops), ("stages", FSTAGE, nst), ("segs", FSEG, nsg), ("flips", FFLIP, nst * nout),
                            ("passes", FPASS, nps), ("pass_entries", np.dtype("<i4"), npe),
                            ("pass_accs", np.dtype("<i4"), npa), ("fin", FFINAL, 1)):
            s[name] = np.frombuffer(blob, dt, k, off)
            off += dt.itemsize * k
        s["flips"] = s["flips"].reshape(nst, nout)
        out.append(s)
    assert off == len(blob)
    return out


def lin(cols, count):
    """XOR of cols[i] over the set bits of 0 .. 2^count - 1."""
    v = np.zeros(1, np.int64)
    for i in range(count):
        v = np.concatenate([v, v ^ int(cols[i])])
    return v


def parity(v):
    v = np.asarray(v, np.int64).copy()
    for s in (16, 8, 4, 2, 1):
        v ^= v >> s
    return v & 1


class Emulator:
    def __init__(self, plan, s, xb, w):
        self.p, self.s, self.xb, self.w = plan, s, xb, w
        self.n, self.m, self.K = plan.n, s["m"], s["K"]

    def tables(self, ps):
        if self.s["path"] == 0:
            return self.p.tables(self.xb, self.w) + (np.arange(len(self.p.accs)),)
        pe_ = self.s["pass_entries"]
        ids = [pe_[ps[k + "_begin"]:ps[k + "_begin"] + ps[k + "_count"]] for k in ("ps", "sh")]
        assert len(ids[0]) + len(ids[1]) <= MAX_PASS_ENTRIES
        val = [[self.p.entry_value(int(e), self.xb, self.w) for e in i] for i in ids]
        return val[0], val[1], self.s["pass_accs"][ps["acc_begin"]:ps["acc_begin"] + ps["acc_count"]]

    def addresses(self, ps, which):
        a, s = lin(ps["g" + which], self.m), lin(ps["s" + which], self.m)
        assert sorted(s) == list(range(1 << self.m))
        o = lin(ps["o" + which], self.s["nout"])
        # 16-byte vectors, and whole lines: the lowest tile bits are the lowest
        # address bits, which nothing else reaches
        low = min(self.p.G, self.m)
        assert list(ps["g" + which][:low]) == [1 << i for i in range(low)]
        assert all(int(v) % (1 << low) == 0 for v in ps["g" + which][low:self.m]) and not np.any(o % (1 << low))
        allad = (o[:, None] ^ a[None, :]).ravel()
        assert sorted(allad) == list(range(1 << self.n))   # tiles partition the state
        return a, s, o

    def stage(self, si, tau):
        st = self.s["stages"][si]
        nb = int(st["nthreadbits"])
        assert nb == self.m - self.K
        slot = pb = 0
        for o in range(self.s["nout"]):
            if (tau >> o) & 1:
                slot ^= int(self.s["flips"][si, o]["slot"])
                pb ^= int(self.s["flips"][si, o]["mask"])
        idx = (lin(st["tau"], nb)[:, None] ^ lin(st["sigma"], self.K)[None, :]) ^ slot
        assert sorted(idx.ravel()) == list(range(1 << self.m))
        return st, idx, lin(st["tmask"].astype(np.int64), nb) ^ pb

    def bit(self, ref, pb):
        ref = int(ref)
        if ref >= 8:
            return ((pb >> (ref - 8)) & 1)[:, None] * np.ones((1, 1 << self.K), np.int64)
        return ((np.arange(1 << self.K) >> ref) & 1)[None, :] * np.ones((len(pb), 1), np.int64)

    def op(self, op, pb, tabs, blocks, adj, acc):
        t, oa, ob = pe.op_type(op)
        tab = tabs[0] if op["flags"] & pe.OPF_PER_SAMPLE else tabs[1]
        if acc is not None and op["flags"] & pe.OPF_HAS_ACC:
            a, l = blocks
            k = tabs[2][op["aux"]]
            if t == pe.OP_M1:
                lo = np.array([r for r in range(1 << self.K) if not (r >> oa) & 1])
                pp, ll = (a[:, lo], a[:, lo | (1 << oa)]), (l[:, lo], l[:, lo | (1 << oa)])
                for i in range(2):
                    for j in range(2):
                        z = (pp[i] * ll[j].conj()).sum()
                        acc[k, 2 * (2 * i + j)] += z.real
                        acc[k, 2 * (2 * i + j) + 1] += z.imag
            else:
                ba, bb = self.bit(oa, pb), self.bit(ob, pb)
                g = (1 - 2 * bb) * ba if op["flags"] & pe.OPF_GEN_CRZ else 1 - 2 * (ba ^ bb)
                acc[k, 0] += (g * (l.conj() * a).imag).sum()
        for a in blocks:
            if t == pe.OP_M1:
                M = tab[op["slot"]]
                M = M.conj().T if adj else M
                lo = np.array([r for r in range(1 << self.K) if not (r >> oa) & 1])
                u, v = a[:, lo].copy(), a[:, lo | (1 << oa)].copy()
                a[:, lo], a[:, lo | (1 << oa)] = M[0, 0] * u + M[0, 1] * v, M[1, 0] * u + M[1, 1] * v
            elif t == pe.OP_CZ:
                a *= 1 - 2 * (self.bit(oa, pb) & self.bit(ob, pb))
            else:
                assert t == pe.OP_PH2
                ph = tab[op["slot"]]
                ph = ph.conj() if adj else ph
                a *= ph[self.bit(oa, pb) + 2 * self.bit(ob, pb)]

    def check_rounds(self, st, ndg):
        """A stage's rounds cover its ops; diagonal ops in the order the kernels walk
        them, runs by position, flags and tables as they are read there."""
        ops, at = self.s["ops"], st["op_begin"]
        for sg in self.s["segs"][st["seg_begin"]:st["seg_end"]]:
            assert sg["op_begin"] == at and sg["op_begin"] <= sg["run_begin"] <= sg["op_end"]
            at = sg["op_end"]
            diag, runs = ops[sg["op_begin"]:sg["run_begin"]], ops[sg["run_begin"]:sg["op_end"]]
            pos = [int(o["a"]) for o in runs]
            assert all(pe.op_type(o)[0] == pe.OP_M1 for o in runs)
            assert pos == sorted(set(pos)) and sg["pmask"] == sum(1 << q for q in pos)
            keys = []
            for o in diag:
                t, a, b = pe.op_type(o)
                assert t in (pe.OP_CZ, pe.OP_PH2)
                la, lb = a < 8, b < 8
                keys.append((10 if t == pe.OP_CZ else 11) if la and lb else 1 + min(int(a), int(b)) if la or lb else 0)
            assert keys == sorted(keys)
            ps = any(int(o["flags"]) & pe.OPF_PER_SAMPLE for k, o in zip(keys, diag) if k == 11)
            assert bool(sg["flags"] & PS) == (ps or any(int(o["flags"]) & pe.OPF_PER_SAMPLE for o in runs))
            assert bool(sg["flags"] & ACC) == any(int(o["flags"]) & pe.OPF_HAS_ACC for o in diag)
            assert bool(sg["flags"] & LL) == (11 in keys)
            dbl = self.p.dtype == 1   # complex128 schedules count double-float's own tables
            want = [11 in keys or (dbl and bool(sg["flags"] & Q)), dbl and bool(sg["flags"] & P_)]
            for k in range(2):
                assert (sg["dg"][k] != NO_DIAGONAL) == want[k] and (not want[k] or sg["dg"][k] < ndg)
        assert at == st["op_end"]
        sg = self.s["segs"][st["seg_begin"]:st["seg_end"]]
        phases = any(pe.op_type(o)[0] == pe.OP_PH2 for o in ops[st["op_begin"]:st["op_end"]])
        assert bool(st["kind"] & 2) == phases
        assert bool(st["kind"] & 1) == (len(sg) == 0 or (len(sg) == 1 and sg[0]["op_begin"] == sg[0]["run_begin"]))
        assert st["pmask"] == (sg[0]["pmask"] if st["kind"] & 1 and len(sg) else 0)

    def logical(self, tau):
        """Logical basis state of [thread, r] of the last stage's blocks of tile tau."""
        f = self.s["fin"][0]
        w = lin(f["tmask"].astype(np.int64), self.m - self.K)
        for o in range(self.s["nout"]):
            if (tau >> o) & 1:
                w = w ^ int(f["omask"][o])
        k = np.zeros((len(w), 1 << self.K), np.int64)
        for j in range(self.n):
            k |= (((w >> j) & 1)[:, None] ^ parity(np.arange(1 << self.K) & int(f["lmask"][j]))[None, :]) << j
        return k

    def forward(self, psi0=None):
        mem = np.zeros(1 << self.n, complex)
        mem[0] = 1
        if psi0 is not None:
            mem[:] = psi0
        passes = self.s["passes"]
        for pi, ps in enumerate(passes):
            tabs = self.tables(ps)
            ai, si_, oi = self.addresses(ps, "in")
            ao, so, oo = self.addresses(ps, "out")
            new = np.zeros_like(mem)
            for tau in range(1 << self.s["nout"]):
                sm = np.zeros(1 << self.m, complex)
                sm[si_] = mem[oi[tau] ^ ai]
                for si in range(ps["stage_begin"], ps["stage_end"]):
                    st, idx, pb = self.stage(si, tau)
                    self.check_rounds(st, int(ps["ndg"]))
                    a = sm[idx]
                    for op in self.s["ops"][st["op_begin"]:st["op_end"]]:
                        self.op(op, pb, tabs, (a,), False, None)
                    sm[idx] = a
                new[oo[tau] ^ ao] = sm[so ^ lin(ps["oslot"], self.s["nout"])[tau]]
                if pi + 1 < len(passes):   # in place: a tile is written where it was read
                    assert set(oo[tau] ^ ao) == set(oi[tau] ^ ai)
                else:
                    k = self.logical(tau)
                    assert np.array_equal(new[k], sm[idx])
            mem = new
        return mem

    def backward(self, psi, gE):
        k = np.arange(1 << self.n)
        O = sum(gE[j] * (1 - 2 * ((k >> j) & 1)) for j in range(self.n))
        mem, lam = psi.copy(), None
        acc = np.zeros((len(self.p.accs), 8))
        passes = self.s["passes"]
        for pi in range(len(passes) - 1, -1, -1):
            ps = passes[pi]
            tabs = self.tables(ps)
            ai, si_, oi = self.addresses(ps, "in")
            ao, so, oo = self.addresses(ps, "out")
            new, newl = np.zeros_like(mem), np.zeros_like(mem)
            for tau in range(1 << self.s["nout"]):
                sm, sl = np.zeros(1 << self.m, complex), np.zeros(1 << self.m, complex)
                sm[so] = mem[oo[tau] ^ ao]
                if lam is not None:
                    sl[so] = lam[oo[tau] ^ ao]
                for si in range(ps["stage_end"] - 1, ps["stage_begin"] - 1, -1):
                    st, idx, pb = self.stage(si, tau)
                    if lam is None and si == ps["stage_end"] - 1:
                        sl[idx] = O[self.logical(tau)] * sm[idx]
                    a, l = sm[idx], sl[idx]
                    for op in self.s["ops"][st["op_begin"]:st["op_end"]][::-1]:
                        self.op(op, pb, tabs, (a, l), True, acc)
                    sm[idx], sl[idx] = a, l
                new[oi[tau] ^ ai], newl[oi[tau] ^ ai] = sm[si_], sl[si_]
                assert set(oo[tau] ^ ao) == set(oi[tau] ^ ai)   # in place
            mem, lam = new, newl
        return self.p.terms_of(acc, self.xb, self.w)


def terms_of(self, acc, xb, w):
    """(dx, dw) from the accumulators: terms Im Tr(W P W^dag rho)."""
    terms = np.zeros(len(self.term_src))
    P = {pe.CK_RX: np.array([[0, 1], [1, 0]], complex), pe.CK_RY: np.array([[0, -1j], [1j, 0]]),
         pe.CK_RZ: np.array([[1, 0], [0, -1]], complex)}
    for k, ac in enumerate(self.accs):
        e = self.entries[ac["entry"]]
        cs = self.consts[e["cfirst"]:e["cfirst"] + e["ccount"]]
        if ac["kind"] == 1:
            terms[cs[0]["term"]] = acc[k, 0]
            continue
        rho = (acc[k, 0::2] + 1j * acc[k, 1::2]).reshape(2, 2)
        W = np.eye(2, dtype=complex)
        for c in cs[::-1]:
            if c["term"] >= 0:
                terms[c["term"]] = np.trace(W @ P[int(c["kind"])] @ W.conj().T @ rho).imag
            W = W @ self.constituent(c, xb, w)
    dx = np.array([terms[self.xocc[self.xocc_ptr[p]:self.xocc_ptr[p + 1]]].sum() for p in range(self.num_x)])
    dw = np.array([terms[self.wocc[self.wocc_ptr[p]:self.wocc_ptr[p + 1]]].sum() for p in range(self.num_w)])
    return dx, dw


pe.Plan.terms_of = terms_of


def check(spec, x, w, gE, psi0, dtype):
    plan = compile_spec(spec, dtype)
    pl, fr = pe.Plan(B.vqc_plan_export(plan)), frames(plan)
    B.vqc_free(plan)
    xs = np.zeros((1, 0)) if x is None else x[:1]
    E, st = orc.forward(spec, x, w, psi0=psi0, want_state=True)
    dx_ref, dw_ref = orc.backward(spec, x, w, gE, psi0=psi0)
    for s in fr:
        em = Emulator(pl, s, xs[0], w)
        p0 = None if psi0 is None else psi0[0]
        if s["mode"] == 0 or s["path"] == 0:   # the resident backward recomputes with its own stages
            assert np.allclose(em.forward(p0), st[0], atol=1e-12)
        if s["mode"] == 1:
            dx, dw = em.backward(st[0], gE[0])
            assert np.allclose(dx, dx_ref[0] if spec.num_x else dx, atol=1e-10)
            assert np.allclose(dw, dw_ref, atol=1e-10)
    return fr


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("tile", [0, 6, 7])
@pytest.mark.parametrize("seed,n,G,psi0", [(801, 7, 60, True), (802, 8, 150, False), (803, 9, 220, True),
                                           (804, 10, 260, False)])
def test_random_circuits(monkeypatch, dtype, tile, seed, n, G, psi0):
    # the whole gate set, small forced tiles (many passes, flips and frame changes)
    if tile:
        monkeypatch.setenv("VQC_HBM_TILE_QUBITS", str(tile))
    w_, p0 = wl.small_random(seed, n, G, batch=1, dtype="c128", with_psi0=psi0)
    check(w_.spec, w_.x, w_.w, w_.gE, p0, dtype)


def layered_inputs(spec):
    rng = np.random.default_rng(5)
    return (rng.uniform(-3, 3, (1, spec.num_x)), rng.uniform(-3, 3, spec.num_w), rng.standard_normal((1, spec.n)))


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("kind", ["cx", "cz", "range", "qaoa", "swap", "diagonal", "empty"])
def test_structured_circuits(monkeypatch, dtype, kind):
    monkeypatch.setenv("VQC_HBM_TILE_QUBITS", "6")
    n = 9
    if kind in ("cx", "cz"):
        spec = wl.layered(n, 3, ("RX", "RY", "RZ"), kind.upper())
    elif kind == "range":
        spec = wl.layered(n, 4, ("RZ", "RY"), "CX", reupload=True, ring_range=lambda l: l % (n - 1) + 1)
    else:
        spec = wl.CircuitSpec(n, n, 2 * n)
        if kind != "empty":
            for q in range(n):
                spec.add("RY", (q,), [("x", q)]) if kind != "diagonal" else spec.add("RZ", (q,), [("x", q)])
            for q in range(n):
                spec.add("RZZ", (q, (q + 4) % n), [("w", q)])
                if kind == "swap":
                    spec.add("SWAP", (q, (q + 2) % n))
                spec.add("CRZ", (q, (q + 1) % n), [("w", n + q)])
            if kind == "qaoa":
                for q in range(n):
                    spec.add("RX", (q,), [("w", q)])
    x, w, gE = layered_inputs(spec)
    check(spec, x, w, gE, None, dtype)


def test_entry_cap(monkeypatch):
    # more runs on one tile's qubits than a pass's tables hold: several passes, same result
    monkeypatch.setenv("VQC_HBM_TILE_QUBITS", "6")
    spec = wl.CircuitSpec(8, 8, 160)
    for j in range(160):
        spec.add("RY", (j % 4,), [("w", j)])
        spec.add("CZ", (j % 4, (j + 1) % 4))
    x, w, gE = layered_inputs(spec)
    fr = check(spec, x, w, gE, None, 0)
    assert all(len(s["passes"]) >= 2 for s in fr if s["path"] == 1)


def test_layered_16_passes():
    # the 16-qubit / 8-layer workload: few passes, most stages full
    spec = wl.config(5, batch=1)[0].spec
    for dtype in (0, 1):
        plan = compile_spec(spec, dtype)
        for s in frames(plan):
            if s["path"] == 1:
                assert len(s["passes"]) <= 6
                assert len(s["stages"]) * s["K"] <= 1.3 * len(s["ops"])
        B.vqc_free(plan)


def narrow(kind, n, k):
    """Circuits of many stages on few directions: every run behind the one before it
    ("rx", "ry"), or next to no runs, CZ gates in changing frames ("signs")."""
    rng = np.random.default_rng(n * k)
    spec = wl.CircuitSpec(n, 1, 1).add("RY", (0,), [("x", 0)])
    for _ in range(k):
        if kind == "rx":
            spec.add("RX", (0,), [("w", 0)]).add("CX", (0, 1))
        elif kind == "ry":
            spec.add("RY", (0,), [("x", 0)]).add("CX", (0, 1)).add("RY", (1,), [("w", 0)]).add("CX", (1, 0))
        else:
            spec.add(("CX", "CZ")[rng.integers(2)], tuple(int(q) for q in rng.permutation(n)[:2]))
    return spec


def launch_bytes(s, n, dtype, dfloat, phases):
    """Shared memory of the launches of a schedule's passes, one tile per CTA: the parts
    that plan_hbm places, each as large as the largest pass needs it."""
    most = {k: max(int(p[k + "_end"] - p[k + "_begin"]) for p in s["passes"]) for k in ("stage", "op", "seg")}
    most.update({k: max(int(p[k]) for p in s["passes"]) for k in ("ps_count", "sh_count", "acc_count", "ndg")})
    rs = 8 if dtype else 4
    ew, T = 20 if dfloat else 8 if dtype else 32, 1 << (s["m"] - s["K"])
    wg, dim = max(1, T // 32), 1 << s["m"]
    nk = -(-dim // (16 // (2 * rs)) // T)
    tables = T >= 32 and dtype and (dfloat or phases)
    parts = [dim * 2 * rs * (2 if s["mode"] else 1), most["sh_count"] * ew * rs, most["ps_count"] * ew * rs,
             most["acc_count"] * wg * 8 * rs if s["mode"] else wg * n * rs, 16 * nk, 16 * T,
             (most["ndg"] << s["K"]) * 2 * rs if tables else 0, 4 * T * most["stage"],
             most["stage"] * FSTAGE.itemsize + FFINAL.itemsize + 8 * most["op"] +
             most["stage"] * s["nout"] * FFLIP.itemsize + most["seg"] * FSEG.itemsize, 8 * (most["stage"] + 1)]
    return sum((b + 15) // 16 * 16 for b in parts)


@pytest.mark.parametrize("kind,k", [("rx", 60), ("rx", 100), ("rx", 400), ("ry", 60), ("ry", 100), ("signs", 2000),
                                    ("signs", 20000)])
@pytest.mark.parametrize("n", [13, 16, 20])
def test_passes_fit_shared_memory(monkeypatch, kind, k, n):
    # 227 KB a CTA; with all of its stages the one pass of most of these takes more
    monkeypatch.setenv("VQC_FORCE_PATH", "hbm")
    spec = narrow(kind, n, k)
    for dtype in (0, 1):
        plan = compile_spec(spec, dtype)
        hbm = [s for s in frames(plan) if s["path"] == 1]
        B.vqc_free(plan)
        assert [s["mode"] for s in hbm] == [0, 1]
        for s in hbm:
            for dfloat in (False, True)[:dtype + 1]:
                assert launch_bytes(s, n, dtype, dfloat, False) <= 232448
            assert sum(p["op_end"] - p["op_begin"] for p in s["passes"]) == len(s["ops"])


@pytest.mark.parametrize("kind,k", [("rx", 130), ("ry", 100), ("signs", 4000)])
def test_split_passes(monkeypatch, kind, k):
    # consecutive passes on one tile: the same result
    monkeypatch.setenv("VQC_FORCE_PATH", "hbm")
    spec = narrow(kind, 13, k)
    rng = np.random.default_rng(17)
    x, w, gE = rng.uniform(-3, 3, (1, 1)), rng.uniform(-3, 3, 1), rng.standard_normal((1, 13))
    fr = check(spec, x, w, gE, None, 1)
    assert any(len(s["passes"]) > 1 for s in fr if s["path"] == 1)


def test_phase_tables_come_first():
    # native complex128 launches hold the tables of two-local phases only
    spec = wl.CircuitSpec(14, 14, 0)
    for l in range(3):
        for q in range(14):
            spec.add("RY", (q,), [("x", q)]).add("RZZ", (q, (q + 1) % 14), [("c", 0.4)])
    plan = compile_spec(spec, 1)
    for s in frames(plan):
        for ps in s["passes"]:
            sg = s["segs"][ps["seg_begin"]:ps["seg_end"]]
            ll = sg[(sg["flags"] & LL) != 0]["dg"][:, 0]
            assert sorted(ll) == list(range(len(ll)))
            every = sg["dg"][sg["dg"] != NO_DIAGONAL]
            assert sorted(every) == list(range(ps["ndg"]))
    B.vqc_free(plan)


@pytest.mark.parametrize("n", [13, 15, 18])
def test_complex128_passes_leave_room_for_two_ctas(n):
    # many gradient slots a pass: fewer entries a pass instead of one CTA per SM
    spec = wl.CircuitSpec(n, n, 12 * n)
    for q in range(n):
        spec.add("RY", (q,), [("x", q)])
    for l in range(6):
        for q in range(n):
            spec.add("RZZ", (q, (q + 1) % n), [("w", 2 * n * l + q)])
        for q in range(n):
            spec.add("RX", (q,), [("w", 2 * n * l + n + q)])
    plan = compile_spec(spec, 1)
    hbm = [s for s in frames(plan) if s["path"] == 1]
    B.vqc_free(plan)
    assert hbm and all(launch_bytes(s, n, 1, True, True) <= 115712 for s in hbm)
