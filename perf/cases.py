"""The work that a user of this package has it do, as measured cases.

A case is one call pattern of ``Circuit`` on one circuit, batch and state type:

  step      E, dx, dw = c.forward_backward(x, w, gE)       a training step whose loss gradient is known
  saved     E, psi = c.forward(..., want_state=True);      a training step that keeps the final states
            dx, dw = c.backward(..., psi_final=psi)
  autograd  E = c(x, w); torch.autograd.grad(E, (x, w), gE)
  expz      E = c.forward(x, w)                            inference
  state     E, psi = c.forward(x, w, want_state=True)
  probs     P = c.probabilities(x, w)
  host      c.prepare_host(x, w, gE)()                     numpy arrays in, numpy arrays out

The circuits are the families of the package's own workloads and tests: layered
ansaetze (rotations per qubit and a ring of CX or CZ), re-uploading ansaetze
with range rings, QAOA-like rings of RZZ and RX, and random circuits over the
whole gate set.  4 to 20 qubits, complex64, complex128 and double-float.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

_REAL = {"c64": torch.float32, "c128": torch.float64, "c128df": torch.float64}
_STATE_BYTES = {"c64": 8, "c128": 16, "c128df": 16}
_STEPS = ("step", "saved", "autograd", "host")   # calls that return gradients


def _case(name, call, dtype, kind, n, layers, batch, rot="RX RY RZ", ent="CX", gates=0, circuit=0):
    return {"name": name, "call": call, "dtype": dtype, "kind": kind, "n": n, "layers": layers,
            "batch": batch, "rot": rot, "ent": ent, "gates": gates, "circuit": circuit}


def listed():
    return [
        # the smallest training step of the package's workloads: latency and launches only
        _case("step_n4_b64", "step", "c64", "layered", 4, 2, 64, rot="RY RZ"),
        # a quantum layer inside a torch model: forward and backward through autograd
        _case("autograd_n8_b1024", "autograd", "c64", "layered", 8, 4, 1024, ent="CZ"),
        # a host program with numpy arrays, an odd batch
        _case("host_n10_b251", "host", "c64", "layered", 10, 3, 251),
        # the re-uploading classifier with range rings: the largest state of the resident backward but one
        _case("saved_n12_b4096", "saved", "c64", "reupload", 12, 6, 4096, rot="RZ RY RZ"),
        # a static circuit over the whole gate set, every angle per sample, states wanted
        _case("state_random_n13_b256", "state", "c64", "random", 13, 0, 256, gates=520, circuit=7),
        # a mid-size ansatz, an odd batch: resident forward, two thread blocks per state backward
        _case("step_n14_b131", "step", "c64", "layered", 14, 6, 131),
        # QAOA-like rings of RZZ and RX with a per-sample encoding
        _case("step_qaoa_n15_b96", "step", "c64", "qaoa", 15, 5, 96),
        # the package's headline workload: 16 qubits, 8 layers, batch 512, states kept
        _case("saved_n16_b512", "saved", "c64", "layered", 16, 8, 512),
        # the same ansatz at complex128 accuracy in double-float, an odd batch
        _case("step_n16_df_b77", "step", "c128df", "layered", 16, 8, 77),
        # inference on a larger state
        _case("expz_n18_b48", "expz", "c64", "layered", 18, 5, 48),
        # a training step on the largest state of the package's regime map, a small odd batch
        _case("step_n20_b9", "step", "c64", "layered", 20, 4, 9),
        # native complex128 on a resident state
        _case("step_n11_c128_b100", "step", "c128", "layered", 11, 4, 100),
    ]


def _cost(case):
    """About proportional to the time of a pass (complex64 amplitude updates)."""
    runs = (case["layers"] + 1) * case["n"] if case["kind"] != "random" else 0.6 * case["gates"]
    per = {"c64": 1.0, "c128df": 7.0, "c128": 24.0}[case["dtype"]] * (4.0 if case["call"] in _STEPS else 1.0)
    return case["batch"] * 2.0 ** case["n"] * runs * per


def draw(rng):
    most = 0.6 * _cost(listed()[7])
    while True:
        kind = rng.choice(["layered", "layered", "layered", "reupload", "qaoa", "random"])
        n = rng.randint(4, 20)
        dtype = rng.choice(["c64", "c64", "c64", "c128df", "c128df", "c128"])
        call = rng.choice(["step", "step", "saved", "autograd", "expz", "state", "probs", "host"])
        batch = int(round(2.0 ** rng.uniform(0, 12)))
        case = _case("", call, dtype, kind, n, rng.randint(1, 8), batch,
                     rot=rng.choice(["RX RY RZ", "RY", "RY RZ", "RZ RY RZ"]), ent=rng.choice(["CX", "CX", "CZ"]),
                     gates=rng.randint(100, 700) if kind == "random" else 0,
                     circuit=rng.randrange(1 << 30) if kind == "random" else 0)
        del case["name"]
        if _cost(case) <= most and batch * 2.0 ** n <= 2.0 ** 25:
            return case


# ------------------------------------------------------------------ circuits and inputs

def _gates(case):
    """(x columns, weights, gates): gates in time order, (name, qubits, params),
    a parameter ("x", column), ("w", index) or ("c", constant)."""
    n, kind = case["n"], case["kind"]
    out = []
    if kind == "random":
        rnd = random.Random(case["circuit"])
        nx = 0
        for _ in range(case["gates"]):
            two, par = rnd.random() < 0.3, rnd.random() < 0.4
            name = rnd.choice((["CRZ", "RZZ"] if par else ["CX", "CZ", "SWAP"]) if two else
                              (["RX", "RY", "RZ", "U3"] if par else ["H", "X", "Y", "Z", "S", "T", "SX"]))
            q = rnd.sample(range(n), 2 if two else 1)
            count = {"U3": 3, "RX": 1, "RY": 1, "RZ": 1, "CRZ": 1, "RZZ": 1}.get(name, 0)
            out.append((name, tuple(q), tuple(("x", nx + k) for k in range(count))))
            nx += count
        return nx, 0, out
    nw = 0
    if kind == "qaoa":
        out += [("H", (q,), ()) for q in range(n)]
    if kind != "reupload":
        out += [("RY", (q,), (("x", q),)) for q in range(n)]
    for layer in range(case["layers"]):
        if kind == "qaoa":
            for i in range(n):
                out.append(("RZZ", (i, (i + 1) % n), (("w", nw),)))
                nw += 1
            for q in range(n):
                out.append(("RX", (q,), (("w", nw),)))
                nw += 1
            continue
        if kind == "reupload":
            out += [("RY", (q,), (("x", q),)) for q in range(n)]
        for q in range(n):
            for r in case["rot"].split():
                out.append((r, (q,), (("w", nw),)))
                nw += 1
        step = layer % (n - 1) + 1 if kind == "reupload" else 1
        out += [(case["ent"], (i, (i + step) % n), ()) for i in range(n)]
    return n, nw, out


def _inputs(case, seed, nx, nw):
    rng = np.random.default_rng(seed)
    b, n = case["batch"], case["n"]
    x = rng.standard_normal((b, nx)) if case["kind"] == "reupload" else rng.uniform(-np.pi, np.pi, (b, nx))
    w = rng.uniform(-np.pi, np.pi, nw)
    g = rng.standard_normal((b, n))
    np_t = np.float32 if case["dtype"] == "c64" else np.float64
    return x.astype(np_t), w.astype(np_t), g.astype(np_t)


def prepare(case, seed):
    from paper_2607_11985_gb300 import workloads as wl
    from paper_2607_11985_gb300.circuit import Circuit
    nx, nw, gates = _gates(case)
    c = Circuit(wl.CircuitSpec(case["n"], nx, nw, gates), case["dtype"])
    x, w, g = _inputs(case, seed, nx, nw)
    if case["call"] == "host":
        return {"call": "host", "step": c.prepare_host(x, w, g)}
    x, w, g = (torch.from_numpy(a).cuda() for a in (x, w, g))
    if case["call"] == "autograd":
        x.requires_grad_()
        w.requires_grad_(nw > 0)
    return {"call": case["call"], "c": c, "x": x, "w": w, "g": g}


def run(state):
    if state["call"] == "host":
        return state["step"]()
    c, x, w, g = state["c"], state["x"], state["w"], state["g"]
    call = state["call"]
    if call == "step":
        return c.forward_backward(x, w, g)
    if call == "saved":
        e, psi = c.forward(x, w, want_state=True)
        return (e, psi) + tuple(c.backward(x, w, g, psi_final=psi))
    if call == "autograd":
        e = c(x, w)
        return (e.detach(),) + torch.autograd.grad(e, (x, w) if w.requires_grad else (x,), g)
    if call == "expz":
        return c.forward(x, w)
    if call == "state":
        return c.forward(x, w, want_state=True)
    return c.probabilities(x, w)


# ------------------------------------------------------------------ what a pass cannot do without

def work(case):
    """Each input read once, each output written once; per amplitude 14 flops for a
    fused single-qubit run, 6 for RZZ, 3 for CRZ and 3 + n for <Z>, and for the
    gradients both states taken back (2 x) and 4 per angle."""
    nx, nw, gates = _gates(case)
    n, b = case["n"], case["batch"]
    real, amp = _STATE_BYTES[case["dtype"]] // 2, _STATE_BYTES[case["dtype"]]
    per, angles, open_run = 0.0, 0, set()
    for name, q, params in gates:
        angles += len(params)
        if len(q) == 1:
            per += 0.0 if q[0] in open_run else 14.0
            open_run.add(q[0])
        else:
            per += {"RZZ": 6.0, "CRZ": 3.0}.get(name, 0.0)
            open_run -= set(q)
    grads = case["call"] in _STEPS
    numbers = b * nx + nw + b * n
    if grads:
        numbers += b * n + b * nx + nw
    if case["call"] == "probs":
        numbers += b * 2 ** n - b * n
    nbytes = numbers * real + (b * 2 ** n * amp if case["call"] in ("saved", "state") else 0)
    flops = per + 3 + n
    if grads:
        flops += 2 * per + 4 * angles + n + 2
    return {"bytes": float(nbytes), "flops": float(flops * b * 2 ** n)}


def tolerance(case):
    """About four times the largest error against exact() seen over the listed and
    drawn cases: 3.3e-6 (complex64, <Z> at 18 qubits, where <Z> is small against
    the norm it sums over), 1.1e-13 (double-float), 6e-15 (complex128)."""
    if case["dtype"] == "c64":
        return {"rel": 1.5e-5, "max": 1.5e-4}
    if case["dtype"] == "c128df":
        return {"rel": 5e-13, "max": 5e-12}
    return {"rel": 4e-14, "max": 4e-13}


# ------------------------------------------------------------------ the same in 64 bits, plain torch

_FIXED = {"H": [[math.sqrt(0.5), math.sqrt(0.5)], [math.sqrt(0.5), -math.sqrt(0.5)]], "X": [[0, 1], [1, 0]],
          "Y": [[0, -1j], [1j, 0]], "Z": [[1, 0], [0, -1]], "S": [[1, 0], [0, 1j]],
          "T": [[1, 0], [0, complex(math.sqrt(0.5), math.sqrt(0.5))]],
          "SX": [[0.5 + 0.5j, 0.5 - 0.5j], [0.5 - 0.5j, 0.5 + 0.5j]]}


def _matrix(name, t):
    """[[a, b], [c, d]] of one gate, each a complex tensor [B or 1, 1, 1]."""
    if name in _FIXED:
        return [[torch.tensor(v, dtype=torch.complex128, device="cuda").reshape(1, 1, 1) for v in row]
                for row in _FIXED[name]]
    t = t.reshape(-1, 1, 1)
    c, s = torch.cos(t / 2) + 0j, torch.sin(t / 2) + 0j
    if name == "RX":
        return [[c, -1j * s], [-1j * s, c]]
    if name == "RY":
        return [[c, -s], [s, c]]
    return [[c - 1j * s, 0 * c], [0 * c, c + 1j * s]]   # RZ


def _halves(psi, q):
    v = psi.view(psi.shape[0], -1, 2, 1 << q)
    return v[:, :, 0], v[:, :, 1]


def _one(psi, q, m):
    u, v = _halves(psi, q)
    m = [[e.reshape(-1, 1, 1) for e in row] for row in m]
    nu, nv = m[0][0] * u + m[0][1] * v, m[1][0] * u + m[1][1] * v
    u.copy_(nu)
    v.copy_(nv)


def _diag(name, q, k):
    """Diagonal of the generator of a two-qubit phase gate over the amplitude index."""
    a, b = ((k >> q[0]) & 1).double(), ((k >> q[1]) & 1).double()
    return a * (1 - 2 * b) if name == "CRZ" else (1 - 2 * a) * (1 - 2 * b)


def exact(case, seed):
    nx, nw, gates = _gates(case)
    x, w, g = (torch.from_numpy(a.astype(np.float64)).cuda() for a in _inputs(case, seed, nx, nw))
    n, b = case["n"], case["batch"]
    k = torch.arange(1 << n, device="cuda")
    flat = []   # U3 as RZ(lambda), RY(theta), RZ(phi) and a scalar phase
    for name, q, params in gates:
        if name == "U3":
            flat += [("RZ", q, params[2]), ("RY", q, params[0]), ("RZ", q, params[1]), ("phase", params[1:], None)]
        else:
            flat.append((name, q, params[0] if params else None))

    def angle(p):
        return x[:, p[1]] if p[0] == "x" else w[p[1]].reshape(1)

    def two(psi, name, q, t):
        if name == "CX":
            return psi[:, k ^ (((k >> q[0]) & 1) << q[1])]
        if name == "SWAP":
            d = ((k >> q[0]) ^ (k >> q[1])) & 1
            return psi[:, k ^ (d << q[0]) ^ (d << q[1])]
        if name == "CZ":
            return psi.mul_((1 - 2 * ((k >> q[0]) & (k >> q[1]) & 1)).double())
        half = -0.5 * t.reshape(-1, 1) * _diag(name, q, k)
        return psi.mul_(torch.polar(torch.ones_like(half), half))

    psi = torch.zeros(b, 1 << n, dtype=torch.complex128, device="cuda")
    psi[:, 0] = 1
    for name, q, p in flat:
        if name == "phase":
            psi.mul_(torch.exp(0.5j * (angle(q[0]) + angle(q[1]))).reshape(-1, 1))
        elif len(q) == 1:
            _one(psi, q[0], _matrix(name, angle(p) if p else None))
        else:
            psi = two(psi, name, q, angle(p) if p else None)
    prob = psi.abs().square()
    signs = torch.stack([(1 - 2 * ((k >> j) & 1)).double() for j in range(n)], 1)
    e = prob @ signs
    call = case["call"]
    if call == "probs":
        return prob
    if call == "expz":
        return e
    if call == "state":
        return e, psi
    final = psi.clone() if call == "saved" else None
    lam = psi * (g @ signs.T)
    del prob
    dx, dw = torch.zeros(b, nx, dtype=torch.float64, device="cuda"), torch.zeros(nw, dtype=torch.float64, device="cuda")
    for name, q, p in reversed(flat):
        if name == "phase":   # common to both states
            continue
        t = angle(p) if p else None
        if p:
            if len(q) == 1:
                (u, v), (lu, lv) = _halves(psi, q[0]), _halves(lam, q[0])
                if name == "RX":
                    term = (lu.conj() * v + lv.conj() * u).imag
                elif name == "RY":
                    term = (lv.conj() * u - lu.conj() * v).real
                else:
                    term = (lu.conj() * u - lv.conj() * v).imag
                term = term.sum((1, 2))
            else:
                term = ((lam.conj() * psi).imag * _diag(name, q, k)).sum(1)
            if p[0] == "x":
                dx[:, p[1]] += term
            else:
                dw[p[1]] += term.sum()
        if len(q) == 1:
            m = _matrix(name, t)
            m = [[m[0][0].conj(), m[1][0].conj()], [m[0][1].conj(), m[1][1].conj()]]
            _one(psi, q[0], m)
            _one(lam, q[0], m)
        else:   # CX, CZ and SWAP are their own inverses
            t = -t if t is not None else None
            psi, lam = two(psi, name, q, t), two(lam, name, q, t)
    dws = dw if nw else None
    if call == "saved":
        return e, final, dx, dws
    if call == "autograd":
        return (e, dx, dw) if nw else (e, dx)
    out = (e, dx, dws)
    return tuple(v.cpu().numpy() if v is not None else None for v in out) if call == "host" else out
