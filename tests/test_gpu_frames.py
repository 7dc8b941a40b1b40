"""GPU parity of the frame-schedule kernels (resident sweeps and HBM passes) where
their rules change: full-warp passes at ragged batches, circuits of one pass with the
state written over psi0, the batches around the cluster / passes line, double-float
runs of every form, diagonal groups of complex128 rounds, and circuits around the
shared-memory limit of the table data.

Every value is compared with the fp64 oracle.  With u the unit roundoff (2^-24, 2^-53;
double-float 2^-46, its products being exact to about four units of 2^-48), one gate
moves a state of norm 1 by at most 8u: a pair update is four products and sums per
component (4u sqrt(2)) of entries good to 2u.  So after G gates (one for each
angle of a U3) |psi - psi_ref| <= d =
8uG, an expectation moves by 2d plus its own sum (32u), and a gradient term Im <lam|P|psi>
with |lam| <= sum |gE| by sum |gE| (4d + 32u) -- times the terms that a column sums,
and over the batch for a shared weight.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as orc  # noqa: E402
from paper_2607_11985_gb300 import binding as B  # noqa: E402
from paper_2607_11985_gb300 import workloads as wl  # noqa: E402
from tests.test_frames_cpu import narrow  # noqa: E402
from tests.test_gpu_parity import C, dev, devc, maxerr, run_bwd, run_fwd  # noqa: E402

pytestmark = pytest.mark.gpu

U = {"c64": 2.0 ** -24, "c128": 2.0 ** -53, "c128df": 2.0 ** -46}


@pytest.fixture(scope="module", autouse=True)
def cuda_ready():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)


def draw(spec, batch, dtype, seed, psi0=False, angles=None):
    rng = np.random.default_rng(seed)

    def a(shape):
        v = rng.uniform(-np.pi, np.pi, shape)
        return wl._round(v if angles is None else rng.choice(angles, shape), dtype)

    w_ = wl.Workload("frames", spec, batch, a((batch, spec.num_x)), a(spec.num_w),
                     wl._round(rng.standard_normal((batch, spec.n)), dtype), dtype, seed)
    p0 = None
    if psi0:
        z = rng.standard_normal((batch, 1 << spec.n)) + 1j * rng.standard_normal((batch, 1 << spec.n))
        p0 = (z / np.linalg.norm(z, axis=1, keepdims=True)).astype(
            np.complex64 if dtype == "c64" else np.complex128).astype(np.complex128)
    return w_, p0


def check(c, w_, p0):
    """Forward with and without the state, backward recomputing and from the saved
    state, one-call forward+backward: each against the oracle."""
    spec, dtype, u = w_.spec, w_.dtype, U[w_.dtype]
    d = 8 * u * sum(max(1, len(ps)) for _, _, ps in spec.gates)
    occ = [sum(1 for _, _, ps in spec.gates for kind, v in ps if kind == k and v == i)
           for k, num in (("x", spec.num_x), ("w", spec.num_w)) for i in range(num)]
    row = np.abs(w_.gE).sum(1) * max(occ, default=0) * (4 * d + 32 * u)
    E_ref, st_ref = orc.forward(spec, w_.x, w_.w, psi0=p0, want_state=True)
    dx_ref, dw_ref = orc.backward(spec, w_.x, w_.w, w_.gE, psi0=p0)
    E, st = run_fwd(c, w_, p0)
    assert maxerr(st, st_ref) <= d
    assert maxerr(E, E_ref) <= 2 * d + 32 * u
    assert maxerr(run_fwd(c, w_, p0, want_state=False), E_ref) <= 2 * d + 32 * u
    grads = [run_bwd(c, w_, p0), run_bwd(c, w_, p0, psi_final=devc(st, dtype))]
    x = dev(w_.x, dtype) if spec.num_x else None
    w = dev(w_.w, dtype) if spec.num_w else None
    E2, dx, dw = c.forward_backward(x, w, dev(w_.gE, dtype), psi0=None if p0 is None else devc(p0, dtype))
    torch.cuda.synchronize()
    assert maxerr(E2.cpu().numpy(), E_ref) <= 2 * d + 32 * u
    grads.append((dx_ref if dx is None else dx.cpu().numpy(), dw_ref if dw is None else dw.cpu().numpy()))
    for dx, dw in grads:
        assert np.all(np.abs(dx - dx_ref) <= row[:, None])
        assert maxerr(dw, dw_ref) <= row.sum()


def mixed(n, kinds, layers=1, num_w=True):
    """RY(x) on every qubit, then per layer runs of the given kinds (an angle for each
    rotation) and the two-qubit gates of `kinds` at near and far distances."""
    spec = wl.CircuitSpec(n=n, num_x=n, num_w=0)
    for q in range(n):
        spec.add("RY", (q,), (("x", q),))
    for l in range(layers):
        for q in range(n):
            for k in kinds:
                if k in wl.TWO_QUBIT:
                    continue
                ps = []
                for _ in range(wl.NPARAMS.get(k, 0)):
                    ps.append(("w", spec.num_w) if num_w else ("c", 0.3 + 0.1 * q))
                    spec.num_w += num_w
                spec.add(k, (q,), ps)
        for k in kinds:
            if k not in wl.TWO_QUBIT:
                continue
            for q in range(n):
                for r in (1, n // 2):
                    ps = []
                    if k in wl.NPARAMS:
                        ps = [("w", spec.num_w)] if num_w else [("c", 0.7)]
                        spec.num_w += num_w
                    if (q + r) % n != q:
                        spec.add(k, (q, (q + r) % n), ps)
    return spec


# complex64 takes 12- and 11-qubit tiles, complex128 12 / 11: the sizes below give one
# pass or several, and runs with and without gradient slots
@pytest.mark.parametrize("dtype,n,batch,kinds,num_w", [
    ("c64", 13, 3, ("RX", "RZ", "CX"), True), ("c64", 14, 1, ("H", "T", "RX", "CX"), False),
    ("c64", 15, 5, ("U3", "CX", "RZZ"), True), ("c128", 13, 2, ("RX", "RY", "RZ", "CX"), True),
    ("c128", 14, 1, ("RY", "CZ", "CRZ"), True), ("c128df", 13, 3, ("RY", "RZ", "CX"), True),
    ("c128df", 14, 1, ("RX", "SWAP", "RZZ"), True)])
def test_full_warp_passes(monkeypatch, dtype, n, batch, kinds, num_w):
    monkeypatch.setenv("VQC_FORCE_PATH", "hbm")
    spec = mixed(n, kinds, num_w=num_w)
    c = C(spec, dtype)
    assert c.info(batch)["fwd_path"] == 1 and c.info(batch)["bwd_path"] == 1
    check(c, *draw(spec, batch, dtype, 7000 + n, psi0=batch == 3))


# passes whose stages exceed a CTA's shared memory all at once: several on one tile
@pytest.mark.parametrize("dtype,kind,n,k", [("c64", "signs", 15, 2000), ("c128", "rx", 14, 100), ("c128", "ry", 13, 100),
                                            ("c128", "signs", 15, 2000), ("c128df", "rx", 13, 400),
                                            ("c128df", "ry", 14, 60)])
def test_passes_of_many_stages(monkeypatch, dtype, kind, n, k):
    monkeypatch.setenv("VQC_FORCE_PATH", "hbm")
    spec = narrow(kind, n, k)
    c = C(spec, dtype)
    assert c.info(2)["fwd_path"] == 1 and c.info(2)["bwd_path"] == 1
    check(c, *draw(spec, 2, dtype, 7050 + n))


# CZ only acts as a sign: a register circuit of one direction needs one pass
@pytest.mark.parametrize("dtype,n,path", [("c64", 14, "hbm"), ("c128", 13, "hbm"), ("c128df", 13, "hbm"),
                                          ("c64", 8, None), ("c128", 3, None)])
@pytest.mark.parametrize("wide", [False, True])
def test_state_written_over_psi0(monkeypatch, dtype, n, path, wide):
    if path:
        monkeypatch.setenv("VQC_FORCE_PATH", path)
    spec = wl.CircuitSpec(n=n, num_x=1, num_w=0)
    for q in range(n if wide else min(n, 2)):
        spec.add("RX", (q,), (("x", 0),)).add("CX", (q, (q + 1) % n))
    c = C(spec, dtype)
    if path:
        assert (c.info(3)["fwd_passes"] > 1) == wide
    w_, p0 = draw(spec, 3, dtype, 7100 + n, psi0=True)
    E_ref, st_ref = orc.forward(spec, w_.x, w_.w, psi0=p0, want_state=True)
    st = devc(p0, dtype)
    E, st2 = c.forward(dev(w_.x, dtype), None, psi0=st, want_state=True, state_out=st)
    torch.cuda.synchronize()
    assert st2.data_ptr() == st.data_ptr()
    d = 8 * U[dtype] * len(spec.gates)
    assert maxerr(st.cpu().numpy(), st_ref) <= d and maxerr(E.cpu().numpy(), E_ref) <= 2 * d + 32 * U[dtype]


@pytest.mark.parametrize("dtype,n,mode", [("c64", 15, 0), ("c64", 14, 1), ("c128", 14, 0), ("c128", 13, 1)])
def test_cluster_up_to_half_the_sms(dtype, n, mode):
    half = torch.cuda.get_device_properties(0).multi_processor_count // 2
    spec = mixed(n, ("RX", "CX"))
    c = C(spec, dtype)
    rows = [0, half - 1]
    u = U[dtype]
    d = 8 * u * len(spec.gates)
    for batch, path in ((half, 2), (half + 1, 1)):
        assert c.info(batch)["fwd_path" if mode == 0 else "bwd_path"] == path
        w_, _ = draw(spec, batch, dtype, 7200 + n)
        if mode == 0:
            E_ref = orc.forward(spec, w_.x[rows], w_.w)
            assert maxerr(run_fwd(c, w_, want_state=False)[rows], E_ref) <= 2 * d + 32 * u
            continue
        dx_ref, _ = orc.backward(spec, w_.x[rows], w_.w, w_.gE[rows])
        dx, dw = run_bwd(c, w_)
        row = np.abs(w_.gE).sum(1) * (4 * d + 32 * u)
        assert np.all(np.abs(dx[rows] - dx_ref) <= row[rows][:, None])
        _, dw_ref = orc.backward_parallel(spec, w_.x, w_.w, w_.gE)
        assert maxerr(dw, dw_ref) <= row.sum()


def test_noalloc_takes_clusters_beyond_its_scratch():
    # 14 qubits, one sample more than the line: the passes' states exceed the built-in
    # scratch, the cluster's partials do not
    half = torch.cuda.get_device_properties(0).multi_processor_count // 2
    spec = mixed(14, ("RX", "CX"))
    c = C(spec, "c64")
    w_, _ = draw(spec, half + 1, "c64", 7300)
    assert c.info(w_.batch)["bwd_path"] == 1
    x, w, gE = dev(w_.x, "c64"), dev(w_.w, "c64"), dev(w_.gE, "c64")
    dx, dw = torch.empty_like(x), torch.empty_like(w)
    B.vqc_backward_noalloc(c.plan, w_.batch, x.data_ptr(), w.data_ptr(), None, None, gE.data_ptr(),
                           dx.data_ptr(), dw.data_ptr(), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    dx2, dw2 = run_bwd(c, w_)
    u = U["c64"]
    row = 2 * np.abs(w_.gE).sum(1) * (32 * u * len(spec.gates) + 32 * u)   # each within one bound
    assert np.all(np.abs(dx.cpu().numpy() - dx2) <= row[:, None])
    assert maxerr(dw.cpu().numpy(), dw2) <= row.sum()


@pytest.mark.parametrize("dtype,n", [("c64", 15), ("c128", 14), ("c128df", 14)])
@pytest.mark.parametrize("saved", [True, False])
def test_noalloc_takes_one_pass_at_a_time(monkeypatch, dtype, n, saved):
    # the rho sums and table entries of the whole circuit exceed the built-in scratch,
    # those of a pass do not: the same sums in the same order, bit by bit
    monkeypatch.setenv("VQC_FORCE_PATH", "hbm")
    spec = mixed(n, ("RX", "RY", "H", "CX"), layers=160 if dtype == "c64" else 115)
    spec.add("RZZ", (0, n - 1), (("x", 1),))
    c = C(spec, dtype)
    w_, _ = draw(spec, 1, dtype, 7350)
    assert B.vqc_workspace_bytes(c.plan, 1, 1) > 1 << 20
    x, w, gE = dev(w_.x, dtype), dev(w_.w, dtype), dev(w_.gE, dtype)
    st = c.forward(x, w, want_state=True)[1] if saved else None
    dx_ref, dw_ref = c.backward(x, w, gE, psi_final=st)
    dx, dw = torch.empty_like(x), torch.empty_like(w)
    B.vqc_backward_noalloc(c.plan, 1, x.data_ptr(), w.data_ptr(), None, st.data_ptr() if saved else None,
                           gE.data_ptr(), dx.data_ptr(), dw.data_ptr(), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert torch.equal(dx, dx_ref) and torch.equal(dw, dw_ref)


def test_noalloc_takes_fewer_ctas():
    # dw partials of a full grid a little beyond the built-in scratch
    num_w = 200
    for _ in range(16):   # (200 x 1.25^15 = 5684 weights: 1 MiB of partials of 46 CTAs)
        spec = wl.CircuitSpec(6, 6, num_w)
        for q in range(6):
            spec.add("RY", (q,), [("x", q)])
        for j in range(num_w):
            spec.add("RX", (j % 6,), [("w", j)])
        c = C(spec, "c64")
        need = B.vqc_workspace_bytes(c.plan, 4096, 1)
        if need > 1 << 20:
            break
        num_w = num_w * 5 // 4
    assert 1 << 20 < need < 2 << 20
    w_, _ = draw(spec, 4096, "c64", 7370)
    x, w, gE = dev(w_.x, "c64"), dev(w_.w, "c64"), dev(w_.gE, "c64")
    dx_ref, dw_ref = c.backward(x, w, gE)
    dx, dw = torch.empty_like(x), torch.empty_like(w)
    B.vqc_backward_noalloc(c.plan, 4096, x.data_ptr(), w.data_ptr(), None, None, gE.data_ptr(), dx.data_ptr(),
                           dw.data_ptr(), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert torch.equal(dx, dx_ref)
    # the same terms in another order: each of at most 4096 additions rounds by u
    bound = 2 * 4096 * U["c64"] * np.abs(w_.gE).sum()
    assert maxerr(dw.cpu().numpy(), dw_ref.cpu().numpy()) <= bound


# runs of every factored form (rotation alone, a diagonal on either side or both, a
# diagonal run), at angles where an entry of the matrix vanishes; groups below a warp
# and small forwards of few stages keep the 2x2 updates
@pytest.mark.parametrize("n,path,layers", [(3, None, 2), (8, None, 2), (8, None, 6), (11, None, 2), (13, "hbm", 1)])
@pytest.mark.parametrize("kinds", [("RY",), ("RY", "RZ"), ("RZ", "RY"), ("RX",), ("H",), ("RZ",), ("U3", "X")])
@pytest.mark.parametrize("dtype", ["c128df", "c128"])
def test_run_forms(monkeypatch, dtype, kinds, n, path, layers):
    if path:
        monkeypatch.setenv("VQC_FORCE_PATH", path)
    spec = mixed(n, kinds + ("CX",), layers=layers)
    c = C(spec, dtype)
    for angles in ((0.0, np.pi, -np.pi, np.pi / 2), None):
        check(c, *draw(spec, 2, dtype, 7400 + n, angles=angles))


# phases and signs with both qubits in the block, one or none, alone and between runs
@pytest.mark.parametrize("n", [2, 5, 9, 11])
@pytest.mark.parametrize("kinds", [("CZ",), ("CRZ",), ("RZZ",), ("RX", "CZ", "RZZ"), ("CRZ", "CX", "RZZ")])
@pytest.mark.parametrize("dtype", ["c128", "c128df", "c64"])
def test_diagonal_groups(dtype, kinds, n):
    spec = mixed(n, kinds, layers=2)
    check(C(spec, dtype), *draw(spec, 3, dtype, 7500 + n, psi0=True))


# few and many table entries: the table data of the larger ones stays in global memory
@pytest.mark.parametrize("dtype,n", [("c64", 9), ("c64", 12), ("c128", 10)])
@pytest.mark.parametrize("layers", [1, 6, 24])
def test_table_data_in_and_out_of_shared_memory(dtype, n, layers):
    spec = mixed(n, ("RX", "RY", "CX"), layers=layers)
    check(C(spec, dtype), *draw(spec, 4, dtype, 7600 + n))


# double-float sweeps on either side of what fits one CTA: with the runs' factors, with
# their matrices only, neither (passes); the built-in scratch takes the first two
@pytest.mark.parametrize("n,layers,path", [(12, 6, 0), (12, 7, 0), (12, 8, 1), (11, 18, 0), (11, 23, 0), (11, 24, 1),
                                           (9, 60, 0)])
def test_double_float_around_the_resident_limit(n, layers, path):
    spec = wl.layered(n, layers, ("RX", "RY", "RZ"), "CX")
    c = C(spec, "c128df")
    assert c.info(9)["bwd_path"] == path
    w_, p0 = draw(spec, 9, "c128df", 7700 + n)
    check(c, w_, p0)
    if path == 0:
        x, w, gE = (dev(a, "c128df") for a in (w_.x, w_.w, w_.gE))
        dx_ref, dw_ref = c.backward(x, w, gE)
        dx, dw = torch.empty_like(x), torch.empty_like(w)
        B.vqc_backward_noalloc(c.plan, 9, x.data_ptr(), w.data_ptr(), None, None, gE.data_ptr(), dx.data_ptr(),
                               dw.data_ptr(), torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        assert torch.equal(dx, dx_ref) and torch.equal(dw, dw_ref)


# native complex128 rings of RZZ whose phase tables do not fit beside the state: the op
# switch instead, on either side of both lines
# (complex64, 12 qubits x 17 layers: the layout to its last 100 bytes)
@pytest.mark.parametrize("dtype,n,layers,path", [
    ("c128", 11, 11, 0), ("c128", 11, 12, 0), ("c128", 11, 13, 1), ("c128", 10, 24, 0), ("c128", 10, 28, 0),
    ("c128", 10, 29, 1), ("c128", 8, 80, 0), ("c64", 12, 17, 0), ("c64", 12, 18, 1)])
def test_phase_tables_around_the_resident_limit(dtype, n, layers, path):
    spec = wl.CircuitSpec(n, n, 2 * n * layers)
    for q in range(n):
        spec.add("RY", (q,), [("x", q)])
    for l in range(layers):
        for q in range(n):
            spec.add("RZZ", (q, (q + 1) % n), [("w", 2 * n * l + q)])
        for q in range(n):
            spec.add("RX", (q,), [("w", 2 * n * l + n + q)])
    c = C(spec, dtype)
    batch = 5 if dtype == "c128" else 100   # (enough for blocks of 16 amplitudes)
    assert c.info(batch)["bwd_path"] == path
    check(c, *draw(spec, batch, dtype, 7800 + n))


# the same on the cluster path: 14 qubits forward, 13 backward
@pytest.mark.parametrize("n,mode,kind,k", [(14, 0, "ry", 400), (13, 1, "layers", 11)])
def test_double_float_around_the_cluster_limit(n, mode, kind, k):
    spec = narrow(kind, n, k) if kind == "ry" else wl.layered(n, k, ("RX", "RY", "RZ"), "CX")
    c = C(spec, "c128df")
    assert c.info(2)["bwd_path" if mode else "fwd_path"] == 2
    check(c, *draw(spec, 2, "c128df", 7900 + n))


# double-float circuits with phases: forward and backward as one launch or as two calls
# (more than one wave of CTAs), which are those of forward and backward
@pytest.mark.parametrize("n,batch", [(9, 3), (9, 1301), (10, 640), (11, 100)])
def test_double_float_phase_steps(n, batch):
    spec = mixed(n, ("RX", "CRZ", "RZZ"))
    c = C(spec, "c128df")
    w_, _ = draw(spec, batch, "c128df", 8000 + n)
    x, w, gE = (dev(a, "c128df") for a in (w_.x, w_.w, w_.gE))
    E, st = c.forward(x, w, want_state=True)
    dx, dw = c.backward(x, w, gE, psi_final=st)
    E2, dx2, dw2 = c.forward_backward(x, w, gE)
    d = 8 * U["c128df"] * len(spec.gates)
    row = np.abs(w_.gE).sum(1) * (4 * d + 32 * U["c128df"])
    assert maxerr(E2.cpu().numpy(), E.cpu().numpy()) <= 4 * d + 64 * U["c128df"]   # each within one bound
    assert np.all(np.abs(dx2.cpu().numpy() - dx.cpu().numpy()) <= 2 * row[:, None])
    assert maxerr(dw2.cpu().numpy(), dw.cpu().numpy()) <= 2 * row.sum()
    if batch > 100:
        assert torch.equal(E, E2) and torch.equal(dx, dx2) and torch.equal(dw, dw2)


# double-float batches of more CTAs than SMs at 8 and 9 qubits: factored or not by the
# layers and by what depends on the sample
@pytest.mark.parametrize("n,layers,reupload", [(8, 2, False), (8, 4, False), (8, 8, False), (9, 2, True), (9, 4, True),
                                               (9, 8, True)])
def test_double_float_large_batches(n, layers, reupload):
    spec = wl.layered(n, layers, ("RX", "RY", "RZ"), "CX", reupload=reupload)
    check(C(spec, "c128df"), *draw(spec, 1303, "c128df", 8100 + n + layers))


# the two complex128 types take workspaces of one size, whichever of them sized it
@pytest.mark.parametrize("n", [4, 8, 9, 10, 11, 12, 13, 14, 15, 16])
@pytest.mark.parametrize("kinds,layers", [(("RX", "RY", "RZ", "CX"), 1), (("RX", "RY", "RZ", "CX"), 8), (("RX", "RZZ"), 2)])
def test_complex128_workspaces(n, kinds, layers):
    spec = mixed(n, kinds, layers=layers)
    native, df = C(spec, "c128"), C(spec, "c128df")
    for batch in (1, 7, 60, 77, 100, 333, 1600):
        for mode in range(4):
            assert B.vqc_workspace_bytes(native.plan, batch, mode) == B.vqc_workspace_bytes(df.plan, batch, mode)


def test_complex128_workspace_of_the_other_type():
    spec = mixed(13, ("RX", "RY", "CX"))
    native = C(spec, "c128")
    for batch in (3, 90):
        w_, _ = draw(spec, batch, "c128df", 8200)
        x, w, gE = (dev(a, "c128df") for a in (w_.x, w_.w, w_.gE))
        c = C(spec, "c128df")
        want = c.forward_backward(x, w, gE)
        E, dx, dw = (torch.empty_like(t) for t in want)
        nbytes = B.vqc_workspace_bytes(native.plan, batch, 3)
        ws = torch.zeros(nbytes, dtype=torch.uint8, device="cuda")
        B.vqc_forward_backward(c.plan, batch, x.data_ptr(), w.data_ptr(), None, gE.data_ptr(), E.data_ptr(), dx.data_ptr(),
                               dw.data_ptr(), ws.data_ptr(), nbytes, torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(want, (E, dx, dw)))


def test_clusters_where_pass_states_exceed_their_cap():
    # 14 qubits, backward: two states of 128 KiB a sample reach 16 GiB at 65536 samples
    spec = mixed(14, ("RX", "CX"))
    c = C(spec, "c64")
    assert c.info(65536)["bwd_path"] == 1 and c.info(65537)["bwd_path"] == 2
    assert B.vqc_workspace_bytes(c.plan, 65537, 1) < 1 << 20
    w_, _ = draw(spec, 65537, "c64", 8300)
    rows = [0, 40000, 65536]
    dx_ref, _ = orc.backward(spec, w_.x[rows], w_.w, w_.gE[rows])
    dx, _ = run_bwd(c, w_)
    d = 8 * U["c64"] * len(spec.gates)
    row = np.abs(w_.gE[rows]).sum(1) * (4 * d + 32 * U["c64"])
    assert np.all(np.abs(dx[rows] - dx_ref) <= row[:, None])


# environment switches set after the circuit was compiled: paths and block sizes that its
# plan was compiled without
@pytest.mark.parametrize("dtype,n", [("c64", 8), ("c128", 9), ("c128df", 9)])
def test_switches_after_compiling(monkeypatch, dtype, n):
    spec = mixed(n, ("RX", "RY", "CX", "RZZ"))
    c = C(spec, dtype)
    data = draw(spec, 3, dtype, 8400 + n, psi0=True)
    assert c.info(3)["fwd_path"] == 0 and c.info(3)["bwd_path"] == 0
    monkeypatch.setenv("VQC_FORCE_PATH", "hbm")
    assert c.info(3)["fwd_path"] == 1 and c.info(3)["bwd_path"] == 1
    check(c, *data)
    monkeypatch.delenv("VQC_FORCE_PATH")
    monkeypatch.setenv("VQC_FORCE_K_FWD", "2")
    monkeypatch.setenv("VQC_FORCE_K_BWD", "1")
    assert c.info(3)["fwd_k"] == 2 and c.info(3)["bwd_k"] == 1
    check(c, *data)
    monkeypatch.delenv("VQC_FORCE_K_FWD")
    monkeypatch.delenv("VQC_FORCE_K_BWD")
    assert c.info(3)["fwd_path"] == 0
    check(c, *data)


def test_switch_in_capture(monkeypatch):
    spec = mixed(8, ("RX", "CX"))
    c = C(spec, "c64")
    w_, _ = draw(spec, 5, "c64", 8500)
    x, w = dev(w_.x, "c64"), dev(w_.w, "c64")
    want = c.forward(x, w)
    monkeypatch.setenv("VQC_FORCE_PATH", "hbm")
    E = torch.empty_like(want)
    nbytes = B.vqc_workspace_bytes(c.plan, 5, 0)
    ws = torch.zeros(nbytes, dtype=torch.uint8, device="cuda")
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):   # (the first call that needs the passes' schedules)
        B.vqc_forward(c.plan, 5, x.data_ptr(), w.data_ptr(), None, E.data_ptr(), None, ws.data_ptr(), nbytes,
                      torch.cuda.current_stream().cuda_stream)
    g.replay()
    torch.cuda.synchronize()
    assert maxerr(E.cpu().numpy(), want.cpu().numpy()) <= 4 * 8 * U["c64"] * len(spec.gates) + 64 * U["c64"]
