"""The dense operators' kernels on systems that keep them: a two-qubit control or a transverse drift
puts the table outside the locally controlled class, so every call here runs the gathered N x N
operators (checked for each table, and by the profiled launches where a kernel has a phase of its own).
Tolerances are those that these kernels are held to elsewhere: FP64 chains 1e-12, its gradients 1e-10;
FP32 and split FP16 2e-4 of an entry (gradients 2e-4 and 1e-3 of the largest), 1e-6 of F."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import redo_oracle as O  # noqa: E402
from paper_1707_02162_gb300 import inputs  # noqa: E402
from tests import _ref  # noqa: E402

pytestmark = pytest.mark.gpu
X = inputs.PAULI["X"]
TOL = {"fp64": 1e-12, "fp32": 2e-4, "fp16x3": 2e-4}
GTOL = {"fp64": 1e-10, "fp32": 2e-4, "fp16x3": 1e-3}
FTOL = {"fp64": 1e-12, "fp32": 1e-6, "fp16x3": 1e-6}


def _pair(n):
    return inputs.embed({0: X / 2, n - 1: X}, n)


def _workload(n, B, M, K=2, base=16):
    w = inputs.config(1, n_qubits=n, B=B, M=M, base=base, digits=2)
    w.Hk = w.Hk[:K].copy()
    w.Hk[K - 1] = _pair(n)
    w.lo, w.hi, w.u = w.lo[:K].copy(), w.hi[:K].copy(), w.u[:, :, :K].copy()
    return w


def _table(w, H0=None, **kw):
    from paper_1707_02162_gb300 import redo
    t = redo.Table(w.H0 if H0 is None else H0, w.Hk, w.dt, w.lo, w.hi, w.base, w.digits, fp32=True, **kw)
    if not kw.get("strang"):              # one-qubit tables would need scratch for their step operators
        assert redo.redo_state_grad_workspace(t.handle, 1) == 0
    return t


class _Launches:
    """Launch counts of the profiled phases inside the block."""

    def __enter__(self):
        from paper_1707_02162_gb300 import redo
        redo.redo_profile_enable(True)
        redo.redo_profile_read()
        return self

    def __exit__(self, *exc):
        from paper_1707_02162_gb300 import redo
        self.n = dict.fromkeys(redo.PHASE_NAMES, 0) | {k: v[1] for k, v in redo.redo_profile_read().items()}
        redo.redo_profile_enable(False)


def _digits(w):
    return _ref.oracle_levels(w)[1]


@pytest.mark.parametrize("variant", ["1", "2", "3"])
def test_dense_tensor_core_variants(monkeypatch, variant):
    w = _workload(6, B=7, M=80, K=3)                # 7 pulses: a ragged last CTA for 2 and 3 chains
    t = _table(w, fp16x3=True, levels=True)
    q = t.quantize(w.u)
    monkeypatch.setenv("REDO_TC_VARIANT", variant)
    with _Launches() as p:
        U, F, _ = t.propagate(q, "fp16x3", target=w.target, reunit_every=16)
        U0, _, _ = t.propagate(q, "fp16x3")
    assert p.n["chain_tc"] == 2
    U64, F64, _ = t.propagate(q, "fp64", target=w.target)
    assert (U - U64).abs().max().item() < TOL["fp16x3"] and (U0 - U64).abs().max().item() < TOL["fp16x3"]
    assert (F - F64).abs().max().item() < FTOL["fp16x3"]
    t.close()


CHAINS = [(3, "fp64", 0), (3, "fp32", 8), (6, "fp64", 7), (6, "fp32", 0), (6, "fp16x3", 0), (6, "fp16x3", 8),
          (7, "fp64", 0), (7, "fp32", 3)]


@pytest.mark.parametrize("levels", [False, True])
@pytest.mark.parametrize("n,prec,reunit", CHAINS)
def test_dense_phase_propagate(n, prec, reunit, levels):
    w = inputs.phase_config(n, B=2, M=24 if n < 7 else 9, base=16, digits=2)
    w.Hk[1] = _pair(n)
    t = _table(w, fp16x3=n == 6, levels=levels)
    t.set_phase_axes(w.extra["sz"])
    with _Launches() as p:
        U, F, _ = t.propagate_phase(t.quantize(w.u), w.extra["phi"], prec, target=w.target, reunit_every=reunit)
    assert (p.n["chain_tc"] > 0) == (prec == "fp16x3")
    T, D = _ref.oracle_table(w)
    dig = _digits(w)
    for b in range(w.B):
        Uo = O.propagate_phase(T, D, dig[b], w.extra["phi"][b], w.extra["sz"])
        assert np.abs(U[b].cpu().numpy() - Uo).max() < TOL[prec]
        assert abs(float(F[b]) - O.fidelity(w.target, Uo)) < FTOL[prec]
    t.close()


@pytest.mark.parametrize("n,M,prec,ck", [(3, 12, "fp64", 0), (3, 12, "fp64", 4), (3, 12, "fp32", 0), (6, 6, "fp64", 2),
                                         (6, 6, "fp32", 2), (7, 5, "fp64", 0), (7, 5, "fp32", 2)])
def test_dense_phase_gradient(n, M, prec, ck):
    w = inputs.phase_config(n, B=2, M=M, base=16, digits=2)
    w.Hk[1] = _pair(n)
    t = _table(w)
    t.set_phase_axes(w.extra["sz"])
    F, gA, gP = t.fidelity_grad_phase(t.quantize(w.u), w.extra["phi"], w.target, prec, checkpoint_every=ck)
    T, D = _ref.oracle_table(w)
    dig = _digits(w)
    rel = 1e-10 if prec == "fp64" else 2e-3         # differences of nearly equal boundary traces
    for b in range(w.B):
        Fo, gAo, gPo = O.phase_gradient(T, D, w.Hk, w.extra["sz"], w.dt, dig[b], w.extra["phi"][b], w.target)
        assert abs(float(F[b]) - Fo) < FTOL[prec]
        assert np.abs(gA[b].cpu().numpy() - gAo).max() <= rel * np.abs(gAo).max()
        assert np.abs(gP[b].cpu().numpy() - gPo).max() <= rel * np.abs(gPo).max()
    t.close()


def _drift(w, seed=3):
    rng = np.random.default_rng(seed)
    return np.stack([np.diag(w.H0).real * rng.uniform(0.5, 1.5) for _ in range(w.B)])


@pytest.mark.parametrize("n,prec,reunit", CHAINS)
def test_dense_drift_propagate(n, prec, reunit):
    w = _workload(n, B=2, M=24 if n < 7 else 9)
    h = _drift(w)
    t = _table(w, H0=np.zeros_like(w.H0), fp16x3=n == 6)
    with _Launches() as p:
        U, F, _ = t.propagate_drift(t.quantize(w.u), h, prec, target=w.target, reunit_every=reunit)
    assert (p.n["chain_tc"] > 0) == (prec == "fp16x3")
    T, _ = _ref.oracle_table(w)
    dig = _digits(w)
    for b in range(w.B):
        Uo = O.propagate(T, np.diag(np.exp(-1j * w.dt * h[b])), dig[b])
        assert np.abs(U[b].cpu().numpy() - Uo).max() < TOL[prec]
        assert abs(float(F[b]) - O.fidelity(w.target, Uo)) < FTOL[prec]
    t.close()


@pytest.mark.parametrize("n,M,prec,ck", [(3, 40, "fp64", 0), (3, 40, "fp64", 4), (3, 40, "fp32", 4), (5, 40, "fp32", 4),
                                         (6, 6, "fp32", 2), (7, 5, "fp64", 2), (7, 5, "fp32", 0)])
def test_dense_drift_gradient(n, M, prec, ck):
    w = _workload(n, B=2, M=M)
    h = _drift(w)
    t = _table(w, H0=np.zeros_like(w.H0))
    F, g = t.fidelity_grad_drift(t.quantize(w.u), h, w.target, prec, checkpoint_every=ck, reunit_every=ck)
    T, _ = _ref.oracle_table(w)
    dig = _digits(w)
    for b in range(w.B):
        Fo, go = O.grape_gradient(T, np.diag(np.exp(-1j * w.dt * h[b])), w.Hk, w.dt, dig[b], w.target)
        assert abs(float(F[b]) - Fo) < FTOL[prec]
        assert np.abs(g[b].cpu().numpy() - go).max() <= GTOL[prec] * np.abs(go).max()
    t.close()


@pytest.mark.parametrize("n,M,ck", [(3, 49, 5), (5, 49, 2), (7, 49, 5), (7, 49, 2)])
@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp16x3"])
def test_dense_reunitarised_gradient_many_segments(n, M, ck, prec):
    # 10 and 25 segments: the grouped scans, with the polar step before them; F to its own tolerance
    if prec == "fp16x3" and n < 7:
        pytest.skip("the split-FP16 gradient needs N >= 128")
    w = _workload(n, B=2, M=M)
    t = _table(w, fp16x3=n == 7)
    F, g = t.fidelity_grad(t.quantize(w.u), w.target, prec, checkpoint_every=ck, reunit_every=ck)
    T, D = _ref.oracle_table(w, method="eig")
    dig = _digits(w)
    for b in range(w.B):
        Fo, go = O.grape_gradient(T, D, w.Hk, w.dt, dig[b], w.target)
        assert abs(float(F[b]) - Fo) < FTOL[prec]
        assert np.abs(g[b].cpu().numpy() - go).max() <= GTOL[prec] * np.abs(go).max()
    t.close()


@pytest.mark.parametrize("nb,keep", [("128", "1"), ("256", "1"), ("128", "0"), ("256", "0")])
@pytest.mark.parametrize("ck", [0, 2])
@pytest.mark.parametrize("rows", ["one", "several"])
def test_dense_tensor_core_gradient_n256(monkeypatch, nb, keep, ck, rows):
    # both operand-block widths, kept and undone states, one nonzero per row of H_k and several
    monkeypatch.setenv("REDO_TCL_NB", nb)
    monkeypatch.setenv("REDO_TCL_KEEP", keep)
    w = _workload(8, B=2, M=5)
    if rows == "several":
        w.Hk[0] = w.Hk[0] + inputs.embed({3: X / 2}, 8)
    t = _table(w, fp16x3=True)
    with _Launches() as p:
        F, g = t.fidelity_grad(t.quantize(w.u), w.target, "fp16x3", checkpoint_every=ck)
    assert min(p.n[k] for k in ("grad_forward_sweep", "grad_scans", "grad_reverse_sweep")) > 0
    T, D = _ref.oracle_table(w, method="eig")
    dig = _digits(w)
    for b in range(w.B):
        Fo, go = O.grape_gradient(T, D, w.Hk, w.dt, dig[b], w.target)
        assert abs(float(F[b]) - Fo) < FTOL["fp16x3"]
        assert np.abs(g[b].cpu().numpy() - go).max() <= GTOL["fp16x3"] * np.abs(go).max()
    U, _, _ = t.propagate(t.quantize(w.u), "fp16x3", reunit_every=2)
    for b in range(w.B):
        assert np.abs(U[b].cpu().numpy() - O.propagate(T, D, dig[b])).max() < TOL["fp16x3"]
    t.close()


@pytest.mark.parametrize("n,B,M", [(3, 3, 40), (6, 3, 20), (7, 2, 20), (7, 160, 5), (9, 2, 6)])
@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp16x3"])
def test_dense_simulate_and_state_gradient(n, B, M, prec):
    # N <= 64: a CTA per pulse; above: every SM on every step, or from one pulse per SM on streamed
    # operators.  Checked against the FP64 propagators of every step, those against the oracle's.
    if prec == "fp16x3" and n not in (6, 9):
        pytest.skip("split FP16 runs the state in FP32; the propagator is tested at these sizes")
    w = _workload(n, B=B, M=M)
    rng = np.random.default_rng(n)
    psi0, psiT = (torch.as_tensor(v / np.linalg.norm(v, axis=-1, keepdims=True), device="cuda") for v in
                  rng.normal(size=(2, B, w.N)) + 1j * rng.normal(size=(2, B, w.N)))
    obs = torch.as_tensor(rng.uniform(-1, 1, w.N), device="cuda")
    t = _table(w, fp16x3=prec == "fp16x3")
    q = t.quantize(w.u)
    e, U = t.simulate(q, psi0, obs, prec, want_U=True)
    T, D = _ref.oracle_table(w, method="eig")
    dig = _digits(w)
    tol = 1e-12 if prec == "fp64" else 2e-5
    for b in (0, B - 1):
        psi = psi0[b].cpu().numpy()
        for m in range(M):
            psi = O.propagate(T, D, dig[b][m:m + 1]) @ psi
            assert abs(float(e[b, m + 1]) - np.abs(psi) ** 2 @ obs.cpu().numpy()) < tol
        assert np.abs(U[b].cpu().numpy() - O.propagate(T, D, dig[b])).max() < TOL[prec]
    if prec != "fp16x3":
        F, g = t.state_grad(q, psi0, psiT, prec)
        for b in (0, B - 1):
            Fo, go = O.state_transfer_gradient(T, D, w.Hk, w.dt, dig[b], psi0[b].cpu().numpy(), psiT[b].cpu().numpy())
            assert abs(float(F[b]) - Fo) < (1e-12 if prec == "fp64" else 2e-5)
            assert np.abs(g[b].cpu().numpy() - go).max() <= GTOL[prec] * np.abs(go).max()
    t.close()


@pytest.mark.parametrize("n,prec,reunit", [(3, "fp64", 0), (3, "fp32", 8), (6, "fp64", 0), (6, "fp16x3", 8),
                                           (7, "fp64", 0), (7, "fp16x3", 0)])
@pytest.mark.parametrize("drift", ["diagonal", "transverse"])
def test_dense_strang_chains(n, prec, reunit, drift):
    w = _workload(n, B=2, M=24 if n < 7 else 9)
    if drift == "transverse":
        w.H0 = w.H0 + 2 * np.pi * 800.0 * inputs.embed({1: X}, n)
    t = _table(w, fp16x3=n >= 6, strang=True)
    U, F, _ = t.propagate(t.quantize(w.u), prec, target=w.target, reunit_every=reunit)
    T, _ = _ref.oracle_table(w)
    Dh = O.half_drift(w.H0, w.dt)
    dig = _digits(w)
    for b in range(w.B):
        Uo = O.propagate_strang(T, Dh, dig[b])
        assert np.abs(U[b].cpu().numpy() - Uo).max() < TOL[prec]
        assert abs(float(F[b]) - O.fidelity(w.target, Uo)) < FTOL[prec]
    t.close()


@pytest.mark.parametrize("n,prec,reunit", CHAINS + [(7, "fp16x3", 3)])
def test_transverse_drift_keeps_dense_products(n, prec, reunit):
    # one-qubit controls, but a drift that is not diagonal
    w = inputs.config(1, n_qubits=n, B=2, M=24 if n < 7 else 9, base=16, digits=2)
    w.Hk, w.lo, w.hi, w.u = w.Hk[:2].copy(), w.lo[:2].copy(), w.hi[:2].copy(), w.u[:, :, :2].copy()
    w.H0 = w.H0 + 2 * np.pi * 800.0 * (inputs.embed({0: X}, n) + inputs.embed({0: X / 2, 1: X}, n))
    t = _table(w, fp16x3=n >= 6)
    q = t.quantize(w.u)
    U, F, _ = t.propagate(q, prec, target=w.target, reunit_every=reunit)
    T, D = _ref.oracle_table(w)
    dig = _digits(w)
    grad = t.fidelity_grad(q, w.target, prec, checkpoint_every=4) if prec != "fp16x3" or n >= 7 else None
    for b in range(w.B):
        Uo = O.propagate(T, D, dig[b])
        assert np.abs(U[b].cpu().numpy() - Uo).max() < TOL[prec]
        assert abs(float(F[b]) - O.fidelity(w.target, Uo)) < FTOL[prec]
        if grad is not None:
            Fo, go = O.grape_gradient(T, D, w.Hk, w.dt, dig[b], w.target)
            assert abs(float(grad[0][b]) - Fo) < FTOL[prec]
            assert np.abs(grad[1][b].cpu().numpy() - go).max() <= GTOL[prec] * np.abs(go).max()
    t.close()
