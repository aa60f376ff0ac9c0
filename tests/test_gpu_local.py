"""Locally controlled systems (every control a sum of one-qubit operators, diagonal drift) take
their own chain and gradient kernels; here against the oracle, over the forms that route accepts:
every dimension, several controls and axes per qubit, identity and z parts, a control that is zero,
digit tables too large for one operator per level, step diagonals, ragged segments, re-unitarised
segments, and controls just outside the class, which keep the dense path.

Tolerances: FP64 products of a few hundred 2 x 2 operators, 1e-12; FP32 chains of M (n + 1)
roundings of 6e-8 each, below 2e-5 at M = 29, n <= 7, and 2e-4 of the largest entry for gradients,
as the dense FP32 paths are held to.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import redo_oracle as O  # noqa: E402
from paper_1707_02162_gb300 import inputs  # noqa: E402
from tests import _ref  # noqa: E402

pytestmark = pytest.mark.gpu

SIG = [np.eye(2), np.array([[0, 1], [1, 0]]), np.array([[0, -1j], [1j, 0]]), np.diag([1.0, -1.0])]


def _workload(n, controls, B, M, seed, base=4, digits=3, dt=1e-2):
    """Coefficients in [-1, 1.5]; dt large enough that a step's rotations are of order 0.1 to 1."""
    rng = np.random.default_rng(seed)
    N = 2 ** n
    if controls == "axes":            # three controls, each a random one-qubit operator on every qubit
        Hk = np.stack([sum(inputs.embed({i: sum(c * s for c, s in zip(rng.normal(size=4), SIG))}, n)
                           for i in range(n)) for _ in range(3)])
    elif controls == "z_and_zero":    # a z control, an x control on the last qubit, and a zero operator
        Hk = np.stack([inputs.embed({0: SIG[3] + 0j}, n), inputs.embed({n - 1: SIG[1] + 0j}, n),
                       np.zeros((N, N), dtype=complex)])
    elif controls == "pi":            # half and full turns: vanishing diagonal or off-diagonal entries
        Hk = np.stack([inputs.embed({0: SIG[1] + 0j}, n), inputs.embed({n - 1: SIG[2] + 0j}, n)])
    else:
        Hk = {"local": inputs.controls_local_xy, "global": inputs.controls_global_xy}[controls](n)
    Hk = np.asarray(Hk, dtype=np.complex128) * (20 if controls != "pi" else 1)
    K = Hk.shape[0]
    H0 = np.diag(rng.normal(size=N) * 15).astype(np.complex128)
    lo, hi = np.full(K, -1.0), np.full(K, 1.5)
    u = rng.uniform(-1.1, 1.6, size=(B, M, K))
    if controls == "pi":
        dt, lo, hi = 1.0, np.full(K, -np.pi / 2), np.full(K, np.pi)
        u = rng.integers(-1, 3, size=(B, M, K)) * (np.pi / 2)
        H0 = H0 / 20
    return inputs.Workload("local", n, H0, Hk, dt, lo, hi, base ** digits, base, digits, u,
                           target=inputs.haar_unitary(rng, N))


def _table(w, **kw):
    from paper_1707_02162_gb300 import redo
    return redo.Table(w.H0, w.Hk, w.dt, w.lo, w.hi, w.base, w.digits, fp32=True, **kw)


def _check(w, prec, tol, gtol, ck=0, reunit=0, **kw):
    t = _table(w, **kw)
    q = t.quantize(w.u)
    U, F, _ = t.propagate(q, prec, target=w.target, reunit_every=reunit)
    Fg, g = t.fidelity_grad(q, w.target, prec, checkpoint_every=ck, reunit_every=reunit)
    T, D = O.build_table(w.H0, w.Hk, w.dt, w.lo, w.hi, w.levels, w.base, w.digits, method="eig")
    _, dig, _, _ = _ref.oracle_levels(w)
    for b in range(w.B):
        Uo = O.propagate(T, D, dig[b])
        assert np.abs(U[b].cpu().numpy() - Uo).max() < tol
        assert abs(float(F[b]) - O.fidelity(w.target, Uo)) < tol
        Fo, go = O.grape_gradient(T, D, w.Hk, w.dt, dig[b], w.target)
        assert abs(float(Fg[b]) - Fo) < tol
        assert np.abs(g[b].cpu().numpy() - go).max() <= gtol * max(np.abs(go).max(), 1e-30)
    t.close()


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 6, 7])
@pytest.mark.parametrize("controls", ["local", "global", "axes", "z_and_zero"])
@pytest.mark.parametrize("prec,tol,gtol", [("fp64", 1e-12, 1e-10), ("fp32", 2e-5, 2e-4)])
def test_local_chain_and_gradient(n, controls, prec, tol, gtol):
    _check(_workload(n, controls, B=3, M=29, seed=n), prec, tol, gtol)


@pytest.mark.parametrize("n,M,ck", [(2, 7, 3), (3, 41, 20), (5, 33, 16), (7, 11, 4)])
@pytest.mark.parametrize("prec,tol,gtol", [("fp64", 1e-12, 1e-10), ("fp32", 2e-5, 2e-4)])
def test_local_ragged_reunitarised_segments(n, M, ck, prec, tol, gtol):
    _check(_workload(n, "axes", B=2, M=M, seed=10 + n), prec, tol, gtol, ck=ck, reunit=ck)


@pytest.mark.parametrize("prec,tol,gtol", [("fp64", 1e-12, 1e-10), ("fp32", 2e-5, 2e-4)])
def test_local_half_turns(prec, tol, gtol):
    # entries of the one-qubit operators that vanish exactly or to rounding
    _check(_workload(3, "pi", B=4, M=17, seed=3, base=4, digits=1), prec, tol, gtol)


def test_local_digit_operators():
    # 16^5 levels: the one-qubit tables keep digits
    _check(_workload(3, "axes", B=2, M=9, seed=5, base=16, digits=5), "fp64", 1e-12, 1e-10)


def test_nearly_local_control_keeps_dense_products():
    w = _workload(3, "local", B=2, M=9, seed=6)
    w.Hk[1] = w.Hk[1] + 20 * inputs.embed({0: SIG[1] + 0j, 2: SIG[1] + 0j}, 3)    # a two-qubit term
    _check(w, "fp64", 1e-12, 1e-10)


def test_local_batches_are_sliced_without_a_seam():
    # the step operators of 600 pulses x 2000 steps do not fit one slice of scratch
    w = inputs.config(1, B=2, M=2000)
    t = _table(w)
    q2 = t.quantize(w.u)
    q = q2[:1].expand(600, -1, -1).contiguous()
    q[-1] = q2[1]
    U, _, _ = t.propagate(q, "fp32", reunit_every=100)
    one, _, _ = t.propagate(q2, "fp32", reunit_every=100)
    assert torch.equal(U[0], one[0]) and torch.equal(U[598], one[0]) and torch.equal(U[599], one[1])
    target = torch.as_tensor(w.target, device="cuda")
    F, g = t.fidelity_grad(q, target, "fp32", checkpoint_every=100, reunit_every=100)
    F1, g1 = t.fidelity_grad(q2, target, "fp32", checkpoint_every=100, reunit_every=100)
    # (two pulses scan their segments in groups, so they agree with the large batch to rounding)
    assert torch.equal(g[0], g[598])
    for b, i in ((0, 0), (599, 1)):
        assert (g[b] - g1[i]).abs().max().item() <= 2e-4 * g1[i].abs().max().item()
    t.close()


def test_local_bad_level_index_counts_once_per_digit():
    from paper_1707_02162_gb300 import redo
    w = _workload(3, "axes", B=1, M=5, seed=8)
    t = _table(w)
    q = t.quantize(w.u).clone()
    q[0, 2, 1], q[0, 3, 0] = w.levels, -1
    st = redo.new_status()
    U, _, _ = t.propagate(q, "fp64", status=st)
    q0 = q.clone()
    q0[0, 2, 1] = q0[0, 3, 0] = 0
    U0, _, _ = t.propagate(q0, "fp64")
    assert int(st[3]) == 2 * w.digits and torch.equal(U, U0)
    t.close()


def _states(rng, B, N):
    v = rng.normal(size=(B, N)) + 1j * rng.normal(size=(B, N))
    return torch.as_tensor(v / np.linalg.norm(v, axis=1, keepdims=True), device="cuda")


def _dense_state_sweeps(t, q, prec, psi0, psiT, obs):
    """The dense sweeps, which a call takes when it brings no scratch for the local ones (N <= 64)."""
    from paper_1707_02162_gb300 import redo
    B, M = q.shape[:2]
    e = torch.empty((B, M + 1), dtype=torch.float64, device="cuda")
    redo.redo_simulate(t.handle, q, prec, 0, psi0, obs, e, None, None)
    F = torch.empty(B, dtype=torch.float64, device="cuda")
    g = torch.empty((B, M, t.K), dtype=torch.float64, device="cuda")
    redo.redo_state_grad(t.handle, q, prec, psi0, psiT, F, g, None)
    return e, F, g


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 6])
@pytest.mark.parametrize("controls", ["local", "global", "axes"])
@pytest.mark.parametrize("prec,tol,gtol", [("fp64", 1e-12, 1e-10), ("fp32", 2e-5, 2e-4)])
def test_local_state_sweeps_match_the_dense_ones(n, controls, prec, tol, gtol):
    w = _workload(n, controls, B=37, M=19, seed=20 + n)     # 37: a ragged last warp at every n
    t = _table(w)
    rng = np.random.default_rng(n)
    psi0, psiT = _states(rng, w.B, w.N), _states(rng, w.B, w.N)
    obs = torch.as_tensor(rng.normal(size=w.N), device="cuda")
    q = t.quantize(w.u)
    e, _ = t.simulate(q, psi0, obs, prec, want_U=False)
    F, g = t.state_grad(q, psi0, psiT, prec)
    eo, Fo, go = _dense_state_sweeps(t, q, "fp64", psi0, psiT, obs)
    scale = float(obs.abs().max())
    assert (e - eo).abs().max().item() < tol * scale
    assert (F - Fo).abs().max().item() < tol
    assert (g - go).abs().max().item() <= gtol * go.abs().max().item()
    t.close()


@pytest.mark.parametrize("n,M", [(7, 6), (9, 4), (10, 3)])
@pytest.mark.parametrize("prec,tol,gtol", [("fp64", 1e-12, 1e-10), ("fp32", 2e-5, 2e-4)])
def test_local_state_sweeps_large(n, M, prec, tol, gtol):
    w = _workload(n, "global", B=2, M=M, seed=30 + n, base=4, digits=2)
    t = _table(w)
    rng = np.random.default_rng(n)
    psi0, psiT = _states(rng, w.B, w.N), _states(rng, w.B, w.N)
    obs = torch.as_tensor(rng.normal(size=w.N), device="cuda")
    q = t.quantize(w.u)
    e, _ = t.simulate(q, psi0, obs, prec, want_U=False)
    F, g = t.state_grad(q, psi0, psiT, prec)
    U, _, _ = t.propagate(q, "fp64")
    psi = torch.einsum("bij,bj->bi", U, psi0)
    assert (e[:, -1] - (psi.abs() ** 2) @ obs).abs().max().item() < tol * float(obs.abs().max())
    a = (psiT.conj() * psi).sum(1)
    assert (F - a.abs() ** 2).abs().max().item() < tol
    from paper_1707_02162_gb300 import redo
    go = torch.empty_like(g)
    redo.redo_state_grad(t.handle, q, "fp64", psi0, psiT, None, go, None)      # the dense streamed sweep
    assert (g - go).abs().max().item() <= gtol * go.abs().max().item()
    t.close()


def test_local_state_gradient_over_several_windows():
    # 9001 steps: three windows of step operators, visited forward and then back
    w = _workload(2, "axes", B=3, M=9001, seed=40, dt=1e-3)
    t = _table(w)
    rng = np.random.default_rng(40)
    psi0, psiT = _states(rng, w.B, w.N), _states(rng, w.B, w.N)
    q = t.quantize(w.u)
    F, g = t.state_grad(q, psi0, psiT, "fp64")
    F1, _ = t.state_grad(q, psi0, psiT, "fp64", want_grad=False)
    _, Fo, go = _dense_state_sweeps(t, q, "fp64", psi0, psiT, torch.ones(w.N, dtype=torch.float64, device="cuda"))
    assert (F - Fo).abs().max().item() < 1e-10 and torch.equal(F, F1)
    assert (g - go).abs().max().item() <= 1e-8 * go.abs().max().item()
    t.close()


@pytest.mark.parametrize("n,B", [(1, 3), (2, 5), (3, 4870), (4, 3), (4, 2450)])
@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("fp32", 2e-5)])
def test_diagonal_controls_expectations(n, B, prec, tol):
    # two diagonal controls (one with an identity part) and a dense drift, one warp per block and full
    # blocks with idle lanes; N = 16 in FP64 keeps the general kernel
    rng = np.random.default_rng(50 + n)
    N, M = 2 ** n, 21
    A = rng.normal(size=(N, N)) + 1j * rng.normal(size=(N, N))
    Hk = np.stack([np.diag(rng.normal(size=N)), np.diag(1.0 + rng.normal(size=N))]).astype(np.complex128)
    w = inputs.Workload("diag", n, (A + A.conj().T) / 2, Hk, 0.1, np.array([-1.0, 0.0]), np.array([1.0, 2.0]), 64, 4, 3,
                        np.stack([rng.uniform(-1, 1, (B, M)), rng.uniform(0, 2, (B, M))], -1))
    rho, obs = rng.uniform(-1, 1, N), rng.uniform(-1, 1, N)
    t = _table(w)
    ex, mean = t.expect_diag(t.quantize(w.u), rho, obs, prec)
    _, mean2 = t.expect_diag(t.quantize(w.u), rho, obs, prec, series=False)
    assert torch.equal(mean, mean2)
    T, D = O.build_table(w.H0, w.Hk, w.dt, w.lo, w.hi, w.levels, w.base, w.digits, method="eig")
    _, dig, _, _ = _ref.oracle_levels(w)
    for b in sorted({0, B // 2, B - 1}):
        eo, _ = O.expect_mixed(T, D, dig[b], np.diag(rho).astype(complex), np.diag(obs).astype(complex))
        assert np.abs(ex[b].cpu().numpy() - eo).max() < tol
        assert abs(float(mean[b]) - eo[1:].mean()) < tol
    t.close()


@pytest.mark.parametrize("n", [2, 3, 5, 7])
@pytest.mark.parametrize("axes", ["species", "general"])
@pytest.mark.parametrize("prec,gtol", [("fp64", 1e-9), ("fp32", 2e-4)])
def test_local_phase_gradients(n, axes, prec, gtol):
    # species S_z (sums of one-qubit parts) and general diagonals, which keep the boundary traces
    from paper_1707_02162_gb300 import redo
    w = inputs.phase_config(n, B=2, M=11, base=8, digits=2)
    sz = w.extra["sz"].copy()
    if axes == "general":
        z = [1.0 - 2.0 * ((np.arange(w.N) >> i) & 1) for i in range(n)]
        sz[0] = sz[0] + 0.25 * z[0] * z[1]
    t = _table(w)
    t.set_phase_axes(sz)
    F, ga, gp = t.fidelity_grad_phase(t.quantize(w.u), w.extra["phi"], w.target, prec, checkpoint_every=4)
    T, D = O.build_table(w.H0, w.Hk, w.dt, w.lo, w.hi, w.levels, w.base, w.digits, method="eig")
    _, dig, _, _ = _ref.oracle_levels(w)
    for b in range(w.B):
        Fo, gao, gpo = O.phase_gradient(T, D, w.Hk, sz, w.dt, dig[b], w.extra["phi"][b], w.target)
        assert abs(float(F[b]) - Fo) < (1e-12 if prec == "fp64" else 2e-5)
        assert np.abs(ga[b].cpu().numpy() - gao).max() <= gtol * np.abs(gao).max()
        assert np.abs(gp[b].cpu().numpy() - gpo).max() <= gtol * np.abs(gpo).max()
    t.close()
