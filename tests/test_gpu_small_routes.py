"""Small FP64 systems change between the one-qubit form and the dense operators with the batch (one pulse
per SM) and the number of factors: both sides of that line against the oracle, and pulse by pulse alike."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import redo_oracle as O  # noqa: E402
from paper_1707_02162_gb300 import inputs, redo  # noqa: E402
from tests import _ref  # noqa: E402

pytestmark = pytest.mark.gpu


def _sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def _table(w, H0=None, **kw):
    return redo.Table(w.H0 if H0 is None else H0, w.Hk, w.dt, w.lo, w.hi, w.base, w.digits, fp32=True, **kw)


@pytest.mark.parametrize("levels", [False, True])
@pytest.mark.parametrize("n", [1, 2, 3, 4])
@pytest.mark.parametrize("extra", [-1, 0])
def test_plain_calls_at_one_pulse_per_sm(n, extra, levels):
    B, M = _sms() + extra, 19
    w = inputs.config(0, n_qubits=n, B=B, M=M, base=4, digits=2)
    t = _table(w, levels=levels)
    q = t.quantize(w.u)
    U, F, _ = t.propagate(q, "fp64", target=w.target)
    Fg, g = t.fidelity_grad(q, w.target, "fp64")
    psi = np.zeros(w.N, dtype=complex)
    psi[0] = 1
    obs = np.linspace(-1, 1, w.N)
    e, Us = t.simulate(q, psi, obs, "fp64")
    T, D = _ref.oracle_table(w)
    _, dig, _, _ = _ref.oracle_levels(w)
    for b in (0, B // 2, B - 1):
        Uo = O.propagate(T, D, dig[b])
        Fo, go = O.grape_gradient(T, D, w.Hk, w.dt, dig[b], w.target)
        eo, _ = O.simulate_expectation(T, D, dig[b], psi, obs)
        assert np.abs(U[b].cpu().numpy() - Uo).max() < 1e-12 and np.abs(Us[b].cpu().numpy() - Uo).max() < 1e-12
        assert abs(float(F[b]) - Fo) < 1e-12 and abs(float(Fg[b]) - Fo) < 1e-12
        assert np.abs(g[b].cpu().numpy() - go).max() <= 1e-10 * np.abs(go).max()
        assert np.abs(e[b].cpu().numpy() - eo).max() < 1e-12
    t.close()


@pytest.mark.parametrize("n", [1, 2, 3])
@pytest.mark.parametrize("extra", [-1, 0])
def test_drift_and_phase_calls_at_one_pulse_per_sm(n, extra):
    B, M = _sms() + extra, 13
    w = inputs.phase_config(n, B=B, M=M, base=4, digits=2)
    t = _table(w, H0=np.zeros_like(w.H0))
    rng = np.random.default_rng(n)
    h = np.diag(w.H0).real * rng.uniform(0.5, 1.5, (B, 1))
    q = t.quantize(w.u)
    U, F, _ = t.propagate_drift(q, h, "fp64", target=w.target)
    Fg, g = t.fidelity_grad_drift(q, h, w.target, "fp64", checkpoint_every=5)
    T, D0 = O.build_table(np.zeros_like(w.H0), w.Hk, w.dt, w.lo, w.hi, w.levels, w.base, w.digits)
    _, dig, _, _ = _ref.oracle_levels(w)
    t.set_phase_axes(w.extra["sz"])
    Up, _, _ = t.propagate_phase(q, w.extra["phi"], "fp64")
    for b in (0, B // 2, B - 1):
        D = np.diag(np.exp(-1j * w.dt * h[b]))
        Fo, go = O.grape_gradient(T, D, w.Hk, w.dt, dig[b], w.target)
        assert np.abs(U[b].cpu().numpy() - O.propagate(T, D, dig[b])).max() < 1e-12
        assert abs(float(F[b]) - Fo) < 1e-12 and abs(float(Fg[b]) - Fo) < 1e-12
        assert np.abs(g[b].cpu().numpy() - go).max() <= 1e-10 * np.abs(go).max()
        Uo = O.propagate_phase(T, D0, dig[b], w.extra["phi"][b], w.extra["sz"])
        assert np.abs(Up[b].cpu().numpy() - Uo).max() < 1e-12
    t.close()


@pytest.mark.parametrize("K,levels", [(1, False), (2, False), (2, True), (3, True)])
@pytest.mark.parametrize("n", [2, 3, 4])
def test_simulations_on_both_sides_of_the_factor_count(n, K, levels):
    B, M = _sms() + 3, 11
    w = inputs.config(1, n_qubits=n, B=B, M=M, base=4, digits=2)
    w.Hk, w.lo, w.hi, w.u = w.Hk[:K].copy(), w.lo[:K].copy(), w.hi[:K].copy(), w.u[:, :, :K].copy()
    t = _table(w, levels=levels)
    q = t.quantize(w.u)
    rng = np.random.default_rng(K)
    psi = rng.normal(size=w.N) + 1j * rng.normal(size=w.N)
    psi /= np.linalg.norm(psi)
    obs = rng.uniform(-1, 1, w.N)
    e, _ = t.simulate(q, psi, obs, "fp64", want_U=False)
    small, _ = t.simulate(q[:5].contiguous(), psi, obs, "fp64", want_U=False)
    assert (e[:5] - small).abs().max().item() < 1e-12
    T, D = _ref.oracle_table(w)
    _, dig, _, _ = _ref.oracle_levels(w)
    eo, _ = O.simulate_expectation(T, D, dig[B - 1], psi, obs)
    assert np.abs(e[B - 1].cpu().numpy() - eo).max() < 1e-12
    t.close()
