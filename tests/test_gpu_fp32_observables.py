"""FP32 simulations of locally controlled systems take observables and states of any length, as their FP64
sums did: the same FP32 states, added in FP32 pairs or in FP64."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1707_02162_gb300 import inputs, redo  # noqa: E402

pytestmark = pytest.mark.gpu


def _workload(n, B, M, seed=1):
    rng = np.random.default_rng(seed)
    w = inputs.config(1, n_qubits=n, B=B, M=M, base=16, digits=2)
    return w, rng


def _table(w):
    return redo.Table(w.H0, w.Hk, w.dt, w.lo, w.hi, w.base, w.digits, fp32=True)


def _states(rng, B, N):
    v = rng.normal(size=(B, N)) + 1j * rng.normal(size=(B, N))
    return torch.as_tensor(v / np.linalg.norm(v, axis=1, keepdims=True), device="cuda")


@pytest.mark.parametrize("n", [1, 3, 6, 7, 9, 10])
@pytest.mark.parametrize("obs_f,psi_f", [(1e45, 1.0), (1e-45, 1.0), (1.0, 1e25), (1.0, 1e-25), (1e30, 1e-30)])
def test_simulated_observables_of_any_length(n, obs_f, psi_f):
    # the same FP32 states summed in FP64 and in FP32 pairs: 2^-40 of the largest weight
    w, rng = _workload(n, B=3, M=7)
    w.Hk, w.lo, w.hi, w.u = w.Hk[:1].copy(), w.lo[:1].copy(), w.hi[:1].copy(), w.u[:, :, :1].copy()
    w.base, w.digits = 4, 2
    t = _table(w)
    q = t.quantize(w.u)
    psi0 = _states(rng, 3, w.N)
    psi0[1] = 0
    psi0[1, w.N // 2] = 1
    obs = torch.as_tensor(rng.uniform(-1, 1, w.N), device="cuda")
    e, _ = t.simulate(q, psi0, obs, "fp32", want_U=False)
    es, _ = t.simulate(q, psi0 * psi_f, obs * obs_f, "fp32", want_U=False)
    # (psi0 * psi_f is rounded to FP32 anew: 2^-24 of each entry)
    tol = 2.0 ** -40 if psi_f == 1.0 else 2.0 ** -21
    assert (es / (obs_f * psi_f * psi_f) - e).abs().max().item() < tol
    t.close()


def test_one_long_state_of_a_batch():
    # a long state sends the sums of its warp's pulses to FP64; all agree to the pairs' 2^-40
    w, rng = _workload(2, B=5, M=7)
    t = _table(w)
    q = t.quantize(w.u)
    psi0 = _states(rng, 5, w.N)
    obs = torch.as_tensor(rng.uniform(-1, 1, w.N), device="cuda")
    e, _ = t.simulate(q, psi0, obs, "fp32", want_U=False)
    psi0[3] *= 2.0 ** 50
    es, _ = t.simulate(q, psi0, obs, "fp32", want_U=False)
    keep = [0, 1, 2, 4]
    assert (es[keep] - e[keep]).abs().max().item() < 2.0 ** -40
    assert (es[3] / 2.0 ** 100 - e[3]).abs().max().item() < 2.0 ** -40
    t.close()
