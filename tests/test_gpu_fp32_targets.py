"""FP32 gradients of locally controlled systems keep the range that FP64 traces gave them: targets and
states of any length.  Lengths that are powers of two come out as exactly that factor of the results."""
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


@pytest.mark.parametrize("n,ck", [(1, 0), (3, 0), (4, 5), (6, 5), (7, 5)])
@pytest.mark.parametrize("e", [90, -90])
def test_gradient_of_scaled_targets(n, ck, e):
    w, _ = _workload(n, B=2, M=17)
    t = _table(w)
    q = t.quantize(w.u)
    f = 2.0 ** e
    UT = torch.as_tensor(w.target, device="cuda")
    F, g = t.fidelity_grad(q, UT, "fp32", checkpoint_every=ck)
    Fs, gs = t.fidelity_grad(q, UT * f, "fp32", checkpoint_every=ck)
    assert torch.equal(gs, g * f * f)
    assert (Fs / f / f - F).abs().max().item() <= 1e-13          # N > 64 adds the overlap's parts in no fixed order
    t.close()


@pytest.mark.parametrize("e", [90, -90])
def test_phase_gradient_of_scaled_targets(e):
    w = inputs.phase_config(3, B=2, M=11, base=8, digits=2)
    t = _table(w)
    q = t.quantize(w.u)
    f = 2.0 ** e
    UT = torch.as_tensor(w.target, device="cuda")
    general = w.extra["sz"] + 0.25 * w.extra["sz"][0] * w.extra["sz"][1]
    for sz in (w.extra["sz"], general):
        t.set_phase_axes(sz)
        a = t.fidelity_grad_phase(q, w.extra["phi"], UT, "fp32", checkpoint_every=4)
        b = t.fidelity_grad_phase(q, w.extra["phi"], UT * f, "fp32", checkpoint_every=4)
        assert all(torch.equal(y, x * f * f) for x, y in zip(a, b))
    t.close()


@pytest.mark.parametrize("n", [1, 3, 6, 8])
@pytest.mark.parametrize("e0,eT", [(80, 90), (-80, -90), (80, -75)])
def test_state_gradient_of_scaled_states(n, e0, eT):
    w, rng = _workload(n, B=3, M=9)
    t = _table(w)
    q = t.quantize(w.u)
    psi0, psiT = _states(rng, 3, w.N), _states(rng, 3, w.N)
    F, g = t.state_grad(q, psi0, psiT, "fp32")
    Fs, gs = t.state_grad(q, psi0 * 2.0 ** e0, psiT * 2.0 ** eT, "fp32")
    f = 4.0 ** (e0 + eT)
    assert torch.equal(Fs, F * f) and torch.equal(gs, g * f)
    t.close()


@pytest.mark.parametrize("n", [1, 3, 6])
@pytest.mark.parametrize("e", [140, -140])
def test_gradients_of_controls_in_other_units(n, e):
    # operators times 2^e on a grid times 2^-e: the same steps, gradients times 2^e
    w, rng = _workload(n, B=3, M=9)
    psi0, psiT = _states(rng, 3, w.N), _states(rng, 3, w.N)
    got = []
    for f in (1.0, 2.0 ** e):
        w2 = inputs.Workload(w.name, n, w.H0, w.Hk * f, w.dt, w.lo / f, w.hi / f, w.levels, w.base, w.digits, w.u / f)
        w2.Hk[0] = w.Hk[0]                            # one term in the first unit
        w2.lo[0], w2.hi[0], w2.u[:, :, 0] = w.lo[0], w.hi[0], w.u[:, :, 0]
        t = _table(w2)
        q = t.quantize(w2.u)
        g = t.fidelity_grad(q, torch.as_tensor(w.target, device="cuda"), "fp32", checkpoint_every=4)[1]
        s = t.state_grad(q, psi0, psiT, "fp32")[1]
        got.append((q, g, s))
        t.close()
    (q, g, s), (q2, g2, s2) = got
    assert torch.equal(q, q2)
    for a, b in ((g, g2), (s, s2)):
        assert torch.equal(b[..., 0], a[..., 0]) and torch.equal(b[..., 1:], a[..., 1:] * 2.0 ** e)
