"""The seam between slices of step operators (512 MiB of scratch) in every call that has one."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1707_02162_gb300 import inputs, redo  # noqa: E402

pytestmark = pytest.mark.gpu


def _table(w, H0=None, **kw):
    return redo.Table(w.H0 if H0 is None else H0, w.Hk, w.dt, w.lo, w.hi, w.base, w.digits, fp32=True, **kw)


# Two slices of step operators: distinct pulses at both ends of the batch, one repeated between.
def _batch(q2, B):
    q = q2[:1].expand(B, -1, -1).contiguous()
    q[-1] = q2[1]
    return q


def _close(a, b, rel):
    return (a - b).abs().max().item() <= rel * b.abs().max().item()


@pytest.mark.parametrize("prec,B,M", [("fp32", 260, 2000), ("fp64", 140, 2000)])
def test_slice_seam_of_drift_and_phase_gradients(prec, B, M):
    w = inputs.phase_config(6, B=2, M=M, base=16, digits=2)
    t = _table(w, H0=np.zeros_like(w.H0))
    t.set_phase_axes(w.extra["sz"])
    q2 = t.quantize(w.u)
    q = _batch(q2, B)
    rng = np.random.default_rng(2)
    h = torch.as_tensor(np.diag(w.H0).real * rng.uniform(0.5, 1.5, (B, 1)), device="cuda")
    phi2 = torch.as_tensor(w.extra["phi"], device="cuda")
    phi = _batch(phi2, B)
    UT = torch.as_tensor(w.target, device="cuda")
    rel = 1e-9 if prec == "fp64" else 5e-3       # FP32: 2000 steps, segments scanned in another order
    F, g = t.fidelity_grad_drift(q, h, UT, prec, checkpoint_every=100, reunit_every=100)
    F1, g1 = t.fidelity_grad_drift(q2, torch.stack([h[0], h[-1]]), UT, prec, checkpoint_every=100, reunit_every=100)
    assert _close(g[0], g1[0], rel) and _close(g[-1], g1[1], rel)
    F2, g2 = t.fidelity_grad_drift(q[B - 3:].contiguous(), h[B - 3:].contiguous(), UT, prec, checkpoint_every=100,
                                   reunit_every=100)
    assert _close(g[B - 3:], g2, rel)
    _, ga, gp = t.fidelity_grad_phase(q, phi, UT, prec, checkpoint_every=100)
    _, ga1, gp1 = t.fidelity_grad_phase(q2, phi2, UT, prec, checkpoint_every=100)
    for a, b in ((ga, ga1), (gp, gp1)):
        assert torch.equal(a[0], a[B - 2]) and _close(a[0], b[0], rel) and _close(a[-1], b[1], rel)
    t.close()


@pytest.mark.parametrize("prec,B,M", [("fp32", 420, 2000), ("fp64", 240, 2000)])
def test_slice_seam_of_simulations(prec, B, M):
    w = inputs.config(1, n_qubits=6, B=2, M=M, base=16, digits=2)
    t = _table(w)
    q2 = t.quantize(w.u)
    rng = np.random.default_rng(3)
    v = rng.normal(size=(B, w.N)) + 1j * rng.normal(size=(B, w.N))
    psi = torch.as_tensor(v / np.linalg.norm(v, axis=1, keepdims=True), device="cuda")
    obs = torch.as_tensor(rng.uniform(-1, 1, w.N), device="cuda")
    e, _ = t.simulate(_batch(q2, B), psi, obs, prec, want_U=False)
    for b, i in ((0, 0), (B - 2, 0), (B - 1, 1)):
        e1, _ = t.simulate(q2[i:i + 1].contiguous(), psi[b:b + 1].contiguous(), obs, prec, want_U=False)
        assert torch.equal(e[b], e1[0])
    t.close()


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_slice_seam_of_state_gradients(prec):
    w = inputs.config(1, n_qubits=6, B=2, M=5, base=16, digits=2)
    t = _table(w)
    B = 2800
    q2 = t.quantize(w.u)
    rng = np.random.default_rng(4)
    v = rng.normal(size=(2, B, w.N)) + 1j * rng.normal(size=(2, B, w.N))
    psi0, psiT = (torch.as_tensor(x / np.linalg.norm(x, axis=1, keepdims=True), device="cuda") for x in v)
    F, g = t.state_grad(_batch(q2, B), psi0, psiT, prec)
    for b, i in ((0, 0), (B - 2, 0), (B - 1, 1)):
        F1, g1 = t.state_grad(q2[i:i + 1].contiguous(), psi0[b:b + 1].contiguous(), psiT[b:b + 1].contiguous(), prec)
        assert torch.equal(F[b], F1[0]) and torch.equal(g[b], g1[0])
    t.close()
