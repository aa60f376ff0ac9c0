"""Single pulses of tens of thousands of steps: several hundred segments in the one-qubit form."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1707_02162_gb300 import inputs, redo  # noqa: E402

pytestmark = pytest.mark.gpu


def _table(w, H0=None, **kw):
    return redo.Table(w.H0 if H0 is None else H0, w.Hk, w.dt, w.lo, w.hi, w.base, w.digits, fp32=True, **kw)


def _dense(t, q, prec):
    """The dense chains, which redo_propagate_noalloc always takes."""
    U = torch.empty((q.shape[0], t.N, t.N), dtype=torch.complex128, device="cuda")
    redo.redo_propagate_noalloc(t.handle, q, prec, U, None, None, None)
    return U


@pytest.mark.parametrize("n,prec,tol", [(2, "fp64", 1e-10), (3, "fp64", 1e-10), (3, "fp32", 2e-3), (4, "fp32", 2e-3),
                                        (5, "fp32", 2e-3)])
def test_long_pulse_in_many_segments(n, prec, tol):
    # 40001 ragged steps: several hundred segments (FP64 rounding of 1.1e-16 a product adds up over the chain's
    # length; FP32 chains this long lose norm, so the bound is loose)
    w = inputs.config(0, n_qubits=n, B=1, M=40001, base=16, digits=2)
    t = _table(w)
    q = t.quantize(w.u)
    U, _, _ = t.propagate(q, prec)
    D = _dense(t, q, "fp64")
    assert (U - D).abs().max().item() < tol
    UT = torch.as_tensor(w.target, device="cuda")
    F, g = t.fidelity_grad(q, UT, prec)
    tau = (UT.conj() * D[0]).sum()
    assert abs(float(F[0]) - float(tau.abs() ** 2) / w.N ** 2) < tol
    F1, g1 = t.fidelity_grad(q, UT, "fp64", checkpoint_every=50)
    assert (g - g1).abs().max().item() <= tol * g1.abs().max().item()
    t.close()
