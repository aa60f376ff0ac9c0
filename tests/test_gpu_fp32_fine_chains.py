"""FP32 propagators of controls on one qubit each, N >= 32: no less exact than the dense FP32 chains."""
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


def _polar(U):
    out = torch.empty_like(U)
    redo.redo_reunitarize(U, out, "fp64", iters=2)
    return out


@pytest.mark.parametrize("n,M", [(5, 200), (6, 200)])
@pytest.mark.parametrize("levels", [False, True])
def test_fp32_chains_of_one_qubit_controls_are_no_less_exact_than_dense(n, M, levels):
    w = inputs.config(1, n_qubits=n, B=8, M=M, base=16, digits=2)
    t = _table(w, levels=levels)
    q = t.quantize(w.u)
    U64, _, _ = t.propagate(q, "fp64")
    U, _, _ = t.propagate(q, "fp32")
    # nearest unitary of each, as re-unitarised calls return it: without it the dense chain's loss of norm
    # is ten times the rest of its error
    err, dense = (float((_polar(x) - U64).abs().square().mean().sqrt()) for x in (U, _dense(t, q, "fp32")))
    assert err <= dense
    t.close()
