"""Systems that are not locally controlled (here a two-qubit control among the x/y ones) keep the dense
operators: the tensor-core chains and sweeps, the two-pass combine and the grouped scans, against
the oracle.  Tolerances are those the dense paths are held to elsewhere."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import redo_oracle as O  # noqa: E402
from paper_1707_02162_gb300 import inputs  # noqa: E402
from tests import _ref  # noqa: E402

pytestmark = pytest.mark.gpu
X = inputs.PAULI["X"]


def _workload(n, B, M, base=16):
    w = inputs.config(1, n_qubits=n, B=B, M=M, base=base, digits=2)
    w.Hk = w.Hk[:3].copy()
    w.Hk[1] = inputs.embed({0: X / 2, n - 1: X}, n)
    w.lo, w.hi, w.u = w.lo[:3].copy(), w.hi[:3].copy(), w.u[:, :, :3].copy()
    return w


def _table(w, **kw):
    from paper_1707_02162_gb300 import redo
    return redo.Table(w.H0, w.Hk, w.dt, w.lo, w.hi, w.base, w.digits, fp32=True, **kw)


@pytest.mark.parametrize("levels", [False, True])
@pytest.mark.parametrize("prec,reunit,tol,ftol", [("fp64", 0, 1e-12, 1e-12), ("fp32", 13, 2e-4, 1e-6),
                                                  ("fp16x3", 13, 2e-4, 1e-6), ("fp16x3", 0, 2e-4, 1e-6)])
def test_dense_chains_n64(levels, prec, reunit, tol, ftol):
    w = _workload(6, B=3, M=160)                     # 13 ragged segments: a two-pass combine
    t = _table(w, fp16x3=True, levels=levels)
    U, F, _ = t.propagate(t.quantize(w.u), prec, target=w.target, reunit_every=reunit)
    T, D = _ref.oracle_table(w)
    _, dig, _, _ = _ref.oracle_levels(w)
    for b in range(w.B):
        Uo = O.propagate(T, D, dig[b])
        assert np.abs(U[b].cpu().numpy() - Uo).max() < tol
        assert abs(float(F[b]) - O.fidelity(w.target, Uo)) < ftol
    t.close()


@pytest.mark.parametrize("n,ck", [(5, 0), (5, 2), (7, 2), (7, 0)])
@pytest.mark.parametrize("prec,gtol", [("fp64", 1e-10), ("fp32", 2e-4), ("fp16x3", 1e-3)])
def test_dense_gradients_many_segments(n, ck, prec, gtol):
    # ck = 2: 25 segments, scanned in groups (two pulses)
    if prec == "fp16x3" and n < 7:
        pytest.skip("the split-FP16 gradient needs N >= 128")
    w = _workload(n, B=2, M=49)
    t = _table(w, fp16x3=n == 7)
    F, g = t.fidelity_grad(t.quantize(w.u), w.target, prec, checkpoint_every=ck)
    T, D = _ref.oracle_table(w, method="eig")
    _, dig, _, _ = _ref.oracle_levels(w)
    for b in range(w.B):
        Fo, go = O.grape_gradient(T, D, w.Hk, w.dt, dig[b], w.target)
        assert abs(float(F[b]) - Fo) < 1e-6
        assert np.abs(g[b].cpu().numpy() - go).max() <= gtol * np.abs(go).max()
    t.close()
