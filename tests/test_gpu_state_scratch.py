"""The state-transfer scratch of a batch serves every smaller batch."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1707_02162_gb300 import inputs, redo  # noqa: E402

pytestmark = pytest.mark.gpu


def _table(w, H0=None, **kw):
    return redo.Table(w.H0 if H0 is None else H0, w.Hk, w.dt, w.lo, w.hi, w.base, w.digits, fp32=True, **kw)


@pytest.mark.parametrize("n", [2, 6, 8])
def test_state_scratch_serves_smaller_batches(n):
    w = inputs.config(1, n_qubits=n, B=1, M=2, base=16, digits=2)
    t = _table(w)
    sizes = [redo.redo_state_grad_workspace(t.handle, B) for B in list(range(1, 400)) + [999, 1000, 5000, 20000, 20001]]
    assert all(a <= b for a, b in zip(sizes, sizes[1:]))
    t.close()
