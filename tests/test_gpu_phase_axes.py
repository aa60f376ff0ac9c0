"""Phase axes set again after a gradient call was captured in a CUDA graph: the replay uses the axes
in force, as an eager call does, also when the new S_kz are not sums of one-qubit parts."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1707_02162_gb300 import inputs  # noqa: E402

pytestmark = pytest.mark.gpu


def _axes(w, n, kind):
    sz = w.extra["sz"].copy()
    if kind == "scaled":
        return -1.5 * sz
    if kind == "general":
        z = [1.0 - 2.0 * ((np.arange(w.N) >> i) & 1) for i in range(n)]
        sz[0] = sz[0] + 0.25 * z[0] * z[1]
    return sz


@pytest.mark.parametrize("first,second", [("species", "scaled"), ("species", "general"), ("general", "scaled")])
@pytest.mark.parametrize("n,prec", [(2, "fp32"), (3, "fp64"), (6, "fp32")])
def test_captured_phase_gradient_follows_the_axes(n, prec, first, second):
    from paper_1707_02162_gb300 import redo
    w = inputs.phase_config(n, B=2, M=11, base=8, digits=2)
    t = redo.Table(w.H0, w.Hk, w.dt, w.lo, w.hi, w.base, w.digits, fp32=True)
    t.set_phase_axes(_axes(w, n, first))
    q = t.quantize(w.u)
    phi = torch.as_tensor(w.extra["phi"], dtype=torch.float64, device="cuda").contiguous()
    target = torch.as_tensor(w.target, dtype=torch.complex128, device="cuda").contiguous()
    before = t.fidelity_grad_phase(q, phi, target, prec, checkpoint_every=4)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        out = t.fidelity_grad_phase(q, phi, target, prec, checkpoint_every=4)
    g.replay()
    assert all(torch.equal(a, b) for a, b in zip(out, before))
    t.set_phase_axes(_axes(w, n, second))
    g.replay()
    torch.cuda.synchronize()
    now = t.fidelity_grad_phase(q, phi, target, prec, checkpoint_every=4)
    assert all(torch.equal(a, b) for a, b in zip(out, now))
    assert not torch.equal(now[2], before[2])
    t.close()
