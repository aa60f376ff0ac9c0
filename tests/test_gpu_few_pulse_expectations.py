"""Expectations of a few FP32 pulses under diagonal controls: weights of any length and not rounded, bad
levels counted once per digit, as in the general kernel."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1707_02162_gb300 import inputs, redo  # noqa: E402

pytestmark = pytest.mark.gpu


def _diag(n, B, M):
    rng = np.random.default_rng(60 + n)
    N = 2 ** n
    A = rng.normal(size=(N, N)) + 1j * rng.normal(size=(N, N))
    Hk = np.stack([np.diag(rng.normal(size=N)), np.diag(1.0 + rng.normal(size=N))]).astype(np.complex128)
    w = inputs.Workload("diag", n, (A + A.conj().T) / 2, Hk, 0.1, np.array([-1.0, 0.0]), np.array([1.0, 2.0]), 64, 4, 3,
                        np.stack([rng.uniform(-1, 1, (B, M)), rng.uniform(0, 2, (B, M))], -1))
    return w, rng.uniform(-1, 1, N), rng.uniform(-1, 1, N)


def _table(w):
    return redo.Table(w.H0, w.Hk, w.dt, w.lo, w.hi, w.base, w.digits, fp32=True)


@pytest.mark.parametrize("n", [1, 3, 4])
@pytest.mark.parametrize("f", [1e45, 1e-45])
def test_few_pulse_expectations_of_any_length(n, f):
    # FP64 sums of the same FP32 states beside FP32 sums of N terms of at most 1: N roundings of 2^-24
    w, rho, obs = _diag(n, B=5, M=50)
    t = _table(w)
    q = t.quantize(w.u)
    e, m = t.expect_diag(q, rho, obs, "fp32")
    es, ms = t.expect_diag(q, rho, obs * f, "fp32")
    tol = w.N * 2.0 ** -24 * np.abs(rho).sum()
    assert (es / f - e).abs().max().item() < tol and (ms / f - m).abs().max().item() < tol
    t.close()


@pytest.mark.parametrize("n", [1, 3, 4])
def test_few_pulse_expectations_do_not_round_the_weights(n):
    w, rho, _ = _diag(n, B=5, M=50)
    t = _table(w)
    q = t.quantize(w.u)
    one, m1 = t.expect_diag(q, rho, np.ones(w.N), "fp32")
    a, ma = t.expect_diag(q, rho, np.full(w.N, 1.0 + 2.0 ** -30), "fp32")
    # FP32 sums of what the weights' second parts add, and FP64 rounding of both results, times 2^30
    tol = (w.N * 2.0 ** -24 + 4 * 2.0 ** -53 * 2.0 ** 30) * np.abs(rho).sum()
    assert ((a - one) * 2.0 ** 30 - one).abs().max().item() < tol
    assert ((ma - m1) * 2.0 ** 30 - m1).abs().max().item() < tol
    t.close()


def test_few_pulse_expectations_count_bad_levels_once_per_digit():
    w, rho, obs = _diag(3, B=2, M=6)
    t = _table(w)
    q = t.quantize(w.u).clone()
    q[0, 2, 1], q[1, 3, 0] = w.levels, -1
    st = redo.new_status()
    t.expect_diag(q, rho, obs, "fp32", status=st)
    assert int(st[3]) == 2 * w.digits
    t.close()
