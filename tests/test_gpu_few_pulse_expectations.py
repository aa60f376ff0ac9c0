"""Expectations of a few FP32 pulses under diagonal controls: weights of any length and not rounded, bad
levels counted once per digit, as in the general kernel; and factor tables that fill shared memory."""
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


@pytest.mark.parametrize("n,base,prec,B", [(4, 128, "fp32", 3), (4, 128, "fp32", 700), (4, 128, "fp32", 2500),
                                           (3, 256, "fp64", 4900), (3, 100, "fp32", 4870)])
def test_large_factor_tables(n, base, prec, B):
    # two controls of base^2 levels: one to three blocks an SM, in blocks of 32 to 256 threads; every
    # pulse as one of a few is
    rng = np.random.default_rng(n)
    N, M, K = 2 ** n, 9, 2
    A = rng.normal(size=(N, N)) + 1j * rng.normal(size=(N, N))
    Hk = np.stack([np.diag(rng.normal(size=N)) for _ in range(K)]).astype(np.complex128)
    t = redo.Table((A + A.conj().T) / 2, Hk, 0.1, -np.ones(K), np.ones(K), base, 2, fp32=True)
    q = torch.randint(0, base * base, (B, M, K), dtype=torch.int32, device="cuda",
                      generator=torch.Generator(device="cuda").manual_seed(7))
    rho, obs = rng.uniform(-1, 1, N), rng.uniform(-1, 1, N)
    e, m = t.expect_diag(q, rho, obs, prec)
    tol = 1e-12 if prec == "fp64" else 2e-5
    for b in sorted({0, B // 2, B - 1}):
        e1, m1 = t.expect_diag(q[b:b + 1].contiguous(), rho, obs, "fp64")
        assert (e[b] - e1[0]).abs().max().item() < tol and abs(float(m[b] - m1[0])) < tol
    t.close()
