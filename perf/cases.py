"""The calls that users of this framework make, over the range in which they make them.

Every case is one call sequence of the Python API on a control problem of the kind the repository
is for: NMR-like spins with a diagonal offset-and-coupling drift, driven by x/y controls on every
qubit ("local") or on all of them together ("global"), plus the driven Ising chain of the freezing
study and the warm-start network.  Sizes, time steps, level grids and re-unitarisation periods are
those of the seeded workloads, the tests and the benchmark, and ranges around them.

Results of reduced-precision calls (FP32, split FP16) are returned at single width, as a caller who
asked for them keeps them; FP64 calls return what the API returns.  Reduced chains longer than a few
thousand operator products are re-unitarised, as the API's documentation asks for.
"""
import math

import numpy as np
import torch

from paper_1707_02162_gb300 import redo
from paper_1707_02162_gb300.warmstart import MLP

OMEGA = 2 * math.pi * 1e4          # largest control amplitude, rad/s


def listed():
    return [
        # One three-qubit pulse of 1000 steps in FP64: the smallest call, what an interactive user or
        # an outer search that looks at one pulse at a time waits for.
        _prop("pulse_single", n=3, ctl="global", B=1, M=1000, prec="fp64"),
        # The benchmark: 256 six-qubit pulses of 2000 steps, level table, split FP16 re-unitarised.
        _prop("pulse_batch", n=6, ctl="local", B=256, M=2000, prec="fp16x3", reunit=64, levels=True),
        # A ragged ordinary batch in single precision with global (shared-coil) controls.
        _prop("pulse_ragged", n=5, ctl="global", B=37, M=611, prec="fp32", reunit=50),
        # One GRAPE evaluation of a single small pulse in FP64 (an optimiser's inner call).
        _grad("grape_single", n=3, ctl="global", B=1, M=200, prec="fp64"),
        # The warm-start study's batch: every instance with its own drift and its own target.
        _grad("grape_batch", n=5, ctl="local", B=256, M=500, prec="fp32", ck=50, reunit=50, drift="pulse",
              target="rotations", dt=2e-6),
        # Eight-qubit GRAPE on the tensor-core precision, close to its target as in mid-run.
        _grad("grape_n256", n=8, ctl="local", B=1, M=200, prec="fp16x3", ck=8, reunit=8, target="near", dt=2e-6),
        # Amplitude/phase controls (six species), FP32 gradient in amplitudes and phases.
        _phase("phase_grad", n=6, B=16, M=200, prec="fp32", grad=True),
        # Noisy-drive ensemble on ten qubits: <Z>(t) of every realisation, state only.
        _sim("ensemble_n1024", n=10, B=64, M=200, prec="fp32", want_U=False),
        # The same study on a small system with the final propagators, FP64.
        _sim("ensemble_small", n=4, B=100, M=500, prec="fp64", want_U=True),
        # State-to-state transfer on eight qubits, a few starting pulses at once.
        _state("state_transfer", n=8, B=8, M=80, prec="fp32"),
        # A tile of the noisy exotic freezing map: many short-register pulses, mean order parameter.
        _freeze("freezing_map", n=3, B=20000, M=1000, prec="fp32"),
        # One training step of the warm-start network at its configured widths.
        _mlp("warm_start_train", width=512, depth=3, outputs=5000, batch=1024),
    ]


def draw(rng):
    """One more case of the same ranges."""
    kind = rng.choices(["prop", "grad", "phase", "sim", "state", "freeze", "mlp"], [30, 28, 10, 12, 8, 6, 6])[0]
    while True:
        c = _draw(kind, rng)
        if c["kind"] == "mlp" or _seconds(c) < 0.05:
            return c


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw(kind, rng):
    ctl = rng.choice(["local", "local", "global"])
    if kind == "prop":
        n = rng.choice([2, 3, 3, 4, 5, 6, 6, 6, 7, 8])
        prec = rng.choice(["fp64", "fp32"] if n < 6 else ["fp64", "fp32", "fp16x3", "fp16x3"])
        levels = n <= 6 and rng.random() < 0.4
        M = _log(rng, 30, 2000 if n <= 6 else 200)
        if prec == "fp16x3":
            M = min(M, 300 if n > 6 else 1000 if not levels else 2000)
        return _prop(None, n=n, ctl=ctl, B=_log(rng, 1, 300), M=M, prec=prec, levels=levels,
                     reunit=_reunit(rng, prec, n, ctl, M), drift="pulse" if n <= 5 and rng.random() < 0.2 else "table",
                     strang=rng.random() < 0.1)
    if kind == "grad":
        n = rng.choice([2, 3, 4, 5, 5, 6, 7, 8])
        prec = rng.choice(["fp64", "fp32"] if n < 7 else ["fp32", "fp16x3", "fp16x3"])
        M = _log(rng, 30, 1000 if n < 7 else 200)
        ck = {"fp64": rng.choice([0, 0, 25]), "fp32": rng.choice([20, 50]), "fp16x3": 8}[prec]
        drift = "pulse" if n <= 5 and rng.random() < 0.3 else "table"
        return _grad(None, n=n, ctl=ctl, B=_log(rng, 1, 256 if n < 7 else 4), M=M, prec=prec, ck=ck,
                     reunit=0 if prec == "fp64" else ck, drift=drift,
                     target="near" if n >= 7 else rng.choice(["haar", "near", "rotations"]) if prec == "fp64" else "near",
                     dt=rng.choice([1e-6, 2e-6]))
    if kind == "phase":
        n = rng.choice([3, 4, 5, 6])
        grad = rng.random() < 0.5
        prec = rng.choice(["fp64", "fp32"] if grad or n < 6 else ["fp32", "fp16x3"])
        M = _log(rng, 30, 200 if grad else 1000)
        return _phase(None, n=n, B=_log(rng, 1, 64), M=M, prec=prec, grad=grad,
                      reunit=0 if grad or prec == "fp64" else 32)
    if kind == "sim":
        n = rng.choice([3, 4, 5, 6, 7, 8, 9, 10])
        prec = rng.choice(["fp64", "fp32"])
        U = n <= 8 and rng.random() < 0.4
        return _sim(None, n=n, B=_log(rng, 1, 200), M=_log(rng, 20, 1000 if n <= 6 else 200), prec=prec, want_U=U,
                    reunit=20 if U and prec == "fp32" else 0)
    if kind == "state":
        n = rng.choice([3, 5, 6, 7, 8, 9])
        prec = rng.choice(["fp64", "fp32"])
        return _state(None, n=n, B=_log(rng, 1, 160), M=_log(rng, 20, 300 if prec == "fp64" else 500 // n), prec=prec)
    if kind == "freeze":
        return _freeze(None, n=rng.choice([2, 3, 3, 4]), B=_log(rng, 50, 20000), M=_log(rng, 200, 1000),
                       prec=rng.choice(["fp64", "fp32", "fp32"]))
    return _mlp(None, width=rng.choice([64, 256, 512]), depth=rng.choice([2, 3]), outputs=rng.choice([100, 1000, 5000]),
                batch=_log(rng, 33, 4096))


def _reunit(rng, prec, n, ctl, M):
    if prec == "fp64":
        return 0
    if prec == "fp32" and M * (2 * n if ctl == "local" else 2) * 2 < 1500 and rng.random() < 0.5:
        return 0
    return rng.choice([20, 50, 64]) if n <= 6 else 20


def _seconds(c):
    """A rough cost, to keep drawn cases below the largest listed ones."""
    n, B, M, K = c["n"], c["B"], c["M"], c["K"]
    dense = 8.0 * 8 ** n
    rate = {"fp64": 0.5e12, "fp32": 1e13, "fp16x3": 2e14}[c["prec"]]
    if c["kind"] in ("sim", "state") and not c.get("want_U"):
        factor = 2.2e-5 * max(4.0 ** (n - 8), 0.1) if c["kind"] == "state" else 4e-6 * max(4.0 ** (n - 8), 1.0)
        return M * K * 2 * factor * (-(-B // 150) if c["kind"] == "state" else 1) * (3 if c["prec"] == "fp64" else 1)
    products = B * M * (K * (1 if c.get("levels") else c.get("digits", 2)) + 1)
    serial = 2e-6 * 16 * (1 + M * K / 500) * (10 if n > 6 else 1)
    return products * dense / rate * (4 if c["kind"] == "grad" or c.get("grad") else 1) + serial


# ---------------------------------------------------------------------------- cases
def _case(kind, name, **kw):
    c = dict(kind=kind, **kw)
    if name:
        c["name"] = name
    return c


def _controls(n, ctl):
    return {"local": 2 * n, "global": 2, "global_x": 1, "local_x": n}[ctl]


def _prop(name, n, ctl, B, M, prec, reunit=0, levels=False, drift="table", strang=False):
    return _case("prop", name, n=n, ctl=ctl, K=_controls(n, ctl), B=B, M=M, prec=prec, reunit=reunit, levels=levels,
                 drift=drift, strang=bool(strang and drift == "table"), dt=1e-6, digits=2,
                 target="haar" if prec == "fp64" or B > 100 else "near")


def _grad(name, n, ctl, B, M, prec, ck=0, reunit=0, drift="table", target="haar", dt=1e-6):
    return _case("grad", name, n=n, ctl=ctl, K=_controls(n, ctl), B=B, M=M, prec=prec, ck=ck, reunit=reunit,
                 drift=drift, target=target, dt=dt, digits=2)


def _phase(name, n, B, M, prec, grad, reunit=0):
    return _case("phase", name, n=n, ctl="local_x", K=n, B=B, M=M, prec=prec, grad=grad, reunit=reunit, dt=1e-6,
                 target="near", levels=prec == "fp16x3", digits=2)


def _sim(name, n, B, M, prec, want_U, reunit=0):
    return _case("sim", name, n=n, ctl="global_x", K=1, B=B, M=M, prec=prec, want_U=want_U, reunit=reunit, dt=1e-6,
                 digits=2)


def _state(name, n, B, M, prec):
    return _case("state", name, n=n, ctl="local", K=2 * n, B=B, M=M, prec=prec, dt=2e-6, target="near", digits=2)


def _freeze(name, n, B, M, prec):
    return _case("freeze", name, n=n, K=1, B=B, M=M, prec=prec, digits=2)


def _mlp(name, width, depth, outputs, batch):
    return _case("mlp", name, width=width, depth=depth, outputs=outputs, batch=batch)


# ---------------------------------------------------------------------------- the control problem
_X = np.array([[0, 1], [1, 0]], dtype=np.complex128) / 2
_Y = np.array([[0, -1j], [1j, 0]], dtype=np.complex128) / 2


def _one_qubit_terms(n, ctl):
    """h[k][i]: the 2 x 2 part of control k on qubit i (qubit 0 is the leading bit); H_k is their sum."""
    z = np.zeros((2, 2), dtype=np.complex128)
    if ctl == "global":
        return np.array([[_X] * n, [_Y] * n])
    if ctl == "global_x":
        return np.array([[_X] * n])
    rows = []
    for i in range(n):
        for s in ((_X, _Y) if ctl == "local" else (_X,)):
            rows.append([s if j == i else z for j in range(n)])
    return np.array(rows)


def _dense(h):
    """The N x N operators of one-qubit terms h [K][n][2][2]."""
    K, n = h.shape[:2]
    out = np.zeros((K, 2 ** n, 2 ** n), dtype=np.complex128)
    for k in range(K):
        for i in range(n):
            if np.any(h[k, i]):
                out[k] += np.kron(np.kron(np.eye(2 ** i), h[k, i]), np.eye(2 ** (n - 1 - i)))
    return out


def _z(n):
    """Signs of every basis state's qubits, [n][N]."""
    idx = np.arange(2 ** n)
    return np.stack([1.0 - 2.0 * ((idx >> (n - 1 - i)) & 1) for i in range(n)])


def _drift(rng, n, count, chain):
    """Diagonals of offsets nu ~ U[-5, 5] kHz and couplings J ~ U[-200, 200] Hz, [count][N], rad/s."""
    z = _z(n)
    h = math.pi * rng.uniform(-5e3, 5e3, size=(count, n)) @ z
    for i in range(n):
        for j in range(i + 1, n):
            if not chain or j == i + 1:
                h += (math.pi / 2) * rng.uniform(-200.0, 200.0, size=(count, 1)) * (z[i] * z[j])
    return h


def _problem(c, seed):
    """The arrays of a case's control problem: everything that both prepare() and exact() start from."""
    n, B, M, K = c["n"], c["B"], c["M"], c["K"]
    rng = np.random.default_rng(seed)
    g = torch.Generator(device="cuda").manual_seed(seed)
    p = dict(n=n, N=2 ** n, levels=64 ** 2, base=64)
    if c["kind"] == "freeze":
        # driven Ising chain in the basis where the x-magnetisation is diagonal
        h0, T = 5 * math.pi, 20 * math.pi * M / 1e4
        had = np.array([[1.0]])
        for _ in range(n):
            had = np.kron(had, np.array([[1, 1], [1, -1]]) / math.sqrt(2.0))
        zz = _z(n)
        p["H0"] = had @ np.diag(-h0 / 20 * sum(zz[i] * zz[i + 1] / 2 for i in range(n - 1))) @ had
        p["m"] = _z(n).sum(0) / 2
        p["Hk"] = np.diag(-p["m"])[None]
        p["dt"], p["base"], p["levels"] = T / M, 100, 100 ** 2
        p["lo"], p["hi"] = np.full(1, -h0), np.full(1, h0)
        om = torch.rand((B, 1), generator=g, device="cuda", dtype=torch.float64) * 24 + 1
        la = torch.rand((B, 1), generator=g, device="cuda", dtype=torch.float64)
        eta = torch.rand((B, M), generator=g, device="cuda", dtype=torch.float64) * 2 - 1
        t = (torch.arange(M, device="cuda", dtype=torch.float64) + 0.5) * p["dt"]
        p["u"] = (h0 * ((1 - la) * torch.cos(om * t) + la * eta))[:, :, None].contiguous()
        return p
    p["dt"] = c["dt"]
    p["h"] = _one_qubit_terms(n, c["ctl"])
    p["Hk"] = _dense(p["h"])
    p["drift"] = _drift(rng, n, B if c.get("drift") == "pulse" else 1, c["kind"] == "sim")
    p["H0"] = np.diag(p["drift"][0]) if c.get("drift") != "pulse" else np.zeros((2 ** n, 2 ** n))
    lo, hi = (0.0, OMEGA) if c["kind"] in ("sim", "phase") else (-OMEGA, OMEGA)
    p["lo"], p["hi"] = np.full(K, lo), np.full(K, hi)
    if c["kind"] == "sim":
        # Omega (1 + xi), xi stationary Ornstein-Uhlenbeck noise (sigma 0.1, correlation time 50 us)
        a = math.exp(-c["dt"] / 50e-6)
        w = torch.randn((B, M), generator=g, device="cuda", dtype=torch.float64)
        w[:, 1:] *= math.sqrt(1 - a * a)
        xi = torch.empty_like(w)
        x = torch.zeros_like(w[:, 0])
        for m in range(M):
            x = a * x + w[:, m]
            xi[:, m] = x
        p["u"] = (OMEGA / 2 * (1 + 0.1 * xi))[:, :, None].contiguous()
        p["psi0"] = torch.zeros(2 ** n, dtype=torch.complex128, device="cuda")
        p["psi0"][0] = 1
        p["obs"] = torch.as_tensor(_z(n)[0], device="cuda").contiguous()
        return p
    rand = torch.rand((B, M, K), generator=g, device="cuda", dtype=torch.float64)
    p["u"] = lo + (hi - lo) * rand
    if c["kind"] == "phase":
        p["phi"] = 2 * math.pi * torch.rand((B, M, K), generator=g, device="cuda", dtype=torch.float64)
    how = c.get("target", "haar")
    if how == "near":
        # where a pulse close by ends, as in the middle of an optimisation (F about 0.6)
        w = 2 * math.sqrt(0.5 / (K * M)) / c["dt"]
        near = p["u"] + w * torch.randn((B, M, K), generator=g, device="cuda", dtype=torch.float64)
        if c["kind"] == "state":
            v = rng.standard_normal((2, B, 2 ** n))
            v = torch.as_tensor(v[0] + 1j * v[1], device="cuda")
            p["psi0"] = v / torch.linalg.vector_norm(v, dim=-1, keepdim=True)
            p["psiT"] = _chain(p, c, near, p["psi0"][:, :, None])[:, :, 0].contiguous()
        elif c["kind"] == "prop" or not c.get("grad", True):
            p["target"] = _propagators(p, c, near[:1])[0].contiguous()     # these calls take one target
        else:
            p["target"] = _propagators(p, c, near).contiguous()
    elif how == "rotations":
        # exp(-i theta.sigma) on every qubit, one target per pulse
        ax = torch.as_tensor(rng.uniform(0.0, math.pi, size=(B, n, 3)), device="cuda")
        r = torch.linalg.vector_norm(ax, dim=-1, keepdim=True)
        x, y, w = (torch.sin(r) * ax / r).unbind(-1)
        cs = torch.cos(r)[..., 0]
        v = torch.stack([torch.complex(cs, -w), torch.complex(-y, -x), torch.complex(y, -x), torch.complex(cs, w)], -1)
        v = v.reshape(B, n, 2, 2)
        t = v[:, 0]
        for i in range(1, n):
            t = torch.einsum("bij,bkl->bikjl", t, v[:, i]).reshape(B, 2 ** (i + 1), 2 ** (i + 1))
        p["target"] = t
    else:
        q, r = np.linalg.qr(rng.standard_normal((2 ** n, 2 ** n)) + 1j * rng.standard_normal((2 ** n, 2 ** n)))
        d = np.diagonal(r)
        p["target"] = torch.as_tensor(q * (d / np.abs(d)), device="cuda")
    return p


# ---------------------------------------------------------------------------- what a user's program does
def prepare(case, seed):
    c = case
    if c["kind"] == "mlp":
        x, y, params, sizes = _mlp_arrays(c, seed)
        return dict(c=c, net=MLP(sizes, params=params.cpu().numpy()), x=x, y=y)
    p = _problem(c, seed)
    n, prec = c["n"], c["prec"]
    table = redo.Table(p["H0"], p["Hk"], p["dt"], p["lo"], p["hi"], p["base"], 2, fp32=prec == "fp32" or c["kind"] == "sim",
                       fp16x3=prec == "fp16x3", levels=c.get("levels", False), strang=c.get("strang", False))
    s = dict(c=c, table=table, **{k: p[k] for k in ("u", "target", "phi", "psi0", "psiT", "obs") if k in p})
    if c["kind"] == "phase":
        table.set_phase_axes(_z(n) / 2)
    if c.get("drift") == "pulse":
        s["drift"] = torch.as_tensor(p["drift"], device="cuda")
    if c["kind"] == "freeze":
        s["m"] = torch.as_tensor(p["m"], device="cuda")
    return s


def run(state):
    s = state
    c = s["c"]
    if c["kind"] == "mlp":
        loss = s["net"].train_step(s["x"], s["y"], 1e-3)
        return dict(loss=loss, grads=s["net"].grads, params=s["net"].params)
    t, prec = s["table"], c["prec"]
    q = t.quantize(s["u"])
    if c["kind"] == "prop":
        if "drift" in s:
            U, F, tau = t.propagate_drift(q, s["drift"], prec, target=s["target"], reunit_every=c["reunit"])
        else:
            U, F, tau = t.propagate(q, prec, target=s["target"], reunit_every=c["reunit"])
        return dict(q=q, **_width(prec, U=U, F=F, tau=tau))
    if c["kind"] == "grad":
        if "drift" in s:
            F, g = t.fidelity_grad_drift(q, s["drift"], s["target"], prec, c["ck"], reunit_every=c["reunit"])
        else:
            F, g = t.fidelity_grad(q, s["target"], prec, c["ck"], reunit_every=c["reunit"])
        return dict(q=q, **_width(prec, F=F, grad=g))
    if c["kind"] == "phase":
        if c["grad"]:
            F, ga, gp = t.fidelity_grad_phase(q, s["phi"], s["target"], prec)
            return dict(q=q, **_width(prec, F=F, grad_amp=ga, grad_phase=gp))
        U, F, tau = t.propagate_phase(q, s["phi"], prec, target=s["target"], reunit_every=c["reunit"])
        return dict(q=q, **_width(prec, U=U, F=F, tau=tau))
    if c["kind"] == "sim":
        e, U = t.simulate(q, s["psi0"], s["obs"], prec, c["reunit"], c["want_U"])
        return dict(q=q, **_width(prec, expect=e, U=U))
    if c["kind"] == "state":
        F, g = t.state_grad(q, s["psi0"], s["psiT"], prec)
        return dict(q=q, **_width(prec, F=F, grad=g))
    _, mean = t.expect_diag(q, s["m"], s["m"], prec, series=False)
    return dict(q=q, **_width(prec, mean=mean))


def _width(prec, **out):
    """Results at the width that their precision is good for."""
    out = {k: v for k, v in out.items() if v is not None}
    if prec == "fp64":
        return out
    return {k: v.to(torch.complex64 if v.is_complex() else torch.float32) for k, v in out.items()}


def work(case):
    """Bytes of inputs and outputs; operations of the problem itself: a step of these controls is a
    2 x 2 operator on every qubit and a diagonal, applied to every column that is carried."""
    c = case
    if c["kind"] == "mlp":
        sizes = _mlp_sizes(c)
        w = sum(a * b + b for a, b in zip(sizes[:-1], sizes[1:]))
        return dict(bytes=4.0 * (6 * w + c["batch"] * (sizes[0] + sizes[-1])), flops=6.0 * w * c["batch"])
    n, N, B, M, K = c["n"], 2.0 ** c["n"], c["B"], c["M"], c["K"]
    wide = 16 if c["prec"] == "fp64" else 8
    table = K * 128 * N * 2 * wide
    controls = B * M * K * (8 + 4)
    step = N * (16.0 * n + 8)                            # flops on one column
    if c["kind"] == "freeze":
        return dict(bytes=controls + B * wide / 2 + table, flops=B * M * N * N * (8.0 * N + 8 + 4))
    if c["kind"] == "sim":
        cols = 1 + (N if c["want_U"] else 0)
        return dict(bytes=controls + table + B * (M + 1) * wide / 2 + (B * N * N * wide if c["want_U"] else 0),
                    flops=B * M * (step * cols + 4 * N))
    cols = 1 if c["kind"] == "state" else N
    if c["kind"] == "prop" or (c["kind"] == "phase" and not c["grad"]):
        extra = B * M * K * 8 if c["kind"] == "phase" else 0
        return dict(bytes=controls + extra + table + (B + 1) * N * N * wide, flops=B * M * step * cols)
    grads = B * M * K * wide / 2 * (3 if c["kind"] == "phase" else 1)
    return dict(bytes=controls + table + grads + (B if c["kind"] != "state" else 2 * B / N) * N * N * wide,
                flops=3 * B * M * step * cols)


# ---------------------------------------------------------------------------- the same in plain 64-bit torch
def _levels(p, u):
    lo, hi = (torch.as_tensor(p[k], device="cuda") for k in ("lo", "hi"))
    delta = (hi - lo) / (p["levels"] - 1)
    q = torch.clamp(torch.round((u - lo) / delta), 0, p["levels"] - 1)
    return q.to(torch.int32), lo + q * delta


def _rotations(p, value, order=None):
    """(V, L): every step's 2 x 2 operator of every qubit, V [B][M][n][2][2], and (order given) the
    logarithmic derivatives dV/du_k V^-1, L [B][M][K][n][2][2]."""
    B, M, K = value.shape
    h = torch.as_tensor(p["h"], device="cuda")
    eye = torch.eye(2, dtype=torch.complex128, device="cuda")
    V = eye.expand(B, M, p["n"], 2, 2)
    done = []
    for k in range(K):
        # (2h)^2 = I where h is not zero: exp(-i a h) = cos(a/2) - i sin(a/2) 2h
        a = value[:, :, k, None, None, None] * p["dt"] / 2
        on = (h[k].abs().amax((-1, -2)) > 0)[:, None, None]
        E = torch.where(on, torch.cos(a) * eye - 2j * torch.sin(a) * h[k], eye.expand(B, M, p["n"], 2, 2))
        V = E @ V
        if order:
            done = [E @ x @ E.conj().transpose(-1, -2) for x in done]
            done.append((-1j * p["dt"] * h[k]).expand(B, M, p["n"], 2, 2))
    return V, (torch.stack(done, 2) if order else None)


def _apply(v, x):
    """Each qubit's operator v [B][n][2][2] on the rows of x [B][N][C]."""
    B, N, C = x.shape
    for i in range(v.shape[1]):
        x = x.reshape(B, 2 ** i, 2, -1)
        w = v[:, i, :, :, None, None]
        a, b = x[:, :, 0], x[:, :, 1]
        x = torch.stack([w[:, 0, 0] * a + w[:, 0, 1] * b, w[:, 1, 0] * a + w[:, 1, 1] * b], 2)
    return x.reshape(B, N, C)


def _phases(p, V, L=None):
    """Turn x rotations into rotations about the phases' axes; derivatives in amplitudes and phases."""
    s = torch.tensor([0.5, -0.5], dtype=torch.float64, device="cuda")
    z = torch.exp(-1j * p["phi"][..., None] * s)                        # [B][M][n][2]
    V = z[..., :, None] * V * z.conj()[..., None, :]
    if L is None:
        return V, None, None
    LA = z[:, :, None, :, :, None] * L * z.conj()[:, :, None, :, None, :]
    S = torch.diag(s).to(torch.complex128)
    LP = torch.zeros_like(L)
    for k in range(L.shape[2]):
        v = V[:, :, k]
        LP[:, :, k, k] = -1j * (S - v @ S @ v.conj().transpose(-1, -2))
    return V, LA, LP


def _diag(p, c, B):
    return torch.exp(-1j * p["dt"] * torch.as_tensor(p["drift"], device="cuda"))[:B].expand(B, -1)[:, :, None]


def _chain(p, c, u, x):
    """The pulses u applied to the columns x [B][N][C]."""
    V = _steps(p, c, u)
    D = _diag(p, c, u.shape[0])
    for m in range(u.shape[1]):
        x = _apply(V[:, m], D * x)
    return x


def _steps(p, c, u):
    V, _ = _rotations(p, _levels(p, u)[1])
    if c["kind"] == "phase":
        V, _, _ = _phases(dict(p, phi=p["phi"][:u.shape[0]]), V)
    return V


def _propagators(p, c, u):
    """Propagators of the pulses u: every step's N x N operator, multiplied pairwise."""
    V = _steps(p, c, u)
    B, M = V.shape[:2]
    out = []
    for b in range(B):
        S = V[b, :, 0]
        for i in range(1, p["n"]):
            S = torch.einsum("mij,mkl->mikjl", S, V[b, :, i]).reshape(M, 2 ** (i + 1), 2 ** (i + 1))
        S = S * _diag(p, c, B)[b, :, 0]
        if c.get("strang"):
            half = torch.exp(-0.5j * p["dt"] * torch.as_tensor(p["drift"][0], device="cuda"))
            S = half[:, None] * S * half.conj()
        while S.shape[0] > 1:
            last = S[S.shape[0] // 2 * 2:]
            S = torch.cat([S[1::2] @ S[:S.shape[0] // 2 * 2:2], last])
        out.append(S[0])
    return torch.stack(out)


def _overlap(target, U):
    return (target.conj() * U).sum((-1, -2))


def _reverse(p, V, D, x, y, tau, norm, Ls):
    """Gradients sum 2/norm Re(conj(tau) dtau) of tau = Tr(y^T x), undoing the chain from its end.
    x, y [B][N][C] (y holds the costate's transpose); Ls: lists of L [B][M][K][n][2][2]."""
    B, M, n = V.shape[:3]
    rho = torch.empty((B, M, n, 2, 2), dtype=torch.complex128, device="cuda")
    for m in range(M - 1, -1, -1):
        for i in range(n):
            X, Yv = x.reshape(B, 2 ** i, 2, -1), y.reshape(B, 2 ** i, 2, -1)
            for a in range(2):
                for b in range(2):
                    rho[:, m, i, a, b] = (X[:, :, a] * Yv[:, :, b]).sum((1, 2))
        x = D.conj() * _apply(V[:, m].conj().transpose(-1, -2), x)
        y = D * _apply(V[:, m].transpose(-1, -2), y)
    return [2.0 / norm * torch.real(tau.conj()[:, None, None] * torch.einsum("bmkiac,bmica->bmk", L, rho)) for L in Ls]


def exact(case, seed):
    c = case
    if c["kind"] == "mlp":
        return _mlp_exact(c, seed)
    p = _problem(c, seed)
    B, M, N = c["B"], c["M"], p["N"]
    q, value = _levels(p, p["u"])
    if c["kind"] == "freeze":
        D = torch.linalg.matrix_exp(torch.as_tensor(-1j * p["dt"] * p["H0"], device="cuda"))
        m = torch.as_tensor(p["m"], device="cuda")
        U = torch.eye(N, dtype=torch.complex128, device="cuda").expand(B, N, N)
        mean = torch.zeros(B, dtype=torch.float64, device="cuda")
        for k in range(M):
            U = torch.exp(1j * p["dt"] * value[:, k] * m)[:, :, None] * (D @ U.transpose(0, 1).reshape(N, -1)).reshape(
                N, B, N).transpose(0, 1)
            mean += ((U.real ** 2 + U.imag ** 2) * m[:, None] * m).sum((1, 2))
        return dict(q=q, mean=mean / M)
    if c["kind"] == "sim":
        V, _ = _rotations(p, value)
        D = _diag(p, c, B)
        x = p["psi0"][:, None].expand(B, N, 1)
        if c["want_U"]:
            x = torch.cat([x, torch.eye(N, dtype=torch.complex128, device="cuda").expand(B, N, N)], 2)
        e = [(x[:, :, 0].abs() ** 2 @ p["obs"])]
        for m in range(M):
            x = _apply(V[:, m], D * x)
            e.append(x[:, :, 0].abs() ** 2 @ p["obs"])
        return dict(q=q, expect=torch.stack(e, 1), **({"U": x[:, :, 1:]} if c["want_U"] else {}))
    D = _diag(p, c, B)
    V, L = _rotations(p, value, order=c["kind"] in ("grad", "state") or c.get("grad"))
    Ls = [L]
    if c["kind"] == "phase":
        V, *Ls = _phases(p, V, L)
    x = p["psi0"][:, :, None] if c["kind"] == "state" else torch.eye(N, dtype=torch.complex128, device="cuda").expand(B, N, N)
    for m in range(M):
        x = _apply(V[:, m], D * x)
    if c["kind"] == "state":
        y = p["psiT"].conj()[:, :, None]
        tau = (y * x).sum((1, 2))
        return dict(q=q, F=tau.abs() ** 2, grad=_reverse(p, V, D, x, y, tau, 1.0, Ls)[0])
    if c.get("strang"):
        half = torch.exp(-0.5j * p["dt"] * torch.as_tensor(p["drift"], device="cuda"))
        x = half[:, :, None] * x * half.conj()[:, None, :]
    tau = _overlap(p["target"], x)
    F = tau.abs() ** 2 / N ** 2
    if c["kind"] == "prop" or not (c["kind"] == "grad" or c["grad"]):
        return dict(q=q, U=x, F=F, tau=tau)
    # tau = Tr(U_T^dag U): the costate's transpose at the end of the chain is conj(U_T)
    y = p["target"].conj().expand(B, N, N)
    g = _reverse(p, V, D, x, y, tau, float(N) ** 2, Ls)
    if c["kind"] == "phase":
        return dict(q=q, F=F, grad_amp=g[0], grad_phase=g[1])
    return dict(q=q, F=F, grad=g[0])


# ---------------------------------------------------------------------------- warm-start network
def _mlp_sizes(c):
    return [23] + [c["width"]] * c["depth"] + [c["outputs"]]


def _mlp_arrays(c, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    sizes = _mlp_sizes(c)
    parts = []
    for a, b in zip(sizes[:-1], sizes[1:]):
        parts += [(torch.rand(a * b, generator=g, device="cuda") * 2 - 1) / math.sqrt(a), torch.zeros(b, device="cuda")]
    x = torch.rand((c["batch"], sizes[0]), generator=g, device="cuda") * 2 - 1
    y = torch.rand((c["batch"], sizes[-1]), generator=g, device="cuda") * 2 - 1
    return x, y, torch.cat(parts), sizes


def _mlp_exact(c, seed):
    x, y, flat, sizes = _mlp_arrays(c, seed)
    flat = flat.double().requires_grad_(True)
    h, at = x.double(), 0
    for i, (a, b) in enumerate(zip(sizes[:-1], sizes[1:])):
        z = h @ flat[at:at + a * b].reshape(b, a).T + flat[at + a * b:at + a * b + b]
        at += a * b + b
        h = torch.nn.functional.gelu(z) if i + 2 < len(sizes) else torch.tanh(z)
    loss = ((h - y.double()) ** 2).mean()
    loss.backward()
    g = flat.grad
    new = flat.detach() - 1e-3 * g / (g.abs() + 1e-8)
    return dict(loss=loss.detach(), grads=g, params=new)
