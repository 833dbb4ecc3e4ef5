"""Performance cases of the propagator: the calls a user of the library makes, timed through its public entry points.

Four families, each over the range of sizes it is used at:

* ``propagate``  -- U(T) of one driven system (``Propagator.set_controls`` + ``propagate``): a control loop sends new
  samples and reads the gate;
* ``gradient``   -- gate infidelity and its gradient for every control sample (``propagate_grad``): one step of a
  gradient-based pulse optimisation (GRAPE);
* ``trajectory`` -- a state at intermediate times (``propagate_trajectory`` with ``psi0``): populations along a pulse;
* ``batched``    -- many independent instances of uneven dimension and length in one launch (``propagate_batched``):
  parameter sweeps and pulse populations.

Precisions follow use: FP64 is the library's default; FP32 is taken where single precision keeps its digits (the
error grows with the number of slices, so its runs are shorter); 3xTF32 is the tensor-core option for dense systems.
"""

import math

import numpy as np
import torch

from paper_2108_07126_gb300.binding import Propagator

TWO_PI = 2.0 * math.pi

SX = np.array([[0, 1], [1, 0]], dtype=np.complex128)
SY = np.array([[0, -1j], [1j, 0]], dtype=np.complex128)
SZ = np.array([[1, 0], [0, -1]], dtype=np.complex128)


def listed():
    return [
        # a short composite pulse on one qubit (two quadratures, fourth-order Magnus): the smallest call, all latency
        {"name": "qubit_pulse_fp64", "family": "propagate", "system": "qubits", "d": 2, "K": 2, "N": 128,
         "integrator": "magnus4_gl2", "prec": "fp64"},
        # the driven two-level system over 1 us in 2^14 midpoint steps: the library's first example
        {"name": "rabi_fp64", "family": "propagate", "system": "rabi", "d": 2, "K": 1, "N": 16384,
         "integrator": "midpoint", "prec": "fp64"},
        # four coupled spins, eight controls, fourth-order Magnus: a long run at the default precision
        {"name": "spins_d16_fp64", "family": "propagate", "system": "qubits", "d": 16, "K": 8, "N": 131072,
         "integrator": "magnus4_gl2", "prec": "fp64"},
        # the same system in single precision, at a length where single precision holds
        {"name": "spins_d16_fp32", "family": "propagate", "system": "qubits", "d": 16, "K": 8, "N": 2048,
         "integrator": "magnus4_gl2", "prec": "fp32"},
        # pulse optimisation on three qubits, 65536 piecewise-constant amplitudes: the gradient workload
        {"name": "grad_d8_fp64", "family": "gradient", "system": "qubits", "d": 8, "K": 6, "N": 65536,
         "integrator": "midpoint", "prec": "fp64"},
        # one step of an interactive optimisation: a short pulse in single precision, odd length
        {"name": "grad_d8_fp32", "family": "gradient", "system": "qubits", "d": 8, "K": 6, "N": 1501,
         "integrator": "midpoint", "prec": "fp32"},
        # gradient of a dense model truncated to an odd dimension, fourth-order Magnus
        {"name": "grad_d23_fp64", "family": "gradient", "system": "dense", "d": 23, "K": 2, "N": 1000,
         "integrator": "magnus4_gl2", "prec": "fp64"},
        # populations along a pulse: every 64th state of a dense model truncated to 12 levels
        {"name": "states_d12_fp64", "family": "trajectory", "system": "dense", "d": 12, "K": 3, "N": 20000,
         "integrator": "magnus4_simpson", "prec": "fp64", "every": 64},
        # a sweep over 64 instances, d = 2..64, in one launch
        {"name": "sweep64_fp32", "family": "batched", "d": 64, "n_inst": 64, "n_min": 100, "n_max": 1500,
         "integrator": "midpoint", "prec": "fp32"},
        # a dense 40-level model at the default precision (the run time against N of the paper's Sec. 5)
        {"name": "dense_d40_fp64", "family": "propagate", "system": "dense", "d": 40, "K": 2, "N": 4000,
         "integrator": "midpoint", "prec": "fp64"},
        # the dense stress system at the default precision
        {"name": "dense_d128_fp64", "family": "propagate", "system": "dense", "d": 128, "K": 4, "N": 608,
         "integrator": "magnus4_gl2", "prec": "fp64"},
        # the dense stress system on the tensor cores
        {"name": "dense_d128_tf32x3", "family": "propagate", "system": "dense", "d": 128, "K": 4, "N": 2048,
         "integrator": "magnus4_gl2", "prec": "fp32_tc_tf32x3"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.randrange(9)
    integ = rng.choice(["midpoint", "magnus4_gl2", "magnus4_simpson"])
    if kind == 0:  # one qubit or a qutrit-like few-level system, any length
        d = rng.choice([2, 2, 3, 4])
        return {"family": "propagate", "system": "dense", "d": d, "K": rng.randint(1, 3), "N": _log(rng, 64, 100000),
                "integrator": integ, "prec": "fp64"}
    if kind == 1:  # spins at the default precision
        q = rng.choice([3, 4])
        return {"family": "propagate", "system": "qubits", "d": 2 ** q, "K": 2 * q, "N": _log(rng, 500, 131072),
                "integrator": integ, "prec": "fp64"}
    if kind == 2:  # small systems in single precision
        return {"family": "propagate", "system": "dense", "d": rng.randint(2, 16), "K": rng.randint(1, 6),
                "N": _log(rng, 100, 1500), "integrator": integ, "prec": "fp32"}
    if kind == 3:  # optimisation steps, small systems
        q = rng.choice([1, 2, 3, 4])
        prec = rng.choice(["fp64", "fp32"])
        return {"family": "gradient", "system": "qubits", "d": 2 ** q, "K": 2 * q,
                "N": _log(rng, 100, 1500) if prec == "fp32" else _log(rng, 100, 30000 if q < 4 else 4000),
                "integrator": rng.choice(["midpoint", "magnus4_gl2"]), "prec": prec}
    if kind == 4:  # optimisation steps, dense models
        return {"family": "gradient", "system": "dense", "d": rng.randint(17, 32), "K": rng.randint(1, 3),
                "N": _log(rng, 50, 1000), "integrator": rng.choice(["midpoint", "magnus4_gl2"]), "prec": "fp64"}
    if kind == 5:  # states along a pulse
        return {"family": "trajectory", "system": "dense", "d": rng.randint(2, 16), "K": rng.randint(1, 4),
                "N": _log(rng, 200, 40000), "integrator": integ, "prec": "fp64", "every": _log(rng, 8, 200)}
    if kind == 6:  # sweeps
        return {"family": "batched", "d": rng.choice([16, 32, 64]), "n_inst": rng.randint(12, 64), "n_min": 100,
                "n_max": _log(rng, 300, 1500), "integrator": rng.choice(["midpoint", "magnus4_gl2"]), "prec": "fp32"}
    if kind == 7:  # dense models at the default precision
        d = rng.randint(17, 128)
        cap = 4000 if d <= 64 else 608
        return {"family": "propagate", "system": "dense", "d": d, "K": rng.randint(1, 4), "N": _log(rng, 60, cap),
                "integrator": integ, "prec": "fp64"}
    # dense models on the tensor cores
    return {"family": "propagate", "system": "dense", "d": rng.randint(65, 128), "K": rng.randint(1, 4),
            "N": _log(rng, 60, 2048), "integrator": integ, "prec": "fp32_tc_tf32x3"}


# ---------------------------------------------------------------- inputs


def _samples(N, integrator):
    return {"midpoint": N, "magnus4_gl2": 2 * N, "magnus4_simpson": 2 * N + 1}[integrator]


def _times(N, dt, integrator):
    j = np.arange(N, dtype=np.float64)
    if integrator == "midpoint":
        return (j + 0.5) * dt
    if integrator == "magnus4_gl2":
        off = math.sqrt(3.0) / 6.0
        return np.stack([(j + 0.5 - off) * dt, (j + 0.5 + off) * dt], 1).reshape(-1)
    return np.arange(2 * N + 1, dtype=np.float64) * (0.5 * dt)


def _embed(op, site, n):
    out = np.ones((1, 1), dtype=np.complex128)
    for s in range(n):
        out = np.kron(out, op if s == site else np.eye(2))
    return out


def _gue(rng, d, norm):
    A = rng.standard_normal((d, d)) + 1j * rng.standard_normal((d, d))
    H = 0.5 * (A + A.conj().T)
    return H * (norm / np.max(np.abs(np.linalg.eigvalsh(H))))


def _haar(rng, d):
    Q, R = np.linalg.qr(rng.standard_normal((d, d)) + 1j * rng.standard_normal((d, d)))
    ph = np.diag(R) / np.abs(np.diag(R))
    return Q * ph[None, :]


def _modes(rng, K, t, amp, n_modes=8):
    """K smooth pulses: sums of Fourier modes of the run's length with normal amplitudes."""
    T = max(float(t[-1]), 1e-9) * 1.01
    tt = torch.as_tensor(t, device="cuda")
    m = torch.arange(1, n_modes + 1, dtype=torch.float64, device="cuda")
    a = torch.as_tensor(rng.normal(0.0, amp, (K, n_modes)), device="cuda")
    ph = torch.as_tensor(rng.uniform(0.0, TWO_PI, (K, n_modes)), device="cuda")
    c = torch.zeros(K, t.size, dtype=torch.float64, device="cuda")
    for i in range(n_modes):
        c += a[:, i:i + 1] * torch.sin(TWO_PI * m[i] * tt[None] / T + ph[:, i:i + 1])
    return c


def _problem(case, seed):
    """(H0, Hk, c, dt) of one system, double precision; c on the GPU."""
    rng = np.random.default_rng([int(seed), int(case["d"]), int(case["N"])])
    d, K, N, integ = case["d"], case["K"], case["N"], case["integrator"]
    if case["system"] == "rabi":
        # resonant drive: 1 GHz splitting, 10 MHz Rabi frequency with a random phase, 1 us
        dt = 1000.0 / N
        t = _times(N, dt, integ)
        c = 0.01 * TWO_PI * np.cos(TWO_PI * t + rng.uniform(0.0, TWO_PI))
        return 0.5 * TWO_PI * SZ, SX[None].copy(), torch.as_tensor(c[None], device="cuda"), dt
    if case["system"] == "qubits":
        q = int(round(math.log2(d)))
        if case["family"] == "gradient":
            # rotating frame, piecewise-constant amplitudes of 20 MHz, 1 ns steps
            w, J, dt = rng.uniform(-5e-3, 5e-3, q), rng.uniform(1e-3, 10e-3, max(q - 1, 1)), 1.0
        else:
            # laboratory frame, 10 ps steps
            w, J, dt = rng.uniform(0.5, 1.5, q), rng.uniform(1e-3, 10e-3, max(q - 1, 1)), 0.01
        H0 = sum(0.5 * TWO_PI * w[i] * _embed(SZ, i, q) for i in range(q))
        for i in range(q - 1):
            H0 = H0 + (TWO_PI * J[i] / 4.0) * _embed(SZ, i, q) @ _embed(SZ, i + 1, q)
        Hk = np.stack([_embed(op, i, q) for i in range(q) for op in (SX, SY)])[:K]
        S = _samples(N, integ)
        if case["family"] == "gradient":
            c = torch.as_tensor(rng.normal(0.0, TWO_PI * 0.02, (K, S)), device="cuda")
        else:
            t = torch.as_tensor(_times(N, dt, integ), device="cuda")
            c = torch.zeros(K, S, dtype=torch.float64, device="cuda")
            for k in range(K):
                for _ in range(3):
                    f = w[k // 2] * (1.0 + rng.uniform(-0.05, 0.05))
                    c[k] += rng.uniform(0.0, TWO_PI * 0.01) * torch.sin(TWO_PI * f * t + rng.uniform(0.0, TWO_PI))
        return H0, Hk, c, dt
    # dense: GUE drift of 100 MHz, GUE controls, smooth pulses of 10 MHz, ||H0|| dt = 0.2
    H0 = _gue(rng, d, TWO_PI * 0.1)
    Hk = np.stack([_gue(rng, d, 1.0) for _ in range(K)])
    dt = 0.2 / (TWO_PI * 0.1)
    return H0, Hk, _modes(rng, K, _times(N, dt, integ), TWO_PI * 0.01), dt


def _batch(case, seed):
    """The instances of a sweep: d in {2, 4, .., d}, N log-uniform, 2 to 6 controls."""
    rng = np.random.default_rng([int(seed), int(case["n_inst"]), int(case["n_max"])])
    dims = [x for x in (2, 4, 8, 16, 32, 64) if x <= case["d"]]
    dt = 0.2 / TWO_PI
    out = []
    for i in range(case["n_inst"]):
        d = dims[i % len(dims)]
        N = int(round(math.exp(rng.uniform(math.log(case["n_min"]), math.log(case["n_max"])))))
        K = int(rng.integers(2, 7))
        H0 = _gue(rng, d, TWO_PI)
        Hk = np.stack([_gue(rng, d, 1.0) for _ in range(K)])
        c = rng.normal(0.0, TWO_PI * 0.02, (K, _samples(N, case["integrator"])))
        out.append((H0, Hk, c, dt, N))
    return out


def _types(prec):
    return (torch.complex128, torch.float64) if prec == "fp64" else (torch.complex64, torch.float32)


def _rounded(H0, Hk, c, prec):
    """The inputs as the call sees them (complex64 / float32 below double precision)."""
    ct, rt = _types(prec)
    return torch.as_tensor(H0).to(ct), torch.as_tensor(Hk).to(ct), torch.as_tensor(c).to(rt)


def prepare(case, seed):
    prec = case["prec"]
    prop = Propagator(0)
    if case["family"] == "batched":
        inst, keep, outs = prop.batch(_batch(case, seed), prec, case["integrator"])
        return {"case": case, "prop": prop, "inst": inst, "keep": keep, "outs": outs}
    H0, Hk, c, dt = _problem(case, seed)
    H0, Hk, c = _rounded(H0, Hk, c, prec)
    prop.set_hamiltonians(H0, Hk, case["integrator"])
    state = {"case": case, "prop": prop, "c": c.cuda(), "dt": dt}
    rng = np.random.default_rng([int(seed), 7])
    if case["family"] == "gradient":
        state["V"] = torch.as_tensor(_haar(rng, case["d"])).to(_types(prec)[0]).cuda()
    if case["family"] == "trajectory":
        psi = rng.standard_normal(case["d"]) + 1j * rng.standard_normal(case["d"])
        state["psi0"] = torch.as_tensor(psi / np.linalg.norm(psi)).to(_types(prec)[0]).cuda()
    return state


def run(state):
    case, prop = state["case"], state["prop"]
    if case["family"] == "batched":
        prop.propagate_batched(state["inst"], case["prec"], case["integrator"])
        return state["outs"]
    prop.set_controls(state["c"], state["dt"], case["N"])
    if case["family"] == "gradient":
        loss, grad = prop.propagate_grad(state["V"], case["prec"])
        return {"loss": loss, "grad": grad}
    if case["family"] == "trajectory":
        return prop.propagate_trajectory(case["prec"], case["every"], state["psi0"])
    return prop.propagate(case["prec"])


# ---------------------------------------------------------------- work


def _basis(K, integrator):
    return 1 + K if integrator == "midpoint" else 1 + 2 * K + K * (K - 1) // 2


def _slices_work(d, K, N, integrator, prec, products):
    """One pass over N slices: samples in, Hamiltonians in, U out; per slice the exponent from its basis and
    `products` complex products (a polynomial of the exponential of a small exponent takes four, the chain one)."""
    ce, re = (16, 8) if prec == "fp64" else (8, 4)
    return {"bytes": K * _samples(N, integrator) * re + (2 + K) * d * d * ce,
            "flops": float(N) * (products * 8 * d ** 3 + 2 * _basis(K, integrator) * d * d)}


def work(case):
    integ, prec = case["integrator"], case["prec"]
    if case["family"] == "batched":
        w = {"bytes": 0, "flops": 0.0}
        for H0, Hk, c, dt, N in _batch(case, 1):
            x = _slices_work(H0.shape[0], Hk.shape[0], N, integ, prec, 5)
            w = {k: w[k] + x[k] for k in w}
        return w
    d, K, N = case["d"], case["K"], case["N"]
    if case["family"] == "gradient":
        # forward chain, adjoint chain and Frechet derivative (three times the products of the exponential)
        w = _slices_work(d, K, N, integ, prec, 5 + 2 + 12)
        w["bytes"] += K * _samples(N, integ) * (8 if prec == "fp64" else 4)
        return w
    w = _slices_work(d, K, N, integ, prec, 5)
    if case["family"] == "trajectory":
        w["bytes"] += -(-N // case["every"]) * d * (16 if prec == "fp64" else 8)
    return w


# ---------------------------------------------------------------- 64-bit reference (plain torch)


def _exponents(H0, Hk, c, dt, integ):
    """Hermitian G_j of slices with samples c: (n, d, d)."""
    def ham(x):  # (K, n) -> (n, d, d)
        return H0[None] + torch.einsum("kn,kab->nab", x.to(H0.dtype), Hk)

    def comm(A, B):
        return A @ B - B @ A

    if integ == "midpoint":
        return dt * ham(c)
    if integ == "magnus4_gl2":
        A, B = ham(c[:, 0::2]), ham(c[:, 1::2])
        return 0.5 * dt * (A + B) + 1j * (math.sqrt(3.0) * dt * dt / 12.0) * comm(A, B)
    A, M, B = ham(c[:, 0:-1:2]), ham(c[:, 1::2]), ham(c[:, 2::2])
    return (dt / 6.0) * (A + 4.0 * M + B) + 1j * (dt * dt / 12.0) * comm(A, B)


def _expm(G):
    """exp(-i G) by a degree-18 Taylor polynomial and squarings."""
    bound = float(torch.linalg.matrix_norm(G.detach(), ord=1).max())
    s = max(0, math.ceil(math.log2(max(bound, 1e-300) / 0.5)))
    X = -1j * G / 2.0 ** s
    eye = torch.eye(G.shape[-1], dtype=G.dtype, device=G.device)
    T = eye + X / 18.0
    for k in range(17, 0, -1):
        T = eye + (X @ T) / k
    for _ in range(s):
        T = T @ T
    return T


def _tree(U):
    while U.shape[0] > 1:
        n = U.shape[0]
        P = U[1:n - n % 2:2] @ U[0:n - n % 2:2]
        U = torch.cat([P, U[n - 1:]]) if n % 2 else P
    return U[0]


def _chunks(c, N, integ, n):
    """Samples of slices [a, b) for consecutive ranges of n slices."""
    for a in range(0, N, n):
        b = min(N, a + n)
        if integ == "midpoint":
            yield c[:, a:b]
        elif integ == "magnus4_gl2":
            yield c[:, 2 * a:2 * b]
        else:
            yield c[:, 2 * a:2 * b + 1]


def _exact_u(H0, Hk, c, dt, N, integ):
    n = max(1, (1 << 24) // (H0.shape[0] ** 2))
    return _tree(torch.stack([_tree(_expm(_exponents(H0, Hk, x, dt, integ))) for x in _chunks(c, N, integ, n)]))


def exact(case, seed):
    integ, prec = case["integrator"], case["prec"]

    def wide(H0, Hk, c):
        a, b, x = _rounded(H0, Hk, c, prec)
        return a.to(torch.complex128).cuda(), b.to(torch.complex128).cuda(), x.double().cuda()

    if case["family"] == "batched":
        out = []
        for H0, Hk, c, dt, N in _batch(case, seed):
            h, k, x = wide(H0, Hk, c)
            out.append(_exact_u(h, k, x, dt, N, integ))
        return out
    H0, Hk, c, dt = _problem(case, seed)
    h, k, x = wide(H0, Hk, c)
    N, d = case["N"], case["d"]
    rng = np.random.default_rng([int(seed), 7])
    if case["family"] == "propagate":
        return _exact_u(h, k, x, dt, N, integ)
    if case["family"] == "gradient":
        V = torch.as_tensor(_haar(rng, d)).to(_types(prec)[0]).to(torch.complex128).cuda()
        x.requires_grad_(True)
        U = _tree(_expm(_exponents(h, k, x, dt, integ)))
        loss = 1.0 - torch.abs(torch.trace(V.conj().T @ U)) ** 2 / d ** 2
        loss.backward()
        return {"loss": float(loss.detach()), "grad": x.grad}
    psi = rng.standard_normal(d) + 1j * rng.standard_normal(d)
    psi = torch.as_tensor(psi / np.linalg.norm(psi)).to(_types(prec)[0]).to(torch.complex128).cuda()
    out = []
    for y in _chunks(x, N, integ, case["every"]):
        psi = _tree(_expm(_exponents(h, k, y, dt, integ))) @ psi
        out.append(psi)
    return torch.stack(out)
