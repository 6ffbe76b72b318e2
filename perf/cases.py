"""The work whose speed this library answers for, as cases that can be timed.

A case is one call (or one short run of calls) of the public interface on inputs a user's
program would have in hand: single gates, whole circuits launched gate by gate, fused or
compiled, the <Z_i> readout, gradients, one training step through torch autograd, and a batch
of small circuits. Sizes and circuit families are those of ``workloads``, the tests and the
benchmark: 12-qubit exact circuits, 20- to 30-qubit states, complex64 and complex128.

What a case fixes is the program: qubit count, precision, circuit structure. What a seed makes
are its inputs: amplitudes, gate matrices and angles. (A compiled pass is kept by a circuit's
structure, so a program that calls one circuit with new matrices compiles it once.)

Numbers that are computed from complex64 amplitudes (energies, gradients) are returned as
float32, whose precision they have; from complex128 amplitudes as float64.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2411_18354_gb300 as qs
import workloads as W
from paper_2411_18354_gb300.autograd import AdjointEnergy

FLAGS = {
    "unfused": 0,
    "fused": qs.QS_FLAG_FUSE,
    "compiled": qs.QS_FLAG_FUSE | qs.QS_FLAG_JIT,
}
TORCH = {"c64": torch.complex64, "c128": torch.complex128}
REAL = {"c64": torch.float32, "c128": torch.float64}
AMP = {"c64": 8, "c128": 16}


def listed():
    return [
        # A small exact simulation: 212 gates on 12 qubits, the whole state in one tile. Latency of one call.
        {"name": "small_n12_c64", "path": "circuit", "circuit": "random", "n": 12, "dtype": "c64", "mode": "fused",
         "count": 212, "cmax": 3, "perm": 0.0, "structure": 0},
        # Gates applied one call at a time to a state that fits the L2 (an interactive or a host-driven program).
        {"name": "gates_n20_c64", "path": "gates", "n": 20, "dtype": "c64", "count": 27, "cmax": 8, "structure": 1},
        # The single-gate sweep at scale, 0-8 controls, targets low, middle and high: the benchmark's headline.
        {"name": "gates_n30_c64", "path": "gates", "n": 30, "dtype": "c64", "count": 27, "cmax": 8, "structure": 1},
        # The same sweep in double precision.
        {"name": "gates_n28_c128", "path": "gates", "n": 28, "dtype": "c128", "count": 27, "cmax": 8, "structure": 1},
        # The 1000-gate random circuit at scale, fused into compiled passes.
        {"name": "random_n28_c64_compiled", "path": "circuit", "circuit": "random", "n": 28, "dtype": "c64",
         "mode": "compiled", "count": 1000, "cmax": 8, "perm": 0.0, "structure": 1},
        # The precision circuit: double precision, a quarter of the gates X / CNOT / Toffoli.
        {"name": "precision_n27_c128", "path": "circuit", "circuit": "random", "n": 27, "dtype": "c128",
         "mode": "fused", "count": 300, "cmax": 6, "perm": 0.25, "structure": 2},
        # The paper's QFT at its own size.
        {"name": "qft_n29_c64_compiled", "path": "circuit", "circuit": "qft", "n": 29, "dtype": "c64",
         "mode": "compiled", "structure": 0},
        # Reading out all <Z_i> and the norm of a double-precision state.
        {"name": "expect_n28_c128", "path": "expect", "n": 28, "dtype": "c128"},
        # One optimisation step of a small variational circuit, through torch autograd.
        {"name": "train_n14_c64", "path": "train", "n": 14, "dtype": "c64", "mode": "compiled", "layers": 4},
        # The gradient benchmark: 24 qubits, 20 layers, 960 parameters.
        {"name": "grad_n24_c64_compiled", "path": "grad", "n": 24, "dtype": "c64", "mode": "compiled", "layers": 20},
        # A reference gradient in double precision.
        {"name": "grad_n20_c128_fused", "path": "grad", "n": 20, "dtype": "c128", "mode": "fused", "layers": 8},
        # Many small circuits at once: energies and gradients of 512 ansatz states.
        {"name": "batch_512_c64_compiled", "path": "batch", "dtype": "c64", "mode": "compiled", "states": 512,
         "nmin": 10, "nmax": 18, "layers": 8, "structure": 4},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["gates", "gates", "circuit", "circuit", "expect", "train", "grad", "batch"])
    dt = rng.choice(["c64", "c128"])
    st = rng.randrange(1, 1 << 16)
    if path == "gates":
        return {"path": path, "n": rng.randint(10, 30 if dt == "c64" else 28), "dtype": dt, "count": 27,
                "cmax": rng.randint(0, 8), "structure": st}
    if path == "circuit":
        kind = rng.choice(["random", "random", "qft", "ansatz"])
        mode = rng.choice(["unfused", "fused", "compiled"])
        case = {"path": path, "circuit": kind, "n": rng.randint(10, 26 if dt == "c64" else 24), "dtype": dt,
                "mode": mode, "structure": st}
        if kind == "random":
            case.update(count=_log(rng, 30, 400), cmax=rng.randint(0, 8), perm=rng.choice([0.0, 0.25]))
        if kind == "ansatz":
            case.update(layers=rng.randint(1, 8))
        return case
    if path == "expect":
        return {"path": path, "n": rng.randint(10, 30 if dt == "c64" else 28), "dtype": dt}
    mode = rng.choice(["unfused", "fused", "compiled"])
    if path == "train":
        return {"path": path, "n": rng.randint(6, 18), "dtype": dt, "mode": mode, "layers": rng.randint(1, 6)}
    if path == "grad":
        return {"path": path, "n": rng.randint(8, 22 if dt == "c64" else 19), "dtype": dt, "mode": mode,
                "layers": rng.randint(1, 8)}
    nmin = rng.randint(4, 14)
    return {"path": path, "dtype": "c64", "mode": rng.choice(["fused", "compiled"]), "states": _log(rng, 8, 256),
            "nmin": nmin, "nmax": rng.randint(nmin, 16), "layers": rng.randint(1, 8), "structure": st}


# ---------------------------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------------------------


def _amplitudes(case, seed, biased=False):
    """A normalised random state as a CUDA tensor. ``biased``: each qubit leans to |0> or |1> (a
    state near a computational one, as a readout meets it), else complex Gaussian."""
    n = case["n"]
    g = torch.Generator(device="cuda").manual_seed(1 + seed)
    v = torch.randn(1 << n, 2, dtype=REAL[case["dtype"]], device="cuda", generator=g)
    if biased:
        w = np.random.default_rng([seed, 5]).uniform(0.3, 1.0, size=n)
        for q in range(n):
            v.view(-1, 2, 2 << q)[:, int(w[q] * 1e6) & 1].mul_(float(w[q]))
    v.mul_(1.0 / float(torch.linalg.vector_norm(v)))
    return torch.view_as_complex(v)


def _random_gates(case, seed):
    """Targets and controls from the case, a Haar matrix for each general gate from the seed."""
    n = case["n"]
    gates = W.random_circuit(n, case["count"], case["cmax"], case["structure"], perm_fraction=case["perm"])
    rng = np.random.default_rng([seed, 1])
    for i in range(len(gates)):
        if gates["kind"][i] == W.KIND_U:
            gates["U"][i] = W.pack_u(W.haar_2x2(rng))
    return gates


def _sweep_gates(case, seed):
    """``count`` gates as (target, control mask, matrix): 0..cmax controls in turn, targets low,
    middle and high."""
    n = case["n"]
    where = np.random.default_rng(case["structure"])
    rng = np.random.default_rng([seed, 2])
    out = []
    for i in range(case["count"]):
        t = (0, n // 2, n - 1)[i % 3]
        c = (i // 3) % (case["cmax"] + 1)
        mask = sum(1 << q for q in W.random_controls(where, n, t, c))
        out.append((t, mask, W.haar_2x2(rng)))
    return out


def _angles(seed, count):
    """Angles as training starts with them: small, so that gradients have not vanished."""
    return np.random.default_rng([seed, 3]).normal(0.0, 0.2, size=count)


def _circuit(case, seed):
    """(gates, theta) of a circuit case."""
    if case["circuit"] == "random":
        return _random_gates(case, seed), None
    if case["circuit"] == "qft":
        return W.qft_circuit(case["n"]), None
    return W.hea_circuit(case["n"], case["layers"]), _angles(seed, 2 * case["n"] * case["layers"])


def _batch_sizes(case):
    return np.random.default_rng(case["structure"]).integers(case["nmin"], case["nmax"] + 1,
                                                             size=case["states"]).astype(np.int32)


def _compile(case, gates, theta, adjoint):
    if case["mode"] == "compiled":
        dt = qs.QS_C64 if case["dtype"] == "c64" else qs.QS_C128
        qs.qs_circuit_compile(case["n"], dt, gates, theta, FLAGS["compiled"], adjoint=adjoint)


def prepare(case, seed):
    path = case["path"]
    s = {"case": case}
    if path in ("gates", "circuit", "expect"):
        s["psi"] = _amplitudes(case, seed, biased=path == "expect")
        s["state"] = qs.State.wrap(s["psi"], case["n"])
    if path == "gates":
        s["gates"] = _sweep_gates(case, seed)
    elif path == "circuit":
        s["gates"], s["theta"] = _circuit(case, seed)
        _compile(case, s["gates"], s["theta"], False)
    elif path in ("grad", "train"):
        s["gates"] = W.hea_circuit(case["n"], case["layers"])
        theta = _angles(seed, 2 * case["n"] * case["layers"])
        _compile(case, s["gates"], theta, True)
        if path == "grad":
            s["theta"] = theta
            s["state"] = qs.State(case["n"], case["dtype"])
        else:
            s["theta"] = torch.tensor(theta, dtype=REAL[case["dtype"]], device="cuda", requires_grad=True)
    elif path == "batch":
        ns = _batch_sizes(case)
        by_n = {int(n): W.hea_circuit(int(n), case["layers"]) for n in set(ns.tolist())}
        counts = [2 * int(n) * case["layers"] for n in ns]
        s["theta"] = torch.tensor(_angles(seed, sum(counts)), dtype=torch.float64, device="cuda")
        s["energy"] = torch.zeros(len(ns), dtype=torch.float64, device="cuda")
        s["grad"] = torch.zeros(sum(counts), dtype=torch.float64, device="cuda")
        s["batch"] = qs.Batch(ns, [by_n[int(n)] for n in ns], counts, case["dtype"])
    return s


def run(s):
    case = s["case"]
    path = case["path"]
    if path == "gates":
        for t, mask, U in s["gates"]:
            s["state"].apply_gate(t, U, mask)
        return s["psi"]
    if path == "circuit":
        s["state"].apply_circuit(s["gates"], s["theta"], FLAGS[case["mode"]])
        return s["psi"]
    if path == "expect":
        z, norm2 = s["state"].expect_z()
        return (z, norm2) if case["dtype"] == "c128" else (z.astype(np.float32), np.float32(norm2))
    if path == "grad":
        s["state"].set_basis(0)
        e, g = s["state"].adjoint_grad(s["gates"], s["theta"], FLAGS[case["mode"]])
        return (e, g) if case["dtype"] == "c128" else (np.float32(e), g.astype(np.float32))
    if path == "train":
        s["theta"].grad = None
        e = AdjointEnergy.apply(s["theta"], case["n"], s["gates"], case["dtype"], FLAGS[case["mode"]])
        e.backward()
        return e.detach().to(s["theta"].dtype), s["theta"].grad
    flags = qs.QS_FLAG_GRAPH | (qs.QS_FLAG_JIT if case["mode"] == "compiled" else 0)
    s["batch"].run(s["theta"], s["energy"], s["grad"], flags)
    return s["energy"].to(REAL[case["dtype"]]), s["grad"].to(REAL[case["dtype"]])


# ---------------------------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------------------------


def _gate_flops(gates, n):
    """Additions and multiplications of the gates' pair updates: 28 per selected pair of a general
    matrix, 12 of a real or diagonal one, 6 of a phase on one side, none of an exchange."""
    total = 0.0
    for g in gates:
        pairs = 2.0 ** (n - 1 - bin(int(g["ctrl_mask"])).count("1"))
        if g["kind"] == W.KIND_X:
            per = 0
        elif g["kind"] in (W.KIND_RY, W.KIND_RZ):
            per = 12
        else:
            a, b, c, d = W.unpack_u(g["U"]).reshape(4)
            per = 6 if (b == 0 and c == 0 and (a == 1 or d == 1)) else 12 if (b == 0 and c == 0) or \
                not np.any(np.abs(np.imag([a, b, c, d]))) else 28
        total += per * pairs
    return total


def _grad_flops(n, layers):
    """Forward, un-apply of psi and lambda, 8 per pair for each derivative, <O> and lambda = O psi."""
    return 3 * _gate_flops(W.hea_circuit(n, layers), n) + 8.0 * 2 * n * layers * 2.0 ** (n - 1) + 8.0 * 2.0 ** n


def work(case):
    path = case["path"]
    amp = AMP[case["dtype"]]
    if path == "gates":
        bytes_, flops = 0.0, 0.0
        for t, mask, _ in _sweep_gates(case, 0):
            sel = 2.0 ** (case["n"] - bin(mask).count("1"))
            bytes_ += 2 * sel * amp
            flops += 28 * sel / 2
        return {"bytes": bytes_, "flops": flops}
    if path == "circuit":
        gates, _ = _circuit(case, 0)
        return {"bytes": 2.0 * 2.0 ** case["n"] * amp, "flops": _gate_flops(gates, case["n"])}
    if path == "expect":
        return {"bytes": 2.0 ** case["n"] * amp, "flops": 4.0 * 2.0 ** case["n"]}
    if path in ("grad", "train"):
        params = 2 * case["n"] * case["layers"]
        return {"bytes": 2.0 * 2.0 ** case["n"] * amp + 16.0 * params, "flops": _grad_flops(case["n"], case["layers"])}
    ns = _batch_sizes(case).tolist()
    params = sum(2 * n * case["layers"] for n in ns)
    flops = {n: _grad_flops(n, case["layers"]) for n in set(ns)}
    return {"bytes": 16.0 * params + 8.0 * len(ns), "flops": sum(flops[n] for n in ns)}


# ---------------------------------------------------------------------------------------------
# The same results from plain torch in 64 bits
# ---------------------------------------------------------------------------------------------


def _pairs(psi, n, target, mask):
    """Views of the two halves of the pairs that a gate selects, of psi[batch, 2^n]."""
    qubits = sorted([q for q in range(n) if (mask >> q) & 1 or q == target], reverse=True)
    shape, at, dim, above = [psi.shape[0]], [slice(None)], None, n
    for q in qubits:
        shape += [1 << (above - q - 1), 2]
        at += [slice(None), slice(None) if q == target else 1]
        dim = len([a for a in at if isinstance(a, slice)]) - 1 if q == target else dim
        above = q
    v = psi.view(shape + [1 << above])[tuple(at)]
    return v.select(dim, 0), v.select(dim, 1)


def _apply(psi, n, target, mask, U):
    """U (a 2x2 list of numbers, or of columns with one number for each state of the batch; None:
    exchange) on the selected pairs of psi[batch, 2^n], in place."""
    x, y = _pairs(psi, n, target, mask)
    if U is None:
        t = x.clone()
        x.copy_(y)
        y.copy_(t)
        return
    (a, b), (c, d) = ([e if isinstance(e, complex) else e.view([-1] + [1] * (x.dim() - 1)) for e in r] for r in U)
    if all(isinstance(e, complex) for e in (b, c)) and b == 0 and c == 0:
        x.mul_(a)
        y.mul_(d)
        return
    nx = a * x
    nx += b * y
    y.mul_(d)
    y += c * x
    x.copy_(nx)


def _matrix(g, theta, inverse=False):
    """The gate's matrix; theta[batch, params] gives each state its own angle."""
    if g["kind"] == W.KIND_X:
        return None
    if g["kind"] == W.KIND_U:
        u = W.unpack_u(g["U"])
        u = u.conj().T if inverse else u
        return [[complex(u[0, 0]), complex(u[0, 1])], [complex(u[1, 0]), complex(u[1, 1])]]
    h = (-0.5 if inverse else 0.5) * theta[:, int(g["param"])]
    c, s = torch.cos(h), torch.sin(h)
    if g["kind"] == W.KIND_RY:
        return [[c, -s], [s, c]]
    return [[torch.complex(c, -s), 0j], [0j, torch.complex(c, s)]]


def _grad64(n, gates, theta):
    """Energies <sum_i Z_i> [batch] and gradients [batch, params] of theta[batch, params]."""
    psi = torch.zeros(theta.shape[0], 1 << n, dtype=torch.complex128, device="cuda")
    psi[:, 0] = 1
    for g in gates:
        _apply(psi, n, int(g["target"]), int(g["ctrl_mask"]), _matrix(g, theta))
    k = torch.arange(1 << n, device="cuda")
    diag = torch.full((1 << n,), float(n), dtype=torch.float64, device="cuda")
    for q in range(n):
        diag -= 2.0 * ((k >> q) & 1)
    energy = (psi.abs().square() * diag).sum(1)
    lam = psi * diag
    grad = torch.zeros_like(theta)
    for g in gates[::-1]:
        t, m = int(g["target"]), int(g["ctrl_mask"])
        if g["kind"] in (W.KIND_RY, W.KIND_RZ):  # dE/dtheta = Im <lambda| P psi>, after the gate
            x, y = _pairs(psi, n, t, m)
            lx, ly = _pairs(lam, n, t, m)
            dims = tuple(range(1, x.dim()))
            if g["kind"] == W.KIND_RZ:
                v = (lx.conj() * x).imag.sum(dims) - (ly.conj() * y).imag.sum(dims)
            else:  # P = Y: (-i y, i x)
                v = (ly.conj() * x).real.sum(dims) - (lx.conj() * y).real.sum(dims)
            grad[:, int(g["param"])] += v
        U = _matrix(g, theta, inverse=True)
        _apply(psi, n, t, m, U)
        _apply(lam, n, t, m, U)
    return energy, grad


def exact(case, seed):
    path = case["path"]
    if path in ("gates", "circuit"):
        n = case["n"]
        psi = _amplitudes(case, seed).to(torch.complex128).view(1, -1)
        if path == "gates":
            for t, mask, u in _sweep_gates(case, seed):
                _apply(psi, n, t, mask, [[complex(u[0, 0]), complex(u[0, 1])], [complex(u[1, 0]), complex(u[1, 1])]])
        else:
            gates, theta = _circuit(case, seed)
            theta = None if theta is None else torch.tensor(theta, device="cuda").view(1, -1)
            for g in gates:
                _apply(psi, n, int(g["target"]), int(g["ctrl_mask"]), _matrix(g, theta))
        return psi.view(-1)
    if path == "expect":
        n = case["n"]
        p = torch.view_as_real(_amplitudes(case, seed, biased=True)).double().square().sum(1)
        z = [float(v[:, 0].sum() - v[:, 1].sum()) for v in (p.view(-1, 2, 1 << q) for q in range(n))]
        return np.array(z), float(p.sum())
    if path in ("grad", "train"):
        theta = torch.tensor(_angles(seed, 2 * case["n"] * case["layers"]), device="cuda")
        if path == "train":
            theta = theta.to(REAL[case["dtype"]]).double()
        e, g = _grad64(case["n"], W.hea_circuit(case["n"], case["layers"]), theta.view(1, -1))
        if path == "grad":
            return float(e[0]), g[0].cpu().numpy()
        return e[0], g[0]
    ns = _batch_sizes(case)
    at = np.concatenate([[0], np.cumsum(2 * ns.astype(np.int64) * case["layers"])])
    theta = torch.tensor(_angles(seed, int(at[-1])), device="cuda")
    energy = torch.zeros(len(ns), dtype=torch.float64, device="cuda")
    grad = torch.zeros(int(at[-1]), dtype=torch.float64, device="cuda")
    for n in sorted(set(ns.tolist())):
        rows = np.nonzero(ns == n)[0]
        cols = torch.tensor(at[rows][:, None] + np.arange(2 * n * case["layers"]), device="cuda")
        e, g = _grad64(n, W.hea_circuit(n, case["layers"]), theta[cols])
        energy[torch.tensor(rows, device="cuda")] = e
        grad[cols.reshape(-1)] = g.reshape(-1)
    return energy, grad
