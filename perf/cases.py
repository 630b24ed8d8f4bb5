"""The work a user of the random-circuit library has it do, as measurable cases.

Each case is one call sequence of the paper's method on seeded inputs:

  circuit    evolve |0...0> by a random circuit and read the 2^n output
             probabilities (Secs. cqs, pt): Clifford+T gates of the paper, or
             the same circuit with parameterised rotations
  step       the whole estimation procedure on one circuit: evolve,
             probabilities, Porter-Thomas statistics, samples, cross entropy
  readout    probabilities, statistics, samples and cross entropy of a state
             loaded from a checkpoint
  cycles     statistics after every cycle of a circuit (Figs. evd, mvd)
  ensemble   independent circuits of uneven size on the batched engine, with
             every instance's entropy and inverse participation ratio
  noisy      trajectories of the depolarising error model on the batched
             engine and their mean output distribution (Fig. pal)
  gradient   d(cross entropy)/d(angle) of a parameterised circuit through the
             torch.autograd binding

Circuits are drawn here from the case's seed by the rules of Sec.
"Convergence to Porter-Thomas" and handed to the library as gate arrays; the
sizes are those of the repository's benchmark, tests and stated
configurations.
"""
import math
import random

import numpy as np
import torch

import paper_1608_00263_gb300 as qs

H, XH, YH, T, CZ, RX, RY, RZ, CPHASE = range(9)

# ---------------------------------------------------------------------------
# circuits (plain Python; the inputs of every case)
# ---------------------------------------------------------------------------


def _rows_for(n):
    """Grid rows of an n-qubit circuit: 3 up to 15 qubits, 4 up to 24, 5 above."""
    return 3 if n <= 15 else 4 if n <= 24 else 5


def _grid(n):
    """Sites of the grid in row-major order; the last row's surplus is dead."""
    rows = _rows_for(n)
    cols = -(-n // rows)
    return rows, cols


def _layout(n, which):
    """CZ pairs of layout `which` (H0 H2 V0 V2 H1 H3 V1 V3)."""
    rows, cols = _grid(n)
    vertical = which in (2, 3, 6, 7)
    offset = (0, 2, 0, 2, 1, 3, 1, 3)[which]
    out = []
    for r in range(rows):
        for c in range(cols):
            if vertical:
                if (r + 2 * c) % 4 != offset or r + 1 >= rows:
                    continue
                a, b = r * cols + c, (r + 1) * cols + c
            else:
                if (c + 2 * r) % 4 != offset or c + 1 >= cols:
                    continue
                a, b = r * cols + c, r * cols + c + 1
            if a < n and b < n:
                out.append((a, b))
    return out


def _circuit(n, depth, rng):
    """H on every qubit, then per cycle one CZ layout and a gate from
    {X^1/2, Y^1/2, T} on each qubit idle now and in a CZ the cycle before (T
    first, then never the previous one again): (kind, q0, q1, cycle, theta)."""
    gates = [(H, q, 0, 0, 0.0) for q in range(n)]
    previous = [None] * n
    busy_before = set()
    for t in range(1, depth + 1):
        pairs = _layout(n, (t - 1) % 8)
        busy = {q for p in pairs for q in p}
        gates += [(CZ, a, b, t, 0.0) for a, b in pairs]
        for q in range(n):
            if q in busy_before and q not in busy:
                kind = T if previous[q] is None else rng.choice([k for k in (XH, YH, T) if k != previous[q]])
                gates.append((kind, q, 0, t, 0.0))
                previous[q] = kind
        busy_before = busy
    return gates


def _rotations(gates, rng, noise=0.05):
    """The circuit with X^1/2, Y^1/2, T and CZ as R_X, R_Y, R_Z and CPHASE at
    their nominal angles plus N(0, noise)."""
    to = {XH: (RX, math.pi / 2), YH: (RY, math.pi / 2), T: (RZ, math.pi / 4), CZ: (CPHASE, math.pi)}
    out = []
    for kind, a, b, t, theta in gates:
        if kind in to:
            kind, theta = to[kind]
            theta += rng.gauss(0.0, noise) if noise else 0.0
        out.append((kind, a, b, t, theta))
    return out


def _trajectory(gates, n, r, rng):
    """One trajectory of the depolarising error model: Paulis (as rotations
    by pi) with probability r / 10 after one-qubit gates, r after CZ, and
    initial bit flips with probability r."""
    pauli = {1: RX, 2: RY, 3: RZ}
    out = [(RX, q, 0, 0, math.pi) for q in range(n) if rng.random() < r]
    for g in gates:
        out.append(g)
        if g[0] == CZ:
            if rng.random() < r:
                e = rng.randrange(1, 16)
                if e // 4:
                    out.append((pauli[e // 4], g[1], 0, g[3], math.pi))
                if e % 4:
                    out.append((pauli[e % 4], g[2], 0, g[3], math.pi))
        elif rng.random() < r / 10:
            out.append((pauli[rng.randrange(1, 4)], g[1], 0, g[3], math.pi))
    return out


def _array(gates):
    """The library's gate records."""
    out = np.zeros(len(gates), dtype=qs.GATE_DTYPE)
    for f, k in (("kind", 0), ("q0", 1), ("q1", 2), ("cycle", 3), ("theta", 4)):
        out[f] = [g[k] for g in gates]
    return out


def _case_circuit(case, seed):
    rng = random.Random("circuit %d" % seed)
    gates = _circuit(case["n"], case["depth"], rng)
    return _rotations(gates, rng) if case.get("gates") == "rotations" else gates


def _instances(case, seed):
    """(n, gates) of every instance of an ensemble: n uniform in the case's
    range and depth uniform in 10..40 by the instance's number, gates from
    the seed."""
    out = []
    for i in range(case["count"]):
        size = random.Random("size %d" % i)
        n, depth = size.randint(case["n_min"], case["n_max"]), size.randint(10, 40)
        out.append((n, _circuit(n, depth, random.Random("instance %d %d" % (seed, i)))))
    return out


def _trajectories(case, seed):
    gates = _circuit(case["n"], case["depth"], random.Random("circuit %d" % seed))
    return [_trajectory(gates, case["n"], 0.005, random.Random("trajectory %d %d" % (seed, i)))
            for i in range(case["count"])]


def _checkpoint(case, seed):
    """A state as a deep circuit leaves it: complex Gaussian amplitudes
    (Porter-Thomas distributed probabilities), normalised."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    a = torch.randn((1 << case["n"]), 2, generator=g, device="cuda", dtype=torch.float32)
    a *= 2.0 ** (-0.5 * (case["n"] + 1))
    return torch.view_as_complex(a)


# ---------------------------------------------------------------------------
# the method in 64 bits (plain torch)
# ---------------------------------------------------------------------------


def _matrix(kind, theta):
    s, c = math.sqrt(0.5), math.cos(theta / 2)
    d = math.sin(theta / 2)
    return {H: (s, s, s, -s), XH: (s, -1j * s, -1j * s, s), YH: (s, -s, s, s),
            RX: (c, -1j * d, -1j * d, c), RY: (c, -d, d, c)}[kind]


def _apply(psi, n, gate, inverse=False):
    kind, a, b, _, theta = gate
    if kind in (CZ, CPHASE):
        lo, hi = min(a, b), max(a, b)
        f = -1.0 if kind == CZ else complex(math.cos(theta), math.sin(theta))
        psi.view(1 << (n - hi - 1), 2, 1 << (hi - lo - 1), 2, 1 << lo)[:, 1, :, 1] *= f.conjugate() if inverse else f
        return
    v = psi.view(1 << (n - a - 1), 2, 1 << a)
    if kind in (T, RZ):
        f = [1.0, complex(math.sqrt(0.5), math.sqrt(0.5))] if kind == T else [
            complex(math.cos(theta / 2), -math.sin(theta / 2)), complex(math.cos(theta / 2), math.sin(theta / 2))]
        for k in (0, 1):
            if f[k] != 1.0:
                v[:, k] *= f[k].conjugate() if inverse else f[k]
        return
    u = _matrix(kind, theta)
    if inverse:
        u = tuple(complex(u[k]).conjugate() for k in (0, 2, 1, 3))
    x = v[:, 0].clone()
    v[:, 0] *= u[0]
    v[:, 0].add_(v[:, 1], alpha=u[1])
    v[:, 1] *= u[3]
    v[:, 1].add_(x, alpha=u[2])


def _zero_state(n):
    psi = torch.zeros(1 << n, dtype=torch.complex128, device="cuda")
    psi[0] = 1.0
    return psi


def _evolve(n, gates):
    psi = _zero_state(n)
    for g in gates:
        _apply(psi, n, g)
    return psi


def _probabilities(psi):
    return psi.real.square().add_(psi.imag.square())


def _statistics(p, kmax):
    """norm, entropy, uniform cross entropy, moments 1..kmax of p / sum p."""
    n, s = p.numel(), p.sum()
    q = p / s
    lq = torch.log(q)
    moments = [float((float(n) ** (k - 1) * q.pow(k)).sum()) for k in range(1, kmax + 1)]
    return [float(s), float(-(torch.where(q > 0, q * lq, torch.zeros_like(q))).sum()), float(-lq.mean())] + moments


def _samples_of(p, m, seed):
    """m indices drawn from p."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    c = torch.cumsum(p, 0)
    u = torch.rand(m, generator=g, device="cuda", dtype=torch.float64) * c[-1]
    return torch.searchsorted(c, u, right=True).clamp_(max=p.numel() - 1)


def _gradient_inputs(case, seed):
    """Circuit with noisy angles, and samples of the nominal circuit."""
    rng = random.Random("gradient %d" % seed)
    plain = _circuit(case["n"], case["depth"], rng)
    gates = _rotations(plain, rng)
    x = _samples_of(_probabilities(_evolve(case["n"], plain)), case["m"], seed)
    return gates, x


def _gradient(n, gates, x):
    """Loss -(1/m) sum ln p(x) and its derivative by every angle (reverse sweep)."""
    psi = _evolve(n, gates)
    p = _probabilities(psi)
    loss = float(-torch.log(p[x]).mean())
    lam = torch.zeros_like(psi)
    lam.index_add_(0, x, -psi[x] / (x.numel() * p[x]))
    del p
    grad = []
    for g in reversed(gates):
        kind, a, b = g[:3]
        if kind == CPHASE:
            lo, hi = min(a, b), max(a, b)
            shape = (1 << (n - hi - 1), 2, 1 << (hi - lo - 1), 2, 1 << lo)
            grad.append(-2.0 * float((lam.view(shape)[:, 1, :, 1].conj() * psi.view(shape)[:, 1, :, 1]).sum().imag))
        elif kind in (RX, RY, RZ):
            shape = (1 << (n - a - 1), 2, 1 << a)
            l0, l1 = lam.view(shape)[:, 0].conj(), lam.view(shape)[:, 1].conj()
            p0, p1 = psi.view(shape)[:, 0], psi.view(shape)[:, 1]
            if kind == RX:
                grad.append(float((l0 * p1).sum().imag + (l1 * p0).sum().imag))
            elif kind == RY:
                grad.append(float(-(l0 * p1).sum().real + (l1 * p0).sum().real))
            else:
                grad.append(float((l0 * p0).sum().imag - (l1 * p1).sum().imag))
        _apply(psi, n, g, inverse=True)
        _apply(lam, n, g, inverse=True)
    return loss, grad[::-1]


# ---------------------------------------------------------------------------
# handles
# ---------------------------------------------------------------------------


class _State:
    """A state handle, released with the object."""

    def __init__(self, n, dtype):
        self.h = qs.qs_state_create(n, dtype)

    def __del__(self):
        qs.qs_state_destroy(self.h)


class _Batch:
    def __init__(self, sizes):
        self.h = qs.qs_batch_create(sizes)

    def __del__(self):
        qs.qs_batch_destroy(self.h)


class _Amplitudes:
    """An instance's 2^n complex64 amplitudes, for torch.as_tensor; keeps the
    batch that owns the memory alive as long as the tensor."""

    def __init__(self, batch, i, n):
        self.batch = batch
        address = qs.qs_batch_state(batch.h, i)
        self.__cuda_array_interface__ = {"shape": (2 << n,), "typestr": "<f4", "data": (address, False), "version": 3}


def _dtype(case):
    return qs.QS_C128 if case.get("dtype") == "c128" else qs.QS_C64


def _mode(case):
    return qs.QS_MODE_FUSED_TC if case.get("form") == "tensor" else qs.QS_MODE_FUSED


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------


def listed():
    return [
        # the smallest circuit of the ensemble recipe (3x4 grid): launches and latency
        {"name": "circuit_n12_d25", "kind": "circuit", "n": 12, "depth": 25},
        # the paper's 20-qubit grid at depth 25, single precision: a state that fits the L2 cache
        {"name": "circuit_n20_d25", "kind": "circuit", "n": 20, "depth": 25},
        # the whole estimation procedure on that grid in double precision, as the paper computes it
        {"name": "step_n20_d25_c128", "kind": "step", "n": 20, "depth": 25, "dtype": "c128", "m": 100000},
        # statistics after every cycle (Figs. evd, mvd), double precision
        {"name": "cycles_n20_d25_c128", "kind": "cycles", "n": 20, "depth": 25, "dtype": "c128"},
        # a ragged grid (4x6 less one site) at an odd depth
        {"name": "circuit_n23_d33", "kind": "circuit", "n": 23, "depth": 33},
        # parameterised gates (forward evolution of circuit-parameter studies), 5x5 grid
        {"name": "rotations_n25_d30", "kind": "circuit", "n": 25, "depth": 30, "gates": "rotations"},
        # the tensor-core form at its default operand precision
        {"name": "tensor_n26_d40", "kind": "circuit", "n": 26, "depth": 40, "form": "tensor"},
        # the benchmark's 30-qubit depth-40 circuit: the largest
        {"name": "circuit_n30_d40", "kind": "circuit", "n": 30, "depth": 40},
        # read-out of a checkpointed state: probabilities, statistics, 10^6 samples, cross entropy
        {"name": "readout_n26_m1e6", "kind": "readout", "n": 26, "m": 1000000},
        # an ensemble of uneven circuits (12..24 qubits, depth 10..40)
        {"name": "ensemble_60", "kind": "ensemble", "count": 60, "n_min": 12, "n_max": 24},
        # error-model trajectories on the 20-qubit grid (Fig. pal) and their mean distribution
        {"name": "noisy_64_n20_d40", "kind": "noisy", "count": 64, "n": 20, "depth": 40},
        # the gradient configuration: 24 qubits, depth 30, 10^5 samples
        {"name": "gradient_n24_d30", "kind": "gradient", "n": 24, "depth": 30, "m": 100000},
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["circuit", "circuit", "circuit", "rotations", "tensor", "step", "readout", "cycles",
                       "ensemble", "noisy", "gradient"])
    depth = rng.randint(8, 40)
    if kind == "circuit":
        dtype = rng.choice(["c64", "c64", "c128"])
        return {"kind": "circuit", "n": rng.randint(12, 29 if dtype == "c64" else 23), "depth": depth, "dtype": dtype}
    if kind == "rotations":
        return {"kind": "circuit", "n": rng.randint(12, 26), "depth": depth, "gates": "rotations"}
    if kind == "tensor":
        return {"kind": "circuit", "n": rng.randint(16, 27), "depth": depth, "form": "tensor"}
    if kind == "step":
        return {"kind": "step", "n": rng.randint(12, 22), "depth": depth, "dtype": "c128", "m": log_int(1000, 300000)}
    if kind == "readout":
        return {"kind": "readout", "n": rng.randint(16, 27), "m": log_int(1000, 1000000)}
    if kind == "cycles":
        return {"kind": "cycles", "n": rng.randint(12, 20), "depth": depth, "dtype": "c128"}
    if kind == "ensemble":
        lo = rng.randint(12, 18)
        return {"kind": "ensemble", "count": log_int(5, 60), "n_min": lo, "n_max": rng.randint(lo, 24)}
    if kind == "noisy":
        return {"kind": "noisy", "count": log_int(5, 64), "n": rng.randint(12, 20), "depth": depth}
    return {"kind": "gradient", "n": rng.randint(12, 24), "depth": rng.randint(8, 30), "m": log_int(1000, 100000),
            "dtype": rng.choice(["c64", "c128"]) if rng.random() < 0.5 else "c64"}


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": dict(case), "seed": seed}
    if kind in ("circuit", "step"):
        n = case["n"]
        gates = _array(_case_circuit(case, seed))
        state = _State(n, _dtype(case))
        # the plan a program makes ahead of the call
        qs.qs_prepare_circuit(state.h, gates, mode=_mode(case))
        single = _dtype(case) == qs.QS_C64
        st.update(state=state, gates=gates, single=single,
                  p=torch.empty(1 << n, dtype=torch.float32 if single else torch.float64, device="cuda"))
    elif kind == "cycles":
        st.update(state=_State(case["n"], _dtype(case)), gates=_array(_case_circuit(case, seed)))
    elif kind == "readout":
        n = case["n"]
        state = _State(n, qs.QS_C64)
        qs.qs_state_copy_in(state.h, _checkpoint(case, seed).cpu().numpy())
        st.update(state=state, p=torch.empty(1 << n, dtype=torch.float64, device="cuda"),
                  x=torch.empty(case["m"], dtype=torch.int64, device="cuda"))
    elif kind == "ensemble":
        inst = _instances(case, seed)
        st.update(batch=_Batch([n for n, _ in inst]), sizes=[n for n, _ in inst], lists=[_array(g) for _, g in inst])
    elif kind == "noisy":
        lists = [_array(g) for g in _trajectories(case, seed)]
        st.update(batch=_Batch([case["n"]] * len(lists)), lists=lists)
    else:
        gates, x = _gradient_inputs(case, seed)
        arr = _array(gates)
        index = np.nonzero(np.isin(arr["kind"], (RX, RY, RZ, CPHASE)))[0]
        theta = torch.tensor(arr["theta"][index], dtype=torch.float64 if _dtype(case) == qs.QS_C128 else torch.float32)
        st.update(state=_State(case["n"], _dtype(case)), gates=arr, index=index, x=x, theta=theta)
    return st


def run(st):
    kind, case = st["case"]["kind"], st["case"]
    if kind in ("circuit", "step"):
        h = st["state"].h
        qs.qs_state_reset(h)
        qs.qs_apply_circuit(h, st["gates"], mode=_mode(case))
        qs.qs_probabilities(h, st["p"], fp64=not st["single"])
        out = {"probabilities": st["p"]}
        if kind == "step":
            out.update(qs.qs_pt_moments(h, 10))
            out["samples"] = qs.qs_sample(h, case["m"], st["seed"])
            out["ce"], out["delta_h"] = qs.qs_cross_entropy(h, out["samples"])
        return out
    if kind == "cycles":
        return {"statistics": qs.qs_cycle_statistics(st["state"].h, st["gates"], 10)}
    if kind == "readout":
        h = st["state"].h
        out = {"probabilities": qs.qs_probabilities(h, st["p"])}
        out.update(qs.qs_pt_moments(h, 10))
        out["samples"] = qs.qs_sample(h, case["m"], st["seed"], st["x"])
        out["ce"], out["delta_h"] = qs.qs_cross_entropy(h, st["x"])
        return out
    if kind == "ensemble":
        b = st["batch"].h
        stats = qs.qs_batch_run(b, st["lists"], kmax=2)
        # the statistics in the precision of the states they are of
        return {"statistics": stats.astype(np.float32),
                "states": [torch.view_as_complex(torch.as_tensor(_Amplitudes(st["batch"], i, n), device="cuda").view(-1, 2))
                           for i, n in enumerate(st["sizes"])]}
    if kind == "noisy":
        b = st["batch"].h
        qs.qs_batch_apply(b, st["lists"])
        # averaged from single-precision states: kept in their precision
        return {"mean": qs.qs_batch_mean_probabilities(b, case["n"]).astype(np.float32)}
    from paper_1608_00263_gb300.autograd import circuit_cross_entropy
    theta = st["theta"].clone().requires_grad_()
    loss = circuit_cross_entropy(theta, st["state"].h, st["gates"], st["index"], st["x"])
    loss.backward()
    return {"loss": loss.detach().to(theta.dtype), "gradient": theta.grad}


def work(case):
    """Inputs read once, outputs written once; operations of the gates: an
    addition per component for H, X^1/2 and Y^1/2, three operations on half
    the amplitudes for T, sign flips counted as one, six per amplitude for
    a rotation."""
    per = {H: 2.0, XH: 2.0, YH: 2.0, T: 1.5, CZ: 0.5, RX: 6.0, RY: 6.0, RZ: 6.0, CPHASE: 1.5}
    size = 16.0 if case.get("dtype") == "c128" else 8.0

    def flops(n, gates):
        return sum(per[g[0]] for g in gates) * (1 << n)

    kind = case["kind"]
    if kind in ("circuit", "step", "cycles"):
        n = case["n"]
        gates = _case_circuit(case, 0)
        if kind == "cycles":
            cycles = case["depth"] + 1
            return {"bytes": 2 * size * (1 << n) * cycles, "flops": flops(n, gates) + 30.0 * (1 << n) * cycles}
        byt = 1.5 * size * (1 << n) + 16.0 * len(gates)
        if kind == "step":
            return {"bytes": byt + 8.0 * case["m"], "flops": flops(n, gates) + 30.0 * (1 << n)}
        return {"bytes": byt, "flops": flops(n, gates)}
    if kind == "readout":
        return {"bytes": 16.0 * (1 << case["n"]) + 16.0 * case["m"], "flops": 30.0 * (1 << case["n"])}
    if kind == "ensemble":
        inst = _instances(case, 0)
        return {"bytes": sum(8.0 * (1 << n) for n, _ in inst), "flops": sum(flops(n, g) for n, g in inst)}
    if kind == "noisy":
        n = case["n"]
        return {"bytes": 8.0 * (1 << n) * case["count"] + 8.0 * (1 << n),
                "flops": sum(flops(n, g) for g in _trajectories(case, 0))}
    rng = random.Random("gradient 0")
    gates = _rotations(_circuit(case["n"], case["depth"], rng), rng)
    return {"bytes": 4 * size * (1 << case["n"]) + 8.0 * case["m"], "flops": 4 * flops(case["n"], gates)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "circuit":
        return {"probabilities": _probabilities(_evolve(case["n"], _case_circuit(case, seed)))}
    if kind in ("step", "readout"):
        if kind == "step":
            p = _probabilities(_evolve(case["n"], _case_circuit(case, seed)))
        else:
            p = _probabilities(_checkpoint(case, seed).to(torch.complex128))
        s = _statistics(p, 10)
        # samples are whole numbers; the cross entropy is that of the samples
        return {"probabilities": p, "norm": s[0], "entropy": s[1], "uniform_ce": s[2], "moments": np.array(s[3:]),
                "samples": None, "ce": None, "delta_h": None}
    if kind == "cycles":
        n, gates = case["n"], _case_circuit(case, seed)
        psi, rows = _zero_state(n), []
        for i, g in enumerate(gates):
            _apply(psi, n, g)
            if i + 1 == len(gates) or gates[i + 1][3] != g[3]:
                rows.append([float(g[3])] + _statistics(_probabilities(psi), 10))
        return {"statistics": np.array(rows)}
    if kind == "ensemble":
        states = [_evolve(n, g) for n, g in _instances(case, seed)]
        return {"statistics": np.array([_statistics(_probabilities(s), 2) for s in states]), "states": states}
    if kind == "noisy":
        mean = 0
        for g in _trajectories(case, seed):
            mean = mean + _probabilities(_evolve(case["n"], g))
        return {"mean": mean / case["count"]}
    gates, x = _gradient_inputs(case, seed)
    loss, grad = _gradient(case["n"], gates, x)
    return {"loss": loss, "gradient": np.array(grad)}
