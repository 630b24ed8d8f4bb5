"""The wide fused pass (complex64, tiles of 11 to 13 qubits) against the FP64
oracle where it can go wrong: one tile and two, every tile size, the first
pass reading a given state instead of generating it, one pass reading and
writing canonical order, state memory the caller holds, and gate lists with
every kind of gate.  Tolerance: the state bound of complex64, 1e-5 relative
L2 (the deviation of an FP32 evolution of a few hundred gates is below 3e-6)."""
import numpy as np
import pytest

import oracle as O
import paper_1608_00263_gb300 as qs
from paper_1608_00263_gb300 import build as qs_build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    qs_build.build()
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


def gate_list(rng, n, count, kinds):
    g = np.zeros(count, dtype=qs.GATE_DTYPE)
    g["kind"] = rng.choice(kinds, size=count)
    for x in g:
        a, b = rng.choice(n, size=2, replace=False)
        x["q0"], x["q1"] = a, b
    g["theta"] = rng.uniform(-7, 7, size=count)
    return g


CT = [qs.QS_H, qs.QS_X_HALF, qs.QS_Y_HALF, qs.QS_T, qs.QS_CZ]
ALL = CT + [qs.QS_RX, qs.QS_RY, qs.QS_RZ, qs.QS_CPHASE]


@pytest.mark.parametrize("kinds", [CT, ALL], ids=["clifford_t", "all"])
@pytest.mark.parametrize("n,tile", [(11, 0), (12, 0), (13, 0), (14, 0), (14, 11), (15, 12), (17, 13), (18, 0)])
def test_state(n, tile, kinds):
    rng = np.random.default_rng(100 * n + tile + len(kinds))
    start = rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)
    start = (start / np.linalg.norm(start)).astype(np.complex64)
    h = qs.qs_state_create(n, qs.QS_C64)
    try:
        for count in (1, 7, 300):
            g = gate_list(rng, n, count, kinds)
            qs.qs_state_copy_in(h, start)
            qs.qs_apply_circuit(h, g, tile_log2=tile)
            ref = start.astype(np.complex128)
            O.apply_circuit(ref, g)
            got = qs.qs_state_copy_out(h, n)
            assert np.linalg.norm(got - ref) < 1e-5 * np.linalg.norm(ref), count
    finally:
        qs.qs_state_destroy(h)


@pytest.mark.parametrize("n", [11, 16, 20])
def test_generated_and_held_states_agree(n):
    """A circuit on |0...0>: generated first pass (created state), and the
    same list on memory the caller holds (every pass loads)."""
    import torch
    rows, cols = (1, n) if n < 12 else (4, -(-n // 4))
    g = O.generate_circuit(rows, cols, 17, 3)
    ref = O.simulate(n, g)
    buf = torch.zeros(1 << n, dtype=torch.complex64, device="cuda")
    buf[0] = 1
    held = qs.qs_state_attach(n, qs.QS_C64, buf)
    made = qs.qs_state_create(n, qs.QS_C64)
    try:
        for h in (held, made):
            qs.qs_apply_circuit(h, g)
            got = qs.qs_state_copy_out(h, n)
            assert np.linalg.norm(got - ref) < 1e-5
    finally:
        qs.qs_state_destroy(held)
        qs.qs_state_destroy(made)


@pytest.mark.parametrize("n", [9, 10, 11, 13, 16])
def test_adjoint_sweep(n):
    """Gradient of every parameterised gate of a list with all gate kinds: the
    complex64 sweep (wide passes from 10 qubits on, tile groups below) against
    the complex128 one, which the adjoint tests pin to exact parameter shifts.
    Tolerance: theirs for complex64, 1e-4 of the largest derivative."""
    rng = np.random.default_rng(40 + n)
    g = np.concatenate([O.generate_circuit(1, n, 0, 0)[:n], gate_list(rng, n, 220, ALL)]).astype(qs.GATE_DTYPE)
    x = rng.integers(0, 1 << n, size=500).astype(np.uint64)
    out = {}
    for dt in (qs.QS_C128, qs.QS_C64):
        h = qs.qs_state_create(n, dt)
        try:
            loss, grad = qs.qs_adjoint_gradient(h, g, x)
            loss2, grad2 = qs.qs_adjoint_gradient(h, g, x)          # the kept plan
            assert loss == loss2 and np.max(np.abs(grad - grad2)) <= 1e-5 * np.max(np.abs(grad))
            g2 = g.copy()
            g2["theta"] *= 1.01                                     # another list: a new plan
            out[dt] = (grad, qs.qs_adjoint_gradient(h, g2, x)[1])
            psi = qs.qs_state_copy_out(h, n, dt)                    # the sweep undoes the circuit
            assert abs(psi[0] - 1) < (1e-4 if dt == qs.QS_C64 else 1e-10)
        finally:
            qs.qs_state_destroy(h)
    for a, b in zip(out[qs.QS_C64], out[qs.QS_C128]):
        assert np.max(np.abs(a - b)) < 1e-4 * np.max(np.abs(b))
        assert np.all(a[g["kind"] < qs.QS_RX] == 0)


@pytest.mark.parametrize("kinds", [CT, ALL], ids=["clifford_t", "all"])
@pytest.mark.parametrize("sizes,tile", [((11, 12, 13, 16, 11), 0), ((14, 11, 12), 11), ((19, 12, 12), 12)])
def test_batch_engines(sizes, tile, kinds):
    """Single tiles that take part of a CTA's threads (tile 0), tiles side by
    side in groups (11, 12), both engines alike."""
    rng = np.random.default_rng(7 * sum(sizes) + tile)
    gl = [np.concatenate([O.generate_circuit(1, n, 0, 0)[:n], gate_list(rng, n, 150, kinds)]).astype(qs.GATE_DTYPE)
          for n in sizes]
    b = qs.qs_batch_create(sizes)
    try:
        qs.qs_batch_set_options(b, tile_log2=tile)
        rows = {}
        for engine in (qs.QS_BATCH_PERSISTENT, qs.QS_BATCH_ROUNDS):
            qs.qs_batch_set_engine(b, engine)
            rows[engine] = qs.qs_batch_run(b, gl, kmax=4)
        assert np.array_equal(rows[qs.QS_BATCH_PERSISTENT], rows[qs.QS_BATCH_ROUNDS])
        for i, n in enumerate(sizes):
            p = O.probabilities(O.simulate(n, gl[i]))
            assert rows[qs.QS_BATCH_ROUNDS][i, 1] == pytest.approx(O.entropy(p), rel=1e-6)
            assert np.allclose(rows[qs.QS_BATCH_ROUNDS][i, 3:], O.moments(p, 4), rtol=1e-5)
    finally:
        qs.qs_batch_destroy(b)
