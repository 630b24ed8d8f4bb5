"""Lists of a few gates on one state against the FP64 oracle: on a state in
memory on both sides of the line between the (re, im) form and the wide pass
(5 gates at 21 qubits, 16 at 22), and on the uniform state that the first pass generates with nothing folded into
it.  Tolerance: the state bound of complex64, 1e-5 relative L2."""
import numpy as np
import pytest

import oracle as O
import paper_1608_00263_gb300 as qs
from paper_1608_00263_gb300 import build as qs_build

pytestmark = pytest.mark.gpu
CT = [qs.QS_H, qs.QS_X_HALF, qs.QS_Y_HALF, qs.QS_T, qs.QS_CZ]
ALL = CT + [qs.QS_RX, qs.QS_RY, qs.QS_RZ, qs.QS_CPHASE]


@pytest.fixture(scope="module", autouse=True)
def built():
    qs_build.build()
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


def gate_list(rng, n, count, kinds):
    g = np.zeros(count, dtype=qs.GATE_DTYPE)
    g["kind"] = rng.choice(kinds, size=count)
    for x in g:
        x["q0"], x["q1"] = rng.choice(n, size=2, replace=False)
    g["theta"] = rng.uniform(-7, 7, size=count)
    return g


@pytest.mark.parametrize("kinds", [CT, ALL], ids=["clifford_t", "all"])
@pytest.mark.parametrize("n", [21, 22])
def test_state_in_memory(n, kinds):
    rng = np.random.default_rng(n)
    start = (rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)) * 2.0 ** (-0.5 * (n + 1))
    start = start.astype(np.complex64)
    h = qs.qs_state_create(n)
    try:
        for count in (1, 5, 6, 16, 17):
            g = gate_list(rng, n, count, kinds)
            for prepare in (False, True):
                qs.qs_state_copy_in(h, start)
                if prepare:
                    qs.qs_prepare_circuit(h, g)
                qs.qs_apply_circuit(h, g)
                ref = start.astype(np.complex128)
                O.apply_circuit(ref, g)
                got = qs.qs_state_copy_out(h, n)
                assert np.linalg.norm(got - ref) < 1e-5 * np.linalg.norm(ref), (count, prepare)
    finally:
        qs.qs_state_destroy(h)


@pytest.mark.parametrize("n", [5, 10, 11, 12, 13, 14, 19, 21, 22])
def test_nothing_folded(n):
    """Every qubit's first gate after the layer is not diagonal, or the list is
    shorter than the layer's width."""
    rng = np.random.default_rng(n)
    layer = np.zeros(n, dtype=qs.GATE_DTYPE)
    layer["kind"], layer["q0"] = qs.QS_H, np.arange(n)
    rot = layer.copy()
    rot["kind"], rot["theta"] = qs.QS_RX, rng.uniform(-3, 3, size=n)
    h = qs.qs_state_create(n)
    try:
        for tail in (rot[:1], rot, np.concatenate([rot, gate_list(rng, n, 60, ALL)])):
            g = np.concatenate([layer, tail]).astype(qs.GATE_DTYPE)
            qs.qs_state_reset(h)
            qs.qs_apply_circuit(h, g)
            assert np.linalg.norm(qs.qs_state_copy_out(h, n) - O.simulate(n, g)) < 1e-5, len(tail)
    finally:
        qs.qs_state_destroy(h)
