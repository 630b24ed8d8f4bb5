"""Gate lists whose (re, im) plans look like wide ones and hold more ops than a
wide pass: 250 gates on the lowest five qubits of a state, in the modes that
plan five register bits of the (re, im) form.  Tolerances: the state bound of
complex64, 1e-5 relative L2; the gradient's, 1e-4 of the largest derivative."""
import numpy as np
import pytest

import oracle as O
import paper_1608_00263_gb300 as qs
from paper_1608_00263_gb300 import build as qs_build

pytestmark = pytest.mark.gpu
CT = [qs.QS_H, qs.QS_X_HALF, qs.QS_Y_HALF, qs.QS_T, qs.QS_CZ]


@pytest.fixture(scope="module", autouse=True)
def built():
    qs_build.build()
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


def low_qubit_list(n, kinds, seed):
    rng = np.random.default_rng(seed)
    g = np.zeros(n + 250, dtype=qs.GATE_DTYPE)
    g["kind"][:n], g["q0"][:n] = qs.QS_H, np.arange(n)
    g["kind"][n:] = rng.choice(kinds, size=250)
    for x in g[n:]:
        x["q0"], x["q1"] = rng.choice(5, size=2, replace=False)
    g["theta"][n:] = rng.uniform(-3, 3, size=250)
    return g


@pytest.mark.parametrize("kinds", [CT, CT + [qs.QS_RZ, qs.QS_CPHASE]], ids=["clifford_t", "phases"])
@pytest.mark.parametrize("n", [11, 12])
def test_tensor_mode_without_blocks(n, kinds):
    g = low_qubit_list(n, kinds, n)
    h = qs.qs_state_create(n, qs.QS_C64)
    try:
        qs.qs_apply_circuit(h, g, mode=qs.QS_MODE_FUSED_TC)
        assert np.linalg.norm(qs.qs_state_copy_out(h, n) - O.simulate(n, g)) < 1e-5
    finally:
        qs.qs_state_destroy(h)


@pytest.mark.parametrize("n", [11, 12, 13, 14, 20])
def test_gradient(n):
    g = low_qubit_list(n, CT + [qs.QS_RZ, qs.QS_CPHASE], n)
    x = np.random.default_rng(n).integers(0, 1 << n, size=300).astype(np.uint64)
    out = {}
    for dt in (qs.QS_C128, qs.QS_C64):
        h = qs.qs_state_create(n, dt)
        try:
            out[dt] = qs.qs_adjoint_gradient(h, g, x)
        finally:
            qs.qs_state_destroy(h)
    (loss, grad), (loss32, grad32) = out[qs.QS_C128], out[qs.QS_C64]
    p = O.probabilities(O.simulate(n, g))
    assert loss == pytest.approx(-np.mean(np.log(p[x])), abs=1e-9)
    assert loss32 == pytest.approx(loss, abs=1e-4)
    assert np.max(np.abs(grad32 - grad)) < 1e-4 * np.max(np.abs(grad))


@pytest.mark.parametrize("first", ["empty", "layer"])
@pytest.mark.parametrize("small", [8, 10])
def test_batch_with_a_small_instance_without_passes(small, first):
    """The others plan five register bits there; both engines against the
    oracle.  Tolerance: the ensemble statistics', 1e-6 (entropy) and 1e-5
    (moments) relative."""
    sizes = (small, 12, 13)
    rng = np.random.default_rng(small)
    layer = lambda n: O.generate_circuit(1, n, 0, 0)[:n]
    for count in (1, 3, 12, 60):
        gl = [layer(small)[:0] if first == "empty" else layer(small)]
        for n in sizes[1:]:
            g = np.zeros(count, dtype=qs.GATE_DTYPE)
            g["kind"] = rng.choice(CT + [qs.QS_RX, qs.QS_RY, qs.QS_RZ, qs.QS_CPHASE], size=count)
            for x in g:
                x["q0"], x["q1"] = rng.choice(n, size=2, replace=False)
            g["kind"][0], g["q0"][0] = qs.QS_RY, 0
            g["theta"] = rng.uniform(-3, 3, size=count)
            gl.append(np.concatenate([layer(n), g]).astype(qs.GATE_DTYPE))
        b = qs.qs_batch_create(sizes)
        try:
            for engine in (qs.QS_BATCH_PERSISTENT, qs.QS_BATCH_ROUNDS):
                qs.qs_batch_set_engine(b, engine)
                rows = qs.qs_batch_run(b, gl, kmax=4)
                for i, n in enumerate(sizes[1:], 1):
                    p = O.probabilities(O.simulate(n, gl[i]))
                    assert rows[i, 1] == pytest.approx(O.entropy(p), rel=1e-6), (engine, count, i)
                    assert np.allclose(rows[i, 3:], O.moments(p, 4), rtol=1e-5), (engine, count, i)
        finally:
            qs.qs_batch_destroy(b)
