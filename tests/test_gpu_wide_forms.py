"""Both splits of the wide pass on one state against the FP64 oracle: five
register bits up to 2^8 tiles, six beyond (the sizes on both sides of the
line, tiles of every size, the first pass generated and loaded).  Tolerance:
the state bound of complex64, 1e-5 relative L2."""
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


@pytest.mark.parametrize("kinds", [CT, ALL], ids=["clifford_t", "all"])
@pytest.mark.parametrize("n,tile,bits", [(19, 11, 5), (20, 11, 6), (20, 12, 5), (21, 12, 6), (21, 13, 5), (22, 13, 6)])
def test_state(n, tile, bits, kinds):
    rng = np.random.default_rng(100 * n + tile)
    g = np.zeros(120, dtype=qs.GATE_DTYPE)
    g["kind"] = rng.choice(kinds, size=len(g))
    for x in g:
        x["q0"], x["q1"] = rng.choice(n, size=2, replace=False)
    g["theta"] = rng.uniform(-7, 7, size=len(g))
    assert qs.qs_plan_circuit(n, qs.QS_C64, g, tile_log2=tile)["reg_log2"] == bits
    layer = np.zeros(n, dtype=qs.GATE_DTYPE)
    layer["kind"], layer["q0"] = qs.QS_H, np.arange(n)
    h = qs.qs_state_create(n, qs.QS_C64)
    try:
        for lists in ([np.concatenate([layer, g])], [layer, g]):
            qs.qs_state_reset(h)
            for part in lists:
                qs.qs_apply_circuit(h, part, tile_log2=tile)
            ref = O.simulate(n, np.concatenate([layer, g]))
            got = qs.qs_state_copy_out(h, n)
            assert np.linalg.norm(got - ref) < 1e-5
    finally:
        qs.qs_state_destroy(h)
