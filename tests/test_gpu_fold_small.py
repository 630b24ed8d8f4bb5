"""The folded diagonal prefix on small tiles: a CTA of 1, 2, 4 or 8 threads (the
states themselves, and small tiles of a larger state) forms the phases of a
uniform state with every count of eighths.  Against the FP64 oracle; the state
bounds: 1e-5 (complex64) and 1e-12 (complex128) relative L2."""
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


@pytest.mark.parametrize("dt,n,tile", [(qs.QS_C64, n, 0) for n in (5, 6, 7, 8, 9)] +
                         [(qs.QS_C64, 10, t) for t in (5, 6, 7, 8)] +
                         [(qs.QS_C128, n, 0) for n in (4, 5, 6, 7, 8)] + [(qs.QS_C128, 10, t) for t in (4, 5, 6, 7)])
def test_every_eighth(dt, n, tile):
    rng = np.random.default_rng(n + tile)
    layer, tail = np.zeros(n, dtype=qs.GATE_DTYPE), np.zeros(n, dtype=qs.GATE_DTYPE)
    layer["kind"], layer["q0"] = qs.QS_H, np.arange(n)
    tail["kind"], tail["q0"], tail["theta"] = qs.QS_RX, np.arange(n), rng.uniform(-3, 3, size=n)
    counts = [1, 2, 3, 5, 6, 7, 4, 1, 3, 7]
    t = np.zeros(sum(counts[:n]), dtype=qs.GATE_DTYPE)
    t["kind"], t["q0"] = qs.QS_T, np.repeat(np.arange(n), counts[:n])
    cz = np.zeros(2 * n, dtype=qs.GATE_DTYPE)
    cz["kind"] = qs.QS_CZ
    for x in cz:
        x["q0"], x["q1"] = rng.choice(n, size=2, replace=False)
    g = np.concatenate([layer, rng.permutation(np.concatenate([t, cz])), tail]).astype(qs.GATE_DTYPE)
    h = qs.qs_state_create(n, dt)
    try:
        for _ in range(2):
            qs.qs_state_reset(h)
            qs.qs_apply_circuit(h, g, tile_log2=tile)
            got = qs.qs_state_copy_out(h, n, dt)
            assert np.linalg.norm(got - O.simulate(n, g)) < (1e-5 if dt == qs.QS_C64 else 1e-12)
    finally:
        qs.qs_state_destroy(h)
