"""Batch statistics where their sums take a branch of their own: terms of
probabilities above the FP32 range (N p > 4096) in some lanes of a batch and in
all, chunks that do not fill a batch of loads, few chunks and many, in both
engines, against the oracle.

Tolerance: the largest probability is a product of up to 20 rotations of three
FP32 shears, 60 * 2^-24 relative in the amplitude, twice that in p and four
times in p^4: 3e-5 relative for the moments.  The entropy is ln N less a sum that
a few such roundings scale: 1e-6 n absolute."""
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


def peaked(n, spread, rng):
    """R_Y on every qubit: product states from |0...0> (one probability of N)
    to nearly uniform ones, with small phases after it."""
    g = np.zeros(2 * n, dtype=qs.GATE_DTYPE)
    g["q0"] = np.tile(np.arange(n), 2)
    g["kind"][:n], g["theta"][:n] = qs.QS_RY, spread * rng.uniform(0.6, 1.0, size=n)
    g["kind"][n:], g["theta"][n:] = qs.QS_RZ, rng.uniform(-3, 3, size=n)
    return g


@pytest.mark.parametrize("sizes", [(11, 12, 13), (14, 16, 17), (20,), (19, 20, 20, 20, 20, 20, 20, 20, 20, 20, 20, 20, 20,
                                                                      20, 20, 20, 20, 20, 20, 20, 20, 20)],
                         ids=["small", "chunks", "one", "many"])
@pytest.mark.parametrize("spread", [0.1, 0.6, 1.5])
def test_peaked_states(sizes, spread):
    rng = np.random.default_rng(len(sizes))
    lists = {n: peaked(n, spread, rng) for n in sorted(set(sizes))}
    want = {n: O.probabilities(O.simulate(n, g)) for n, g in lists.items()}
    if spread == 0.1:
        assert any((1 << n) * p.max() > 4096 for n, p in want.items())
    b = qs.qs_batch_create(sizes)
    try:
        rows = {}
        for engine in (qs.QS_BATCH_PERSISTENT, qs.QS_BATCH_ROUNDS):
            qs.qs_batch_set_engine(b, engine)
            rows[engine] = qs.qs_batch_run(b, [lists[n] for n in sizes], kmax=4)
        assert np.array_equal(rows[qs.QS_BATCH_PERSISTENT], rows[qs.QS_BATCH_ROUNDS])
        for i, n in enumerate(sizes):
            assert rows[qs.QS_BATCH_ROUNDS][i, 1] == pytest.approx(O.entropy(want[n]), abs=1e-6 * n)
            assert np.allclose(rows[qs.QS_BATCH_ROUNDS][i, 3:], O.moments(want[n], 4), rtol=3e-5)
    finally:
        qs.qs_batch_destroy(b)
