"""The sampler's prefix table, written by the read-out of a state that was
sampled before, against the one formed for the sample (a state that was
not): the same samples, whole numbers, at partial chunks, one chunk, and
several; also after the state changed without a read-out of its own, and for
a second sample of the same state."""
import numpy as np
import pytest

import paper_1608_00263_gb300 as qs
from paper_1608_00263_gb300 import build as qs_build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    qs_build.build()
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


def state_values(n, seed):
    rng = np.random.default_rng(seed)
    a = rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)
    return (a / np.linalg.norm(a)).astype(np.complex64)


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("n", [3, 7, 8, 9, 13, 18])
def test_same_samples(n, fp64):
    k = 5000
    first, second, third = (state_values(n, s) for s in (1, 2, 3))

    def fresh(values):
        h = qs.qs_state_create(n, qs.QS_C64)
        qs.qs_state_copy_in(h, values)
        x = qs.qs_sample(h, k, 77)
        qs.qs_state_destroy(h)
        return np.asarray(x)

    h = qs.qs_state_create(n, qs.QS_C64)
    out = np.empty(1 << n, dtype=np.float64 if fp64 else np.float32)
    got = []
    for values, read in ((first, True), (second, True), (third, False)):
        qs.qs_state_copy_in(h, values)
        if read:
            qs.qs_probabilities(h, out, fp64=fp64)
        got.append(np.asarray(qs.qs_sample(h, k, 77)))
    again = np.asarray(qs.qs_sample(h, k, 77))
    qs.qs_state_destroy(h)
    for values, x in zip((first, second, third), got):
        assert np.array_equal(x, fresh(values))
    assert np.array_equal(again, got[-1])
