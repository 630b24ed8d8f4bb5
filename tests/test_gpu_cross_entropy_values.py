"""Cross entropy of samples on amplitudes whose probability has no ordinary
exponent field: zero, subnormal, infinite and NaN of either sign, alone and
among ordinary ones.

Tolerance: a probability and its logarithm carry a few units in the last place,
a product of eight mantissas eight roundings, and the sum of m <= 4000 terms
less than m: 1e-12 of the mean magnitude of the terms covers them."""
import numpy as np
import pytest

import paper_1608_00263_gb300 as qs
from paper_1608_00263_gb300 import build as qs_build

pytestmark = pytest.mark.gpu
N = 10
NEG_NAN = {np.complex64: np.uint32(0xFFC00000).view(np.float32), np.complex128: np.uint64(0xFFF8 << 48).view(np.float64)}


@pytest.fixture(scope="module", autouse=True)
def built():
    qs_build.build()
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


def special(value, dtype):
    part = np.dtype(dtype).type(0).real.dtype.type
    v = np.zeros(1, dtype=dtype)
    re, im = {"zero": (0, 0), "subnormal": (1e-42, 0) if part is np.float32 else (1e-160, 1e-161),
              "inf": (0.5, np.inf), "minus_inf": (-np.inf, 0), "nan": (np.nan, 0.25),
              "negative_nan": (NEG_NAN[dtype], 0.25), "negative_nan_im": (0, NEG_NAN[dtype]),
              "inf_nan": (np.inf, NEG_NAN[dtype])}[value]
    v.real[0], v.imag[0] = re, im
    return v[0]


@pytest.mark.parametrize("dt,dtype", [(qs.QS_C64, np.complex64), (qs.QS_C128, np.complex128)])
@pytest.mark.parametrize("value", ["zero", "subnormal", "inf", "minus_inf", "nan", "negative_nan", "negative_nan_im",
                                   "inf_nan"])
def test_special_amplitude(value, dt, dtype):
    rng = np.random.default_rng(5)
    a = (rng.standard_normal(1 << N) + 1j * rng.standard_normal(1 << N)).astype(dtype) / np.sqrt(2.0 ** (N + 1)).astype(
        dtype)
    a[77] = special(value, dtype)
    h = qs.qs_state_create(N, dt)
    try:
        qs.qs_state_copy_in(h, a)
        for m, at in ((1, [0]), (8, [3]), (300, [0, 17, 299]), (4000, [2047])):
            x = rng.integers(78, 1 << N, size=m).astype(np.uint64)
            x[at] = 77
            v = a[x.astype(np.int64)].astype(np.complex128)
            with np.errstate(all="ignore"):
                terms = -np.log(v.real * v.real + v.imag * v.imag)
            want = np.mean(terms)
            got = qs.qs_cross_entropy(h, x)[0]
            if np.isfinite(want):
                assert abs(got - want) <= 1e-12 * np.mean(np.abs(terms)), m
            else:
                assert got == want or (np.isnan(got) and np.isnan(want)), (m, got, want)
    finally:
        qs.qs_state_destroy(h)
