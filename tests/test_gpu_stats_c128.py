"""Statistics of complex128 states against extended precision where the table
logarithm and the shared powers can go wrong: probabilities at the edges of
the table's intervals and of powers of two, exponents below and above its
range, zero amplitudes, and states smaller than a block, with remainders and
of several elements per thread.

Tolerance: a term's error is a few units in the last place (at most nine
roundings for y^10, one for each exponent product and logarithm), and the
sums' rounding is below sqrt(N) of those of their largest terms: 4e-14
relative covers 2^17 terms with a factor of ten."""
import numpy as np
import pytest

import paper_1608_00263_gb300 as qs
from paper_1608_00263_gb300 import build as qs_build

pytestmark = pytest.mark.gpu
TOL = 4e-14


@pytest.fixture(scope="module", autouse=True)
def built():
    qs_build.build()
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


def amplitudes(n, kind):
    rng = np.random.default_rng(n)
    size = 1 << n
    a = (rng.standard_normal(size) + 1j * rng.standard_normal(size)) * 2.0 ** (-0.5 * (n + 1))
    if kind == "edges":
        # |a|^2 at and beside the borders of table intervals and powers of two
        i = rng.integers(0, 2049, size)
        p = (1 + i / 2048) * 2.0 ** (rng.integers(-6, 3, size) - n)
        a = np.sqrt(p * (1 + rng.integers(-2, 3, size) * 2.0 ** -52)) * rng.choice([1, -1, 1j, -1j], size)
    elif kind in ("wide", "zeros"):
        a *= 2.0 ** rng.integers(-60, 1, size)
        a[rng.integers(0, size)] = 1e-170          # |a|^2 subnormal or zero
        a[rng.integers(0, size)] = 2.0 ** -0.25
        if kind == "zeros":
            a[rng.integers(0, size, 1 + size // 8)] = 0
    return a


@pytest.mark.parametrize("kind", ["gauss", "edges", "wide", "zeros"])
@pytest.mark.parametrize("n", [1, 7, 8, 12, 17])
def test_statistics(n, kind):
    a = amplitudes(n, kind)
    h = qs.qs_state_create(n, qs.QS_C128)
    qs.qs_state_copy_in(h, a)
    got = qs.qs_pt_moments(h, 10)
    qs.qs_state_destroy(h)
    p = (a.real * a.real + a.imag * a.imag).astype(np.longdouble)
    size, s = 1 << n, p.sum()
    if s == 0:      # a state without a norm has no distribution
        assert got["norm"] == 0 and got["entropy"] == 0 and not np.any(got["moments"])
        return
    q = p / s
    nz = q[q > 0]
    assert abs(got["norm"] - s) <= TOL * s
    assert abs(got["entropy"] + (nz * np.log(nz)).sum()) <= TOL * n
    want = [(np.longdouble(size) ** (k - 1) * q ** k).sum() for k in range(1, 11)]
    assert np.all(np.abs(got["moments"] - want) <= TOL * np.array(want))
    if (p > 0).all():
        ce = -np.log(q).mean()
        assert abs(got["uniform_ce"] - ce) <= TOL * max(abs(ce), n)
    else:
        assert np.isinf(got["uniform_ce"]) and got["uniform_ce"] > 0
