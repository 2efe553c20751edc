"""Reciprocals of the pivots over the whole range of FP64: mantissas next to powers
of two, exponents around the ends of the integer path's range and of FP64's.

The inverse of a diagonal matrix is the pivots' reciprocals (times 1).  Real: the
integer step is off by half a unit of the last place and 2^-62, so at most one unit
against the correctly rounded quotient.  Complex: conj(z) / |z|^2 takes |z|^2 (two
roundings), its reciprocal and a product, Smith's division about as much; 8 u
against a reference of 3 u."""
from __future__ import annotations

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as _t
    if not _t.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1708_04539_gb300 import build
    build.build()
    return _t


def mantissas(rng, n):
    m = 1.0 + rng.random(n)
    near = np.array([1.0, np.nextafter(1.0, 2), np.nextafter(2.0, 1), 1.0 + 2.0 ** -24,
                     2.0 - 2.0 ** -24, 1.0 + 2.0 ** -29, 2.0 - 2.0 ** -29, 1.5])
    m[:n // 2] = rng.choice(near, n // 2)
    return m * rng.choice([-1.0, 1.0], n)


def inverse(torch, values):
    import paper_1708_04539_gb300 as ps
    n = values.size
    i = np.arange(n, dtype=np.int64)
    h = ps.SelInv(n, np.arange(n + 1, dtype=np.int64), i, i)
    h.factor(torch.from_numpy(values).cuda())
    h.selinv()
    out = h.get_selected()
    h.close()
    return out


def test_real(torch):
    rng = np.random.default_rng(1)
    # biased exponents: 1 .. 2044 (1 / d stays finite), the edges 64 and 1982 often
    e = np.concatenate([np.repeat([1, 2, 62, 63, 64, 65, 66, 1981, 1982, 1983, 1984, 2043, 2044], 60),
                        rng.integers(1, 2045, 3000)])
    d = np.ldexp(mantissas(rng, e.size), e - 1023)
    got, ref = inverse(torch, d), 1.0 / d
    assert (np.abs(got - ref) <= np.spacing(np.abs(ref))).all()


def test_complex(torch):
    rng = np.random.default_rng(2)
    e = np.concatenate([np.repeat([200, 638, 639, 640, 641, 1399, 1400, 1401, 1402, 1800], 60),
                        rng.integers(200, 1800, 3000)])
    other = e - rng.choice([0, 1, 5, 30, 60, 150], e.size)
    x, y = (np.ldexp(mantissas(rng, e.size), k - 1023) for k in (e, other))
    swap = rng.random(e.size) < 0.5
    z = np.where(swap, y, x) + 1j * np.where(swap, x, y)
    got, ref = inverse(torch, z), 1.0 / z
    # (moduli through a common power of two: |z|^2 may leave the range)
    s = np.ldexp(1.0, e - 1023)
    assert (np.abs((got - ref) * s) <= 8 * 2.0 ** -53 * np.abs(ref * s)).all()
