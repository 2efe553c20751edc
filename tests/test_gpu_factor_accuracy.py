"""Accuracy of the split factorisation's products that are not six-slice ones:
panel solves that stay on the FP64 pipe, and products of eight slices."""
from __future__ import annotations

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

U64 = 2.0 ** -53


@pytest.fixture(scope="module")
def torch():
    import torch as _t
    if not _t.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1708_04539_gb300 import build
    build.build()
    return _t


def csc(a, rng):
    """(colptr, rowind, values) of a dense array's non-zero pattern."""
    r, c = np.nonzero(a.T)[1], np.nonzero(a.T)[0]
    colptr = np.zeros(a.shape[0] + 1, dtype=np.int64)
    np.cumsum(np.bincount(c, minlength=a.shape[0]), out=colptr[1:])
    return colptr, r.astype(np.int64), np.ascontiguousarray(a[r, c])


@pytest.mark.parametrize("complex_values", [False, True])
@pytest.mark.parametrize("s", [20, 40])
def test_one_sided_level_solves_in_fp64(torch, s, complex_values):
    """General pattern, split factorisation: on a level with a supernode that
    has only one of R_L and R_U every panel is solved in FP64.  The first
    supernode's panels take no Schur update, so they agree with the FP64
    factorisation's to rounding: a solve against s columns errs by at most s u of
    its largest terms (diagonally dominant: of the order of the panel's largest
    entry) on each side, 8 s u in all; six slices err by 2^-43 = 1024 u a term."""
    import paper_1708_04539_gb300 as ps
    rng = np.random.default_rng(s)
    n, k = 136, 96
    a = np.zeros((n, n), dtype=complex if complex_values else float)
    a[:k, :k] = rng.uniform(-1, 1, (k, k))
    a[k:, k:] = np.triu(rng.uniform(-1, 1, (n - k, n - k)), 1)
    if complex_values:
        a = a + 1j * np.where(a != 0, rng.uniform(-1, 1, (n, n)), 0)
    np.fill_diagonal(a, np.abs(a).sum(0) + np.abs(a).sum(1) + 1)
    colptr, rowind, values = csc(a, rng)
    order = np.arange(n, dtype=np.int64)
    got = []
    for kw in ({}, {"factor_precision": ps.PREC_OZAKI_FP16, "factor_split_mflops": -1}):
        h = ps.SelInv.general(n, colptr, rowind, rperm=order, cperm=order, max_supernode=s,
                              relax_pct=0, **kw)
        st = h.structure()
        h.factor(torch.from_numpy(values).cuda())
        got.append(h.get_selected(layout=ps.LAYOUT_FACTORS))
        h.close()
    c, cu = np.diff(st["rows_ptr"]), np.diff(st["urows_ptr"])
    assert st["sn_width"][0] == s and c[0] == cu[0] == k - s
    assert ((c == 0) != (cu == 0)).any()
    w = slice(st["sn_offset"][0] + s * s, st["sn_offset"][0] + s * s + 2 * s * (k - s))
    ref, x = got[0][w], got[1][w]
    for part in (slice(0, s * (k - s)), slice(s * (k - s), None)):
        assert np.abs(x[part] - ref[part]).max() <= 8 * s * U64 * np.abs(ref[part]).max()


@pytest.mark.parametrize("kind", ["real", "complex", "symmetric"])
@pytest.mark.parametrize("s,c", [(33, 140), (64, 133), (65, 64), (256, 60)])
def test_eight_slice_outputs_keep_their_bits(torch, kind, s, c):
    """Panels over an identity block, so that the solved panels are A's own: every
    row has entries of 1 and of 2^-20.  Their digits hold 63 bits below the
    row's power of two (2 at most) and the other operand is one digit, so an entry
    is off by at most 2^-63 and its own rounding."""
    import paper_1708_04539_gb300 as ps
    n = s + c
    nb = int(1.2e8 / ((2.0 * c * c * s + 2.0 * c * s * s) * (4 if kind == "complex" else 1)
                      * (0.5 if kind == "symmetric" else 1))) + 1
    rng = np.random.default_rng(s)

    def panel():
        x = rng.uniform(0.5, 1, (c, s)) * np.where(rng.random((c, s)) < 0.2, 1.0, 2.0 ** -20)
        return x + (1j * rng.uniform(-1, 1, (c, s)) * 2.0 ** -18 if kind == "complex" else 0)
    low = panel()
    up = low if kind == "symmetric" else panel()
    a = np.zeros((n, n), dtype=low.dtype)
    a[s:, :s], a[:s, s:] = low, up.T
    a[:s, :s] = np.eye(s)
    a[s:, s:] = 4.0 * n * np.eye(c)
    colptr = np.arange(n + 1, dtype=np.int64) * n  # (the whole pattern, zeros too)
    rowind = np.tile(np.arange(n, dtype=np.int64), n)
    h = ps.SelInv(n, colptr, rowind, np.arange(n, dtype=np.int64), max_supernode=s,
                  symmetric=kind == "symmetric", factor_precision=ps.PREC_OZAKI_FP16,
                  factor_split_mflops=100000)
    st = h.structure()
    assert st["sn_width"][0] == s
    h.factor(torch.from_numpy(np.tile(a.T.reshape(-1), (nb, 1))).cuda())
    assert any(r["kind"] == "ozaki_gemm" and r["level"] == 0 for r in h.profile(1))
    h.factor(torch.from_numpy(np.tile(a.T.reshape(-1), (nb, 1))).cuda())
    for b in (0, nb - 1):
        fac = h.get_selected(batch=b, layout=ps.LAYOUT_FACTORS)
        o = st["sn_offset"][0] + s * s
        for got, ref in ((fac[o:o + c * s], low), (fac[o + c * s:o + 2 * c * s], up)):
            got = got.reshape(s, c).T
            for x, r in ((got.real, ref.real), (got.imag, ref.imag)):
                assert (np.abs(x - r) <= 2.0 ** -63 + U64 * np.abs(r)).all()
    h.close()
