"""Accuracy of the split factorisation's products that are not six-slice ones:
panel solves that stay on the FP64 pipe."""
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
