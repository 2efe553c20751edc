"""The eight-slice normalisation of split levels at the edges of its K blocks
(32), column tiles (64) and row tiles (128), against the oracle.

Tolerance: the split sweep's own products carry 42 bits of each row and
column (2^-42 = 2.3e-13 a product, a few hundred products at random signs:
below 1e-11 of the largest selected entry), so 1e-11 leaves the
normalisation's 56 bits nothing to hide behind.
"""
from __future__ import annotations

import numpy as np
import pytest

import gen
import oracle
from helpers import selected_error

pytestmark = pytest.mark.gpu
TOL = 1e-11


@pytest.fixture(scope="module")
def torch():
    import torch as _t
    if not _t.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1708_04539_gb300 import build
    build.build()
    return _t


def split_everywhere(h):
    import paper_1708_04539_gb300 as ps
    nlev = int(h.structure()["nlevels"])
    h.plan_set([(lev, 3, 0) for lev in range(nlev)], ps.PREC_OZAKI_FP16)


@pytest.mark.parametrize("kind", ["real", "complex", "symmetric"])
@pytest.mark.parametrize("s,rest", [(33, 1), (63, 40), (64, 64), (65, 130), (96, 129), (128, 5),
                                    (191, 70), (255, 64), (256, 150)])
def test_widths(torch, kind, s, rest):
    import paper_1708_04539_gb300 as ps
    from paper_1708_04539_gb300.binding import supernodal_coordinates
    n = s + rest
    ii, jj = np.meshgrid(np.arange(n), np.arange(n), indexing="ij")
    p = gen.problems._finish_small(n, ii.reshape(-1), jj.reshape(-1), 700 + s, kind == "complex",
                                   f"dense_{n}", s, symmetric_values=kind == "symmetric")
    h = ps.SelInv.from_problem(p, symmetric=kind == "symmetric")
    split_everywhere(h)
    h.factor(torch.from_numpy(p.values).cuda())
    h.selinv(precision=ps.PREC_OZAKI_FP16)
    assert any(r["kind"] == "ozaki_gemm" and r["side"] == 1 for r in h.profile(0))
    sel = oracle.selected_inverse(p, relax_pct=20)
    orows, ocols = sel.sym.lu_pattern()
    grows, gcols = supernodal_coordinates(h.structure())
    gi, oi = np.argsort(grows * n + gcols), np.argsort(orows * n + ocols)
    got, ref = h.get_selected(layout=ps.LAYOUT_SUPERNODAL), sel.values_lu_order()
    h.close()
    assert selected_error(got[gi], ref[oi], orows[oi], ocols[oi], n) < TOL


@pytest.mark.parametrize("complex_values", [False, True])
def test_general_pattern(torch, complex_values):
    """C_L != C_U: panels of different heights."""
    import paper_1708_04539_gb300 as ps
    p = gen.general_random(260, 0.25, 71, complex_values=complex_values, max_sn=96)
    h = ps.SelInv.from_general_problem(p)
    split_everywhere(h)
    h.factor(torch.from_numpy(p.values).cuda())
    h.selinv(precision=ps.PREC_OZAKI_FP16)
    got = h.get_selected()
    h.close()
    ref = oracle.gextract(oracle.general_selected_inverse(p), p.colptr, p.rowind)
    assert np.abs(got - ref).max() < TOL * np.abs(ref).max()


def test_non_finite_values_are_seen(torch):
    """An infinity in A reaches the selected inverse as non-finite values."""
    import paper_1708_04539_gb300 as ps
    p = gen.dense(200, 72, max_sn=100)
    v = p.values.copy()
    v[5] = np.inf
    h = ps.SelInv.from_problem(p)
    split_everywhere(h)
    h.factor(torch.from_numpy(v).cuda())
    h.selinv(precision=ps.PREC_OZAKI_FP16)
    assert not np.isfinite(h.get_selected()).all()
    h.close()
