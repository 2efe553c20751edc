"""Schur products of a level beside the next level's LU: the corner (the
parents' diagonal blocks) on the main stream, the rest on another, each with
its own scatter.  Corners of 96 rows, no multiple of the product tiles' 128,
enough instances for the overlap, and several factorisations with other values,
so that what an earlier one left in the scratch is not right by chance.

Tolerances: those of the factorisation's other parity tests, 1e-10 for sliced
products of 42 bits, 1e-12 for eight slices.
"""
from __future__ import annotations

import numpy as np
import pytest

import gen
import oracle
from helpers import selected_error

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as _t
    if not _t.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1708_04539_gb300 import build
    build.build()
    return _t


@pytest.mark.parametrize("kind,n,nb", [
    ("real", 224, 130), ("complex", 224, 70), ("symmetric", 224, 256),  # corner tiles only
    ("real", 325, 41), ("complex", 325, 21), ("symmetric", 325, 81)])
@pytest.mark.parametrize("mflops,tol", [(0, 1e-10), (100000, 1e-12)], ids=["split", "eight"])
def test_bulk_beside_the_next_level(torch, kind, nb, n, mflops, tol):
    import paper_1708_04539_gb300 as ps
    from paper_1708_04539_gb300.binding import supernodal_coordinates
    ii, jj = np.meshgrid(np.arange(n), np.arange(n), indexing="ij")
    p = gen.problems._finish_small(n, ii.reshape(-1), jj.reshape(-1), 40 + n, kind == "complex",
                                   f"dense_{n}", 96, symmetric_values=kind == "symmetric")
    h = ps.SelInv.from_problem(p, symmetric=kind == "symmetric",
                               factor_precision=ps.PREC_OZAKI_FP16, factor_split_mflops=mflops)
    base = p.values
    s = oracle.analyze(p, relax_pct=20)
    orows, ocols = s.lu_pattern()
    grows, gcols = supernodal_coordinates(h.structure())
    gi, oi = np.argsort(grows * n + gcols), np.argsort(orows * n + ocols)
    for k in range(3):
        scale = np.linspace(0.5, 2.0, nb) * 3.0 ** k
        vals = np.ascontiguousarray(base[None, :] * scale[:, None])
        h.factor(torch.from_numpy(vals).cuda())
        # (symmetric six-slice products of real values scatter themselves)
        if k == 0 and n > 224 and (kind, mflops) != ("symmetric", 0):
            assert any(x["kind"] == "scatter_sub" and x["side"] == 2 for x in h.profile(1))
            h.factor(torch.from_numpy(vals).cuda())
        for b in (0, nb // 2, nb - 1):
            f = oracle.lu(s, p.colptr, p.rowind, vals[b])
            ref = np.concatenate([f.diag, f.low, f.up])
            got = h.get_selected(batch=b, layout=ps.LAYOUT_FACTORS)
            assert selected_error(got[gi], ref[oi], orows[oi], ocols[oi], n) < tol
    h.close()
