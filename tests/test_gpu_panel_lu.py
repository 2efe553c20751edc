"""The panel LU of the diagonal blocks and their triangular inverses at the
edges of its panels (32 columns), line groups (32 lines, 96 in large
launches) and inverse merges (32, 64, 128), against the oracle's factors.

Tolerance: as for the factorisation's other parity tests, 1e-12 of the
largest selected entry of the row and column; the selected inverse (which
reads the inverses) 1e-10.
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


def check(p, h, batches):
    import paper_1708_04539_gb300 as ps
    from paper_1708_04539_gb300.binding import supernodal_coordinates
    st = h.structure()
    s = oracle.analyze(p, relax_pct=20)
    orows, ocols = s.lu_pattern()
    grows, gcols = supernodal_coordinates(st)
    gi, oi = np.argsort(grows * p.n + gcols), np.argsort(orows * p.n + ocols)
    for b in batches:
        vals = p.values if p.values.ndim == 1 else p.values[b]
        f = oracle.lu(s, p.colptr, p.rowind, vals)
        ovals = np.concatenate([f.diag, f.low, f.up])
        got = h.get_selected(batch=b, layout=ps.LAYOUT_FACTORS)
        assert selected_error(got[gi], ovals[oi], orows[oi], ocols[oi], p.n) < 1e-12
        ref = oracle.selinv(f).values_lu_order()
        got = h.get_selected(batch=b, layout=ps.LAYOUT_SUPERNODAL)
        assert selected_error(got[gi], ref[oi], orows[oi], ocols[oi], p.n) < 1e-10


@pytest.mark.parametrize("kind", ["real", "complex", "symmetric"])
@pytest.mark.parametrize("s,rest", [(1, 3), (31, 40), (32, 33), (33, 20), (63, 5), (64, 0), (65, 40),
                                    (97, 1), (128, 30), (160, 17), (255, 0), (256, 40)])
def test_widths(torch, kind, s, rest):
    import paper_1708_04539_gb300 as ps
    n = s + rest
    ii, jj = np.meshgrid(np.arange(n), np.arange(n), indexing="ij")
    p = gen.problems._finish_small(n, ii.reshape(-1), jj.reshape(-1), 900 + s, kind == "complex",
                                   f"dense_{n}", s, symmetric_values=kind == "symmetric")
    h = ps.SelInv.from_problem(p, symmetric=kind == "symmetric")
    h.factor(torch.from_numpy(p.values).cuda())
    h.selinv()
    check(p, h, [0])
    h.close()


@pytest.mark.parametrize("s,complex_values", [(20, False), (32, True), (70, False)])
def test_many_instances(torch, s, complex_values):
    """Enough tasks for the launches of 96 lines per CTA."""
    import paper_1708_04539_gb300 as ps
    p = gen.dense(s + 45, 950 + s, complex_values=complex_values, max_sn=s)
    nb = 160
    rng = np.random.default_rng(3)
    vals = p.values[None, :] * rng.uniform(0.5, 2.0, size=(nb, 1))
    p.values = np.ascontiguousarray(vals)
    h = ps.SelInv.from_problem(p)
    h.factor(torch.from_numpy(p.values).cuda())
    h.selinv()
    check(p, h, [0, 77, nb - 1])
    h.close()


@pytest.mark.parametrize("kind", ["real", "complex", "symmetric"])
@pytest.mark.parametrize("s", [20, 70])
@pytest.mark.parametrize("nb", [9, 20])
def test_lanes_per_line(torch, kind, s, nb):
    """Launches whose lines take two lanes or one (one instance: four), with
    ragged last panels and line groups."""
    import paper_1708_04539_gb300 as ps
    n = s + 45
    ii, jj = np.meshgrid(np.arange(n), np.arange(n), indexing="ij")
    p = gen.problems._finish_small(n, ii.reshape(-1), jj.reshape(-1), 970 + s, kind == "complex",
                                   f"dense_{n}", s, symmetric_values=kind == "symmetric")
    p.values = np.ascontiguousarray(p.values[None, :] * np.linspace(0.5, 2.0, nb)[:, None])
    h = ps.SelInv.from_problem(p, symmetric=kind == "symmetric", check_level=1)
    h.factor(torch.from_numpy(p.values).cuda())
    h.selinv()
    check(p, h, [0, nb - 1])
    h.close()


@pytest.mark.parametrize("kind", ["real", "complex", "symmetric"])
def test_large_schur_tiles(torch, kind):
    """Levels with enough Schur work for 32 x 32 tiles and a K split: ragged
    tiles (133 rows) over supernodes of 90 columns, 24 instances."""
    import paper_1708_04539_gb300 as ps
    n, nb = 90 + 133, 24
    ii, jj = np.meshgrid(np.arange(n), np.arange(n), indexing="ij")
    p = gen.problems._finish_small(n, ii.reshape(-1), jj.reshape(-1), 990, kind == "complex",
                                   f"dense_{n}", 90, symmetric_values=kind == "symmetric")
    p.values = np.ascontiguousarray(p.values[None, :] * np.linspace(0.5, 2.0, nb)[:, None])
    h = ps.SelInv.from_problem(p, symmetric=kind == "symmetric", check_level=1)
    h.factor(torch.from_numpy(p.values).cuda())
    h.selinv()
    check(p, h, [0, nb - 1])
    h.close()


@pytest.mark.parametrize("density,max_sn", [(0.02, 16), (0.3, 64)])
def test_general_schur(torch, density, max_sn):
    """C_L != C_U: the Schur tiles through the two row structures' maps."""
    import paper_1708_04539_gb300 as ps
    p = gen.general_random(300, density, 77, max_sn=max_sn)
    h = ps.SelInv.from_general_problem(p, check_level=1)
    h.factor(torch.from_numpy(p.values).cuda())
    h.selinv()
    got = h.get_selected()
    ref = oracle.gextract(oracle.general_selected_inverse(p), p.colptr, p.rowind)
    assert np.abs(got - ref).max() < 1e-10 * np.abs(ref).max()
    h.close()


@pytest.mark.parametrize("kind,nb", [("real", 40), ("complex", 12), ("symmetric", 80)])
@pytest.mark.parametrize("s", [30, 96])
def test_eight_slice_levels(torch, kind, nb, s):
    """Split factorisation, levels below its threshold of Schur work but with
    more FP64 work than a few launches: products of eight slices, held to the
    FP64 tolerance."""
    import paper_1708_04539_gb300 as ps
    n = s + 133
    nb = nb * (5 if s == 30 else 1)
    ii, jj = np.meshgrid(np.arange(n), np.arange(n), indexing="ij")
    p = gen.problems._finish_small(n, ii.reshape(-1), jj.reshape(-1), 995, kind == "complex",
                                   f"dense_{n}", s, symmetric_values=kind == "symmetric")
    p.values = np.ascontiguousarray(p.values[None, :] * np.linspace(0.5, 2.0, nb)[:, None])
    h = ps.SelInv.from_problem(p, symmetric=kind == "symmetric",
                               factor_precision=ps.PREC_OZAKI_FP16, factor_split_mflops=100000)
    h.factor(torch.from_numpy(p.values).cuda())
    h.selinv()
    assert any(r["kind"] == "ozaki_gemm" for r in h.profile(1))
    h.factor(torch.from_numpy(p.values).cuda())
    h.selinv()
    check(p, h, [0, nb - 1])
    h.close()
