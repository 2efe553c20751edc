"""The fused launch of an FP64 level (gather of G and steps 3-5) at the edges
of its 16 x 16 output tiles and 32-long contraction chunks, for every form of
handle: real, complex, symmetric values, general patterns, several instances,
checked maps.

Tolerance: as for the sweep's other parity tests, 1e-10 of the largest
selected entry of the row and column, against the oracle and between the
fused launch and the gather and products of the per-supernode schedule.
"""
from __future__ import annotations

import numpy as np
import pytest

import gen
from test_gpu_general import check_against_oracle, run_general
from test_gpu_panel_lu import check

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as _t
    if not _t.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1708_04539_gb300 import build
    build.build()
    return _t


@pytest.mark.parametrize("kind", ["real", "complex", "symmetric"])
@pytest.mark.parametrize("s,c", [(1, 1), (1, 40), (2, 16), (5, 17), (15, 31), (16, 32), (17, 33),
                                 (31, 64), (33, 65), (40, 95), (48, 7), (66, 130)])
def test_tiles(torch, kind, s, c):
    """Supernodes of s columns over all the later rows (c, c - s, ...)."""
    import paper_1708_04539_gb300 as ps
    n = s + c
    ii, jj = np.meshgrid(np.arange(n), np.arange(n), indexing="ij")
    p = gen.problems._finish_small(n, ii.reshape(-1), jj.reshape(-1), 700 + n, kind == "complex",
                                   f"dense_{n}", s, symmetric_values=kind == "symmetric")
    h = ps.SelInv.from_problem(p, symmetric=kind == "symmetric", check_level=s % 2)
    h.factor(torch.from_numpy(p.values).cuda())
    h.selinv()
    assert any(r["kind"] == "small_level" for r in h.profile(0))
    check(p, h, [0])
    h.close()


@pytest.mark.parametrize("make", [
    lambda: gen.general_random(260, 0.02, 711, max_sn=12),
    lambda: gen.general_random(200, 0.03, 712, complex_values=True, max_sn=33),
    lambda: gen.general_random(90, 0.08, 713, triangle="upper", row_scramble=False),
    lambda: gen.general_random(90, 0.08, 714, triangle="lower", row_scramble=False),
], ids=["real", "complex", "upper", "lower"])
@pytest.mark.parametrize("check_level", [0, 1])
def test_general(torch, make, check_level):
    """C_L != C_U: G is c_U x c_L; a triangular pattern has one of them empty."""
    import paper_1708_04539_gb300 as ps
    p = make()
    h, st, fac, sn, pa = run_general(torch, p, check_level=check_level)
    check_against_oracle(p, st, fac, sn, pa)
    h.close()
    g, st2, fac2, sn2, pa2 = run_general(torch, p, schedule=ps.SCHED_PER_SUPERNODE)
    g.close()
    scale = np.abs(sn2).max()
    assert np.abs(sn - sn2).max() <= 1e-10 * scale


@pytest.mark.parametrize("complex_values", [False, True])
def test_instances(torch, complex_values):
    """Several instances, whose tasks are shared (one grid row each)."""
    import paper_1708_04539_gb300 as ps
    p = gen.upwind_3d(7, 720, max_sn=20) if not complex_values else gen.stencil27_complex(5, 721, max_sn=20)
    rng = np.random.default_rng(5)
    p.values = np.ascontiguousarray(p.values[None, :] * rng.uniform(0.5, 2.0, size=(9, 1)))
    h = ps.SelInv.from_problem(p)
    h.factor(torch.from_numpy(p.values).cuda())
    h.selinv()
    check(p, h, [0, 4, 8])
    h.close()
