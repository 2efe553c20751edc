"""FP64 sweep levels beyond the fused launch's size: gather and products, against
the oracle.  Tolerances as for the sweep's other parity tests."""
from __future__ import annotations

import numpy as np
import pytest

import gen
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


@pytest.mark.parametrize("kind,nb", [("real", 76), ("complex", 19), ("symmetric", 76)])
def test_large_level(torch, kind, nb):
    """Just over 2e10 flops on one level (513 rows of 256 columns), the others fused."""
    import paper_1708_04539_gb300 as ps
    n = 256 + 513
    ii, jj = np.meshgrid(np.arange(n), np.arange(n), indexing="ij")
    p = gen.problems._finish_small(n, ii.reshape(-1), jj.reshape(-1), 80, kind == "complex",
                                   f"dense_{n}", 256, symmetric_values=kind == "symmetric")
    p.values = np.ascontiguousarray(p.values[None, :] * np.linspace(0.5, 2.0, nb)[:, None])
    h = ps.SelInv.from_problem(p, symmetric=kind == "symmetric")
    h.factor(torch.from_numpy(p.values).cuda())
    h.selinv()
    kinds = [r["kind"] for r in h.profile(0)]
    assert kinds.count("gather") == 1 and "small_level" in kinds
    h.selinv()
    check(p, h, [0, nb - 1])
    h.close()
