"""A factorisation that does not fit the device is refused, again and again, and
the handle works for smaller batches afterwards."""
from __future__ import annotations

import numpy as np
import pytest

import gen

pytestmark = pytest.mark.gpu


def test_batch_beyond_the_device():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1708_04539_gb300 import build
    build.build()
    import paper_1708_04539_gb300 as ps
    p = gen.conv_diff_2d(24, seed=5)
    h = ps.SelInv.from_problem(p)
    v = torch.from_numpy(p.values).cuda()

    def result():
        h.factor(v)
        h.selinv()
        return h.get_selected()
    ref = result()
    free, _ = torch.cuda.mem_get_info()
    # the first buffer alone exceeds the device (the values are not read before it)
    nb = free // (8 * int(h.structure()["storage_size"])) * 2 + 1
    for _ in range(2):
        rc = h._lib.pselinv_factor(h._h, ps.F64, nb, v.data_ptr(), None)
        assert rc == -4  # PSELINV_ERR_OOM
        with pytest.raises(ps.PselinvError):
            h.selinv()
    np.testing.assert_allclose(result(), ref, rtol=0, atol=1e-13 * np.abs(ref).max())
    h.close()
