"""The tensor-core applies' wait_limit means the same time in the group kernel (static screen) and in
the pair-list kernel: the first wait of every CTA runs out (the test hook sends no MMA), both report
MRA_ETIMEOUT, and the next apply is as without it.  16,384 polls take about 60 ms in either; a factor
of four between them allows for the rest of the call."""
import time

import numpy as np
import pytest

from paper_0706_0747_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_0706_0747_gb300 import mra  # noqa: E402


def test_one_meaning_of_wait_limit():
    tree, _ = mra.build_tree(W.unit_mass([70.0, 150.0], [[0.45, 0.52, 0.5], [0.62, 0.41, 0.47]]), 4, 1e-4, 3, init_level=1)
    mra.compress(tree)
    op = mra.make_operator(0.0, 1.0, 1e-4, 4, 3)
    took = []
    for screen in ("static", "pair"):
        ref = mra.apply_ns(op, tree, precision="tc", screen=screen)[0].export()[2]
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        with pytest.raises(mra.MraError) as e:
            mra.apply_ns(op, tree, precision="tc", screen=screen, wait_limit=16384, test_flags=mra.TEST_WITHHOLD_MMA)
        took.append(time.perf_counter() - t0)
        assert e.value.code == mra.ETIMEOUT
        again = mra.apply_ns(op, tree, precision="tc", screen=screen)[0].export()[2]
        assert np.array_equal(again, ref)
    assert max(took) < min(4 * min(took), 1.0), took
