"""Algorithm 1 skips a term of the density that is not a number, or whose centre lies beyond all bounds: the
blocks are those of the other terms, bit for bit (the mesh is given, the kept term reaches every box)."""
import numpy as np
import pytest

from paper_0706_0747_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_0706_0747_gb300 import mra  # noqa: E402

GOOD = ([2.0], [3.0], [[0.4, 0.5, 0.6]], [0.5])


@pytest.mark.parametrize("k", [3, 8])
@pytest.mark.parametrize("bad", [([np.nan], [5.0], [[0.3, 0.3, 0.3]], [0.0]), ([1.0], [5.0], [[0.3, np.nan, 0.3]], [0.0]),
                                 ([1.0], [5.0], [[0.3, np.nan, 0.3]], [2.0]), ([1.0], [5.0], [[np.inf, 0.1, 0.3]], [2.0]),
                                 ([1.0], [5.0], [[0.2, 0.1, -1e200]], [2.0]), ([1.0], [np.inf], [[0.2, 0.1, 0.3]], [0.0])])
def test_terms_that_are_skipped(k, bad):
    def blocks(*parts):
        coef, expo, cen, r2 = (sum(v, []) for v in zip(*parts))
        d = W.Density(coef=coef, expo=expo, centers=cen, r2coef=r2)
        return mra.build_tree(d, k, 1e-6, 2, uniform_level=2)[0].export()[2]

    ref = blocks(GOOD)
    assert np.isfinite(ref).all() and np.abs(ref).max() > 1
    assert np.array_equal(blocks(GOOD, bad), ref)
    assert np.array_equal(blocks(bad, GOOD), ref)
