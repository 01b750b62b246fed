"""The group applies in FP32 and on the tensor cores held to their rounding, against the FP64 apply of the same
operator and tree: a piece, a translation or a product of FP16 halves left out would show.

Tolerances: FP16 hi + lo operands keep 22 bits, six of them enter a product, and sums are FP32: 2e-6
(hi lo products left out: 1e-3).  FP32: three stages of 24-bit factors and sums, 1e-6."""
import numpy as np
import pytest

from oracle import tree as OT
from tests.helpers import oracle_to_arrays

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_0706_0747_gb300 import mra  # noqa: E402

EPS, J = 1e-4, 4
DENS = OT.Density([3.0, 1.2, 5.0], [40.0, 400.0, 2500.0], [[0.42, 0.55, 0.5], [0.8, 0.2, 0.9], [0.26, 0.24, 0.51]])


@pytest.mark.parametrize("mu", [0.0, 1.5])
@pytest.mark.parametrize("k", range(1, 9))
def test_groups_to_rounding(k, mu):
    op = mra.make_operator(mu, 1.0, EPS, k, J)
    depth = 3 if k <= 2 else J
    for levels, kw in ((depth, {"init_level": 1}), (2, {"uniform_level": 2}), (1, {"uniform_level": 1}), (0, {"uniform_level": 0})):
        t, _ = OT.build_tree(DENS, k, 1e-3, levels, **kw)
        tg = mra.tree_import(k, *oracle_to_arrays(t, k))
        mra.compress(tg)
        for unscreened in (False, True):
            ref, st = mra.apply_ns(op, tg, precision="fp64", unscreened=unscreened)
            ref = ref.export()[2]
            assert st["n_items"] > 0
            for precision, tol in (("tc", 2e-6), ("fp32", 1e-6)):
                got, stp = mra.apply_ns(op, tg, precision=precision, unscreened=unscreened)
                assert (stp["n_items"], stp["n_pairs"]) == (st["n_items"], st["n_pairs"])
                assert np.linalg.norm(got.export()[2] - ref) <= tol * np.linalg.norm(ref), (levels, unscreened, precision)
