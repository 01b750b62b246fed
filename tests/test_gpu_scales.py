"""Magnitudes of the inputs: the operator is linear and its screens are relative, so a tree times a power
of two gives the outputs times it.

Tolerances: FP16 hi + lo operands and FP32 sums lose nothing under a power of two, so scaled outputs
agree to FP32's rounding of the sums, 1e-6 relative; against FP64 the tensor cores' 2e-6
(six operands rounded to 22 bits and FP32 sums, as test_gpu_orders.py).  The ladder may add eps ||g|| / 4
of rounding to each run, in an order of sums that is not fixed: eps."""
import numpy as np
import pytest

from oracle import tree as OT
from tests.helpers import oracle_to_arrays

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_0706_0747_gb300 import mra  # noqa: E402

DENS = OT.Density([3.0, 1.2], [40.0, 400.0], [[0.42, 0.55, 0.5], [0.8, 0.2, 0.9]])


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


def scaled(k, arrays, factor):
    c, leaf, b = arrays
    t = mra.tree_import(k, c, leaf, b * factor)
    mra.compress(t)
    return t


@pytest.mark.parametrize("k", [3, 8])
@pytest.mark.parametrize("precision,screen", [("tc", "static"), ("tc", "pair"), ("tc_ladder", "static"),
                                              ("tc_ladder", "pair")])
def test_zero_blocks_leave_small_inputs_whole(k, precision, screen):
    """Leaves that are exactly zero beside leaves of any magnitude."""
    t, _ = OT.build_tree(DENS, k, 1e-3, 3, init_level=2)
    c, leaf, b = oracle_to_arrays(t, k)
    b[(c[:, 0] >= 2) & ((c[:, 1] + c[:, 2] + c[:, 3]) % 3 == 0)] = 0.0
    op = mra.make_operator(0.0, 1.0, 1e-5, k, 3)
    ref = mra.apply_ns(op, scaled(k, (c, leaf, b), 1.0), precision="fp64", screen=screen)[0].export()[2]
    one = None
    for e in (0, -27, -33, 27):
        g, _ = mra.apply_ns(op, scaled(k, (c, leaf, b), 2.0 ** e), precision=precision, screen=screen)
        out = g.export()[2] * 2.0 ** -e
        one = out if one is None else one
        assert rel(out, one) <= (1e-6 if precision == "tc" else 1e-5), e
        if precision == "tc":
            assert rel(out, ref) <= 2e-6, e
