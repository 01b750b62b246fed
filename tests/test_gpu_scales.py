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


@pytest.mark.parametrize("precision", ["tc", "tc_fast"])
def test_step2_at_the_edge_of_fp32(precision):
    """A coarse leaf whose refinement (Step 2) passes FP32's range is refused, one close to it is not."""
    k = 6
    t, _ = OT.build_tree(OT.Density([1.0], [4000.0], [[0.51, 0.49, 0.26]]), k, 1e-4, 5, init_level=1)
    c, leaf, b = oracle_to_arrays(t, k)
    b /= np.abs(b).max()
    op = mra.make_operator(0.0, 1.0, 1e-5, k, 5)
    # a coarse leaf: the lowest entry of its children 110 and 111 is (0.71 + 0.61)^2 0.71 = 1.23 of `top`
    i = int(np.flatnonzero(leaf)[0])
    assert c[i, 0] < c[:, 0].max() - 1
    for top, refused in ((1e30, False), (3.2e38, True)):
        x = b * 1e-3 * top
        x[i] = 0.0
        x[i, :2, :2, 0] = top
        tg = mra.tree_import(k, c, leaf, x)
        mra.compress(tg)
        ref, st = mra.apply_ns(op, tg, precision="fp64")
        assert st["n_ghosts"] > 0
        if refused:
            with pytest.raises(mra.MraError) as e:
                mra.apply_ns(op, tg, precision=precision)
            assert e.value.code == mra.EINVAL and "FP32" in str(e.value)
        else:
            got = mra.apply_ns(op, tg, precision=precision)[0]
            assert rel(got.export()[2], ref.export()[2]) <= 2e-6


@pytest.mark.parametrize("precision,screen", [("tc", "static"), ("tc", "pair"), ("tc_ladder", "static")])
def test_inputs_just_below_the_largest_float(precision, screen):
    """A root block whose scales leave FP32's exponents while their ratios do not: every term counts."""
    k = 4
    op = mra.make_operator(0.0, 1.0, 1e-5, k, 0)
    x = np.random.default_rng(5).uniform(-1e38, 1e38, (1, k, k, k))
    for top in (1e37, 1.7e38, 3.39e38):
        x[0, 0, 0, 0] = top
        tg = mra.tree_import(k, np.zeros((1, 4), np.int32), np.ones(1, np.int32), x)
        mra.compress(tg)
        ref, st = mra.apply_ns(op, tg, precision="fp64", screen=screen)
        got, stt = mra.apply_ns(op, tg, precision=precision, screen=screen)
        assert stt["n_items"] == st["n_items"] > 0
        assert rel(got.export()[2], ref.export()[2]) <= (2e-6 if precision == "tc" else 1e-5), top
