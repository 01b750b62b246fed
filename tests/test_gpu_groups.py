"""The sibling-group apply of the static screen (apply_oct.cu, apply_oct_tc.cu) against the oracle
where it can go wrong: every order k, trees of one node, uniform trees (every neighbour inside or
outside the cube), ragged trees with leaf and internal siblings in one group, the unscreened
schedule (every class of every term, pieces beyond one chunk), and a batch of different depths.

Tolerances: FP64 1e-12 relative as the other parity tests; FP32 sums of at most 216 k^3 products
of 24-bit factors in three nested stages, 1e-5; the tensor cores the 10 eps gate."""
import numpy as np
import pytest

from oracle import apply as OA, operator as OO, tree as OT
from tests.helpers import arrays_to_dict, oracle_to_arrays, rel_l2

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_0706_0747_gb300 import mra  # noqa: E402

EPS, J = 1e-3, 3
DENS = OT.Density([3.0, 1.2], [40.0, 400.0], [[0.42, 0.55, 0.5], [0.8, 0.2, 0.9]])


def trees(k):
    ragged, _ = OT.build_tree(DENS, k, EPS, J, init_level=1)
    uniform, _ = OT.build_tree(DENS, k, EPS, 2, uniform_level=2)
    root, _ = OT.build_tree(DENS, k, EPS, 0, uniform_level=0)
    out = [ragged, uniform, root]
    for t in out:
        OT.compress(t, k)
    return out


def on_gpu(t, k):
    tg = mra.tree_import(k, *oracle_to_arrays(t, k))
    mra.compress(tg)
    return tg


@pytest.mark.parametrize("k", [1, 2, 3, 5, 7, 8, 9, 10, 11, 12])
def test_groups_every_order(k):
    op_o, op_g = OO.Operator(0.0, 1.0, EPS, k, J), mra.make_operator(0.0, 1.0, EPS, k, J)
    ts = trees(k)[: 3 if k <= 8 else 1]
    for t in ts:
        st_o = {}
        ref = OA.apply_ns(op_o, t, stats=st_o)
        tg = on_gpu(t, k)
        for precision, tol in (("fp64", 1e-12), ("fp32", 1e-5), ("tc", 10 * EPS)):
            if precision == "tc" and k > 8:
                continue
            g, st = mra.apply_ns(op_g, tg, precision=precision)
            assert (st["n_items"], st["n_pairs"], st["n_ghosts"]) == \
                (st_o["n_items"], st_o["n_pairs"], st_o["n_refined"])
            c, _, b, _ = g.export()
            assert rel_l2(arrays_to_dict(c, b), ref) <= tol, (k, precision)
    for precision in ("fp64", "tc")[: 2 if k <= 8 else 1]:
        tg = [on_gpu(t, k) for t in ts]
        plan = mra.plan_create(op_g, tg, precision=precision)
        plan.execute()
        for b, t in enumerate(tg):
            one, _ = mra.apply_ns(op_g, t, precision=precision)
            assert np.array_equal(plan.output(b).export()[2], one.export()[2])


@pytest.mark.parametrize("k", [4, 6])
def test_groups_unscreened(k):
    op_o, op_g = OO.Operator(1.5, 1.0, EPS, k, J), mra.make_operator(1.5, 1.0, EPS, k, J)
    t = trees(k)[0]
    ref = OA.apply_ns(op_o, t, screen=False)
    tg = on_gpu(t, k)
    for precision, tol in (("fp64", 1e-12), ("tc", 10 * EPS)):
        c, _, b, _ = mra.apply_ns(op_g, tg, precision=precision, unscreened=True)[0].export()
        assert rel_l2(arrays_to_dict(c, b), ref) <= tol
