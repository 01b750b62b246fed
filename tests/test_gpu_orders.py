"""Kernels with an instance per order k (Algorithm 1, the pointwise multiply, the d = 2 apply, Step 2
in two floats) against the oracle at every order, and the schedule network at widths and addresses
that rule out whole 16-byte words.

Tolerances.  FP64 results: sums of at most 216 k^3 products, 1e-12 relative as the other parity tests.
The tensor-core apply against FP64: six operands rounded to 22 bits, 6 x 2^-22, and FP32 sums, 2e-6
(a Step-2 block wrong beyond its FP32 rounding would show).  Network: as test_gpu_schedule.py."""
import numpy as np
import pytest

from oracle import d2 as D, mlp as OM, product as OP, tree as OT
from tests.helpers import arrays_to_dict, oracle_to_arrays, rel_l2

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_0706_0747_gb300 import mra, workloads as W  # noqa: E402
from tests.test_gpu_d2 import apply_both, as_dicts  # noqa: E402


def many_terms(n, r2):
    """n Gaussians (one chunk of 32, its edge, or two), every third with an r^2 factor."""
    rng = np.random.default_rng(n)
    return dict(coef=rng.uniform(-2.0, 3.0, n), expo=10.0 ** rng.uniform(0.5, 3.0, n), centers=rng.random((n, 3)),
                r2coef=np.where(np.arange(n) % 3 == 0, 40.0 * r2, 0.0))


@pytest.mark.parametrize("k,n,r2", [(1, 3, False), (2, 33, True), (3, 1, True), (4, 32, False), (5, 64, True), (6, 7, False),
                                    (7, 33, False), (8, 31, True), (9, 5, True), (10, 32, True), (11, 2, False),
                                    (12, 33, True)])
def test_build_every_order(k, n, r2):
    kw = many_terms(n, r2)
    depth = 2 if k <= 4 else 3
    tg, hit = mra.build_tree(W.Density(**kw), k, 1e-4, depth, init_level=1)
    to, hit_o = OT.build_tree(OT.Density(**kw), k, 1e-4, depth, init_level=1)
    c, leaf, b, _ = tg.export()
    assert hit == hit_o
    co, lo, bo = oracle_to_arrays(to, k)
    assert np.array_equal(c, co) and np.array_equal(leaf != 0, lo != 0)
    assert np.abs(b - bo)[leaf != 0].max() <= 1e-12 * np.abs(bo).max()


@pytest.mark.parametrize("k", range(1, 13))
def test_multiply_every_order(k):
    kw = dict(coef=[2.0, -1.0], r2coef=[0.0, 3.0], expo=[5.0, 40.0], centers=[[0.4, 0.5, 0.6], [0.7, 0.2, 0.5]],
              charges=[-0.5], positions=[[0.31, 0.52, 0.77]])
    t, _ = OT.build_tree(OT.Density([1.0], [30.0], [[0.45, 0.5, 0.55]]), k, 1e-2, 2, init_level=1)
    out = mra.tree_multiply(mra.tree_import(k, *oracle_to_arrays(t, k)), mra.Potential(**kw), scale=0.75)
    ref = OP.multiply(t, k, OP.Potential(**kw), scale=0.75)
    c, leaf, b, _ = out.export()
    got = arrays_to_dict(c, b)
    keys = [key for key, node in ref.items() if node.leaf]
    scale = max(np.abs(ref[key].s).max() for key in keys)
    for key in keys:
        assert np.abs(got[key] - ref[key].s).max() <= 1e-12 * scale


@pytest.mark.parametrize("k", range(1, 13))
def test_stored_wavelets_every_order(k):
    """Blocks, norms and the inverse; a tree of one node has neither."""
    for depth in (0, 3):
        t, _ = OT.build_tree(OT.Density([1.0, 2.0], [30.0, 300.0], [[0.45, 0.5, 0.55], [0.8, 0.3, 0.2]]), k, 1e-2, depth,
                             init_level=min(depth, 1))
        tg = mra.tree_import(k, *oracle_to_arrays(t, k))
        _, leaf, leaves, _ = tg.export()
        mra.compress(tg, store_d=True)
        OT.compress(t, k)
        _, _, b, dn = tg.export()
        bo = oracle_to_arrays(t, k)[2]
        top = np.abs(bo).max()
        assert np.abs(b - bo).max() <= 1e-12 * top
        keys = [tuple(int(v) for v in c) for c in tg.export()[0]]
        for key, d in zip(keys, dn):
            if not t[key].leaf:
                assert abs(d - t[key].dnorm) <= 1e-12 * top * k ** 1.5
        mra.reconstruct(tg, mode="inverse")
        assert np.abs(tg.export()[2] - leaves)[leaf != 0].max() <= 1e-12 * top


@pytest.mark.parametrize("k", range(1, 13))
def test_apply2_every_order(k):
    """Leaf and internal siblings in a group, inputs refined from one and several levels above."""
    dens = D.Density2([1.0, 0.7], [60.0, 3000.0], [[0.4, 0.55], [0.71, 0.27]])
    to, _ = D.build_tree(dens, k, 1e-3, 4 if k <= 6 else 3, init_level=1)
    g, st, ghat, sto, *_ = apply_both(to, k, (0.0, 0.5, 1e-4, k, 4))
    assert (st["n_items"], st["n_pairs"]) == (sto["n_items"], sto["n_pairs"])
    assert rel_l2(as_dicts(g)[0], ghat) <= 1e-12


@pytest.mark.parametrize("k", [2, 3, 5, 6, 7, 8])
def test_step2_two_floats(k):
    """A narrow peak beside coarse leaves: missing inputs one to three levels below their leaf."""
    dens = W.Density(coef=[1.0], expo=[4000.0], centers=[[0.51, 0.49, 0.26]], r2coef=[0.0])
    t, _ = mra.build_tree(dens, k, 1e-4, 5, init_level=1)
    mra.compress(t)
    op = mra.make_operator(0.0, 1.0, 1e-5, k, 5)
    ref, _ = mra.apply_ns(op, t, precision="fp64")
    got, st = mra.apply_ns(op, t, precision="tc")
    assert st["n_ghosts"] > 0 or k == 2  # (k = 2 refines the whole cube)
    a, b = got.export()[2], ref.export()[2]
    assert np.linalg.norm(a - b) <= 2e-6 * np.linalg.norm(b)


@pytest.mark.parametrize("n_in,rows,shift", [(16, 1, 0), (16, 33, 1), (13, 31, 0), (18, 65, 2), (130, 40, 0), (16, 257, 3)])
def test_network_widths(n_in, rows, shift):
    rng = np.random.default_rng(n_in + rows)
    theta = OM.flatten([rng.normal(0.0, np.sqrt(2.0 / s[1]), s) if len(s) == 2 else rng.normal(0.0, 0.1, s)
                        for s in OM.param_shapes(n_in)]).astype(np.float32)
    x = rng.normal(0.0, 1.0, (rows, n_in)).astype(np.float32)
    t = np.zeros((rows, 12), dtype=np.float32)
    t[:, 1::3] = rng.random((rows, 4)) * 0.5
    t[:, 2::3] = t[:, 1::3] + 0.25
    net = mra.mlp_create(n_in=n_in, params=theta)
    room = torch.zeros(shift + rows * n_in, device="cuda")  # rows that start `shift` floats off a 16-byte boundary
    room[shift:] = torch.from_numpy(x.ravel()).cuda()
    xd = room[shift:].view(rows, n_in)
    y = torch.empty((rows, 12), device="cuda")
    net.forward(xd, y)
    loss, g = net.loss_grad(xd, torch.from_numpy(t).cuda())
    p64 = theta.astype(np.float64)
    ref, _ = OM.forward(OM.unflatten(p64, n_in), x.astype(np.float64))
    assert np.abs(y.cpu().numpy() - ref).max() <= 1e-3 * np.abs(ref).max()
    loss_o, g_o = OM.loss_grad(p64, x.astype(np.float64), t.astype(np.float64), n_in)
    assert abs(loss - loss_o) <= 1e-5 * abs(loss_o)
    o = 0
    for shp in OM.param_shapes(n_in):
        a, b = g[o:o + int(np.prod(shp))], g_o[o:o + int(np.prod(shp))]
        assert np.abs(a - b).max() <= 2e-3 * np.abs(b).max() + 1e-7, shp
        o += int(np.prod(shp))
