"""The sibling groups in batches: with room for the partial sums of a few groups at a time (an allocator that
refuses large blocks) the results are bit for bit those of one launch, for an apply and a plan."""
import numpy as np
import pytest

from paper_0706_0747_gb300 import workloads as W
from tests.test_gpu_network_memory import LimitAlloc

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_0706_0747_gb300 import mra  # noqa: E402

DENS = dict(coef=[3.0, 1.2, 0.4], expo=[40.0, 400.0, 3000.0], centers=[[0.42, 0.55, 0.5], [0.8, 0.2, 0.9], [0.3, 0.31, 0.7]],
            r2coef=[0.0, 0.0, 0.0])


@pytest.mark.parametrize("precision,k", [("fp64", 6), ("fp32", 7), ("tc", 8)])
def test_batches_of_groups(precision, k):
    mra.release_cached()
    out = []
    for limit in (1 << 40, 60 << 20):
        A = LimitAlloc(limit)
        t, _ = mra.build_tree(W.Density(**DENS), k, 1e-5, 4, init_level=4 if precision == "tc" else 3, allocator=A.hook)
        mra.compress(t)
        op = mra.make_operator(0.0, 1.0, 1e-6, k, 4, allocator=A.hook)
        g, st = mra.apply_ns(op, t, precision=precision)
        plan = mra.plan_create(op, [t, t], precision=precision)
        plan.execute()
        out.append((st["n_items"], g.export()[2], plan.output(0).export()[2], plan.output(1).export()[2]))
        assert (A.refused > 0) == (limit == 60 << 20)
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("k", [8, 12])
def test_d2_level_by_level(k):
    """d = 2 with room for the matrices of a few levels at a time (20 k^4 doubles a level)."""
    dens = W.unit_mass2(np.array([300.0, 5000.0]), np.array([[0.4, 0.55], [0.71, 0.27]]))
    out = []
    for limit in (1 << 40, 8 << 20 if k == 12 else 3 << 20):
        A = LimitAlloc(limit)
        t, _ = mra.build_tree2(dens, k, 1e-5, 6, init_level=4, allocator=A.hook)
        mra.compress2(t)
        op = mra.make_operator2(0.0, 0.5, 1e-3, k, 6, allocator=None)
        g, st = mra.apply_ns2(op, t)
        out.append((st["n_items"], st["n_ghosts"], g.export()[2]))
        assert (A.refused > 0) == (limit < 1 << 40)
    for a, b in zip(*out):
        assert np.array_equal(a, b)


def constant_net(logits):
    theta = np.zeros(mra.mlp_create().n_params, dtype=np.float32)
    theta[-12:] = np.tile(logits, 4)
    return mra.mlp_create(params=theta)


def test_learned_apply_without_room_for_the_groups():
    """The learned screen prepares the groups beside the pair lists; where they find no room the pair lists serve."""
    k, out = 6, []
    for limit in (1 << 40, 20 << 20):
        mra.release_cached()
        A = LimitAlloc(limit)
        t, _ = mra.build_tree(W.Density(**DENS), k, 1e-5, 4, init_level=3, allocator=A.hook)
        mra.compress(t)
        op = mra.make_operator(0.0, 1.0, 1e-6, k, 4)
        for logits in ([10.0, 0.0, 0.0], [-10.0, 0.0, 1.0]):  # every pair narrowed; none
            g, st = mra.apply_ns(op, t, precision="fp64", screen="learned", schedule=constant_net(logits), margin=0)
            out.append((st["n_items"], g.export()[2]))
        assert (A.refused > 0) == (limit == 20 << 20)
    assert [a[0] for a in out[:2]] == [a[0] for a in out[2:]]
    assert np.array_equal(out[0][1], out[2][1])
    assert np.abs(out[1][1] - out[3][1]).max() <= 1e-12 * np.abs(out[1][1]).max()


def test_learned_plan_keeps_one_way():
    """A plan whose network narrows pairs holds no more than a plan of the exact screen, and one whose network
    keeps every term no more than a static one, but for the network's own."""
    k = 6

    def held(screen, logits=None):
        mra.release_cached()
        A = LimitAlloc(1 << 40)
        t, _ = mra.build_tree(W.Density(**DENS), k, 1e-4, 4, init_level=2, allocator=A.hook)
        mra.compress(t)
        op = mra.make_operator(0.0, 1.0, 1e-5, k, 4)
        net = None
        if logits:
            net = constant_net(logits)
        plan = mra.plan_create(op, [t], precision="tc", use_graph=False, screen=screen, schedule=net, margin=0)
        plan.execute()
        out = plan.output(0).export()[2]
        info = plan.info()
        torch.cuda.synchronize()
        mra.release_cached()  # what is cached, not held
        size = A.held
        return size, out, info["n_pairs"], info["n_items"]

    pair, empty = held("pair"), held("learned", [10.0, 0.0, 0.0])
    static, full = held("static"), held("learned", [-10.0, 0.0, 1.0])
    for a, b in ((pair, empty), (static, full)):
        assert b[0] <= a[0] and b[2:] == a[2:] and np.array_equal(a[1], b[1])
