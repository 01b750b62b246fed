"""Memory of the network's training pass: each network has its own buffers whatever stream it trains on,
and a batch trains with what room the allocator has.

Tolerances: networks trained side by side on two streams end with the bits of networks trained one
after the other (no sum of the weight gradients depends on scheduling).  With fewer row slices the
gradient's FP32 sums of at most 4,096 rows are formed in another order: 1e-4 of a tensor's maximum."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_0706_0747_gb300 import mra  # noqa: E402


HOOKS = []  # the library keeps blocks that were freed: a hook outlives its last handle


class LimitAlloc:
    """torch caching-allocator hook that refuses blocks of more than `limit` bytes."""

    def __init__(self, limit):
        self.limit, self.refused, self.sizes = limit, 0, {}

        def _alloc(nbytes, stream, ctx):
            if nbytes > self.limit:
                self.refused += 1
                return None
            p = torch.cuda.caching_allocator_alloc(int(nbytes), torch.cuda.current_device(), stream or 0)
            self.sizes[p] = int(nbytes)
            return p

        def _free(ptr, stream, ctx):
            self.sizes.pop(ptr)
            torch.cuda.caching_allocator_delete(ptr)

        self._fa, self._ff = mra.ALLOC_FN(_alloc), mra.FREE_FN(_free)
        self.hook = mra.Alloc(self._fa, self._ff, None)
        HOOKS.append(self)

    @property
    def held(self):
        return sum(self.sizes.values())


def batch(seed, rows=4096):
    rng = np.random.default_rng(seed)
    t = rng.random((rows, 12)).astype(np.float32)
    t[:, ::3] = t[:, ::3] < 0.3
    return (torch.from_numpy(rng.normal(0.0, 1.0, (rows, 16)).astype(np.float32)).cuda(), torch.from_numpy(t).cuda())


def test_two_networks_on_two_streams():
    data, steps = [batch(1), batch(2)], 50
    alone = []
    for i, (x, t) in enumerate(data):
        net = mra.mlp_create(seed=i)
        for _ in range(steps):
            net.train_step(x, t, 1e-3)
        alone.append(net.get_params())
    nets = [mra.mlp_create(seed=i) for i in range(2)]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for _ in range(steps):
        for net, s, (x, t) in zip(nets, streams, data):
            net.train_step(x, t, 1e-3, stream=s)
    torch.cuda.synchronize()
    for net, ref in zip(nets, alone):
        assert np.array_equal(net.get_params(), ref)


def test_training_with_little_room():
    x, t = batch(3)
    ref = mra.mlp_create(seed=7).loss_grad(x, t)
    A = LimitAlloc(5 << 19)  # the activations of 4,096 rows fit (2 MB each), 64 slices of gradients (9.5 MB) do not
    loss, g = mra.mlp_create(seed=7, allocator=A.hook).loss_grad(x, t)
    assert A.refused > 0
    assert abs(loss - ref[0]) <= 1e-6 * abs(ref[0])
    assert np.abs(g - ref[1]).max() <= 1e-4 * np.abs(ref[1]).max()
