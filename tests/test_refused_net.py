"""Net calls that are refused: a forward pass whose activations cannot be allocated, loss weights without a positive
sum, a tensor-core wait that runs out."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1508_07982_gb300 import lbm as mod
    return mod


class _Hook:
    """torch's caching allocator that refuses the k-th allocation, once."""

    def __init__(self, lbm):
        import torch
        self.torch, self.calls, self.fail_at, self.live = torch, 0, None, {}
        self.hook = lbm.Allocator(lbm.ALLOC_FN(self._alloc), lbm.RELEASE_FN(self._release), None)

    def _alloc(self, nbytes, stream, user):
        self.calls += 1
        if self.calls == self.fail_at:
            return None
        p = self.torch.cuda.caching_allocator_alloc(int(nbytes), stream=int(stream or 0))
        self.live[p] = int(nbytes)
        return p

    def _release(self, ptr, nbytes, stream, user):
        assert self.live.pop(int(ptr)) == int(nbytes)
        self.torch.cuda.caching_allocator_delete(int(ptr))


def _volumes(n):
    import torch
    g = torch.Generator(device="cuda").manual_seed(n)
    x = torch.zeros((n, 6, 6, 6, 16), dtype=torch.bfloat16, device="cuda")
    x[..., :6] = torch.randn((n, 6, 6, 6, 6), generator=g, device="cuda").to(torch.bfloat16)
    return x, torch.randn((n, 6, 6, 6, 4), generator=g, device="cuda")


@pytest.mark.parametrize("entry", ["forward", "predict", "train_step"])
def test_no_gradient_follows_a_forward_pass_that_was_refused(lbm, entry):
    """Three layers hold six buffers; growing them fails at each in turn."""
    (xs, ts), (xl, tl) = _volumes(2), _volumes(5)
    for k in range(1, 7):
        h = _Hook(lbm)
        net = lbm.Net(3, 6, 4, seed=5, allocator=h.hook)
        before, params = dict(h.live), net.params()
        z = net.forward(xs).float().cpu().numpy()
        loss = net.gradient(ts)
        assert len(h.live) == len(before) + 6
        h.calls, h.fail_at = 0, k
        with pytest.raises(lbm.LBMError) as e:
            net.train_step(xl, tl) if entry == "train_step" else getattr(net, entry)(xl)
        assert e.value.status == lbm.LBM_ENOMEM
        assert h.live == before
        for t in (ts, tl):
            with pytest.raises(lbm.LBMError) as e:
                net.gradient(t)
            assert e.value.status == lbm.LBM_EINVAL
        assert np.array_equal(net.params(), params)
        assert np.array_equal(net.forward(xs).float().cpu().numpy(), z)
        assert net.gradient(ts) == pytest.approx(loss, rel=1e-12)
        net.gradient(ts)
        net.close()
        assert h.live == {}


@pytest.mark.parametrize("reason", ["zero", "negative", "nan", "timeout"])
@pytest.mark.parametrize("entry", ["gradient", "train_step"])
def test_a_refused_gradient_keeps_the_gradients_and_parameters(lbm, reason, entry):
    import torch
    x, t = _volumes(3)
    net = lbm.Net(3, 6, 4, seed=6)
    net.train_step(x, t)
    grads, params = net.grads(), net.params()
    assert np.isfinite(grads).all() and np.abs(grads).max() > 0.0
    weight = {"zero": 0.0, "negative": -1.0, "nan": float("nan"), "timeout": 1.0}[reason] * torch.ones(x.shape[:-1], device="cuda")
    net.forward(x)
    net.set_wait_test(reason == "timeout")
    with pytest.raises(lbm.LBMError) as e:
        net.gradient(t, weight=weight) if entry == "gradient" else net.train_step(x, t, weight=weight)
    assert e.value.status == (lbm.LBM_ETIMEOUT if reason == "timeout" else lbm.LBM_EINVAL)
    net.set_wait_test(False)
    assert np.array_equal(net.grads(), grads) and np.array_equal(net.params(), params)
    # and the next gradient is that of a net with the same parameters (sums of 648 voxels in another order)
    ref = lbm.Net(3, 6, 4, seed=6)
    ref.set_params(params)
    out = []
    for n in (net, ref):
        n.forward(x)
        out.append((n.gradient(t), n.grads()))
        n.close()
    assert out[0][0] == pytest.approx(out[1][0], rel=1e-12)
    assert np.abs(out[0][1] - out[1][1]).max() <= 648 * 2.0 ** -23 * np.abs(out[1][1]).max()
