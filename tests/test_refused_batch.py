"""A batch whose launch tables cannot be allocated: every refusal is reported, nothing is kept of the tables, and the
next step builds them whole."""
import numpy as np
import pytest

from paper_1508_07982_gb300 import inputs

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


def _members(lbm, precision):
    fs = [lbm.Forest(c, precision=precision) for c in inputs.batch_cases(n=3, seed=3)]
    for f in fs:
        f.init_uniform()
    return fs


@pytest.mark.parametrize("entry", ["step", "launches"])
@pytest.mark.parametrize("precision", ["fp64", "fp32s"])
def test_a_refused_table_leaves_no_partial_step(lbm, precision, entry):
    alone = _members(lbm, precision)
    for f in alone:
        f.step_coarse(3)
    want = [[f.get_pdfs(L) for L in range(f.nlev)] for f in alone]
    h = _Hook(lbm)
    whole = lbm.Batch(_members(lbm, precision), allocator=h.hook)
    launches = whole.launches_per_coarse_step()
    total = h.calls
    assert total >= 4 * launches
    whole.close()
    for k in {1, 2, 3, 4, 5, total // 2, total - 1, total}:
        h.calls, h.fail_at = 0, k
        members = _members(lbm, precision)
        b = lbm.Batch(members, allocator=h.hook)
        with pytest.raises(lbm.LBMError) as e:
            b.step(1) if entry == "step" else b.launches_per_coarse_step()
        assert e.value.status == lbm.LBM_ENOMEM and h.calls == k
        assert h.live == {}, "tables of a step that was not built"
        assert b.launches_per_coarse_step() == launches
        b.step(3)
        for f, w in zip(members, want):
            for L in range(f.nlev):
                assert np.array_equal(f.get_pdfs(L), w[L], equal_nan=True)
        b.close()
        assert h.live == {}
