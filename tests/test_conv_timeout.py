"""The bounded waits of the tcgen05 convolution: whichever wait of a unit's last two planes runs out, in whichever warp,
all four draining warps leave together.  On the CPU every interleaving of the flag protocol is walked through; on the
GPU the waits run out with nothing in flight (the net's wait test)."""
import os
import re

import pytest

WARPS = 4


def _stuck(flag_of):
    """Whether some interleaving of two successive drains leaves a warp at the warps' barrier for ever.  A drain is: set
    its flag if the wait ran out, meet the other warps, read the flag and leave if it is set."""
    # state: per warp (drain, step), step 0 wait, 1 at the barrier, 2 released; the flags
    start = (((0, 0),) * WARPS, (0, 0))
    seen, todo = {start}, [start]
    while todo:
        warps, flags = todo.pop()
        nexts = []
        if all(w[1] == 1 for w in warps):
            nexts.append((tuple((d, 2) for d, _ in warps), flags))
        for i, (d, s) in enumerate(warps):
            def go(w, f=flags):
                nexts.append((warps[:i] + (w,) + warps[i + 1:], f))
            if d == 2:
                continue
            if s == 0:
                go((d, 1))
                go((d, 1), tuple(1 if k == flag_of(d) else v for k, v in enumerate(flags)))
            elif s == 2:
                go((2, 0) if flags[flag_of(d)] else (d + 1, 0))
        if not nexts and any(d < 2 for d, _ in warps):
            return True
        for n in nexts:
            if n not in seen:
                seen.add(n)
                todo.append(n)
    return False


def test_the_warps_that_drain_agree_in_every_interleaving():
    assert _stuck(lambda d: 0)                 # one flag for both: a late reader can leave alone
    assert not _stuck(lambda d: d & 1)
    src = open(os.path.join(os.path.dirname(__file__), "..", "paper_1508_07982_gb300", "csrc", "net.cu")).read()
    drain = src[src.index("auto drain = [&](int z)"):]
    drain = drain[:drain.index("tcgen05.fence::after_thread_sync")]
    assert "const int h = z & 1;" in drain
    used = re.findall(r"(\*fail|fail\[\w+\])", drain)
    assert used == ["fail[h]", "fail[h]"], used


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(1, 1, 5, 5), (2, 2, 9, 61), (3, 3, 8, 8), (400, 18, 18, 18)])
def test_a_wait_that_runs_out_in_units_of_any_depth(shape):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1508_07982_gb300 import lbm
    g = torch.Generator(device="cuda").manual_seed(9)
    x = torch.zeros(shape + (16,), dtype=torch.bfloat16, device="cuda")
    x[..., :6] = torch.randn(shape + (6,), generator=g, device="cuda").to(torch.bfloat16)
    net = lbm.Net(2, 6, 4, seed=3)
    z = net.forward(x)
    for _ in range(3):
        net.set_wait_test(True)
        with pytest.raises(lbm.LBMError) as e:
            net.forward(x)
        assert e.value.status == lbm.LBM_ETIMEOUT
        net.set_wait_test(False)
        assert torch.equal(net.forward(x), z)
    net.close()
