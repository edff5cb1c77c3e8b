"""What the launches of a coarse step depend on: not the launch configuration (the tuner times the one mapping once),
but the schedule, side branches of a graph or one launch after another, which must not change a bit."""
import time

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


@pytest.mark.parametrize("batch", [False, True])
def test_the_tuner_times_the_steps_once(lbm, batch):
    """A run over every launch configuration would take 20 times as long as the steps themselves."""
    import torch
    case = inputs.periodic_case(n=128, B=16, collision="trt", omega=1.7)
    f = lbm.Forest(case, precision="fp32s")
    f.init_uniform((0.01, 0.0, 0.0))
    b = lbm.Batch([f]) if batch else f
    step = b.step if batch else b.step_coarse
    n = 2000
    for _ in range(2):
        step(2)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        step(n)
        torch.cuda.synchronize()
        steps = time.perf_counter() - t0
    t0 = time.perf_counter()
    _, _, ms = b.autotune(n)
    assert time.perf_counter() - t0 < 6 * steps
    assert 0.2 < ms * n * 1e-3 / steps < 2.0
    if batch:
        b.close()
    f.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32s", "fp16s"])
@pytest.mark.parametrize("H,B,inlet", [(32, 8, False), (32, 16, True), (64, 32, False)])
def test_side_branches_and_a_series_of_launches_give_the_same_bits(lbm, precision, H, B, inlet):
    """Bricks without a marked link, bricks that the sphere cuts, and coupled cells at every interface; with lbm_timing
    the same launches run one after another."""
    case = inputs.sphere_channel_case(H=H, B=B, inlet_outlet=inlet)
    graph, series = (lbm.Forest(case, precision=precision) for _ in range(2))
    for f in (graph, series):
        f.init_uniform(case["u_init"])
    graph.step_coarse(5)
    series.timing_begin(5)
    series.step_coarse(5)
    _, launches, _, explosions, _, side = series.timing_end(explode=True, side=True)
    assert (launches > 0).all() and (explosions[1:] > 0).all() and (precision == "fp64" or (side > 0).all())
    for L in range(graph.nlev):
        assert np.array_equal(graph.get_pdfs(L), series.get_pdfs(L), equal_nan=True), L
    assert np.array_equal(graph.reduce_mass_momentum(), series.reduce_mass_momentum())
    graph.close()
    series.close()
