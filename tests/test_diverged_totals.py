"""The totals of a state with one NaN population: the components it does not enter stay finite."""
import ctypes

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


@pytest.mark.parametrize("q", [0, 1, 5, 10, 15])
@pytest.mark.parametrize("precision", ["fp64", "fp32s", "fp16s"])
def test_a_nan_enters_the_totals_through_its_own_direction(lbm, precision, q):
    """The step records the moments its collision starts from, so after one step the NaN has moved one cell and enters
    the mass and the components of its direction; a step later all populations of that cell are NaN and enter all."""
    case = inputs.periodic_case(n=16, B=8, collision="trt", omega=1.6)
    f = lbm.Forest(case, precision=precision)
    f.init_uniform((0.02, -0.01, 0.03))
    e, _, _ = lbm.lbm_lattice()
    pd = f.get_pdfs(0)
    pd[q, 700] = np.nan
    f.set_pdfs(0, pd)
    out = (ctypes.c_double * 4)()
    for step in range(2):
        f.step_coarse(1)
        assert lbm.library().lbm_reduce_mass_momentum(f.h, out) == lbm.LBM_ENONFINITE
        hit = [True] + [bool(e[q][a]) or step == 1 for a in range(3)]
        assert np.isnan(np.array(out)).tolist() == hit
        assert (~np.isfinite(f.get_pdfs(0))).any(axis=0).sum() == (1 if step == 0 else 19)
        assert np.isnan(f.get_pdfs(0)).sum() == (1 if step == 0 else 19) * 19
    f.close()
