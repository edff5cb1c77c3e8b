"""The velocity read-out of cells whose directions along one axis hold values far below the others'."""
from fractions import Fraction

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


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("rho0", [1.0, 1.7])
@pytest.mark.parametrize("precision", ["fp32s", "fp16s"])
def test_a_small_component_keeps_the_bits_of_its_own_values(lbm, precision, rho0, axis):
    """The stored value of a population f is f - w rho0 rounded to the storage type.  A component
    is a sum over the ten directions that move along its axis: FP64 additions are off by at most 18 x 2^-53 of the sum
    of those values' sizes, and the division by 2^-53 of the result."""
    case = inputs.periodic_case(n=8, B=8)
    case["rho0"] = rho0
    f = lbm.Forest(case, precision=precision)
    f.init_uniform()
    e, w, _ = lbm.lbm_lattice()
    rng = np.random.default_rng(7 + axis)
    n = 512
    v = 500.0 * rng.uniform(0.5, 1.0, (19, n)) * rng.choice([-1.0, 1.0], (19, n))
    along = np.asarray(e)[:, axis] != 0
    v[along] *= 2.0 ** -(np.arange(n) % 45)
    v[np.flatnonzero(along)[0], ::5] = 0.0
    base = (w * rho0)[:, None]
    pd = base + v
    f.set_pdfs(0, pd)
    with np.errstate(over="ignore", under="ignore"):
        stored = (pd - base).astype(np.float32 if precision == "fp32s" else np.float16).astype(np.float64)
    _, u = f.get_macroscopic(0)
    for i in range(n):
        j = sum(int(e[q][axis]) * Fraction(float(stored[q, i])) for q in range(19)) / Fraction(rho0)
        size = float(sum(abs(Fraction(float(stored[q, i]))) for q in range(19) if along[q])) / rho0
        assert abs(float(Fraction(float(u[axis, i])) - j)) <= 18 * 2.0 ** -53 * size + 2.0 ** -53 * abs(float(j)), (i, u[axis, i], float(j))
    f.close()
