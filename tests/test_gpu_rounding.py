"""How results are rounded: where a value is formed in more bits than it is stored in, or by a
division or root of the library's own, it is the correctly rounded one."""
import numpy as np
import pytest

import oracle as O
from paper_2203_12946_gb300 import elbm as E
from paper_2203_12946_gb300 import inputs
from test_gpu_parity import LAT, _cuda, dev_ref  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["f16dev", "bf16dev"])
@pytest.mark.parametrize("D,dims", [(2, (1, 1, 1)), (2, (523, 301, 1)), (3, (41, 33, 29))])
def test_16_bit_start_is_rounded_once(D, dims, storage):
    """16-bit starts hold the FP64 equilibrium rounded once: within half a unit in the last place
    of the stored value, plus the 2^-44 of f^eq that the evaluation may be off.  A value rounded
    to FP32 on the way misses that by up to 2^-25 of itself, at one value in 2^14."""
    X, Y, Z = inputs.grid(dims)
    rng = np.random.default_rng(17)
    rho, u = 1.0 + 0.1 * rng.standard_normal(X.size), 0.08 * rng.standard_normal((D, X.size))
    want = O.init_equilibrium(D, rho, u)
    with E.Simulation(LAT[D], dims, 0.97, storage=storage) as sim:
        sim.init_equilibrium(rho, u)
        got = sim.get_populations()
    if storage == "f16dev":
        unit = np.spacing(np.abs(got)).astype(np.float64)
        got = got.astype(np.float64)
    else:
        got = (got.astype(np.uint32) << 16).view(np.float32).astype(np.float64)
        unit = 2.0 ** (np.floor(np.log2(np.maximum(np.abs(got), 2.0 ** -126))) - 7)
    assert np.all(np.abs(got - (want - dev_ref(D)[:, None])) <= 0.5 * unit + 2.0 ** -44 * want)
