"""Calls that take a kernel of their own by mode, size or addressing, against the general path or
the FP64 oracle."""
import numpy as np
import pytest

from paper_2203_12946_gb300 import elbm as E
from test_gpu_dispatch import raw_state
from test_gpu_parity import LAT, _cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,dims", [(2, (37, 5, 1)), (3, (7, 5, 3))])
def test_lbgk_adjoint_of_vanishing_populations(D, dims):
    """The LBGK reverse step does not depend on the departures: populations of 3e-22, whose
    departures overflow FP32 when squared, leave it finite and equal to the FP64 adjoint (6e-7 in
    the norm, the FP32 tolerance of test_gpu_adjoint)."""
    torch = pytest.importorskip("torch")
    f = raw_state(D, dims, "f32")
    f[:, ::3] = np.where(np.random.default_rng(3).random(f[:, ::3].shape) < 0.2, np.float32(3e-22), f[:, ::3])
    g = np.random.default_rng(4).standard_normal(f.shape).astype(np.float32)

    def adjoint(storage, dtype):
        with E.Simulation(LAT[D], dims, 0.97, storage=storage, alpha_mode=E.ELBM_ALPHA_LBGK) as sim:
            sim.set_populations(f.astype(dtype))
            return sim.adjoint_step(sim.state_copy(), torch.from_numpy(g.astype(dtype)).cuda()).cpu().numpy()

    want, got = adjoint("f64", np.float64), adjoint("f32", np.float32)
    assert np.all(np.isfinite(want))
    assert np.linalg.norm(got - want) <= 6e-7 * np.linalg.norm(want)
