"""GPU paths that the library chooses by size, type or alignment, at the sizes where the choice
or the split of the work changes, against the general path or the FP64 oracle."""
import numpy as np
import pytest

from paper_2203_12946_gb300 import elbm as E
from test_gpu_parity import LAT, MODES, _cuda, dev_ref, noisy_state, stored  # noqa: F401

pytestmark = pytest.mark.gpu


def raw_state(D, dims, storage, eps=4e-3, seed=5):
    """A noisy state as the storage holds it (set_populations input)."""
    f = noisy_state(D, dims, eps, seed=seed)
    if storage == "f64":
        return f
    if storage in ("f32", "f32dev"):
        return stored(D, f, storage)[0]
    d = f - dev_ref(D)[:, None]
    if storage == "f16dev":
        return d.astype(np.float16)
    torch = pytest.importorskip("torch")
    return torch.from_numpy(d).to(torch.bfloat16).view(torch.int16).numpy().view(np.uint16)


def run(D, dims, f0, chunks, storage, force=None, **kw):
    """Raw populations after the given step() calls, as bytes."""
    torch = pytest.importorskip("torch")
    with E.Simulation(LAT[D], dims, 0.97, storage=storage, **kw) as sim:
        sim.set_populations(f0)
        if force is not None:
            sim.set_force(np.asarray(force)[:D])
        for n in chunks:
            sim.step(n)
        assert sim.steps == sum(chunks)
        out = sim.state_copy()
        sim.synchronize()
        return torch.as_tensor(out).cpu().view(torch.uint8).numpy().copy()


@pytest.mark.parametrize("storage", ["f32", "f32dev", "f16dev", "bf16dev"])
@pytest.mark.parametrize("dims", [(1, 1, 1), (5, 7, 1), (31, 3, 1), (33, 2, 1), (64, 64, 1), (65, 9, 1), (97, 31, 1),
                                  (128, 33, 1), (129, 12, 1), (7, 304, 1), (64, 305, 1)])
def test_several_steps_per_launch_equal_single_steps(dims, storage):
    """Small D2Q9 domains take up to four steps per launch under AUTO: any split of the steps
    gives the bits of one launch per step (DIRECT)."""
    f0 = raw_state(2, dims, storage)
    for force, mode in ((None, "higher"), ((1e-4, -2e-4, 0.0), "higher"), (None, "iterate1")):
        kw = dict(storage=storage, force=force, alpha_mode=MODES[mode][0])
        want = run(2, dims, f0, [13], kernel=E.ELBM_KERNEL_DIRECT, **kw)
        for chunks in ([13], [1, 2, 3, 7], [4, 9], [5, 8]):
            assert np.array_equal(run(2, dims, f0, chunks, **kw), want), (force, mode, chunks)
