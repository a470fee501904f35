"""Calls that take a kernel of their own by mode, size or addressing, against the general path or
the FP64 oracle."""
import numpy as np
import pytest

import oracle as O
from paper_2203_12946_gb300 import elbm as E
from test_gpu_dispatch import raw_state
from test_gpu_parity import LAT, _cuda, dev_ref  # noqa: F401

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


def step_error(D, dims, storage, force=None):
    """Largest error of one step without the cutoff against the oracle on the same stored state, in
    units of what test_gpu_dispatch allows it: 1e-12 relative in FP64, 2e-6 in FP32, and half a unit
    of the stored FP16 deviation on top for 16-bit storage."""
    raw = raw_state(D, dims, storage)
    c = dev_ref(D)[:, None] if storage.endswith("dev") else 0.0
    want = O.step(D, dims, c + raw.astype(np.float64), 0.97, cutoff=False, force=force)[0]
    with E.Simulation(LAT[D], dims, 0.97, storage=storage, cutoff=False) as sim:
        sim.set_populations(raw)
        sim.set_force(force)
        sim.step(1)
        got = c + sim.get_populations().astype(np.float64)
    tol = (1e-12 if storage == "f64" else 2e-6) * np.abs(want)
    if storage == "f16dev":
        tol = tol + 2.0 ** -11 * np.abs(want - c) + 2.0 ** -25
    return np.max(np.abs(got - want) / tol)


# one node per thread: nz above the grid's limit; two nodes per thread (D2Q9, FP32 arithmetic): ny
@pytest.mark.parametrize("force", [False, True])
@pytest.mark.parametrize("D,dims,storage", [
    *[(3, d, st) for st in ("f64", "f32", "f32dev", "f16dev") for d in [(2, 2, 65537), (1, 1, 65536), (3, 1, 65601)]],
    *[(2, d, st) for st in ("f32", "f32dev", "f16dev") for d in [(2, 65537, 1), (1, 65536, 1), (65, 65536, 1)]]])
def test_step_beyond_the_grid_limit(D, dims, storage, force):
    """Sides above 65,535 take a grid over all nodes and 64-bit indices."""
    assert step_error(D, dims, storage, np.array([1e-4, -2e-4, 5e-5])[:D] if force else None) <= 1.0


@pytest.mark.parametrize("storage", ["f32", "f32dev"])
@pytest.mark.parametrize("dims", [(81, 81, 82), (82, 82, 81)])
def test_step_around_the_l2_line(dims, storage):
    """D3Q27 steps of FP32 take another instantiation where both buffers fill 112 MiB or less: 538,002
    and 544,644 nodes are the last and the first such box on either side of 543,706."""
    assert step_error(3, dims, storage) <= 1.0


@pytest.mark.parametrize("storage", ["f32", "f32dev", "f16dev"])
@pytest.mark.parametrize("force", [False, True])
@pytest.mark.parametrize("dims", [(1, 1, 65537), (2, 3, 65536)])
def test_adjoint_step_beyond_the_grid_limit(dims, storage, force):
    """nz above 65,535 takes a grid over all nodes and 64-bit indices: against the FP64 adjoint of the
    same state (6e-7 in the norm, the FP32 tolerance of test_gpu_adjoint), and the force's derivative,
    a sum over the nodes in FP64 of FP32 values, to 1e-5 of the sum of their sizes over sqrt(N)."""
    torch = pytest.importorskip("torch")
    F = np.array([1e-4, -2e-4, 5e-5]) if force else None
    raw = raw_state(3, dims, storage)
    c = dev_ref(3)[:, None] if storage.endswith("dev") else 0.0
    g = np.random.default_rng(7).standard_normal(raw.shape).astype(np.float32)

    def adjoint(st, state, g):
        with E.Simulation(E.ELBM_D3Q27, dims, 0.97, storage=st, cutoff=False) as sim:
            sim.set_populations(state)
            sim.set_force(F)
            dF = torch.zeros(3, dtype=torch.float64, device="cuda") if force else None
            h = sim.adjoint_step(sim.state_copy(), torch.from_numpy(g).cuda(), dF).cpu().numpy()
            return h, None if dF is None else dF.cpu().numpy()

    want, dF_want = adjoint("f64", c + raw.astype(np.float64), g.astype(np.float64))
    got, dF = adjoint(storage, raw, g)
    assert np.linalg.norm(got - want) <= 6e-7 * np.linalg.norm(want)
    if force:
        assert np.max(np.abs(dF - dF_want)) <= 1e-5 * np.sqrt(raw.shape[1])


def test_adjoint_step_beyond_4_gb():
    """More than 2^32 bytes of FP32 gradient take 64-bit indices: a periodic tiling of a small state
    and gradient stays the tiling of the small result."""
    torch = pytest.importorskip("torch")
    small, tiles = (64, 32, 1), (172, 344, 1)
    big = tuple(s * t for s, t in zip(small, tiles))
    raw = raw_state(2, small, "f32")
    g = torch.from_numpy(np.random.default_rng(7).standard_normal(raw.shape).astype(np.float32)).cuda()

    def tiled(t):
        return t.view(9, small[1], small[0]).repeat(1, tiles[1], tiles[0])

    with E.Simulation(E.ELBM_D2Q9, small, 0.97, storage="f32", cutoff=False) as a:
        want = tiled(a.adjoint_step(torch.from_numpy(raw).cuda(), g))
    with E.Simulation(E.ELBM_D2Q9, big, 0.97, storage="f32", cutoff=False) as b:
        assert b.pop_bytes > 2 ** 32
        state, grad = tiled(torch.from_numpy(raw).cuda()).contiguous(), tiled(g).contiguous()
        got = b.adjoint_step(state, grad)
        torch.cuda.synchronize()
        assert bool((torch.abs(got - want) <= 4e-6 * torch.abs(want).max()).all())


@pytest.mark.parametrize("offset", [0, 16, 8, 1])
@pytest.mark.parametrize("D,dims,storage", [(2, (1, 1, 1), "f16dev"), (2, (227, 1, 1), "f32"), (3, (41, 13, 9), "f64")])
def test_ensemble_copies_leave_their_neighbours_alone(D, dims, storage, offset):
    """Populations of an ensemble's domain into a part of a device buffer: the batch works on a stream
    of its own, so the buffer is filled and the device waited for before the copy."""
    torch = pytest.importorskip("torch")
    raw = raw_state(D, dims, storage)
    with E.Ensemble(LAT[D], [dims, dims], [0.9, 0.9], storage=storage) as ens:
        n = raw.nbytes
        E.elbm_batch_set_populations(ens.b, 1, raw, E.ELBM_MEM_HOST)
        out = torch.full((n + 64,), 0xA5, dtype=torch.uint8, device="cuda")
        torch.cuda.synchronize()
        E.elbm_batch_get_populations(ens.b, 1, out[offset:offset + n], E.ELBM_MEM_DEVICE)
        torch.cuda.synchronize()
        want = np.full(n + 64, 0xA5, np.uint8)
        want[offset:offset + n] = np.ascontiguousarray(raw).view(np.uint8).ravel()
        assert np.array_equal(out.cpu().numpy(), want)
