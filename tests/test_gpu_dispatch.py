"""GPU paths that the library chooses by size, type or alignment, at the sizes where the choice
or the split of the work changes, against the general path or the FP64 oracle."""
import numpy as np
import pytest

import oracle as O
from paper_2203_12946_gb300 import elbm as E
from paper_2203_12946_gb300 import inputs
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


# one node per thread: blocks of consecutive nodes of a plane, smaller ones for small domains
# (plane sizes around the block sizes 32 to 256, planes of one node); D2Q9 FP32: rows around the
# 64-node runs of a warp, whose interior ones take the second node's address from the first's
@pytest.mark.parametrize("D,storage,dims", [
    *[(2, "f64", d) for d in [(1, 1, 1), (33, 1, 1), (1, 63, 1), (13, 5, 1), (96, 96, 1), (257, 3, 1)]],
    *[(3, "f64", d) for d in [(1, 1, 1), (8, 4, 65), (43, 3, 2)]],
    *[(3, st, d) for st in ("f32", "f32dev", "f16dev")
      for d in [(1, 1, 1), (1, 127, 1), (129, 1, 2), (16, 8, 3), (3, 43, 2), (1, 1, 67), (40, 33, 31)]],
    *[(2, st, (nx, 3, 1)) for st in ("f32", "f32dev", "f16dev")
      for nx in (1, 2, 31, 32, 33, 63, 64, 65, 66, 127, 128, 129, 191, 193, 257, 320)]])
def test_one_step_at_block_edges(D, storage, dims):
    """One step without the cutoff (every node solves for alpha) against the oracle on the same
    stored state: 1e-12 relative in FP64, 2e-6 in FP32 (test_gpu_parity), and half a unit of the
    stored FP16 deviation, 2^-11 of it, on top of that for 16-bit storage."""
    raw = raw_state(D, dims, storage)
    c = dev_ref(D)[:, None] if storage.endswith("dev") else 0.0
    want = O.step(D, dims, c + raw.astype(np.float64), 0.97, cutoff=False)[0]
    with E.Simulation(LAT[D], dims, 0.97, storage=storage, cutoff=False) as sim:
        sim.set_populations(raw)
        sim.step(1)
        got = c + sim.get_populations().astype(np.float64)
    tol = (1e-12 if storage == "f64" else 2e-6) * np.abs(want)
    if storage == "f16dev":
        tol = tol + 2.0 ** -11 * np.abs(want - c) + 2.0 ** -25
    assert np.all(np.abs(got - want) <= tol)


@pytest.mark.parametrize("D,small,tiles", [(3, (32, 32, 16), (11, 11, 21)), (2, (64, 32, 1), (172, 344, 1))])
def test_populations_beyond_4_gb(D, small, tiles):
    """More than 2^32 bytes of FP32 populations take element offsets instead of byte offsets: a
    periodic tiling of a small state stays the tiling of the small domain's result."""
    torch = pytest.importorskip("torch")
    raw = raw_state(D, small, "f32")
    big = tuple(s * t for s, t in zip(small, tiles))
    with E.Simulation(LAT[D], small, 0.97, storage="f32") as a:
        a.set_populations(raw)
        a.step(2)
        want = a.state_copy().view(torch.float32).view(a.Q, *small[::-1])
    with E.Simulation(LAT[D], big, 0.97, storage="f32") as b:
        assert b.pop_bytes > 2 ** 32
        start = torch.from_numpy(raw).cuda().view(b.Q, *small[::-1]).repeat(1, *tiles[::-1])
        start = start.contiguous().view(-1).view(torch.uint8)
        want = want.repeat(1, *tiles[::-1])
        b.restore(start)
        b.step(2)
        got = b.state_copy().view(torch.float32).view(b.Q, *big[::-1])
        assert bool((torch.abs(got - want) <= 4e-6 * torch.abs(want)).all())
    with E.Ensemble(LAT[D], [small, big], [0.97, 0.97], storage="f32") as c:
        torch.cuda.synchronize()
        E.elbm_batch_set_populations(c.b, 1, start, E.ELBM_MEM_DEVICE)
        E.elbm_batch_set_populations(c.b, 0, raw, E.ELBM_MEM_HOST)
        c.step(2)
        E.elbm_batch_get_populations(c.b, 1, start, E.ELBM_MEM_DEVICE)
        c.synchronize()
        got = start.view(torch.float32).view(3 ** D, *big[::-1])
        assert bool((torch.abs(got - want) <= 4e-6 * torch.abs(want)).all())


@pytest.mark.parametrize("storage", ["f32", "f32dev"])
@pytest.mark.parametrize("D,dims", [(2, (1, 1, 1)), (2, (255, 1, 1)), (2, (257, 3, 1)), (3, (5, 3, 17)), (3, (41, 33, 29))])
def test_fp32_start_is_rounded_once(D, dims, storage):
    """FP32 starts hold the FP64 equilibrium rounded once: within half a unit in the last place
    of the stored value, plus the 2^-44 of f^eq that the double-float evaluation may be off."""
    X, Y, Z = inputs.grid(dims)
    rng = np.random.default_rng(11)
    rho, u = 1.0 + 0.1 * rng.standard_normal(X.size), 0.08 * rng.standard_normal((D, X.size))
    want = O.init_equilibrium(D, rho, u)
    c = dev_ref(D)[:, None] if storage == "f32dev" else 0.0
    with E.Simulation(LAT[D], dims, 0.97, storage=storage) as sim:
        sim.init_equilibrium(rho, u)
        got = sim.get_populations()
    tol = 0.5 * np.spacing(np.abs(got)).astype(np.float64) + 2.0 ** -44 * want
    assert np.all(np.abs(got.astype(np.float64) - (want - c)) <= tol)


@pytest.mark.parametrize("storage", ["f32", "f32dev"])
@pytest.mark.parametrize("D,dims", [(2, (1, 1, 1)), (2, (255, 1, 1)), (2, (257, 3, 1)), (3, (5, 3, 17)), (3, (41, 33, 29))])
def test_kinetic_energy_of_fp32_states(D, dims, storage):
    """Energy of an FP32 state to 1e-12 (FP64 sums of exact products), its gradient rounded once
    to FP32 (2^-23 of the largest entry)."""
    raw = raw_state(D, dims, storage)
    c = dev_ref(D)[:, None] if storage == "f32dev" else 0.0
    L_o, g_o = O.kinetic_energy(D, c + raw.astype(np.float64))
    with E.Simulation(LAT[D], dims, 0.97, storage=storage) as sim:
        sim.set_populations(raw)
        L, g = sim.kinetic_energy(with_grad=True)
    assert abs(L - L_o) <= 1e-12 * L_o
    assert np.max(np.abs(g.cpu().numpy().astype(np.float64) - g_o)) <= 2.0 ** -23 * np.max(np.abs(g_o))


@pytest.mark.parametrize("storage", ["f32", "f32dev"])
@pytest.mark.parametrize("force", [False, True])
@pytest.mark.parametrize("D,dims", [(2, (65, 9, 1)), (2, (1, 129, 1)), (3, (1, 1, 3)), (3, (17, 8, 5))])
def test_adjoint_step_on_both_sides_of_the_series(D, dims, storage, force):
    """The FP32 adjoint takes a power series where |x| allows it and the general form elsewhere:
    states whose |x| lies below, around and above the line, against the FP64 adjoint, which is the
    general form (6e-7 in the norm, the FP32 tolerance of test_gpu_adjoint)."""
    torch = pytest.importorskip("torch")
    F = np.array([1e-4, -2e-4, 5e-5])[:D] if force else None

    def adjoint(st, state, g):
        with E.Simulation(LAT[D], dims, 0.97, storage=st, cutoff=False) as sim:
            sim.set_populations(state)
            sim.set_force(F)
            dF = torch.zeros(D, dtype=torch.float64, device="cuda") if force else None
            return sim.adjoint_step(sim.state_copy(), torch.from_numpy(g).cuda(), dF).cpu().numpy()

    for eps in (1e-3, 0.02, 0.04, 0.06):
        raw = raw_state(D, dims, storage, eps=eps)
        c = dev_ref(D)[:, None] if storage == "f32dev" else 0.0
        g = np.random.default_rng(7).standard_normal(raw.shape).astype(np.float32)
        want = adjoint("f64", c + raw.astype(np.float64), g.astype(np.float64))
        got = adjoint(storage, raw, g)
        assert np.linalg.norm(got - want) <= 6e-7 * np.linalg.norm(want), eps


@pytest.mark.parametrize("D,dims,storage", [(2, (128, 64, 1), "f32"), (2, (300, 200, 1), "f16dev"), (3, (24, 20, 16), "f32")])
def test_kernels_of_a_stream_see_each_other_and_the_callers(D, dims, storage):
    """Kernels may become resident before the previous one of the stream has ended; what they
    read and write stays ordered with each other's, the caller's kernels on the same stream, and
    those of another stream ordered by events: the bits of a run that synchronises every call."""
    torch = pytest.importorskip("torch")
    raw = raw_state(D, dims, storage)

    def go(sync, other):
        wait = torch.cuda.synchronize if sync else (lambda: None)
        with E.Simulation(LAT[D], dims, 0.97, storage=storage) as sim:
            sim.set_populations(raw)
            states = []
            for k in range(12):
                sim.step(1 + k % 3)
                wait()
                buf = sim.state_copy()
                wait()
                if other is not None and k % 2:
                    other.wait_stream(sim.stream)
                    with torch.cuda.stream(other):
                        moved = buf.view(sim.Q, -1).roll(dims[0] * buf.element_size(), 1)
                    sim.stream.wait_stream(other)
                    moved.record_stream(sim.stream)
                    buf.record_stream(other)
                else:
                    moved = buf.view(sim.Q, -1).roll(dims[0] * buf.element_size(), 1)
                wait()
                sim.restore(moved.contiguous().view(-1))
                wait()
                states.append(sim.state_copy())
                wait()
            torch.cuda.synchronize()
            return torch.stack(states).cpu()

    want = go(True, None)
    assert torch.equal(go(False, None), want)
    assert torch.equal(go(False, torch.cuda.Stream()), want)


@pytest.mark.parametrize("where", ["plain", "captured"])
@pytest.mark.parametrize("offset", [0, 16, 8, 1])
@pytest.mark.parametrize("D,dims,storage", [(2, (1, 1, 1), "f16dev"), (2, (7, 1, 1), "f32"), (2, (227, 1, 1), "f32"),
                                            (2, (3641, 1, 1), "f16dev"), (3, (41, 13, 9), "f64")])
def test_device_copies_of_populations(D, dims, storage, offset, where):
    """Copies between device buffers, by the library's kernel where both ends lie on 16 bytes and
    by the driver elsewhere: sizes with and without bytes left over, around one block's 8 KB,
    nothing written beside them; also under capture."""
    torch = pytest.importorskip("torch")
    raw = raw_state(D, dims, storage)
    with E.Simulation(LAT[D], dims, 0.97, storage=storage) as sim, \
            E.Ensemble(LAT[D], [dims, dims], [0.9, 0.9], storage=storage) as ens:
        n = sim.pop_bytes
        out = torch.full((n + 64,), 0xA5, dtype=torch.uint8, device="cuda")
        dst = out[offset:offset + n]
        sim.set_populations(raw)
        if where == "captured":
            E.elbm_get_populations(sim.h, dst, E.ELBM_MEM_DEVICE)  # a first call outside
            out.fill_(0xA5)
            torch.cuda.synchronize()
            graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
            E.elbm_set_stream(sim.h, side.cuda_stream)
            with torch.cuda.graph(graph, stream=side):
                E.elbm_get_populations(sim.h, dst, E.ELBM_MEM_DEVICE)
            graph.replay()
        else:
            E.elbm_get_populations(sim.h, dst, E.ELBM_MEM_DEVICE)
        torch.cuda.synchronize()
        want = np.full(n + 64, 0xA5, np.uint8)
        want[offset:offset + n] = np.ascontiguousarray(raw).view(np.uint8).ravel()
        assert np.array_equal(out.cpu().numpy(), want)
        if where == "captured":
            return
        sim.set_populations(np.zeros_like(raw))
        E.elbm_set_populations(sim.h, dst, E.ELBM_MEM_DEVICE)
        E.elbm_batch_set_populations(ens.b, 1, dst, E.ELBM_MEM_DEVICE)
        assert np.array_equal(sim.get_populations(), raw)
        assert np.array_equal(ens.get_populations(1), raw)
        out.fill_(0xA5)
        E.elbm_batch_get_populations(ens.b, 1, dst, E.ELBM_MEM_DEVICE)
        torch.cuda.synchronize()
        assert np.array_equal(out.cpu().numpy(), want)
