"""How results are rounded: where a value is formed in more bits than it is stored in, or by a
division or root of the library's own, it is the correctly rounded one."""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

import oracle as O
from paper_2203_12946_gb300 import build as B
from paper_2203_12946_gb300 import elbm as E
from paper_2203_12946_gb300 import inputs
from test_gpu_parity import LAT, _cuda, dev_ref  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    """Calls a function of device_probes.cu, or with D of lattice_probes.cu, built with the
    library's flags: arrays go in as device copies, the outputs (shape, dtype) come back as arrays."""
    torch = pytest.importorskip("torch")
    libs = {}

    def load(D):
        if D not in libs:
            lib = str(tmp_path_factory.mktemp("probes") / f"probes{D}.so")
            src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "lattice_probes.cu" if D else "device_probes.cu")
            subprocess.run([B.nvcc(), *B.ARCH, *B.NVCC_FLAGS, f"-DELBM_DIM={D}", "-shared", "-o", lib, src, "-cudart", "static"], check=True)
            libs[D] = ctypes.CDLL(lib)
        return libs[D]

    def call(name, ins, outs, *scalars, D=0):
        so = load(D)
        a = [torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in ins]
        o = [torch.from_numpy(np.zeros(shape, dtype)).cuda() for shape, dtype in outs]
        torch.cuda.synchronize()
        assert getattr(so, name)(*[ctypes.c_void_p(t.data_ptr()) for t in a + o], *scalars) == 0
        return [t.cpu().numpy() for t in o]

    return call


def same(a, b):
    return np.array_equal(a, b, equal_nan=True)


def doubles(rng, n, lo, hi):
    """Random significands and signs, binary exponents in [lo, hi)."""
    return np.ldexp(rng.uniform(1.0, 2.0, n), rng.integers(lo, hi, n)) * rng.choice([-1.0, 1.0], n)


# around the exponents where the library's forms end, and what they do not take
EDGES = np.array([0.0, -0.0, 5e-324, 1e-310, 2.0 ** -1022, 2.0 ** -501, 2.0 ** -500, 2.0 ** 500, 2.0 ** 1023,
                  np.nextafter(2.0 ** -500, 0), np.nextafter(2.0 ** 500, 0), 1.0, np.nextafter(1.0, 0), np.nextafter(2.0, 0),
                  1.7976931348623157e308, np.inf, np.nan])


def test_fp64_division_is_ieee(probe):
    """The FP64 collision's quotient against the correctly rounded one: the same number wherever
    the exact quotient is further than 2^-49 of a unit from the middle between two, so at every
    one of 2^20 random pairs (2^-28 of a chance that one of them is not), and outside the range of
    the library's form, which leaves those to the IEEE operation."""
    rng = np.random.default_rng(1)
    n = 1 << 18
    e = np.concatenate([EDGES, -EDGES, doubles(rng, 40, -520, -480), doubles(rng, 40, 480, 520)])
    a = np.concatenate([doubles(rng, n, -3, 3), doubles(rng, n, -60, 4), doubles(rng, n, -520, 520), doubles(rng, n, -1074, 1024),
                        np.repeat(e, e.size)])
    b = np.concatenate([doubles(rng, n, -3, 3), doubles(rng, n, -12, 8), doubles(rng, n, -520, 520), doubles(rng, n, -1074, 1024),
                        np.tile(e, e.size)])
    out, ieee = probe("probe_div", [a, b], [(a.shape, np.float64)] * 2, a.size)
    with np.errstate(all="ignore"):
        assert same(ieee, a / b)
    assert same(out, ieee)


def test_fp64_square_root_is_ieee(probe):
    """As test_fp64_division_is_ieee: 1/(2s) here is good to 2^-50."""
    rng = np.random.default_rng(2)
    n = 1 << 19
    e = np.concatenate([EDGES, -EDGES])
    a = np.concatenate([rng.uniform(1.0, 1.2, n), np.abs(doubles(rng, n, -520, 520)), np.abs(doubles(rng, n, -1074, 1024)), e])
    out, ieee = probe("probe_sqrt", [a], [(a.shape, np.float64)] * 2, a.size)
    with np.errstate(all="ignore"):
        assert same(ieee, np.sqrt(a))
    assert same(out, ieee)


def test_fp64_reciprocal_of_the_density(probe):
    """1/rho of the moments: r0 (1 + e + e^2) with |e| < 2^-22 is off by 2^-66 of it before its one
    rounding, against 2^-53 or more between two numbers: within one unit in the last place of the
    correctly rounded reciprocal, and that reciprocal but for one density in 2^12 at most; what the
    FP32 range cannot take is IEEE."""
    rng = np.random.default_rng(3)
    n = 1 << 20
    edges = np.concatenate([EDGES, -EDGES])
    rho = np.concatenate([rng.uniform(0.5, 2.0, n), doubles(rng, n, -120, 120), edges])
    (out,) = probe("probe_rcp64", [rho], [(rho.shape, np.float64)], rho.size, D=2)
    with np.errstate(all="ignore"):
        want = 1.0 / rho
    fp32 = (np.abs(rho) > 1e-30) & (np.abs(rho) < 1e30)
    assert np.all(np.abs(out[fp32] - want[fp32]) <= np.spacing(np.abs(want[fp32])))
    assert np.count_nonzero(out[fp32] != want[fp32]) <= 2 * n >> 12
    assert same(out[~fp32], want[~fp32])


@pytest.mark.parametrize("dev", [False, True])
@pytest.mark.parametrize("D", [2, 3])
def test_node_sums_are_exact_at_the_edges_of_their_forms(probe, D, dev):
    """rho and rho u of a node's FP32 values (deviations: with the reference) are the exact sums
    rounded once, by the split into two parts (up to 15 binades between a node's values, the
    largest in 2^-63 .. 2^65) and by the fixed-point form past it: values over 0 to 20 binades,
    exactly 15 and 16, all at the top of a binade, zeros among them, largest values on both sides
    of the range; not-finite values are refused."""
    rng = np.random.default_rng(31)
    Q, n = 3 ** D, 512
    top = np.float32(2.0 - 2.0 ** -23)  # largest significand

    def spread(b, at=-4):
        v = np.ldexp(rng.uniform(1.0, 2.0, (Q, n)), at - rng.integers(0, b + 1, (Q, n)))
        v[0], v[-1] = np.ldexp(rng.uniform(1.0, 2.0, n), at), np.ldexp(rng.uniform(1.0, 2.0, n), at - b)
        return v * rng.choice([-1.0, 1.0], (Q, n))

    blocks = [spread(b) for b in (0, 1, 8, 14, 15, 16, 17, 20)]
    blocks += [np.full((Q, n), 0.25) * top, np.full((Q, n), -0.25) * top, 0.25 * top * rng.choice([-1.0, 1.0], (Q, n))]
    blocks += [spread(15) * (rng.random((Q, n)) < p) for p in (0.9, 0.5, 0.1, 0.0)]
    low, high = (-14, 8) if dev else (-64, 66)  # binades of the largest value; 2^-63 and 2^64 end the split
    blocks += [spread(b, at) for at in (low, low + 1, low + 2, high - 2, high - 1, high) for b in (0, 15, 16)]
    v = np.concatenate(blocks, axis=1).astype(np.float32)
    R = float(np.float32(6.0 ** -D)) if dev else 0.0
    bad = np.repeat(v[:, :1], 3, axis=1)
    bad[[0, Q // 2, Q - 1], [0, 1, 2]] = np.inf, np.nan, -np.inf
    (out,) = probe("probe_exact_sums", [np.concatenate([v, bad], axis=1)], [((1 + D, v.shape[1] + 3), np.float64)],
                   v.shape[1] + 3, ctypes.c_float(R), D=D)
    assert np.all(out[:, -3:] == -1.0)
    vel = np.array([[(i // 3 ** (D - 1 - a)) % 3 - 1 for a in range(D)] for i in range(Q)])
    for k in range(v.shape[1]):
        col = v[:, k].astype(np.float64)
        assert out[0, k] == math.fsum([*col, 6 ** D * R]), k
        for a in range(D):
            assert out[1 + a, k] == math.fsum(vel[:, a] * col), (k, a)


@pytest.mark.parametrize("share", [0.5, 0.1, 0.01])
@pytest.mark.parametrize("q", [9, 27])
def test_sums_over_omega_minus_keep_their_digits(probe, q, share):
    """S_3..S_6, the sums of f x^k over x < 0, whose terms have one sign: within four roundings of
    a term and one of each addition of their exact value, however small the negative departures are
    next to the positive ones."""
    rng = np.random.default_rng(q)
    n = 4096
    f = (rng.uniform(0.2, 1.0, (q, n)) / q).astype(np.float32)
    x = rng.uniform(1e-3, 0.04, (q, n)) * np.where(rng.random((q, n)) < 0.5, 1.0, -share)
    x = x.astype(np.float32)
    (got,) = probe("probe_power_sums", [f, x], [((4, n), np.float32)], n, q)
    fd, xm = f.astype(np.float64), np.minimum(x.astype(np.float64), 0.0)
    for j in range(4):
        want = (fd * xm ** (3 + j)).sum(0)
        assert np.all(np.abs(got[j] - want) <= (4 + (q + 1) // 2 + 1) * 2.0 ** -24 * np.abs(want)), 3 + j


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


@pytest.mark.parametrize("storage", ["f32", "f32dev"])
@pytest.mark.parametrize("D,dims", [(2, (251, 200, 1)), (3, (41, 33, 29))])
def test_kinetic_energy_gradient_where_it_cancels(D, dims, storage):
    """dL/df_i = c_i . u - |u|^2 / 2 with u on the circle (sphere) where it vanishes for one c_i, to
    the rounding of the state: half a unit in the last place of the FP32 entry, and the few FP64
    roundings of u and of the sum (2^-50 of its terms)."""
    rng = np.random.default_rng(23)
    N = int(np.prod(dims))
    ux, uz = rng.uniform(-0.1, 0.1, N), rng.uniform(-0.05, 0.05, N) * (D == 3)
    u = np.stack([ux, 1.0 - np.sqrt(1.0 + 2.0 * ux - ux * ux - uz * uz), uz])[:D]
    f = O.init_equilibrium(D, rng.uniform(0.9, 1.1, N), u)
    c = dev_ref(D)[:, None] if storage == "f32dev" else np.zeros((1, 1))
    raw = (f - c).astype(np.float32)
    with E.Simulation(LAT[D], dims, 0.97, storage=storage) as sim:
        sim.set_populations(raw)
        got = sim.kinetic_energy(with_grad=True)[1].cpu().numpy()
    F = c.astype(np.longdouble) + raw.astype(np.longdouble)
    vel = [[(i // 3 ** (D - 1 - a)) % 3 - 1 for a in range(D)] for i in range(3 ** D)]
    rho = F.sum(0)
    v = [sum(ci[a] * F[i] for i, ci in enumerate(vel)) / rho for a in range(D)]
    uu = sum(w * w for w in v)
    size = (sum(np.abs(w) for w in v) + uu).astype(np.float64)
    for i, ci in enumerate(vel):
        want = sum(ci[a] * v[a] for a in range(D)) - uu / 2
        tol = 0.5 * np.spacing(np.abs(got[i])).astype(np.float64) + 2.0 ** -50 * size
        assert np.all(np.abs(got[i].astype(np.longdouble) - want) <= tol), ci


@pytest.mark.parametrize("D,dims", [(2, (131, 40, 1)), (3, (21, 13, 9))])
def test_fp32_start_of_thin_matter_is_rounded_once(D, dims):
    """As test_fp32_start_is_rounded_once (test_gpu_dispatch), for densities of 1e-28 to 1e-20, whose
    second FP32 part is small but counts."""
    N = int(np.prod(dims))
    rng = np.random.default_rng(37)
    rho, u = 10.0 ** rng.uniform(-28, -20, N), 0.08 * rng.standard_normal((D, N))
    want = O.init_equilibrium(D, rho, u)
    with E.Simulation(LAT[D], dims, 0.97, storage="f32") as sim:
        sim.init_equilibrium(rho, u)
        got = sim.get_populations()
    assert np.all(np.abs(got - want) <= 0.5 * np.spacing(got).astype(np.float64) + 2.0 ** -44 * want)
