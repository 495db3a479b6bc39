"""The initial equilibrium on fields that are small somewhere, every
precision, against extended precision: spins of any size down to what the
storage rounds to zero, a fluid at rest at the reference density (its
deviations are exactly zero), slow flows (deviations down to the rounding of
the density).

Tolerances, from the arithmetic: a stored single- or half-precision value is
the rounding of an expression known to ~2^-45 of itself: half a last place and
a thousandth; a trace's deviation is the difference of values that the double
expression knows to 11 roundings of w_i P_i n, w_i < 1/2: 2^-50 n.  64-bit
storage: as test_gpu_sitesums, relative to the component, and the smallest
number where that ends."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LD = np.longdouble


@pytest.fixture(scope="module")
def q():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1309_1656_gb300 import qlbm
    return qlbm


def directions(d):
    return [(x, y, z) for z in ((-1, 0, 1) if d == 3 else (0,)) for y in (-1, 0, 1) for x in (-1, 0, 1)
            if abs(x) + abs(y) + abs(z) < 3]


def weights(k, d):
    return np.array([k[("w_rest", "w_axis", "w_diag")[sum(map(abs, v))]] for v in directions(d)])


def equilibrium(k, d, rho4, u, eps):
    K = LD(k["xi"]) ** 2 / 2
    j = [u[a].astype(LD) / k["xi"] for a in range(d)]
    a2 = 0 if eps is None else (eps.astype(LD) - k["c"]) / (k["m"] - LD(k["c"]) ** 2)
    out = []
    for v, w in zip(directions(d), weights(k, d)):
        t = sum(v[a] * j[a] for a in range(d))
        P = (1 - k["c"] * a2 + a2 * K * sum(map(abs, v)) + 2 * K * k["alpha3"] * t + 4 * K * K * k["alpha4"] * t * t +
             K * k["alpha5"] * sum(a * a for a in j))
        out.append(w * P * rho4.astype(LD))
    return np.stack(out)


def check(q, prec, d, dims, rho4, u, eps):
    with q.Lattice(d, dims, 0.8, 1.0, precision=prec) as lat:
        k = {name: LD(v) for name, v in lat.info().items()}
        lat.init_equilibrium(rho4, u, eps)
        img = lat.save_checkpoint()
        got = lat.get_state()
    want = equilibrium(k, d, rho4, u, eps)
    if prec in ("fp64", "df64"):
        rel, least = (2.0 ** -48, 2.0 ** -1072) if prec == "fp64" else (2.0 ** -46, 2.0 ** -126)
        assert np.all(np.abs(got - want) <= rel * np.abs(rho4).astype(LD) + least)
        return None
    w = weights(k, d)
    want[:, 0] -= w[:, None]
    stored = img.view(np.float32 if prec == "fp32" else np.float16).reshape(len(w), -1, 4).transpose(0, 2, 1)
    slack = np.zeros_like(want)
    slack[:, 0] = 2.0 ** -50 * np.abs(rho4[0])
    assert np.all(np.abs(stored.astype(LD) - want) <= 0.501 * np.spacing(np.abs(stored)).astype(LD) + slack)
    return stored


@pytest.mark.parametrize("prec", ["fp64", "df64", "fp32", "fp16dev"])
@pytest.mark.parametrize("d,dims", [(2, (45, 27, 1)), (3, (33, 7, 5))])
def test_spins_of_any_size(q, prec, d, dims):
    # every octave of the double range below 1, among others at the same site;
    # more of them where single and half precision end
    rng = np.random.default_rng(3)
    N = int(np.prod(dims))
    rho4 = rng.uniform(0.95, 1.05, (4, N))
    for c in (1, 2, 3):
        s = np.where(rng.random(N) < 0.5, rng.integers(0, 1074, N), rng.integers(0, 160, N))
        rho4[c] *= np.ldexp(rng.choice([-1.0, 1.0], N), -s)
    rho4[1, :1074] = np.ldexp(rng.uniform(0.5, 1.0, 1074), -np.arange(1074))
    rho4[2, ::13] = 0.0
    check(q, prec, d, dims, rho4, rng.uniform(-0.1, 0.1, (d, N)), None)


@pytest.mark.parametrize("prec", ["fp64", "df64", "fp32", "fp16dev"])
@pytest.mark.parametrize("d,dims", [(2, (45, 27, 1)), (3, (33, 7, 5))])
def test_fluid_at_rest(q, prec, d, dims):
    rng = np.random.default_rng(4)
    N = int(np.prod(dims))
    rho4 = 0.1 * rng.standard_normal((4, N))
    rho4[0] = 1.0
    rho4[0, 5::7] = np.nextafter(1.0, 2.0)      # almost
    rho4[0, 6::7] = np.nextafter(1.0, 0.0)
    u = np.zeros((d, N))
    u[:, ::2] = -0.0
    stored = check(q, prec, d, dims, rho4, u, None)
    if stored is not None:
        assert np.all(stored[:, 0, rho4[0] == 1.0] == 0)


@pytest.mark.parametrize("prec", ["fp32", "fp16dev"])
@pytest.mark.parametrize("given", [False, True])
@pytest.mark.parametrize("d,dims", [(2, (45, 27, 1)), (3, (33, 7, 5))])
def test_slow_flows(q, prec, given, d, dims):
    # velocities and density waves from 2^-10 down to 2^-60
    rng = np.random.default_rng(5)
    N = int(np.prod(dims))
    rho4 = 0.1 * rng.standard_normal((4, N))
    rho4[0] = 1.0 + rng.choice([-1.0, 0.0, 1.0], N) * 2.0 ** -rng.integers(10, 60, N)
    u = rng.standard_normal((d, N)) * 2.0 ** -rng.integers(10, 60, N)
    eps = None
    if given:
        with q.Lattice(d, dims, 0.8, 1.0, precision=prec) as lat:
            eps = lat.info()["c"] * (1.0 + rng.standard_normal(N) * 2.0 ** -rng.integers(10, 60, N))
    check(q, prec, d, dims, rho4, u, eps)
