"""The FP64 step on the integer pipes against the step in extended precision,
where its layout and its fixed-point form can go wrong: rows around the 8-site
chunks of a warp, both parities and the two-buffer step, components of very
different size, zero components, and sites outside the form's range (stepped
in double).

The reference is the step of Sec. 3.3 in numpy's long double with the handle's
own constants (the double-precision oracle's rounding, tens of 2^-53 on random
populations, is larger than what is looked for here).  Tolerance per step,
relative to the component's largest value on the lattice: 64 x 2^-53.  The
step errs by at most ~4 x 2^-53 of it (two basis terms, the 96-bit products,
one rounding); the sites stepped in double by the sums of b <= 19 terms, the
equilibrium's ~12 roundings and the update's three."""
import numpy as np
import pytest

from paper_1309_1656_gb300 import fields

pytestmark = pytest.mark.gpu

TOL = 64 * 2.0 ** -53


@pytest.fixture(scope="module")
def q():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1309_1656_gb300 import qlbm
    return qlbm


def worst(got, exp):
    """Largest error of the four components, each relative to its largest value."""
    return max(float(np.max(np.abs(got[:, c] - exp[:, c])) / max(np.max(np.abs(exp[:, c])), 1e-300)) for c in range(4))


def reference(q, d, dims, tau, st, n, dt=1.0, phi=None):
    """n steps in long double; phi [3][N or 1]: rotation vector of the field term (Eqs. DiscrAvr, WeqAlgo, CollisionStep, TransportStep)."""
    with q.Lattice(d, dims, tau, 1.0, dt=dt, precision="fp64") as lat:
        k = {name: np.longdouble(v) for name, v in lat.info().items()}
    nx, ny, nz = dims
    e = [(x, y, z) for z in ((-1, 0, 1) if d == 3 else (0,)) for y in (-1, 0, 1) for x in (-1, 0, 1)
         if abs(x) + abs(y) + abs(z) < 3]
    w = [k[("w_rest", "w_axis", "w_diag")[sum(map(abs, v))]] for v in e]
    omega, W = np.longdouble(dt / tau), st.astype(np.longdouble)
    K = k["xi"] ** 2 / 2
    for _ in range(n):
        rho = W.sum(0)
        j = [sum(v[a] * W[i, 0] for i, v in enumerate(e)) / rho[0] for a in range(3)]
        jj = sum(a * a for a in j)
        E = sum(sum(map(abs, v)) * W[i, 0] for i, v in enumerate(e)) / rho[0]
        a2 = (K * (E - jj) - k["c"]) / (k["m"] - k["c"] ** 2)
        new = []
        for i, v in enumerate(e):
            t = sum(v[a] * j[a] for a in range(3))
            P = (1 - k["c"] * a2 + a2 * K * sum(map(abs, v)) + 2 * K * k["alpha3"] * t +
                 4 * K * K * k["alpha4"] * t * t + K * k["alpha5"] * jj)
            c = W[i] + omega * (w[i] * P * rho - W[i])
            if phi is not None:     # Rodrigues
                th = np.sqrt((phi * phi).sum(0))
                a = phi / th
                s, dot = c[1:], (a * c[1:]).sum(0)
                cross = np.stack([a[1] * s[2] - a[2] * s[1], a[2] * s[0] - a[0] * s[2], a[0] * s[1] - a[1] * s[0]])
                c = np.concatenate([c[:1], np.cos(th) * s + np.sin(th) * cross + (1 - np.cos(th)) * dot * a])
            c = c.reshape(4, nz, ny, nx)
            new.append(np.roll(c, (v[2], v[1], v[0]), (1, 2, 3)).reshape(4, -1))
        W = np.stack(new)
    return W


def step(q, d, dims, tau, st, n, dt=1.0):
    with q.Lattice(d, dims, tau, 1.0, dt=dt, precision="fp64") as lat:
        lat.set_state(st)
        lat.step(n)
        return lat.get_state()


@pytest.mark.parametrize("tau", [0.5, 0.8, 10.0])
@pytest.mark.parametrize("d,dims", [(2, (1, 1, 1)), (2, (7, 3, 1)), (2, (8, 1, 1)), (2, (9, 5, 1)), (2, (33, 64, 1)),
                                    (3, (2, 3, 1)), (3, (8, 4, 5)), (3, (15, 2, 3)), (3, (17, 9, 4))])
def test_rows_around_a_chunk(q, d, dims, tau):
    st = fields.random_populations(d, dims, seed=17)
    st[:, 1:] -= 0.5 * st[:, 1:].mean(axis=0)
    for n in (1, 2, 3):
        assert worst(step(q, d, dims, tau, st, n), reference(q, d, dims, tau, st, n)) < n * TOL


@pytest.mark.parametrize("scale,spin", [(1.0, 0.0), (1.0, 1e-12), (2.0 ** -80, 1.0), (2.0 ** 60, 1e-3)])
@pytest.mark.parametrize("d,dims", [(2, (21, 6, 1)), (3, (11, 5, 3))])
def test_component_sizes(q, d, dims, scale, spin):
    st = fields.random_populations(d, dims, seed=23) * scale
    st[:, 1:] *= spin
    st[:, 2] = 0.0
    for n in (1, 2):
        got = step(q, d, dims, 0.7, st, n)
        assert worst(got, reference(q, d, dims, 0.7, st, n)) < n * TOL
        assert not got[:, 2].any()


@pytest.mark.parametrize("d,dims", [(2, (19, 4, 1)), (3, (9, 4, 3))])
def test_sites_outside_the_form(q, d, dims):
    # a fast site (|j| > 1/2), a tiny one and an ordinary rest: warps with and
    # without sites that are stepped in double
    st = fields.random_populations(d, dims, seed=29)
    b = st.shape[0]
    st[b - 1, 0, 3] += 2.0
    st[:, :, 20] *= 2.0 ** -1000
    assert worst(step(q, d, dims, 0.9, st, 1), reference(q, d, dims, 0.9, st, 1)) < TOL
    # omega > 2 leaves the form for the whole lattice
    st = fields.random_populations(d, dims, seed=31)
    got = step(q, d, dims, 1.0, st, 1, dt=2.5)
    assert worst(got, reference(q, d, dims, 1.0, st, 1, dt=2.5)) < 2 * TOL


# the flag looks at tr rho, |S| and beta0 eps (the double step's test): a
# rest population beyond the range leaves all three finite (E2/n = J/n = 0)
@pytest.mark.parametrize("value,direction,code", [(np.nan, 4, -5), (np.inf, 4, 0), (1e200, 4, 0), (-1e3, 4, -6),
                                                  (np.inf, 8, -5), (np.nan, 0, -5)])
def test_flags(q, value, direction, code):
    st = fields.random_populations(2, (24, 3, 1), seed=37)
    st[direction, 0, 30] = value
    with q.Lattice(2, (24, 3, 1), 0.8, 1.0, precision="fp64") as lat:
        lat.set_state(st)
        lat.step(1)
        got = 0
        try:
            lat.sync()
        except q.QLBMError as e:
            got = e.code
        assert got == code


@pytest.mark.parametrize("d,dims", [(2, (26, 7, 1)), (3, (13, 6, 5))])
def test_two_buffer_step_is_the_same(q, d, dims):
    # a rollout that keeps every state steps between two buffers
    st = fields.random_populations(d, dims, seed=41)
    with q.Lattice(d, dims, 0.7, 1.0, precision="fp64") as lat:
        lat.set_state(st)
        lat.rollout(5, 1)
        got = lat.get_state()
    assert np.array_equal(got, step(q, d, dims, 0.7, st, 5))


@pytest.mark.parametrize("scale", [1.0, 0.25])
@pytest.mark.parametrize("d,dims", [(2, (32, 4, 1)), (3, (16, 4, 2))])
def test_density_near_a_power_of_two(q, d, dims, scale):
    # 1/n at both ends of its normalised range: n = scale (1 +- 2^-k), k = 1..53
    st = fields.random_populations(d, dims, seed=43)
    b, N = st.shape[0], st.shape[2]
    st *= 0.5 / st[:, 0].sum(0)
    k = np.arange(N) % 54
    n = np.where(np.arange(N) < N // 2, 1.0 + 2.0 ** -k.astype(float), 1.0 - 2.0 ** -(k + 1.0))
    st[b // 2, 0] += n - st[:, 0].sum(0)
    st *= scale
    for steps in (1, 2):
        got = step(q, d, dims, 0.8, st, steps)
        assert worst(got, reference(q, d, dims, 0.8, st, steps)) < steps * TOL
    with q.Lattice(d, dims, 0.8, 1.0, precision="fp64") as lat:
        lat.set_state(st)
        r, u, eps = lat.moments()
        xi = lat.info()["xi"]
    e = [(x, y, z) for z in ((-1, 0, 1) if d == 3 else (0,)) for y in (-1, 0, 1) for x in (-1, 0, 1)
         if abs(x) + abs(y) + abs(z) < 3]
    f = st[:, 0].astype(np.longdouble)
    j = [sum(v[a] * f[i] for i, v in enumerate(e)) / f.sum(0) for a in range(d)]
    E = sum(sum(map(abs, v)) * f[i] for i, v in enumerate(e)) / f.sum(0)
    assert np.max(np.abs(u - xi * np.stack(j))) < TOL
    assert np.max(np.abs(eps - 0.5 * xi * xi * (E - sum(a * a for a in j)))) < 4 * TOL


@pytest.mark.parametrize("kind", ["uniform", "site"])
@pytest.mark.parametrize("prec", ["fp64", "fp64df"])
@pytest.mark.parametrize("d,dims", [(2, (19, 4, 1)), (3, (9, 4, 3))])
def test_magnetic_field(q, d, dims, prec, kind):
    # the rotation folded into the relaxation, and by warps that step in double
    st = fields.random_populations(d, dims, seed=47)
    st[:, 1] *= 1e-3                    # spin components of different size
    N = st.shape[2]
    B = fields.normal(7, 1, 3 * N).reshape(3, N)
    if kind == "uniform":
        B = B[:, :1].copy()
    phi = 2 * np.longdouble(0.4) * B.astype(np.longdouble)
    for n in (1, 2):
        # for one step also a site outside the fixed-point form (its density
        # is negative after the second)
        st[-1, 0, 3] += 2.0 if n == 1 else -2.0
        with q.Lattice(d, dims, 0.7, 1.0, precision=prec) as lat:
            if kind == "site":
                lat.set_magnetic_field_array(0.4, B)
            else:
                lat.set_magnetic_field(0.4, B[:, 0])
            lat.set_state(st)
            lat.step(n)
            got = lat.get_state()
        exp = reference(q, d, dims, 0.7, st, n, phi=phi)
        # the rotation mixes the components: relative to the largest
        assert np.max(np.abs(got - exp)) < n * TOL * np.abs(exp).max()


def test_double_float_precision_beyond_omega_2(q):
    # QLBM_FP64_DF is stepped by the same kernel there, in double
    st = fields.random_populations(3, (9, 4, 3), seed=53)
    with q.Lattice(3, (9, 4, 3), 1.0, 1.0, dt=2.5, precision="fp64df") as lat:
        lat.set_state(st)
        lat.step(1)
        got = lat.get_state()
    assert worst(got, reference(q, 3, (9, 4, 3), 1.0, st, 1, dt=2.5)) < 2 * TOL
