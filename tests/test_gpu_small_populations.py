"""The FP64 step population by population: each result against the step in
long double, relative to the terms it is a sum of rather than to the largest
value around it, where populations or spin components of a site are far apart
and at small omega = dt / tau.

Tolerance.  With v the population before the step, M the component's sum, A_i
= 1 + |alpha2| (c + K |i|^2) + |c3 t| + |c4 t^2| + |c5 jj| the sum of the
absolute terms of P_i and T = |v| + omega w_i A_i |M|, a step in double errs by
2^-53 of: v, the product omega h M and their sum once each, and the
coefficients' own roundings, at most ~4 of omega w_i A_i |M|: 8 x 2^-53 T.  Sums
M of populations of one sign err by a few 2^-53 of M more: 16 x 2^-53 T in all.
The fixed-point form (omega from 0.65 on) errs by 1.3 x 2^-56 of the component's
largest value at the site, which is at most b times |M| for populations of one
sign: within the same bound there, as omega w_i A_i >= 0.65 / 36 x A_i and A_i
is at least 1.  A field's rotation R mixes the bounds: sum_b |R_ab| T_b, and
8 x 2^-53 sum_b |R_ab| max |W_b| for the fixed-point form's common alignment of
what it mixes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LD = np.longdouble
U = LD(2) ** -53


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


def rotation(phi):
    """Rodrigues' matrix [3][3][N] of the rotation vectors phi [3][N], and the
    products a_i a_j of its axis."""
    th = np.sqrt((phi * phi).sum(0))
    a = phi / np.where(th > 0, th, 1)
    R = np.zeros((3, 3, phi.shape[1]), dtype=LD)
    for i in range(3):
        for j in range(3):
            R[i, j] = 2 * np.sin(th / 2) ** 2 * a[i] * a[j] + (np.cos(th) if i == j else 0)
    for i, j, k in ((0, 1, 2), (1, 2, 0), (2, 0, 1)):
        R[i, j] -= np.sin(th) * a[k]
        R[j, i] += np.sin(th) * a[k]
    return R, np.abs(a[:, None] * a[None])


def step_and_bound(k, d, dims, omega, st, phi=None):
    nx, ny, nz = dims
    e = directions(d)
    omega, W = LD(omega), st.astype(LD)
    w = [k[("w_rest", "w_axis", "w_diag")[sum(map(abs, v))]] for v in e]
    K = LD(0.5 * (6.0 * float(k["m"]) / ((d + 2.0) * float(k["c"]))))      # as the handle has it (beta0 = 1)
    rho = W.sum(0)
    j = [sum(v[a] * W[i, 0] for i, v in enumerate(e)) / rho[0] for a in range(3)]
    jj = sum(a * a for a in j)
    E = sum(sum(map(abs, v)) * W[i, 0] for i, v in enumerate(e)) / rho[0]
    a2 = (K * (E - jj) - k["c"]) / (k["m"] - k["c"] ** 2)
    big = np.abs(W).max(0)
    out, bound = [], []
    for i, v in enumerate(e):
        m = sum(map(abs, v))
        t = sum(v[a] * j[a] for a in range(3))
        terms = [1 + 0 * t, -k["c"] * a2, a2 * K * m, 2 * K * k["alpha3"] * t, 4 * K * K * k["alpha4"] * t * t,
                 K * k["alpha5"] * jj]
        P, A = sum(terms), 1 + np.abs(a2) * (k["c"] + K * m) + sum(np.abs(x) for x in terms[3:])
        c = W[i] + omega * (w[i] * P * rho - W[i])
        b = 16 * U * (np.abs(W[i]) + omega * w[i] * A * np.abs(rho))
        if phi is not None:
            R, aa = rotation(phi)
            mix = lambda M, x: np.concatenate([x[:1], np.einsum("abn,bn->an", M, x[1:])])
            c, b = mix(R, c), mix(np.abs(R), b + 8 * U * big)
            b[0] -= 8 * U * big[0]
            if phi.shape[1] == 1:       # (the uniform field's matrix is formed with 1 - cos: 2^-53 a_i a_j)
                b[1:] += np.einsum("abn,bn->an", 2 * U * aa, np.abs(W[i, 1:]) + omega * w[i] * A * np.abs(rho[1:]))
        roll = lambda x: np.roll(x.reshape(4, nz, ny, nx), (v[2], v[1], v[0]), (1, 2, 3)).reshape(4, -1)
        out.append(roll(c))
        bound.append(roll(b))
    return np.stack(out), np.stack(bound)


def run(q, d, dims, omega, st, prec="fp64", field=None):
    with q.Lattice(d, dims, 1.0 / omega, 1.0, precision=prec) as lat:
        k = {name: LD(v) for name, v in lat.info().items()}
        if field is not None:
            if field.shape[1] == 1:
                lat.set_magnetic_field(0.4, field[:, 0])
            else:
                lat.set_magnetic_field_array(0.4, field)
        lat.set_state(st)
        lat.step(1)
        got = lat.get_state()
    assert np.isfinite(got).all()
    phi = None if field is None else 2 * LD(0.4) * field.astype(LD)
    want, bound = step_and_bound(k, d, dims, 1.0 / LD(1.0 / omega), st, phi)
    assert np.all(np.abs(got - want) <= bound)


def one_outweighs(d, dims, small):
    """Rest populations of 1 and all others near `small`, every component of
    one sign."""
    rng = np.random.default_rng(11 + d)
    b = len(directions(d))
    st = small * rng.uniform(0.5, 1.5, (b, 4, int(np.prod(dims))))
    st[b // 2] = rng.uniform(0.5, 1.0, st[b // 2].shape)
    st[:, 2] *= -1
    return st


@pytest.mark.parametrize("omega", [1.9, 1.25, 0.75, 0.66, 0.5, 0.1, 0.01, 0.001])
@pytest.mark.parametrize("small", [1e-2, 1e-6, 1e-12])
@pytest.mark.parametrize("d,dims", [(2, (21, 5, 1)), (3, (9, 5, 3))])
def test_small_populations(q, d, dims, small, omega):
    run(q, d, dims, omega, one_outweighs(d, dims, small))


# rotations about a coordinate axis leave one component alone; others mix
# all three, weakly for the small field
@pytest.mark.parametrize("omega", [1.25, 0.5, 0.01])
@pytest.mark.parametrize("axis", [(0, 0, 1), (0, 1, 0), (0.7, 0, 0), (0.3, -0.4, 0.5), (1e-7, 2e-7, 1e-7)])
@pytest.mark.parametrize("site", [False, True])
@pytest.mark.parametrize("d,dims", [(2, (21, 5, 1)), (3, (9, 5, 3))])
def test_small_spin_components_in_a_field(q, d, dims, site, axis, omega):
    rng = np.random.default_rng(5)
    b, N = len(directions(d)), int(np.prod(dims))
    st = np.empty((b, 4, N))
    w = np.array([(1 / 3, 1 / 18, 1 / 36)[sum(map(abs, v))] for v in directions(d)])
    st[:] = w[:, None, None] * rng.uniform(0.8, 1.2, st.shape)
    st[:, 1, :] *= 10.0 ** -rng.integers(0, 14, N)
    st[:, 2, :] *= 10.0 ** -rng.integers(0, 14, N)
    st[:, 3, :] *= 10.0 ** -rng.integers(0, 14, N)
    st[:, 2, ::7] = 0.0
    B = np.array(axis, dtype=float)[:, None]
    if site:
        B = B * rng.uniform(0.5, 1.5, N)
    run(q, d, dims, omega, st, field=B)


# at an omega this small the step leaves the state as it is, but for streaming
@pytest.mark.parametrize("tau", [1e200, 1e270, 1e290, 1e300])
@pytest.mark.parametrize("prec", ["fp64", "fp64df"])
@pytest.mark.parametrize("d,dims", [(2, (21, 5, 1)), (3, (9, 5, 3))])
def test_endless_relaxation(q, d, dims, prec, tau):
    run(q, d, dims, 1.0 / tau, one_outweighs(d, dims, 0.1), prec=prec)
