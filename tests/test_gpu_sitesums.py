"""Moments, global sums and the initial equilibrium on the integer pipes, every
precision, against extended precision, where their layouts and ranges end:
rows around 8-site chunks and 128-site blocks, both buffer parities, sites
outside the fixed-point range (formed in double), zero and tiny components.

Tolerances, from the arithmetic: a sum of b <= 19 values in double errs by at
most 19 x 2^-53 of the sum of their magnitudes, the fixed-point one by less;
the ratios add a few roundings: 64 x 2^-53 in all.  A stored initial value is
the rounding of an expression known to 2^-40 of it: half a last place of the
storage type, and a thousandth."""
import numpy as np
import pytest

from paper_1309_1656_gb300 import fields

pytestmark = pytest.mark.gpu

TOL = 64 * 2.0 ** -53
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


def spoil(st):
    """Sites beyond the integer form among ordinary ones: n < 0, fast, tiny."""
    N = st.shape[2]
    if N > 24:
        st[0, 0, 5] = -3.0
        st[-1, 0, 13] += 1.0
        st[:, 1:, 20] *= 2.0 ** -40
        st[:, 3, 22] = 0.0
    return st


@pytest.mark.parametrize("prec", ["fp64", "fp64df", "df64", "fp32", "fp16dev"])
@pytest.mark.parametrize("steps", [0, 1])
@pytest.mark.parametrize("d,dims", [(2, (1, 1, 1)), (2, (7, 5, 1)), (2, (129, 3, 1)), (3, (9, 4, 3)), (3, (16, 2, 5))])
def test_moments_and_sums(q, prec, steps, d, dims):
    st = fields.random_populations(d, dims, seed=3)
    if not steps:
        st = spoil(st)
    with q.Lattice(d, dims, 0.8, 1.0, precision=prec) as lat:
        lat.set_state(st)
        lat.step(steps)
        W = lat.get_state().astype(LD)
        r, u, eps = lat.moments()
        total = lat.conserved()
        xi = lat.info()["xi"]
    e = np.array(directions(d), dtype=LD)
    f, size = W[:, 0], np.abs(W).sum(0)
    n = f.sum(0)
    assert np.all(np.abs(r - W.sum(0)) <= TOL * size)
    cond = size[0] / np.abs(n)          # cancellation in n
    j = [(e[:, a, None] * f).sum(0) / n for a in range(3)]
    ok = np.abs(n) > 1e-3
    for a in range(d):
        assert np.all(np.abs(u[a] - xi * j[a])[ok] <= (TOL * xi * cond * (1 + np.abs(j[a])))[ok])
    E = ((e * e).sum(1)[:, None] * f).sum(0) / n
    want = 0.5 * xi * xi * (E - sum(a * a for a in j))
    assert np.all(np.abs(eps - want)[ok] <= (4 * TOL * cond * cond * (1 + np.abs(want)))[ok])
    N = W.shape[2]
    sums = list(W.sum(0).sum(1) / N) + [xi * (e[:, a, None] * f).sum() / N for a in range(3)]
    sums.append(0.5 * xi * xi * ((e * e).sum(1)[:, None] * f).sum() / N)
    scale = float(size.sum(1).max() / N)
    bound = 4 * TOL * scale * xi * xi * (1 if prec not in ("fp32", "fp16dev") else 16)
    assert np.max(np.abs(total - np.array(sums, dtype=LD))) <= bound


@pytest.mark.parametrize("prec", ["fp64", "df64", "fp32", "fp16dev"])
@pytest.mark.parametrize("d,dims", [(2, (37, 5, 1)), (2, (130, 2, 1)), (3, (33, 3, 2))])
def test_initial_equilibrium(q, prec, d, dims):
    fl = fields.random_fields(d, dims, seed=9, umax=0.3)
    rho4, u, eps = fl["rho4"], fl["u"], fl["eps"]
    N = rho4.shape[1]
    quiet = np.arange(N) % 3 == 0       # near the reference: small deviations
    rho4[0, quiet] = 1.0 + 1e-3 * (rho4[0, quiet] - 1.0)
    rho4[1:, quiet] *= 1e-2
    u[:, quiet] *= 1e-2
    rho4[:, 7] *= 64.0                  # beyond the fixed-point ranges
    u[0, 8] = 1.5
    rho4[1:, 10] *= 2.0 ** -40
    rho4[2, 11:20] = 0.0
    with q.Lattice(d, dims, 0.8, 1.0, precision=prec) as lat:
        k = lat.info()
        eps[quiet] = k["c"] * (1.0 + 1e-2 * (eps[quiet] - 1.5))
        lat.init_equilibrium(rho4, u, eps)
        img = lat.save_checkpoint()
        got = lat.get_state()
    k = {name: LD(v) for name, v in k.items()}
    K = k["xi"] ** 2 / 2
    j = [u[a].astype(LD) / k["xi"] for a in range(d)]
    jj = sum(a * a for a in j)
    a2 = (eps.astype(LD) - k["c"]) / (k["m"] - k["c"] ** 2)
    want, w = [], []
    for v in directions(d):
        m = sum(map(abs, v))
        t = sum(v[a] * j[a] for a in range(d))
        P = (1 - k["c"] * a2 + a2 * K * m + 2 * K * k["alpha3"] * t + 4 * K * K * k["alpha4"] * t * t +
             K * k["alpha5"] * jj)
        w.append(k[("w_rest", "w_axis", "w_diag")[m]])
        want.append(w[-1] * P * rho4.astype(LD))
    want = np.stack(want)
    if prec in ("fp64", "df64"):
        scale = np.abs(rho4).astype(LD)
        assert np.all(np.abs(got - want) <= (2.0 ** -48 if prec == "fp64" else 2.0 ** -46) * scale)
        return
    want[:, 0] -= np.array(w)[:, None]
    stored = img.view(np.float32 if prec == "fp32" else np.float16).reshape(len(w), N, 4).transpose(0, 2, 1)
    ulp = np.spacing(np.abs(stored)).astype(LD)
    # the deviation's own uncertainty: 2^-47 of the density it is a difference of
    slack = np.zeros_like(want)
    slack[:, 0] = 2.0 ** -47 * np.abs(rho4[0])
    assert np.all(np.abs(stored.astype(LD) - want) <= 0.501 * ulp + slack)


@pytest.mark.parametrize("prec", ["fp64", "df64", "fp32"])
@pytest.mark.parametrize("d,dims", [(2, (33, 5, 1)), (3, (17, 3, 4))])
def test_tiny_spins(q, prec, d, dims):
    # spins from 2^-50 down to single precision's subnormals and to zero, each
    # component a size of its own, and now and then a site summed in double
    rng = np.random.default_rng(61)
    st = fields.random_populations(d, dims, seed=13)
    N = st.shape[2]
    for c in (1, 2, 3):
        st[:, c] *= 2.0 ** -rng.integers(50, 150, N)
    st[:, 1, ::11] = 0.0
    if N > 40:
        st[0, 0, ::40] = -3.0
    with q.Lattice(d, dims, 0.8, 1.0, precision=prec) as lat:
        lat.set_state(st)
        W = lat.get_state().astype(LD)
        r, u, eps = lat.moments()
        total = lat.conserved()
    assert np.all(np.abs(r - W.sum(0)) <= TOL * np.abs(W).sum(0))
    if prec != "fp32":      # (its global sums are formed in double-float, to single precision's range)
        for c in (1, 2, 3):
            assert abs(total[c] - W[:, c].sum() / N) <= 4 * TOL * np.abs(W[:, c]).sum() / N
