"""Reverse sweep and init gradients at the sizes where the staged copies and
the folded sums can go wrong: rows shorter and longer than a block, periodic
images in one-site directions, and a single site."""
import numpy as np
import pytest

from paper_1309_1656_gb300 import fields

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def q():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1309_1656_gb300 import qlbm
    return qlbm


STEP_SHAPES = [(3, (1, 1, 1)), (3, (31, 2, 1)), (3, (33, 1, 2)), (3, (127, 2, 2)), (3, (129, 2, 3)), (3, (300, 1, 2)),
               (2, (129, 3, 1))]


@pytest.mark.parametrize("prec", ["fp32", "fp16dev"])
@pytest.mark.parametrize("d,dims", STEP_SHAPES)
def test_step_adjoint_single_precision_sites(q, oracle_mod, prec, d, dims):
    # A result passes through at most ~64 single-precision roundings (sums of
    # b directions, four components, the transposed moments) of terms up to
    # about four times the largest result: 64 x 2^-24 x 4 = 1.6e-5.
    tau, beta0 = 0.8, 1.0
    fl = fields.random_fields(d, dims, seed=7)
    with q.Lattice(d, dims, tau, beta0, precision=prec) as lat:
        lat.init_equilibrium(fl["rho4"], fl["u"], fl["eps"])
        w = lat.get_state()
        lam_next = np.random.default_rng(3).normal(size=w.shape)
        lam, g = lat.step_adjoint(lam_next)
    lam_o, g_o = oracle_mod.adjoint_step(d, dims, tau, beta0, w, lam_next)
    assert np.max(np.abs(lam - lam_o)) < 1.6e-5 * np.max(np.abs(lam_o))
    assert abs(g - g_o) < 64 * 2.0**-24 / tau**2 * np.max(np.abs(w)) * np.sum(np.abs(lam_next))


def vectors(d):
    z = (0,) if d == 2 else (-1, 0, 1)
    return [(x, y, k) for k in z for y in (-1, 0, 1) for x in (-1, 0, 1) if d == 2 or x * x + y * y + k * k < 3]


@pytest.mark.parametrize("with_eps", [False, True])
@pytest.mark.parametrize("d,dims", [(2, (1, 1, 1)), (2, (129, 3, 1)), (3, (1, 1, 1)), (3, (5, 4, 3)), (3, (130, 2, 2))])
def test_init_adjoint_against_extended_precision(q, oracle_mod, d, dims, with_eps):
    # The initialisation is linear in rho4 and quadratic in u: W = w P rho with
    # P found here from the oracle's own W at rho4 = (1, 0, 0, 0) by exact
    # finite differences of a quadratic.  Bound: 64 roundings of 2^-53 on the
    # sum of the absolute terms (double), and the differences' own rounding,
    # 2^-53 |W| / h with h = 1/8 and the same number of terms.
    beta0, N = 1.1, int(np.prod(dims))
    b = len(vectors(d))
    fl = fields.random_fields(d, dims, seed=14)
    eps = fl["eps"] if with_eps else None
    lam = np.random.default_rng(2).normal(size=(b, 4, N))
    gr, gu, ge = np.zeros((4, N)), np.zeros((d, N)), np.zeros(N)
    with q.Lattice(d, dims, 0.7, beta0) as lat:
        q.qlbm_init_equilibrium_adjoint(lat.h, fl["rho4"], fl["u"], eps, lam, gr, gu, ge)
        eps_in = fl["eps"] if with_eps else None

    one = np.zeros((4, N))
    one[0] = 1.0
    wp = lambda u, e: oracle_mod.init_equilibrium(d, dims, beta0, one, u, e)[:, 0, :].astype(np.longdouble)
    L = lam.astype(np.longdouble)
    base = wp(fl["u"], eps_in)
    pb = np.einsum("cn,qcn->qn", fl["rho4"].astype(np.longdouble), L)
    scale = np.abs(fl["rho4"]).max() * np.abs(L).sum(axis=(0, 1)).max()
    tol = 64 * 2.0**-53 * 8 * float(scale)
    assert np.max(np.abs(gr - np.einsum("qn,qcn->cn", base, L))) < tol
    for a in range(d):
        up, dn = fl["u"].copy(), fl["u"].copy()
        up[a] += 0.125
        dn[a] -= 0.125
        assert np.max(np.abs(gu[a] - ((wp(up, eps_in) - wp(dn, eps_in)) * pb).sum(axis=0) * 4)) < 8 * tol
    if with_eps:
        e = fl["eps"]
        ref = ((wp(fl["u"], e + 0.125) - wp(fl["u"], e - 0.125)) * pb).sum(axis=0) * 4
        assert np.max(np.abs(ge - ref)) < 8 * tol
