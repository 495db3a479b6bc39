"""Fermi-Dirac recovery where the fast path's range checks divide a warp: sites
inside and outside of them side by side."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def q():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1309_1656_gb300 import qlbm
    return qlbm


@pytest.mark.parametrize("prec", ["fp64", "fp64df"])
@pytest.mark.parametrize("d,dims", [(2, (41, 3, 1)), (3, (33, 2, 3))])
def test_fd_params_mixed_ranges(q, oracle_mod, prec, d, dims):
    # occupations down to and below 2^-39, |S| zero, tiny (its square above and
    # below 2^-120) and nearly n, degenerate sites (nu > 1), a site without a
    # solution now and then; the bound of the ordinary comparison, 1e-9
    N = int(np.prod(dims))
    rng = np.random.default_rng(d)
    n = rng.choice([1.0, 0.7, 4e-12, 3e-12, 1e-12, 1e-9, 60.0], N, p=[0.5, 0.2, 0.05, 0.05, 0.05, 0.05, 0.1])
    frac = rng.choice([0.0, 0.1, 0.9, 0.999, 1e-10, 1e-17, 1e-25], N)
    axis = rng.normal(size=(3, N))
    axis /= np.linalg.norm(axis, axis=0)
    rho4 = np.concatenate([n[None], n * frac * axis])
    eps = rng.uniform(0.8, 1.3, N) * 0.5 * d
    bad = np.arange(5, N, 37)
    rho4[1:, bad] = 1.2 * n[bad] * axis[:, bad]
    with q.Lattice(d, dims, 0.8, 1.0, precision=prec) as lat:
        lat.init_equilibrium(rho4, 0.01 * rng.normal(size=(d, N)), eps)
        r4, u, e = lat.moments()
        beta, mu_up, mu_dn, ax, nfail = lat.fd_params()
    assert np.isnan(beta).sum() == nfail and np.all(np.isnan(beta[bad]))
    ok = np.isfinite(beta)
    ok[bad] = True
    assert np.all(ok[n < 60.0])         # (n = 60 can lie below the degenerate limit)
    for s in np.flatnonzero(np.isfinite(beta)):
        # against the equations themselves (near |S| = 0 the splitting of the
        # oracle's own solve is 6e-9 off)
        nS = np.linalg.norm(r4[1:, s])
        nu, nd, en = oracle_mod.fd_moments(d, beta[s], mu_up[s], mu_dn[s])
        assert nu == pytest.approx(0.5 * (r4[0, s] + nS), rel=1e-9)
        assert nd == pytest.approx(0.5 * (r4[0, s] - nS), rel=1e-9)
        assert en == pytest.approx(e[s], rel=1e-9)
        S = r4[1:, s]
        assert np.allclose(ax[:, s], S / (np.linalg.norm(S) or 1.0), atol=1e-9)


@pytest.mark.parametrize("d,dims", [(2, (41, 3, 1)), (3, (33, 2, 3))])
def test_fd_params_at_the_ends_of_the_tables(q, oracle_mod, d, dims):
    # beta mu spread over 2^-20 on both sides of 1 and of -8, where the
    # polynomials begin and end; the bound of the ordinary comparison, 1e-9
    N = int(np.prod(dims))
    rng = np.random.default_rng(40 + d)
    nu = rng.choice([1.0, -8.0], (2, N)) + rng.integers(-16, 17, (2, N)) * 2.0**-24
    beta = rng.uniform(0.9, 1.1, N)
    axis = np.zeros((3, N))
    axis[2] = 1.0
    with q.Lattice(d, dims, 0.8, 1.0, precision="fp64") as lat:
        q.qlbm_init_fd_params(lat.h, beta, nu[0] / beta, nu[1] / beta, axis, np.zeros((d, N)))
        r4, u, e = lat.moments()
        b, mu_up, mu_dn, ax, nfail = lat.fd_params()
    assert nfail == 0
    for s in range(N):
        nS = np.linalg.norm(r4[1:, s])
        a, c, en = oracle_mod.fd_moments(d, b[s], mu_up[s], mu_dn[s])
        assert a == pytest.approx(0.5 * (r4[0, s] + nS), rel=1e-9)
        assert c == pytest.approx(0.5 * (r4[0, s] - nS), rel=1e-9)
        assert en == pytest.approx(e[s], rel=1e-9)
