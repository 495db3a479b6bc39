"""Step through the Fermi-Dirac parameters under a caller's stream capture."""
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


@pytest.mark.parametrize("d,dims", [(2, (40, 6, 1)), (3, (12, 5, 4))])
def test_fd_path_first_step_inside_a_capture(q, d, dims):
    # the matrices of the two-kernel form are allocated by the first step; a
    # caller's capture of that step survives it
    import torch
    from paper_1309_1656_gb300 import fields
    fl = fields.random_fields(d, dims, seed=3)
    s = torch.cuda.Stream()
    with q.Lattice(d, dims, 0.8, 1.0, stream=s.cuda_stream) as lat, q.Lattice(d, dims, 0.8, 1.0) as ref:
        for x in (lat, ref):
            x.init_equilibrium(fl["rho4"], fl["u"], fl["eps"])
            q.qlbm_set_equilibrium_path(x.h, q.QLBM_EQ_FD_PARAMS)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            lat.step(2)
        for _ in range(2):
            g.replay()
        torch.cuda.synchronize()
        ref.step(4)
        assert np.array_equal(lat.get_state(), ref.get_state())
