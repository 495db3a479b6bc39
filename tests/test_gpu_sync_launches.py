"""qlbm_sync waits and reads the flag word and launches nothing (a kernel would
need the handle's device to be the calling thread's current one)."""
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


def kernels(f):
    """Names of the library's kernels that f() launches."""
    import torch
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as p:
        f()
        torch.cuda.synchronize()
    return [e.name for e in p.events() if "k_" in e.name and "cuda" not in e.name.lower().split("k_")[0]]


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_sync_launches_nothing(q, prec):
    dims = (24, 3, 1)
    st = fields.random_populations(2, dims, seed=5)
    with q.Lattice(2, dims, 0.8, 1.0, precision=prec) as lat:
        lat.set_state(st)
        lat.step(1)
        kernels(lambda: lat.step(1))        # (the profiler's first use can record nothing)
        if not kernels(lambda: lat.step(1)):
            pytest.skip("no kernel records from the profiler here")
        assert kernels(lat.sync) == []
        st[4, 0, 30] = np.nan
        lat.set_state(st)
        lat.step(1)
        with pytest.raises(q.QLBMError):
            lat.sync()
        lat.sync()      # the flags are cleared
