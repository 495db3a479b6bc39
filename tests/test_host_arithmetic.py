"""Index and number arithmetic of the kernels, run on the host: sizes that no
test could allocate, and comparisons with exact arithmetic."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1309_1656_gb300 import _build


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    here = os.path.dirname(os.path.abspath(__file__))
    lib = str(tmp_path_factory.mktemp("host") / "libhost.so")
    subprocess.run([_build.nvcc(), "-O2", "-std=c++17", "--expt-relaxed-constexpr", "-Xcompiler", "-fPIC", "-shared",
                    "-I", _build.INCLUDE, os.path.join(here, "host_kernels.cu"), "-o", lib], check=True)
    return ctypes.CDLL(lib)


# rows of at most one chunk, rows of two, and square lattices, around the
# sizes where 32 threads per chunk pass 2^32 and up to the most sites a handle
# has
@pytest.mark.parametrize("threads", [64, 128, 256])
@pytest.mark.parametrize("nx,rows", [(1, 1), (9, 5), (1, 2**27), (1, 2**27 + 5), (8, 2**27 + 1), (9, 2**26 + 3),
                                     (2**15 + 1, 2**15 + 1), (1, 2**31 - 64)])
def test_every_chunk_has_one_warp(host, nx, rows, threads):
    total = host.chunks_of_lattice(nx, rows)
    assert total == (nx + 7) // 8 * rows
    per_block = threads // 32
    blocks = (total + per_block - 1) // per_block
    for block in {0, blocks // 3, blocks // 2, blocks - 1}:
        for warp in range(per_block):
            # (a warp beyond the last chunk must see a number not below total)
            assert host.chunk_of_warp(ctypes.c_uint(block), ctypes.c_uint(warp), threads) == block * per_block + warp


def test_fermi_dirac_intervals_end_inside_the_tables(host):
    # every float of the last 2^-18 below 1, those around -8 and the seams
    host.fd_table_offset.restype = ctypes.c_double
    ends = [np.float32(1.0)] + [np.float32(-8.0 + 0.25 * i) for i in range(36)]
    xs = [v for e in ends for v in (e, np.nextafter(e, np.float32(9)), np.nextafter(e, np.float32(-9)))]
    xs += list(1.0 - np.arange(1, 65) * np.float32(2.0**-24))
    n = host.fd_table_intervals()
    for x in map(float, xs):
        if -8.0 <= x < 1.0:
            assert 0 <= host.fd_table_interval(ctypes.c_float(x)) < n
            # (a point at a seam may fall to either side of it by rounding)
            assert abs(host.fd_table_offset(ctypes.c_float(x))) <= 0.125 + 2.0**-20
