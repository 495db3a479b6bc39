"""Index and number arithmetic of the kernels, run on the host: sizes that no
test could allocate, and comparisons with exact arithmetic."""
import ctypes
import fractions
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_1309_1656_gb300 import _build


def compile_host(path, flags="-fPIC"):
    here = os.path.dirname(os.path.abspath(__file__))
    lib = str(path / "libhost.so")
    subprocess.run([_build.nvcc(), "-O2", "-std=c++17", "--expt-relaxed-constexpr", "-Xcompiler", flags, "-shared",
                    "-I", _build.INCLUDE, os.path.join(here, "host_kernels.cu"), "-o", lib], check=True)
    return lib


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    return ctypes.CDLL(compile_host(tmp_path_factory.mktemp("host")))


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


OMEGAS = [0.0, 2.0**-60, 0.1, 0.5, 1.0 - 2.0**-53, 1.0, 1.0 + 2.0**-52, 1.25, 1.9, 2.0 - 2.0**-52, 2.0]


def test_one_minus_omega(host):
    host.one_minus_omega.restype = ctypes.c_longlong
    for omega in OMEGAS:
        want = (1 - fractions.Fraction(omega)) * 2**62
        assert abs(host.one_minus_omega(ctypes.c_double(omega)) - want) <= 1


def test_one_minus_omega_stays_within_64_bits(tmp_path):
    # signed overflow traps in this build (in a process of its own)
    lib = compile_host(tmp_path, "-fPIC,-fsanitize=signed-integer-overflow,-fsanitize-undefined-trap-on-error")
    code = "import ctypes; f = ctypes.CDLL(%r).one_minus_omega; [f(ctypes.c_double(w)) for w in %r]" % (lib, OMEGAS)
    assert subprocess.run([sys.executable, "-c", code]).returncode == 0


@pytest.mark.parametrize("d", [2, 3])
def test_coefficients_of_a_tiny_omega_are_normal_doubles(host, d):
    # (their words are put together in integers; below, the step is in double)
    for k in range(0, 1075):
        assert host.least_coefficient_exponent(d, ctypes.c_double(2.0**-k)) in [0] + list(range(-1022, -61))
    assert all(host.least_coefficient_exponent(d, ctypes.c_double(w)) for w in (2.0**-900, 1e-9, 0.5, 1.0, 2.0))
