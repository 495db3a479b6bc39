// Host entry points to the device headers' arithmetic (functions compiled for
// both sides), for the checks that need no GPU: loaded by
// test_host_arithmetic.py.
#include "../paper_1309_1656_gb300/csrc/consts.cu"
#include "../paper_1309_1656_gb300/csrc/fdparams.cuh"
#include "../paper_1309_1656_gb300/csrc/fix64.cuh"

using namespace qlbm;

// The chunks that the warps of block `block` take, and the number of blocks a
// launch over `nx` x `rows` sites has.
extern "C" int chunk_of_warp(unsigned block, unsigned warp, int threads)
{
    return chunk_of_thread(block, 32 * warp + 31, threads);
}
extern "C" int chunks_of_lattice(int nx, int rows)
{
    Grid g = {};
    g.nx = nx;
    g.ny = rows;
    g.nz = 1;
    return make_chunks(g).total;
}

// Interval of the Fermi-Dirac polynomial tables, their number, and the
// distance of x from the interval's centre (1/8 at most).
extern "C" int fd_table_interval(float x) { return fd_interval(x); }
extern "C" int fd_table_intervals() { return FD_PINT; }
extern "C" double fd_table_offset(float x) { return (double)x - (FD_PX0 + 0.125 + 0.25 * fd_interval(x)); }

// 1 - omega as the FP64 step's constants hold it (q62).
extern "C" long long one_minus_omega(double omega) { return fx_one_minus(omega); }

// Smallest exponent of a coefficient h_i that is not zero, for the update in
// double of a D2Q9 or D3Q19 step at `omega`; 0 where the form is not taken.
extern "C" int least_coefficient_exponent(int d, double omega)
{
    HostConsts k;
    FixConst fc;
    if (compute_constants(d, 1.0, &k) != 0) return 1;
    return make_fix_const(k, omega, true, &fc) ? fc.h_unit : 0;
}
