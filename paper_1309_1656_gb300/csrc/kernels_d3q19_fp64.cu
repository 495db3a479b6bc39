// D3Q19 (Sec. 3.1, d = 3, b = 19) kernels for FP64 storage: the dispatch tables of FP64 storage with the
// FP64 step and QLBM_FP64_DF's, in a translation unit of its own so the instantiations
// compile in parallel.
#include "launch.cuh"

namespace qlbm {
const LatticeOps *ops_d3q19_fp64() { return Launchers<3, CodecF64>::table(); }

// QLBM_FP64_DF: the FP64 operations, the fixed-point step with single
// precision's exponent range (kernels_d3q19_fp64_fix.cu), no reverse mode.
const LatticeOps *ops_d3q19_fp64df()
{
    static const LatticeOps t = [] {
        LatticeOps o = *Launchers<3, CodecF64>::table();
        o.step = &step_f64df<3>;
        o.adjoint = nullptr;
        o.push = nullptr;
        o.lam_import = nullptr;
        o.lam_export = nullptr;
        return o;
    }();
    return &t;
}
}  // namespace qlbm
