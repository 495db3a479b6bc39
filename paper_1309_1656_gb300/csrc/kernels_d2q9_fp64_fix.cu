// D2Q9 kernels of the FP64 step on the integer pipes (fix64.cuh): the AA
// steps and the two-buffer step of the reverse mode, compiled apart from the
// rest of the FP64 dispatch table.
#include "fix64.cuh"
#include "launch.cuh"

namespace qlbm {

template <int D> bool step_fix(qlbm_ctx *h, int mode, const void *src, void *dst, const void *rho, cudaError_t *err)
{
    FixConst fc;
    if (h->mag != FIELD_NONE || !make_fix_const(h->hc, h->dt / h->tau, &fc)) return false;
    using L = Launchers<D, CodecF64>;
    const Chunks ch = make_chunks(h->g);
    const Planes<double, Lattice<D>::Q> s = L::template planes_of<double>(h, src), d = L::template planes_of<double>(h, dst);
    const Coll<double> k = make_coll<double>(h);
    const dim3 blk(kFixBlock), grd((unsigned)((ch.total + kFixBlock / 32 - 1) / (kFixBlock / 32)));
    const DQuad *r = static_cast<const DQuad *>(rho);
    const int df = h->prec == QLBM_FP64_DF && !rho;     // the step through the parameters is the FP64 one
    auto launch = [&](auto kernel) { *err = launch_chained(kernel, grd, blk, 0, h->stream, s, d, h->g, fc, k, ch, df, r, h->flags); };
    if (mode == FIX_PUSH) launch(k_step_fix<D, FIX_PUSH, false>);
    else if (mode == FIX_ODD) launch(rho ? k_step_fix<D, FIX_ODD, true> : k_step_fix<D, FIX_ODD, false>);
    else launch(rho ? k_step_fix<D, FIX_EVEN, true> : k_step_fix<D, FIX_EVEN, false>);
    return true;
}
template bool step_fix<2>(qlbm_ctx *, int, const void *, void *, const void *, cudaError_t *);

}  // namespace qlbm
