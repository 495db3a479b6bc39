// D2Q9 kernels of the FP64 step on the integer pipes (fix64.cuh): the AA
// steps and the two-buffer step of the reverse mode, compiled apart from the
// rest of the FP64 dispatch table.
#include "fix64.cuh"
#include "launch.cuh"

namespace qlbm {

template <int D> bool step_fix(qlbm_ctx *h, int mode, const void *src, void *dst, const void *rho, cudaError_t *err)
{
    FixConst fc;
    const double omega = h->dt / h->tau;
    const bool dbl = omega < fix_double_below(h->prec, h->mag);
    // FP64 storage has a kernel of its own for omega > 2; QLBM_FP64_DF is
    // stepped by this one alone, there in double
    if (!make_fix_const(h->hc, omega, dbl, &fc) && h->prec != QLBM_FP64_DF) return false;
    using L = Launchers<D, CodecF64>;
    const Chunks ch = make_chunks(h->g);
    const Planes<double, Lattice<D>::Q> s = L::template planes_of<double>(h, src), d = L::template planes_of<double>(h, dst);
    const Coll<double> k = make_coll<double>(h);
    const dim3 blk(kFixBlock), grd((unsigned)((ch.total + kFixBlock / 32 - 1) / (kFixBlock / 32)));
    const DQuad *r = static_cast<const DQuad *>(rho);
    // (the step through the parameters is the FP64 one)
    const FixRange rg = make_fix_range(h->prec == QLBM_FP64_DF && !rho);
    FixField uq;
    make_fix_field(h->rot, &uq);
    auto go = [&](auto fcn, auto dbl) {
        constexpr int F = decltype(fcn)::value;
        constexpr bool U = decltype(dbl)::value;
        auto launch = [&](auto kernel) {
            return launch_chained(kernel, grd, blk, 0, h->stream, s, d, h->g, fc, k, ch, rg, r, uq, h->flags);
        };
        if (mode == FIX_PUSH) return launch(k_step_fix<D, FIX_PUSH, false, F, U>);
        if (mode == FIX_ODD) return launch(rho ? k_step_fix<D, FIX_ODD, true, F, U> : k_step_fix<D, FIX_ODD, false, F, U>);
        return launch(rho ? k_step_fix<D, FIX_EVEN, true, F, U> : k_step_fix<D, FIX_EVEN, false, F, U>);
    };
    *err = with_field(h->mag, [&](auto fcn) { return dbl ? go(fcn, std::true_type{}) : go(fcn, std::false_type{}); });
    return true;
}
template bool step_fix<2>(qlbm_ctx *, int, const void *, void *, const void *, cudaError_t *);
template <int D> cudaError_t step_f64df(qlbm_ctx *h, bool odd)
{
    cudaError_t e = cudaErrorNotSupported;
    step_fix<D>(h, odd ? FIX_ODD : FIX_EVEN, h->pop, h->pop, nullptr, &e);
    return e;
}
template cudaError_t step_f64df<2>(qlbm_ctx *h, bool odd);

}  // namespace qlbm
