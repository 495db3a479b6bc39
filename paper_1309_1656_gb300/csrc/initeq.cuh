// Initial equilibrium (Eq. WeqAlgo from given rho, u, eps) on the integer
// pipes.  In double, each of a site's 4b values takes a product and (for the
// deviation codecs) a subtraction and a conversion on a pipe of 64 cycles per
// warp instruction; here the h_i = w_i P_i are the step's fixed-point
// coefficients (fix64.cuh, omega = 1), the products 64-bit integers, and each
// stored value is rounded once from ~58 bits.  Single- and half-precision
// values are, bit for bit, what rounding the double expression gives (a
// time-stepped state remembers every last bit): where a value is too near a
// rounding boundary to be sure, its direction's f or spins are formed in
// double by the site's thread, one such direction after another.  Those are
// ~1e-4 of the values at fluctuations of 2 %, and every f of a flow slow
// enough (|u| of 1e-5 and less) for its deviations to be made of the double
// expression's own roundings.  Spins of any size stay in integers down to
// what rounds to zero (FP32: but for the octaves of subnormal results).
// One thread per site, one vector store per direction.  Everything in double
// -> this: D3Q19 128^3 FP64 938 -> 284 us; FP32 with fluctuations 1223 -> 353,
// slow flow 1224 -> 520, at rest 1363 -> 307, spin blob 1363 -> 513; D2Q9
// 2048^2 FP16 shear layer 1297 -> 301, spin blob 1480 -> 306.
#pragma once

#include "fix64.cuh"
#include "kernels.cuh"
#include "quadsum.cuh"

namespace qlbm {

// A double as m 2^unit, m of 62 bits and a sign (0 for zero); false for
// magnitudes outside [2^(lo - 1023), 2^(hi - 1023)) other than zero.
__device__ __forceinline__ bool fx_mantissa(double v, int lo, int hi, long long &m, int &unit)
{
    const unsigned h = (unsigned)__double2hiint(v), l = (unsigned)__double2loint(v);
    const int e = (int)((h >> 20) & 0x7ffu);
    const bool zero = (((h & 0x7fffffffu) | l) == 0u);
    const unsigned long long a = ((unsigned long long)((h & 0xfffffu) | 0x100000u) << 32) | l;
    const long long s = (long long)((int)h >> 31);
    m = zero ? 0 : (((long long)(a << 9)) ^ s) - s;
    unit = zero ? -1084 + 1023 : e - 1084;
    return zero || (e >= lo && e < hi);
}

// How far a fixed-point value t may be off from the double expression
// (poly_P_d and the products below), in t's units: the single- and half-
// precision codecs store exactly what rounding that expression gives, because
// a value this close to a rounding boundary is formed in double instead.
// With x_k the terms of P_i besides 1, the double expression errs by at most
// 2^-53 (11 + 10 sum |x_k|) w_i |rho_c|, sum |x_k| <= 8 |d| + 7 |j|_1, and
// rho_c <= 2^60 units; the fixed-point path by less than 32 units and the
// rounding of j and d to doubles.
struct InitEps {
    unsigned e[3];      // by class: w_0 < 1/2, w_1 < 1/8, w_2 < 1/32
};
template <int D> __device__ __forceinline__ InitEps init_eps(const FxSplit (&j)[3], long long d60)
{
    unsigned n = (unsigned)abs((int)(d60 >> 32)) >> 21;         // 128 |d|
#pragma unroll
    for (int a = 0; a < D; ++a) n += (unsigned)abs(j[a].hi) >> 25;      // 128 |j_a|
    n += 24u;
    return InitEps{64u * n + 32u, 16u * n + 32u, 4u * n + 32u};
}

// |t| normalised to m (leading bit 63): its upper word, and lz; false where t
// has no bit in its upper word (too small to be judged).
__device__ __forceinline__ bool fx_normal(long long t, unsigned &sign, unsigned &m1, unsigned &m0, int &lz)
{
    const unsigned s = (unsigned)(int)(t >> 63), a1 = (unsigned)(t >> 32) ^ s, a0 = (unsigned)t ^ s;
    sign = s & 0x80000000u;
    lz = __clz((int)a1);
    m1 = __funnelshift_l(a0, a1, lz);
    m0 = a0 << (lz & 31);
    return a1 != 0u;
}
__device__ __forceinline__ float fx_pow2(int k) { return __int_as_float((k + 127) << 23); }

// t 2^unit (below 2^120) rounded to a float; false where a number within eps
// of t rounds to another float, and for subnormal results.
__device__ __forceinline__ bool fx_round_float(long long t, int unit, unsigned eps, unsigned &sign, float &out)
{
    unsigned m1, m0;
    int lz;
    bool ok = fx_normal(t, sign, m1, m0, lz);
    // distance of the 40 dropped bits from their midpoint, in units of 2^8
    // (eps < 2^16: below 2^30 for lz <= 22, tested above that)
    const unsigned thr = __funnelshift_l(eps << 24, eps >> 8, lz) + 2u;
    const unsigned q = __funnelshift_r(m0, m1, 8) + 0x80000000u;
    const int k = unit + 32 - lz;       // |t| 2^unit = m1 2^k
    ok = ok && lz <= __clz((int)eps) + 6 && q + thr > 2u * thr && k + 31 >= -126;
    // the last bit stands for all below (never a tie here)
    out = __uint_as_float(sign | (__float_as_uint(__uint2float_rn(m1 | 1u)) + ((unsigned)k << 23)));
    return ok;
}

// The same for a half, subnormal ones included, returned as a float that
// rounds to it (24 leading bits, the rest in the last one).  unit > -120.
__device__ __forceinline__ bool fx_round_half(long long t, int unit, unsigned eps, unsigned &sign, float &out)
{
    unsigned m1, m0;
    int lz;
    const bool ok = fx_normal(t, sign, m1, m0, lz);
    // bits that a half keeps: 11, fewer below 2^-14, none below 2^-24 (kept
    // < -1: zero; 0: halfway to the smallest ends the octave below)
    const int e = unit + 63 - lz, kept = e < -14 ? 25 + e : 11;
    // eps, and what m1 leaves out, in m1's last place
    // (eps < 2^15: below 2^30; the bits of m0 taken in as well cost more, 294 ->
    // 330 us at 4.2e6 sites, than the fewer sites in double gain)
    const unsigned thr = ((eps >> ((32 - lz) & 31)) + 3u) << (kept & 31);
    out = __uint2float_rn((m1 & 0xffffff00u) | 0x100u) * fx_pow2(unit + 32 - lz);
    out = __int_as_float(__float_as_int(out) | (int)sign);
    return ok && (kept < -1 || (kept >= 0 && (m1 << (kept & 31)) + 0x80000000u + thr > 2u * thr));
}

// Stores the vector of direction q (class cls): t[c] 2^unit[c] the components
// of w_i P_i rho; w: the weights by class in q62, the traces of the deviation
// codecs' reference.  Returns which parts have a rounding that is not certain
// (1: f, 2: a spin component) and are to be formed in double (zero[c]: what is
// stored of the component, the deviation of f, is zero).
template <class Codec> struct InitStore;
template <> struct InitStore<CodecF64> {
    // exponents from 64: t's last place is a normal double
    static constexpr int MIN_EXP = 64, MAX_EXP = 1023 + 900, MIN_N = 64, MAX_N = 1023 + 900, ZERO_EXP = 0;
    static __device__ __forceinline__ unsigned put(const CodecF64 &, DQuad *p, const long long (&t)[4], const int (&unit)[4],
                                                   const bool (&)[4], int, const long long (&)[3], const InitEps &)
    {
        // half of the conversions on the double pipe, half beside it
        stq(p, fx_to_double(t[0], unit[0] * (1 << 20)), fx_to_double(t[1], unit[1] * (1 << 20)),
            fx_to_double_int(t[2], unit[2]), fx_to_double_int(t[3], unit[3]));
        return 0u;
    }
};
template <> struct InitStore<CodecDF> {
    static constexpr int MIN_EXP = 0, MAX_EXP = 1023 + 90, MIN_N = 1023 - 60, MAX_N = MAX_EXP, ZERO_EXP = 0;
    // hi rounded to 24 bits, lo the rounded remainder
    static __device__ __forceinline__ df pair(long long t, int unit)
    {
        const long long s = t >> 63;
        const unsigned long long a = (unsigned long long)((t ^ s) - s);
        const int lz = __clzll((long long)a);
        const unsigned long long m = (a << (lz & 63)) >> 1;                    // leading bit at 62
        const unsigned h = (unsigned)((m + (1ull << 38)) >> 39);               // <= 2^24
        const int rem = (int)((long long)(m - ((unsigned long long)h << 39)) >> 7);     // units of 2^-32 of h's last place
        // h 2^k + rem 2^(k - 32), 2^k in two factors (both parts are 0 from
        // k = -252 on)
        const int k = max(unit + 1 - lz + 39, -252);
        const int k1 = k >> 1;
        const float p1 = fx_pow2(k1), p2 = fx_pow2(k - k1);
        const float hi = (float)h * p1 * p2, lo = (float)rem * 0x1p-32f * p1 * p2;
        const int sg = (int)s & (int)0x80000000;
        return df(__int_as_float(__float_as_int(hi) ^ sg), __int_as_float(__float_as_int(lo) ^ sg));
    }
    static __device__ __forceinline__ unsigned put(const CodecDF &codec, float4 *p, const long long (&t)[4],
                                                   const int (&unit)[4], const bool (&)[4], int, const long long (&)[3],
                                                   const InitEps &)
    {
        codec.store4(p, pair(t[0], unit[0]), pair(t[1], unit[1]), pair(t[2], unit[2]), pair(t[3], unit[3]));
        return 0u;
    }
};
template <class Codec> struct InitStore {
    // the deviation codecs: f - w is formed in f's units (2^-59 n: n within
    // [1/16, 16)); spins of any size: below 2^(ZERO_EXP - 1023) all their
    // values (|w_i P_i| < 1) round to zero
    static constexpr bool HALF = sizeof(typename Codec::S) == 2;
    static constexpr int MIN_EXP = 0, MAX_EXP = 1023 + 30, MIN_N = 1023 - 4, MAX_N = 1023 + 4;
    static constexpr int ZERO_EXP = 1023 - (HALF ? 26 : 151);
    static __device__ __forceinline__ unsigned put(const Codec &codec, typename Codec::V *p, const long long (&t)[4],
                                                   const int (&unit)[4], const bool (&zero)[4], int cls,
                                                   const long long (&w)[3], const InitEps &eps)
    {
        float v[4];
        unsigned bad = 0u;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            long long x = t[c];
            if (c == 0) {
                const int sh = unit[0] + 62;    // w q62 in units of 2^unit, unit = -59 - 4 .. -59 + 3
                x -= sh >= 0 ? w[cls] >> sh : w[cls] << -sh;
            }
            unsigned sign;
            const bool r = HALF ? fx_round_half(x, unit[c], eps.e[cls], sign, v[c])
                                : fx_round_float(x, unit[c], eps.e[cls], sign, v[c]);
            if (zero[c]) v[c] = c ? __uint_as_float(sign) : 0.f;
            else if (!r) bad |= c ? 2u : 1u;
        }
        codec.store4(p, v[0], v[1], v[2], v[3]);
        return bad;
    }
};

// 2 bits per direction: its component along axis a, plus 1.
template <int D> constexpr unsigned long long direction_code(int a)
{
    unsigned long long r = 0;
    for (int q = 0; q < Lattice<D>::Q; ++q)
        r |= (unsigned long long)((a == 0 ? cx<D>(q) : a == 1 ? cy<D>(q) : cz<D>(q)) + 1) << (2 * q);
    return r;
}

// fc: the fixed-point constants for omega = 1 (h_i = w_i P_i).
template <int D, class Codec>
__global__ void __launch_bounds__(kStepBlock, 4)
k_init_eq(const Planes<typename Codec::S, Lattice<D>::Q> pl, Grid g, InitConsts ic, FixConst fc, Codec codec,
          const double *__restrict__ rho4, const double *__restrict__ u, const double *__restrict__ eps)
{
    using St = InitStore<Codec>;
    constexpr int Q = Lattice<D>::Q;
    SiteIdx si;
    if (!site_of_block(g, si)) return;
    const int64_t N = g.N, s = si.s;
    const double rho[4] = {rho4[s], rho4[N + s], rho4[2 * N + s], rho4[3 * N + s]};
    double uu[3] = {u[s], u[N + s], 0.0};
    if (D == 3) uu[2] = u[2 * N + s];
    // the moments as fixed-point numbers; range checks on the high words of
    // the doubles (the conversions saturate beyond)
    long long m[4];
    int unit[4];
    bool zero[4];
    bool ok = fx_mantissa(rho[0], St::MIN_N, St::MAX_N, m[0], unit[0]) && m[0] > 0;
    // a fluid at rest at the reference density has no deviation at all (in
    // double: P_i = 1, w_i 1 1 - w_i = 0)
    auto bits = [](double v) { return (unsigned long long)__double_as_longlong(v); };
    zero[0] = !eps && ic.rest && bits(rho[0]) == 0x3ffull << 52 && (bits(uu[0]) | bits(uu[1]) | bits(uu[2])) << 1 == 0ull;
#pragma unroll
    for (int c = 1; c < 4; ++c) {
        ok = fx_mantissa(rho[c], St::MIN_EXP, St::MAX_EXP, m[c], unit[c]) && ok;
        zero[c] = m[c] == 0 || (int)((unsigned)__double2hiint(rho[c]) >> 20 & 0x7ffu) < St::ZERO_EXP;
    }
    FxSplit j[3];
    long long jj = 0;
#pragma unroll
    for (int a = 0; a < D; ++a) {
        ok = ok && (__double2hiint(uu[a]) & 0x7fffffff) < __double2hiint(ic.umax);
        j[a] = fx_split(__double2ll_rn(uu[a] * ic.rxi));
        jj += fx_mul(j[a], j[a]);
    }
    // d = E2/n - |j|^2 - d0 = (beta0 eps - c) / K
    long long d60 = 0;
    if (eps) {
        const double d = (ic.beta0 * eps[s] - ic.c) * ic.rK;
        ok = ok && (__double2hiint(d) & 0x7fffffff) < ((1023 + 60) << 20);
        d60 = __double2ll_rn(d);
    }
    FixCoef cf;
    ok = fx_basis<D>(j, jj, d60, fc, cf) && ok;
    // directions to be formed in double: their f, their spins
    constexpr unsigned all = (1u << Q) - 1u;
    unsigned bad_f = ok ? 0u : all, bad_s = bad_f;
    if (ok) {
        FxSplit ms[4];
        int ut[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            ms[c] = fx_split(m[c]);
            ut[c] = unit[c] + 2;
        }
        const InitEps ie = init_eps<D>(j, d60);
        fx_each_h<D>(cf, [&](int q, long long h) {
            const FxSplit hs = fx_split(h);
            const long long t[4] = {fx_mul(hs, ms[0]), fx_mul(hs, ms[1]), fx_mul(hs, ms[2]), fx_mul(hs, ms[3])};
            const unsigned bad = St::put(codec, pl.p[q] + s, t, ut, zero, cnorm2<D>(q), fc.al, ie);
            if (bad & 1u) bad_f |= 1u << q;
            if (bad & 2u) bad_s |= 1u << q;
        });
        if (!(bad_f | bad_s)) return;
    }
    // in double, a direction at a time, each lane its own (unrolled, this code
    // does not fit the instruction caches beside the above: 500 us instead of
    // 353 at D3Q19 128^3 FP32 with fluctuations); f and the spins by
    // themselves: near the reference f's rounding is seldom certain, the
    // spins' is
    const int64_t sr = s + g.zero;      // (read again, not kept from above)
    const double r[4] = {rho4[sr], rho4[N + sr], rho4[2 * N + sr], rho4[3 * N + sr]};
    const double e = eps ? eps[sr] : ic.eps0, be = ic.beta0 * e;
    const double j0 = u[sr] / ic.xi, j1 = u[N + sr] / ic.xi, j2 = D == 3 ? u[2 * N + sr] / ic.xi : 0.0;
    const double sq = fma(j2, j2, fma(j1, j1, j0 * j0)), a2 = (be - ic.c) * ic.inv_mc2, a1 = fma(-ic.c, a2, 1.0);
    const double b1 = fma(a2, ic.K, a1), b2 = fma(a2 * ic.K, 2.0, a1);
    auto along = [](int i, double v) { return i == 0 ? 0.0 : i > 0 ? v : -v; };
#pragma unroll 1
    for (unsigned todo = bad_f | bad_s; todo; todo &= todo - 1u) {
        const int q = __ffs((int)todo) - 1;
        const int ix = (int)(direction_code<D>(0) >> (2 * q) & 3u) - 1, iy = (int)(direction_code<D>(1) >> (2 * q) & 3u) - 1,
                  iz = (int)(direction_code<D>(2) >> (2 * q) & 3u) - 1;
        const int cls = abs(ix) + abs(iy) + abs(iz);
        // P_i as poly_P_d forms it, rounding by rounding
        const double t = along(ix, j0) + along(iy, j1) + along(iz, j2);
        const double P = fma(ic.c5, sq, fma(ic.c4 * t, t, fma(ic.c3, t, cls == 0 ? a1 : cls == 1 ? b1 : b2)));
        const double wp = (cls == 0 ? ic.w[0] : cls == 1 ? ic.w[1] : ic.w[2]) * P;
        auto *p = pl.p[0] + (int64_t)q * g.P + s;
        if constexpr (Codec::DEV) {
            typename Codec::S *v = reinterpret_cast<typename Codec::S *>(p);
            if (bad_f >> q & 1u) v[0] = codec.from_double(wp * r[0], 0, cls);
            if (bad_s >> q & 1u) {
#pragma unroll
                for (int c = 1; c < 4; ++c) v[c] = codec.from_double(wp * r[c], c, cls);
            }
        } else {
            codec.store4(p, codec.load(codec.from_double(wp * r[0], 0, cls)),
                         codec.load(codec.from_double(wp * r[1], 1, cls)),
                         codec.load(codec.from_double(wp * r[2], 2, cls)),
                         codec.load(codec.from_double(wp * r[3], 3, cls)));
        }
    }
}

}  // namespace qlbm
