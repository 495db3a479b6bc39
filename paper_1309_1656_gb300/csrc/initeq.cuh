// Initial equilibrium (Eq. WeqAlgo from given rho, u, eps) on the integer
// pipes.  In double, each of a site's 4b values takes a product and (for the
// deviation codecs) a subtraction and a conversion on a pipe of 64 cycles per
// warp instruction; here the h_i = w_i P_i are the step's fixed-point
// coefficients (fix64.cuh, omega = 1), the products 64-bit integers, and each
// stored value is rounded once from ~58 bits.  Single- and half-precision
// values are, bit for bit, what rounding the double expression gives (a
// time-stepped state remembers every last bit): a site with a value too near
// a rounding boundary to be sure is formed in double by its thread (~1e-4 of
// the sites at 2 % fluctuations).  One thread per site, one vector store per
// direction.  D3Q19 128^3: FP64 938 -> 284 us, FP32 1217 ->
// 405 us; D2Q9 4096^2 FP16 5142 -> 1258 us.
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

// t 2^unit (|unit + 32| < 120) rounded to a float; false where a number
// within eps of t rounds to another float.
__device__ __forceinline__ bool fx_round_float(long long t, int unit, unsigned eps, float &out)
{
    unsigned sign, m1, m0;
    int lz;
    bool ok = fx_normal(t, sign, m1, m0, lz);
    // distance of the 40 dropped bits from their midpoint, in units of 2^8
    // (eps < 2^16: below 2^30 for lz <= 22, tested above that)
    const unsigned thr = __funnelshift_l(eps << 24, eps >> 8, lz) + 2u;
    const unsigned q = __funnelshift_r(m0, m1, 8) + 0x80000000u;
    ok = ok && lz <= __clz((int)eps) + 6 && q + thr > 2u * thr;
    // the last bit stands for all below (never a tie here)
    out = __uint2float_rn(m1 | 1u) * fx_pow2(unit + 32 - lz);
    out = __int_as_float(__float_as_int(out) | (int)sign);
    return ok;
}

// The same for a half, returned as a float that rounds to it (24 leading bits,
// the rest in the last one).
__device__ __forceinline__ bool fx_round_half(long long t, int unit, unsigned eps, float &out)
{
    unsigned sign, m1, m0;
    int lz;
    bool ok = fx_normal(t, sign, m1, m0, lz);
    // bits that a half keeps: 11, fewer below 2^-14
    const int e = unit + 63 - lz, kept = e < -14 ? 25 + e : 11;
    // eps and the bits below, in m1's last place (eps < 2^15: below 2^30)
    const unsigned thr = ((eps >> ((32 - lz) & 31)) + 3u) << (kept & 31);
    ok = ok && kept > 0 && (m1 << (kept & 31)) + 0x80000000u + thr > 2u * thr;
    out = __uint2float_rn((m1 & 0xffffff00u) | 0x100u) * fx_pow2(unit + 32 - lz);
    out = __int_as_float(__float_as_int(out) | (int)sign);
    return ok;
}

// Stores the vector of direction q (class cls): t[c] 2^unit[c] the components
// of w_i P_i rho; w: the weights by class in q62, the traces of the deviation
// codecs' reference.  False, with nothing stored, where a component's rounding
// is not certain (zero[c]: the component is zero).
template <class Codec> struct InitStore;
template <> struct InitStore<CodecF64> {
    static constexpr int MIN_EXP = kFxMinExp, MAX_EXP = 1023 + 900, MIN_N = kFxMinExp, MAX_N = 1023 + 900;
    static __device__ __forceinline__ bool put(const CodecF64 &, DQuad *p, const long long (&t)[4], const int (&unit)[4],
                                               const bool (&)[4], int, const long long (&)[3], const InitEps &)
    {
        // half of the conversions on the double pipe, half beside it
        stq(p, fx_to_double(t[0], unit[0] * (1 << 20)), fx_to_double(t[1], unit[1] * (1 << 20)),
            fx_to_double_int(t[2], unit[2]), fx_to_double_int(t[3], unit[3]));
        return true;
    }
};
template <> struct InitStore<CodecDF> {
    static constexpr int MIN_EXP = 1023 - 60, MAX_EXP = 1023 + 90, MIN_N = MIN_EXP, MAX_N = MAX_EXP;
    // hi rounded to 24 bits, lo the rounded remainder
    static __device__ __forceinline__ df pair(long long t, int unit)
    {
        const long long s = t >> 63;
        const unsigned long long a = (unsigned long long)((t ^ s) - s);
        const int lz = __clzll((long long)a);
        const unsigned long long m = (a << (lz & 63)) >> 1;                    // leading bit at 62
        const unsigned h = (unsigned)((m + (1ull << 38)) >> 39);               // <= 2^24
        const int rem = (int)((long long)(m - ((unsigned long long)h << 39)) >> 7);     // units of 2^-32 of h's last place
        const int k = unit + 1 - lz + 39;           // h 2^k + rem 2^(k - 32), 2^k in two factors
        const int k1 = k >> 1;
        const float p1 = fx_pow2(k1), p2 = fx_pow2(k - k1);
        const float hi = (float)h * p1 * p2, lo = (float)rem * 0x1p-32f * p1 * p2;
        const int sg = (int)s & (int)0x80000000;
        return df(__int_as_float(__float_as_int(hi) ^ sg), __int_as_float(__float_as_int(lo) ^ sg));
    }
    static __device__ __forceinline__ bool put(const CodecDF &codec, float4 *p, const long long (&t)[4],
                                               const int (&unit)[4], const bool (&)[4], int, const long long (&)[3],
                                               const InitEps &)
    {
        codec.store4(p, pair(t[0], unit[0]), pair(t[1], unit[1]), pair(t[2], unit[2]), pair(t[3], unit[3]));
        return true;
    }
};
template <class Codec> struct InitStore {
    // the deviation codecs: f - w is formed in f's units (2^-59 n: n within
    // [1/16, 16)); components above 2^-30 or zero
    static constexpr bool HALF = sizeof(typename Codec::S) == 2;
    static constexpr int MIN_EXP = 1023 - 30, MAX_EXP = 1023 + 30, MIN_N = 1023 - 4, MAX_N = 1023 + 4;
    static __device__ __forceinline__ bool put(const Codec &codec, typename Codec::V *p, const long long (&t)[4],
                                               const int (&unit)[4], const bool (&zero)[4], int cls,
                                               const long long (&w)[3], const InitEps &eps)
    {
        float v[4];
        bool ok = true;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            long long x = t[c];
            if (c == 0) {
                const int sh = unit[0] + 62;    // w q62 in units of 2^unit, unit = -59 - 4 .. -59 + 3
                x -= sh >= 0 ? w[cls] >> sh : w[cls] << -sh;
            }
            const bool r = HALF ? fx_round_half(x, unit[c], eps.e[cls], v[c]) : fx_round_float(x, unit[c], eps.e[cls], v[c]);
            if (c && zero[c]) v[c] = 0.f;
            else ok = ok && r;
        }
        if (ok) codec.store4(p, v[0], v[1], v[2], v[3]);
        return ok;
    }
};

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
    zero[0] = false;
#pragma unroll
    for (int c = 1; c < 4; ++c) {
        ok = fx_mantissa(rho[c], St::MIN_EXP, St::MAX_EXP, m[c], unit[c]) && ok;
        zero[c] = m[c] == 0;
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
            ok = St::put(codec, pl.p[q] + s, t, ut, zero, cnorm2<D>(q), fc.al, ie) && ok;
        });
        if (ok) return;
    }
    // the whole site in double
    const double e = eps ? eps[s] : ic.eps0, be = ic.beta0 * e;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int cls = cnorm2<D>(q);
        const double wp = ic.w[cls] * poly_P_d<D>(ic, q, uu[0] / ic.xi, uu[1] / ic.xi, uu[2] / ic.xi, be);
        codec.store4(pl.p[q] + s, codec.load(codec.from_double(wp * rho[0], 0, cls)),
                     codec.load(codec.from_double(wp * rho[1], 1, cls)),
                     codec.load(codec.from_double(wp * rho[2], 2, cls)),
                     codec.load(codec.from_double(wp * rho[3], 3, cls)));
    }
}

}  // namespace qlbm
