// The FP64 step on the integer pipes (QLBM_FP64 and QLBM_FP64_DF storage).
//
// GB300's double-precision pipe takes 64 cycles per warp instruction and
// sub-partition (measured, whatever the number of warps; integer add, logic
// and minimum take 1, shifts and 32-bit multiplies 2, the 32 x 32 -> 64-bit
// multiply 4).  The step of k_step_aa<D, CodecF64> is bound by that pipe
// alone: ~445 double-precision instructions per D3Q19 site, at 128^3 1485 us
// for 2.55 GB that the copy rate moves in 376 us.  This file does the same
// step (Eqs. DiscrAvr, WeqAlgo, CollisionStep, TransportStep) in fixed point
// with more digits than a double has:
//
//   * a component's b values at a site are aligned to their largest one's
//     exponent: X = v / U as 64-bit integers with |X| < 2^58 (a double up to
//     32 times smaller than the largest is represented exactly, smaller ones
//     to 2^-58 of the largest); sums of b of them are exact in 64 bits;
//   * the equilibrium's coefficients h_i = omega w_i P_i are formed from the
//     ratios J/n and E2/n with 2^-60 steps, as sums of ten basis values
//     (class constants, i.j and its products), and
//       W_i' = (1 - omega) W_i + h_i M,   M = sum_j W_j of the component,
//     is a pair of 64 x 64-bit products, rounded to 2^-56 of the largest;
//   * one conversion per value rounds it to a double (the only use of the
//     double pipe, which runs beside the integer ones).
//
// Each result errs by at most ~1.2 x 2^-53 of its component's largest value
// at the site (0.13 rms; the double-precision step, which rounds h, h M - W
// and W', by up to 8 x 2^-53, 0.5 rms, at omega = 0.5, and more above).  At
// smaller omega the double step is more accurate than that on populations
// small beside the largest; there the last line is done in double
// (fix_double_below).
// Warps with a site outside the form's range (non-finite or extreme values,
// n <= 0, |j| >= 3/8, E2/n a unit off, |h| >= 1) step in double, with the same
// flags as k_step_aa.
//
// Layout: four lanes per site, lane c holding component c (f, s_x, s_y, s_z)
// of its b populations.  A site's vector of four doubles is 32 bytes, so a
// warp's 8-byte accesses cover 256 consecutive bytes (8 sites), every value
// is read and written once, and a thread keeps 19 values instead of 76.
// Blocks of two warps (a 64 x 64 lattice reaches every SM); 16 warps per SM
// at 128 registers for D3Q19 (20 at 96 spill: 548 us).
//
// Measured (double-precision kernel -> this one), updated in integers: D3Q19
// 128^3 1485 -> 504 us, D2Q9 2048^2 1512 -> 527 us, D2Q9 64^2 8.2 -> 2.3 us; in
// double: 1485 -> 659 us, 1516 -> 594 us, 64^2 2.9 and 2048 x 2 9.0 -> 2.8 us per
// step.  The former is bound by issue (57 % of the cycles), the integer pipe (62 %
// busy), the multiply pipe (60 %) and the conversions (51 %) together, at 1360
// instructions per warp of 8 sites; the latter by the double pipe.
#pragma once

#include <math.h>
#include <string.h>

#include "internal.h"
#include "step.cuh"

namespace qlbm {

#ifdef __CUDA_ARCH__
// a b + c, and a b: one multiply-add each (written out: from the C expression
// the compiler adds separately, 22 instructions more per updated value)
__device__ __forceinline__ long long fx_mad(int a, int b, long long c)
{
    long long r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
}
__device__ __forceinline__ unsigned long long fx_umad(unsigned a, unsigned b, unsigned long long c)
{
    unsigned long long r;
    asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
}
__device__ __forceinline__ int fx_clz(unsigned a) { return __clz((int)a); }
// v >> s for any s >= 0 (0 from 64 on)
__device__ __forceinline__ unsigned long long fx_shr(unsigned long long v, int s)
{
    unsigned long long r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(s));
    return r;
}
// 1/x to ~1 ulp
__device__ __forceinline__ float fx_rcp(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float fx_float(unsigned b) { return __uint_as_float(b); }
__device__ __forceinline__ unsigned fx_bits(float v) { return __float_as_uint(v); }
#else   // the same functions for the host (arithmetic checks without a GPU)
inline long long fx_mad(int a, int b, long long c) { return (long long)a * b + c; }
inline unsigned long long fx_umad(unsigned a, unsigned b, unsigned long long c)
{
    return (unsigned long long)a * b + c;
}
inline int fx_clz(unsigned a) { return a ? __builtin_clz(a) : 32; }
inline unsigned long long fx_shr(unsigned long long v, int s) { return s > 63 ? 0 : v >> s; }
inline float fx_rcp(float x) { return 1.0f / x; }
inline float fx_float(unsigned b)
{
    float v;
    memcpy(&v, &b, 4);
    return v;
}
inline unsigned fx_bits(float v)
{
    unsigned b;
    memcpy(&b, &v, 4);
    return b;
}
#endif

#define FX_FN __host__ __device__ __forceinline__

// sum X_q, sum i X_q and sum |i|^2 X_q.
template <int D>
FX_FN void fx_sums(const long long (&X)[Lattice<D>::Q], long long &M, long long (&J)[3], long long &E)
{
    constexpr int Q = Lattice<D>::Q;
    long long e1 = 0, e2 = 0;
    J[0] = J[1] = J[2] = 0;
#pragma unroll
    for (int q = 0; q < Q / 2; ++q) {
        const long long s = X[q] + X[Q - 1 - q], d = X[Q - 1 - q] - X[q];
        if (cnorm2<D>(q) == 1) e1 += s;
        else e2 += s;
        // direction Q - 1 - q is -q's: d carries the sign of its components
        if (cx<D>(q)) J[0] += cx<D>(q) < 0 ? d : -d;
        if (cy<D>(q)) J[1] += cy<D>(q) < 0 ? d : -d;
        if (cz<D>(q)) J[2] += cz<D>(q) < 0 ? d : -d;
    }
    M = e1 + e2 + X[Q / 2];
    E = e1 + 2 * e2;
}

// v = hi 2^32 + lo with lo signed: products of two splits then need signed
// 32 x 32 -> 64-bit multiply-adds only.  v < 2^63 - 2^31 (hi would wrap).
struct FxSplit {
    int hi, lo;
};
FX_FN FxSplit fx_split(long long v)
{
    FxSplit r;
    r.lo = (int)v;
    r.hi = (int)(v >> 32) + (int)((unsigned)r.lo >> 31);
    return r;
}
// Constants of the fixed-point step, "qN" meaning the value times 2^N:
//   h_i of class m = |i|^2:  h = al[m] + be[m] d + ga[m] |j|^2 + (linear and
//   quadratic terms in i.j),  d = E2/n - |j|^2 - d0,  d0 = c/K,
//   al = omega w,  be = omega w (m K - c) K / (m4 - c^2),  ga = omega w c5
// (P_i of Eq. WeqAlgo with alpha1 and alpha2 written out: alpha2 is
// K d / (m4 - c^2)), and for the axis class c3 = omega w_1 c3, c4 = omega w_1
// c4; the diagonal class has w_2 = w_1 / 2 (D3Q19) or w_1 / 4 (D2Q9) exactly,
// so its terms are shifts of these.
struct FixConst {
    FxSplit omc;            // q62: 1 - omega
    long long al[3];        // q62
    FxSplit be[3];          // q62
    FxSplit ga[2];          // q62, rest and axis class
    FxSplit c3, c4;         // q62
    long long d0;           // q60
    int h_unit;             // h_i as formed: units of 2^h_unit
    int valid;              // 0: every site in double
};
constexpr long long kFxOne = 1LL << 62;   // 1.0 in q62

// The smallest and largest biased exponent of a nonzero component's largest
// value that the fixed-point step takes (no result near the ends of the
// double range; below the 1e30 that the step flags as non-finite).
constexpr int kFxMinExp = 128, kFxMaxExp = 1023 + 90;
constexpr int kFxZeroExp = 2000;    // aligned to this exponent everything is shifted out

// The double with words (hi, lo) in units of 2^(eb - 1080), truncated.
FX_FN long long fx_align(unsigned hi, unsigned lo, int eb)
{
    const int e = (int)((hi >> 20) & 0x7ffu);
    // subnormals and zeros get a leading one they do not have; they are
    // shifted out (e = 0, eb >= kFxMinExp)
    const unsigned long long m = ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32) | lo;
    const long long x = (long long)fx_shr(m << 11, eb - e + 6);
    const long long s = (long long)((int)hi >> 31);
    return (x ^ s) - s;
}

FX_FN long long fx_wide(int a, int b) { return (long long)a * b; }
// a b / 2^64 without the product of the low words (at most a quarter of the
// last place): qA x qB -> q(A + B - 64).
FX_FN long long fx_mul(FxSplit a, FxSplit b)
{
    return fx_mad(a.hi, b.hi, fx_mad(a.hi, b.lo, fx_wide(a.lo, b.hi)) >> 32);
}

// t (units 2^(eb - 1078)) rounded to a double: one conversion, which takes
// the double pipe the step otherwise leaves idle (64 cycles against ~15
// integer instructions), and the exponent moved by shift = (eb - 1078) << 20.
FX_FN double fx_to_double(long long t, int shift)
{
    const double v = (double)t;
#ifdef __CUDA_ARCH__
    const int hi = __double2hiint(v);
    return __hiloint2double(hi ? hi + shift : 0, __double2loint(v));
#else
    return ldexp(v, shift / (1 << 20));
#endif
}

// t 2^unit as a double in integer operations (fx_to_double without the
// double pipe).
__device__ __forceinline__ double fx_to_double_int(long long t, int unit)
{
    const long long s = t >> 63;
    const unsigned long long a = (unsigned long long)((t ^ s) - s);
    if (a == 0ull) return 0.0;
    const int lz = __clzll((long long)a);       // >= 1: |t| < 2^63
    const unsigned long long m = (a << (lz - 1)) + 0x200u;      // leading bit at 62
    // leading bit 2^(63 - lz) of t: exponent unit + 63 - lz, one of it from the
    // leading bit itself (bit 20 of the high word)
    const unsigned hi = (unsigned)(m >> 42) + ((unsigned)(unit + 63 - lz + 1023 - 1) << 20);
    return __hiloint2double((int)(hi | ((unsigned)s & 0x80000000u)), (int)(unsigned)(m >> 10));
}

// omc X + h m in units of 4 U, rounded to nearest but for the products of the
// low words, which are left out (2^-58 of the largest value at most; they
// would take 3 of 9 multiplications on the pipe that bounds the kernel).
// |omc|, |h| <= 2^62 and |m| <= 19 * 2^58 keep the cross terms in 64 bits.
FX_FN long long fx_update(long long X, FxSplit omc, long long h, FxSplit m)
{
    const FxSplit x = fx_split(X), g = fx_split(h);
    const long long cross =
        fx_mad(m.hi, g.lo, fx_mad(m.lo, g.hi, fx_mad(x.hi, omc.lo, fx_mad(x.lo, omc.hi, 0x80000000LL))));
    return fx_mad(m.hi, g.hi, fx_mad(x.hi, omc.hi, cross >> 32));
}

// 1/x in q61 for nn = x 2^64, x in [1/2, 1): a single-precision reciprocal
// and two Newton steps r <- r + r (1 - x r) in integers, each product cut
// below 2^-62.
FX_FN long long fx_recip(unsigned long long nn)
{
    const unsigned nh = (unsigned)(nn >> 32), nl = (unsigned)nn;
    // 24 leading bits of x as a float in [1/2, 1); its reciprocal in q30
    const unsigned rb = fx_bits(fx_rcp(fx_float(0x3f000000u | ((nh >> 8) & 0x7fffffu))));
    const unsigned R0 = ((rb < 0x3fffffffu ? rb : 0x3fffffffu) << 7 | 0x40000000u) & 0x7fffffffu;
    const unsigned long long p = fx_umad(nh, R0, fx_umad(nl, R0, 0) >> 32);      // q62: x r
    const long long e0 = kFxOne - (long long)p;
    const long long r1 = ((long long)R0 << 32) + (fx_wide((int)R0, (int)(e0 >> 10)) >> 20);      // q62
    const unsigned rh = (unsigned)((unsigned long long)r1 >> 32), rl = (unsigned)r1;
    const unsigned long long x1 = fx_umad(nh, rh, fx_umad(nh, rl, 0) >> 32) + (fx_umad(nl, rh, 0) >> 32);
    const int e1 = (int)(kFxOne - (long long)x1);       // < 2^20
    const long long r = r1 + (fx_wide((int)(rh >> 1), e1) >> 29);       // q62, up to 2^63
    return (long long)((unsigned long long)r >> 1);
}

// J/n and E2/n - |j|^2 of a site.
struct FixRatios {
    FxSplit j[3];       // q64
    long long jj;       // q64: |j|^2
    long long ej;       // q60: E2/n - |j|^2
};

// From n, J, E2 (all in the same units); false outside the range of the form
// (decided on high words): |j_a| < 3/8 (so |j|^2 < 1/2), 0 <= E2/n < 15/8.
template <int D> FX_FN bool fx_ratios(long long n, const long long (&J)[3], long long E, FixRatios &o)
{
    const int nh = (int)(n >> 32), Eh = (int)(E >> 32), lim = (nh >> 2) + (nh >> 3);
    auto mag = [](long long v) { return abs((int)(v >> 32)); };
    bool ok = Eh >= 0 && (Eh >> 1) < nh - (nh >> 4) && mag(J[0]) < lim && mag(J[1]) < lim;
    if (D == 3) ok = ok && mag(J[2]) < lim;
    const int lz = fx_clz((unsigned)nh);    // 1..31 where ok
    const FxSplit r = fx_split(fx_recip((unsigned long long)n << lz));
    o.jj = 0;
#pragma unroll
    for (int a = 0; a < D; ++a) {
        o.j[a] = fx_split(fx_mul(fx_split(J[a] << lz), r) << 3);
        o.jj += fx_mul(o.j[a], o.j[a]);
    }
    o.ej = 2 * fx_mul(fx_split((E >> 1) << (lz - 1)), r) - (o.jj >> 4);
    return ok;
}

// h_i of all directions as ten basis values (q62).
struct FixCoef {
    long long b0, b1, b2;           // class constants
    long long B[3];                 // axis class: c3 j_a
    long long qd[3];                // axis class: c4 j_a^2
    long long qo[3];                // axis class: c4 j_a j_b, (a, b) = (0,1), (0,2), (1,2)
};

// From j (q64), |j|^2 (q64) and d = E2/n - |j|^2 - d0 (q60); false where |d|
// is not well below 1 or an |h_i| might reach 1 (the terms not looked at are bounded by
// |j_a| < 3/8, see make_fix_const).
template <int D>
FX_FN bool fx_basis(const FxSplit (&j)[3], long long jj, long long d60, const FixConst &k, FixCoef &c)
{
    auto mag = [](long long v) { return abs((int)(v >> 32)); };
#pragma unroll
    for (int a = 0; a < D; ++a) {
        c.B[a] = fx_mul(k.c3, j[a]);
        c.qd[a] = fx_mul(k.c4, fx_split(fx_mul(j[a], j[a])));
    }
    c.qo[0] = fx_mul(k.c4, fx_split(fx_mul(j[0], j[1])));
    if (D == 3) {
        c.qo[1] = fx_mul(k.c4, fx_split(fx_mul(j[0], j[2])));
        c.qo[2] = fx_mul(k.c4, fx_split(fx_mul(j[1], j[2])));
    }
    const FxSplit d = fx_split(d60 << 3), s = fx_split(jj);     // q63, q64
    const long long g1 = fx_mul(k.ga[1], s);
    c.b0 = k.al[0] + fx_mul(k.ga[0], s) + 2 * fx_mul(k.be[0], d);
    c.b1 = k.al[1] + g1 + 2 * fx_mul(k.be[1], d);
    c.b2 = k.al[2] + (g1 >> (D == 3 ? 1 : 2)) + 2 * fx_mul(k.be[2], d);
    constexpr int q62 = 1 << 30;
    return mag(d60) < (1 << 28) - (1 << 20) && mag(c.b0) < q62 && mag(c.b1) < q62 / 2 && mag(c.b2) < q62 / 4;
}

template <int D> FX_FN bool fx_coefficients(long long n, const long long (&J)[3], long long E, const FixConst &k,
                                            FixCoef &c)
{
    FixRatios r;
    const bool ok = fx_ratios<D>(n, J, E, r);
    return fx_basis<D>(r.j, r.jj, r.ej - k.d0, k, c) && ok;
}

// Calls f(q, h_q) for every direction, h_q in q62: the terms are shared
// within the pairs +-a and the quadruples +-a +-b.
template <int D, class F> FX_FN void fx_each_h(const FixCoef &c, F &&f)
{
    constexpr int Q = Lattice<D>::Q, sh = D == 3 ? 1 : 2;       // w_2 = w_1 >> sh
    f(Q / 2, c.b0);
#pragma unroll
    for (int a = 0; a < D; ++a) {
        const int q = direction_of<D>(a == 0, a == 1, a == 2);
        const long long A = c.b1 + c.qd[a];
        f(q, A + c.B[a]);
        f(Q - 1 - q, A - c.B[a]);
    }
#pragma unroll
    for (int a = 0; a < D - 1; ++a)
#pragma unroll
        for (int b = a + 1; b < D; ++b) {
            const long long A = c.b2 + ((c.qd[a] + c.qd[b]) >> sh), C = c.qo[a + b - 1] >> (sh - 1);
            const long long S = (c.B[a] + c.B[b]) >> sh, T = (c.B[a] - c.B[b]) >> sh;
            const long long P = A + C, M = A - C;
            const int qp = direction_of<D>(a == 0, a == 1 || b == 1, b == 2);
            const int qm = direction_of<D>(a == 0, a == 1 ? 1 : (b == 1 ? -1 : 0), b == 2 ? -1 : 0);
            f(qp, P + S);
            f(Q - 1 - qp, P - S);
            f(qm, M + T);
            f(Q - 1 - qm, M - T);
        }
}

// Double-double arithmetic for the constants (host): rounding them to double
// first would leave errors of 2^-53 in every h_i, the same at every site and
// step.  std::fma rounds once on every host.
struct Dd {
    double h, l;
    Dd(double a, double b = 0.0) : h(a + b), l(b - (h - a)) {}      // |a| >= |b|
};
inline Dd operator+(Dd a, Dd b)
{
    const double s = a.h + b.h, v = s - a.h;
    return Dd(s, ((a.h - (s - v)) + (b.h - v)) + (a.l + b.l));
}
inline Dd operator-(Dd a) { return Dd(-a.h, -a.l); }
inline Dd operator*(Dd a, Dd b)
{
    const double p = a.h * b.h;
    return Dd(p, fma(a.h, b.h, -p) + (a.h * b.l + a.l * b.h));
}
inline Dd reciprocal(Dd a)
{
    const Dd r(1.0 / a.h);
    return r + r * (Dd(1.0) + -(a * r));
}

// Host: 1 - omega in q62 for omega in [0, 2] (omega - 1 is exact from 1 on,
// and neither branch leaves 64 bits: 2.0 itself is 2^63).
inline long long fx_one_minus(double omega)
{
    const double q62 = 4611686018427387904.0;
    return omega < 1.0 ? kFxOne - llrint(omega * q62) : -llrint((omega - 1.0) * q62);
}

// Host: the constants, false where they leave the form's range (then the
// double-precision kernel steps the lattice).  normalise: h_i for omega 2^k in
// [1/2, 1) instead of a smaller omega, so that it keeps its digits (for the
// update in double, which takes it in units of 2^-(62 + k): from 2^-900 on, so
// that h_i's last place is a normal double).
inline bool make_fix_const(const HostConsts &k, double omega, bool normalise, FixConst *o)
{
    *o = FixConst{};
    if (!(omega >= 0x1p-900 && omega <= 2.0)) return false;
    o->h_unit = -62;
    if (normalise && omega < 0.5) {
        int e;
        omega = frexp(omega, &e);
        o->h_unit += e;
    }
    bool ok = k.w[2] * (k.d == 3 ? 2.0 : 4.0) == k.w[1];     // the diagonal class is shifts of the axis class
    auto fix = [&](Dd v, double scale, double lim) {
        ok = ok && v.h < lim && v.h > -lim;
        return ok ? llrint(v.h * scale) + llrint(v.l * scale) : 0LL;
    };
    const double q62 = 4611686018427387904.0;
    const Dd K(k.K), c(k.c), inv = reciprocal(Dd(k.m) + -(c * c)), om(omega);
    o->omc = fx_split(fx_one_minus(omega));
    for (int m = 0; m < 3; ++m) {
        const Dd ow = om * Dd(k.w[m]);
        o->al[m] = fix(ow, q62, 1.0);
        o->be[m] = fx_split(fix(ow * (Dd(m) * K + -c) * K * inv, q62, 1.99));
        if (m < 2) o->ga[m] = fx_split(fix(ow * K * Dd(k.alpha5), q62, 1.99));
    }
    // with |j_a| < 3/8 and class constants below 1, 1/2 and 1/4, |h_i| < 1:
    // B = c3 3/8 and q = c4 9/64 bound the linear and quadratic terms
    const Dd c3 = om * Dd(k.w[1]) * Dd(2.0) * K * Dd(k.alpha3), c4 = om * Dd(k.w[1]) * Dd(4.0) * K * K * Dd(k.alpha4);
    const double B = fabs(c3.h) * 0.375, q = fabs(c4.h) * 0.140625, half = k.d == 3 ? 0.5 : 0.25;
    ok = ok && 0.5 + q + B < 0.99 && 0.25 + half * (2 * q + 2 * B) + 2 * half * q < 0.99;
    o->c3 = fx_split(fix(c3, q62, 1.99));
    o->c4 = fx_split(fix(c4, q62, 1.99));
    o->d0 = fix(c * reciprocal(K), q62 / 4.0, 2.0);
    o->valid = ok;
    return ok;
}

// n / d for n < 2^31 as a multiplication: (n * m) >> s.
struct FastDiv {
    unsigned m;
    int s;
};
inline FastDiv make_fast_div(unsigned d)
{
    int k = 0;
    while ((1ull << k) < d) ++k;
    FastDiv f;
    f.s = 31 + k;
    f.m = (unsigned)(((1ull << f.s) + d - 1) / d);
    return f;
}
FX_FN int fast_div(int n, FastDiv f) { return (int)(((unsigned long long)(unsigned)n * f.m) >> f.s); }

// The lattice as rows of 8-site chunks, one warp each (a chunk is 8
// consecutive x of a row, the last one of a row partly idle).
struct Chunks {
    int per_row, total;
    FastDiv row, y;     // divisions by per_row and by ny
};
inline Chunks make_chunks(const Grid &g)
{
    Chunks c;
    c.per_row = (g.nx + 7) / 8;
    c.total = (int)((int64_t)c.per_row * g.ny * g.nz);
    c.row = make_fast_div((unsigned)c.per_row);
    c.y = make_fast_div((unsigned)g.ny);
    return c;
}
constexpr int kFixBlock = 64;

// The chunk of a thread's warp, `threads` per block.  Warps are counted, not
// threads: 32 threads per chunk wrap 32 bits from 2^27 chunks on (2^30 sites,
// or 2^27 rows of up to 8), and chunks come up to the 2^31 - 64 sites of a
// lattice.
FX_FN int chunk_of_thread(unsigned block, unsigned thread, int threads)
{
    return (int)(block * (unsigned)(threads / 32) + (thread >> 5));
}

__device__ __forceinline__ long long fx_from_lane0(long long v)
{
    return __shfl_sync(0xffffffffu, v, 0, 4);   // the site's lane 0 (component f)
}

// The magnetic-field term: the rotation of the spins by the unit quaternion
// (w, x, y, z) of site s.  Lane c = 1..3 holds component c; in cyclic order
// p, q, r = its own component of the vector part, the next and the one after,
// its row of the rotation matrix is
//   1 - 2 (q^2 + r^2)  (own),  2 (p q - w r)  (next),  2 (p r + w q)  (after);
// lane 0 (f) has the identity's.  For the uniform field the host gives each
// lane's row in that order.
struct FixField {
    double r[4][3];
};
inline void make_fix_field(const double (&rot)[9], FixField *o)
{
    for (int c = 0; c < 4; ++c)
        for (int b = 0; b < 3; ++b) o->r[c][b] = c ? rot[3 * (c - 1) + (c - 1 + b) % 3] : (b ? 0.0 : 1.0);
}
FX_FN int fx_next_lane(int c) { return c == 3 ? 1 : c + 1; }
FX_FN int fx_prev_lane(int c) { return c <= 1 ? 3 : c - 1; }
template <int FIELD>
__device__ __forceinline__ void fx_rotation_row(const FixField &uq, const DQuad *qf, int s, int c, double (&r)[3])
{
    if constexpr (FIELD == FIELD_SITE) {
        const double *v = reinterpret_cast<const double *>(qf + s);
        const int own = c ? c : 1;
        const double w = v[0], p = v[own], q = v[fx_next_lane(own)], t = v[fx_prev_lane(own)];
        r[0] = 1.0 - 2.0 * (q * q + t * t);
        r[1] = 2.0 * (p * q - w * t);
        r[2] = 2.0 * (p * t + w * q);
        if (c == 0) {
            r[0] = 1.0;
            r[1] = r[2] = 0.0;
        }
    } else if constexpr (FIELD == FIELD_UNIFORM) {
#pragma unroll
        for (int b = 0; b < 3; ++b) r[b] = uq.r[c][b];
    } else {
        r[0] = r[1] = r[2] = 0.0;
    }
}
// The exponent of a rotated component.  The three components (own, next,
// after) keep alignments e[b] of their own; the result is in units of
// 2^(E - 1080) with 2^E at least sum_b |r_b| 2^e_b and at most twice that, so
// that a component small beside the others keeps its digits as far as the
// rotation does not mix them in.  e[b] <= 0: the component is zero.
FX_FN int fx_mixed_exponent(const unsigned (&rh)[3], const int (&e)[3])
{
    int top = 0, x[3];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        const int er = (int)((rh[b] >> 20) & 0x7ffu);       // |r_b| < 2^(er - 1022)
        x[b] = er && e[b] > 0 ? e[b] + er - 1022 : -4000;
        top = x[b] > top ? x[b] : top;
    }
    // sum_b |r_b| 2^(e_b - top), each term below 1 (the largest at least 1/2)
    float t = 0.f;
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        const int k = x[b] - top;
        if (k > -100) t += fx_float((((rh[b] & 0xfffffu) + 1u) << 3) + (unsigned)((126 + k) << 23));
    }
    // (the sum of X_b r_b stays below 2^58 where t 2^top <= 2^E)
    const int E = top + (t > 1.f ? (t > 2.f ? 2 : 1) : (t > 0.51f ? 0 : -1));
    return E > 64 ? E : 64;     // (the results' exponents stay positive)
}
// r 2^(e - E) in q62 (at most 1).
FX_FN FxSplit fx_scaled_row(unsigned rh, unsigned rl, int e, int E)
{
    const bool none = ((rh >> 20) & 0x7ffu) == 0u || e <= 0;
    return fx_split(none ? 0 : fx_align(rh, rl, 1018 + E - e));
}
__device__ __forceinline__ FxSplit fx_shfl(FxSplit v, int lane)
{
    return FxSplit{__shfl_sync(0xffffffffu, v.hi, lane, 4), __shfl_sync(0xffffffffu, v.lo, lane, 4)};
}

// The step of one component in double (collide's formulas), for warps with a
// site outside the fixed-point form; lane c = 0 holds f, 1..3 the spins.
// FD: the equilibrium is built from the component R of a rebuilt density
// matrix instead of M (the flag then looks at n only).  FIELD: the spins are
// rotated, r the lane's row (fx_rotation_row).
template <int D, bool FD, bool FIELD>
__device__ __forceinline__ unsigned fx_collide_double(unsigned long long (&w)[Lattice<D>::Q], const Coll<double> &k,
                                                      double R, const double (&r)[3])
{
    constexpr int Q = Lattice<D>::Q;
    double M = 0.0, J[3] = {0.0, 0.0, 0.0}, E = 0.0;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const double v = __longlong_as_double((long long)w[q]);
        M += v;
        if (cx<D>(q)) J[0] += cx<D>(q) * v;
        if (cy<D>(q)) J[1] += cy<D>(q) * v;
        if (cz<D>(q)) J[2] += cz<D>(q) * v;
        if (cnorm2<D>(q)) E += cnorm2<D>(q) * v;
    }
    const unsigned all = 0xffffffffu;
    const double n = __shfl_sync(all, M, 0, 4), rn = 1.0 / n;
    const double jx = __shfl_sync(all, J[0], 0, 4) * rn, jy = __shfl_sync(all, J[1], 0, 4) * rn;
    const double jz = D == 3 ? __shfl_sync(all, J[2], 0, 4) * rn : 0.0;
    const double jj = jx * jx + jy * jy + jz * jz;
    const double be = k.K * (__shfl_sync(all, E, 0, 4) * rn - jj);
    const double a2 = (be - k.c) * k.inv_mc2, a2K = a2 * k.K;
    const double b0 = fma(k.c5, jj, 1.0 - k.c * a2);
    const double bq[3] = {b0, b0 + a2K, b0 + 2.0 * a2K};
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const double v = __longlong_as_double((long long)w[q]);
        const double t = cx<D>(q) * jx + cy<D>(q) * jy + cz<D>(q) * jz;
        const double h = k.w[cnorm2<D>(q)] * fma(t, fma(k.c4, t, k.c3), bq[cnorm2<D>(q)]);
        w[q] = (unsigned long long)__double_as_longlong(fma(k.omega, fma(h, FD ? R : M, -v), v));
    }
    if constexpr (FIELD) {
        const int c = threadIdx.x & 3;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const double v = __longlong_as_double((long long)w[q]);
            const double v1 = __shfl_sync(all, v, fx_next_lane(c), 4), v2 = __shfl_sync(all, v, fx_prev_lane(c), 4);
            if (c) w[q] = (unsigned long long)__double_as_longlong(r[0] * v + r[1] * v1 + r[2] * v2);
        }
    }
    double sum = (threadIdx.x & 3) ? fabs(M) : fabs(be);
    sum += __shfl_xor_sync(all, sum, 1, 4);
    sum += __shfl_xor_sync(all, sum, 2, 4);
    unsigned flag = 0u;
    if (!(n > 0.0)) flag |= n == n ? FLAG_NONPOSITIVE : FLAG_NONFINITE;
    if (!FD && !(sum < 1e30)) flag |= FLAG_NONFINITE;
    return flag;
}

// One step of FP64 storage (QLBM_FP64 and QLBM_FP64_DF): an
// even or odd AA step in place (addressing as k_step_aa; src and dst the same
// planes) or the two-buffer step of the reverse mode (as k_step_push), with
// the same arithmetic in all three.
// With FD the equilibrium is built from a density matrix per site (rho, Eq.
// WeqDiscr) instead of the populations' own; P_i keeps their u and eps.
// With a field the rotation R is folded into the relaxation: sum_b (1 - omega)
// R_ab X_b + h (R M)_a, the other two components from the neighbouring lanes,
// each with its own alignment (fx_mixed_exponent).
// DBL: the populations are updated in double from the integer sums and
// coefficients (fix_double_below).
// rg: the largest high word (magnitude) of a component that counts as zero,
// and the smallest that is non-finite; QLBM_FP64_DF has single precision's
// exponent range there (2^-126, 2^128).
struct FixRange {
    unsigned zero, bad;
};
inline FixRange make_fix_range(bool single) { return single ? FixRange{(897u << 20) - 1u, 1151u << 20} : FixRange{0u, ~0u}; }
enum : int { FIX_EVEN = 0, FIX_ODD = 1, FIX_PUSH = 2 };
// The omega below which the populations are updated in double, two multiply-
// adds each.  The fixed-point update errs by up to 1.3 x 2^-56 of the
// component's largest value whatever omega is, the double step by a few 2^-53
// of omega h M and by 2^-54 of the result: for a population much smaller than
// the largest the double step is the better one where omega is small.  The
// line lies where its errors reach the double step's on such populations, in
// 2^-53 of the terms of each result (largest and root mean square; fixed point,
// double step; one population of 1 and the others near 1e-6, D2Q9): omega =
// 0.75: 1.5 0.35, 2.3 0.51; 0.65: 2.0 0.42, 2.2 0.51; 0.6: 2.2 0.46, 2.1 0.51;
// 0.5: 2.5 0.52, 2.0 0.51; with a field 0.7: 1.7
// 0.22, 2.0 0.28; 0.65: 2.0 0.23, 1.7 0.28.  (Populations near equilibrium: 0.4:
// 2.9 0.44, 3.3 0.65.)  In double D3Q19 128^3 takes 659 us instead of 504, with a
// field 1436 instead of 702, D2Q9 64^2 2.9 instead of 2.3 (the double pipe; 1485,
// 2207 and 8.2 with everything in double).  The change h M - omega W in
// integers at omega's own scale and one addition in double instead was as
// exact and slower (749 us; 64^2 2.96).  QLBM_FP64_DF with a field, stated to
// 1e-14 of the largest, keeps the fixed-point update further down.
inline double fix_double_below(int prec, int field)
{
    return field == FIELD_NONE ? 0.65 : prec == QLBM_FP64 ? 0.7 : 0.0625;
}
template <int D, int MODE, bool FD, int FIELD, bool DBL>
__global__ void __launch_bounds__(kFixBlock, D == 3 ? 8 : 14)
k_step_fix(const Planes<double, Lattice<D>::Q> src, const Planes<double, Lattice<D>::Q> dst, Grid g, FixConst fc,
           Coll<double> k, Chunks ch, FixRange rg, const DQuad *__restrict__ rho, FixField uq,
           unsigned *__restrict__ flags)
{
    constexpr int Q = Lattice<D>::Q;
    const unsigned all = 0xffffffffu;
    wait_for_previous();
    const int chunk = chunk_of_thread(blockIdx.x, threadIdx.x, kFixBlock);
    if (chunk >= ch.total) return;      // the whole warp
    const int c = threadIdx.x & 3;
    const int row = fast_div(chunk, ch.row);
    SiteIdx si;
    const int x = (chunk - row * ch.per_row) * 8 + ((threadIdx.x & 31) >> 2);
    const bool active = x < g.nx;
    si.x = active ? x : g.nx - 1;       // idle lanes work on the row's last site and store nothing
    si.z = fast_div(row, ch.y);
    si.y = row - si.z * g.ny;
    si.s = row * g.nx + si.x;
    const NbOff nb = nb_offsets(g, si);
    // component c of the stored vector at s
    auto at = [c](DQuad *plane, int s) { return reinterpret_cast<unsigned long long *>(plane + s) + c; };
    // population q is read from slot q at x (even, push) or slot opposite(q)
    // at x - e_q (odd)
    auto load = [&](int q) {
        return MODE == FIX_ODD ? *at(src.p[opposite<D>(q)], nb_at(nb, si.s, -cx<D>(q), -cy<D>(q), -cz<D>(q)))
                               : *at(src.p[q], si.s);
    };
    unsigned long long w[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) w[q] = load(q);
    // alignment to the component's largest value
    unsigned mx = 0u;
#pragma unroll
    for (int q = 0; q < Q; ++q) mx = max(mx, (unsigned)(w[q] >> 32) & 0x7fffffffu);
    unsigned flag = mx >= rg.bad ? FLAG_NONFINITE : 0u;
    // a component that counts as zero is shifted out altogether
    const bool zero = mx <= rg.zero;
    const int eb = zero ? kFxZeroExp : (int)(mx >> 20);
    double r[3];
    fx_rotation_row<FIELD>(uq, k.qf, si.s, c, r);
    double R = 0.0;
    if (FD) R = reinterpret_cast<const double *>(rho + si.s)[c];
    bool fine = fc.valid && __all_sync(all, zero || (eb >= kFxMinExp && eb <= kFxMaxExp));
    if (fine) {
        long long X[Q], M, J[3], E;
#pragma unroll
        for (int q = 0; q < Q; ++q) X[q] = fx_align((unsigned)(w[q] >> 32), (unsigned)w[q], eb);
        fx_sums<D>(X, M, J, E);
        // the coefficients from f's sums (formed by the site's four lanes alike)
#pragma unroll
        for (int a = 0; a < D; ++a) J[a] = fx_from_lane0(J[a]);
        FixCoef cf;
        fine = __all_sync(all, fx_coefficients<D>(fx_from_lane0(M), J, fx_from_lane0(E), fc, cf));
        if (fine && DBL) {
            const double m = FD ? R : fx_to_double(M, zero ? 0 : (eb - 1080) * (1 << 20));
            if constexpr (FIELD == FIELD_NONE) {
                fx_each_h<D>(cf, [&](int q, long long h) {
                    const double v = zero ? 0.0 : __longlong_as_double((long long)w[q]);
                    w[q] = (unsigned long long)__double_as_longlong(
                        fma(fx_to_double_int(h, fc.h_unit), m, fma(-k.omega, v, v)));
                });
            } else {
                const int n1 = fx_next_lane(c), n2 = fx_prev_lane(c);
                // f: (f - omega f) + h n; spins: (1 - omega) R s + h R S
                const double m1 = __shfl_sync(all, m, n1, 4), m2 = __shfl_sync(all, m, n2, 4), omc = 1.0 - k.omega;
                const double rm = c ? r[0] * m + r[1] * m1 + r[2] * m2 : m;     // of R S
#pragma unroll
                for (int b = 0; b < 3; ++b) r[b] *= omc;
                if (c == 0) r[0] = -k.omega;
                fx_each_h<D>(cf, [&](int q, long long h) {
                    const double v = zero ? 0.0 : __longlong_as_double((long long)w[q]);
                    const double v1 = __shfl_sync(all, v, n1, 4), v2 = __shfl_sync(all, v, n2, 4);
                    const double t = fma(r[1], v1, r[2] * v2);
                    w[q] = (unsigned long long)__double_as_longlong(
                        fma(fx_to_double_int(h, fc.h_unit), rm, fma(r[0], v, c ? t : v)));
                });
            }
        } else if (fine) {
            if (FD) {       // rho's component in the units of M
                const int rh = __double2hiint(R), e = (rh >> 20) & 0x7ff;
                const bool none = e <= eb - 70;     // below U / 2^13
                fine = __all_sync(all, none || (e < eb + 5 && !zero));
                M = none ? 0 : __double2ll_rn(__hiloint2double(rh + (1080 - eb) * (1 << 20), __double2loint(R)));
            }
            if constexpr (FIELD == FIELD_NONE) {
                const int shift = (eb - 1078) * (1 << 20);
                const FxSplit m = fx_split(M);
                fx_each_h<D>(cf, [&](int q, long long h) {
                    w[q] = (unsigned long long)__double_as_longlong(
                        fx_to_double(fx_update(X[q], fc.omc, h, m), shift));
                });
            } else {
                const int n1 = fx_next_lane(c), n2 = fx_prev_lane(c), e0 = zero ? 0 : eb;
                const int e[3] = {e0, __shfl_sync(all, e0, n1, 4), __shfl_sync(all, e0, n2, 4)};
                const unsigned rh[3] = {(unsigned)__double2hiint(r[0]), (unsigned)__double2hiint(r[1]),
                                        (unsigned)__double2hiint(r[2])};
                const int E = fx_mixed_exponent(rh, e), shift = (E - 1078) * (1 << 20);
                FxSplit rt[3];
#pragma unroll
                for (int b = 0; b < 3; ++b) rt[b] = fx_scaled_row(rh[b], (unsigned)__double2loint(r[b]), e[b], E);
                FxSplit m = fx_split(M);
                const FxSplit m1 = fx_shfl(m, n1), m2 = fx_shfl(m, n2);
                const long long rm = fx_mul(rt[0], m) + fx_mul(rt[1], m1) + fx_mul(rt[2], m2);
                if (c) m = fx_split(rm ? (rm + 1) << 2 : 0);       // (a zero component stays zero)
#pragma unroll
                for (int b = 0; b < 3; ++b)
                    rt[b] = c ? fx_split(fx_mul(fc.omc, rt[b]) << 2) : (b ? FxSplit{0, 0} : fc.omc);
                fx_each_h<D>(cf, [&](int q, long long h) {
                    const FxSplit x = fx_split(X[q]), x1 = fx_shfl(x, n1), x2 = fx_shfl(x, n2), g = fx_split(h);
                    long long t = fx_mad(x.hi, rt[0].lo, fx_mad(x.lo, rt[0].hi, 0x80000000LL));
                    t = fx_mad(x1.hi, rt[1].lo, fx_mad(x1.lo, rt[1].hi, t));
                    t = fx_mad(x2.hi, rt[2].lo, fx_mad(x2.lo, rt[2].hi, t));
                    t = fx_mad(m.hi, g.lo, fx_mad(m.lo, g.hi, t)) >> 32;
                    t = fx_mad(x2.hi, rt[2].hi, fx_mad(x1.hi, rt[1].hi, fx_mad(x.hi, rt[0].hi, t)));
                    w[q] = (unsigned long long)__double_as_longlong(fx_to_double(fx_mad(m.hi, g.hi, t), shift));
                });
            }
        }
    }
    if (!fine) {
#pragma unroll
        for (int q = 0; q < Q; ++q) w[q] = zero ? 0ull : load(q);
        flag |= fx_collide_double<D, FD, FIELD != FIELD_NONE>(w, k, R, r);
    }
    let_next_start();
    if (active) {
        const int so = si.s + g.zero;   // store addresses formed anew (see k_step_aa)
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            // to slot opposite(q) at x (even), or slot q at x + e_q (odd, push)
            if (MODE == FIX_EVEN) *at(dst.p[opposite<D>(q)], so) = w[q];
            else *at(dst.p[q], nb_at(nb, so, cx<D>(q), cy<D>(q), cz<D>(q))) = w[q];
        }
        if (flag) atomicOr(flags, flag);
    }
}

}  // namespace qlbm
