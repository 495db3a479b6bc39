// The FP64 step on the integer pipes (QLBM_FP64 storage, no field).
//
// GB300's double-precision pipe takes 64 issue cycles per warp instruction
// (measured: one DFMA per 64.0 cycles and sub-partition, whatever the number
// of warps; integer add, logic and minimum 1, shifts and 32-bit multiplies 2,
// the 32x32->64 multiply 4).  The step of k_step_aa<D, CodecF64> is bound by
// that pipe alone: ~445 double-precision instructions per D3Q19 site, at
// 128^3 1485 us for 2.55 GB that the copy rate moves in 376 us.  This file
// does the same step (Eqs. DiscrAvr, WeqAlgo, CollisionStep, TransportStep)
// without one double-precision instruction, in fixed point with more digits
// than a double has:
//
//   * a component's b values at a site are aligned to their largest one's
//     exponent: X = v / U as 64-bit integers with |X| < 2^58 (a double up to
//     32 times smaller than the largest is represented exactly, smaller ones
//     to 2^-58 of the largest); sums of b of them are exact in 64 bits;
//   * the equilibrium's coefficients h_i = omega w_i P_i are formed from the
//     ratios J/n and E2/n with 2^-60 steps, as sums of ten basis values
//     (class constants, i.j and its products), and
//       W_i' = (1 - omega) W_i + h_i M,   M = sum_j W_j of the component,
//     is one pair of 64 x 64-bit products whose 96 leading bits are kept;
//   * the result is normalised and rounded once to a double.
//
// Measured: D3Q19 128^3 1484 -> 835 us (even step), 2048 x 2 D2Q9 9.2 -> 4.1 us.
//
// Each step above errs by at most ~2^-57 of the component's largest value at
// the site, the result by its own rounding besides; the double-precision step
// rounds h, h M - W and W' (tests/test_gpu_fix64.py compares both with the
// 64-bit oracle).  Sites outside the fixed-point form's range (non-finite
// or extreme values, n <= 0, |j| >= 1/2, |h| >= 1) are stepped in double by
// their warp, with the same flags as k_step_aa.
//
// Layout: four lanes per site, lane c holding component c (f, s_x, s_y, s_z)
// of its b populations.  A site's vector of four doubles is 32 bytes, so a
// warp's 8-byte accesses cover 256 consecutive bytes (8 sites), every value
// is read and written once, and a thread keeps 19 values instead of 76 (20
// resident warps per SM instead of 8).
#pragma once

#include <math.h>

#include "internal.h"
#include "step.cuh"

namespace qlbm {

#ifdef __CUDA_ARCH__
__device__ __forceinline__ long long fx_mulhi(long long a, long long b) { return __mul64hi(a, b); }
__device__ __forceinline__ unsigned long long fx_umulhi(unsigned long long a, unsigned long long b)
{
    return __umul64hi(a, b);
}
__device__ __forceinline__ int fx_mulhi32(int a, int b) { return __mulhi(a, b); }
__device__ __forceinline__ int fx_clz(unsigned a) { return __clz((int)a); }
__device__ __forceinline__ int fx_clz64(unsigned long long a) { return __clzll((long long)a); }
__device__ __forceinline__ unsigned fx_shf_l(unsigned lo, unsigned hi, int s) { return __funnelshift_l(lo, hi, s); }
__device__ __forceinline__ unsigned fx_shf_r(unsigned lo, unsigned hi, int s) { return __funnelshift_r(lo, hi, s); }
// v >> s for any s >= 0 (0 from 64 on)
__device__ __forceinline__ unsigned long long fx_shr(unsigned long long v, int s)
{
    unsigned long long r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(s));
    return r;
}
__device__ __forceinline__ float fx_rcp(float x) { return __frcp_rn(x); }
#else   // the same functions for the host (arithmetic checks without a GPU)
inline long long fx_mulhi(long long a, long long b) { return (long long)(((__int128)a * b) >> 64); }
inline unsigned long long fx_umulhi(unsigned long long a, unsigned long long b)
{
    return (unsigned long long)(((unsigned __int128)a * b) >> 64);
}
inline int fx_mulhi32(int a, int b) { return (int)(((long long)a * b) >> 32); }
inline int fx_clz(unsigned a) { return a ? __builtin_clz(a) : 32; }
inline int fx_clz64(unsigned long long a) { return a ? __builtin_clzll(a) : 64; }
inline unsigned fx_shf_l(unsigned lo, unsigned hi, int s)
{
    s &= 31;
    return s ? (hi << s) | (lo >> (32 - s)) : hi;
}
inline unsigned fx_shf_r(unsigned lo, unsigned hi, int s)
{
    s &= 31;
    return s ? (lo >> s) | (hi << (32 - s)) : lo;
}
inline unsigned long long fx_shr(unsigned long long v, int s) { return s > 63 ? 0 : v >> s; }
inline float fx_rcp(float x) { return 1.0f / x; }
#endif

#define FX_FN __host__ __device__ __forceinline__

// Constants of the fixed-point step, "qN" meaning the value times 2^N:
//   h_i of class m = |i|^2:  h = al[m] + be[m] d + ga[m] |j|^2 + (linear and
//   quadratic terms in i.j),  d = E2/n - |j|^2,
//   al = omega w (1 - (m K - c) c inv),  be = omega w (m K - c) K inv,
//   ga = omega w c5,  inv = 1/(m4 - c^2)  (P_i of Eq. WeqAlgo with alpha1 and
//   alpha2 written out), and for the axis class c3 = omega w_1 c3,
//   c4 = omega w_1 c4; the diagonal class has w_2 = w_1 / 2 (D3Q19) or
//   w_1 / 4 (D2Q9) exactly, so its terms are shifts of these.
struct FixConst {
    long long omc;          // q62: 1 - omega
    long long al[3], be[3]; // q62
    long long ga[2];        // q62, rest and axis class
    long long c4;           // q62
    long long c3;           // q63
};
constexpr long long kFxOne = 1LL << 62;   // 1.0 in q62

// The smallest and largest biased exponent of a nonzero component's largest
// value that the fixed-point step takes (no result near the ends of the
// double range; below the 1e30 that the step flags as non-finite).
constexpr int kFxMinExp = 128, kFxMaxExp = 1023 + 90;

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

// v = hi 2^32 + lo with lo signed.
struct FxSplit {
    int hi, lo;
};
FX_FN FxSplit fx_split(long long v)
{
    FxSplit r;
    r.lo = (int)v;
    r.hi = (int)(v >> 32) - (r.lo >> 31);
    return r;
}

// The value t 2^32 + f (t the 64 leading bits, units 2^(e0 - 1078)) rounded
// to a double; e0 = 25 stands for a component that is zero throughout.
FX_FN unsigned long long fx_to_double(long long t, unsigned f, int e0)
{
    const unsigned s = (unsigned)(int)(t >> 63);
    unsigned a1 = (unsigned)(t >> 32) ^ s, a0 = (unsigned)t ^ s, a = f ^ s;
    int lz = fx_clz(a1), ex = e0;
    if (a1 == 0u && e0 != 25) {     // below 2^-24 of the largest value, or cancelled
        a1 = a0;
        a0 = a;
        a = 0u;
        ex -= 32;
        if (a1 == 0u) {
            a1 = a0;
            a0 = 0u;
            ex -= 32;
            if (a1 == 0u) return 0ull;
        }
        lz = fx_clz(a1);
    }
    const unsigned m1 = fx_shf_l(a0, a1, lz), m0 = fx_shf_l(a, a0, lz);
    unsigned long long r = ((unsigned long long)(m1 >> 11) << 32) | fx_shf_r(m0, m1, 11);
    r += (m0 >> 10) & 1u;
    r += (unsigned long long)(unsigned)((ex + 7 - lz) << 20) << 32;
    return r | ((unsigned long long)(s & 0x80000000u) << 32);
}

// omc X + h m as (t, f) of fx_to_double: units of 4 U, and the next 32 bits
// (of the products of the low words their high words).  |omc|, |h| <= 2^62 and
// |m| <= 19 * 2^58 keep the cross terms in 64 bits.
FX_FN void fx_update(long long X, FxSplit omc, long long h, FxSplit m, long long &t, unsigned &f)
{
    const FxSplit x = fx_split(X), g = fx_split(h);
    const long long cross = (long long)x.lo * omc.hi + (long long)x.hi * omc.lo + (long long)m.lo * g.hi +
                            (long long)m.hi * g.lo + ((long long)fx_mulhi32(x.lo, omc.lo) + fx_mulhi32(m.lo, g.lo));
    t = (long long)x.hi * omc.hi + (long long)m.hi * g.hi + (cross >> 32);
    f = (unsigned)cross;
}

// 1/x in q61 for nn = x 2^64, x in [1/2, 1): a single-precision reciprocal
// and two Newton steps r <- r + r (1 - x r) in integers.
FX_FN long long fx_recip(unsigned long long nn)
{
    const float xf = (float)(unsigned)(nn >> 40) * 0x1p-24f;
    const unsigned R0 = (unsigned)(fx_rcp(xf) * 1073741824.f);      // q30
    const unsigned nh = (unsigned)(nn >> 32), nl = (unsigned)nn;
    const unsigned long long p = (unsigned long long)nh * R0 + (((unsigned long long)nl * R0) >> 32);   // q62: x r
    const long long e0 = kFxOne - (long long)p;
    const unsigned long long r1 =
        ((unsigned long long)R0 << 32) + (unsigned long long)(((long long)R0 * (int)(e0 >> 10)) >> 20);  // q62
    const long long e1 = kFxOne - (long long)fx_umulhi(nn, r1);
    return (long long)((r1 + (unsigned long long)(((long long)(unsigned)(r1 >> 32) * e1) >> 30)) >> 1);
}

// h_i of all directions as ten basis values (q62).
struct FixCoef {
    long long b0, b1, b2;           // class constants
    long long B[3];                 // axis class: c3 j_a
    long long qd[3];                // axis class: c4 j_a^2
    long long qo[3];                // axis class: c4 j_a j_b, (a, b) = (0,1), (0,2), (1,2)
};

// From n, J, E2 (all in the same units); false outside the range of the form.
template <int D> FX_FN bool fx_coefficients(long long n, const long long (&J)[3], long long E, const FixConst &k,
                                            FixCoef &c)
{
    bool ok = n > 0;
    const long long half = n >> 1;
#pragma unroll
    for (int a = 0; a < D; ++a) ok = ok && J[a] < half && J[a] > -half;
    ok = ok && E >= 0 && (E >> 1) < n - (n >> 4);
    if (!ok) return false;
    const int lz = fx_clz64((unsigned long long)n);     // >= 1
    const long long r = fx_recip((unsigned long long)n << lz);
    long long j[3];     // q60
#pragma unroll
    for (int a = 0; a < D; ++a) j[a] = fx_mulhi(J[a] << (lz - 1), r);
    const long long e = fx_mulhi((E >> 1) << (lz - 1), r) << 3;     // q62
    long long sq[3], jj = 0;                                        // q62
#pragma unroll
    for (int a = 0; a < D; ++a) {
        sq[a] = fx_mulhi(j[a] << 3, j[a] << 3);
        jj += sq[a];
        c.B[a] = fx_mulhi(k.c3, j[a] << 2) << 1;
        c.qd[a] = fx_mulhi(k.c4, sq[a]) << 2;
    }
    c.qo[0] = fx_mulhi(k.c4, fx_mulhi(j[0] << 3, j[1] << 3)) << 2;
    if (D == 3) {
        c.qo[1] = fx_mulhi(k.c4, fx_mulhi(j[0] << 3, j[2] << 3)) << 2;
        c.qo[2] = fx_mulhi(k.c4, fx_mulhi(j[1] << 3, j[2] << 3)) << 2;
    }
    const long long d = e - jj, g1 = fx_mulhi(k.ga[1], jj) << 2;
    c.b0 = k.al[0] + ((fx_mulhi(k.be[0], d) + fx_mulhi(k.ga[0], jj)) << 2);
    c.b1 = k.al[1] + (fx_mulhi(k.be[1], d) << 2) + g1;
    c.b2 = k.al[2] + (fx_mulhi(k.be[2], d) << 2) + (g1 >> (D == 3 ? 1 : 2));
    // |h_i| < 1 for every direction: axis 1/2 + 1/8 + 1/4, diagonal at most
    // 1/4 + 1/8 + 1/8 + 1/4 (magnitudes by or-ing, exact for powers of two)
    auto mag = [](long long v) { return v ^ (v >> 63); };
    long long q = mag(c.qd[0]) | mag(c.qd[1]) | mag(c.qo[0]), B = mag(c.B[0]) | mag(c.B[1]);
    if (D == 3) {
        q |= mag(c.qd[2]) | mag(c.qo[1]) | mag(c.qo[2]);
        B |= mag(c.B[2]);
    }
    return mag(c.b0) < kFxOne && mag(c.b1) < kFxOne / 2 && ((mag(c.b2) | B) < kFxOne / 4) && q < kFxOne / 8;
}

// h_q (q62) of direction q (compile-time after unrolling).
template <int D> FX_FN long long fx_h(const FixCoef &c, int q)
{
    const int ex = cx<D>(q), ey = cy<D>(q), ez = cz<D>(q), cls = cnorm2<D>(q);
    constexpr int sh = D == 3 ? 1 : 2;      // w_2 = w_1 >> sh
    if (cls == 0) return c.b0;
    if (cls == 1) {
        const int a = ex ? 0 : (ey ? 1 : 2);
        const long long A = c.b1 + c.qd[a];
        return (ex + ey + ez > 0) ? A + c.B[a] : A - c.B[a];
    }
    const int a = ex ? 0 : 1, b = ez ? 2 : 1;
    const int ea = a == 0 ? ex : ey, eb = b == 2 ? ez : ey;
    const long long qo = c.qo[a + b - 1] >> (sh - 1);
    const long long A = c.b2 + ((c.qd[a] + c.qd[b]) >> sh) + (ea * eb > 0 ? qo : -qo);
    const long long L = (ea > 0 ? c.B[a] : -c.B[a]) + (eb > 0 ? c.B[b] : -c.B[b]);
    return A + (L >> sh);
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

// Host: the constants, false where they leave the form's range (then the
// double-precision kernel steps the lattice).
inline bool make_fix_const(const HostConsts &k, double omega, FixConst *o)
{
    if (!(omega > 0.0 && omega <= 2.0)) return false;
    bool ok = k.w[2] * (k.d == 3 ? 2.0 : 4.0) == k.w[1];     // the diagonal class is shifts of the axis class
    auto fix = [&](Dd v, double scale, double lim) {
        ok = ok && v.h < lim && v.h > -lim;
        return ok ? llrint(v.h * scale) + llrint(v.l * scale) : 0LL;
    };
    const double q62 = 4611686018427387904.0;
    const Dd K(k.K), c(k.c), inv = reciprocal(Dd(k.m) + -(c * c)), om(omega);
    o->omc = kFxOne - (omega < 1.0 ? llrint(omega * q62) : 2 * llrint(omega * q62 * 0.5));
    for (int m = 0; m < 3; ++m) {
        const Dd ow = om * Dd(k.w[m]), t = Dd(m) * K + -c;
        o->al[m] = fix(ow * (Dd(1.0) + -(t * c * inv)), q62, 1.99);
        o->be[m] = fix(ow * t * K * inv, q62, 1.99);
        if (m < 2) o->ga[m] = fix(ow * K * Dd(k.alpha5), q62, 1.99);
    }
    o->c4 = fix(om * Dd(k.w[1]) * Dd(4.0) * K * K * Dd(k.alpha4), q62, 1.99);
    o->c3 = fix(om * Dd(k.w[1]) * Dd(2.0) * K * Dd(k.alpha3), 2.0 * q62, 0.99);
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
constexpr int kFixBlock = 128;

__device__ __forceinline__ long long fx_from_lane0(long long v)
{
    return __shfl_sync(0xffffffffu, v, 0, 4);   // the site's lane 0 (component f)
}

// The step of one component in double (collide's formulas), for warps with a
// site outside the fixed-point form; lane c = 0 holds f, 1..3 the spins.
template <int D>
__device__ __forceinline__ unsigned fx_collide_double(unsigned long long (&w)[Lattice<D>::Q], const Coll<double> &k)
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
        w[q] = (unsigned long long)__double_as_longlong(fma(k.omega, fma(h, M, -v), v));
    }
    double sum = (threadIdx.x & 3) ? fabs(M) : fabs(be);
    sum += __shfl_xor_sync(all, sum, 1, 4);
    sum += __shfl_xor_sync(all, sum, 2, 4);
    unsigned flag = 0u;
    if (!(n > 0.0)) flag |= n == n ? FLAG_NONPOSITIVE : FLAG_NONFINITE;
    if (!(sum < 1e30)) flag |= FLAG_NONFINITE;
    return flag;
}

// One step of FP64 storage: an even or odd AA step in place (addressing as
// k_step_aa; src and dst the same planes) or the two-buffer step of the
// reverse mode (as k_step_push), with the same arithmetic in all three.
enum : int { FIX_EVEN = 0, FIX_ODD = 1, FIX_PUSH = 2 };
template <int D, int MODE>
__global__ void __launch_bounds__(kFixBlock, D == 3 ? 5 : 8)
k_step_fix(const Planes<double, Lattice<D>::Q> src, const Planes<double, Lattice<D>::Q> dst, Grid g, FixConst fc,
           Coll<double> k, Chunks ch, unsigned *__restrict__ flags)
{
    constexpr int Q = Lattice<D>::Q;
    const unsigned all = 0xffffffffu;
    const int chunk = (int)((blockIdx.x * kFixBlock + threadIdx.x) >> 5);
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
    const int eb = mx ? (int)(mx >> 20) : kFxMinExp;
    bool ok = eb >= kFxMinExp && eb <= kFxMaxExp;
    unsigned flag = 0u;
    if (__all_sync(all, ok)) {
        long long X[Q], M = 0, J[3] = {0, 0, 0}, e1 = 0, e2 = 0;
#pragma unroll
        for (int q = 0; q < Q; ++q) X[q] = fx_align((unsigned)(w[q] >> 32), (unsigned)w[q], eb);
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
        // the coefficients from f's sums (formed by the site's four lanes alike)
#pragma unroll
        for (int a = 0; a < D; ++a) J[a] = fx_from_lane0(J[a]);
        FixCoef cf;
        ok = fx_coefficients<D>(fx_from_lane0(M), J, fx_from_lane0(e1 + 2 * e2), fc, cf);
        if (__all_sync(all, ok)) {
            const FxSplit omc = fx_split(fc.omc), m = fx_split(M);
            const int e0 = mx ? eb : 25;
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                long long t;
                unsigned f;
                fx_update(X[q], omc, fx_h<D>(cf, q), m, t, f);
                w[q] = fx_to_double(t, f, e0);
            }
        } else {
#pragma unroll
            for (int q = 0; q < Q; ++q) w[q] = load(q);
            flag = fx_collide_double<D>(w, k);
        }
    } else {
        flag = fx_collide_double<D>(w, k);
    }
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
