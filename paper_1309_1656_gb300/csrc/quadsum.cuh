// Read-only site sums on the integer pipes, for every storage codec: the
// moments (Eq. DiscrAvr), the global sums (Eqs. GlobalDensity, GlobalVelocity,
// GlobalTotalEnergy) and the negative-equilibrium diagnostic.
//
// Formed in double, these kernels are bound by the double-precision pipe (64
// cycles per warp instruction and sub-partition, conversions included): ~150
// of them per D3Q19 site to convert the 76 populations and add them up, 3-4
// times what reading the populations takes.  Here each of a site's four
// lanes aligns its component's b values to their largest one's exponent and
// adds them as 64-bit integers (fix64.cuh: exact sums of values held to 2^-58
// of the largest), and only results are converted to double, 2 to 4
// conversions per lane.  The deviation codecs add the reference equilibrium's
// sums to f's, whose values are aligned to 1.  A warp with a site outside the
// form's range (non-finite or extreme values; for the ratios also n <= 0,
// |j| >= 3/8) forms its sums in double.
#pragma once

#include "fix64.cuh"
#include "kernels.cuh"

namespace qlbm {

// One stored value as the integer sums take it: key() orders magnitudes, its
// bits from KEY_EXP on are the biased exponent (bias BIAS); align() gives the
// value in units of 2^(e - BIAS - 57) for a largest exponent e >= MIN_EXP.  A
// component below that is taken times 2^LIFT (exact, subnormals included),
// where LIFT is not 0.
template <class Codec> struct QuadValue;
template <> struct QuadValue<CodecF64> {
    using Raw = unsigned long long;
    static constexpr int LIFT = 0, KEY_EXP = 20, BIAS = 1023, MIN_EXP = kFxMinExp, MAX_EXP = kFxMaxExp;
    static __device__ __forceinline__ Raw load(const CodecF64 &, const DQuad *p, int c)
    {
        return reinterpret_cast<const unsigned long long *>(p)[c];
    }
    static __device__ __forceinline__ unsigned key(Raw w) { return (unsigned)(w >> 32) & 0x7fffffffu; }
    static __device__ __forceinline__ Raw lift(Raw w) { return w; }
    static __device__ __forceinline__ long long align(Raw w, int e) { return fx_align((unsigned)(w >> 32), (unsigned)w, e); }
    static __device__ __forceinline__ double value(const CodecF64 &, Raw w, int, int)
    {
        return __longlong_as_double((long long)w);
    }
};

// A float's bits aligned likewise; subnormals are shifted out (MIN_EXP).
__device__ __forceinline__ long long fx_align_float(unsigned b, int e)
{
    const unsigned long long m = (unsigned long long)(((b & 0x7fffffu) | 0x800000u) << 8) << 32;
    const long long x = (long long)fx_shr(m, e - (int)((b >> 23) & 0xffu) + 6);
    const long long s = (long long)((int)b >> 31);
    return (x ^ s) - s;
}
__device__ __forceinline__ unsigned fx_lift_float(unsigned b) { return __float_as_uint(__uint_as_float(b) * 0x1p96f); }
struct QuadValueFloat {
    using Raw = unsigned;
    static constexpr int LIFT = 96, KEY_EXP = 23, BIAS = 127, MIN_EXP = 66, MAX_EXP = 127 + 90;
    static __device__ __forceinline__ unsigned key(Raw w) { return w & 0x7fffffffu; }
    static __device__ __forceinline__ Raw lift(Raw w) { return fx_lift_float(w); }
    static __device__ __forceinline__ long long align(Raw w, int e) { return fx_align_float(w, e); }
};
template <> struct QuadValue<CodecF32> : QuadValueFloat {
    static __device__ __forceinline__ Raw load(const CodecF32 &, const float4 *p, int c)
    {
        return reinterpret_cast<const unsigned *>(p)[c];
    }
    static __device__ __forceinline__ double value(const CodecF32 &k, Raw w, int comp, int cls)
    {
        return k.to_double(__uint_as_float(w), comp, cls);
    }
};
template <> struct QuadValue<CodecF16Dev> : QuadValueFloat {
    static __device__ __forceinline__ Raw load(const CodecF16Dev &, const uint2 *p, int c)
    {
        return __float_as_uint(__half2float(reinterpret_cast<const __half *>(p)[c]));
    }
    static __device__ __forceinline__ double value(const CodecF16Dev &k, Raw w, int comp, int cls)
    {
        return k.to_double(__uint_as_float(w), comp, cls);
    }
};
template <> struct QuadValue<CodecDF> {
    using Raw = uint2;      // hi, lo
    static constexpr int LIFT = 96, KEY_EXP = 23, BIAS = 127, MIN_EXP = 66, MAX_EXP = 127 + 90;
    static __device__ __forceinline__ Raw load(const CodecDF &k, const float4 *p, int c)
    {
        return make_uint2(reinterpret_cast<const unsigned *>(p)[c], reinterpret_cast<const unsigned *>(p + k.lo)[c]);
    }
    static __device__ __forceinline__ unsigned key(Raw w) { return max(w.x & 0x7fffffffu, w.y & 0x7fffffffu); }
    static __device__ __forceinline__ Raw lift(Raw w) { return make_uint2(fx_lift_float(w.x), fx_lift_float(w.y)); }
    static __device__ __forceinline__ long long align(Raw w, int e) { return fx_align_float(w.x, e) + fx_align_float(w.y, e); }
    static __device__ __forceinline__ double value(const CodecDF &k, Raw w, int comp, int cls)
    {
        return k.to_double(df(__uint_as_float(w.x), __uint_as_float(w.y)), comp, cls);
    }
};

// sum w_i and sum w_i |i|^2 in q58, the reference's part of n and E2 of a
// deviation codec (f aligned to exponent 126, i.e. to 1).
struct QuadRef {
    long long n, E;
};
inline QuadRef make_quad_ref(const HostConsts &k)
{
    const double na = k.d == 2 ? 4.0 : 6.0, nd = k.d == 2 ? 4.0 : 12.0, q58 = 288230376151711744.0;
    auto fix = [&](Dd v) { return (long long)(llrint(v.h * q58) + llrint(v.l * q58)); };
    const Dd a = Dd(na) * Dd(k.w[1]), d = Dd(nd) * Dd(k.w[2]);
    return QuadRef{fix(Dd(k.w[0]) + a + d), fix(a + Dd(2.0) * d)};
}

// The sums of one lane's component: integers in units of 2^unit where fine
// (J and E2 mean something in lane 0 only), doubles otherwise (the same in
// every lane of the warp).
struct QuadSums {
    bool fine;
    int unit;
    long long M, J[3], E;
    double dM, dJ[3], dE;
};

template <int D, class Codec, bool SWAPPED>
__device__ __forceinline__ QuadSums quad_sums(const Planes<typename Codec::S, Lattice<D>::Q> &pl, const Grid &g,
                                              const SiteIdx &si, const Codec &codec, const QuadRef &ref)
{
    using V = QuadValue<Codec>;
    constexpr int Q = Lattice<D>::Q;
    const int c = threadIdx.x & 3;
    QuadSums o;
    typename V::Raw w[Q];
    {
        const NbOff nb = nb_offsets(g, si);
#pragma unroll
        for (int q = 0; q < Q; ++q)     // population q
            w[q] = SWAPPED ? V::load(codec, pl.p[opposite<D>(q)] + nb_at(nb, si.s, -cx<D>(q), -cy<D>(q), -cz<D>(q)), c)
                           : V::load(codec, pl.p[q] + si.s, c);
    }
    unsigned mx = 0u;
#pragma unroll
    for (int q = 0; q < Q; ++q) mx = max(mx, V::key(w[q]));
    int em = (int)(mx >> V::KEY_EXP), lifted = 0;
    if (V::LIFT && mx && em < V::MIN_EXP && !(Codec::DEV && c == 0)) {
        lifted = V::LIFT;
        mx = 0u;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            w[q] = V::lift(w[q]);
            mx = max(mx, V::key(w[q]));
        }
        em = (int)(mx >> V::KEY_EXP);
    }
    int e = em;
    bool ok = em >= V::MIN_EXP && em <= V::MAX_EXP;
    if (Codec::DEV && c == 0) {
        e = V::BIAS - 1;
        ok = em <= e;
    }
    if (mx == 0u) {
        e = V::BIAS - 1;
        ok = true;
    }
    o.fine = __all_sync(0xffffffffu, ok);
    o.unit = e - V::BIAS - 57 - lifted;
    if (o.fine) {
        long long X[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) X[q] = V::align(w[q], e);
        fx_sums<D>(X, o.M, o.J, o.E);
        if (Codec::DEV && c == 0) {
            o.M += ref.n;
            o.E += ref.E;
        }
    } else {
        o.dM = o.dJ[0] = o.dJ[1] = o.dJ[2] = o.dE = 0.0;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const double v = V::value(codec, w[q], c, cnorm2<D>(q));
            o.dM += v;
            if (cx<D>(q)) o.dJ[0] += cx<D>(q) * v;
            if (cy<D>(q)) o.dJ[1] += cy<D>(q) * v;
            if (cz<D>(q)) o.dJ[2] += cz<D>(q) * v;
            if (cnorm2<D>(q)) o.dE += cnorm2<D>(q) * v;
        }
        if (lifted) {
            constexpr double down = V::LIFT ? 0x1p-96 : 1.0;
            o.dM *= down;
            o.dE *= down;
#pragma unroll
            for (int a = 0; a < 3; ++a) o.dJ[a] *= down;
        }
    }
    return o;
}

// v 2^unit as a double (one conversion).
__device__ __forceinline__ double quad_double(long long v, int unit)
{
    return fx_to_double(v, unit * (1 << 20));
}

// The sums as doubles, for warps that leave the integer form after all.
__device__ __forceinline__ void quad_to_double(QuadSums &s)
{
    s.fine = false;
    s.dM = quad_double(s.M, s.unit);
    s.dE = quad_double(s.E, s.unit);
#pragma unroll
    for (int a = 0; a < 3; ++a) s.dJ[a] = quad_double(s.J[a], s.unit);
}

// Site of a lane in chunk `chunk`; false for lanes beyond the row's end
// (they work on the row's last site).
__device__ __forceinline__ bool quad_site(const Grid &g, const Chunks &ch, int chunk, SiteIdx &si)
{
    const int row = fast_div(chunk, ch.row);
    const int x = (chunk - row * ch.per_row) * 8 + ((threadIdx.x & 31) >> 2);
    const bool active = x < g.nx;
    si.x = active ? x : g.nx - 1;
    si.z = fast_div(row, ch.y);
    si.y = row - si.z * g.ny;
    si.s = row * g.nx + si.x;
    return active;
}

constexpr int kQuadBlock = 128;

// Ratios of the warp's sites from lane 0's sums; false (for the whole warp)
// where a site leaves their range.
template <int D> __device__ __forceinline__ bool quad_ratios(const QuadSums &s, FixRatios &r)
{
    long long J[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) J[a] = a < D ? fx_from_lane0(s.J[a]) : 0;
    const bool ok = fx_ratios<D>(fx_from_lane0(s.M), J, fx_from_lane0(s.E), r);
    return __all_sync(0xffffffffu, ok);
}

// ---------------------------------------------------------------------------
// Single and half precision: one thread per site (76 values of 4 bytes fit
// its registers), so that the ratios and the conversions of the results are
// done once per site instead of by four lanes.  Moments of D3Q19 128^3 FP32:
// in double 916 us, four lanes 246, one thread 144 (376 bytes per site take
// 116); D2Q9 4096^2 FP16 3589 -> 658 us.
// ---------------------------------------------------------------------------
struct SiteSums {
    bool fine;          // integers hold (else the doubles)
    int unit[4];
    long long M[4], J[3], E;
    double dM[4], dJ[3], dE;
};

template <int D, class Codec, bool SWAPPED>
__device__ __forceinline__ void site_sums(const Planes<typename Codec::S, Lattice<D>::Q> &pl, const Grid &g,
                                          const SiteIdx &si, const Codec &codec, const QuadRef &ref, SiteSums &o)
{
    using V = QuadValueFloat;
    constexpr int Q = Lattice<D>::Q;
    float f[4][Q];
    gather<D, Codec, SWAPPED>(pl, g, si, codec, f[0], f[1], f[2], f[3]);
    o.fine = true;
    bool lifted[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        unsigned mx = 0u;
#pragma unroll
        for (int q = 0; q < Q; ++q) mx = max(mx, V::key(__float_as_uint(f[c][q])));
        int em = (int)(mx >> V::KEY_EXP);
        int e = V::BIAS - 1;
        lifted[c] = c && mx && em < V::MIN_EXP;
        if (c == 0) {
            o.fine = o.fine && em <= e;
        } else if (mx) {
            if (lifted[c]) {
                mx = 0u;
#pragma unroll
                for (int q = 0; q < Q; ++q) {
                    f[c][q] *= 0x1p96f;
                    mx = max(mx, V::key(__float_as_uint(f[c][q])));
                }
                em = (int)(mx >> V::KEY_EXP);
            }
            o.fine = o.fine && em >= V::MIN_EXP && em <= V::MAX_EXP;
            e = em;
        }
        o.unit[c] = e - V::BIAS - 57 - (lifted[c] ? V::LIFT : 0);
        if (c == 0) {
            long long X[Q];
#pragma unroll
            for (int q = 0; q < Q; ++q) X[q] = V::align(__float_as_uint(f[0][q]), e);
            fx_sums<D>(X, o.M[0], o.J, o.E);
            o.M[0] += ref.n;
            o.E += ref.E;
        } else {
            o.M[c] = 0;
#pragma unroll
            for (int q = 0; q < Q; ++q) o.M[c] += V::align(__float_as_uint(f[c][q]), e);
        }
    }
    if (!o.fine) {
        o.dE = o.dJ[0] = o.dJ[1] = o.dJ[2] = 0.0;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            o.dM[c] = 0.0;
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const double v = codec.to_double(f[c][q], c, cnorm2<D>(q));
                o.dM[c] += v;
                if (c) continue;
                if (cx<D>(q)) o.dJ[0] += cx<D>(q) * v;
                if (cy<D>(q)) o.dJ[1] += cy<D>(q) * v;
                if (cz<D>(q)) o.dJ[2] += cz<D>(q) * v;
                if (cnorm2<D>(q)) o.dE += cnorm2<D>(q) * v;
            }
            if (lifted[c]) o.dM[c] *= 0x1p-96;
        }
    }
}
__device__ __forceinline__ void site_to_double(SiteSums &s)
{
    if (!s.fine) return;
    s.fine = false;
#pragma unroll
    for (int c = 0; c < 4; ++c) s.dM[c] = quad_double(s.M[c], s.unit[c]);
#pragma unroll
    for (int a = 0; a < 3; ++a) s.dJ[a] = quad_double(s.J[a], s.unit[0]);
    s.dE = quad_double(s.E, s.unit[0]);
}

// xi 2^-62 and xi^2/2 2^-62 (moments from q62 ratios), xi and xi^2/2.
struct MomentScale {
    double u62, e62, u, e;
};

// n and S (s.dM), u and eps of a site from its sums.
template <int D>
__device__ __forceinline__ void site_finish(SiteSums &s, const MomentScale &sc, double (&uu)[3], double &eps)
{
    FixRatios r;
    if (s.fine && fx_ratios<D>(s.M[0], s.J, s.E, r)) {
#pragma unroll
        for (int c = 0; c < 4; ++c) s.dM[c] = quad_double(s.M[c], s.unit[c]);
#pragma unroll
        for (int a = 0; a < D; ++a) uu[a] = (double)((((long long)r.j[a].hi << 32) + r.j[a].lo) >> 2) * sc.u62;
        eps = (double)(r.ej << 2) * sc.e62;
        return;
    }
    site_to_double(s);
    const double rn = 1.0 / s.dM[0];
    const double jx = s.dJ[0] * rn, jy = s.dJ[1] * rn, jz = D == 3 ? s.dJ[2] * rn : 0.0;
    uu[0] = sc.u * jx;
    uu[1] = sc.u * jy;
    uu[2] = sc.u * jz;
    eps = sc.e * (s.dE * rn - (jx * jx + jy * jy + jz * jz));
}

template <int D, class Codec, bool SWAPPED>
__global__ void __launch_bounds__(kStepBlock, 4)
k_moments_site(const Planes<typename Codec::S, Lattice<D>::Q> pl, Grid g, Codec codec, QuadRef ref, MomentScale sc,
               double *__restrict__ rho4, double *__restrict__ u, double *__restrict__ eps)
{
    SiteIdx si;
    if (!site_of_block(g, si)) return;
    SiteSums s;
    site_sums<D, Codec, SWAPPED>(pl, g, si, codec, ref, s);
    double uu[3], ee;
    site_finish<D>(s, sc, uu, ee);
    const int64_t N = g.N, i = si.s;
    if (rho4)
#pragma unroll
        for (int c = 0; c < 4; ++c) rho4[c * N + i] = s.dM[c];
    if (u)
#pragma unroll
        for (int a = 0; a < D; ++a) u[a * N + i] = uu[a];
    if (eps) eps[i] = ee;
}

// ---------------------------------------------------------------------------
// Moments of Eq. DiscrAvr (one warp per chunk).  D3Q19 128^3 FP64: 555 -> 277
// us (680 bytes per site take 210).
// ---------------------------------------------------------------------------
template <int D, class Codec, bool SWAPPED>
__global__ void __launch_bounds__(kQuadBlock)
k_moments(const Planes<typename Codec::S, Lattice<D>::Q> pl, Grid g, Codec codec, Chunks ch, QuadRef ref, MomentScale sc,
          double *__restrict__ rho4, double *__restrict__ u, double *__restrict__ eps)
{
    const int chunk = chunk_of_thread(blockIdx.x, threadIdx.x, kQuadBlock), c = threadIdx.x & 3;
    if (chunk >= ch.total) return;      // the whole warp
    SiteIdx si;
    const bool active = quad_site(g, ch, chunk, si);
    QuadSums s = quad_sums<D, Codec, SWAPPED>(pl, g, si, codec, ref);
    // lane 0: n and eps; lane a + 1: spin component a and velocity component a
    double M, v;
    FixRatios r;
    if (s.fine && !quad_ratios<D>(s, r)) quad_to_double(s);
    if (s.fine) {
        M = quad_double(s.M, s.unit);
        long long t = r.ej << 2;        // q62
#pragma unroll
        for (int a = 0; a < D; ++a)
            if (c == a + 1) t = (((long long)r.j[a].hi << 32) + r.j[a].lo) >> 2;
        v = (double)t * (c == 0 ? sc.e62 : sc.u62);
    } else {
        const unsigned all = 0xffffffffu;
        const double rn = 1.0 / __shfl_sync(all, s.dM, 0, 4);
        const double jx = __shfl_sync(all, s.dJ[0], 0, 4) * rn, jy = __shfl_sync(all, s.dJ[1], 0, 4) * rn;
        const double jz = D == 3 ? __shfl_sync(all, s.dJ[2], 0, 4) * rn : 0.0;
        const double e2n = __shfl_sync(all, s.dE, 0, 4) * rn;
        M = s.dM;
        v = c == 0 ? sc.e * (e2n - (jx * jx + jy * jy + jz * jz)) : sc.u * (c == 1 ? jx : (c == 2 ? jy : jz));
    }
    if (!active) return;
    const int64_t N = g.N;
    if (rho4) rho4[c * N + si.s] = M;
    if (c == 0) {
        if (eps) eps[si.s] = v;
    } else if (u && c <= D) {
        u[(c - 1) * N + si.s] = v;
    }
}

// ---------------------------------------------------------------------------
// Negative-definite equilibria (Sec. 3.2 end, Sec. 3.3 end): W_i^eq =
// w_i rho P_i (Eq. WeqAlgo) can have a negative eigenvalue, and the scheme
// neither clips it nor adapts tau.  This read-only diagnostic forms, from
// the current state, the moments and every P_i that the next collision uses
// and flags direction i when W_i^eq has a negative eigenvalue.  The
// eigenvalues of w_i P_i rho are w_i P_i (n +- |S|)/2 (w_i > 0), so the
// smallest is negative exactly when P_i n < |P_i| |S|: for n > 0, when P_i < 0,
// or when P_i > 0 and n < |S|.  The signs of the P_i come from the fixed-point
// coefficients (2^-58 absolute), n and |S| are compared in double.  mask[s]
// (if not NULL) receives bit i for each flagged direction; *count
// accumulates the number of flagged (site, direction) pairs (one atomic per
// warp).  D3Q19 90 x 101 x 75 FP64: 429 -> 133 us.
// ---------------------------------------------------------------------------
template <int D, class Codec, bool SWAPPED>
__global__ void __launch_bounds__(kQuadBlock)
k_negative_eq(const Planes<typename Codec::S, Lattice<D>::Q> pl, Grid g, Codec codec, Chunks ch, QuadRef ref,
              FixConst fc, InitConsts ic, unsigned long long *__restrict__ count, unsigned *__restrict__ mask)
{
    constexpr int Q = Lattice<D>::Q;
    const unsigned all = 0xffffffffu;
    const int chunk = chunk_of_thread(blockIdx.x, threadIdx.x, kQuadBlock), c = threadIdx.x & 3;
    if (chunk >= ch.total) return;      // the whole warp
    SiteIdx si;
    const bool active = quad_site(g, ch, chunk, si);
    QuadSums s = quad_sums<D, Codec, SWAPPED>(pl, g, si, codec, ref);
    FixRatios r;
    FixCoef cf;
    if (s.fine) {
        bool ok = quad_ratios<D>(s, r);
        if (ok) ok = __all_sync(all, fx_basis<D>(r.j, r.jj, r.ej - fc.d0, fc, cf));
        if (!ok) quad_to_double(s);
    }
    unsigned m = 0u;
    if (s.fine) {
        const double M = quad_double(s.M, s.unit);
        double sq = c == 0 ? 0.0 : M * M;
        sq += __shfl_xor_sync(all, sq, 1, 4);
        sq += __shfl_xor_sync(all, sq, 2, 4);
        // of lane 0: n < |S|, by the root where the squares are close (pure
        // states: it halves the squares' rounding, and a zero eigenvalue does
        // not count; ~20 double-precision instructions elsewhere too if taken
        // always)
        const double MM = M * M;
        bool polar = MM < sq;
        if (c == 0 && abs(__double2hiint(MM) - __double2hiint(sq)) <= 1) polar = M < sqrt(sq);
        fx_each_h<D>(cf, [&](int q, long long h) {
            if (h < 0 || (polar && h > 0)) m |= 1u << q;
        });
    } else {
        const double n = __shfl_sync(all, s.dM, 0, 4), rn = 1.0 / n;
        const double jx = __shfl_sync(all, s.dJ[0], 0, 4) * rn, jy = __shfl_sync(all, s.dJ[1], 0, 4) * rn;
        const double jz = D == 3 ? __shfl_sync(all, s.dJ[2], 0, 4) * rn : 0.0;
        const double be = ic.K * (__shfl_sync(all, s.dE, 0, 4) * rn - (jx * jx + jy * jy + jz * jz));
        double sq = c == 0 ? 0.0 : s.dM * s.dM;
        sq += __shfl_xor_sync(all, sq, 1, 4);
        sq += __shfl_xor_sync(all, sq, 2, 4);
        const double normS = sqrt(sq);
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const double P = poly_P_d<D>(ic, q, jx, jy, jz, be);
            if (P * n < fabs(P) * normS) m |= 1u << q;
        }
    }
    if (c || !active) m = 0u;
    else if (mask) mask[si.s] = m;
    const unsigned k = __reduce_add_sync(all, (unsigned)__popc(m));
    if ((threadIdx.x & 31) == 0 && k) atomicAdd(count, (unsigned long long)k);
}

// ---------------------------------------------------------------------------
// Global sums of Eqs. GlobalDensity, GlobalVelocity, GlobalTotalEnergy:
// per-block partials, then one block over the partials.  A site's sums are
// exact integers; each lane adds two of them per site in double (its
// component's, and E2 or a component of J), two conversions and two
// additions per lane.  The launch shape is fixed per handle, so the result
// is deterministic.  D3Q19 128^3 FP64: 630 -> 218 us
// (608 bytes per site take 188).
// ---------------------------------------------------------------------------
template <int D, class Codec, bool SWAPPED>
__global__ void __launch_bounds__(kRedBlock)
k_conserved_partial(const Planes<typename Codec::S, Lattice<D>::Q> pl, Grid g, Codec codec, Chunks ch, QuadRef ref,
                    double *__restrict__ partials)
{
    const unsigned all = 0xffffffffu;
    const int c = threadIdx.x & 3;
    const unsigned nw = gridDim.x * (kRedBlock / 32);
    double acc[2] = {0.0, 0.0};
    wait_for_previous();
    // (unsigned: the step beyond the last chunk can pass 2^31)
    for (unsigned k = (unsigned)chunk_of_thread(blockIdx.x, threadIdx.x, kRedBlock); k < (unsigned)ch.total; k += nw) {
        SiteIdx si;
        const bool active = quad_site(g, ch, (int)k, si);
        const QuadSums s = quad_sums<D, Codec, SWAPPED>(pl, g, si, codec, ref);
        double M, v;
        if (s.fine) {
            const int unit = __shfl_sync(all, s.unit, 0, 4);
            long long t = fx_from_lane0(s.E);
#pragma unroll
            for (int a = 0; a < D; ++a) {
                const long long J = fx_from_lane0(s.J[a]);
                if (c == a + 1) t = J;
            }
            M = quad_double(s.M, s.unit);
            v = quad_double(t, unit);
        } else {
            M = s.dM;
            v = __shfl_sync(all, s.dE, 0, 4);
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const double J = __shfl_sync(all, s.dJ[a], 0, 4);
                if (c == a + 1) v = J;
            }
        }
        if (active) {
            acc[0] += M;
            acc[1] += v;
        }
    }
    let_next_start();
    if (D == 2 && c == 3) acc[1] = 0.0;
    // over the warp's eight sites, then over the block's warps
    __shared__ double sh[kRedBlock / 32][8];
#pragma unroll
    for (int i = 0; i < 2; ++i)
        for (int o = 4; o < 32; o <<= 1) acc[i] += __shfl_xor_sync(all, acc[i], o);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane < 4) {
        sh[warp][c] = acc[0];
        sh[warp][c == 0 ? 7 : 3 + c] = acc[1];
    }
    __syncthreads();
    if (threadIdx.x < 8) {
        double t = 0.0;
        for (int w = 0; w < kRedBlock / 32; ++w) t += sh[w][threadIdx.x];
        partials[(int64_t)blockIdx.x * 8 + threadIdx.x] = t;
    }
}

}  // namespace qlbm
