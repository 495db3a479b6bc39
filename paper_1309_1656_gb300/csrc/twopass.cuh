// Two-pass AA step for the double-float codec.  Holding all 4b double-float
// values of a site takes the whole register file of a thread (255 registers,
// 8 warps per SM), and with so few warps the loads and the long arithmetic
// do not overlap.  This kernel streams the populations through the moment
// sums (pass 1), keeping their hi parts (4b floats) in registers and their
// lo parts in shared memory (4b x 4 B per thread: 38.9 KB per D3Q19 block),
// forms the coefficients, then takes the lo parts of each direction
// together with its opposite back from shared memory (pass 2), updates the
// pair and stores it.  Every value is read from HBM once.  In the AA pattern the read locations of a direction
// and of its opposite are exactly the pair's two write locations (even step:
// slots q and opposite(q) at x; odd step: slot opposite(q) at x - e_q and
// slot q at x + e_q), so updating pair by pair in place is race-free within
// the thread, and across threads as in the one-pass kernel.
#pragma once

#include "dfloat.cuh"
#include "kernels.cuh"

namespace qlbm {

template <class Codec> struct TwoPass {
    static constexpr bool value = false;
};
template <> struct TwoPass<CodecDF> {
    static constexpr bool value = true;
    // Blocks of 128 per SM: D3Q19 keeps 76 hi floats per thread (128
    // registers), D2Q9 36 (96).  Re-reading whole values in pass 2 instead
    // missed in L2 for ~40 % of the re-read bytes (D3Q19).
    template <int D> static constexpr int min_blocks() { return D == 2 ? 5 : 4; }
};

// A population's update with the magnetic-field term: the rotation r of
// (1 - omega) s + h omega S taken as (1 - omega) r s + h (r omega S), m =
// (1 - omega) r and the rotated omega S (in c) formed once per site, one
// four-term product sum per component.  Updated first and rotated then, it
// takes 22 + 43 single-precision operations per component, this 46 (D2Q9
// 1501 x 777, uniform field: 146 -> 132 us per step).
__device__ __forceinline__ void df_update_rotated(const DFCoef &c, df h, const df (&m)[9], df &f, df &x, df &y, df &z)
{
    f = dfma(h, c.on, c.omc * f);
    const df a = x, b = y, d = z;
    x = dot4(m[0], a, m[1], b, m[2], d, h, c.oSx);
    y = dot4(m[3], a, m[4], b, m[5], d, h, c.oSy);
    z = dot4(m[6], a, m[7], b, m[8], d, h, c.oSz);
}

// Location of population p of site si: slot and site index.
template <int D, bool SWAPPED>
__device__ __forceinline__ int read_slot(int p) { return SWAPPED ? opposite<D>(p) : p; }

template <int D, bool SWAPPED>
__device__ __forceinline__ int read_site(const Grid &g, const SiteIdx &si, int p)
{
    // swapped buffer: population p sits in slot opposite(p) at x - e_p
    return SWAPPED ? neighbour(g, si, -cx<D>(p), -cy<D>(p), -cz<D>(p)) : si.s;
}

template <int D, bool ODD, int FIELD>
__global__ void __launch_bounds__(kStepBlock, TwoPass<CodecDF>::min_blocks<D>())
k_step_aa_df2(const Planes<df, Lattice<D>::Q> pl, Grid g, Coll<df> k, CodecDF codec, unsigned *__restrict__ flags)
{
    constexpr int Q = Lattice<D>::Q;
    // lo parts, kept from pass 1 in shared memory (a thread reads back only
    // what it wrote: no barrier)
    __shared__ float4 lo_stage[Q][kStepBlock];
    SiteIdx si;
    wait_for_previous();
    if (!site_of_block(g, si)) return;
    float hf[Q], hx[Q], hy[Q], hz[Q];   // hi parts, kept from pass 1 in registers
    DFSums a;
    a.zero();
#pragma unroll
    for (int p = 0; p < Q; ++p) {
        const float4 *v = pl.p[read_slot<D, ODD>(p)] + read_site<D, ODD>(g, si, p);
        const float4 h = v[0], l = v[codec.lo];
        hf[p] = h.x;
        hx[p] = h.y;
        hy[p] = h.z;
        hz[p] = h.w;
        lo_stage[p][threadIdx.x] = l;
        df_accumulate<D>(a, p, df(h.x, l.x), df(h.y, l.y), df(h.z, l.z), df(h.w, l.w));
    }
    DFCoef c = df_coefficients<D>(a, k);
    // the field's rotation: the uniform one, or the site's own, formed in
    // double from its unit quaternion and rounded to double-float pairs
    df rm[9];
    if constexpr (FIELD != FIELD_NONE) {
        if constexpr (FIELD == FIELD_SITE) {
            double w, x, y, z, r[9];
            load_quat(k.qf + si.s, w, x, y, z);
            quat_rotation(w, x, y, z, r);
#pragma unroll
            for (int i = 0; i < 9; ++i) rm[i] = df(r[i]);
        } else {
#pragma unroll
            for (int i = 0; i < 9; ++i) rm[i] = k.rot[i];
        }
        const df Sx = c.oSx, Sy = c.oSy, Sz = c.oSz;
        c.oSx = rm[0] * Sx + rm[1] * Sy + rm[2] * Sz;
        c.oSy = rm[3] * Sx + rm[4] * Sy + rm[5] * Sz;
        c.oSz = rm[6] * Sx + rm[7] * Sy + rm[8] * Sz;
#pragma unroll
        for (int i = 0; i < 9; ++i) rm[i] = c.omc * rm[i];
    }
    // g.zero (0 at run time) makes pass 2's addresses distinct expressions,
    // so the compiler re-loads the lo parts instead of keeping pass 1's.
    SiteIdx s2 = si;
    s2.s += g.zero;
    s2.x += g.zero;
    let_next_start();
#pragma unroll
    for (int q = 0; q <= (Q - 1) / 2; ++q) {
        const int qb = Q - 1 - q;
        // (index through g.zero: the compiler re-reads shared memory instead
        // of keeping pass 1's lo values in registers)
        const float4 l = lo_stage[q][threadIdx.x + g.zero];
        df f(hf[q], l.x), x(hx[q], l.y), y(hy[q], l.z), z(hz[q], l.w);
        df fb, xb, yb, zb;
        if (qb != q) {
            const float4 lb = lo_stage[qb][threadIdx.x + g.zero];
            fb = df(hf[qb], lb.x);
            xb = df(hx[qb], lb.y);
            yb = df(hy[qb], lb.z);
            zb = df(hz[qb], lb.w);
        }
        df hp, hm;
        df_pair_h<D>(c, k, q, hp, hm);
        if constexpr (FIELD == FIELD_NONE) {
            df_update(c, hp, f, x, y, z);
            if (qb != q) df_update(c, hm, fb, xb, yb, zb);
        } else {
            df_update_rotated(c, hp, rm, f, x, y, z);
            if (qb != q) df_update_rotated(c, hm, rm, fb, xb, yb, zb);
        }
        // population p goes to slot opposite(p) at x (even) or slot p at x + e_p (odd)
        codec.store4(pl.p[ODD ? q : qb] + (ODD ? neighbour(g, s2, cx<D>(q), cy<D>(q), cz<D>(q)) : s2.s), f, x, y,
                     z);
        if (qb != q)
            codec.store4(pl.p[ODD ? qb : q] + (ODD ? neighbour(g, s2, cx<D>(qb), cy<D>(qb), cz<D>(qb)) : s2.s), fb,
                         xb, yb, zb);
    }
    if (c.flag) atomicOr(flags, c.flag);
}

}  // namespace qlbm
