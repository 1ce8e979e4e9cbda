// Pair terms of the pair sums, two pairs per instruction (cluster.cu, tile.cu).
//
// The pair sums are bound by instruction issue: each pair costs some fifty
// FP32 operations, three MUFU results and a few tests, and nothing comes
// from memory but one atom per several pairs.  Blackwell issues an FP32
// operation on two operand pairs as one instruction (FFMA2, FADD2, FMUL2), so
// a lane takes two pairs at a time: the displacement, r^2, the Newton step,
// the Ewald, LJ and switching polynomials are packed; the MUFU results, the
// cutoff tests and the selects are per pair.  The MUFU inputs are normal
// numbers for every pair that counts, so the flushing forms are taken (the
// others add range tests).
//
// Every pair keeps the roundings of pairsum_w (common.cuh), operation by
// operation, and the kernels keep the order of every FP32 sum, so that a
// trajectory repeats bit for bit what one pair per instruction gives: pairs
// that cross a truncated cutoff, and thinning decisions near a tie, would
// turn any other rounding into visible differences within a few steps.
#pragma once
#include "common.cuh"

constexpr float MAGIC = 12582912.f;  // 1.5 2^23: adding and subtracting it rounds to the nearest integer
constexpr float PAIR_FAR = 1e15f;    // coordinate of an atom placed out of reach

// Scalars of the packed pair terms (each twice where an operand of a
// two-pair instruction), filled on the host.
struct PairConsts {
    float2 beta, c2b;               // Ewald beta, 2 beta / sqrt(pi)
    float2 mron;                    // -r' of the switching function
    float2 invL[3], mLhi[3], mLlo[3];
    float rc2, band;                // centre of the rounding band of r_c^2 and its half width (with a margin)
    float inv_span, r_off, rc2_lo;
    int chi_step;
};

inline PairConsts make_pair_consts(const Params& p) {
    auto d = [](float x) { return make_float2(x, x); };
    PairConsts k;
    k.beta = d(p.ebeta);
    k.c2b = d(p.e2b_sqrtpi);
    k.mron = d(-p.r_on);
    const bool cut = p.rc2_lo < INFINITY;
    k.rc2 = cut ? 0.5f * p.rc2_lo + 0.5f * p.rc2_hi : 0.f;
    k.band = cut ? 0.51f * (p.rc2_hi - p.rc2_lo) : -1.f;
    for (int c = 0; c < 3; ++c) {
        k.invL[c] = d(p.periodic ? p.invL[c] : 0.f);  // (open boundaries: no image)
        k.mLhi[c] = d(-p.Lhi[c]);
        k.mLlo[c] = d(-p.Llo[c]);
    }
    k.inv_span = p.inv_span;
    k.r_off = p.r_off;
    // without a cutoff every pair counts but those with an atom out of reach
    k.rc2_lo = cut ? p.rc2_lo : 0.01f * PAIR_FAR * PAIR_FAR;
    k.chi_step = p.chi_step;
    return k;
}

__device__ __forceinline__ float2 two(float x) { return make_float2(x, x); }
// a + b rounded by itself: a packed product and a packed sum are contracted
// into one fused operation, the explicitly rounded scalar sum is not.
__device__ __forceinline__ float2 add2_apart(float2 a, float2 b) {
    return make_float2(__fadd_rn(a.x, b.x), __fadd_rn(a.y, b.y));
}
__device__ __forceinline__ float rsqrt_ftz(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float ex2_ftz(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rcp_ftz(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// pairsum_w of two pairs at squared distances r2 (any value: a pair that does
// not count is masked by the caller).  nqq: -k q_i q_j; l12, ml6: 12 c12 and
// -6 c6 of the pairs.  EW: Ewald direct, else bare Coulomb; CJ: Coulomb is
// switched too.
template <int PART, bool EW, bool CJ>
__device__ __forceinline__ float2 pair_w2(const PairConsts& k, float2 r2, float2 nqq, float2 l12, float2 ml6) {
    const float2 y = make_float2(rsqrt_ftz(r2.x), rsqrt_ftz(r2.y));
    const float2 ir = __fmul2_rn(y, __ffma2_rn(__fmul2_rn(__fmul2_rn(r2, two(-0.5f)), y), y, two(1.5f)));
    const float2 ir2 = __fmul2_rn(ir, ir);
    const float2 r = __fmul2_rn(r2, ir);
    float2 wc;
    if (EW) {
        const float2 x = __fmul2_rn(k.beta, r);
        const float2 ea = __fmul2_rn(__fmul2_rn(x, x), two(-1.4426950408889634f));
        const float2 e = make_float2(ex2_ftz(ea.x), ex2_ftz(ea.y));
        const float2 ta = __ffma2_rn(x, two(0.3275911f), two(1.f));
        const float2 t = make_float2(rcp_ftz(ta.x), rcp_ftz(ta.y));
        float2 s = __ffma2_rn(t, two(1.061405429f), two(-1.453152027f));
        s = __ffma2_rn(t, s, two(1.421413741f));
        s = __ffma2_rn(t, s, two(-0.284496736f));
        s = __ffma2_rn(t, s, two(0.254829592f));
        const float2 u = __ffma2_rn(__fmul2_rn(k.c2b, e), ir, __fmul2_rn(__fmul2_rn(__fmul2_rn(t, s), e), ir2));
        wc = __fmul2_rn(__fmul2_rn(nqq, u), ir);
    } else {
        wc = __fmul2_rn(__fmul2_rn(nqq, ir2), ir);
    }
    const float2 ir6 = __fmul2_rn(__fmul2_rn(ir2, ir2), ir2);
    const float2 nwl = __fmul2_rn(__fmul2_rn(__ffma2_rn(l12, ir6, ml6), ir6), ir2);
    const float2 wl = make_float2(-nwl.x, -nwl.y);
    if (PART == 5) return add2_apart(wc, wl);
    float2 mc;  // 1 - chi
    if (k.chi_step) {
        mc = make_float2(r.x >= k.r_off ? 0.f : 1.f, r.y >= k.r_off ? 0.f : 1.f);
    } else {
        const float2 x = __fadd2_rn(r, k.mron);
        const float2 s = make_float2(__saturatef(x.x * k.inv_span), __saturatef(x.y * k.inv_span));
        const float2 q = __ffma2_rn(s, __ffma2_rn(s, two(6.f), two(-15.f)), two(10.f));
        const float2 chi = __fmul2_rn(__fmul2_rn(__fmul2_rn(s, s), s), q);
        mc = add2_apart(two(1.f), make_float2(-chi.x, -chi.y));
    }
    return CJ ? __fmul2_rn(add2_apart(wc, wl), mc) : add2_apart(__fmul2_rn(wl, mc), wc);
}

__device__ __forceinline__ float2 norm2(float2 dx, float2 dy, float2 dz) {
    return __ffma2_rn(dz, dz, __ffma2_rn(dx, dx, __fmul2_rn(dy, dy)));
}

// Minimum image of two displacements d + e (high and low parts' differences),
// as pair_disp.
__device__ __forceinline__ void image2(const PairConsts& k, int c, float2& d, float2& e) {
    const float2 n = __fadd2_rn(add2_apart(__fmul2_rn(d, k.invL[c]), two(MAGIC)), two(-MAGIC));
    d = __ffma2_rn(n, k.mLhi[c], d);
    e = __ffma2_rn(n, k.mLlo[c], e);
}

// The eight i atoms of a warp's group in shared memory, two per record.
struct __align__(16) IPair {
    float2 hx, hy, hz, lx, ly, lz;  // split positions
    float2 kq;                      // k q
    int2 mol;                       // molecules
};
struct __align__(16) IGroup {
    IPair a[4];
    float4 lj[4][BOUNCE_MAXT];      // 12 c12 (x, y) and -6 c6 (z, w) of both atoms with each type of j
};

// Record of i atom a of the group (hi.w = charge, lo.w = type); an atom that
// does not exist (molecule < 0) is placed out of reach.  Lanes of one warp,
// followed by __syncwarp.
__device__ __forceinline__ void igroup_set(IGroup& g, const Params& p, int a, float4 hi, float4 lo, int mol) {
    IPair& r = g.a[a >> 1];
    const int h = a & 1;
    if (mol < 0) {
        hi = make_float4(PAIR_FAR, PAIR_FAR, PAIR_FAR, 0.f);
        lo = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    (&r.hx.x)[h] = hi.x;
    (&r.hy.x)[h] = hi.y;
    (&r.hz.x)[h] = hi.z;
    (&r.lx.x)[h] = lo.x;
    (&r.ly.x)[h] = lo.y;
    (&r.lz.x)[h] = lo.z;
    (&r.kq.x)[h] = p.kcoul * hi.w;
    (&r.mol.x)[h] = mol;
    const int t = type_of(lo) * BOUNCE_MAXT;
#pragma unroll
    for (int b = 0; b < BOUNCE_MAXT; ++b) {
        (&g.lj[a >> 1][b].x)[h] = 12.f * p.c12[t + b];
        (&g.lj[a >> 1][b].z)[h] = -6.f * p.c6[t + b];
    }
}

// A j atom of a lane: split position (h.w = charge), molecule, type, and the
// index rule (pairs with the group's atoms a < above).
struct JAtom {
    float4 h, l;
    int mol, type, above;
};

// The pairs of a lane's j atom with the group's eight atoms: w d added to gi
// (two atoms per entry) and to gj (the eight atoms in turn), the pairs that
// count added to npair.  A pair counts when the molecules differ and r^2 <
// rc2_lo (an atom out of reach never does); GEN: also a < j.above, and with
// the minimum image per pair.  near receives the smallest |r^2 - r_c^2|, for
// the exact test of pairs in the rounding band of the cutoff.
template <int PART, bool EW, bool CJ, bool GEN>
__device__ __forceinline__ void group_pairs(const PairConsts& k, const IGroup& g, const JAtom& j, float2 (&gi)[4][3],
                                            float3& gj, float& near, int& npair) {
    const float2 nhx = two(-j.h.x), nhy = two(-j.h.y), nhz = two(-j.h.z);
    const float2 nlx = two(-j.l.x), nly = two(-j.l.y), nlz = two(-j.l.z);
    const float2 nq = two(-j.h.w);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const IPair& a = g.a[c];
        float2 dx = __fadd2_rn(a.hx, nhx), dy = __fadd2_rn(a.hy, nhy), dz = __fadd2_rn(a.hz, nhz);
        float2 ex = __fadd2_rn(a.lx, nlx), ey = __fadd2_rn(a.ly, nly), ez = __fadd2_rn(a.lz, nlz);
        if (GEN) {
            image2(k, 0, dx, ex);
            image2(k, 1, dy, ey);
            image2(k, 2, dz, ez);
        }
        dx = __fadd2_rn(dx, ex);
        dy = __fadd2_rn(dy, ey);
        dz = __fadd2_rn(dz, ez);
        const float2 r2 = norm2(dx, dy, dz);
        bool in0 = a.mol.x != j.mol && r2.x < k.rc2_lo, in1 = a.mol.y != j.mol && r2.y < k.rc2_lo;
        if (GEN) {
            in0 = in0 && j.above > 2 * c && a.mol.x >= 0;
            in1 = in1 && j.above > 2 * c + 1 && a.mol.y >= 0;
        }
        near = fminf(near, fminf(fabsf(r2.x - k.rc2), fabsf(r2.y - k.rc2)));
        const float4 t = g.lj[c][j.type];
        float2 w = pair_w2<PART, EW, CJ>(k, r2, __fmul2_rn(a.kq, nq), make_float2(t.x, t.y), make_float2(t.z, t.w));
        w.x = in0 ? w.x : 0.f;
        w.y = in1 ? w.y : 0.f;
        npair += (in0 ? 1 : 0) + (in1 ? 1 : 0);
        gi[c][0] = __ffma2_rn(w, dx, gi[c][0]);
        gi[c][1] = __ffma2_rn(w, dy, gi[c][1]);
        gi[c][2] = __ffma2_rn(w, dz, gi[c][2]);
        gj.x = fmaf(-w.y, dx.y, fmaf(-w.x, dx.x, gj.x));
        gj.y = fmaf(-w.y, dy.y, fmaf(-w.x, dy.x, gj.y));
        gj.z = fmaf(-w.y, dz.y, fmaf(-w.x, dz.x, gj.z));
    }
}

// Warp sums of the eight atoms' i sides: on return lane 4 b + d (d < 3) holds
// component d of atom igroup_atom(b).  Halves of the atoms are exchanged over
// three butterfly stages (12 + 6 + 3 shuffles) and the three components left
// are summed over the four lanes of an atom (6), 27 shuffles where 24 full
// warp sums take 120; the tree of each sum is that of the full butterfly.
__device__ __forceinline__ int igroup_atom(int b) { return ((b & 4) >> 2) | (b & 2) | ((b & 1) << 2); }
__device__ __forceinline__ float igroup_reduce(const float2 (&gi)[4][3]) {
    const int lane = threadIdx.x & 31;
    const uint32_t F = 0xffffffffu;
    float v[4][3];  // bit 4 of the lane picks the odd or even atom
    {
        const bool up = lane & 16;
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const float keep = up ? gi[c][d].y : gi[c][d].x, give = up ? gi[c][d].x : gi[c][d].y;
                v[c][d] = keep + __shfl_xor_sync(F, give, 16);
            }
    }
    float u[2][3];  // bit 3 picks the even or odd pair
    {
        const bool up = lane & 8;
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const float keep = up ? v[2 * c + 1][d] : v[2 * c][d], give = up ? v[2 * c][d] : v[2 * c + 1][d];
                u[c][d] = keep + __shfl_xor_sync(F, give, 8);
            }
    }
    float w[3];  // bit 2 picks the lower or upper pairs
    {
        const bool up = lane & 4;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const float keep = up ? u[1][d] : u[0][d], give = up ? u[0][d] : u[1][d];
            w[d] = keep + __shfl_xor_sync(F, give, 4);
        }
    }
#pragma unroll
    for (int o = 2; o > 0; o >>= 1)
#pragma unroll
        for (int d = 0; d < 3; ++d) w[d] += __shfl_xor_sync(F, w[d], o);
    const int d = lane & 3;
    return d == 0 ? w[0] : (d == 1 ? w[1] : w[2]);
}
