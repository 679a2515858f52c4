// Hopping term on FP64 fields in block fixed-point integer arithmetic.
//
// GB300 issues FP64 at 2 lanes per clock and SM (measured 0.63 T FMA/s against
// 37 T FP32 FMA/s); 64-bit integer multiply-adds (IMAD.WIDE, 32 x 32 + 64)
// run at 64.  One site's FP64 hopping term is ~900 FP64 operations and was
// bound by that pipe: 1673 us at 32^3 x 64, 558 us at 24^3 x 48, 131 us at
// 16^3 x 32, 55 us at 4^4.  Here the SU(3) products and the sum over the eight
// hops run on the integer pipes; FP64 keeps the spin projection (12 additions
// per hop) and the epilogue: 580, 193, 46 and 8 us (516, 172, 41 and 8 without the
// check of the components, see below).  What bounds it now: dependent issue and the
// loads at the 20 warps per SM that 96 registers allow (issue 46 % active, FP64
// pipe 45 % busy, DRAM 25 to 28 % on 16^3 x 32).
//
// Numbers.  A link element is u = Fu 2^(eu - 62) with a 62-bit integer Fu and
// one exponent eu per link: |u| <= 2^eu, and the absolute values of the six
// reals of any row or column add to at most 2.46 2^eu (eu = 0 for every SU(3)
// link, whose rows add to at most sqrt(6)).  It is stored as two signed limbs, Fu =
// u1 2^32 + u0, |u1| <= 2^30, |u0| <= 2^31, converted once when the gauge field
// is loaded.  The projected half-spinor row of a hop (6 reals, FP64) is
// converted to 60-bit integers Fh = h1 2^32 + h0, |h1| <= 2^28, with one shared
// exponent.  Then
//   sum Fu Fh = 2^64 (sum u1 h1 + 2^-32 sum (u1 h0 + u0 h1)) + ...
// with two 64-bit accumulators per real sum; the omitted u0 h0 terms are below
// a quarter of the last place each.  |sum (u1 h0 + u0 h1)| <= 2.46 2^61 + 6 2^59
// < 2^63, |sum u1 h1| <= 2.46 2^58, and the sum over the eight hops (exponent XA
// of the site's accumulators, raised when a larger hop arrives) stays below
// 2^63.  The last place of a hop is 2^-58 of twice its largest component: the
// result is one rounding of a value good to about 2^-57 of the site's scale,
// where FP64 arithmetic rounds after every operation.  Against 113-bit
// arithmetic (relative 2-norm, 6 x 10 x 14 x 18): Gaussian fields 7.0e-17 (FP64
// arithmetic 1.5e-16), fields falling by e^3 per time slice 7.8e-17 (1.4e-16); a
// point source after two applications of D (10 x 10 x 6 x 18, mean of 16) 7.2e-17
// (8.2e-17).
//
// Hops whose half spinor is zero contribute nothing.  Infinities, NaN,
// half spinors below 2^-523 or from 2^477 in magnitude, and links outside
// 2^-60 .. 2^60 leave the site to FP64 arithmetic (fx_site_f64, fx_number_f64).
//
// Components.  One last place serves all numbers that share an exponent, so a
// component far below the others would keep fewer bits than in FP64 arithmetic,
// whose errors are relative to the component's own terms.  Every real sum
// therefore carries the sum T of the absolute values of its hops' transported
// numbers (at most that of its products' absolute values), and a site with a sum of
// T < 2^54.5 last places is left to FP64 arithmetic too.  From there on the errors,
// at most 35 last places (2.8 per hop and one per alignment; 1.1 in the root mean
// square), are below 13 2^-53 T (0.4 2^-53 T), as those of FP64 arithmetic are.
// Measured, a component's error over 2^-53 and the sum of its products' absolute
// values, root mean square: Gaussian fields 0.13 (FP64 arithmetic 0.27), e^3 per time
// slice 0.34 (0.43), point sources 0.36 (0.46), one colour on links within 0.1 and
// 0.01 of 1 0.29 and 0.31 (0.33 and 0.34).  A Gaussian field has the eight terms
// of a component that small at about one site in 10^6; fields of one colour on links
// that hardly mix colours have them at every site (740 us at 24^3 x 48).  A row
// without a nonzero term is zero either way.
#pragma once

#include "dslash.cuh"

namespace wd {

struct FxArgs {
    DslashArgs<double> d;     // the FP64 links serve the sites that fall back
    int recon;                // their format
    int dagger;
    const char *fx_out, *fx_in;   // fixed-point links: 9 planes (re, im limbs) per direction
    size_t fx_dir_bytes;
    const int16_t *ex_out, *ex_in;   // link exponents [direction][stride]
    const int *any_exp;       // nonzero: some link exponent of the field is not 0
};

// 2^-523 and 2^477 as biased FP64 exponents: far enough from the ends of the
// range that no product or sum of a hop leaves it
constexpr int FX_MIN_EXP = 500, FX_MAX_EXP = 1500;
constexpr int FX_BAD_EXP = -32768;     // link exponent of a link that cannot be converted
constexpr int FX_LINK_EXP = 60;
constexpr int FX_PLANES = 9;
// the least sum of a component's absolute values, in units of 2^48 last places
constexpr int FX_MIN_MAG = 90;

// c + a b, 32 x 32 -> 64 bits signed, as the carry pair that assembles into
// one IMAD.WIDE (mad.wide.s32 becomes a product and a separate addition, and
// the C++ expression is reordered across the sums)
__device__ __forceinline__ long long imadw(int a, int b, long long c) {
    unsigned lo;
    int hi;
    asm("mad.lo.cc.u32 %0, %2, %3, %4;\n\tmadc.hi.s32 %1, %2, %3, %5;"
        : "=&r"(lo), "=r"(hi)
        : "r"(a), "r"(b), "r"((unsigned)c), "r"((int)(c >> 32)));
    return (long long)(((unsigned long long)(unsigned)hi << 32) | lo);
}
// arithmetic shift right by min(d, 63), and the logical one (0 from 64 on)
__device__ __forceinline__ long long sar64(long long v, int d) { return v >> min(d, 63); }
__device__ __forceinline__ unsigned long long shr64(unsigned long long v, unsigned d) {
    unsigned long long r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(d));
    return r;
}

// Fh of the FP64 value v against the block exponent word eh ((E << 20) |
// 0xFFFFF with E its biased exponent, at least v's): +-(mantissa 2^7) >> (E -
// e), negated if flip's sign bit is set.  Zeros and values 2^-60 below the
// block give 0.
__device__ __forceinline__ long long fx_fixed(double v, unsigned eh, int flip) {
    const int hi = __double2hiint(v), lo = __double2loint(v);
    const unsigned s = (eh - (unsigned)(hi & 0x7FFFFFFF)) >> 20;
    const unsigned m = ((unsigned)hi & 0xFFFFFu) | 0x100000u;
    unsigned long long x = (((unsigned long long)m << 32) | (unsigned)lo) << 7;
    x = shr64(x, s);
    const long long sg = (long long)((hi ^ flip) >> 31);
    return ((long long)x ^ sg) - sg;
}
// the signed limbs of f
__device__ __forceinline__ void fx_split(long long f, int &l1, int &l0) {
    l0 = (int)f;
    l1 = (int)(f >> 32) + (int)((unsigned)l0 >> 31);
}

// v 2^(x - 1080) rounded to FP64 (x in about 500 .. 1600): the conversion
// instruction, then the exponent field
__device__ __forceinline__ double fx_to_double(long long v, int x) {
    const double d = __ll2double_rn(v);
    const int hi = __double2hiint(d);
    return __hiloint2double(v == 0 ? 0 : hi + (x - 1080) * (1 << 20), __double2loint(d));
}

__device__ __forceinline__ double2 ld_nc_d2(const char *p) {
    const uint4 v = ld_nc_v4(p);
    return make_double2(__hiloint2double((int)v.y, (int)v.x), __hiloint2double((int)v.w, (int)v.z));
}

// neighbour of site h in direction mu, forward or backward
__device__ __forceinline__ unsigned fx_neighbour(const Geom &g, unsigned h, const int c[4], int mu,
                                                 bool fwd, bool &wrap) {
    if (mu == 0) {
        int xn = fwd ? c[0] + 1 : c[0] - 1;
        wrap = fwd ? xn == g.L[0] : xn < 0;
        if (wrap) xn = fwd ? 0 : g.L[0] - 1;
        return h + (unsigned)((xn >> 1) - (c[0] >> 1));
    }
    const int cm = mu == 1 ? c[1] : mu == 2 ? c[2] : c[3];
    const unsigned step = g.step[mu], back = g.back[mu];
    wrap = cm == (fwd ? g.L[mu] - 1 : 0);
    return fwd ? (wrap ? h - back : h + step) : (wrap ? h + back : h - step);
}

// The hops run as a loop over one body: mu, the sense and the row are the same
// for a warp, so every choice on them is a uniform branch (unrolled by
// direction and sense, warps waited on instruction fetch: 2.4 stalled cycles
// per instruction).

// the nine link elements of the hop from site `site`, in the order of the
// product: U forward, its transpose backward (32-bit byte offsets from a
// warp-uniform base)
__device__ __forceinline__ void fx_links(const FxArgs &A, unsigned site, int mu, bool fwd,
                                         uint4 U[3][3]) {
    const size_t plane = (size_t)A.d.g.stride * 16;
    const char *pu = (fwd ? A.fx_out : A.fx_in) + mu * A.fx_dir_bytes;
    const size_t pi = (fwd ? 3 : 1) * plane, pj = (fwd ? 1 : 3) * plane;
    const unsigned o = site * 16u;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) U[i][j] = ld_stream_v4(pu + i * pi + j * pj + o);
}

// whether row k enters gamma_mu with a minus sign: row 0 of gamma_y, row 1 of
// gamma_z
__device__ __forceinline__ bool fx_row_neg(int mu, int k) {
    return mu == 1 ? k == 0 : mu == 2 && k == 1;
}

// row k of the half spinor at neighbour hn, [colour][re, im]: p_k + s (i) q with
// the partner spin q = 3 - k (x, y) or 2 + k (z, t)
__device__ __forceinline__ void fx_half_row(const FxArgs &A, unsigned hn, int mu, int k, bool fwd,
                                            double r[6]) {
    const size_t plane = (size_t)A.d.g.stride * 16;
    const char *pp = (const char *)A.d.in + k * plane;
    const char *pq = (const char *)A.d.in + (mu < 2 ? 3 - k : 2 + k) * plane;
    const unsigned o = hn * 16u;
    const bool neg = (fwd != (A.dagger != 0)) != fx_row_neg(mu, k);
    const double s = __hiloint2double(neg ? (int)0xBFF00000u : 0x3FF00000, 0);
    const double ns = __hiloint2double(neg ? 0x3FF00000 : (int)0xBFF00000u, 0);
    double2 p[3], q[3];
#pragma unroll
    for (int cc = 0; cc < 3; ++cc) {
        p[cc] = ld_nc_d2(pp + (4 * cc) * plane + o);
        q[cc] = ld_nc_d2(pq + (4 * cc) * plane + o);
    }
    if ((mu & 1) == 0) {   // p + s i q
#pragma unroll
        for (int cc = 0; cc < 3; ++cc) {
            r[2 * cc] = fma(ns, q[cc].y, p[cc].x);
            r[2 * cc + 1] = fma(s, q[cc].x, p[cc].y);
        }
    } else {               // p + s q
#pragma unroll
        for (int cc = 0; cc < 3; ++cc) {
            r[2 * cc] = fma(s, q[cc].x, p[cc].x);
            r[2 * cc + 1] = fma(s, q[cc].y, p[cc].y);
        }
    }
}

// r *= the boundary phase of direction mu (it commutes with the link)
__device__ __forceinline__ void fx_phase(const FxArgs &A, int mu, bool fwd, double r[6]) {
    const double pr = A.d.ph[2 * mu], pi = fwd ? A.d.ph[2 * mu + 1] : -A.d.ph[2 * mu + 1];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const double t = r[2 * i] * pr - r[2 * i + 1] * pi;
        r[2 * i + 1] = r[2 * i] * pi + r[2 * i + 1] * pr;
        r[2 * i] = t;
    }
}

// any bit of r but the signs set (bits, not values: FP64 comparisons would
// cost as much as the sums)
__device__ __forceinline__ unsigned fx_bits(const double r[6]) {
    unsigned any = 0;
#pragma unroll
    for (int i = 0; i < 6; ++i)
        any |= ((unsigned)__double2hiint(r[i]) & 0x7FFFFFFFu) | (unsigned)__double2loint(r[i]);
    return any;
}
__device__ __forceinline__ unsigned fx_max(const double r[6]) {
    unsigned mx = 0;
#pragma unroll
    for (int i = 0; i < 6; ++i) mx = max(mx, (unsigned)__double2hiint(r[i]) & 0x7FFFFFFFu);
    return mx;
}

// the row transported, u[colour][re, im], in units of the block exponent eh
__device__ __forceinline__ void fx_product(const uint4 U[3][3], const double r[6], unsigned eh,
                                           bool fwd, long long u[6]) {
    // backward: conj(U)^T h = conj(U^T conj(h)); i are the limbs of the
    // imaginary parts entering the product, j those of their negatives
    const int cj = fwd ? 0 : (int)0x80000000u;
    int r1[3], r0[3], i1[3], i0[3], j1[3], j0[3];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        const long long re = fx_fixed(r[2 * b], eh, 0), im = fx_fixed(r[2 * b + 1], eh, cj);
        fx_split(re, r1[b], r0[b]);
        fx_split(im, i1[b], i0[b]);
        fx_split(-im, j1[b], j0[b]);
    }
    // the leading and the middle sums of the real and the imaginary part; the
    // middle ones start at half a last place
    long long ph[3], pm[3], qh[3], qm[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        ph[i] = qh[i] = 0;
        pm[i] = qm[i] = 1ll << 31;
    }
#pragma unroll
    for (int b = 0; b < 3; ++b)
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const int u1r = (int)U[i][b].y, u0r = (int)U[i][b].x;
            const int u1i = (int)U[i][b].w, u0i = (int)U[i][b].z;
            ph[i] = imadw(u1r, r1[b], ph[i]);
            pm[i] = imadw(u1r, r0[b], pm[i]);
            qh[i] = imadw(u1r, i1[b], qh[i]);
            qm[i] = imadw(u1r, i0[b], qm[i]);
            pm[i] = imadw(u0r, r1[b], pm[i]);
            qm[i] = imadw(u0r, i1[b], qm[i]);
            ph[i] = imadw(u1i, j1[b], ph[i]);
            pm[i] = imadw(u1i, j0[b], pm[i]);
            qh[i] = imadw(u1i, r1[b], qh[i]);
            qm[i] = imadw(u1i, r0[b], qm[i]);
            pm[i] = imadw(u0i, j1[b], pm[i]);
            qm[i] = imadw(u0i, r1[b], qm[i]);
        }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        u[2 * i] = imadw((int)(pm[i] >> 32), 1, ph[i]);
        u[2 * i + 1] = imadw((int)(qm[i] >> 32), 1, qh[i]);
    }
    if (!fwd) {
#pragma unroll
        for (int i = 0; i < 3; ++i) u[2 * i + 1] = -u[2 * i + 1];
    }
}

// a += u, and the row's term of spin 2 or 3 without the projector's sign, b +=
// -i u (x, z) or u (y, t), subtracted if minus
__device__ __forceinline__ void fx_accumulate(long long a[6], long long b[6], const long long u[6],
                                              int mu, bool minus) {
#pragma unroll
    for (int i = 0; i < 6; ++i) a[i] += u[i];
    if ((mu & 1) == 0) {
        if (minus) {
#pragma unroll
            for (int i = 0; i < 3; ++i) { b[2 * i] -= u[2 * i + 1]; b[2 * i + 1] += u[2 * i]; }
        } else {
#pragma unroll
            for (int i = 0; i < 3; ++i) { b[2 * i] += u[2 * i + 1]; b[2 * i + 1] -= u[2 * i]; }
        }
    } else if (minus) {
#pragma unroll
        for (int i = 0; i < 6; ++i) b[i] -= u[i];
    } else {
#pragma unroll
        for (int i = 0; i < 6; ++i) b[i] += u[i];
    }
}

// |re|, |im| (one less for negative ones) in units of 2^48, in the halves of a
// word: at most 2.46 2^10 of a hop, 2.46 2^13 of a component's eight
__device__ __forceinline__ unsigned fx_mag(long long re, long long im) {
    const unsigned hr = (unsigned)((unsigned long long)re >> 32);
    const unsigned hi = (unsigned)((unsigned long long)im >> 32);
    unsigned m, s;
    asm("prmt.b32 %0, %1, %2, 0x7632;" : "=r"(m) : "r"(hr), "r"(hi));
    asm("prmt.b32 %0, %1, %2, 0xFFBB;" : "=r"(s) : "r"(hr), "r"(hi));   // the signs
    return m ^ s;
}
// both halves shifted right by d >= 0
__device__ __forceinline__ unsigned fx_mag_shift(unsigned t, int d) {
    return d > 15 ? 0u : (t >> d) & ((0xFFFFu >> d) * 0x10001u);
}
// whether both halves reach FX_MIN_MAG
__device__ __forceinline__ bool fx_mag_ok(unsigned t) {
    return ((t + (0x8000u - FX_MIN_MAG) * 0x10001u) & 0x80008000u) == 0x80008000u;
}
// ta, tb (a word per colour, 32 apart) += the magnitudes of the terms that
// fx_accumulate adds to a and b
__device__ __forceinline__ void fx_magnitudes(unsigned *ta, unsigned *tb, const long long u[6],
                                              int mu) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const unsigned m = fx_mag(u[2 * i], u[2 * i + 1]);
        atomicAdd(ta + 32 * i, m);
        atomicAdd(tb + 32 * i, (mu & 1) ? m : __byte_perm(m, 0, 0x1032));
    }
}

__device__ __forceinline__ bool fx_out_of_range(int eb, int eu) {
    return eb < FX_MIN_EXP || eb > FX_MAX_EXP || eu == FX_BAD_EXP;
}
__device__ __forceinline__ int fx_link_exp(const FxArgs &A, bool any_exp, unsigned site, int mu,
                                           bool fwd) {
    if (!any_exp) return 0;
    return (fwd ? A.ex_out : A.ex_in)[(size_t)mu * A.d.g.stride + site];
}
// The vote, to which every lane of the warp comes in every hop, makes this a branch
// (as predicated instructions the FP64 products of the phase would take the pipe in
// every hop).
__device__ __forceinline__ bool fx_wraps(const FxArgs &A, int mu, bool wrap) {
    return (A.d.phase_on >> mu & 1u) && __any_sync(0xffffffffu, wrap) && wrap;
}

// FP64 arithmetic, for the sites that the fixed-point form leaves to it.  Element
// (i, j) of the matrix of the hop's product, U forward, its adjoint backward
// (12-real links: row 2 is rebuilt as in load_link)
template <int RECON>
__device__ __forceinline__ double2 fx_elem_f64(const FxArgs &A, unsigned site, int mu, bool fwd,
                                               int i, int j) {
    const size_t plane = (size_t)A.d.g.stride * 16;
    const char *base = (fwd ? A.d.gauge_out : A.d.gauge_in) + mu * A.d.dir_bytes + site * 16u;
    const int r = fwd ? i : j, c = fwd ? j : i;
    double2 e;
    if (RECON == 18 || r < 2) {
        e = ld_nc_d2(base + (3 * r + c) * plane);
    } else {
        const int c1 = c == 2 ? 0 : c + 1, c2 = c == 0 ? 2 : c - 1;
        const double2 a1 = ld_nc_d2(base + c1 * plane), a2 = ld_nc_d2(base + c2 * plane);
        const double2 b1 = ld_nc_d2(base + (3 + c1) * plane), b2 = ld_nc_d2(base + (3 + c2) * plane);
        e.x = a1.x * b2.x; e.x -= a1.y * b2.y; e.x -= a2.x * b1.x; e.x += a2.y * b1.y;
        e.y = a2.x * b1.y; e.y += a2.y * b1.x; e.y -= a1.x * b2.y; e.y -= a1.y * b2.x;
    }
    // (on the sign bit: a conditional negation of a double is an FP64 instruction)
    return make_double2(e.x, __hiloint2double(__double2hiint(e.y) ^ (fwd ? 0 : (int)0x80000000u),
                                              __double2loint(e.y)));
}
// colour i of the transported row r
template <int RECON>
__device__ __forceinline__ double2 fx_colour_f64(const FxArgs &A, unsigned site, int mu, bool fwd,
                                                 int i, const double r[6]) {
    double2 u;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const double2 e = fx_elem_f64<RECON>(A, site, mu, fwd, i, j);
        u.x = j == 0 ? pmul(e.x, r[0]) : pmac(e.x, r[2 * j], u.x);
        u.y = j == 0 ? pmul(e.x, r[1]) : pmac(e.x, r[2 * j + 1], u.y);
        u.x = pmsub(e.y, r[2 * j + 1], u.x);
        u.y = pmac(e.y, r[2 * j], u.y);
    }
    return u;
}
__device__ __forceinline__ double2 fx_phase_f64(const FxArgs &A, int mu, bool fwd, double2 u) {
    const double pr = A.d.ph[2 * mu], pi = fwd ? A.d.ph[2 * mu + 1] : -A.d.ph[2 * mu + 1];
    return make_double2(u.x * pr - u.y * pi, u.x * pi + u.y * pr);
}

// Work split: the four warps of a 128-thread block take 32 consecutive sites,
// warp (k, dir) row k of the half spinors of their four forward or four
// backward hops.  One thread per site needs 24 64-bit accumulators (152
// registers, 12 warps per SM); without the check of the components it measured the
// same at 32^3 x 64 (518 against 515 us) and loses below: 188 / 172 us at 24^3 x 48,
// 48 / 41 at 16^3 x 32, 24 / 11 at 8^4.  Row k goes into
// spin k (accumulator a) and spin 3 - k for directions x and y, 2 + k for z
// and t (accumulator b, exchanged between the two rows' warps in between); the
// forward and the backward warp add up at the end, where one keeps spin k and
// the other spin 2 + k.  Both exchanges go through shared memory.
constexpr int FX_BLOCK = 128;
constexpr int FX_SITES = 32;      // sites per block

struct FxShared {
    long long v[2][4][6][32];
    // Magnitudes: words of one thread at a time, in shared memory because six
    // registers more spill (197 against 210 us at 24^3 x 48); its additions need no
    // result, so they go out as atomics (200 as loads and stores).
    unsigned ta[4][3][32], tb[4][3][32];
    int xa[2][4][32];
};

// The sites marked by any of the four warps, in FP64 arithmetic and the same split,
// so that a site costs what it costs in the plain hop.  A hop with every site
// marked before the first product (a field near 1e-290): 160 us at 16^3 x 32, 731
// at 24^3 x 48; marked after the products, 165 and 740; FP64 arithmetic alone with
// a thread per site, 131 and 563.
// (Every thread its whole site: 442 and 2127 us.)  Every thread of the block calls it.
template <int RECON>
__device__ __noinline__ void fx_site_f64(const FxArgs &A, unsigned h, int w, FxShared &sh, bool bad,
                                         double v[6]) {
    const int lane = threadIdx.x & 31, k = w & 1;
    const bool fwd = w < 2;
    sh.xa[0][w][lane] = bad;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 4; ++q) bad = bad || sh.xa[0][q][lane] != 0;
    int c[4];
    site_coords(A.d.g, h, A.d.parity, c);
    double a[6], b[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) a[i] = b[i] = 0;
#pragma unroll 1
    for (int mu = 0; mu < 4; ++mu) {
        if (mu == 2) {   // row k goes on with spin 2 + k
#pragma unroll
            for (int i = 0; i < 6; ++i) sh.v[0][w][i][lane] = __double_as_longlong(b[i]);
            __syncwarp();
            __syncthreads();
#pragma unroll
            for (int i = 0; i < 6; ++i) b[i] = __longlong_as_double(sh.v[0][w ^ 1][i][lane]);
        }
        bool wrap;
        const unsigned hn = fx_neighbour(A.d.g, h, c, mu, fwd, wrap), site = fwd ? h : hn;
        wrap = wrap && bad && (A.d.phase_on >> mu & 1u);
        const bool phase = __any_sync(0xffffffffu, wrap);   // (a branch, as in fx_wraps)
        if (!bad) continue;
        double r[6];
        fx_half_row(A, hn, mu, k, fwd, r);
        const double sb = fx_row_neg(mu, k) ? -1.0 : 1.0;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            double2 u = fx_colour_f64<RECON>(A, site, mu, fwd, i, r);
            if (phase && wrap) u = fx_phase_f64(A, mu, fwd, u);
            a[2 * i] += u.x;
            a[2 * i + 1] += u.y;
            b[2 * i] = fma(sb, (mu & 1) ? u.x : u.y, b[2 * i]);
            b[2 * i + 1] = fma((mu & 1) ? sb : -sb, (mu & 1) ? u.y : u.x, b[2 * i + 1]);
        }
    }
#pragma unroll
    for (int i = 0; i < 6; ++i) sh.v[1][w][i][lane] = __double_as_longlong(fwd ? b[i] : a[i]);
    __syncwarp();
    __syncthreads();
    if (!bad) return;
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        const double got = __longlong_as_double(sh.v[1][w ^ 2][i][lane]), own = fwd ? a[i] : b[i];
        v[i] = fwd ? own + got : A.dagger ? got - own : own - got;
    }
}

// every thread of the block calls it, the four warps of one lane on the same
// site h: v = spin k (forward warps) or 2 + k of H in, [colour][re, im]
__device__ __forceinline__ void fx_site(const FxArgs &A, unsigned h, int w, FxShared &sh,
                                             double v[6]) {
    const int lane = threadIdx.x & 31, k = w & 1;
    const bool fwd = w < 2;
    int c[4];
    site_coords(A.d.g, h, A.d.parity, c);
    const bool any_exp = __ldg(A.any_exp) != 0;
    long long a[6], b[6];
    unsigned *ta = &sh.ta[w][0][lane], *tb = &sh.tb[w][0][lane];   // as a and b
#pragma unroll
    for (int i = 0; i < 6; ++i) a[i] = b[i] = 0;
#pragma unroll
    for (int i = 0; i < 3; ++i) ta[32 * i] = tb[32 * i] = 0;
    int xa = -(1 << 20);
    bool bad = false, any_a = false, any_b = false;   // any term in a, in b
#pragma unroll 1
    for (int mu = 0; mu < 4; ++mu) {
        if (mu == 2) {   // row k goes on with spin 2 + k
#pragma unroll
            for (int i = 0; i < 6; ++i) sh.v[0][w][i][lane] = b[i];
            sh.xa[0][w][lane] = xa;
            __syncwarp();
            __syncthreads();
            const int xo = sh.xa[0][w ^ 1][lane];
#pragma unroll
            for (int i = 0; i < 6; ++i) b[i] = sh.v[0][w ^ 1][i][lane];
            tb = &sh.tb[w ^ 1][0][lane];
            any_b = xo >= 0;
            if (xo != xa) {   // b comes in the other row's units
                const int x = max(xo, xa);
                if (xa >= 0) {
#pragma unroll
                    for (int i = 0; i < 6; ++i) a[i] = sar64(a[i], x - xa);
#pragma unroll
                    for (int i = 0; i < 3; ++i) ta[32 * i] = fx_mag_shift(ta[32 * i], x - xa);
                }
                if (xo >= 0) {
#pragma unroll
                    for (int i = 0; i < 6; ++i) b[i] = sar64(b[i], x - xo);
#pragma unroll
                    for (int i = 0; i < 3; ++i) tb[32 * i] = fx_mag_shift(tb[32 * i], x - xo);
                }
                xa = x;
            }
        }
        bool wrap;
        const unsigned hn = fx_neighbour(A.d.g, h, c, mu, fwd, wrap), site = fwd ? h : hn;
        uint4 U[3][3];
        fx_links(A, site, mu, fwd, U);
        const int eu = fx_link_exp(A, any_exp, site, mu, fwd);
        double r[6];
        fx_half_row(A, hn, mu, k, fwd, r);
        if (fx_wraps(A, mu, wrap)) fx_phase(A, mu, fwd, r);
        const int eb = (int)(fx_max(r) >> 20);
        if (fx_out_of_range(eb, eu)) {
            if (fx_bits(r) != 0 || eu == FX_BAD_EXP) bad = true;
            continue;
        }
        if (eb + eu > xa) {   // a larger hop
            const int x = eb + eu;
            if (xa >= 0) {
                const int d = x - xa;
#pragma unroll
                for (int i = 0; i < 6; ++i) {
                    a[i] = sar64(a[i], d);
                    b[i] = sar64(b[i], d);
                }
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    ta[32 * i] = fx_mag_shift(ta[32 * i], d);
                    tb[32 * i] = fx_mag_shift(tb[32 * i], d);
                }
            }
            xa = x;
        }
        any_a = any_b = true;
        long long u[6];
        fx_product(U, r, ((unsigned)(xa - eu) << 20) | 0xFFFFFu, fwd, u);
        fx_accumulate(a, b, u, mu, fx_row_neg(mu, k));
        fx_magnitudes(ta, tb, u, mu);
    }
    // the forward warp keeps a and gives b, the backward warp the reverse; what
    // has no term comes without an exponent, a bad site is marked in it
    const int xg = (fwd ? any_b : any_a) ? xa : -1;
    const int xk = (fwd ? any_a : any_b) ? xa : -1;
#pragma unroll
    for (int i = 0; i < 6; ++i) sh.v[1][w][i][lane] = fwd ? b[i] : a[i];
    sh.xa[1][w][lane] = bad ? (1 << 24) : xg;
    __syncwarp();
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 4; ++q) bad = bad || sh.xa[1][q][lane] == (1 << 24);
    const int xb = sh.xa[1][w ^ 2][lane], xm = max(xk, xb);
    if (!bad && xm >= 0) {
        // the warp's own and the partner's, the one with the smaller exponent shifted
        const unsigned *to = fwd ? &sh.ta[w][0][lane] : &sh.tb[w ^ 1][0][lane];
        const unsigned *tg = fwd ? &sh.ta[w ^ 2][0][lane] : &sh.tb[w ^ 3][0][lane];
        const unsigned *big = xk >= xb ? to : tg, *small = xk >= xb ? tg : to;
#pragma unroll
        for (int i = 0; i < 3; ++i)
            bad = bad || !fx_mag_ok(big[32 * i] + fx_mag_shift(small[32 * i], xm - min(xk, xb)));
    }
    // opposite projectors: spins 2, 3 take forward minus backward, times the
    // forward one's sign (-1 for H, +1 for H^dag)
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        long long got = sh.v[1][w ^ 2][i][lane], own = fwd ? a[i] : b[i];
        if (xk != xb) {
            got = xb >= 0 ? sar64(got, xm - xb) : 0;
            own = xk >= 0 ? sar64(own, xm - xk) : 0;
        }
        const long long sum = fwd ? own + got : A.dagger ? got - own : own - got;
        v[i] = fx_to_double(sum, xm);
    }
    __syncwarp();
    if (!__syncthreads_or(bad)) return;
    double t[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) t[i] = v[i];
    if (A.recon == 12) fx_site_f64<12>(A, h, w, sh, bad, t);
    else fx_site_f64<18>(A, h, w, sh, bad, t);
#pragma unroll
    for (int i = 0; i < 6; ++i) v[i] = t[i];
}

// The same with one hop per warp, for lattices whose blocks leave the chip nearly
// empty: there a launch is a warp's chain of four hops, on four warps per SM.
// Sixteen warps take 32 sites, warp w = 4 mu + 2 backward + k row k of one hop,
// and leave the product and its exponent in shared memory; then twelve warps
// each add the eight terms of one complex number j = 4 colour + spin, in units
// of the largest exponent.
//
// A hop, with the host's share, one warp per row and sense / one per hop (before
// the check of the components):
//   blocks    4 (4^4)   64 (8^4)   128 (8^3 x 16)   192   324 (12^4)   2048
//   us     10.9 / 8.0  11.0 / 8.7    11.3 / 8.7   13.2 / 13.0  14.8 / 17.7  42 / 67
// so the line lies where one block per SM ends (fx_one_hop_per_warp): blocks of 16
// warps with 82 registers run one at a time on an SM.
constexpr int FXW_BLOCK = 512;

struct FxWideShared {
    long long u[16][6][32];
    int xa[16][32];      // exponent, negative: no term, 1 << 24: a bad site
};

// complex number 4 cc + s of H in at site h in FP64 arithmetic
template <int RECON>
__device__ __noinline__ double2 fx_number_f64(const FxArgs &A, unsigned h, int cc, int s) {
    int c[4];
    site_coords(A.d.g, h, A.d.parity, c);
    double2 v = make_double2(0.0, 0.0);
#pragma unroll 1
    for (int t = 0; t < 8; ++t) {
        const int mu = t >> 1, k = s < 2 ? s : t < 4 ? 3 - s : s - 2;
        const bool fwd = (t & 1) == 0;
        bool wrap;
        const unsigned hn = fx_neighbour(A.d.g, h, c, mu, fwd, wrap), site = fwd ? h : hn;
        double r[6];
        fx_half_row(A, hn, mu, k, fwd, r);
        double2 u = fx_colour_f64<RECON>(A, site, mu, fwd, cc, r);
        if (wrap && (A.d.phase_on >> mu & 1u)) u = fx_phase_f64(A, mu, fwd, u);
        const bool swap = s >= 2 && (mu & 1) == 0;
        const bool minus = s >= 2 && fx_row_neg(mu, k) != (fwd == (A.dagger == 0));
        const double sg = minus ? -1.0 : 1.0;
        v.x = fma(sg, swap ? u.y : u.x, v.x);
        v.y = fma(swap ? -sg : sg, swap ? u.x : u.y, v.y);
    }
    return v;
}

// v = complex number w (w < 12) of H in at site h, [re, im]
__device__ __forceinline__ void fx_site_wide(const FxArgs &A, unsigned h, int w, FxWideShared &sh,
                                             double v[2]) {
    const int lane = threadIdx.x & 31;
    {
        const int mu = w >> 2, k = w & 1;
        const bool fwd = (w & 2) == 0;
        int c[4];
        site_coords(A.d.g, h, A.d.parity, c);
        bool wrap;
        const unsigned hn = fx_neighbour(A.d.g, h, c, mu, fwd, wrap), site = fwd ? h : hn;
        uint4 U[3][3];
        fx_links(A, site, mu, fwd, U);
        const int eu = fx_link_exp(A, __ldg(A.any_exp) != 0, site, mu, fwd);
        double r[6];
        fx_half_row(A, hn, mu, k, fwd, r);
        if (fx_wraps(A, mu, wrap)) fx_phase(A, mu, fwd, r);
        const int eb = (int)(fx_max(r) >> 20);
        int xa = eb + eu;
        if (fx_out_of_range(eb, eu)) {
            xa = fx_bits(r) != 0 || eu == FX_BAD_EXP ? 1 << 24 : -1;
        } else {
            long long u[6];
            fx_product(U, r, ((unsigned)eb << 20) | 0xFFFFFu, fwd, u);
#pragma unroll
            for (int i = 0; i < 6; ++i) sh.u[w][i][lane] = u[i];
        }
        sh.xa[w][lane] = xa;
    }
    __syncthreads();
    if (w >= 12) return;
    const int s = w & 3, cc = w >> 2;
    int xm = -1, xt[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) {   // t = 2 mu + backward
        const int k = s < 2 ? s : t < 4 ? 3 - s : s - 2;
        xt[t] = sh.xa[2 * t + k][lane];
        xm = max(xm, xt[t]);
    }
    long long re = 0, im = 0;
    int mr = 0, mi = 0;   // the sums of the absolute values, in units of 2^32
    bool bad = xm == 1 << 24;
    if (!bad) {
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            if (xt[t] < 0) continue;
            const int mu = t >> 1, k = s < 2 ? s : t < 4 ? 3 - s : s - 2;
            const long long ur = sar64(sh.u[2 * t + k][2 * cc][lane], xm - xt[t]);
            const long long ui = sar64(sh.u[2 * t + k][2 * cc + 1][lane], xm - xt[t]);
            // -i u (x, z) or u (y, t) for spins 2 and 3, with the row's sign; H:
            // backward minus forward, H^dag the reverse
            const bool swap = s >= 2 && (mu & 1) == 0;
            const bool minus =
                s >= 2 && fx_row_neg(mu, k) != ((t & 1) == (A.dagger != 0 ? 1 : 0));
            const long long br = swap ? ui : ur, bi = swap ? -ur : ui;
            re += minus ? -br : br;
            im += minus ? -bi : bi;
            const int hr = (int)(br >> 32), hi = (int)(bi >> 32);
            mr += hr ^ (hr >> 31);
            mi += hi ^ (hi >> 31);
        }
        bad = xm >= 0 && min(mr, mi) < FX_MIN_MAG << 16;
    }
    if (bad) {
        const double2 f = A.recon == 12 ? fx_number_f64<12>(A, h, cc, s)
                                        : fx_number_f64<18>(A, h, cc, s);
        v[0] = f.x;
        v[1] = f.y;
        return;
    }
    v[0] = fx_to_double(re, xm);
    v[1] = fx_to_double(im, xm);
}

}  // namespace wd
