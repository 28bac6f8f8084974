// Block fixed-point arithmetic ("FX"): FP64-accurate sums of products on the
// integer multiply-add pipe.
//
// GB300 issues an FP64 FMA on 2 lanes per clock and SM, an IMAD.WIDE
// (32 x 32 + 64 -> 64 bits) on 64 (measured: 2.0 and 63.8), so a product
// built from three IMAD.WIDE is ten times cheaper than one FP64 FMA.  A
// number is a signed integer t times a power of two shared by a whole site
// (spinors, |t| < 2^57; clover blocks, 2^55) or by the field (links, whose
// entries are at most 1 = 2^55), kept as two limbs, t = h 2^28 + l.  A sum of
// products keeps two 64-bit accumulators:
//     sum a b = 2^56 sum ah bh + 2^28 sum (ah bl + al bh) + (sum al bl),
// the last term (below 1/4 unit of the result per product) is dropped, and
// the result is sum ah bh + (mid >> 28) in units of 2^56.  Every step is
// exact integer arithmetic but for that term and the final rounding, about
// 2^-57 of the largest component of the site: several times less than the FP64
// forms lose in their chains of roundings (2^-53 of the running sum per FMA) --
// against the size of the site, that is: a component 2^-20 of its site's largest
// keeps 37 bits where FP64 keeps 53.
#pragma once

#include "qcd_internal.cuh"

namespace qcd {

constexpr int FX_BITS = 55;  // links and clover blocks: |t| <= 2^FX_BITS
constexpr int FX_VBITS = 57; // spinors: |t| < 2^FX_VBITS
constexpr int FX_LIMB = 28;
// Links of a larger squared Frobenius norm (SU(3): 3) keep the FP64 forms.
// With it every product of links below stays in range: |A B| <= 3, |A B C| <=
// 5.2 entry by entry, so that limbs stay below 2^31 and sums below 2^63.
constexpr float FX_LINK_FRO2 = 3.001f;
// Rounding here is relative to the largest entry of a link (2^-55) and of a site
// (2^-57), FP64's to each term of a sum.  The two agree where a link turns no
// vector into one much smaller than itself and mixes the colours, so a field keeps
// the FP64 forms if it has a link that
//   has a squared norm below this (uniformly small entries, zero links);
constexpr float FX_LINK_FRO2_MIN = 0.5f;
//   is further than this from a multiple of a unitary matrix (the rows' squared
//   norms and products, against their mean squared norm: diag(1, 1e-12, 1), a
//   small or a dependent row; its action stays within 5 per cent of the mean);
constexpr float FX_LINK_UNITARY = 1.f / 64;
//   or has an entry whose square is below this (2^-32: unit, diagonal and block
//   diagonal links, whose colours stay apart).  A random SU(3) link has one with
//   a probability of some 1e-18.
constexpr float FX_LINK_ENTRY2 = 5.4e-20f;

// a += x y as one instruction (written in C the sums are reassociated into
// products and 64-bit additions, three instructions each)
__device__ __forceinline__ void fx_mac(long long &a, int x, int y)
{
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(a) : "r"(x), "r"(y));
}
__device__ __forceinline__ long long fx_mul(int x, int y) { return (long long)x * y; }

// the limbs of t
__device__ __forceinline__ int fx_lo(long long t) { return ((int)(unsigned)t << 4) >> 4; }
__device__ __forceinline__ int fx_hi(long long t) { return (int)((t + (1ll << (FX_LIMB - 1))) >> FX_LIMB); }

// One complex number as limbs
struct fxc {
    int rh, rl, ih, il;
};
__device__ __forceinline__ fxc fx_unpack(int4 v) { return fxc{v.x, v.y, v.z, v.w}; }
__device__ __forceinline__ int4 fx_pack(long long r, long long i) { return make_int4(fx_hi(r), fx_lo(r), fx_hi(i), fx_lo(i)); }

// FP64 -> FP32 on the integer pipe: a conversion instruction keeps the two FP64
// lanes as long as an FMA, and the kernels that build the links and the clover
// blocks in four precisions waited on those (24^3x48, links 0.28 -> 0.23 ms,
// clover blocks 0.81 -> 0.70 ms a parity; with the links' check and rounding
// and denormals kept 0.21 and 0.73).
// Rounded to nearest even as (float)d; odd = true: cut off, the last bit set if
// anything was lost, so that rounding the result to IEEE half equals rounding d.
// Only for zero and FP32's normal range: *slow is set for anything else.
template <bool ODD>
__device__ __forceinline__ float f32_int(double d, bool &slow)
{
    const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
    const unsigned mag = hi & 0x7fffffffu, r = lo << 3;
    const bool zero = (mag | lo) == 0;
    slow = slow || (!zero && mag - (897u << 20) >= (254u << 20));
    unsigned u = ((mag - (896u << 20)) << 3) | (lo >> 29);
    if (ODD) u |= r != 0;
    else u += r + (u & 1) > 0x80000000u;
    return __uint_as_float((zero ? 0u : u) | (hi & 0x80000000u));
}

// rint-free conversion of a double with |d| <= 1: t = d 2^55, rounded to nearest
// (2^-56 absolute, a sixteenth of a unit in the last place of 1).
// Larger, infinite or NaN values set *bad (links of SU(3) have none).
__device__ __forceinline__ long long fx_from_unit(double d, int &bad)
{
    const long long b = __double_as_longlong(d);
    const int hi = (int)(b >> 32);
    const int ex = (hi >> 20) & 0x7ff;
    bad |= (b & 0x7fffffffffffffffll) > __double_as_longlong(1.0 + 1e-9);
    if (ex == 0) return 0;  // zero and denormals (far below a unit)
    long long m = (b & 0xfffffffffffffll) | 0x10000000000000ll;  // 2^52 <= m < 2^53
    const int sh = 1023 - ex;                                    // |d| = m 2^(-52 - sh)
    m = (((m << 4) >> (sh < 0 ? 0 : sh > 63 ? 63 : sh)) + 1) >> 1;
    return b < 0 ? -m : m;
}

// Whether a link, its entries f rounded to FP32, is one that the fixed-point forms
// take (the constants above; false for NaN)
__device__ __forceinline__ bool fx_link_ok(const float2 f[9])
{
    float n[3], small = 1.f;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        n[i] = 0.f;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const float e = f[3 * i + j].x * f[3 * i + j].x + f[3 * i + j].y * f[3 * i + j].y;
            n[i] += e;
            small = fminf(small, e);
        }
    }
    const float fro = n[0] + n[1] + n[2], tol = FX_LINK_UNITARY * fro;
    bool ok = fro <= FX_LINK_FRO2 && fro >= FX_LINK_FRO2_MIN && small >= FX_LINK_ENTRY2;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        ok = ok && fabsf(3.f * n[i] - fro) <= tol;
        const int k = i == 2 ? 0 : i + 1;  // row i times row k
        float re = 0.f, im = 0.f;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const float2 a = f[3 * i + j], b = f[3 * k + j];
            re += a.x * b.x + a.y * b.y;
            im += a.y * b.x - a.x * b.y;
        }
        ok = ok && 9.f * (re * re + im * im) <= tol * tol;
    }
    return ok;
}

// The link m (row by row) as direction mu of site cb; true if it is out of range
__device__ __forceinline__ bool fx_store_link(const double2 m[9], int4 *ux, int cb, int mu)
{
    int bad = 0;
    float2 f[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        ux[soa(cb, 36, mu * 9 + k)] = fx_pack(fx_from_unit(m[k].x, bad), fx_from_unit(m[k].y, bad));
        bool tiny = false;  // below FP32's normal range (above it is bad): too small to count
        f[k].x = f32_int<false>(m[k].x, tiny);
        if (tiny) f[k].x = 0.f;
        tiny = false;
        f[k].y = f32_int<false>(m[k].y, tiny);
        if (tiny) f[k].y = 0.f;
    }
    return bad || !fx_link_ok(f);
}

// ---------------------------------------------------------------- 3x3 matrices
// A link product in FX: entries at most 1 (field scale 2^-55)
struct M3x {
    fxc m[3][3];
};

// (A B)_ij in the operands' scale: t_C = t_A t_B 2^-55.  For entries up to 1 every
// accumulator stays below 2^62 (three complex products, limbs up to 2^29.6
// after one product of three terms).
__device__ __forceinline__ void fx_mul_elem(const M3x &A, const M3x &B, int i, int j, long long &tr, long long &ti)
{
    // mid sums start at half a unit of their final shift
    long long mr = 1ll << 26, mi = 1ll << 26, hr = 0, hi = 0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const fxc a = A.m[i][k], b = B.m[k][j];
        fx_mac(mr, a.rh, b.rl);
        fx_mac(mr, a.rl, b.rh);
        fx_mac(mr, -a.ih, b.il);
        fx_mac(mr, -a.il, b.ih);
        fx_mac(mi, a.rh, b.il);
        fx_mac(mi, a.rl, b.ih);
        fx_mac(mi, a.ih, b.rl);
        fx_mac(mi, a.il, b.rh);
        fx_mac(hr, a.rh, b.rh);
        fx_mac(hr, -a.ih, b.ih);
        fx_mac(hi, a.rh, b.ih);
        fx_mac(hi, a.ih, b.rh);
    }
    tr = (hr << 1) + (mr >> 27);
    ti = (hi << 1) + (mi >> 27);
}

// ---------------------------------------------------------------- spinors
// A real as limbs, with the additions the spin projection needs (limb by limb:
// the sum of two numbers below 2^57 has limbs up to 2^30 and below 2^29)
struct fx2 {
    int h, l;
};
__device__ __forceinline__ fx2 operator+(fx2 a, fx2 b) { return {a.h + b.h, a.l + b.l}; }
__device__ __forceinline__ fx2 operator-(fx2 a, fx2 b) { return {a.h - b.h, a.l - b.l}; }
__device__ __forceinline__ fx2 operator-(fx2 a) { return {-a.h, -a.l}; }

// Unit exponents: the value of t is t 2^e.  FX_ZERO is below every one of them (a
// sum of nothing); a site with an infinite or NaN component has FX_NAN, and so
// has every result that reads it.
constexpr int FX_ZERO = -100000, FX_NAN = 100000;

// the limbs of a signed t, the low one unsigned (the partner's low limb is
// balanced wherever two low limbs would meet)
__device__ __forceinline__ fx2 fx_split(long long t) { return {(int)(t >> FX_LIMB), (int)t & ((1 << FX_LIMB) - 1)}; }

__device__ __forceinline__ int fx_clamp63(int s) { return s > 63 ? 63 : s; }

// a double's exponent field, and its t in units of 2^(E - 1023 - 56) for a site
// whose largest exponent field is E >= 1 (bits below one unit cut off).  Field 0
// (zero and denormals) has field 1's unit and no leading one.  (S_ee calls in FP64 at
// 16^3x32, with denormals cut to zero / so / with a test a site and a scaling where it
// matters: 111.4 / 113.7 / 117.5 us; hopping term 42.5 / 42.5 / 45.1.)
__device__ __forceinline__ int fx_field(double d) { return (__double2hiint(d) >> 20) & 0x7ff; }
template <int UP, bool ROUND>  // the mantissa's 53 bits up by UP; rounded or cut
__device__ __forceinline__ unsigned long long fx_mant(double d, int E)
{
    const int hi = __double2hiint(d), ex = (hi >> 20) & 0x7ff, one = min(ex, 1);
    const unsigned mh = ((unsigned)hi & 0xfffffu) | ((unsigned)one << 20);
    const unsigned long long m = (((unsigned long long)mh << 32) | (unsigned)__double2loint(d)) << (UP + ROUND);
    const unsigned long long t = m >> fx_clamp63(E - 1 - ex + one);
    return ROUND ? (t + 1) >> 1 : t;
}
__device__ __forceinline__ fx2 fx_limbs(double d, int E)
{
    const int sg = (__double2hiint(d) >> 31) | 1;
    const fx2 v = fx_split((long long)fx_mant<FX_VBITS - 53, false>(d, E));
    return {v.h * sg, v.l * sg};
}
// the same as one signed integer in units of 2^(E - 1023 - 54), rounded to nearest or
// cut, |t| <= 2^55 (for operands stored with balanced limbs)
template <bool ROUND>
__device__ __forceinline__ long long fx_int(double d, int E)
{
    const long long m = (long long)fx_mant<2, ROUND>(d, E);
    return __double2hiint(d) < 0 ? -m : m;
}
// the same for a float pair: field of the leading float, widened
__device__ __forceinline__ int fx_field(df d)
{
    const int ex = (__float_as_int(d.hi) >> 23) & 0xff;
    return ex == 0xff ? 0x7ff : ex + 896;
}
__device__ __forceinline__ long long fx_float(float f, int E)  // E >= 897
{
    // (denormals by way of 2^24 f: with the mantissa masked as above, the batched
    // kernels spilled more, 106.7 -> 108.6 ms for 48 problems)
    const bool tiny = fabsf(f) < 1.17549435e-38f;
    const int b = __float_as_int(tiny ? f * 16777216.f : f), ex = (b >> 23) & 0xff;
    const long long m = (long long)((b & 0x7fffff) | 0x800000) << (FX_VBITS - 24);
    const long long t = m >> (ex ? fx_clamp63(E - 896 - ex + (tiny ? 24 : 0)) : 63);
    return b < 0 ? -t : t;
}
__device__ __forceinline__ fx2 fx_limbs(df d, int E) { return fx_split(fx_float(d.hi, E) + fx_float(d.lo, E)); }
// the least E of an arithmetic type
template <class T>
constexpr int FX_FIELD_MIN = std::is_same<T, df>::value ? 897 : 1;

// a spinor in FP64 or DF64 arithmetic as limbs; returns its unit exponent
template <class T>
__device__ __forceinline__ int fx_from_spinor(const Spinor<T> &p, Spinor<fx2> &o)
{
    int E = FX_FIELD_MIN<T>;
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int i = 0; i < 3; ++i) E = max(E, max(fx_field(p.s[a][i].r), fx_field(p.s[a][i].i)));
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int i = 0; i < 3; ++i) o.s[a][i] = cx<fx2>{fx_limbs(p.s[a][i].r, E), fx_limbs(p.s[a][i].i, E)};
    return E == 0x7ff ? FX_NAN : E - (1023 + FX_VBITS - 1);
}

__device__ __forceinline__ double fx_pow2(int e)  // 2^e; the caller keeps e in the normal range
{
    return __longlong_as_double((long long)(1023 + e) << 52);
}

// ---------------------------------------------------------------- fields
// A fixed-point spinor field, the operators' input: 12 int4 (re h, re l, im h,
// im l) per site in the site-blocked order, and one unit exponent per site in
// the place of the FP16 norms.

__device__ __forceinline__ void fx_store(const SpinorPtr &v, int cb, const Spinor<fx2> &s, int e)
{
    int4 *p = (int4 *)v.p;
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        const cx<fx2> z = s.s[k / 3][k % 3];
        p[soa(cb, 12, k)] = make_int4(z.r.h, z.r.l, z.i.h, z.i.l);
    }
    ((int *)v.norm)[cb] = e;
}

template <>  // written by conversions only; the operators load it themselves (stencil_fx.cuh)
struct Prec<QCD_FX> {
    using T = double;
    static constexpr int SP_NC = 12;
    static __device__ __forceinline__ void store(const SpinorPtr &v, int cb, const Spinor<T> &s)
    {
        Spinor<fx2> o;
        const int e = fx_from_spinor(s, o);
        fx_store(v, cb, o, e);
    }
};

}  // namespace qcd
