// The hopping term and the clover term for FP64 and DF64 in fixed point
// (fx.cuh), two threads a site: lane 16 a + s of a warp takes spin row a of the
// projected half spinors of site s, and the chiral block a of the clover term.
//
// A thread multiplies one colour vector by the link of each hop (both rows
// share every link word: the two lanes read the same address) and gathers the
// upper spin a and the lower spins its row feeds; one exchange between the two
// lanes leaves it with the spins a and 2 + a of the result.  The clover blocks
// need both rows of one chirality: one exchange before the 6x6 product, one
// after.  The raw words of hop d + 1 (15 of 16 bytes) are loaded before hop d is
// computed: 168 registers, twelve warps an SM in blocks of 128 threads.  MULT at
// 24^3x48, L2 evicted: 175 us (DRAM traffic 0.68 GB, 100 us of HBM time).  Without
// the hop in flight the kernels waited on one chain of loads after the other,
// whatever the occupancy: 265 us at 128 registers, 270 at 80; one thread a site
// 260 us at 168 registers, 290 at 128, 287 with the words staged by cp.async.
//
// The integer accumulators stay below 2^63: a projected pair is below 2^58, a
// link of Frobenius norm sqrt(3) takes it to 2^59.2 in the result's units, eight
// hops to 2^62.2; clover sums (twelve products of limbs 2^27 x 2^30) to 2^61.6.
#pragma once

#include "stencil.cuh"

namespace qcd {

// the two spins a and 2 + a that a thread holds of a spinor
template <class T>
struct HalfSp {
    cx<T> u[3], d[3];
};

__device__ __forceinline__ int fx_row() { return (threadIdx.x >> 4) & 1; }
// the site of this thread among the blockDim.x / 2 of its block
__device__ __forceinline__ int fx_site() { return (int)((threadIdx.x >> 5) << 4) + (int)(threadIdx.x & 15); }

__device__ __forceinline__ long long fx_swap(long long v) { return __shfl_xor_sync(0xffffffffu, v, 16); }
__device__ __forceinline__ int fx_swap(int v) { return __shfl_xor_sync(0xffffffffu, v, 16); }
__device__ __forceinline__ cx<long long> fx_swap(cx<long long> v) { return mk(fx_swap(v.r), fx_swap(v.i)); }
__device__ __forceinline__ fx2 fx_swap(fx2 v) { return fx2{fx_swap(v.h), fx_swap(v.l)}; }

// component index of (spin a or 2 + a, colour i)
__device__ __forceinline__ int fx_comp(int a, int lower, int i) { return 6 * lower + 3 * a + i; }

// ---- loads and stores of a thread's half -------------------------------------
template <int P>
__device__ __forceinline__ void load_half(const SpinorPtr &v, int cb, int a, HalfSp<typename Prec<P>::T> &o)
{
    constexpr bool COH = P >= COHERENT;
    constexpr int B = COH ? P - COHERENT : P;
    static_assert(B == QCD_F64 || B == QCD_DF64, "FP64-sized vectors");
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        const size_t at = soa(cb, 12, fx_comp(a, j / 3, j % 3));
        cx<typename Prec<P>::T> z;
        if constexpr (B == QCD_F64) {
            const double2 *p = (const double2 *)v.p + at;
            const double2 q = COH ? __ldcg(p) : __ldg(p);
            z = mk(q.x, q.y);
        } else {
            const float4 *p = (const float4 *)v.p + at;
            z = f4c(COH ? __ldcg(p) : __ldg(p));
        }
        (j < 3 ? o.u[j] : o.d[j - 3]) = z;
    }
}
template <int P>
__device__ __forceinline__ void store_half(const SpinorPtr &v, int cb, int a, const HalfSp<typename Prec<P>::T> &o)
{
    constexpr int B = P >= COHERENT ? P - COHERENT : P;
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        const size_t at = soa(cb, 12, fx_comp(a, j / 3, j % 3));
        const auto z = j < 3 ? o.u[j] : o.d[j - 3];
        if constexpr (B == QCD_F64) ((double2 *)v.p)[at] = make_double2(z.r, z.i);
        else ((float4 *)v.p)[at] = c4f(z);
    }
}

// ---- conversions ------------------------------------------------------------
// both threads of a site agree on its exponent
template <class T>
__device__ __forceinline__ int fx_from_half(const HalfSp<T> &p, HalfSp<fx2> &o)
{
    int E = FX_FIELD_MIN<T>;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        E = max(E, max(fx_field(p.u[i].r), fx_field(p.u[i].i)));
        E = max(E, max(fx_field(p.d[i].r), fx_field(p.d[i].i)));
    }
    E = max(E, fx_swap(E));
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        o.u[i] = cx<fx2>{fx_limbs(p.u[i].r, E), fx_limbs(p.u[i].i, E)};
        o.d[i] = cx<fx2>{fx_limbs(p.d[i].r, E), fx_limbs(p.d[i].i, E)};
    }
    return E == 0x7ff ? FX_NAN : E - (1023 + FX_VBITS - 1);
}

// v scaled below 2^57; e follows
__device__ __forceinline__ void fx_normalise(HalfSp<long long> &v, int &e)
{
    unsigned mh = 0, ml = 0;
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        const cx<long long> z = j < 3 ? v.u[j] : v.d[j - 3];
        const long long c[2] = {z.r, z.i};
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const unsigned h = (unsigned)((unsigned long long)c[k] >> 32), s = (unsigned)((int)h >> 31);
            mh |= h ^ s;
            ml |= (unsigned)c[k] ^ s;
        }
    }
    mh |= (unsigned)fx_swap((int)mh);
    ml |= (unsigned)fx_swap((int)ml);
    const int lz = mh ? __clz(mh) : 32 + min(__clz(ml), 31);
    const int up = lz - 1;  // the largest to 2^62 or more, then six bits down
    constexpr int DN = 63 - FX_VBITS;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        v.u[i] = mk((v.u[i].r << up) >> DN, (v.u[i].i << up) >> DN);
        v.d[i] = mk((v.d[i].r << up) >> DN, (v.d[i].i << up) >> DN);
    }
    if (e > FX_ZERO / 2 && e < FX_NAN / 2) e += DN - up;
}
__device__ __forceinline__ void fx_split(const HalfSp<long long> &v, HalfSp<fx2> &o)
{
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        o.u[i] = cx<fx2>{fx_split(v.u[i].r), fx_split(v.u[i].i)};
        o.d[i] = cx<fx2>{fx_split(v.d[i].r), fx_split(v.d[i].i)};
    }
}

__device__ __forceinline__ void fx_store_half(const SpinorPtr &v, int cb, int a, const HalfSp<fx2> &s, int e)
{
    int4 *p = (int4 *)v.p;
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        const cx<fx2> z = j < 3 ? s.u[j] : s.d[j - 3];
        p[soa(cb, 12, fx_comp(a, j / 3, j % 3))] = make_int4(z.r.h, z.r.l, z.i.h, z.i.l);
    }
    if (a == 0) ((int *)v.norm)[cb] = e;
}

// v 2^e in the arithmetic type T (v is scratch)
template <class T>
__device__ __forceinline__ void fx_to_half(HalfSp<long long> &v, int e, HalfSp<T> &o)
{
    auto each = [&](auto f) {
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            o.u[i] = mk(f(v.u[i].r), f(v.u[i].i));
            o.d[i] = mk(f(v.d[i].r), f(v.d[i].i));
        }
    };
    if constexpr (std::is_same<T, df>::value) {
        // float pairs without the FP64 pipe: the site scaled to 57 bits, the top
        // 24 exactly and the next 31 rounded to a float
        fx_normalise(v, e);
        const int es = e + FX_VBITS - 24;
        if (es > -100 && es < 100) {
            const float s = __int_as_float((127 + es) << 23), s31 = 4.656612873077392578125e-10f * s;  // 2^-31 s
            each([&](long long x) {
                return fast_two_sum((float)(int)(x >> (FX_VBITS - 24)) * s,
                                    (float)((int)(x >> (FX_VBITS - 55)) & 0x7fffffff) * s31);
            });
            return;
        }
    }
    if (e >= FX_NAN / 2) {
        each([&](long long) { return T(__longlong_as_double(0x7ff8000000000000ll)); });
    } else if (e >= -1000) {
        const double s = fx_pow2(e);
        each([&](long long x) { return T((double)x * s); });
    } else {  // below the normal range (sites under 2^-900) in two steps
        const double s1 = fx_pow2(-1000), s2 = e < -2000 ? 0.0 : fx_pow2(e + 1000);
        each([&](long long x) { return T((double)x * s1 * s2); });
    }
}

// the half of a fixed-point field in T
template <class T>
__device__ __forceinline__ void fx_load_half(const SpinorPtr &v, int cb, int a, HalfSp<T> &o)
{
    const int4 *p = (const int4 *)v.p;
    HalfSp<long long> t;
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        const int4 q = __ldg(p + soa(cb, 12, fx_comp(a, j / 3, j % 3)));
        (j < 3 ? t.u[j] : t.d[j - 3]) = mk(((long long)q.x << FX_LIMB) + q.y, ((long long)q.z << FX_LIMB) + q.w);
    }
    fx_to_half(t, __ldg((const int *)v.norm + cb), o);
}

// ---- hops ---------------------------------------------------------------------
// The raw words of hop D = 2 mu + backward (S the sign of its projector): the
// one or two spins the thread's row is projected from, and the link
struct FxRaw {
    int4 s[6], l[9];
};
template <int D, int S, bool COH>
__device__ __forceinline__ void fx_row_load(const GaugePtr &U, const SpinorPtr &in, int out_par, int cb, int nb, int a,
                                            FxRaw &R)
{
    constexpr int MU = D >> 1;
    constexpr bool BWD = D & 1;
    const int4 *own = (const int4 *)in.p + soa(nb, 12, 0) + a * 3 * SB;
    const int4 *opp = (const int4 *)in.p + soa(nb, 12, 9) - a * 3 * SB;
    auto ld = [](const int4 *p) { return COH ? __ldcg(p) : __ldg(p); };
    const int4 *lp = (const int4 *)U.a[BWD ? 1 - out_par : out_par] + soa(BWD ? nb : cb, 36, MU * 9);
#pragma unroll
    for (int k = 0; k < 9; ++k) R.l[k] = ld_stream(lp + k * SB);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        if constexpr (MU == 3) {
            R.s[i] = ld(own + ((S > 0 ? 6 : 0) + i) * SB);
        } else {
            R.s[i] = ld(own + i * SB);
            R.s[3 + i] = MU == 2 ? ld(own + (6 + i) * SB) : ld(opp + i * SB);
        }
    }
}

// The thread's row q of U h, in units of 2^(E - 55 + 56), sh = E - the
// neighbour's exponent.  Row a: h = p_a + S i p_3-a (x), p_a + S sa p_3-a (y),
// p_a + S i sa p_2+a (z), p_2+a or p_a (t), sa = +1 for a = 0, -1 for a = 1.
template <int D, int S>
__device__ __forceinline__ void fx_row_mul(const FxRaw &R, int sa, bool flip, int sh, cx<long long> q[3])
{
    constexpr int MU = D >> 1;
    constexpr bool BWD = D & 1;
    cx<fx2> h[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const int4 v = R.s[i];
        const cx<fx2> p{fx2{v.x, v.y}, fx2{v.z, v.w}};
        if constexpr (MU == 3) {
            h[i] = p;
        } else {
            const int4 w = R.s[3 + i];
            const int s = MU == 0 ? 1 : sa;
            const cx<fx2> r{fx2{w.x * s, w.y * s}, fx2{w.z * s, w.w * s}};
            if (MU == 1) h[i] = S > 0 ? p + r : p - r;
            else h[i] = S > 0 ? p + ti(r) : p - ti(r);
        }
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        long long mr, mi, hr, hi;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            // U_ij, or conj(U_ji) for the backward hop
            const int4 u = R.l[BWD ? 3 * j + i : 3 * i + j];
            const int pih = BWD ? -u.z : u.z, pil = BWD ? -u.w : u.w, nih = BWD ? u.z : -u.z, nil = BWD ? u.w : -u.w;
            const cx<fx2> x = h[j];
            if (j == 0) {
                mr = fx_mul(u.x, x.r.l);
                mi = fx_mul(u.x, x.i.l);
                hr = fx_mul(u.x, x.r.h);
                hi = fx_mul(u.x, x.i.h);
            } else {
                fx_mac(mr, u.x, x.r.l);
                fx_mac(mi, u.x, x.i.l);
                fx_mac(hr, u.x, x.r.h);
                fx_mac(hi, u.x, x.i.h);
            }
            fx_mac(mr, u.y, x.r.h);
            fx_mac(mi, u.y, x.i.h);
            fx_mac(hr, nih, x.i.h);
            fx_mac(hi, pih, x.r.h);
            fx_mac(mr, nih, x.i.l);
            fx_mac(mi, pih, x.r.l);
            fx_mac(mr, nil, x.i.h);
            fx_mac(mi, pil, x.r.h);
        }
        q[i] = mk((hr + (mr >> FX_LIMB)) >> sh, (hi + (mi >> FX_LIMB)) >> sh);
        if (MU == 3 && flip) q[i] = -q[i];
    }
}

// acc 2^E = H in at site cb, this thread's spins a and 2 + a
template <bool DAG, bool COH>
__device__ __forceinline__ void fx_hopping(const Geom &g, const GaugePtr &U, const SpinorPtr &in, int out_par, int cb,
                                           int a, HalfSp<long long> &acc, int &E)
{
    int c[4];
    site_coords(g, out_par, cb, c);
    const int lex = lex_of(g, c);
    constexpr int SF = DAG ? -1 : 1;
    const int sa = a ? -1 : 1;
    auto nb = [&](int d) { return lex_hop(g, lex, c, d >> 1, (d & 1) ? -1 : +1) >> 1; };
    auto ex = [&](int d) { return COH ? __ldcg((const int *)in.norm + nb(d)) : __ldg((const int *)in.norm + nb(d)); };
    E = FX_ZERO;
#pragma unroll
    for (int d = 0; d < 8; ++d) E = max(E, ex(d));
    const bool up = g.t_bc < 0 && c[3] == g.L[3] - 1, dn = g.t_bc < 0 && c[3] == 0;
    cx<long long> q[3], X[3], Y[3];  // X: what row a adds to spin 3 - a; Y: to spin 2 + a
    FxRaw R0, R1;
#define QCD_FX_LOAD(D, S, R) fx_row_load<D, S, COH>(U, in, out_par, cb, nb(D), a, R)
#define QCD_FX_HOP(D, S, FLIP, R, DN, SN, RN)                           \
    QCD_FX_LOAD(DN, SN, RN);                                            \
    fx_row_mul<D, S>(R, sa, FLIP, fx_clamp63(E - ex(D)), q)
#define QCD_FX_LAST(D, S, FLIP, R) fx_row_mul<D, S>(R, sa, FLIP, fx_clamp63(E - ex(D)), q)
    QCD_FX_LOAD(2, SF, R0);
    // y: upper g, lower spin 3 - a gets S sa g (sa applied once to both hops)
    QCD_FX_HOP(2, SF, false, R0, 3, -SF, R1);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        acc.u[i] = q[i];
        X[i] = SF > 0 ? q[i] : -q[i];
    }
    QCD_FX_HOP(3, -SF, false, R1, 0, SF, R0);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        acc.u[i] = acc.u[i] + q[i];
        X[i] = SF > 0 ? X[i] - q[i] : X[i] + q[i];
        if (a) X[i] = -X[i];
    }
    // x: lower spin 3 - a gets -S i g
    QCD_FX_HOP(0, SF, false, R0, 1, -SF, R1);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        acc.u[i] = acc.u[i] + q[i];
        X[i] = SF > 0 ? X[i] - ti(q[i]) : X[i] + ti(q[i]);
    }
    QCD_FX_HOP(1, -SF, false, R1, 4, SF, R0);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        acc.u[i] = acc.u[i] + q[i];
        X[i] = SF > 0 ? X[i] + ti(q[i]) : X[i] - ti(q[i]);
    }
    // z: lower spin 2 + a gets -S i sa g
    QCD_FX_HOP(4, SF, false, R0, 5, -SF, R1);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        acc.u[i] = acc.u[i] + q[i];
        Y[i] = SF > 0 ? tmi(q[i]) : ti(q[i]);
    }
    QCD_FX_HOP(5, -SF, false, R1, 6, SF, R0);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        acc.u[i] = acc.u[i] + q[i];
        Y[i] = SF > 0 ? Y[i] + ti(q[i]) : Y[i] - ti(q[i]);
        if (a) Y[i] = -Y[i];
    }
    // t: the projector's factor 2 (see project); S > 0 the lower spin, S < 0 the upper
    QCD_FX_HOP(6, SF, up, R0, 7, -SF, R1);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        if (SF > 0) Y[i] = Y[i] + twice(q[i]);
        else acc.u[i] = acc.u[i] + twice(q[i]);
    }
    QCD_FX_LAST(7, -SF, dn, R1);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        if (SF > 0) acc.u[i] = acc.u[i] + twice(q[i]);
        else Y[i] = Y[i] + twice(q[i]);
        acc.d[i] = Y[i] + fx_swap(X[i]);  // the other row's share of spin 2 + a
    }
#undef QCD_FX_HOP
#undef QCD_FX_LOAD
#undef QCD_FX_LAST
    // links are in units of 2^-55, a product is cut by 2^56
    if (E > FX_ZERO / 2 && E < FX_NAN / 2) E += 2 * FX_LIMB - FX_BITS;
}

// ---- clover ---------------------------------------------------------------------
// out 2^e = the clover term of x 2^e (the site's two blocks have their unit
// exponents in C.e)
__device__ __forceinline__ void fx_clover(const CloverPtr &C, int par, int cb, int a, const HalfSp<fx2> &x, int &e,
                                          HalfSp<long long> &out)
{
    const int4 *p = (const int4 *)C.p[par] + soa(cb, 36, 0) + a * 18 * SB;
    const int e0 = __ldg(C.e[par] + 2 * cb), e1 = __ldg(C.e[par] + 2 * cb + 1), em = max(e0, e1);
    const int sh = fx_clamp63(em - (a ? e1 : e0));
    // chi_+ = up - dn (block 0), chi_- = up + dn (block 1), rows 0 and 1
    cx<fx2> v[6];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const cx<fx2> s = x.u[i] + x.d[i], d = x.u[i] - x.d[i];
        const cx<fx2> mine = a ? s : d, give = a ? d : s;
        const cx<fx2> got{fx_swap(give.r), fx_swap(give.i)};
        v[i] = a ? got : mine;
        v[3 + i] = a ? mine : got;
    }
    long long mr[6], mi[6], hr[6], hi[6];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int4 d = ld_stream(p + k * SB);
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const int i = 2 * k + b, dh = b ? d.z : d.x, dl = b ? d.w : d.y;
            mr[i] = fx_mul(dh, v[i].r.l);
            mi[i] = fx_mul(dh, v[i].i.l);
            hr[i] = fx_mul(dh, v[i].r.h);
            hi[i] = fx_mul(dh, v[i].i.h);
            fx_mac(mr[i], dl, v[i].r.h);
            fx_mac(mi[i], dl, v[i].i.h);
        }
    }
    int k = 0;
#pragma unroll
    for (int i = 1; i < 6; ++i)
#pragma unroll
        for (int j = 0; j < i; ++j) {
            const int4 o = ld_stream(p + (3 + k) * SB);
            const int nih = -o.z, nil = -o.w;
            // y_i += A_ij v_j
            fx_mac(mr[i], o.x, v[j].r.l);
            fx_mac(mr[i], o.y, v[j].r.h);
            fx_mac(mr[i], nih, v[j].i.l);
            fx_mac(mr[i], nil, v[j].i.h);
            fx_mac(mi[i], o.x, v[j].i.l);
            fx_mac(mi[i], o.y, v[j].i.h);
            fx_mac(mi[i], o.z, v[j].r.l);
            fx_mac(mi[i], o.w, v[j].r.h);
            fx_mac(hr[i], o.x, v[j].r.h);
            fx_mac(hr[i], nih, v[j].i.h);
            fx_mac(hi[i], o.x, v[j].i.h);
            fx_mac(hi[i], o.z, v[j].r.h);
            // y_j += conj(A_ij) v_i
            fx_mac(mr[j], o.x, v[i].r.l);
            fx_mac(mr[j], o.y, v[i].r.h);
            fx_mac(mr[j], o.z, v[i].i.l);
            fx_mac(mr[j], o.w, v[i].i.h);
            fx_mac(mi[j], o.x, v[i].i.l);
            fx_mac(mi[j], o.y, v[i].i.h);
            fx_mac(mi[j], nih, v[i].r.l);
            fx_mac(mi[j], nil, v[i].r.h);
            fx_mac(hr[j], o.x, v[i].r.h);
            fx_mac(hr[j], o.z, v[i].i.h);
            fx_mac(hi[j], o.x, v[i].i.h);
            fx_mac(hi[j], nih, v[i].r.h);
            ++k;
        }
    // up = (y+ + y-)/2, dn = (y- - y+)/2, the 1/2 in the exponent
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const cx<long long> y0 = mk((hr[i] + (mr[i] >> FX_LIMB)) >> sh, (hi[i] + (mi[i] >> FX_LIMB)) >> sh);
        const cx<long long> y1 =
            mk((hr[3 + i] + (mr[3 + i] >> FX_LIMB)) >> sh, (hi[3 + i] + (mi[3 + i] >> FX_LIMB)) >> sh);
        const cx<long long> mine = a ? y1 : y0, got = fx_swap(a ? y0 : y1);
        out.u[i] = mine + got;
        out.d[i] = a ? mine - got : got - mine;
    }
    if (e > FX_ZERO / 2 && e < FX_NAN / 2) e += em + 2 * FX_LIMB - 1;
}

// the clover term of a spinor in T's arithmetic, in place
template <class T>
__device__ __forceinline__ void fx_clover_half(const CloverPtr &C, int par, int cb, int a, HalfSp<T> &s)
{
    HalfSp<fx2> x;
    HalfSp<long long> y;
    int e = fx_from_half(s, x);
    fx_clover(C, par, cb, a, x, e, y);
    fx_to_half(y, e, s);
}

// acc 2^E = H in, or with CLOVER the clover term (F^-1, or what C holds) of it
template <bool DAG, bool CLOVER, bool COH>
__device__ __forceinline__ void fx_hop(const Geom &g, const GaugePtr &U, const CloverPtr &C, const SpinorPtr &in,
                                       int out_par, int cb, int a, HalfSp<long long> &acc, int &E)
{
    fx_hopping<DAG, COH>(g, U, in, out_par, cb, a, acc, E);
    if constexpr (CLOVER) {
        HalfSp<fx2> x;
        fx_normalise(acc, E);
        fx_split(acc, x);
        fx_clover(C, out_par, cb, a, x, E, acc);
    }
}

// ---- sums over a thread's half ---------------------------------------------------
// o = s x + t y
template <class T>
__device__ __forceinline__ void axpby_half(HalfSp<T> &o, T s, const HalfSp<T> &x, T t, const HalfSp<T> &y)
{
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        o.u[i] = mk(s * x.u[i].r + t * y.u[i].r, s * x.u[i].i + t * y.u[i].i);
        o.d[i] = mk(s * x.d[i].r + t * y.d[i].r, s * x.d[i].i + t * y.d[i].i);
    }
}
// re + i im += <x|y>
template <class T>
__device__ __forceinline__ void dot_half(const HalfSp<T> &x, const HalfSp<T> &y, double &re, double &im)
{
    T r = 0, m = 0;
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        const cx<T> a = j < 3 ? x.u[j] : x.d[j - 3], b = j < 3 ? y.u[j] : y.d[j - 3];
        r += a.r * b.r + a.i * b.i;
        m += a.r * b.i - a.i * b.r;
    }
    re += to_d(r);
    im += to_d(m);
}
template <class T>
__device__ __forceinline__ void norm_half(const HalfSp<T> &x, double &n)
{
    T s = 0;
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        const cx<T> a = j < 3 ? x.u[j] : x.d[j - 3];
        s += a.r * a.r + a.i * a.i;
    }
    n += to_d(s);
}

}  // namespace qcd
