// Adjoint pieces: lambda = D^-dag g through gamma5-hermiticity
// (D^dag = gamma5 D gamma5, so D^-dag = gamma5 D^-1 gamma5), and the link
// gradient ("force") of f(U) = -Re<lambda, D[U] x> for fixed x, lambda, in the
// convention G = df/dRe U + i df/dIm U.  With x = D^-1 b and lambda = D^-dag g,
// -Re<lambda, dD x> is the change of Re<g, x>, so G is the gradient of a loss
// whose gradient with respect to x is g.
//
// Hopping part (Eq. 4): U_mu(m) enters (1 - g_mu) U_mu(m) x(m+mu) at m and
// (1 + g_mu) U_mu(m)^dag x(m) at m+mu; with bc the boundary phase,
//   G_mu(m) += kappa bc [ sum_s ((1-g_mu) lambda(m))_s (x) conj(x_s(m+mu))
//                       + sum_s x_s(m) (x) conj(((1+g_mu) lambda(m+mu))_s) ].
// Clover part: f_clov = csw kappa Re sum_n sum_{mu<nu} Tr(S^T F_munu), with
// S_ij = sum_ab conj(lambda_ai) sigma_munu,ab x_bj; since F = (Q - Q^dag)/(8i),
// this is Re sum Tr(Y Q) with Y = csw kappa (S^T + conj(S))/(8i).  Every
// plaquette of Q enters at its four corners, so the derivative with respect
// to one link collects the two plaquettes of each plane through it with Y
// inserted at each corner (a staple with insertions).
#include "blas.cuh"
#include "stencil.cuh"

namespace qcd {

namespace {

using C = cx<double>;

struct M3 {
    C m[3][3];
};

__device__ __forceinline__ M3 zero3()
{
    M3 r;
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j) r.m[i][j] = mk(0.0, 0.0);
    return r;
}

__device__ __forceinline__ M3 mul(const M3 &a, const M3 &b)
{
    M3 c;
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j) {
            C s = mk(0.0, 0.0);
            for (int k = 0; k < 3; ++k) fma_(s, a.m[i][k], b.m[k][j]);
            c.m[i][j] = s;
        }
    return c;
}

__device__ __forceinline__ M3 dagm(const M3 &a)
{
    M3 c;
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j) c.m[i][j] = conj(a.m[j][i]);
    return c;
}

__device__ __forceinline__ void addm(M3 &a, const M3 &b)
{
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j) a.m[i][j] = a.m[i][j] + b.m[i][j];
}

// canonical links [V][4][3][3] complex128
__device__ __forceinline__ M3 link(const double2 *U, int s, int mu)
{
    M3 r;
    const double2 *p = U + ((size_t)s * 4 + mu) * 9;
    for (int k = 0; k < 9; ++k) r.m[k / 3][k % 3] = mk(p[k].x, p[k].y);
    return r;
}

__device__ __forceinline__ int site_shift(const Geom &g, int s, int mu, int d)
{
    int c[4], t = s;
    for (int k = 0; k < 4; ++k) {
        c[k] = t % g.L[k];
        t /= g.L[k];
    }
    c[mu] = (c[mu] + d + g.L[mu]) % g.L[mu];
    return lex_of(g, c);
}

__device__ __forceinline__ void load_spinor(const double2 *v, int s, C out[4][3])
{
    const double2 *p = v + (size_t)s * 12;
    for (int k = 0; k < 12; ++k) out[k / 3][k % 3] = mk(p[k].x, p[k].y);
}

// (1 - sg * gamma_mu) v in the Dirac basis
__device__ void one_minus_gamma(const C v[4][3], int mu, int sg, C o[4][3])
{
    for (int i = 0; i < 3; ++i) {
        C g0, g1, g2, g3;  // gamma_mu v
        if (mu == 0) {
            g0 = tmi(v[3][i]); g1 = tmi(v[2][i]); g2 = ti(v[1][i]); g3 = ti(v[0][i]);
        } else if (mu == 1) {
            g0 = -v[3][i]; g1 = v[2][i]; g2 = v[1][i]; g3 = -v[0][i];
        } else if (mu == 2) {
            g0 = tmi(v[2][i]); g1 = ti(v[3][i]); g2 = ti(v[0][i]); g3 = tmi(v[1][i]);
        } else {
            g0 = v[0][i]; g1 = v[1][i]; g2 = -v[2][i]; g3 = -v[3][i];
        }
        const double s = (double)sg;
        o[0][i] = v[0][i] - s * g0;
        o[1][i] = v[1][i] - s * g1;
        o[2][i] = v[2][i] - s * g2;
        o[3][i] = v[3][i] - s * g3;
    }
}

// sigma_munu for the six planes (mu < nu) in the order (x,y) (x,z) (x,t)
// (y,z) (y,t) (z,t): each row has one non-zero entry, a phase:
// (sigma v)_a = phase[a] * v[perm[a]].  Worked out from
// sigma_jk = -eps_jkl diag(s_l, s_l) and sigma_k4 = [[0, -s_k], [-s_k, 0]].
__constant__ int c_sig_perm[6][4] = {
    {0, 1, 2, 3}, {1, 0, 3, 2}, {3, 2, 1, 0}, {1, 0, 3, 2}, {3, 2, 1, 0}, {2, 3, 0, 1}};
// phases as (re, im)
__constant__ double c_sig_ph[6][4][2] = {
    {{-1, 0}, {1, 0}, {-1, 0}, {1, 0}},     // sigma_xy = -diag(s3, s3)
    {{0, -1}, {0, 1}, {0, -1}, {0, 1}},     // sigma_xz = +diag(s2, s2)
    {{-1, 0}, {-1, 0}, {-1, 0}, {-1, 0}},   // sigma_xt = [[0,-s1],[-s1,0]]
    {{-1, 0}, {-1, 0}, {-1, 0}, {-1, 0}},   // sigma_yz = -diag(s1, s1)
    {{0, 1}, {0, -1}, {0, 1}, {0, -1}},     // sigma_yt = [[0,-s2],[-s2,0]]
    {{-1, 0}, {1, 0}, {-1, 0}, {1, 0}}};    // sigma_zt = [[0,-s3],[-s3,0]]

__device__ __forceinline__ int plane_index(int mu, int nu)
{
    // mu < nu
    return mu == 0 ? nu - 1 : (mu == 1 ? nu + 1 : 5);
}

// Y_p(n) = csw kappa (S^T + conj(S)) / (8i) for the six planes
__device__ __forceinline__ void force_Y_site(const Geom &g, const double2 *__restrict__ x,
                                             const double2 *__restrict__ lam, double ck, double2 *Y, int s)
{
    C X[4][3], L[4][3];
    load_spinor(x, s, X);
    load_spinor(lam, s, L);
    for (int p = 0; p < 6; ++p) {
        C S[3][3];
        for (int i = 0; i < 3; ++i)
            for (int j = 0; j < 3; ++j) {
                C acc = mk(0.0, 0.0);
                for (int a = 0; a < 4; ++a) {
                    const C ph = mk(c_sig_ph[p][a][0], c_sig_ph[p][a][1]);
                    const C sx = ph * X[c_sig_perm[p][a]][j];
                    fmac_(acc, L[a][i], sx);  // conj(lambda_ai) (sigma x)_aj
                }
                S[i][j] = acc;
            }
        double2 *out = Y + ((size_t)s * 6 + p) * 9;
        for (int i = 0; i < 3; ++i)
            for (int j = 0; j < 3; ++j) {
                const C t = S[j][i] + conj(S[i][j]);
                const C y = (ck * 0.125) * tmi(t);  // t / (8i)
                out[i * 3 + j] = make_double2(y.r, y.i);
            }
    }
}

// Y of the ordered plane (mu, nu), mu != nu, at site s: for mu > nu the loop
// runs the other way round, which is the same as inserting Y_{nu mu}^dag.
__device__ __forceinline__ M3 Yeff(const double2 *Y, int s, int mu, int nu)
{
    M3 r;
    const bool fwd = mu < nu;
    const int p = fwd ? plane_index(mu, nu) : plane_index(nu, mu);
    const double2 *q = Y + ((size_t)s * 6 + p) * 9;
    for (int k = 0; k < 9; ++k) r.m[k / 3][k % 3] = mk(q[k].x, q[k].y);
    return fwd ? r : dagm(r);
}

__device__ __forceinline__ void force_link_one(const Geom &g, const double2 *__restrict__ U,
                                               const double2 *__restrict__ x, const double2 *__restrict__ lam,
                                               const double2 *__restrict__ Y, double kappa, int with_clover, double2 *G,
                                               int tid)
{
    const int m = tid >> 2, mu = tid & 3;
    const int mp = site_shift(g, m, mu, +1);
    M3 Gm = zero3();
    // ---- hopping part
    {
        int c[4], t = m;
        for (int k = 0; k < 4; ++k) {
            c[k] = t % g.L[k];
            t /= g.L[k];
        }
        const double bc = (mu == 3 && c[3] == g.L[3] - 1) ? (double)g.t_bc : 1.0;
        C Lm[4][3], Xp[4][3], Xm[4][3], Lp[4][3], PL[4][3], QL[4][3];
        load_spinor(lam, m, Lm);
        load_spinor(x, mp, Xp);
        load_spinor(x, m, Xm);
        load_spinor(lam, mp, Lp);
        one_minus_gamma(Lm, mu, +1, PL);  // (1 - g_mu) lambda(m)
        one_minus_gamma(Lp, mu, -1, QL);  // (1 + g_mu) lambda(m+mu)
        const double f = kappa * bc;
        for (int i = 0; i < 3; ++i)
            for (int j = 0; j < 3; ++j) {
                C acc = mk(0.0, 0.0);
                for (int s = 0; s < 4; ++s) {
                    fmac_(acc, Xp[s][j], PL[s][i]);  // PL_si conj(Xp_sj)
                    fmac_(acc, QL[s][j], Xm[s][i]);  // Xm_si conj(QL_sj)
                }
                Gm.m[i][j] = f * acc;
            }
    }
    // ---- clover part: the two plaquettes of each plane (mu, nu) through U_mu(m)
    if (with_clover) {
        for (int nu = 0; nu < 4; ++nu) {
            if (nu == mu) continue;
            {  // above: corners m, m+mu, m+mu+nu, m+nu
                const int mn = site_shift(g, m, nu, +1);
                const int mpn = site_shift(g, mp, nu, +1);
                const M3 Unu_mp = link(U, mp, nu), Umu_mn_d = dagm(link(U, mn, mu)), Unu_m_d = dagm(link(U, m, nu));
                const M3 W = mul(Unu_mp, Umu_mn_d);  // U_nu(m+mu) U_mu(m+nu)^dag
                const M3 A = mul(W, Unu_m_d);
                M3 R = mul(A, Yeff(Y, m, mu, nu));
                addm(R, mul(Yeff(Y, mp, mu, nu), A));
                addm(R, mul(mul(Unu_mp, Yeff(Y, mpn, mu, nu)), mul(Umu_mn_d, Unu_m_d)));
                addm(R, mul(mul(W, Yeff(Y, mn, mu, nu)), Unu_m_d));
                addm(Gm, dagm(R));  // U_mu(m) enters undaggered: G += R^dag
            }
            {  // below: corners m-nu, m-nu+mu, m+mu, m
                const int q = site_shift(g, m, nu, -1);
                const int qp = site_shift(g, q, mu, +1);
                const M3 Unu_q_d = dagm(link(U, q, nu)), Umu_q = link(U, q, mu), Unu_qp = link(U, qp, nu);
                const M3 V = mul(Unu_q_d, Umu_q);  // U_nu(q)^dag U_mu(q)
                const M3 B = mul(V, Unu_qp);
                M3 R = mul(mul(Unu_q_d, Yeff(Y, q, mu, nu)), mul(Umu_q, Unu_qp));
                addm(R, mul(mul(V, Yeff(Y, qp, mu, nu)), Unu_qp));
                addm(R, mul(B, Yeff(Y, mp, mu, nu)));
                addm(R, mul(Yeff(Y, m, mu, nu), B));
                addm(Gm, R);  // U_mu(m) enters daggered: G += R
            }
        }
    }
    double2 *out = G + (size_t)tid * 9;
    for (int k = 0; k < 9; ++k) out[k] = make_double2(Gm.m[k / 3][k % 3].r, Gm.m[k / 3][k % 3].i);
}

// run != NULL: nothing to do unless *run is set (any grid covers all sites)
__global__ void k_force_Y(Geom g, const double2 *__restrict__ x, const double2 *__restrict__ lam, double ck, double2 *Y,
                          const int *run)
{
    if (run && !*run) return;
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < g.V; s += gridDim.x * blockDim.x)
        force_Y_site(g, x, lam, ck, Y, s);
}
__global__ void k_force_link(Geom g, const double2 *__restrict__ U, const double2 *__restrict__ x,
                             const double2 *__restrict__ lam, const double2 *__restrict__ Y, double kappa,
                             int with_clover, double2 *G, const int *run)
{
    if (run && !*run) return;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < 4 * g.V; t += gridDim.x * blockDim.x)
        force_link_one(g, U, x, lam, Y, kappa, with_clover, G, t);
}

// ---------------------------------------------------------------- fixed-point form
// For links within the fixed-point range (fx.cuh) the clover part runs on the
// integer pipe, with fewer products.  Y is anti-Hermitian, so with
//   Z_nu(n) = U_nu(n) Y(n+nu) + Y(n) U_nu(n)   (one per direction and plane)
// the four insertions into each of a link's two plaquettes in a plane pair up:
//   G_mu(m) += +-[ U_nu(m) (U_mu(m+nu) Z_nu(m+mu)^dag) - Z_nu(m) (U_mu(m+nu) U_nu(m+mu)^dag)
//                - Z_nu(q)^dag (U_mu(q) U_nu(q+mu)) + U_nu(q)^dag (U_mu(q) Z_nu(q+mu)) ],
// q = m - nu, + for mu < nu: 8 products a plane instead of 18, and 24 a site for
// Z.  The hopping part keeps FP64 and uses the projector's rank: with h the
// two projected spin rows, sum_s ((1-g)lambda)_s conj(x_s) = sum_a h_a(lambda)
// conj(h_a(x)).  16^3x32: 8.4 ms before, 1.27 ms now (the caller's links
// into fixed point 0.03, Y 0.19, Z 0.20, links 0.84, issue-bound at half a slot
// per cycle).

// (sigma_p v)_a = ph v[perm]: ph as a power of i (the tables above)
__device__ constexpr int sig_perm(int p, int a)
{
    return p == 0 ? a : p == 1 || p == 3 ? a ^ 1 : p == 5 ? a ^ 2 : 3 - a;
}
__device__ constexpr int sig_pow(int p, int a)  // 0: 1, 1: i, 2: -1, 3: -i
{
    return p == 0 || p == 5 ? ((a & 1) ? 0 : 2) : p == 1 ? ((a & 1) ? 1 : 3) : p == 4 ? ((a & 1) ? 3 : 1) : 2;
}

// Y of plane P at a site: (imaginary diagonal 0..2, then (re, im) of (1,0), (2,0),
// (2,1)), anti-Hermitian: [plane][9][2][Vh_pad] by parity
template <int P>
__device__ __forceinline__ void force_y_plane(const Geom &g, const Spinor<double> &X, const Spinor<double> &L, double f,
                                              double *out, size_t stride)
{
    C S[3][3];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            C acc = mk(0.0, 0.0);
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                const C v = X.s[sig_perm(P, a)][j];
                const int ph = sig_pow(P, a);
                fmac_(acc, L.s[a][i], ph == 0 ? v : ph == 1 ? ti(v) : ph == 2 ? -v : tmi(v));
            }
            S[i][j] = acc;
        }
    // y_ij = -i f (S_ji + conj(S_ij))
#pragma unroll
    for (int i = 0; i < 3; ++i) out[i * stride] = -2.0 * f * S[i][i].r;
#pragma unroll
    for (int i = 1; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < i; ++j) {
            const C t = S[j][i] + conj(S[i][j]);
            const int k = 3 + 2 * (i + j - 1);
            out[k * stride] = f * t.i;
            out[(k + 1) * stride] = -f * t.r;
        }
}

// The caller's links in fixed point; *wide is set if one is out of range
// (thread = link in the caller's order: a warp reads 4.6 KB in a row)
__global__ void __launch_bounds__(128) k_force_Ux(Geom g, const double2 *__restrict__ U, int4 *Ue, int4 *Uo, int *wide)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x, s = t >> 2;
    if (s >= g.V) return;
    int par = 0, q = s;
    for (int k = 0; k < 4; ++k) {
        par ^= (q % g.L[k]) & 1;
        q /= g.L[k];
    }
    double2 m[9];
    for (int k = 0; k < 9; ++k) m[k] = __ldg(U + (size_t)t * 9 + k);
    if (fx_store_link(m, par ? Uo : Ue, s >> 1, t & 3)) *wide = 1;
}

__global__ void __launch_bounds__(128) k_force_Yx(Geom g, const double2 *__restrict__ x, const double2 *__restrict__ lam,
                                                  double f, double *Y, const int *wide)
{
    const int cb = blockIdx.x * blockDim.x + threadIdx.x, par = blockIdx.y;
    if (cb >= g.Vh || *wide) return;
    int c[4];
    site_coords(g, par, cb, c);
    const int s = lex_of(g, c);
    Spinor<double> X, L;
    load_spinor(x, s, X.s);
    load_spinor(lam, s, L.s);
    const size_t st = 2 * (size_t)g.Vh_pad;
    double *o = Y + (size_t)par * g.Vh_pad + cb;
    force_y_plane<0>(g, X, L, f, o, st);
    force_y_plane<1>(g, X, L, f, o + 9 * st, st);
    force_y_plane<2>(g, X, L, f, o + 18 * st, st);
    force_y_plane<3>(g, X, L, f, o + 27 * st, st);
    force_y_plane<4>(g, X, L, f, o + 36 * st, st);
    force_y_plane<5>(g, X, L, f, o + 45 * st, st);
}

// a link, or a Z matrix, of the fixed-point fields (nc int4 a site, the matrix
// at k0), daggered on loading
__device__ __forceinline__ void load_m3x(const int4 *p, int cb, int nc, int k0, bool dg, M3x &r)
{
    const int sg = dg ? -1 : 1;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const int4 v = __ldg(p + soa(cb, nc, k0 + (dg ? 3 * j + i : 3 * i + j)));
            r.m[i][j] = fxc{v.x, v.y, v.z * sg, v.w * sg};
        }
}

// cb of the site c + a + b (unit steps, +-mu): every index of one parity
__device__ __forceinline__ int cb_step(const Geom &g, const int c[4], int mu, int dm, int nu, int dn)
{
    int lex = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        int v = c[k] + (k == mu ? dm : 0) + (k == nu ? dn : 0);
        v = v < 0 ? v + g.L[k] : v >= g.L[k] ? v - g.L[k] : v;
        lex += v * g.st[k];
    }
    return lex >> 1;
}

// direction nu's Z of the plane it spans with mu: index 3 nu + (mu without nu)
__device__ __forceinline__ int z_index(int nu, int mu) { return 3 * nu + (mu < nu ? mu : mu - 1); }

struct ForceZ {
    int4 *z[2];  // [parity]: 12 matrices a site
    int *e;      // unit exponents [12][2][Vh_pad]
};

__global__ void __launch_bounds__(128, 3) k_force_Z(Geom g, GaugePtr U, const double *__restrict__ Y, ForceZ Z,
                                                    const int *wide)
{
    const int cb = blockIdx.x * blockDim.x + threadIdx.x, zi = blockIdx.y, par = blockIdx.z;
    if (cb >= g.Vh || *wide) return;
    const int nu = zi / 3, k3 = zi - 3 * nu, mu = k3 < nu ? k3 : k3 + 1;
    const int plane = mu < nu ? plane_index(mu, nu) : plane_index(nu, mu);
    int c[4];
    site_coords(g, par, cb, c);
    const int up = cb_step(g, c, nu, 1, nu, 0);
    const size_t st = 2 * (size_t)g.Vh_pad;
    const double *y0 = Y + (size_t)plane * 9 * st + (size_t)par * g.Vh_pad + cb;
    const double *y1 = Y + (size_t)plane * 9 * st + (size_t)(1 - par) * g.Vh_pad + up;
    double a[9], b[9];
    int E = FX_FIELD_MIN<double>;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        a[k] = __ldg(y0 + k * st);
        b[k] = __ldg(y1 + k * st);
        E = max(E, max(fx_field(a[k]), fx_field(b[k])));
    }
    // the anti-Hermitian matrix of nine reals, in units of 2^(E - 1023 - 54)
    auto full = [&](const double v[9], M3x &m) {
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const int4 d = fx_pack(0, fx_int<true>(v[i], E));
            m.m[i][i] = fx_unpack(d);
#pragma unroll
            for (int j = 0; j < i; ++j) {
                const int k = 3 + 2 * (i + j - 1);
                const int4 o = fx_pack(fx_int<true>(v[k], E), fx_int<true>(v[k + 1], E));
                m.m[i][j] = fx_unpack(o);
                m.m[j][i] = fxc{-o.x, -o.y, o.z, o.w};
            }
        }
    };
    M3x Um, M;
    load_m3x((const int4 *)U.a[par], cb, 36, nu * 9, false, Um);
    long long tr[3][3], tI[3][3];
    full(b, M);
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) fx_mul_elem(Um, M, i, j, tr[i][j], tI[i][j]);
    full(a, M);
    unsigned mh = 0, ml = 0;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            long long r, s;
            fx_mul_elem(M, Um, i, j, r, s);
            tr[i][j] += r;
            tI[i][j] += s;
            const long long t[2] = {tr[i][j], tI[i][j]};
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const unsigned h = (unsigned)((unsigned long long)t[q] >> 32), sg = (unsigned)((int)h >> 31);
                mh |= h ^ sg;
                ml |= (unsigned)t[q] ^ sg;
            }
        }
    // scaled below 2^55
    const int up1 = (mh ? __clz(mh) : 32 + min(__clz(ml), 31)) - 1;
    constexpr int DN = 63 - FX_BITS;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j)
            Z.z[par][soa(cb, 108, zi * 9 + 3 * i + j)] = fx_pack((tr[i][j] << up1) >> DN, (tI[i][j] << up1) >> DN);
    Z.e[(size_t)(zi * 2 + par) * g.Vh_pad + cb] = E == 0x7ff ? FX_NAN : E - (1023 + 54) + DN - up1;
}

// G_mu(m) of the sites of parity blockIdx.z, direction blockIdx.y
__global__ void __launch_bounds__(128, 3) k_force_link_x(Geom g, GaugePtr U, ForceZ Z, const double2 *__restrict__ x,
                                                         const double2 *__restrict__ lam, double kappa, int with_clover,
                                                         double2 *G, const int *wide)
{
    const int cb = blockIdx.x * blockDim.x + threadIdx.x, mu = blockIdx.y, par = blockIdx.z;
    if (cb >= g.Vh || *wide) return;
    int c[4];
    site_coords(g, par, cb, c);
    const int op = 1 - par;
    const int mp = cb_step(g, c, mu, 1, mu, 0);
    // ---- clover part in units of 2^E
    long long tr[3][3], tI[3][3];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) tr[i][j] = tI[i][j] = 0;
    int E = FX_ZERO;
    if (with_clover) {
#pragma unroll 1
        for (int k = 0; k < 12; ++k) {  // four terms P (Q T) of each of three planes
            const int n3 = k >> 2, t = k & 3, nu = n3 < mu ? n3 : n3 + 1;
            const int zi = z_index(nu, mu);
            // t = 0: U_nu(m), U_mu(m+nu), Z(m+mu)^dag      t = 1: Z(m), U_mu(m+nu), U_nu(m+mu)^dag
            // t = 2: Z(q)^dag, U_mu(q), U_nu(q+mu)          t = 3: U_nu(q)^dag, U_mu(q), Z(q+mu)
            const int q = cb_step(g, c, nu, -1, nu, 0);
            const bool low = t >= 2, zp = t == 1 || t == 2;  // P is the Z matrix
            const int4 *pp = zp ? Z.z[low ? op : par] : (const int4 *)U.a[low ? op : par];
            const int4 *pt = zp ? (const int4 *)U.a[low ? par : op] : Z.z[low ? par : op];
            const int sp = low ? q : cb, st = low ? cb_step(g, c, mu, 1, nu, -1) : mp;
            const int sq = low ? q : cb_step(g, c, nu, 1, nu, 0);
            const int e = __ldg(Z.e + (size_t)(zi * 2 + ((t == 1 || t == 3) ? par : op)) * g.Vh_pad + (zp ? sp : st));
            M3x B;
            {
                M3x Q, T;
                load_m3x((const int4 *)U.a[op], sq, 36, mu * 9, false, Q);
                load_m3x(pt, st, zp ? 36 : 108, zp ? nu * 9 : zi * 9, !low, T);
#pragma unroll
                for (int i = 0; i < 3; ++i)
#pragma unroll
                    for (int j = 0; j < 3; ++j) {
                        long long r, s;
                        fx_mul_elem(Q, T, i, j, r, s);
                        B.m[i][j] = fx_unpack(fx_pack(r, s));
                    }
            }
            M3x Pm;
            load_m3x(pp, sp, zp ? 108 : 36, zp ? zi * 9 : nu * 9, low, Pm);
            const int En = max(E, e), sa = fx_clamp63(En - E), sb = fx_clamp63(En - e);
            const bool neg = zp != (mu > nu);
#pragma unroll
            for (int i = 0; i < 3; ++i)
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    long long r, s;
                    fx_mul_elem(Pm, B, i, j, r, s);
                    r >>= sb;
                    s >>= sb;
                    tr[i][j] = (tr[i][j] >> sa) + (neg ? -r : r);
                    tI[i][j] = (tI[i][j] >> sa) + (neg ? -s : s);
                }
            E = En;
        }
    }
    // ---- hopping part
    C Gm[3][3];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) Gm[i][j] = mk(0.0, 0.0);
    int cp[4] = {c[0], c[1], c[2], c[3]};
#pragma unroll
    for (int k = 0; k < 4; ++k)
        if (k == mu) cp[k] = c[k] + 1 == g.L[k] ? 0 : c[k] + 1;
    const int m = lex_of(g, c), m1 = lex_of(g, cp);
    // (1 - g_mu): lambda(m) (x) conj(x(m+mu)); (1 + g_mu): x(m) (x) conj(lambda(m+mu))
#pragma unroll 1
    for (int k = 0; k < 2; ++k) {
        Spinor<double> A, B;
        load_spinor(k ? x : lam, m, A.s);
        load_spinor(k ? lam : x, m1, B.s);
        C ha[2][3], hb[2][3];
        project_rt(mu, k ? -1 : 1, A, ha);
        project_rt(mu, k ? -1 : 1, B, hb);
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = 0; j < 3; ++j)
#pragma unroll
                for (int a = 0; a < 2; ++a) fmac_(Gm[i][j], hb[a][j], ha[a][i]);
    }
    // mu = t: the projector's factor 2 (see project)
    const double f = kappa * ((mu == 3 && c[3] == g.L[3] - 1) ? (double)g.t_bc : 1.0) * (mu == 3 ? 2.0 : 1.0);
    const bool nan = E >= FX_NAN / 2;
    const double s1 = nan ? __longlong_as_double(0x7ff8000000000000ll) : fx_pow2(E < -1000 ? -1000 : E);
    const double s2 = E >= -1000 ? 1.0 : E < -2000 ? 0.0 : fx_pow2(E + 1000);
    double2 *out = G + ((size_t)m * 4 + mu) * 9;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j)
            out[3 * i + j] = make_double2(::fma(f, Gm[i][j].r, (double)tr[i][j] * s1 * s2),
                                          ::fma(f, Gm[i][j].i, (double)tI[i][j] * s1 * s2));
}

// v -> gamma5 v on canonical full-lattice vectors, gamma5 = -[[0,1],[1,0]];
// in and out may be the same buffer (no __restrict__: each thread reads its
// site completely before writing it)
__global__ void k_gamma5(int V, const double2 *in, double2 *out)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= V) return;
    const double2 *p = in + (size_t)s * 12;
    double2 v[12];
    for (int k = 0; k < 12; ++k) v[k] = p[k];
    double2 *o = out + (size_t)s * 12;
    for (int k = 0; k < 6; ++k) {
        o[k] = make_double2(-v[k + 6].x, -v[k + 6].y);
        o[k + 6] = make_double2(-v[k].x, -v[k].y);
    }
}

}  // namespace

int force(qcd_ctx *c, const void *x, const void *lam, void *G, const void *U_canon)
{
    // FP64 form: Y as full matrices; fixed-point form: Y as nine reals, Z and its
    // exponents, and the links that the caller passes (not the loaded ones) in
    // fixed point (34 us at 16^3x32).  Whether they are in its range is known on
    // the device only, so the FP64 kernels follow and return at once if they are.
    const size_t vp = (size_t)c->g.Vh_pad;
    const size_t yx = 54 * 2 * vp * sizeof(double), zx = 2 * vp * 108 * 16, ex = 24 * vp * sizeof(int);
    const size_t y64 = (size_t)c->g.V * 6 * 9 * 16, fx = yx + zx + ex + 2 * vp * 36 * 16;
    // Where the device has no room for the fixed-point form's 2784 bytes a site, the
    // context keeps the FP64 form with its 864.
    auto hold = [&](size_t bytes) -> int {
        if (c->force_bytes >= bytes) return QCD_OK;
        if (c->force_buf) {
            cudaStreamSynchronize(c->stream);
            cudaFree(c->force_buf);
            for (auto &p : c->pool)
                if (p == c->force_buf) p = nullptr;
            c->force_buf = nullptr;
            c->force_bytes = 0;
        }
        const int rc = dev_alloc(c, &c->force_buf, bytes);
        if (rc == QCD_OK) c->force_bytes = bytes;
        return rc;
    };
    int rc = QCD_OK;
    bool use_fx = c->fx_links && !c->force_fp64;
    if (use_fx && (rc = hold(fx > y64 ? fx : y64)) == QCD_ENOMEM) {
        c->force_fp64 = true;
        use_fx = false;
    }
    if (!use_fx) rc = hold(y64);
    if (rc) return rc;
    int *wide = nullptr;
    if (use_fx) {
        wide = c->flag_dev + 1;
        QCD_CUDA_CHECK(cudaMemsetAsync(wide, 0, sizeof(int), c->stream));
        double *Y = (double *)c->force_buf;
        ForceZ Z;
        Z.z[0] = (int4 *)((char *)c->force_buf + yx);
        Z.z[1] = Z.z[0] + vp * 108;
        Z.e = (int *)((char *)c->force_buf + yx + zx);
        int4 *ux = (int4 *)((char *)c->force_buf + yx + zx + ex);
        GaugePtr U;
        for (int p = 0; p < 2; ++p) {
            U.a[p] = ux + (size_t)p * vp * 36;
            U.b[p] = nullptr;
        }
        const unsigned nb = nblocks(c->g.Vh, 128);
        const int with = c->csw != 0.0;
        {
            ProfScope p0(c, QCD_K_OTHER, 0.0);
            k_force_Ux<<<nblocks(4L * c->g.V, 128), 128, 0, c->stream>>>(c->g, (const double2 *)U_canon, ux, ux + vp * 36, wide);
            QCD_CUDA_CHECK(cudaGetLastError());
        }
        if (with) {
            ProfScope p1(c, QCD_K_OTHER, 0.0);
            k_force_Yx<<<dim3(nb, 2), 128, 0, c->stream>>>(c->g, (const double2 *)x, (const double2 *)lam,
                                                            0.125 * c->csw * c->kappa, Y, wide);
            QCD_CUDA_CHECK(cudaGetLastError());
        }
        if (with) {
            ProfScope p2(c, QCD_K_OTHER, 0.0);
            k_force_Z<<<dim3(nb, 12, 2), 128, 0, c->stream>>>(c->g, U, Y, Z, wide);
            QCD_CUDA_CHECK(cudaGetLastError());
        }
        ProfScope p3(c, QCD_K_OTHER, 0.0);
        k_force_link_x<<<dim3(nb, 4, 2), 128, 0, c->stream>>>(c->g, U, Z, (const double2 *)x, (const double2 *)lam,
                                                              c->kappa, with, (double2 *)G, wide);
        QCD_CUDA_CHECK(cudaGetLastError());
    }
    // one wave where they most likely have nothing to do
    const auto blocks = [&](unsigned all) { return wide && all > 4u * c->num_sms ? 4u * c->num_sms : all; };
    {
        ProfScope prof(c, QCD_K_OTHER, 0.0);
        k_force_Y<<<blocks(nblocks(c->g.V, 128)), 128, 0, c->stream>>>(c->g, (const double2 *)x, (const double2 *)lam,
                                                              c->csw * c->kappa, (double2 *)c->force_buf, wide);
        QCD_CUDA_CHECK(cudaGetLastError());
    }
    {
        ProfScope prof(c, QCD_K_OTHER, 0.0);
        k_force_link<<<blocks(nblocks(4L * c->g.V, 64)), 64, 0, c->stream>>>(
            c->g, (const double2 *)U_canon, (const double2 *)x, (const double2 *)lam, (const double2 *)c->force_buf,
            c->kappa, c->csw != 0.0, (double2 *)G, wide);
        QCD_CUDA_CHECK(cudaGetLastError());
    }
    return QCD_OK;
}

int gamma5_full(qcd_ctx *c, const void *in, void *out)
{
    ProfScope prof(c, QCD_K_OTHER, 0.0);
    k_gamma5<<<nblocks(c->g.V, 128), 128, 0, c->stream>>>(c->g.V, (const double2 *)in, (double2 *)out);
    QCD_CUDA_CHECK(cudaGetLastError());
    return QCD_OK;
}

}  // namespace qcd
