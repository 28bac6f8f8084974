// Gauge-field ingest (the conversion [U, F] -> [U^SP, F^SP] of Alg. 1) and
// the clover term: F(n) = 1 - (csw kappa/2) sum_{mu!=nu} sigma_munu F_munu(n)
// with F_munu = (Q_munu - Q_munu^dag)/(8i) from the four plaquette leaves,
// built and inverted site by site in FP64 (Sec. II-B: "inverted easily"),
// stored as two 6x6 Hermitian blocks (Sec. III-A).
//
// Chiral blocks.  In the Dirac basis used here sigma_jk = -eps_jkl
// diag(s_l, s_l) and sigma_k4 = [[0, -s_k], [-s_k, 0]].  Both commute with
// gamma5; on chi_+ = (psi_up - psi_dn)/sqrt2 and chi_- = (psi_up + psi_dn)/sqrt2
// they act as sigma_jk -> -eps_jkl s_l and sigma_k4 -> +-s_k.  Hence
//   A_+- = 1 + csw kappa sum_l s_l (x) (B_l -+ E_l),
//   B_1 = F_yz, B_2 = F_zx, B_3 = F_xy, E_k = F_kt,
// each a 6x6 Hermitian matrix indexed 3*spin + colour.
#include "ctx.cuh"
#include "fx.cuh"

namespace qcd {

// ---------------------------------------------------------------- links
__device__ __forceinline__ float4 df_pair(double2 z)
{
    const df r(z.x), i(z.y);
    return make_float4(r.hi, r.lo, i.hi, i.lo);
}

// FX: the third copy of a link is its fixed-point form (fx.cuh); otherwise, for
// fields with links beyond that form's range, float pairs.
template <bool FX>
__global__ void k_gauge_convert(Geom g, const double2 *__restrict__ U, double2 *U64e, double2 *U64o, float4 *U32e,
                                float4 *U32o, uint4 *U16ae, uint4 *U16ao, uint2 *U16be, uint2 *U16bo, void *UXe,
                                void *UXo, int *wide)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= g.V) return;
    int c[4], t = s;
    for (int mu = 0; mu < 4; ++mu) {
        c[mu] = t % g.L[mu];
        t /= g.L[mu];
    }
    const int par = (c[0] + c[1] + c[2] + c[3]) & 1;
    const int cb = s >> 1;
    double2 *u64 = par ? U64o : U64e;
    float4 *u32 = par ? U32o : U32e;
    uint4 *u16a = par ? U16ao : U16ae;
    uint2 *u16b = par ? U16bo : U16be;
    void *ux = par ? UXo : UXe;
    for (int mu = 0; mu < 4; ++mu) {
        double2 m[9];
        for (int k = 0; k < 9; ++k) m[k] = U[((size_t)s * 4 + mu) * 9 + k];
        for (int k = 0; k < 9; ++k) u64[soa(cb, 36, mu * 9 + k)] = m[k];
        if constexpr (FX) {
            if (fx_store_link(m, (int4 *)ux, cb, mu)) *wide = 1;
        } else {
            for (int k = 0; k < 9; ++k) ((float4 *)ux)[soa(cb, 36, mu * 9 + k)] = df_pair(m[k]);
        }
        // first two columns: a = (m00, m10, m20), b = (m01, m11, m21)
        const double2 a0 = m[0], a1 = m[3], a2 = m[6], b0 = m[1], b1 = m[4], b2 = m[7];
        const double2 ab[6] = {a0, a1, a2, b0, b1, b2};
        float2 f[6];
        bool slow = false;
#pragma unroll
        for (int k = 0; k < 6; ++k) f[k] = make_float2(f32_int<false>(ab[k].x, slow), f32_int<false>(ab[k].y, slow));
        if (slow)
#pragma unroll
            for (int k = 0; k < 6; ++k) f[k] = make_float2((float)ab[k].x, (float)ab[k].y);
#pragma unroll
        for (int k = 0; k < 3; ++k)
            u32[soa(cb, 12, mu * 3 + k)] = make_float4(f[2 * k].x, f[2 * k].y, f[2 * k + 1].x, f[2 * k + 1].y);
        auto hh = [](float2 z) { return h2u(__floats2half2_rn(z.x, z.y)); };
        u16a[soa(cb, 4, mu)] = make_uint4(hh(f[0]), hh(f[1]), hh(f[2]), hh(f[3]));
        u16b[soa(cb, 4, mu)] = make_uint2(hh(f[4]), hh(f[5]));
    }
}

int gauge_convert(qcd_ctx *c, const void *U_dev)
{
    auto go = [&](auto kernel) -> int {
        kernel<<<nblocks(c->g.V, 256), 256, 0, c->stream>>>(
            c->g, (const double2 *)U_dev, (double2 *)c->U64[0], (double2 *)c->U64[1], (float4 *)c->U32[0],
            (float4 *)c->U32[1], (uint4 *)c->U16a[0], (uint4 *)c->U16a[1], (uint2 *)c->U16b[0], (uint2 *)c->U16b[1],
            c->UX[0], c->UX[1], c->flag_dev);
        QCD_CUDA_CHECK(cudaGetLastError());
        return QCD_OK;
    };
    QCD_CUDA_CHECK(cudaMemsetAsync(c->flag_dev, 0, sizeof(int), c->stream));
    int rc = go(k_gauge_convert<true>);
    if (rc) return rc;
    int wide = 0;
    QCD_CUDA_CHECK(cudaMemcpyAsync(&wide, c->flag_dev, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
    QCD_CUDA_CHECK(cudaStreamSynchronize(c->stream));
    c->fx_links = !wide;
    return wide ? go(k_gauge_convert<false>) : QCD_OK;
}

// ---------------------------------------------------------------- clover
// F_munu from ten 3x3 products per plane: with K = (L1 - L4^dag) + (L3 - L2^dag)
// the leaves' sum Q obeys Q - Q^dag = K - K^dag, and the four leaves of K pair
// by their first and last links,
//   K = [U_mu(n) P1 - U_mu(n-mu)^dag P1'] U_nu(n)^dag
//     - [U_mu(n) P2 - U_mu(n-mu)^dag P2'] U_nu(n-nu),
//   P1  = U_nu(n+mu) U_mu(n+nu)^dag,          P1' = U_nu(n-mu) U_mu(n-mu+nu),
//   P2  = U_nu(n+mu-nu)^dag U_mu(n-nu)^dag,   P2' = U_nu(n-mu-nu)^dag U_mu(n-mu-nu)
// (twelve products leaf by leaf).  One loop runs over the four P, daggers taken
// while loading, so that the code stays within the instruction cache (unrolled,
// the warps waited on fetches: 1.65 ms a parity at 24^3x48 against 1.22, now 1.16).  The
// products run in an algebra: AlgX, the fixed-point form of fx.cuh on the
// integer pipe, whose accumulators hold every product of links with a Frobenius
// norm up to sqrt(3) (each of SU(3) has exactly that); AlgD, FP64, for fields
// with larger links.
struct M3 {
    cx<double> m[3][3];
};

struct AlgX {
    using M = M3x;
    using T = long long;
    // the link, or its conjugate transpose, its real parts times sr and its
    // imaginary parts times si
    static __device__ __forceinline__ M load(const GaugePtr &U, int par, int cb, int mu, bool dg, int sr, int si)
    {
        const int4 *p = (const int4 *)U.a[par];
        M r;
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const int4 v = __ldg(p + soa(cb, 36, mu * 9 + (dg ? 3 * j + i : 3 * i + j)));
                r.m[i][j] = fxc{v.x * sr, v.y * sr, v.z * si, v.w * si};
            }
        return r;
    }
    static __device__ __forceinline__ void elem(const M &A, const M &B, int i, int j, T &r, T &s)
    {
        fx_mul_elem(A, B, i, j, r, s);
    }
    static __device__ __forceinline__ void set(M &A, int i, int j, T r, T s) { A.m[i][j] = fx_unpack(fx_pack(r, s)); }
    static constexpr double UNIT = 1.0 / (double)(1ll << FX_BITS);
};

struct AlgD {
    using M = M3;
    using T = double;
    static __device__ __forceinline__ M load(const GaugePtr &U, int par, int cb, int mu, bool dg, int sr, int si)
    {
        const double2 *p = (const double2 *)U.a[par];
        M r;
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const double2 v = __ldg(p + soa(cb, 36, mu * 9 + (dg ? 3 * j + i : 3 * i + j)));
                r.m[i][j] = mk(sr * v.x, si * v.y);
            }
        return r;
    }
    static __device__ __forceinline__ void elem(const M &A, const M &B, int i, int j, T &r, T &s)
    {
        cx<double> z = mk(0.0, 0.0);
#pragma unroll
        for (int k = 0; k < 3; ++k) fma_(z, A.m[i][k], B.m[k][j]);
        r = z.r;
        s = z.i;
    }
    static __device__ __forceinline__ void set(M &A, int i, int j, T r, T s) { A.m[i][j] = mk(r, s); }
    static constexpr double UNIT = 1.0;
};

// F_munu at site n of parity par (coordinates c): the three real diagonal
// entries, then (re, im) of the entries (1,0), (2,0), (2,1) below it
template <class Alg>
__device__ __forceinline__ void field_strength(const Geom &g, const GaugePtr &U, int par, const int c[4], int mu, int nu,
                                               double ck, double F[9])
{
    using M = typename Alg::M;
    using T = typename Alg::T;
    auto at = [&](int dm, int dn) {  // cb of n + dm mu + dn nu
        int lex = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int d = k == mu ? dm : k == nu ? dn : 0;
            int x = c[k] + d;
            x = x < 0 ? x + g.L[k] : x >= g.L[k] ? x - g.L[k] : x;
            lex += x * g.st[k];
        }
        return lex >> 1;
    };
    const int op = 1 - par;
    T Fd[3] = {0, 0, 0}, Fr[3] = {0, 0, 0}, Fi[3] = {0, 0, 0};  // of K - K^dag: Im diagonal; entries (1,0), (2,0), (2,1)
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {  // the bracket of U_nu(n)^dag, then of U_nu(n-nu)
        M R;
        {
            T Rr[3][3], Ri[3][3];
#pragma unroll
            for (int i = 0; i < 3; ++i)
#pragma unroll
                for (int j = 0; j < 3; ++j) Rr[i][j] = Ri[i][j] = 0;
#pragma unroll 1
            for (int k = 0; k < 2; ++k) {  // + U_mu(n) P, - U_mu(n-mu)^dag P'
                const int dm = k ? -1 : 1;
                M P;
                {
                    // X Y: U_nu(n+dm mu [-nu]) (daggered below) times U_mu of the other end
                    const M X = Alg::load(U, h ? par : op, at(dm, h ? -1 : 0), nu, h, 1, h ? -1 : 1);
                    const M Y = Alg::load(U, k ? par : op, at(k ? -1 : 0, h ? -1 : 1), mu, !k, 1, k ? 1 : -1);
#pragma unroll
                    for (int i = 0; i < 3; ++i)
#pragma unroll
                        for (int j = 0; j < 3; ++j) {
                            T r, s;
                            Alg::elem(X, Y, i, j, r, s);
                            Alg::set(P, i, j, r, s);
                        }
                }
                // with the signs of both brackets: dagger in k, minus in k and in h
                const M A = Alg::load(U, k ? op : par, at(k ? -1 : 0, 0), mu, k, k ^ h ? -1 : 1, h ? -1 : 1);
#pragma unroll
                for (int i = 0; i < 3; ++i)
#pragma unroll
                    for (int j = 0; j < 3; ++j) {
                        T r, s;
                        Alg::elem(A, P, i, j, r, s);
                        Rr[i][j] += r;
                        Ri[i][j] += s;
                    }
            }
#pragma unroll
            for (int i = 0; i < 3; ++i)
#pragma unroll
                for (int j = 0; j < 3; ++j) Alg::set(R, i, j, Rr[i][j], Ri[i][j]);
        }
        const M B = Alg::load(U, h ? op : par, at(0, h ? -1 : 0), nu, !h, 1, h ? 1 : -1);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            T r, s;
            Alg::elem(R, B, i, i, r, s);
            Fd[i] += s;
#pragma unroll
            for (int j = 0; j < i; ++j) {
                T r2, s2;
                Alg::elem(R, B, i, j, r, s);
                Alg::elem(R, B, j, i, r2, s2);
                Fr[i + j - 1] += r - r2;
                Fi[i + j - 1] += s + s2;
            }
        }
    }
    // ck (K - K^dag)/(8i)
    const double f = 0.125 * Alg::UNIT * ck;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        F[i] = 2.0 * f * (double)Fd[i];
        F[3 + 2 * i] = f * (double)Fi[i];
        F[4 + 2 * i] = -f * (double)Fr[i];
    }
}

// A Hermitian 6x6 matrix as its diagonal and its lower triangle, row by row
struct Herm6 {
    double d[6];
    cx<double> o[15];
};
__device__ __forceinline__ constexpr int tri(int i, int j) { return i * (i - 1) / 2 + j; }

// A -> A^-1 by A = L D L^dag (no pivoting; the clover blocks are close to the
// identity), in place: L, then M = L^-1 over it, then M^dag D^-1 M.  (The kernel
// has a frame of 288 bytes in local memory, the 36 reals of a block, without spills.)
// Returns false on a (near-)zero pivot.
__device__ __forceinline__ bool herm_inverse6(Herm6 &A)
{
    double amax = 0.0;
#pragma unroll
    for (int i = 0; i < 6; ++i) amax = fmax(amax, fabs(A.d[i]));
    double inv[6];
    bool ok = true;
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        // column j: w_ij = A_ij - sum_k L_ik D_k conj(L_jk); L_ij = w_ij / D_j
        cx<double> v[6];  // D_k conj(L_jk)
        double dj = A.d[j];
#pragma unroll
        for (int k = 0; k < j; ++k) {
            const cx<double> l = A.o[tri(j, k)];
            v[k] = mk(A.d[k] * l.r, -(A.d[k] * l.i));
            dj = ::fma(-v[k].r, l.r, dj);
            dj = ::fma(v[k].i, l.i, dj);
        }
        ok = ok && fabs(dj) > 1e-12 * amax && isfinite(dj);
        A.d[j] = dj;
        inv[j] = 1.0 / dj;
#pragma unroll
        for (int i = j + 1; i < 6; ++i) {
            cx<double> s = A.o[tri(i, j)];
#pragma unroll
            for (int k = 0; k < j; ++k) fma_(s, -A.o[tri(i, k)], v[k]);
            A.o[tri(i, j)] = inv[j] * s;
        }
    }
    // M = L^-1 (unit lower triangular): M_ij = -(L_ij + sum_{j<k<i} L_ik M_kj),
    // row by row (row i uses its own L entries and the finished rows above)
#pragma unroll
    for (int i = 1; i < 6; ++i) {
        cx<double> row[6];
#pragma unroll
        for (int j = 0; j < i; ++j) {
            cx<double> s = A.o[tri(i, j)];
#pragma unroll
            for (int k = j + 1; k < i; ++k) fma_(s, A.o[tri(i, k)], A.o[tri(k, j)]);
            row[j] = -s;
        }
#pragma unroll
        for (int j = 0; j < i; ++j) A.o[tri(i, j)] = row[j];
    }
    // (A^-1)_ij = sum_{k >= i} conj(M_ki) M_kj / D_k, i >= j: row i needs M's
    // rows from i on only, so the result replaces M row by row
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        cx<double> w[6];  // conj(M_ki) / D_k
#pragma unroll
        for (int k = i + 1; k < 6; ++k) {
            const cx<double> m = A.o[tri(k, i)];
            w[k] = mk(inv[k] * m.r, -(inv[k] * m.i));
        }
        double dd = inv[i];
#pragma unroll
        for (int k = i + 1; k < 6; ++k) {
            dd = ::fma(w[k].r, A.o[tri(k, i)].r, dd);
            dd = ::fma(-w[k].i, A.o[tri(k, i)].i, dd);
        }
        A.d[i] = dd;
#pragma unroll
        for (int j = 0; j < i; ++j) {
            cx<double> s = inv[i] * A.o[tri(i, j)];
#pragma unroll
            for (int k = i + 1; k < 6; ++k) fma_(s, w[k], A.o[tri(k, j)]);
            A.o[tri(i, j)] = s;
        }
    }
    return ok;
}

struct CloverOut {
    double2 *f64;
    float4 *f32;
    uint4 *f16;
    void *x;  // fixed point, or float pairs where the links are out of its range
    int *e;   // the fixed-point blocks' unit exponents, two per site
};

// store one block (diag reals then the lower triangle) in all precisions
template <bool FX>
__device__ __forceinline__ void store_block(const Herm6 &A, int blk, int cb, const CloverOut &O)
{
    double2 *p64 = O.f64;
    float4 *p32 = O.f32;
    uint4 *p16 = O.f16;
    double r[36];
#pragma unroll
    for (int i = 0; i < 6; ++i) r[i] = A.d[i];
#pragma unroll
    for (int k = 0; k < 15; ++k) {
        r[6 + 2 * k] = A.o[k].r;
        r[7 + 2 * k] = A.o[k].i;
    }
#pragma unroll
    for (int q = 0; q < 18; ++q) p64[soa(cb, 36, blk * 18 + q)] = make_double2(r[2 * q], r[2 * q + 1]);
    if constexpr (FX) {
        int E = FX_FIELD_MIN<double>;
#pragma unroll
        for (int k = 0; k < 36; ++k) E = max(E, fx_field(r[k]));
#pragma unroll
        for (int q = 0; q < 18; ++q)
            // (cut: rounded, the blocks of an 8^4 build took 5 us of 121 longer)
            ((int4 *)O.x)[soa(cb, 36, blk * 18 + q)] = fx_pack(fx_int<false>(r[2 * q], E), fx_int<false>(r[2 * q + 1], E));
        O.e[2 * cb + blk] = E - (1023 + 54);
    } else {
#pragma unroll
        for (int q = 0; q < 18; ++q)
            ((float4 *)O.x)[soa(cb, 36, blk * 18 + q)] = df_pair(make_double2(r[2 * q], r[2 * q + 1]));
    }
    float f[36];
    unsigned w[18];
    bool slow = false;
#pragma unroll
    for (int k = 0; k < 36; ++k) f[k] = f32_int<false>(r[k], slow);
    // halves, rounded from FP64: element e = 36 blk + j of the site is half e & 7
    // of uint4 e >> 3, so block 0 ends and block 1 begins in the middle of uint4 4
#pragma unroll
    for (int k = 0; k < 18; ++k)
        w[k] = h2u(__floats2half2_rn(f32_int<true>(r[2 * k], slow), f32_int<true>(r[2 * k + 1], slow)));
#pragma unroll
    for (int q = 0; q < 9; ++q) p32[soa(cb, 18, blk * 9 + q)] = make_float4(f[4 * q], f[4 * q + 1], f[4 * q + 2], f[4 * q + 3]);
    const int q0 = blk ? 5 : 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int a = 4 * q;
        p16[soa(cb, 9, q0 + q)] = blk ? make_uint4(w[a + 2], w[a + 3], w[a + 4], w[a + 5]) : make_uint4(w[a], w[a + 1], w[a + 2], w[a + 3]);
    }
    ((uint2 *)p16)[soa(cb, 9, 4) * 2 + blk] = blk ? make_uint2(w[0], w[1]) : make_uint2(w[16], w[17]);
    if (slow)  // (rare) entries beyond FP32's normal range: over again from the stored block
#pragma unroll 1
        for (int j = 0; j < 36; ++j) {
            const int e = 36 * blk + j;
            const double v = ((const double *)(p64 + soa(cb, 36, e >> 1)))[e & 1];
            ((float *)(p32 + soa(cb, 18, e >> 2)))[e & 3] = (float)v;
            ((__half *)(p16 + soa(cb, 9, e >> 3)))[e & 7] = __double2half(v);
        }
}

// Field strengths of the sites [first, end) of one parity, times csw kappa:
// [plane][9][stride] doubles
struct FsBuf {
    double *p;
    int first, end;
    size_t stride;
};

// Both kernels replace one that walked the planes twice per site in FP64 with
// its matrices in local memory: 24^3x48, both parities, 23.5 ms before, 3.8 ms
// now (k_field_strength 2.3 ms, issue-bound at 0.45 of a slot per cycle with
// twelve warps an SM; k_clover_build 1.5 ms, the inverses on the FP64 pipe).
// Field strengths: thread = (site, plane), blockIdx.y the plane; planes (0,1)
// (0,2) (0,3) (1,2) (1,3) (2,3).
template <class Alg>
__global__ void __launch_bounds__(128, 3) k_field_strength(Geom g, GaugePtr U, int par, double ck, FsBuf FS)
{
    const int cb = FS.first + blockIdx.x * blockDim.x + threadIdx.x, w = blockIdx.y;
    if (cb >= FS.end) return;
    const int mu = w < 3 ? 0 : w < 5 ? 1 : 2, nu = w < 3 ? w + 1 : w < 5 ? w - 1 : 3;
    int c[4];
    site_coords(g, par, cb, c);
    double f[9];
    field_strength<Alg>(g, U, par, c, mu, nu, ck, f);
#pragma unroll
    for (int k = 0; k < 9; ++k) FS.p[((size_t)w * 9 + k) * FS.stride + (cb - FS.first)] = f[k];
}

// The chiral block blockIdx.y (0: A_+, gamma5 = +1; 1: A_-) of every one of these
// sites, assembled from the field strengths, stored, inverted, stored.
template <bool FX>
__global__ void __launch_bounds__(128) k_clover_build(FsBuf FS, CloverOut F, CloverOut Fi, int *bad)
{
    const int cb = FS.first + blockIdx.x * blockDim.x + threadIdx.x, blk = blockIdx.y;
    if (cb >= FS.end) return;
    auto fs = [&](int plane, int k) { return __ldg(FS.p + ((size_t)plane * 9 + k) * FS.stride + (cb - FS.first)); };
    // G_l = B_l -+ E_l: B_1 = F_yz, B_2 = -F_xz, B_3 = F_xy, E = F_xt, F_yt, F_zt
    double G1[9], G2[9], G3[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const double e1 = fs(2, k), e2 = fs(4, k), e3 = fs(5, k);
        G1[k] = fs(3, k) + (blk ? e1 : -e1);
        G2[k] = (blk ? e2 : -e2) - fs(1, k);
        G3[k] = fs(0, k) + (blk ? e3 : -e3);
    }
    auto ent = [](const double G[9], int i, int j) {  // G_ij of the Hermitian G
        if (i == j) return mk(G[i], 0.0);
        const int k = 3 + 2 * (i + j - 1);
        return i > j ? mk(G[k], G[k + 1]) : mk(G[k], -G[k + 1]);
    };
    // A = 1 + s_1 (x) G1 + s_2 (x) G2 + s_3 (x) G3, indexed 3 spin + colour
    Herm6 A;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        A.d[i] = 1.0 + G3[i];
        A.d[3 + i] = 1.0 - G3[i];
#pragma unroll
        for (int j = 0; j < i; ++j) {
            A.o[tri(i, j)] = ent(G3, i, j);
            A.o[tri(3 + i, 3 + j)] = -ent(G3, i, j);
        }
#pragma unroll
        for (int j = 0; j < 3; ++j) A.o[tri(3 + i, j)] = ent(G1, i, j) + ti(ent(G2, i, j));
    }
    store_block<FX>(A, blk, cb, F);
    if (!herm_inverse6(A)) {
        atomicExch(bad, 1);
#pragma unroll
        for (int i = 0; i < 6; ++i) A.d[i] = 0.0;
#pragma unroll
        for (int k = 0; k < 15; ++k) A.o[k] = mk(0.0, 0.0);
    }
    store_block<FX>(A, blk, cb, Fi);
}

int clover_build(qcd_ctx *c, double kappa, double csw)
{
    GaugePtr U;
    for (int p = 0; p < 2; ++p) {
        U.a[p] = c->fx_links ? c->UX[p] : c->U64[p];
        U.b[p] = nullptr;
    }
    QCD_CUDA_CHECK(cudaMemsetAsync(c->flag_dev, 0, sizeof(int), c->stream));
    auto out = [&](void *const f[4][2], int *const e[2], int par) {
        return CloverOut{(double2 *)f[QCD_F64][par], (float4 *)f[QCD_F32][par], (uint4 *)f[QCD_F16][par],
                         f[QCD_DF64][par], e[par]};
    };
    // the field strengths of one parity at a time
    // (the buffer at least as large as the operator calls need it, so that the
    // first of them does not free it, wait and allocate again; where the device has
    // no room for that, of a part of the sites at a time)
    constexpr size_t SITE = 54 * sizeof(double);
    int n = c->g.Vh_pad;
    const size_t fs = n * SITE, ops = (size_t)c->g.V * 12 * 16 * 2;
    int rc = ensure_staging(c, fs > ops ? fs : ops);
    while (rc == QCD_ENOMEM && n > 128) {
        n = (n / 2 + 127) / 128 * 128;
        rc = ensure_staging(c, n * SITE);
    }
    if (rc) return rc;
    for (int par = 0; par < 2; ++par)
        for (int first = 0; first < c->g.Vh; first += n) {
            const FsBuf FS{(double *)c->staging, first, first + n < c->g.Vh ? first + n : c->g.Vh, (size_t)n};
            const unsigned nb = nblocks(FS.end - first, 128);
            const dim3 gs(nb, 6), gc(nb, 2);
            const double ck = csw * kappa;
            const CloverOut F = out(c->C, c->Cx, par), Fi = out(c->Ci, c->Cix, par);
            if (c->fx_links) {
                k_field_strength<AlgX><<<gs, 128, 0, c->stream>>>(c->g, U, par, ck, FS);
                k_clover_build<true><<<gc, 128, 0, c->stream>>>(FS, F, Fi, c->flag_dev);
            } else {
                k_field_strength<AlgD><<<gs, 128, 0, c->stream>>>(c->g, U, par, ck, FS);
                k_clover_build<false><<<gc, 128, 0, c->stream>>>(FS, F, Fi, c->flag_dev);
            }
            QCD_CUDA_CHECK(cudaGetLastError());
        }
    int bad = 0;
    QCD_CUDA_CHECK(cudaMemcpyAsync(&bad, c->flag_dev, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
    QCD_CUDA_CHECK(cudaStreamSynchronize(c->stream));
    if (bad) {
        set_error_message("clover block with a zero pivot (kappa=%g, csw=%g)", kappa, csw);
        return QCD_ECLOVER_SINGULAR;
    }
    return QCD_OK;
}

}  // namespace qcd
