// The hopping stencil H_{p,1-p} (Eq. 4) and the kernels built on it:
//   M_HOP   out = H in                       (qcd_dslash_eo)
//   M_MULT  out = F^-1 H in                  (MULT = H~, Sec. II-B)
//   M_DHAT  out = a*y + cc*F^-1 H in + d*z   (second half of D^ = 1 - k^2 H~_eo H~_oe,
//                                             with the dot products of Alg. 2 fused)
//   M_SRC   out = F^-1 (a*y + cc*H in)       (b^_e, Eq. 6, and x_o, Eq. 7)
//   M_FULL  out = a*F y + cc*H in + d*z      (D = F - kappa H on one parity, residuals)
//   M_RECON out = F^-1 (a*y + cc*H in) and |a*y + cc*H in - F out|^2 (FP64 only)
//
// One thread computes one output site (and one right-hand side: the
// right-hand sides of a site sit in the same block so that its links and
// clover entries are fetched from HBM once and hit L1 for the others).
// For each of the 8 directions the neighbour spinor is projected with
// (1 -/+ gamma_mu) to two spin components before the colour multiply
// (the rank-2 structure of Eq. 4), the link is rebuilt from 12 reals for
// FP32/FP16 (Sec. III-A), multiplied, and expanded back.
#include "stencil.cuh"

namespace qcd {

// per-precision instantiations (stencil_<prec>.cu) and the multi-RHS kernel
int dispatch_f64(const StencilCall &sc, const StencilArgs &A, dim3 grid, dim3 block, cudaStream_t s, int v);
int dispatch_fx(const StencilCall &sc, const StencilArgs &A, dim3 grid, dim3 block, cudaStream_t s);
int dispatch_f32(const StencilCall &sc, const StencilArgs &A, dim3 grid, dim3 block, cudaStream_t s, int v);
int dispatch_f32_rg(const StencilCall &sc, const StencilArgs &A, int bx, cudaStream_t s, int v);
int dispatch_f16(const StencilCall &sc, const StencilArgs &A, dim3 grid, dim3 block, cudaStream_t s, int v);
int dispatch_df64(const StencilCall &sc, const StencilArgs &A, dim3 grid, dim3 block, cudaStream_t s, int v);
int launch_mrhs(const StencilCall &sc, const StencilArgs &A, int nrhs, cudaStream_t s, int variant, int tile,
                int num_sms);

// Algorithmic bytes per output site of one stencil launch (each input read
// once, the output written once), by precision: spinor, link, clover.
static void site_bytes(int prec, double &spinor, double &link, double &clover)
{
    if (prec == QCD_F64 || prec == QCD_DF64) { spinor = 192; link = 144; clover = 576; }
    else if (prec == QCD_F32) { spinor = 96; link = 48; clover = 288; }
    else { spinor = 52; link = 24; clover = 144; }
}

static bool runs_fx(const qcd_ctx *c, int prec) { return c->fx_links && (prec == QCD_F64 || prec == QCD_DF64); }

unsigned tune_key(const qcd_ctx *c, const StencilCall &sc)
{
    const unsigned nr = sc.nrhs < 1 ? 1 : (sc.nrhs > 31 ? 31 : sc.nrhs);
    return (unsigned)sc.prec | ((unsigned)sc.mode << 2) | ((unsigned)sc.red << 5) | ((unsigned)(sc.dagger != 0) << 7) |
           (nr << 8) | (runs_fx(c, sc.prec) ? TUNE_KEY_FX : 0u);
}

double stencil_bytes(const qcd_ctx *c, const StencilCall &sc)
{
    double sp, lk, cl;
    site_bytes(sc.prec, sp, lk, cl);
    const int nrhs = sc.nrhs < 1 ? 1 : sc.nrhs;
    double per_site = nrhs * 2 * sp + 8 * lk;  // in, out, links
    if (sc.mode != M_HOP) per_site += cl;
    if (sc.mode == M_DHAT || sc.mode == M_SRC || sc.mode == M_FULL || sc.mode == M_RECON) per_site += nrhs * sp;  // y
    if (sc.mode == M_RECON) per_site += cl;  // F as well as F^-1
    if (sc.d != 0.0 && (sc.mode == M_DHAT || sc.mode == M_FULL)) per_site += nrhs * sp;   // z
    if (sc.red == R_DOT_AUX || (sc.red == R_OMEGA && sc.aux.p != sc.y.p)) per_site += nrhs * sp;
    return per_site * c->g.Vh;
}

bool is_mrhs(const StencilCall &sc)
{
    return sc.prec == QCD_F32 && sc.nrhs > 1 && sc.red == R_NONE && (sc.mode == M_MULT || sc.mode == M_HOP);
}

bool canon_out(const qcd_ctx *c, const StencilCall &s, const void *dst)
{
    return (runs_fx(c, s.prec) || (s.prec == QCD_F32 && (uintptr_t)dst % 16 == 0)) && s.red == R_NONE &&
           (s.mode == M_HOP || s.mode == M_MULT || s.mode == M_DHAT || s.mode == M_FULL);
}

// the threads that five blocks of 128 an SM hold
static long one_wave(const qcd_ctx *c) { return 640L * c->num_sms; }

// The launch shape where the tuner has no entry: sites per block (for the
// multi-RHS kernel the right-hand sides per block) and register budget.
// FP32 and FP16 with more threads than one wave at the compiler's budget holds: the
// 80-register kernels, six such blocks.  Solves with every such launch at one shape,
// budget / 80 registers: 20^3x40 10.43 / 9.98 ms, 24^3x48 18.55 / 17.65, FP16 inner
// level at 40^3x80 104.8 / 96.6.  Below, the
// SMs are not full and spills only lengthen the chain: 16^3x32 5.74 / 5.91 ms,
// 12^3x24 4.42 / 4.54.  Where dot products are fused, 256 sites per block (half
// the partials of 128) once that leaves most SMs a block: 128 / 256 sites 12^3x24
// 3.86 / 3.79 ms, 16^3x32 4.97 / 4.82, 24^3x48 17.48 / 17.27; 8^3x16 2.64 / 2.76.
static void default_shape(const qcd_ctx *c, const StencilCall &sc, int &variant, int &bx)
{
    const int nrhs = sc.nrhs < 1 ? 1 : sc.nrhs;
    variant = 0;
    bx = 128;
    if (nrhs > 1) bx = is_mrhs(sc) ? nrhs : nrhs <= 4 ? 64 : 32;
    // fixed point (two threads a site, 168 registers): blocks of 128 threads, three
    // an SM; 256 threads fit once (MULT at 24^3x48 175 / 223 us)
    if (runs_fx(c, sc.prec)) {
        bx = nrhs > 1 ? 32 : 64;
        // down to one warp a block while SMs would stay without one
        while (nrhs == 1 && bx > 16 && (int)nblocks(c->g.Vh, bx) < c->num_sms) bx >>= 1;
    }
    const bool low = sc.prec == QCD_F32 || sc.prec == QCD_F16;
    if (low && !is_mrhs(sc) && (long)c->g.Vh * nrhs > one_wave(c)) variant = 1;
    if (low && sc.red != R_NONE && c->g.Vh >= 128 * c->num_sms) bx = 256;
}

int launch_stencil(qcd_ctx *c, const StencilCall &sc)
{
    StencilArgs A;
    A.g = c->g;
    const int p = sc.prec;
    // FP64 and DF64 in fixed point where the links allow it
    A.fx = runs_fx(c, p);
    const int pf = A.fx ? QCD_DF64 : p;  // the precision slot of the fields
    for (int par = 0; par < 2; ++par) {
        A.U.a[par] = pf == QCD_F64 ? c->U64[par] : pf == QCD_F32 ? c->U32[par] : pf == QCD_DF64 ? c->UX[par] : c->U16a[par];
        A.U.b[par] = c->U16b[par];
        A.C.p[par] = (sc.mode == M_FULL) ? c->C[pf][par] : c->Ci[pf][par];
        A.C.e[par] = (sc.mode == M_FULL) ? c->Cx[par] : c->Cix[par];
        A.Cf.p[par] = c->C[pf][par];
        A.Cf.e[par] = c->Cx[par];
    }
    A.y_fx = sc.y.prec == QCD_FX;
    HVec in = sc.in;
    if (A.fx && in.prec != QCD_FX) {
        // the caller's input in FP64 or DF64: one conversion pass (each site
        // converted once instead of by its eight neighbours)
        if (sc.nrhs > 1) {
            set_error_message("several right-hand sides in FP64 or DF64 take fixed-point input");
            return QCD_EINVAL;
        }
        HVec fx;
        int rc = get_work(c, QCD_FX, FX_IN, &fx);
        if (rc || (rc = convert_half(c, in, fx, sc.done))) return rc;
        in = fx;
    }
    A.out = sc.out.sp();
    A.in = in.sp();
    A.y = sc.y.sp();
    A.aux = sc.aux.sp();
    A.z = sc.z.sp();
    A.out_par = sc.out_par;
    A.a = sc.a;
    A.cc = sc.cc;
    A.d = sc.d;
    A.af = (float)sc.a;
    A.ccf = (float)sc.cc;
    A.df32 = (float)sc.d;
    A.has_z = sc.d != 0.0;
    A.rhs_stride = sc.rhs_stride;
    A.norm_stride = sc.norm_stride;
    A.nrhs = sc.nrhs < 1 ? 1 : sc.nrhs;
    A.red = sc.red_args;
    A.done = sc.done;
    A.canon = sc.canon;
    A.canon_stride = sc.canon_stride;
    // A large FP32 or FP16 stencil does not start beside the blocks of the pack before
    // it: there it took half as long again, and the D^ half behind it too (probably
    // because an SM that is never empty keeps the split of L1 and shared memory that
    // the pack's 14 KB a block asked for).  Overlapped / apart, FP32 D^ call: 24^3x48
    // 144.7 / 106.3 us, 18^3x36 52.4 / 39.0, 16^3x32 35.8 / 30.0 but its MULT call 17.0 / 20.4,
    // 12^3x24 19.3 / 22.6: from one wave on.  FP16: 24^3x48 87.6 / 81.9, 18^3x36 33.5 / 35.1,
    // two right-hand sides 40.1 / 42.3 at 16^3x32, 82.3 / 76.1 at 20^3x40: from two waves
    // of six blocks an SM on.  (FP64 MULT call 24^3x48 228.7 / 230.1.)
    const long threads = (long)c->g.Vh * A.nrhs;
    A.apart = sc.after_pack &&
              ((p == QCD_F32 && threads > one_wave(c)) || (p == QCD_F16 && threads > 2L * 768 * c->num_sms));
    A.done_stride = sc.done_stride;
    A.red_pstride = sc.red_pstride;
    A.skip = nullptr;
    const int nrhs = sc.nrhs < 1 ? 1 : sc.nrhs;
    if (nrhs > 16) {
        set_error_message("nrhs > 16 per launch");
        return QCD_EINVAL;
    }
    if (sc.rhs_grid) {
        // a lockstep second half: the single-RHS entry's register budget and
        // sites per block, so that every right-hand side repeats the
        // single-RHS launch's arithmetic and reduction order
        if (p != QCD_F32 || sc.mode != M_DHAT || (sc.red != R_DOT_AUX && sc.red != R_OMEGA) ||
            sc.done_stride < 1 || !sc.red_pstride) {
            set_error_message("rhs_grid: FP32 D^ second halves with per-RHS states and partials only");
            return QCD_EINVAL;
        }
        StencilCall one = sc;
        one.nrhs = 1;
        one.rhs_grid = false;
        int v, b;
        default_shape(c, one, v, b);
        auto it = c->tune.find(tune_key(c, one));
        if (it != c->tune.end()) {
            v = it->second.variant;
            b = it->second.bx;
        }
        if (v != 1) v = 0;  // the rolled and pipelined hops have no lockstep form: the plain kernel
        if ((size_t)nblocks(c->g.Vh, b) * 4 > sc.red_pstride) {
            set_error_message("rhs_grid: %u partials per right-hand side do not fit", nblocks(c->g.Vh, b));
            return QCD_EINVAL;
        }
        const int rc = dispatch_f32_rg(sc, A, b, c->stream, v);
        if (rc != QCD_OK) return rc;
        c->launches += 1;
        QCD_CUDA_CHECK(cudaGetLastError());
        return QCD_OK;
    }
    int bx, variant;  // bx: sites per block, or for the multi-RHS kernel the RHS tile
    default_shape(c, sc, variant, bx);
    if (sc.force_variant >= 0) {
        variant = sc.force_variant;
        bx = sc.force_bx;
    } else {
        auto it = c->tune.find(tune_key(c, sc));
        if (it != c->tune.end()) {
            variant = it->second.variant;
            bx = it->second.bx / (A.fx ? 2 : 1);  // threads a block
        }
    }
    const int cap = A.fx ? 192 : 384;  // sites times right-hand sides of a block (fixed point: two threads each)
    if (!is_mrhs(sc) && bx * nrhs > cap) {
        // more right-hand sides than a block of the generic kernels holds:
        // launch them in groups (no reduction spans the groups)
        if (sc.red != R_NONE) {
            set_error_message("a fused reduction over %d right-hand sides is not supported", nrhs);
            return QCD_EINVAL;
        }
        const int per = cap / bx;
        for (int r0 = 0; r0 < nrhs; r0 += per) {
            StencilCall g = sc;
            g.nrhs = nrhs - r0 < per ? nrhs - r0 : per;
            g.force_variant = variant;
            g.force_bx = bx;
            HVec *vs[5] = {&g.out, &g.in, &g.y, &g.z, &g.aux};
            for (HVec *v : vs) {
                if (v->p) v->p = (char *)v->p + (size_t)r0 * sc.rhs_stride * 16;
                if (v->norm) v->norm += (size_t)r0 * sc.norm_stride;
            }
            if (g.canon) g.canon = (char *)g.canon + (size_t)r0 * sc.canon_stride * (p == QCD_F32 ? 4 : 8);
            const int rc = launch_stencil(c, g);
            if (rc != QCD_OK) return rc;
        }
        return QCD_OK;
    }
    dim3 block(bx, nrhs);
    dim3 grid(nblocks(c->g.Vh, bx));
    if (!is_mrhs(sc) && sc.red != R_NONE && (int)grid.x > c->partial_blocks) {
        set_error_message("reduction grid too large");
        return QCD_EINVAL;
    }
    // the second half of an even-odd operator with its fused dots (D^_ee:
    // M_DHAT; S_ee: M_FULL with a reduction) is timed apart from the MULTs
    const bool second_half = sc.mode == M_DHAT || (sc.mode == M_FULL && sc.red != R_NONE);
    const int cls = p == QCD_F32    ? (second_half ? QCD_K_DHAT_F32 : QCD_K_MULT_F32)
                    : p == QCD_F16  ? QCD_K_MULT_F16
                    : p == QCD_DF64 ? QCD_K_MULT_DF64
                                    : QCD_K_MULT_F64;
    ProfScope prof(c, cls, stencil_bytes(c, sc));
    A.skip = prof.flag;
    int rc;
    const int rv = variant;
    if (is_mrhs(sc)) rc = launch_mrhs(sc, A, nrhs, c->stream, rv, bx, c->num_sms);
    else if (A.fx) rc = dispatch_fx(sc, A, grid, dim3(2 * bx, nrhs), c->stream);
    else if (p == QCD_F64) rc = dispatch_f64(sc, A, grid, block, c->stream, rv);
    else if (p == QCD_F32) rc = dispatch_f32(sc, A, grid, block, c->stream, rv);
    else if (p == QCD_DF64) rc = dispatch_df64(sc, A, grid, block, c->stream, rv);
    else rc = dispatch_f16(sc, A, grid, block, c->stream, rv);
    if (rc != QCD_OK) return rc;
    QCD_CUDA_CHECK(cudaGetLastError());
    return QCD_OK;
}

}  // namespace qcd
