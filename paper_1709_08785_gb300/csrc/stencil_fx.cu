// The FP64 and DF64 stencil kernels in fixed point (stencil_fx.cuh): the modes
// of stencil_impl.cuh with two threads a site.
#include "stencil_fx.cuh"

namespace qcd {

namespace {

// where the result goes: out in P, out as a fixed-point field, or the caller's
// canonical complex128 vectors, on a 16-byte boundary or off it
enum { TO_P = 0, TO_FX = 1, TO_CANON = 2, TO_CANON8 = 3 };

template <int P, int MODE, int RED, bool DAG, int OUT>
__device__ __forceinline__ void fx_body(const StencilArgs &A)
{
    using T = typename Prec<P>::T;
    pdl_enter();
    const bool lead = blockIdx.x == 0 && threadIdx.x == 0 && threadIdx.y == 0;
    if (A.done && *A.done) {
        if (A.skip && lead) *A.skip = 1;
        return;
    }
    if (A.skip && lead) *A.skip = 0;
    const int r = threadIdx.y, a = fx_row();
    const int site = blockIdx.x * (blockDim.x >> 1) + fx_site();
    // a thread past the lattice takes part in the exchanges at the last site
    // and neither stores nor sums
    const bool live = site < A.g.Vh;
    const int cb = live ? site : A.g.Vh - 1;
    auto vec = [&](const SpinorPtr &v) { return rhs_ptr(v, r, A.rhs_stride, A.norm_stride); };
    double red[4] = {0.0, 0.0, 0.0, 0.0};
    HalfSp<long long> acc;
    int E;
    fx_hop<DAG, MODE == M_MULT || MODE == M_DHAT, false>(A.g, A.U, A.C, vec(A.in), A.out_par, cb, a, acc, E);
    if constexpr (OUT == TO_FX) {
        HalfSp<fx2> o;
        fx_normalise(acc, E);
        fx_split(acc, o);
        if (live) fx_store_half(vec(A.out), cb, a, o, E);
        return;
    }
    HalfSp<T> v;
    fx_to_half(acc, E, v);
    HalfSp<T> y;
    if constexpr (MODE != M_HOP && MODE != M_MULT) {
        if (A.y_fx) fx_load_half(vec(A.y), cb, a, y);
        else load_half<P>(vec(A.y), cb, a, y);
    }
    if constexpr (MODE == M_DHAT || MODE == M_FULL) {
        HalfSp<T> fy = y;
        if constexpr (MODE == M_FULL) fx_clover_half(A.C, A.out_par, cb, a, fy);
        axpby_half(v, T(A.cc), v, T(A.a), fy);
        if (A.has_z) {
            HalfSp<T> z;
            load_half<P>(vec(A.z), cb, a, z);
            axpby_half(v, T(1), v, T(A.d), z);
        }
        if constexpr (RED == R_OMEGA) {  // <out|aux>, |out|^2 (aux is usually y)
            if (A.aux.p != A.y.p) load_half<P>(vec(A.aux), cb, a, y);
            if (live) {
                dot_half(v, y, red[0], red[1]);
                norm_half(v, red[2]);
            }
        }
    } else if constexpr (MODE == M_SRC) {
        axpby_half(v, T(A.cc), v, T(A.a), y);
        fx_clover_half(A.C, A.out_par, cb, a, v);
    } else if constexpr (MODE == M_RECON) {
        // x_o = F^-1 u, u = b_o + kappa H_oe x_e, and the odd rows of the residual,
        // u - F x_o, from the same hopping term
        axpby_half(v, T(A.cc), v, T(A.a), y);  // u
        y = v;
        fx_clover_half(A.C, A.out_par, cb, a, y);
        if (live) store_half<P>(vec(A.out), cb, a, y);
        fx_clover_half(A.Cf, A.out_par, cb, a, y);  // F x_o
        axpby_half(v, T(1), v, T(-1), y);
    }
    if constexpr (RED == R_DOT_AUX) {  // <aux|out>
        load_half<P>(vec(A.aux), cb, a, y);
        if (live) dot_half(y, v, red[0], red[1]);
    } else if constexpr (RED == R_NORM) {
        if (live) norm_half(v, red[0]);
    }
    if constexpr (RED != R_NONE) grid_reduce<RED == R_OMEGA ? 3 : RED == R_DOT_AUX ? 2 : 1>(red, A.red);
    if constexpr (MODE == M_RECON) return;
    if (!live) return;
    if constexpr (OUT == TO_CANON || OUT == TO_CANON8) {
        // 16 bytes a lane; the six stores of a warp cover its 16 sites' 3 KB (off the
        // 16-byte boundary the same numbers in halves)
        double *o = (double *)A.canon + r * A.canon_stride + (size_t)cb * 24;
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            const cx<T> z = j < 3 ? v.u[j] : v.d[j - 3];
            double *to = o + 2 * fx_comp(a, j / 3, j % 3);
            if constexpr (OUT == TO_CANON) {
                *(double2 *)to = make_double2(to_d(z.r), to_d(z.i));
            } else {
                to[0] = to_d(z.r);
                to[1] = to_d(z.i);
            }
        }
    } else {
        store_half<P>(vec(A.out), cb, a, v);
    }
}

// 168 registers asked for, not only allowed: three blocks of 128 threads an SM
// either way, but under a launch bound the compiler takes 150-odd and moves the
// next hop's loads down to their use (MULT at 24^3x48 319 us against 174; 160: 205,
// 176 registers, eight warps fewer: 207).  With it, before the two threads a site
// and the prefetch: MULT 260 -> 174 us, FP64 source pass 347 -> 263, residual 381 ->
// 258, float-pair second halves 328 / 368 -> 229 / 282.
template <int P, int MODE, int RED, bool DAG, int OUT>
__global__ void __maxnreg__(168) fx_kernel(StencilArgs A)
{
    fx_body<P, MODE, RED, DAG, OUT>(A);
}

template <int P>
int dispatch_fx_p(const StencilCall &sc, const StencilArgs &A, dim3 grid, dim3 block, cudaStream_t s)
{
#define QCD_CASE(MODE, RED)                                                                              \
    if (sc.mode == MODE && sc.red == RED) {                                                              \
        launch_pdl(fx_kernel<P, MODE, RED, false, TO_P>, grid, block, 0, s, A);                          \
        return QCD_OK;                                                                                   \
    }
    QCD_CASE(M_DHAT, R_NONE)
    QCD_CASE(M_DHAT, R_DOT_AUX)
    QCD_CASE(M_DHAT, R_OMEGA)
    QCD_CASE(M_DHAT, R_NORM)
    QCD_CASE(M_SRC, R_NONE)
    QCD_CASE(M_SRC, R_NORM)
    QCD_CASE(M_FULL, R_NONE)
    QCD_CASE(M_FULL, R_NORM)
    QCD_CASE(M_FULL, R_DOT_AUX)
    QCD_CASE(M_FULL, R_OMEGA)
    if constexpr (P == QCD_F64) {  // the FP64 reconstruction with its residual
        QCD_CASE(M_RECON, R_NORM)
    }
#undef QCD_CASE
    set_error_message("unsupported stencil mode %d / reduction %d", sc.mode, sc.red);
    return QCD_EINVAL;
}

}  // namespace

// block.x: two threads a site.  The hopping term and MULT are the same in FP64
// and DF64: to canonical vectors, or MULT (the first half of D^) to a fixed-point field.
int dispatch_fx(const StencilCall &sc, const StencilArgs &A, dim3 grid, dim3 block, cudaStream_t s)
{
#define QCD_OUT(MODE, DAG, OUT) launch_pdl(fx_kernel<QCD_F64, MODE, R_NONE, DAG, OUT>, grid, block, 0, s, A)
#define QCD_CANON(MODE, DAG)                                    \
    do {                                                        \
        if ((size_t)A.canon % 16) QCD_OUT(MODE, DAG, TO_CANON8); \
        else QCD_OUT(MODE, DAG, TO_CANON);                      \
        return QCD_OK;                                          \
    } while (0)
    if (sc.red == R_NONE && (sc.mode == M_HOP || sc.mode == M_MULT)) {
        if (A.canon) {
            if (sc.mode == M_MULT && sc.dagger) QCD_CANON(M_MULT, true);
            if (sc.mode == M_MULT) QCD_CANON(M_MULT, false);
            if (sc.dagger) QCD_CANON(M_HOP, true);
            QCD_CANON(M_HOP, false);
        }
        if (sc.mode == M_MULT && !sc.dagger && sc.out.prec == QCD_FX) {
            QCD_OUT(M_MULT, false, TO_FX);
            return QCD_OK;
        }
        set_error_message("the FP64 and DF64 hopping terms give canonical vectors, MULT fixed-point fields too");
        return QCD_EINVAL;
    }
    if (sc.dagger) {
        set_error_message("dagger is only available for the hopping and MULT kernels");
        return QCD_EINVAL;
    }
    if (A.canon && sc.mode == M_DHAT) QCD_CANON(M_DHAT, false);
    if (A.canon && sc.mode == M_FULL) QCD_CANON(M_FULL, false);
#undef QCD_CANON
#undef QCD_OUT
    return sc.prec == QCD_DF64 ? dispatch_fx_p<QCD_DF64>(sc, A, grid, block, s)
                               : dispatch_fx_p<QCD_F64>(sc, A, grid, block, s);
}

}  // namespace qcd
