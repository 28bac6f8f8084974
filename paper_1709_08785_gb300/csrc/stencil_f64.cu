// The stencil kernels instantiated for FP64 storage and arithmetic.
#include "stencil_impl.cuh"

namespace qcd {

int dispatch_f64(const StencilCall &sc, const StencilArgs &A, dim3 grid, dim3 block, cudaStream_t s, int v)
{
    return dispatch<QCD_F64>(sc, A, grid, block, s, v);
}

// fixed point in, fixed point out: the hopping term and MULT
int dispatch_fxout(const StencilCall &sc, const StencilArgs &A, dim3 grid, dim3 block, cudaStream_t s)
{
    if (sc.mode == M_MULT) {
        if (sc.dagger) launch_pdl(stencil_kernel_fxout<M_MULT, true>, grid, block, 0, s, A);
        else launch_pdl(stencil_kernel_fxout<M_MULT, false>, grid, block, 0, s, A);
    } else {
        if (sc.dagger) launch_pdl(stencil_kernel_fxout<M_HOP, true>, grid, block, 0, s, A);
        else launch_pdl(stencil_kernel_fxout<M_HOP, false>, grid, block, 0, s, A);
    }
    return QCD_OK;
}

}  // namespace qcd
