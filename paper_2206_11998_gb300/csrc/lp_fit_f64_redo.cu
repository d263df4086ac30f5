// lp_fit_f64_redo.cu -- the FP64 redo of the stencils the FP32 pass listed.
#include "lp_fit_redo.cuh"

namespace lp {

namespace {
constexpr unsigned REDO_BLOCKS = 152u * 4u;
}

cudaError_t launch_step_redo(int dim, const FitArgs& a, const StepOut& o, cudaStream_t s)
{
    const bool gate = o.features || a.c.estimator == LP_EST_MLP;
    if (dim == 3) {
        if (gate) k_step_redo<3, true><<<REDO_BLOCKS, FIT_THREADS, 0, s>>>(a, o);
        else k_step_redo<3, false><<<REDO_BLOCKS, FIT_THREADS, 0, s>>>(a, o);
    } else if (dim == 2) {
        if (gate) k_step_redo<2, true><<<REDO_BLOCKS, FIT_THREADS, 0, s>>>(a, o);
        else k_step_redo<2, false><<<REDO_BLOCKS, FIT_THREADS, 0, s>>>(a, o);
    } else {
        if (gate) k_step_redo<1, true><<<REDO_BLOCKS, FIT_THREADS, 0, s>>>(a, o);
        else k_step_redo<1, false><<<REDO_BLOCKS, FIT_THREADS, 0, s>>>(a, o);
    }
    return cudaGetLastError();
}

cudaError_t launch_derivs_redo(int dim, int F, const FitArgs& a, const DerivOut& o, cudaStream_t s)
{
    if (dim == 3 && F == 1) k_derivs_redo<3, 1><<<REDO_BLOCKS, FIT_THREADS, 0, s>>>(a, o);
    else if (dim == 3) k_derivs_redo<3, 5><<<REDO_BLOCKS, FIT_THREADS, 0, s>>>(a, o);
    else if (dim == 2) k_derivs_redo<2, 5><<<REDO_BLOCKS, FIT_THREADS, 0, s>>>(a, o);
    else k_derivs_redo<1, 5><<<REDO_BLOCKS, FIT_THREADS, 0, s>>>(a, o);
    return cudaGetLastError();
}

cudaError_t launch_onesided_redo(int dim, const FitArgs& a, double* out, int f_real, cudaStream_t s)
{
    if (dim == 3) k_onesided_redo<3, 5><<<REDO_BLOCKS, FIT_THREADS, 0, s>>>(a, out, f_real);
    else if (dim == 2) k_onesided_redo<2, 5><<<REDO_BLOCKS, FIT_THREADS, 0, s>>>(a, out, f_real);
    else k_onesided_redo<1, 5><<<REDO_BLOCKS, FIT_THREADS, 0, s>>>(a, out, f_real);
    return cudaGetLastError();
}

}  // namespace lp
