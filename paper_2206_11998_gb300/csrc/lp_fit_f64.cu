// lp_fit_f64.cu -- FP64 instantiations of the fit and step kernels.
#include "lp_fit_kern.cuh"

namespace lp {

LP_DEFINE_FIT_LAUNCHERS(double, f64)

cudaError_t launch_onesided_f64(int dim, const FitArgs& a, double* out, int f_real, cudaStream_t s)
{
    if (a.n == 0) return cudaSuccess;
    const unsigned b = fit_blocks(a);
    if (dim == 3) k_onesided<3, 5><<<b, FIT_THREADS, 0, s>>>(a, out, f_real);
    else if (dim == 2) k_onesided<2, 5><<<b, FIT_THREADS, 0, s>>>(a, out, f_real);
    else k_onesided<1, 5><<<b, FIT_THREADS, 0, s>>>(a, out, f_real);
    return cudaGetLastError();
}

}  // namespace lp
