// lp_fit_f32.cu -- FP32 instantiations of the fit and step kernels.
#include "lp_fit_kern.cuh"

namespace lp {

LP_DEFINE_FIT_LAUNCHERS(float, f32)

namespace {
template <int DIM>
cudaError_t onesided(const FitArgs& a, double* out, int f_real, cudaStream_t s)
{
    const unsigned b = fit_blocks<float>(a);
    if (!onesided_staged(DIM, a.n)) {
        k_onesided<float, DIM, 5><<<b, FIT_THREADS, 0, s>>>(a, out, f_real);
        return cudaGetLastError();
    }
    k_onesided_sides<DIM, 5><<<b, FIT_THREADS, 0, s>>>(a, out, f_real);
    k_onesided_check<DIM, 5><<<b, FIT_THREADS, 0, s>>>(a);
    k_onesided_fill<DIM, 5><<<152u * 4u, FIT_THREADS, 0, s>>>(a, out, f_real);
    return cudaGetLastError();
}
}  // namespace

cudaError_t launch_onesided_f32(int dim, const FitArgs& a, double* out, int f_real, cudaStream_t s)
{
    if (a.n == 0) return cudaSuccess;
    return dim == 3 ? onesided<3>(a, out, f_real, s) : (dim == 2 ? onesided<2>(a, out, f_real, s)
                                                                 : onesided<1>(a, out, f_real, s));
}

}  // namespace lp
