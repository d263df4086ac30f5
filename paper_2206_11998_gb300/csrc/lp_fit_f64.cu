// lp_fit_f64.cu -- FP64 instantiations of the fit and step kernels.
#include "lp_fit_kern.cuh"

namespace lp {

LP_DEFINE_FIT_LAUNCHERS(double, f64)

namespace {

// Particles by falling neighbour count (a counting sort over 0..KMAX).  A warp of
// FP64 fits takes the time of its longest list: in key order a warp of the gas
// cloud has lists of 45 on average and 55 at most, and 24 of 32 lanes at work.
// The longest first, so that the last warps to finish are short ones.
constexpr int ORDER_BINS = KMAX + 1;
__global__ void k_count_bins(int64_t n, const uint32_t* __restrict__ count, unsigned int* bins)
{
    __shared__ unsigned int h[ORDER_BINS];
    for (int q = threadIdx.x; q < ORDER_BINS; q += blockDim.x) h[q] = 0;
    __syncthreads();
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        atomicAdd(&h[KMAX - min(count[i], (uint32_t)KMAX)], 1u);
    __syncthreads();
    for (int q = threadIdx.x; q < ORDER_BINS; q += blockDim.x)
        if (h[q]) atomicAdd(bins + q, h[q]);
}

// (bins: the counts, then one running place per bin)
__global__ void k_count_order(int64_t n, const uint32_t* __restrict__ count, unsigned int* bins, uint32_t* order)
{
    __shared__ unsigned int first[ORDER_BINS];
    if (threadIdx.x == 0) {
        unsigned int run = 0;
        for (int q = 0; q < ORDER_BINS; ++q) { first[q] = run; run += bins[q]; }
    }
    __syncthreads();
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const bool on = i < n;
    const unsigned bin = on ? KMAX - min(count[i], (uint32_t)KMAX) : 0xffffffffu;
    const unsigned peers = __match_any_sync(0xffffffffu, bin);
    const int leader = __ffs(peers) - 1, lane = (int)(threadIdx.x & 31u);
    unsigned int base = 0;
    if (on && lane == leader) base = atomicAdd(bins + ORDER_BINS + bin, (unsigned)__popc(peers));
    base = __shfl_sync(0xffffffffu, base, leader);
    if (on) order[first[bin] + base + __popc(peers & ((1u << lane) - 1u))] = (uint32_t)i;
}

}  // namespace

cudaError_t order_by_count(int64_t n, const uint32_t* count, unsigned int* bins, uint32_t* order, cudaStream_t s)
{
    cudaError_t e = cudaMemsetAsync(bins, 0, 2 * ORDER_BINS * sizeof(unsigned int), s);
    if (e != cudaSuccess) return e;
    const unsigned b = (unsigned)((n + 255) / 256);
    k_count_bins<<<b < 304u ? b : 304u, 256, 0, s>>>(n, count, bins);
    k_count_order<<<b, 256, 0, s>>>(n, count, bins, order);
    return cudaGetLastError();
}

cudaError_t launch_onesided_f64(int dim, const FitArgs& a, double* out, int f_real, cudaStream_t s)
{
    if (a.n == 0) return cudaSuccess;
    const unsigned b = fit_blocks<double>(a);
    if (dim == 3) k_onesided<3, 5><<<b, FitBlock<double>::v, 0, s>>>(a, out, f_real);
    else if (dim == 2) k_onesided<2, 5><<<b, FitBlock<double>::v, 0, s>>>(a, out, f_real);
    else k_onesided<1, 5><<<b, FitBlock<double>::v, 0, s>>>(a, out, f_real);
    return cudaGetLastError();
}

}  // namespace lp
