// lp_fit_f64.cu -- FP64 instantiations of the fit and step kernels (32-thread
// blocks), and the order of particles by cost that they run in.
#include "lp_fit_kern.cuh"

namespace lp {

LP_DEFINE_FIT_LAUNCHERS(double, f64)

namespace {

// Particles by falling cost (a counting sort).  A warp of FP64 fits takes the
// time of its longest list: in key order a warp of the gas cloud has lists of 45
// on average and 55 at most, and 24 of 32 lanes at work.  The fits that will take
// the correction pass, a second pass over the list, come first, by list length:
// they are 4 % of that cloud, and one of them made its whole warp run the pass
// in three warps of four.  They are told by the FP32 ratio (20 us at 60k; a wrong
// guess near the threshold only costs its warp).  The longest first, so that
// the last warps to finish are short ones.
constexpr int COST_MAX = 2 * KMAX + 1;            // list length, plus KMAX + 1 with the pass
constexpr int ORDER_BINS = COST_MAX + 1;

template <int DIM>
__global__ void __launch_bounds__(FIT_THREADS, 5) k_cost(FitArgs a, uint32_t* cost, unsigned int* bins)
{
    __shared__ uint32_t stage[64][NB_PITCH];
    __shared__ unsigned int h[ORDER_BINS];
    for (int q = threadIdx.x; q < ORDER_BINS; q += blockDim.x) h[q] = 0;
    __syncthreads();
    const bool guess = a.c.refine == LP_REFINE_AUTO;
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (guess) stage_rows<64>(stage, a.idx, a.c.k_max, i < a.n ? i : -1);
    if (i < a.n) {
        const int cnt = (int)a.count[i];
        uint32_t k = (uint32_t)min(cnt, KMAX);
        if (guess && cnt >= NU<DIM>::v) {
            Src<float, DIM, 1> src(a, i);
            const NbStaged<64> nb{a.idx + i * (int64_t)a.c.k_max, &stage[0][threadIdx.x]};
            if (gram_ratio(src, nb, cnt, inv_scale(last_d2(src, nb, cnt))) < (float)a.c.refine_ratio)
                k += KMAX + 1;
        }
        cost[i] = COST_MAX - k;
        atomicAdd(&h[COST_MAX - k], 1u);
    }
    __syncthreads();
    for (int q = threadIdx.x; q < ORDER_BINS; q += blockDim.x)
        if (h[q]) atomicAdd(bins + q, h[q]);
}

// (bins: the counts, then one running place per bin)
__global__ void k_cost_order(int64_t n, const uint32_t* __restrict__ cost, unsigned int* bins, uint32_t* order)
{
    __shared__ unsigned int first[ORDER_BINS];
    if (threadIdx.x < 32) {                       // exclusive sums of the counts, 32 bins at a time
        unsigned int run = 0;
        for (int q0 = 0; q0 < ORDER_BINS; q0 += 32) {
            const int q = q0 + (int)threadIdx.x;
            const unsigned int v = q < ORDER_BINS ? bins[q] : 0u;
            unsigned int x = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned int y = __shfl_up_sync(0xffffffffu, x, o);
                if ((int)threadIdx.x >= o) x += y;
            }
            if (q < ORDER_BINS) first[q] = run + x - v;
            run += __shfl_sync(0xffffffffu, x, 31);
        }
    }
    __syncthreads();
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const bool on = i < n;
    const unsigned bin = on ? cost[i] : 0xffffffffu;
    const unsigned peers = __match_any_sync(0xffffffffu, bin);
    const int leader = __ffs(peers) - 1, lane = (int)(threadIdx.x & 31u);
    unsigned int base = 0;
    if (on && lane == leader) base = atomicAdd(bins + ORDER_BINS + bin, (unsigned)__popc(peers));
    base = __shfl_sync(0xffffffffu, base, leader);
    if (on) order[first[bin] + base + __popc(peers & ((1u << lane) - 1u))] = (uint32_t)i;
}

}  // namespace

cudaError_t order_by_cost(int dim, const FitArgs& a, unsigned int* bins, uint32_t* cost, uint32_t* order, cudaStream_t s)
{
    cudaError_t e = cudaMemsetAsync(bins, 0, 2 * ORDER_BINS * sizeof(unsigned int), s);
    if (e != cudaSuccess) return e;
    const unsigned b = fit_blocks<float>(a);
    if (dim == 3) k_cost<3><<<b, FIT_THREADS, 0, s>>>(a, cost, bins);
    else if (dim == 2) k_cost<2><<<b, FIT_THREADS, 0, s>>>(a, cost, bins);
    else k_cost<1><<<b, FIT_THREADS, 0, s>>>(a, cost, bins);
    k_cost_order<<<(unsigned)((a.n + 255) / 256), 256, 0, s>>>(a.n, cost, bins, order);
    return cudaGetLastError();
}

cudaError_t launch_onesided_f64(int dim, const FitArgs& a, double* out, int f_real, cudaStream_t s)
{
    if (a.n == 0) return cudaSuccess;
    const unsigned b = fit_blocks<double>(a);
    if (dim == 3) k_onesided<double, 3, 5><<<b, FitBlock<double>::v, 0, s>>>(a, out, f_real);
    else if (dim == 2) k_onesided<double, 2, 5><<<b, FitBlock<double>::v, 0, s>>>(a, out, f_real);
    else k_onesided<double, 1, 5><<<b, FitBlock<double>::v, 0, s>>>(a, out, f_real);
    return cudaGetLastError();
}

}  // namespace lp
