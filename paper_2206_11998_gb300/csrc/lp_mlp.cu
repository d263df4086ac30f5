// lp_mlp.cu -- the learned state estimator: an 8 -> 32 (ReLU) -> 1 (sigmoid)
// network on stencil features, trained on the GPU from the flags that the
// plain estimator of Sec. 2.1 produces on the method's own runs.
//
// Weights are used in BF16 with FP32 accumulation; FP32 master weights and
// Adam moments live in the context.  Parameter layout (MLP_NPARAM floats):
//   W1[32][8] (row j: hidden unit j), b1[32], w2[32], b2.
// Loss: mean class-weighted binary cross-entropy, weight pos_weight on flagged
// samples.
#include <cuda_bf16.h>
#include <string.h>

#include <type_traits>

#include "lp_mlp.cuh"

namespace lp {
namespace {

__device__ inline float bf(const __nv_bfloat16* w, int i) { return __bfloat162float(w[i]); }

// ---------------------------------------------------------------------------
// Loss and gradient over samples, a block of MT_THREADS.  A warp takes MT_TILE
// samples at a time: forward with two lanes per sample (16 hidden units each),
// backward with a lane per hidden unit, which keeps its unit's ten sums in
// registers over all the samples the warp takes (the unit's activation is
// formed again, eight FMAs, instead of passing 32 values per sample through
// shared memory).  The warps' sums meet in shared memory once per call and go
// to the gradient with one atomic per parameter and block.
// ---------------------------------------------------------------------------
constexpr int MT_THREADS = 256;
constexpr int MT_WARPS = MT_THREADS / 32;
constexpr int MT_TILE = 16;
constexpr int MT_BLOCK = MT_WARPS * MT_TILE;      // samples a block takes at a time
constexpr int MT_ROW = 12;                        // staged sample: x[8], dz, padding
constexpr int MT_HALF = 16 * MLP_IN + 4;          // W1 of 16 units, the halves 4 banks apart

struct MlpShared {
    alignas(16) float W1[2 * MT_HALF];
    float b1[MLP_H], w2[MLP_H], b2;
    alignas(16) float xs[MT_WARPS][MT_TILE][MT_ROW];
    float red[MT_WARPS][MLP_NPARAM + 1];          // per warp: gradient sums, loss
};

// the BF16 value of parameter q into the shared weights
__device__ __forceinline__ void mlp_put(MlpShared& sm, int q, float v)
{
    if (q < OFF_B1) sm.W1[(q / (16 * MLP_IN)) * MT_HALF + q % (16 * MLP_IN)] = v;
    else if (q < OFF_W2) sm.b1[q - OFF_B1] = v;
    else if (q < OFF_B2) sm.w2[q - OFF_W2] = v;
    else sm.b2 = v;
}

struct MlpSample {
    float4 x0, x1;
    float y;
    bool on;
};

// the sample of this lane in tile `tile` of the nb samples at X, y
__device__ __forceinline__ MlpSample mlp_load(const float* __restrict__ X, const float* __restrict__ y, int64_t nb,
                                              int64_t tile)
{
    MlpSample v;
    const int64_t s = tile * MT_TILE + (int64_t)(lane_id() >> 1);
    v.on = s < nb;
    v.x0 = v.x1 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    v.y = 0.0f;
    if (v.on) {
        // (X may lie at any float)
        const float* p = X + s * MLP_IN;
        v.x0 = make_float4(__ldg(p), __ldg(p + 1), __ldg(p + 2), __ldg(p + 3));
        v.x1 = make_float4(__ldg(p + 4), __ldg(p + 5), __ldg(p + 6), __ldg(p + 7));
        v.y = __ldg(y + s);
    }
    return v;
}

// whether the features of the warp's samples are finite (false, too, where their sum overflows)
__device__ __forceinline__ bool mlp_finite(const MlpSample& v)
{
    const float sum = ((v.x0.x + v.x0.y) + (v.x0.z + v.x0.w)) + ((v.x1.x + v.x1.y) + (v.x1.z + v.x1.w));
    return __all_sync(0xffffffffu, fabsf(sum) < INFINITY);
}

// adds the mean loss and its gradient over the nb samples at X, y (mean over
// n_norm) to loss and grad; `first`: this lane's sample of the warp's first tile.
// All threads of the grid's blocks take part; weights in sm.
__device__ void mlp_block_grad(MlpShared& sm, MlpSample first, const float* __restrict__ X,
                               const float* __restrict__ y, int64_t nb, int64_t n_norm, float pos_weight, float* grad,
                               float* loss)
{
    const unsigned lane = lane_id();
    const int w = (int)(threadIdx.x >> 5), half = (int)(lane & 1u);
    const int64_t warps = (int64_t)gridDim.x * MT_WARPS, tiles = (nb + MT_TILE - 1) / MT_TILE;
    const int64_t t0 = (int64_t)blockIdx.x * MT_WARPS + w;
    float (*xs)[MT_ROW] = sm.xs[w];
    const float* W1 = sm.W1 + half * MT_HALF;
    // this lane's unit in the backward pass
    float wu[MLP_IN], gu[MLP_IN];
    const float* Wu = sm.W1 + ((int)lane / 16) * MT_HALF + ((int)lane % 16) * MLP_IN;
#pragma unroll
    for (int k = 0; k < MLP_IN; ++k) { wu[k] = Wu[k]; gu[k] = 0.0f; }
    const float bu = sm.b1[lane], w2u = sm.w2[lane];
    float gb = 0.0f, gw2 = 0.0f, gb2 = 0.0f, ls = 0.0f;
    MlpSample v = first;
    for (int64_t t = t0; t < tiles; t += warps) {
        // (used after the forward pass; taken there, the training took 1.5 % longer)
        const bool finite = mlp_finite(v);
        const float x[MLP_IN] = {v.x0.x, v.x0.y, v.x0.z, v.x0.w, v.x1.x, v.x1.y, v.x1.z, v.x1.w};
        float z = 0.0f;
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            const float4 a0 = *reinterpret_cast<const float4*>(W1 + j * MLP_IN);
            const float4 a1 = *reinterpret_cast<const float4*>(W1 + j * MLP_IN + 4);
            const float wj[MLP_IN] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
            float a = sm.b1[16 * half + j];
#pragma unroll
            for (int k = 0; k < MLP_IN; ++k) a = fmaf(wj[k], x[k], a);
            z = fmaf(sm.w2[16 * half + j], a > 0.0f ? a : 0.0f, z);
        }
        z = sm.b2 + (z + __shfl_xor_sync(0xffffffffu, z, 1));
        float dz = 0.0f;
        if (v.on) {
            const float cw = v.y > 0.5f ? pos_weight : 1.0f;
            // log sigmoid(z) and log(1 - sigmoid(z)) without overflow
            const float p = 1.0f / (1.0f + __expf(-z));
            dz = cw * (p - v.y) / (float)n_norm;
            if (half == 0) {
                const float t1 = log1pf(__expf(-fabsf(z)));
                const float lp_ = z >= 0.0f ? -t1 : z - t1;
                const float lq = z >= 0.0f ? -z - t1 : -t1;
                ls += cw * (-v.y * lp_ - (1.0f - v.y) * lq) / (float)n_norm;
                gb2 += dz;
            }
        }
        float* row = xs[lane >> 1];
        if (half == 0) {
            *reinterpret_cast<float4*>(row) = v.x0;
            row[8] = dz;
        } else {
            *reinterpret_cast<float4*>(row + 4) = v.x1;
        }
        __syncwarp();
        if (t + warps < tiles) v = mlp_load(X, y, nb, t + warps);
        // (a dead unit's dh is 0, and 0 times a feature that is not finite would be NaN:
        // in tiles with such features dead units are left out)
        auto backward = [&](auto careful) {
#pragma unroll 4
            for (int s = 0; s < MT_TILE; ++s) {
                const float4 x0 = *reinterpret_cast<const float4*>(xs[s]);
                const float4 x1 = *reinterpret_cast<const float4*>(xs[s] + 4);
                const float d = xs[s][8];
                const float q[MLP_IN] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
                float a = bu;
#pragma unroll
                for (int k = 0; k < MLP_IN; ++k) a = fmaf(wu[k], q[k], a);
                const bool live = a > 0.0f;
                gw2 = fmaf(d, live ? a : 0.0f, gw2);
                if (decltype(careful)::value && !live) continue;
                const float dh = live ? d * w2u : 0.0f;
                gb += dh;
#pragma unroll
                for (int k = 0; k < MLP_IN; ++k) gu[k] = fmaf(dh, q[k], gu[k]);
            }
        };
        if (finite) backward(std::false_type{});
        else backward(std::true_type{});
        __syncwarp();
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        gb2 += __shfl_xor_sync(0xffffffffu, gb2, o);
        ls += __shfl_xor_sync(0xffffffffu, ls, o);
    }
    float* red = sm.red[w];
#pragma unroll
    for (int k = 0; k < MLP_IN; ++k) red[(int)lane * MLP_IN + k] = gu[k];
    red[OFF_B1 + lane] = gb;
    red[OFF_W2 + lane] = gw2;
    if (lane == 0) { red[OFF_B2] = gb2; red[MLP_NPARAM] = ls; }
    __syncthreads();
    for (int q = threadIdx.x; q <= MLP_NPARAM; q += MT_THREADS) {
        float g = 0.0f;
#pragma unroll
        for (int u = 0; u < MT_WARPS; ++u) g += sm.red[u][q];
        atomicAdd(q < MLP_NPARAM ? grad + q : loss, g);
    }
}

__global__ void __launch_bounds__(MT_THREADS) k_mlp_grad(const float* __restrict__ X, const float* __restrict__ y,
                                                         int64_t n, float pos_weight,
                                                         const __nv_bfloat16* __restrict__ wb, float* grad, float* loss)
{
    __shared__ MlpShared sm;
    for (int q = threadIdx.x; q < MLP_NPARAM; q += MT_THREADS) mlp_put(sm, q, bf(wb, q));
    __syncthreads();
    const MlpSample v = mlp_load(X, y, n, (int64_t)blockIdx.x * MT_WARPS + (threadIdx.x >> 5));
    mlp_block_grad(sm, v, X, y, n, n, pos_weight, grad, loss);
}

__device__ __forceinline__ void adam_update(float g, float& m1, float& m2, float& w, float c1, float c2, float lr,
                                            float beta1, float beta2, float eps)
{
    m1 = beta1 * m1 + (1.0f - beta1) * g;
    m2 = beta2 * m2 + (1.0f - beta2) * g * g;
    w = w - lr * (m1 / c1) / (sqrtf(m2 / c2) + eps);
}

// Whole training in one cooperative launch: every block keeps the weights and
// the Adam state, adds its share of a minibatch's gradient to a buffer in
// global memory, meets the others at a grid barrier and takes the same Adam
// step from the same sums.  One barrier a minibatch: three gradient buffers take
// turns, the next one zeroed (by block 0) while the current one is summed; its
// last readers passed the barrier before.  A minibatch of 8192 samples took a
// launch for the gradient (9.9 us), one for Adam (2.4 us) and the gaps between
// them; what is left is the barrier and the latency of the sums.
struct MlpTrainArgs {
    const float* X;
    const float* y;
    int64_t n, batch;
    int epochs;
    float pos_weight, lr, beta1, beta2, eps;
    float* master;
    float* m1;
    float* m2;
    __nv_bfloat16* wb;
    float* gbuf;                  // [3][MLP_NPARAM + 1], zero: gradient, batch loss
    float* loss;                  // [epochs]: sums of the batch losses
    unsigned int* arrived;        // zero
    long long* step;              // Adam steps taken; written with the weights
    unsigned int* lost;           // set (and ST_TIMEOUT in the status word) where the barrier gave up
    unsigned int* status;
    unsigned int polls;           // reads of the barrier's count before a block gives up (0: at once)
};

__global__ void __launch_bounds__(MT_THREADS) k_mlp_train(MlpTrainArgs a)
{
    __shared__ MlpShared sm;
    __shared__ int lost;
    constexpr int PER = (MLP_NPARAM + MT_THREADS - 1) / MT_THREADS;
    const int tid = (int)threadIdx.x;
    float w[PER], m1[PER], m2[PER];
#pragma unroll
    for (int u = 0; u < PER; ++u) {
        const int q = tid + u * MT_THREADS;
        w[u] = m1[u] = m2[u] = 0.0f;
        if (q < MLP_NPARAM) {
            w[u] = a.master[q];
            m1[u] = a.m1[q];
            m2[u] = a.m2[q];
            mlp_put(sm, q, bf(a.wb, q));
        }
    }
    const long long step0 = *a.step;            // (block 0 writes it after the last barrier)
    // (an earlier launch of the call gave up: the shared copy, since a block of this
    // one may set the flag while others start)
    if (tid == 0) lost = *reinterpret_cast<volatile unsigned int*>(a.lost) != 0u;
    const int64_t t0 = (int64_t)blockIdx.x * MT_WARPS + (tid >> 5);
    auto size = [&](int64_t b0) { return a.n - b0 < a.batch ? a.n - b0 : a.batch; };
    MlpSample v = mlp_load(a.X, a.y, size(0), t0);
    __syncthreads();
    if (lost) return;
    unsigned it = 0;
    for (int ep = 0; ep < a.epochs; ++ep) {
        double total = 0.0;                     // (of block 0's first thread)
        for (int64_t b0 = 0; b0 < a.n; b0 += a.batch, ++it) {
            float* g = a.gbuf + (it % 3u) * (MLP_NPARAM + 1);
            if (blockIdx.x == 0)
                for (int q = tid; q <= MLP_NPARAM; q += MT_THREADS)
                    a.gbuf[((it + 1u) % 3u) * (MLP_NPARAM + 1) + q] = 0.0f;
            const int64_t nb = size(b0);
            mlp_block_grad(sm, v, a.X + b0 * MLP_IN, a.y + b0, nb, nb, a.pos_weight, g, g + MLP_NPARAM);
            // the next minibatch's samples, in flight over the barrier
            const int64_t b1 = b0 + a.batch < a.n ? b0 + a.batch : 0;
            v = mlp_load(a.X + b1 * MLP_IN, a.y + b1, size(b1), t0);
            // (the release is cumulative: it covers the block's sums, ordered before it
            // by the barrier)
            __syncthreads();
            if (tid == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" : : "l"(a.arrived) : "memory");
            const float step = (float)(step0 + (long long)it + 1);
            const float c1 = 1.0f - powf(a.beta1, step), c2 = 1.0f - powf(a.beta2, step);
            if (tid == 0) {
                const unsigned want = (it + 1u) * gridDim.x;
                unsigned polls = 0, seen;
                do
                    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(a.arrived) : "memory");
                while ((int)(seen - want) < 0 && ++polls < a.polls);
                if ((int)(seen - want) < 0 || a.polls == 0u) {
                    lost = 1;
                    atomicOr(a.lost, 1u);
                    atomicOr(a.status, ST_TIMEOUT);
                }
            }
            __syncthreads();
            if (lost) return;
            if (blockIdx.x == 0 && tid == 0) total += (double)__ldcg(g + MLP_NPARAM);
            float gq[PER];
#pragma unroll
            for (int u = 0; u < PER; ++u) gq[u] = tid + u * MT_THREADS < MLP_NPARAM ? __ldcg(g + tid + u * MT_THREADS) : 0.0f;
#pragma unroll
            for (int u = 0; u < PER; ++u) {
                const int q = tid + u * MT_THREADS;
                if (q >= MLP_NPARAM) continue;
                adam_update(gq[u], m1[u], m2[u], w[u], c1, c2, a.lr, a.beta1, a.beta2, a.eps);
                mlp_put(sm, q, __bfloat162float(__float2bfloat16_rn(w[u])));
            }
            __syncthreads();
        }
        if (blockIdx.x == 0 && tid == 0) a.loss[ep] = (float)total;
    }
    if (blockIdx.x != 0) return;
#pragma unroll
    for (int u = 0; u < PER; ++u) {
        const int q = tid + u * MT_THREADS;
        if (q >= MLP_NPARAM) continue;
        a.master[q] = w[u];
        a.m1[q] = m1[u];
        a.m2[q] = m2[u];
        a.wb[q] = __float2bfloat16_rn(w[u]);
    }
    if (tid == 0) *a.step = step0 + (long long)it;
}

// Adam on the FP32 master weights; refreshes the BF16 copy and clears the gradient
constexpr int ADAM_THREADS = 352;
static_assert(ADAM_THREADS >= MLP_NPARAM, "one block, a thread per parameter");
__global__ void __launch_bounds__(ADAM_THREADS) k_mlp_adam(float* master, float* grad, float* m1, float* m2,
                                                           long long* taken, float lr, float beta1, float beta2,
                                                           float eps, __nv_bfloat16* wb)
{
    const int q = (int)threadIdx.x;
    const float step = (float)(*taken + 1);
    __syncthreads();
    if (q == 0) *taken += 1;
    if (q >= MLP_NPARAM) return;
    float w = master[q];
    const float c1 = 1.0f - powf(beta1, step), c2 = 1.0f - powf(beta2, step);
    adam_update(grad[q], m1[q], m2[q], w, c1, c2, lr, beta1, beta2, eps);
    master[q] = w;
    wb[q] = __float2bfloat16_rn(w);
    grad[q] = 0.0f;
}

__global__ void k_mlp_infer(const float* __restrict__ X, int64_t n, const __nv_bfloat16* __restrict__ wb,
                            float* __restrict__ p)
{
    int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (s >= n) return;
    float x[MLP_IN];
#pragma unroll
    for (int k = 0; k < MLP_IN; ++k) x[k] = X[s * MLP_IN + k];
    p[s] = mlp_prob(x, wb);
}

__global__ void k_set_bf16(const float* master, __nv_bfloat16* wb, long long* step)
{
    int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q == 0) *step = 0;
    if (q < MLP_NPARAM) wb[q] = __float2bfloat16_rn(master[q]);
}

}  // namespace
}  // namespace lp

using namespace lp;

// blocks for n samples: one to an SM, so that a cooperative launch fits beside
// nothing else and its barrier stays short
static inline unsigned mlp_blocks(int64_t n)
{
    const int64_t b = (n + MT_BLOCK - 1) / MT_BLOCK;
    return (unsigned)(b < 152 ? b : 152);
}

static inline __nv_bfloat16* wbf(lp_ctx* c) { return static_cast<__nv_bfloat16*>(c->mlp_bf16); }

#define LP_CUDA_MLP(call)                                      \
    do {                                                       \
        if ((call) != cudaSuccess) return LP_ERR_CUDA;         \
    } while (0)

extern "C" {

lp_status lp_mlp_set_params(lp_ctx* c, const float* params)
{
    if (!c || !params) return LP_ERR_ARG;
    LP_CUDA_MLP(cudaMemcpy(c->mlp_master, params, MLP_NPARAM * sizeof(float), cudaMemcpyHostToDevice));
    LP_CUDA_MLP(cudaMemset(c->mlp_m1, 0, MLP_NPARAM * sizeof(float)));
    LP_CUDA_MLP(cudaMemset(c->mlp_m2, 0, MLP_NPARAM * sizeof(float)));
    LP_CUDA_MLP(cudaMemset(c->mlp_grad, 0, MLP_NPARAM * sizeof(float)));
    k_set_bf16<<<2, 256>>>(c->mlp_master, wbf(c), c->mlp_step);
    LP_CUDA_MLP(cudaGetLastError());
    LP_CUDA_MLP(cudaDeviceSynchronize());
    c->mlp_ready = 1;
    c->launches += 1;
    return LP_OK;
}

lp_status lp_mlp_get_params(lp_ctx* c, float* master, float* bf16_as_float)
{
    if (!c) return LP_ERR_ARG;
    LP_CUDA_MLP(cudaDeviceSynchronize());
    if (master) LP_CUDA_MLP(cudaMemcpy(master, c->mlp_master, MLP_NPARAM * sizeof(float), cudaMemcpyDeviceToHost));
    if (bf16_as_float) {
        __nv_bfloat16 h[MLP_NPARAM];
        LP_CUDA_MLP(cudaMemcpy(h, wbf(c), sizeof(h), cudaMemcpyDeviceToHost));
        for (int q = 0; q < MLP_NPARAM; ++q) bf16_as_float[q] = __bfloat162float(h[q]);
    }
    return LP_OK;
}

lp_status lp_mlp_grad(lp_ctx* c, const float* X, const float* y, int64_t n, double pos_weight, float* grad,
                      float* loss, lp_stream stream)
{
    if (!c || !X || !y || !grad || !loss || n < 1) return LP_ERR_ARG;
    if (!c->mlp_ready) return LP_ERR_STATE;
    cudaStream_t s = (cudaStream_t)stream;
    LP_CUDA_MLP(cudaMemsetAsync(grad, 0, MLP_NPARAM * sizeof(float), s));
    LP_CUDA_MLP(cudaMemsetAsync(loss, 0, sizeof(float), s));
    k_mlp_grad<<<mlp_blocks(n), MT_THREADS, 0, s>>>(X, y, n, (float)pos_weight, wbf(c), grad, loss);
    c->launches += 1;
    return cudaGetLastError() == cudaSuccess ? LP_OK : LP_ERR_CUDA;
}

lp_status lp_mlp_train(lp_ctx* c, const float* X, const float* y, int64_t n, int32_t epochs, int32_t batch,
                       double lr, double pos_weight, float* epoch_loss, lp_stream stream)
{
    if (!c || !X || !y || n < 1 || epochs < 1 || batch < 1 || !(lr > 0.0)) return LP_ERR_ARG;
    if (!c->mlp_ready) return LP_ERR_STATE;
    cudaStream_t s = (cudaStream_t)stream;
    MlpTrainArgs a;
    a.X = X; a.y = y; a.n = n; a.batch = batch;
    a.pos_weight = (float)pos_weight; a.lr = (float)lr; a.beta1 = 0.9f; a.beta2 = 0.999f; a.eps = 1e-8f;
    a.master = c->mlp_master; a.m1 = c->mlp_m1; a.m2 = c->mlp_m2; a.wb = wbf(c);
    a.lost = reinterpret_cast<unsigned int*>(c->mlp_work);
    a.loss = c->mlp_work + 1;
    a.gbuf = a.loss + MLP_EPOCHS;
    a.arrived = reinterpret_cast<unsigned int*>(a.gbuf + 3 * (MLP_NPARAM + 1));
    a.status = reinterpret_cast<unsigned int*>(c->counters + C_STATUS);
    a.step = c->mlp_step;
    a.polls = c->mlp_polls;
    const int64_t nbatches = (n + batch - 1) / batch, most = n < batch ? n : batch;
    // launches of at most MLP_EPOCHS epochs, whose losses the work area holds
    for (int32_t e0 = 0; e0 < epochs; e0 += MLP_EPOCHS) {
        a.epochs = epochs - e0 < MLP_EPOCHS ? epochs - e0 : MLP_EPOCHS;
        // (the barrier counts in 32 bits, compared modulo 2^32; the flag stays set
        // over the launches of one call, so that none trains on after one gave up)
        const int kept = e0 > 0 ? 1 : 0;
        LP_CUDA_MLP(cudaMemsetAsync(c->mlp_work + kept, 0, (MLP_WORK - kept) * sizeof(float), s));
        void* args[] = {&a};
        LP_CUDA_MLP(cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(k_mlp_train), dim3(mlp_blocks(most)),
                                                dim3(MT_THREADS), args, 0, s));
        c->launches += 1;
        if (epoch_loss) {
            float h[1 + MLP_EPOCHS];                 // the flag, the losses
            LP_CUDA_MLP(cudaMemcpyAsync(h, c->mlp_work, (size_t)(1 + a.epochs) * sizeof(float), cudaMemcpyDeviceToHost,
                                        s));
            LP_CUDA_MLP(cudaStreamSynchronize(s));
            unsigned int lost;                       // (its bits: as a float 1 is denormal, and may compare equal to 0)
            memcpy(&lost, h, sizeof(lost));
            if (lost != 0u) return LP_ERR_TIMEOUT;
            for (int32_t e = 0; e < a.epochs; ++e) epoch_loss[e0 + e] = h[1 + e] / (float)nbatches;
        }
    }
    return LP_OK;
}

lp_status lp_mlp_wait_limit(lp_ctx* c, uint32_t polls)
{
    if (!c) return LP_ERR_ARG;
    c->mlp_polls = polls;
    return LP_OK;
}

lp_status lp_mlp_adam_step(lp_ctx* c, const float* grad, double lr, lp_stream stream)
{
    if (!c || !grad || !(lr > 0.0)) return LP_ERR_ARG;
    if (!c->mlp_ready) return LP_ERR_STATE;
    cudaStream_t s = (cudaStream_t)stream;
    LP_CUDA_MLP(cudaMemcpyAsync(c->mlp_grad, grad, MLP_NPARAM * sizeof(float), cudaMemcpyDeviceToDevice, s));
    k_mlp_adam<<<1, ADAM_THREADS, 0, s>>>(c->mlp_master, c->mlp_grad, c->mlp_m1, c->mlp_m2, c->mlp_step, (float)lr, 0.9f,
                                 0.999f, 1e-8f, wbf(c));
    c->launches += 1;
    return cudaGetLastError() == cudaSuccess ? LP_OK : LP_ERR_CUDA;
}

lp_status lp_mlp_infer(lp_ctx* c, const float* X, int64_t n, float* p, lp_stream stream)
{
    if (!c || !X || !p || n < 0) return LP_ERR_ARG;
    if (!c->mlp_ready) return LP_ERR_STATE;
    if (n == 0) return LP_OK;
    k_mlp_infer<<<(unsigned)((n + 255) / 256), 256, 0, (cudaStream_t)stream>>>(X, n, wbf(c), p);
    c->launches += 1;
    return cudaGetLastError() == cudaSuccess ? LP_OK : LP_ERR_CUDA;
}

}  // extern "C"
