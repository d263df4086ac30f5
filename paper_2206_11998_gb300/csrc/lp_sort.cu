// lp_sort.cu -- Sec. 2.2 steps 2-3 on the GPU: bounding cube, Morton (Z-curve)
// keys, LSD radix sort, gather of the state into key order, and the per-level
// cell tables that stand in for the paper's octree.
#include <string.h>

#include <mutex>

#include "lp_internal.cuh"

namespace lp {

namespace {

constexpr int RS_THREADS = 256;
constexpr int RS_ITEMS = 8;
constexpr int RS_TILE = RS_THREADS * RS_ITEMS;
static_assert(RS_TILE == RS_TILE_KEYS, "the histogram is sized for this tile");
static_assert(RS_BINS == 2 * RS_THREADS, "each thread owns two digits of the histogram");
constexpr uint32_t RS_MASK = RS_BINS - 1;


__device__ inline double from_order_key(unsigned long long k)
{
    uint64_t b = (k & 0x8000000000000000ull) ? (k & 0x7fffffffffffffffull) : ~k;
    return __longlong_as_double((long long)b);
}

constexpr int EXT_ITEMS = 16;

// order key of the double with bit pattern b (order_key without FP64
// instructions), and whether b is a NaN (NaNs take no part in an extent, as
// with fmin / fmax)
__device__ __forceinline__ uint64_t order_key_bits(uint64_t b)
{
    if ((b << 1) == 0) b = 0;                   // -0 as +0
    return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}
__device__ __forceinline__ bool is_nan_bits(uint64_t b) { return (b & 0x7fffffffffffffffull) > 0x7ff0000000000000ull; }

constexpr uint64_t KEY_POS_INF = 0xfff0000000000000ull;   // order_key(+inf)
constexpr uint64_t KEY_NEG_INF = 0x000fffffffffffffull;   // order_key(-inf)

// extent of one run of particles, as order keys: lo[k], hi[k] of the
// coordinates and wlo, whi of m V
struct ExtKeys {
    uint64_t lo[3], hi[3], wlo, whi;
    __device__ __forceinline__ void init()
    {
#pragma unroll
        for (int k = 0; k < 3; ++k) { lo[k] = KEY_POS_INF; hi[k] = KEY_NEG_INF; }
        wlo = KEY_POS_INF;
        whi = KEY_NEG_INF;
    }
    template <int DIM>
    __device__ __forceinline__ void add(const double* const (&xs)[3], int64_t i)
    {
#pragma unroll
        for (int k = 0; k < DIM; ++k) {
            const uint64_t b = (uint64_t)__double_as_longlong(xs[k][i]);
            if (is_nan_bits(b)) continue;
            const uint64_t q = order_key_bits(b);
            lo[k] = q < lo[k] ? q : lo[k];
            hi[k] = q > hi[k] ? q : hi[k];
        }
    }
    __device__ __forceinline__ void add_w(double w)
    {
        const uint64_t bw = (uint64_t)__double_as_longlong(w);
        if (!is_nan_bits(bw)) {
            const uint64_t q = order_key_bits(bw);
            wlo = q < wlo ? q : wlo;
            whi = q > whi ? q : whi;
        }
    }
    template <int DIM>
    __device__ void flush(unsigned long long* e) const
    {
#pragma unroll
        for (int k = 0; k < DIM; ++k) {
            atomicMin(e + k, (unsigned long long)lo[k]);
            atomicMax(e + 3 + k, (unsigned long long)hi[k]);
        }
    }
    __device__ void flush_w(unsigned long long* e) const
    {
        atomicMin(e + 6, (unsigned long long)wlo);
        atomicMax(e + 7, (unsigned long long)whi);
    }
};

// the m V extent of the particles of a block (gather order, simulations
// kept together), to ext[8 s + 6..7] of their simulation s: reduced over each
// warp whose particles share a simulation, then over the block when all its
// warps do (one pair of atomics per block: the extent words are the same few
// addresses for every block, so their atomics would otherwise queue);
// atomics per warp or per lane otherwise.  Every thread of the block calls it
// (valid: this thread has a particle); blockDim.x <= 32 * EXT_WARPS.
constexpr int EXT_WARPS = 8;
__device__ __forceinline__ void block_w_extent(bool valid, double w, uint32_t sim, unsigned long long* ext)
{
    __shared__ uint64_t swlo[EXT_WARPS], swhi[EXT_WARPS];
    __shared__ uint32_t ssim[EXT_WARPS];
    ExtKeys r;
    r.init();
    if (valid) r.add_w(w);
    else sim = 0xffffffffu;
    const uint32_t s0 = __shfl_sync(0xffffffffu, sim, 0);
    const bool uniform = __all_sync(0xffffffffu, sim == s0 || sim == 0xffffffffu);
    const unsigned wid = threadIdx.x >> 5;
    if (uniform) {
        for (int o = 16; o > 0; o >>= 1) {
            const uint64_t a = __shfl_xor_sync(0xffffffffu, r.wlo, o);
            const uint64_t b = __shfl_xor_sync(0xffffffffu, r.whi, o);
            r.wlo = a < r.wlo ? a : r.wlo;
            r.whi = b > r.whi ? b : r.whi;
        }
    } else if (sim != 0xffffffffu) {
        r.flush_w(ext + 8 * (int64_t)sim);                  // a warp across simulations
    }
    if (lane_id() == 0) {
        ssim[wid] = uniform ? s0 : 0xfffffffeu;             // 0xfffffffe: flushed already
        swlo[wid] = r.wlo;
        swhi[wid] = r.whi;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const int nw = (int)((blockDim.x + 31) / 32);
        uint32_t sb = 0xffffffffu;
        bool one = true;
        for (int q = 0; q < nw; ++q) {
            const uint32_t sq = ssim[q];
            if (sq == 0xffffffffu) continue;                // no particle
            if (sq == 0xfffffffeu || (sb != 0xffffffffu && sq != sb)) { one = false; break; }
            sb = sq;
        }
        if (one) {
            if (sb != 0xffffffffu) {
                ExtKeys t;
                t.init();
                for (int q = 0; q < nw; ++q)
                    if (ssim[q] == sb) {
                        t.wlo = swlo[q] < t.wlo ? swlo[q] : t.wlo;
                        t.whi = swhi[q] > t.whi ? swhi[q] : t.whi;
                    }
                t.flush_w(ext + 8 * (int64_t)sb);
            }
        } else {
            for (int q = 0; q < nw; ++q) {
                ExtKeys t;
                t.init();
                t.wlo = swlo[q];
                t.whi = swhi[q];
                if (ssim[q] < 0xfffffffeu) t.flush_w(ext + 8 * (int64_t)ssim[q]);
            }
        }
    }
}

__global__ void k_init_extent(unsigned long long* ext, int nsim, unsigned int* ticket)
{
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t == 0) *ticket = 0u;
    if (t < 8 * nsim) {
        int w = t & 7;
        ext[t] = (w < 3 || w == 6) ? ~0ull : 0ull;
    }
}

// Bounding cube of a simulation (what the keys need) from its extent lo, hi
// (order keys).
__device__ inline void finalize_cube(const DevCfg& c, const unsigned long long (&lo)[3],
                                     const unsigned long long (&hi)[3], Grid* g)
{
    double L = 0.0, org[3] = {0.0, 0.0, 0.0};
    for (int k = 0; k < c.dim; ++k) {
        double ext_k;
        if (c.periodic[k]) { org[k] = c.box_lo[k]; ext_k = c.Lper[k]; }
        else { org[k] = from_order_key(lo[k]); ext_k = __dsub_rn(from_order_key(hi[k]), org[k]); }
        L = fmax(L, ext_k);
    }
    if (!(L > 0.0)) L = 1.0;
    g->L = L;
    g->inv = __ddiv_rn(ldexp(1.0, c.mbits), L);
    for (int k = 0; k < 3; ++k) {
        g->lo[k] = org[k];
        split(org[k], g->lo_h[k], g->lo_l[k]);
    }
    g->inv_f = (float)g->inv;
    g->L_f = (float)L;
}

// one particle's entries of the cell tables (see k_tables)
struct TableArgs {
    int dim, mbits;
    int64_t n;                    // 0: no tables
    const uint64_t* keys;
    const int* grange;
    const int64_t* level_off;
    unsigned long long* cells;
};
template <bool CLEAR>
__device__ __forceinline__ void table_entries(const TableArgs& a, int64_t i)
{
    const uint64_t k = a.keys[i];
    const uint64_t kp = i > 0 ? a.keys[i - 1] : 0;
    const uint64_t kn = i + 1 < a.n ? a.keys[i + 1] : 0;
    uint32_t* half = reinterpret_cast<uint32_t*>(a.cells);
    for (int l = a.grange[0]; l <= a.grange[1]; ++l) {
        const int sh = a.dim * (a.mbits - l);
        const uint64_t c = k >> sh;
        const bool first = i == 0 || (kp >> sh) != c;
        const int64_t e = a.level_off[l] + (int64_t)c;
        if (CLEAR) {
            if (first) a.cells[e] = 0ull;
        } else {
            const bool last = i + 1 == a.n || (kn >> sh) != c;
            if (first) half[2 * e] = (uint32_t)i;
            if (last) half[2 * e + 1] = (uint32_t)(i + 1);
        }
    }
}

// The start of a build: the last build's table entries cleared (old), and the
// extent of the positions, ext[8 s + 0..2] min x_k, [8 s + 3..5] max x_k (order
// keys) of simulation s, from which the last block to finish forms the bounding
// cubes (the extent of m V, ext[8 s + 6..7], is taken by the gather, which
// reads m and V anyway: the keys need only the positions).  The extent words
// are at their initial values on entry and are put back for the next build.
// One simulation: grid-stride accumulation and a warp reduction; several:
// EXT_ITEMS particles per thread, reduced over the warp when the warp's
// particles share a simulation (they are stored by simulation), with atomics
// per run otherwise.  The comparisons are integer ones on the order keys (FP64
// min / max would run on the scarce FP64 units).  As kernels of their own the
// clearing, the words' initialisation and the cubes cost a launch each (2 to 3
// us, and as much between launches).
template <int DIM>
__global__ void k_begin(int64_t n, const double* __restrict__ x0, const double* __restrict__ x1,
                        const double* __restrict__ x2, const uint32_t* __restrict__ sim_of, unsigned long long* ext,
                        DevCfg c, int nsim, Grid* grids, unsigned int* ticket, TableArgs old)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < old.n; i += (int64_t)gridDim.x * blockDim.x)
        table_entries<true>(old, i);
    ExtKeys r;
    r.init();
    const double* const xs[3] = {x0, x1, x2};
    uint32_t sim = 0;
    if (!sim_of) {
        for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
            r.add<DIM>(xs, i);
    } else {
        // EXT_ITEMS particles per thread (strided by the block size, so loads
        // stay coalesced); a change of simulation flushes the running extent
        sim = 0xffffffffu;
        const int64_t base = (int64_t)blockIdx.x * blockDim.x * EXT_ITEMS + threadIdx.x;
        for (int q = 0; q < EXT_ITEMS; ++q) {
            const int64_t i = base + (int64_t)q * blockDim.x;
            if (i >= n) break;
            const uint32_t si = sim_of[i];
            if (si != sim) {
                if (sim != 0xffffffffu) r.flush<DIM>(ext + 8 * (int64_t)sim);
                sim = si;
                r.init();
            }
            r.add<DIM>(xs, i);
        }
    }
    // over the warp when its particles share a simulation, then over the
    // block when all its warps do (one set of atomics per block: the extent
    // words are the same few addresses for every block); per lane otherwise
    __shared__ uint64_t slo[EXT_WARPS][3], shi[EXT_WARPS][3];
    __shared__ uint32_t ssim[EXT_WARPS];
    const uint32_t s0 = __shfl_sync(0xffffffffu, sim, 0);
    const bool uniform = __all_sync(0xffffffffu, sim == s0 || sim == 0xffffffffu);
    const unsigned wid = threadIdx.x >> 5;
    if (uniform) {
        for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
            for (int k = 0; k < DIM; ++k) {
                const uint64_t a = __shfl_xor_sync(0xffffffffu, r.lo[k], o);
                const uint64_t b = __shfl_xor_sync(0xffffffffu, r.hi[k], o);
                r.lo[k] = a < r.lo[k] ? a : r.lo[k];
                r.hi[k] = b > r.hi[k] ? b : r.hi[k];
            }
        }
    } else if (sim != 0xffffffffu) {
        r.flush<DIM>(ext + 8 * (int64_t)sim);
    }
    if (lane_id() == 0) {
        ssim[wid] = uniform ? s0 : 0xfffffffeu;             // 0xfffffffe: flushed already
#pragma unroll
        for (int k = 0; k < DIM; ++k) { slo[wid][k] = r.lo[k]; shi[wid][k] = r.hi[k]; }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const int nw = (int)((blockDim.x + 31) / 32);
        uint32_t sb = 0xffffffffu;
        bool one = true;
        for (int q = 0; q < nw; ++q) {
            const uint32_t sq = ssim[q];
            if (sq == 0xffffffffu) continue;                    // no particle
            if (sq == 0xfffffffeu || (sb != 0xffffffffu && sq != sb)) { one = false; break; }
            sb = sq;
        }
        for (int q = 0; q < nw; ++q) {
            const uint32_t sq = ssim[q];
            if (sq >= 0xfffffffeu) continue;
            ExtKeys t;
            t.init();
    #pragma unroll
            for (int k = 0; k < DIM; ++k) { t.lo[k] = slo[q][k]; t.hi[k] = shi[q][k]; }
            if (one) {
                // merge every warp into the first, flushed once at the end
                for (int q2 = q + 1; q2 < nw; ++q2) {
                    if (ssim[q2] != sb) continue;
    #pragma unroll
                    for (int k = 0; k < DIM; ++k) {
                        t.lo[k] = slo[q2][k] < t.lo[k] ? slo[q2][k] : t.lo[k];
                        t.hi[k] = shi[q2][k] > t.hi[k] ? shi[q2][k] : t.hi[k];
                    }
                }
                t.flush<DIM>(ext + 8 * (int64_t)sb);
                break;
            }
            t.flush<DIM>(ext + 8 * (int64_t)sq);
        }
    }
    // the last block: every block's words are in
    __shared__ bool last_block;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last_block = atomicAdd(ticket, 1u) == gridDim.x - 1u;
    }
    __syncthreads();
    if (!last_block) return;
    __threadfence();
    for (int q = threadIdx.x; q < nsim; q += blockDim.x) {
        unsigned long long* e = ext + 8 * (int64_t)q;
        unsigned long long lo[3], hi[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) { lo[k] = __ldcg(e + k); hi[k] = __ldcg(e + 3 + k); }
#pragma unroll
        for (int k = 0; k < 3; ++k) { e[k] = ~0ull; e[3 + k] = 0ull; }
        e[6] = ~0ull;
        e[7] = 0ull;
        finalize_cube(c, lo, hi, grids + q);
    }
    if (threadIdx.x == 0) *ticket = 0u;
}

// floor(log2(v)) of a positive normal value
__device__ __forceinline__ int exponent_of(double v) { return (int)((__double_as_longlong(v) >> 52) & 0x7ff) - 1023; }

// floor(log2(A / r)) for the radius r = (k^dim w)^(1/dim): with q = A^dim / (k^dim w)
// it is floor(floor(log2 q) / dim), so the exponent of q gives it (FP64 pow and
// log2 took a single block 11 us).  Outside the range where the powers are
// normal numbers, the functions.
__device__ inline int level_of(int dim, double A, double k, double w)
{
    double a = A, b = k;
    for (int d = 1; d < dim; ++d) { a *= A; b *= k; }
    const double q = a / (b * w);
    if (!(q >= 0x1p-1000) || !(q <= 0x1p1000) || !(a <= 0x1p1000) || !(a >= 0x1p-1000) || !(b * w >= 0x1p-1000))
        return (int)floor(log2(A / (k * pow(w, 1.0 / dim))));
    const int e = exponent_of(q);
    return e >= 0 ? e / dim : -((dim - 1 - e) / dim);
}

// The range of cell levels of each simulation, and over all of them (one
// block).  lmin is the finest level whose cell edge L / 2^l is at least the
// largest radius present; lmax the finest whose edge is at least half the
// smallest radius (the queries use cells down to half a radius).  Also zeroes
// the lengths and work counters of the query and the fit pass that follow
// (fresh_query, fresh_fit: they need no memsets of their own), and puts the
// words that k_begin and k_cfl leave for the next step to their initial values,
// whatever they hold: overlapping calls on one context may leave anything there,
// and a count of finished blocks that is off would never come right by itself.
constexpr int LEVEL_THREADS = 256;
__global__ void __launch_bounds__(LEVEL_THREADS) k_finalize_levels(DevCfg c, int lmax_cap, int nsim,
                                                                   unsigned long long* ext_all, Grid* grids,
                                                                   int* grange, unsigned long long* counters,
                                                                   unsigned int* tickets, unsigned long long* dtmin)
{
    __shared__ int slo[LEVEL_THREADS], shi[LEVEL_THREADS];
    if (threadIdx.x < 8) {
        const int zero[8] = {C_QFB_LEN, C_GROUP_LEN, C_QUEUE_TILE, C_REDO_LEN, C_PLAIN_LEN, C_REFINE_LEN,
                             C_QUEUE_CENTRAL, C_QUEUE_PLAIN};
        counters[zero[threadIdx.x]] = 0ull;
    }
    if (threadIdx.x < 2) tickets[threadIdx.x] = 0u;
    int lo_all = 1 << 20, hi_all = 0;
    for (int sim = threadIdx.x; sim < nsim; sim += LEVEL_THREADS) {
        unsigned long long* ext = ext_all + 8 * sim;
        Grid* g = grids + sim;
        const double L = g->L;
        dtmin[sim] = DTMIN_INIT;
#pragma unroll
        for (int k = 0; k < 3; ++k) { ext[k] = ~0ull; ext[3 + k] = 0ull; }
        const bool fixed = c.radius_mode == LP_RADIUS_FIXED;
        // the radius is k w^(1/dim), the fixed one with w = 1.  Margins wider than
        // the per-particle float radius margin (1e-5) keep every particle's level
        // inside [lmin, lmax]
        const double k = fixed ? c.radius : c.kappa;
        const double wlo = fixed ? 1.0 : from_order_key(ext[6]), whi = fixed ? 1.0 : from_order_key(ext[7]);
        const bool some = wlo > 0.0 && k > 0.0, bounded = whi > 0.0 && k > 0.0 && !isinf(whi) && !isinf(k);
        int lmax = some ? level_of(c.dim, 2.0 * L, k * (1.0 - 1e-4), wlo)
                        : lmax_cap + 1;               // empty or degenerate simulation: the finest
        int lmin = bounded ? level_of(c.dim, L, k * (1.0 + 1e-4), whi) : 0;
        lmax = max(0, min(lmax, lmax_cap));
        lmin = max(0, min(lmin, lmax));
        g->lmax = lmax;
        g->lmin = lmin;
        lo_all = min(lo_all, lmin);
        hi_all = max(hi_all, lmax);
    }
    slo[threadIdx.x] = lo_all;
    shi[threadIdx.x] = hi_all;
    __syncthreads();
    for (int h = LEVEL_THREADS / 2; h > 0; h >>= 1) {
        if ((int)threadIdx.x < h) {
            slo[threadIdx.x] = min(slo[threadIdx.x], slo[threadIdx.x + h]);
            shi[threadIdx.x] = max(shi[threadIdx.x], shi[threadIdx.x + h]);
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        grange[0] = slo[0];
        grange[1] = shi[0];
    }
}

// key = simulation << (DIM mbits) | Morton code of the quantised position (1D:
// the order key of x)
template <int DIM>
__device__ __forceinline__ uint64_t key_of(const double* const (&xs)[3], int64_t i, const Grid* g, uint32_t sim, int mbits)
{
    if (DIM == 1) return order_key(xs[0][i]);
    const double inv = g->inv;
    const uint32_t qmax = (1u << mbits) - 1u;
    uint32_t q[3] = {0, 0, 0};
#pragma unroll
    for (int k = 0; k < DIM; ++k) {
        // floor(t) clamped to [0, qmax] (negative and NaN give 0, +inf gives
        // qmax), read from t's bits: the conversion instruction would run on
        // the FP64 units, which the subtraction and the product already keep busy
        const double t = __dmul_rn(__dsub_rn(xs[k][i], g->lo[k]), inv);
        q[k] = floor_clamped(t, qmax);
    }
    return ((uint64_t)sim << (DIM * mbits)) | morton<DIM>(q);
}

template <int DIM>
__global__ void k_keys(int64_t n, const double* __restrict__ x0, const double* __restrict__ x1,
                       const double* __restrict__ x2, const Grid* __restrict__ grids,
                       const uint32_t* __restrict__ sim_of, int mbits,
                       uint64_t* __restrict__ keys, uint32_t* __restrict__ vals)
{
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double* xs[3] = {x0, x1, x2};
    const uint32_t sim = sim_of ? sim_of[i] : 0u;
    keys[i] = key_of<DIM>(xs, i, grids + sim, sim, mbits);
    vals[i] = (uint32_t)i;
}

// ---- LSD radix sort, RS_BITS-bit digits ----------------------------------

// Up to RS_FEW tiles, the downsweep's blocks sum the tiles' counts themselves
// (FEW: counts by tile, read coalesced, independent loads) instead of a scan kernel
// between: three passes 42 -> 33 us at 20k particles and 43 -> 39 at 131k (65 tiles),
// and a launch less each, 14 and 15 us of the step.  A tile more costs a pass 0.04 us:
// at 96 both take the same without the launch, at 245 the kernel takes 57 -> 73.
constexpr int64_t RS_FEW = 96;

template <bool FEW>
__global__ void k_rs_upsweep(int64_t n, const uint64_t* __restrict__ keys, int shift,
                             uint32_t* __restrict__ counts, int64_t nblocks)
{
    __shared__ uint32_t h[RS_BINS];
    h[threadIdx.x] = 0;
    h[threadIdx.x + RS_THREADS] = 0;
    __syncthreads();
    int64_t base = (int64_t)blockIdx.x * RS_TILE;
    for (int r = 0; r < RS_ITEMS; ++r) {
        int64_t i = base + r * RS_THREADS + threadIdx.x;
        if (i < n) atomicAdd(&h[(keys[i] >> shift) & RS_MASK], 1u);
    }
    __syncthreads();
    for (int d = (int)threadIdx.x; d < RS_BINS; d += RS_THREADS)
        counts[FEW ? (int64_t)blockIdx.x * RS_BINS + d : (int64_t)d * nblocks + blockIdx.x] = h[d];
}

// Per digit d (one block each): exclusive scan of the block counts
// counts[d * nblocks + b] along b, in place, and the digit's total in totals[d].
__global__ void __launch_bounds__(1024) k_rs_scan(uint32_t* counts, int64_t nblocks, uint32_t* totals)
{
    __shared__ uint32_t wsum[32];
    uint32_t* row = counts + (int64_t)blockIdx.x * nblocks;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    uint32_t carry = 0;
    for (int64_t b0 = 0; b0 < nblocks; b0 += 1024) {
        const int64_t b = b0 + t;
        const uint32_t v = b < nblocks ? row[b] : 0u;
        uint32_t x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wsum[w] = x;
        __syncthreads();
        if (w == 0) {
            uint32_t z = wsum[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, z, o);
                if (lane >= o) z += y;
            }
            wsum[lane] = z;                    // inclusive over warps
        }
        __syncthreads();
        const uint32_t before = (w ? wsum[w - 1] : 0u) + x - v;
        if (b < nblocks) row[b] = carry + before;
        carry += wsum[31];
        __syncthreads();
    }
    if (t == 0) totals[blockIdx.x] = carry;
}

// Scatter of one tile of RS_TILE keys: each warp ranks its 512 consecutive keys
// round by round (match on the digit), the warps' digit counts are scanned
// once per tile, and every key goes to digit base + block offset + rank.
template <bool FEW>
__global__ void __launch_bounds__(RS_THREADS)
k_rs_downsweep(int64_t n, const uint64_t* __restrict__ kin, const uint32_t* __restrict__ vin,
               uint64_t* __restrict__ kout, uint32_t* __restrict__ vout, int shift,
               const uint32_t* __restrict__ counts, const uint32_t* __restrict__ totals, int64_t nblocks)
{
    constexpr int NW = RS_THREADS / 32;
    __shared__ uint32_t wc[NW][RS_BINS];
    __shared__ uint32_t dbase[RS_BINS];
    const int t = threadIdx.x, w = t >> 5, lane = t & 31;
    // digit bases: exclusive scan of the digit totals, thread t owning digits
    // 2t and 2t + 1, plus this tile's offset within each digit
    {
        uint32_t v0 = 0, v1 = 0, c0 = 0, c1 = 0;
        if (FEW) {
#pragma unroll 8
            for (int b = 0; b < (int)nblocks; ++b) {
                const uint2 h = reinterpret_cast<const uint2*>(counts)[(int64_t)b * (RS_BINS / 2) + t];
                if (b == (int)blockIdx.x) { c0 = v0; c1 = v1; }
                v0 += h.x;
                v1 += h.y;
            }
        } else {
            v0 = totals[2 * t];
            v1 = totals[2 * t + 1];
            c0 = counts[(int64_t)(2 * t) * nblocks + blockIdx.x];
            c1 = counts[(int64_t)(2 * t + 1) * nblocks + blockIdx.x];
        }
        const uint32_t v = v0 + v1;
        uint32_t x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wc[0][w] = x;
        __syncthreads();
        uint32_t add = 0;
        for (int ww = 0; ww < w; ++ww) add += wc[0][ww];
        const uint32_t b0 = add + x - v;
        dbase[2 * t] = b0 + c0;
        dbase[2 * t + 1] = b0 + v0 + c1;
    }
    __syncthreads();
    for (int d = lane; d < RS_BINS; d += 32) wc[w][d] = 0;
    __syncwarp();
    const int64_t base = (int64_t)blockIdx.x * RS_TILE + (int64_t)w * (32 * RS_ITEMS);
    const unsigned lt = (1u << lane) - 1u;
    uint64_t key[RS_ITEMS];
    uint32_t val[RS_ITEMS], loc[RS_ITEMS];
#pragma unroll
    for (int r = 0; r < RS_ITEMS; ++r) {
        const int64_t i = base + r * 32 + lane;
        const bool valid = i < n;
        key[r] = valid ? kin[i] : 0ull;
        val[r] = valid ? vin[i] : 0u;
        const uint32_t d = valid ? (uint32_t)((key[r] >> shift) & RS_MASK) : RS_BINS + lane;
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        const bool leader = (__ffs(peers) - 1) == lane;
        loc[r] = valid ? wc[w][d] + __popc(peers & lt) : 0u;
        __syncwarp();
        if (valid && leader) wc[w][d] += __popc(peers);
        __syncwarp();
    }
    __syncthreads();
    // per digit: offsets of the warps' runs in tile order
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int d = t + h * RS_THREADS;
        uint32_t run = dbase[d];
#pragma unroll
        for (int ww = 0; ww < NW; ++ww) {
            const uint32_t c = wc[ww][d];
            wc[ww][d] = run;
            run += c;
        }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < RS_ITEMS; ++r) {
        const int64_t i = base + r * 32 + lane;
        if (i < n) {
            const uint32_t d = (uint32_t)((key[r] >> shift) & RS_MASK);
            const uint32_t pos = wc[w][d] + loc[r];
            kout[pos] = key[r];
            vout[pos] = val[r];
        }
    }
}

// The whole front of a build for one simulation of at most FS_MAX particles, by
// one block: the last build's table entries cleared, the extent, the cube, the
// keys and every pass of the radix sort, keys and indices in shared memory.
// Launched one by one these are 4 + 3 launches per digit, 28 for the 64-bit keys
// of 1D, each a few microseconds whatever n is: of a 1D step of 1000 particles
// they were 180 of 218 us.  Keys already in order (1D particles keep theirs)
// need no pass; with more particles than FS_MAX the passes of one SM cost more
// than the launches of all.  The order is that of the general path: stable, by
// the same digits.
constexpr int FS_THREADS = 1024;
constexpr int FS_ITEMS = 8;
constexpr int FS_MAX = FS_THREADS * FS_ITEMS;
constexpr int FS_WARPS = FS_THREADS / 32;
struct FrontShared {
    uint64_t key[FS_MAX];
    uint16_t val[FS_MAX];
    uint16_t wc[FS_WARPS][RS_BINS];       // per warp digit counts, then places
    uint32_t wsum[FS_WARPS];
    uint64_t lo[3][FS_WARPS], hi[3][FS_WARPS];
    Grid grid;
};
static_assert(FS_MAX <= 65535 && RS_BINS <= FS_THREADS, "16-bit places, a thread per digit");

template <int DIM>
__global__ void __launch_bounds__(FS_THREADS) k_front_small(int n, const double* __restrict__ x0,
                                                            const double* __restrict__ x1,
                                                            const double* __restrict__ x2, DevCfg c, Grid* grid,
                                                            unsigned long long* ext, TableArgs old, int lo_bit,
                                                            int hi_bit, uint64_t* __restrict__ keys,
                                                            uint32_t* __restrict__ vals)
{
    extern __shared__ __align__(16) unsigned char fs_smem[];
    FrontShared& sm = *reinterpret_cast<FrontShared*>(fs_smem);
    const int t = (int)threadIdx.x, w = t >> 5, lane = t & 31;
    const unsigned lt = (1u << lane) - 1u;
    for (int64_t i = t; i < old.n; i += FS_THREADS) table_entries<true>(old, i);
    if (t < 2) ext[6 + t] = t == 0 ? ~0ull : 0ull;        // the gather takes the extent of m V
    const double* const xs[3] = {x0, x1, x2};
    ExtKeys r;
    r.init();
    for (int i = t; i < n; i += FS_THREADS) r.add<DIM>(xs, i);
#pragma unroll
    for (int k = 0; k < DIM; ++k) {
        for (int o = 16; o > 0; o >>= 1) {
            const uint64_t a = __shfl_xor_sync(0xffffffffu, r.lo[k], o);
            const uint64_t b = __shfl_xor_sync(0xffffffffu, r.hi[k], o);
            r.lo[k] = a < r.lo[k] ? a : r.lo[k];
            r.hi[k] = b > r.hi[k] ? b : r.hi[k];
        }
        if (lane == 0) { sm.lo[k][w] = r.lo[k]; sm.hi[k][w] = r.hi[k]; }
    }
    __syncthreads();
    if (w == 0) {
        unsigned long long lo[3] = {~0ull, ~0ull, ~0ull}, hi[3] = {0ull, 0ull, 0ull};
#pragma unroll
        for (int k = 0; k < DIM; ++k) {
            uint64_t a = sm.lo[k][lane], b = sm.hi[k][lane];
            for (int o = 16; o > 0; o >>= 1) {
                const uint64_t a2 = __shfl_xor_sync(0xffffffffu, a, o), b2 = __shfl_xor_sync(0xffffffffu, b, o);
                a = a2 < a ? a2 : a;
                b = b2 > b ? b2 : b;
            }
            lo[k] = a;
            hi[k] = b;
        }
        if (lane == 0) {
            finalize_cube(c, lo, hi, &sm.grid);
            // (the levels are set after the gather)
            for (int k = 0; k < 3; ++k) {
                grid->lo[k] = sm.grid.lo[k];
                grid->lo_h[k] = sm.grid.lo_h[k];
                grid->lo_l[k] = sm.grid.lo_l[k];
            }
            grid->L = sm.grid.L;
            grid->inv = sm.grid.inv;
            grid->inv_f = sm.grid.inv_f;
            grid->L_f = sm.grid.L_f;
        }
    }
    __syncthreads();
    // warp w holds positions [w 32 items, (w + 1) 32 items), 32 per round
    const int items = (n + FS_THREADS - 1) / FS_THREADS;
    const int base = w * 32 * items + lane;
    uint64_t key[FS_ITEMS];
    uint32_t val[FS_ITEMS];
#pragma unroll
    for (int q = 0; q < FS_ITEMS; ++q) {
        const int i = base + 32 * q;
        if (q >= items || i >= n) continue;
        key[q] = key_of<DIM>(xs, i, &sm.grid, 0u, c.mbits);
        val[q] = (uint32_t)i;
        sm.key[i] = key[q];
    }
    __syncthreads();
    bool sorted = true;
#pragma unroll
    for (int q = 0; q < FS_ITEMS; ++q) {
        const int i = base + 32 * q;
        if (q < items && i + 1 < n) sorted = sorted && (key[q] >> lo_bit) <= (sm.key[i + 1] >> lo_bit);
    }
    if (!__syncthreads_and(sorted)) {
        for (int shift = lo_bit; shift < hi_bit; shift += RS_BITS) {
            for (int d = lane; d < RS_BINS; d += 32) sm.wc[w][d] = 0;
            __syncwarp();
            uint32_t loc[FS_ITEMS];
#pragma unroll
            for (int q = 0; q < FS_ITEMS; ++q) {
                if (q >= items) break;
                const bool valid = base + 32 * q < n;
                const uint32_t d = valid ? (uint32_t)((key[q] >> shift) & RS_MASK) : RS_BINS + lane;
                const unsigned peers = __match_any_sync(0xffffffffu, d);
                const bool leader = (__ffs(peers) - 1) == lane;
                loc[q] = valid ? sm.wc[w][d] + __popc(peers & lt) : 0u;
                __syncwarp();
                if (valid && leader) sm.wc[w][d] += (uint16_t)__popc(peers);
                __syncwarp();
            }
            __syncthreads();
            // digit t: its warps' counts to places, after the smaller digits
            uint32_t total = 0;
            if (t < RS_BINS)
                for (int u = 0; u < FS_WARPS; ++u) total += sm.wc[u][t];
            uint32_t x = total;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            if (lane == 31) sm.wsum[w] = x;
            __syncthreads();
            if (t < RS_BINS) {
                uint32_t run = x - total;
                for (int u = 0; u < w; ++u) run += sm.wsum[u];
                for (int u = 0; u < FS_WARPS; ++u) {
                    const uint32_t k = sm.wc[u][t];
                    sm.wc[u][t] = (uint16_t)run;
                    run += k;
                }
            }
            __syncthreads();
#pragma unroll
            for (int q = 0; q < FS_ITEMS; ++q) {
                if (q >= items || base + 32 * q >= n) continue;
                const uint32_t pos = sm.wc[w][(uint32_t)((key[q] >> shift) & RS_MASK)] + loc[q];
                sm.key[pos] = key[q];
                sm.val[pos] = (uint16_t)val[q];
            }
            __syncthreads();
#pragma unroll
            for (int q = 0; q < FS_ITEMS; ++q) {
                const int i = base + 32 * q;
                if (q >= items || i >= n) continue;
                key[q] = sm.key[i];
                val[q] = sm.val[i];
            }
        }
    }
#pragma unroll
    for (int q = 0; q < FS_ITEMS; ++q) {
        const int i = base + 32 * q;
        if (q >= items || i >= n) continue;
        keys[i] = key[q];
        vals[i] = val[q];
    }
}

template <int DIM>
cudaError_t launch_front_small(int n, const double* x0, const double* x1, const double* x2, const DevCfg& c, Grid* grid,
                               unsigned long long* ext, const TableArgs& old, int lo_bit, int hi_bit, uint64_t* keys,
                               uint32_t* vals, cudaStream_t s)
{
    k_front_small<DIM><<<1, FS_THREADS, sizeof(FrontShared), s>>>(n, x0, x1, x2, c, grid, ext, old, lo_bit, hi_bit, keys,
                                                                  vals);
    return cudaGetLastError();
}

cudaError_t front_small(int dim, int n, const double* x0, const double* x1, const double* x2, const DevCfg& c, Grid* grid,
                        unsigned long long* ext, const TableArgs& old, int lo_bit, int hi_bit, uint64_t* keys,
                        uint32_t* vals, cudaStream_t s)
{
    if (dim == 3) return launch_front_small<3>(n, x0, x1, x2, c, grid, ext, old, lo_bit, hi_bit, keys, vals, s);
    if (dim == 2) return launch_front_small<2>(n, x0, x1, x2, c, grid, ext, old, lo_bit, hi_bit, keys, vals, s);
    return launch_front_small<1>(n, x0, x1, x2, c, grid, ext, old, lo_bit, hi_bit, keys, vals, s);
}

// gather the state into key order and split it into float hi/lo pairs
template <int DIM>
__global__ void k_gather(int64_t n, const uint32_t* __restrict__ perm, lp_particles p, DevCfg c,
                         double* sx0, double* sx1, double* sx2, double* sV, double* su0, double* su1,
                         double* su2, double* sP, double* sm, uint32_t* sid, float4* rec, float4* pos4,
                         const uint32_t* __restrict__ sim_of, unsigned long long* ext)
{
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    {
        const uint32_t jw = i < n ? perm[i] : 0u;
        block_w_extent(i < n, i < n ? __dmul_rn(p.m[jw], p.V[jw]) : 0.0, (i < n && sim_of) ? sim_of[jw] : 0u, ext);
    }
    if (i >= n) return;
    uint32_t j = perm[i];
    float r[4 * REC_F4];
#pragma unroll
    for (int q = 0; q < 4 * REC_F4; ++q) r[q] = 0.0f;
    double* sx[3] = {sx0, sx1, sx2};
    double* su[3] = {su0, su1, su2};
#pragma unroll
    for (int k = 0; k < DIM; ++k) {
        double v = p.x[k][j];
        sx[k][i] = v;
        split(v, r[REC_XH + k], r[REC_XL + k]);
    }
    double V = p.V[j], P = p.P[j];
    sV[i] = V;
    sP[i] = P;
    constexpr int F = DIM + 2;
    split(V, r[rec_fh(0, F)], r[rec_fl(0, F)]);
    split(P, r[rec_fh(F - 1, F)], r[rec_fl(F - 1, F)]);
#pragma unroll
    for (int k = 0; k < DIM; ++k) {
        double v = p.u[k][j];
        su[k][i] = v;
        split(v, r[rec_fh(1 + k, F)], r[rec_fl(1 + k, F)]);
    }
#pragma unroll
    for (int q = 0; q < REC_F4; ++q) rec[i * REC_F4 + q] = make_float4(r[4 * q], r[4 * q + 1], r[4 * q + 2], r[4 * q + 3]);
    const double m = p.m[j];
    // (r[rec_fh(0, F)] is RN(V))
    pos4[2 * i] = make_float4(r[REC_XH], r[REC_XH + 1], r[REC_XH + 2],
                              query_radius_ff(c, DIM, to_float_rn(m), r[rec_fh(0, F)]));
    pos4[2 * i + 1] = make_float4(r[REC_XL], r[REC_XL + 1], r[REC_XL + 2], 0.0f);
    sm[i] = m;
    sid[i] = p.id[j];
}

// The same gather in two kernels, for the end-to-end path (lp_step_host),
// where the fields are still being copied from the host while the neighbour
// query runs: the geometry (positions, m, V, id, the query's float positions
// and radius, the m V extent) before the query, the fields (u, P and the packed
// fit record) after it.  Together they write what k_gather writes, bit for bit.
template <int DIM>
__global__ void k_gather_geom(int64_t n, const uint32_t* __restrict__ perm, lp_particles p, DevCfg c,
                              double* sx0, double* sx1, double* sx2, double* sV, double* sm, uint32_t* sid,
                              float4* pos4, const uint32_t* __restrict__ sim_of, unsigned long long* ext)
{
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    {
        const uint32_t jw = i < n ? perm[i] : 0u;
        block_w_extent(i < n, i < n ? __dmul_rn(p.m[jw], p.V[jw]) : 0.0, (i < n && sim_of) ? sim_of[jw] : 0u, ext);
    }
    if (i >= n) return;
    const uint32_t j = perm[i];
    double* sx[3] = {sx0, sx1, sx2};
    float xh[3] = {0.0f, 0.0f, 0.0f}, xl[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int k = 0; k < DIM; ++k) {
        const double v = p.x[k][j];
        sx[k][i] = v;
        split(v, xh[k], xl[k]);
    }
    const double V = p.V[j], m = p.m[j];
    sV[i] = V;
    sm[i] = m;
    sid[i] = p.id[j];
    pos4[2 * i] = make_float4(xh[0], xh[1], xh[2], query_radius_ff(c, DIM, to_float_rn(m), to_float_rn(V)));
    pos4[2 * i + 1] = make_float4(xl[0], xl[1], xl[2], 0.0f);
}

template <int DIM>
__global__ void k_gather_fields(int64_t n, const uint32_t* __restrict__ perm, lp_particles p,
                                const double* sx0, const double* sx1, const double* sx2, const double* sV,
                                double* su0, double* su1, double* su2, double* sP, float4* rec)
{
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint32_t j = perm[i];
    float r[4 * REC_F4];
#pragma unroll
    for (int q = 0; q < 4 * REC_F4; ++q) r[q] = 0.0f;
    const double* sx[3] = {sx0, sx1, sx2};
    double* su[3] = {su0, su1, su2};
#pragma unroll
    for (int k = 0; k < DIM; ++k) split(sx[k][i], r[REC_XH + k], r[REC_XL + k]);
    constexpr int F = DIM + 2;
    const double P = p.P[j];
    sP[i] = P;
    split(sV[i], r[rec_fh(0, F)], r[rec_fl(0, F)]);
    split(P, r[rec_fh(F - 1, F)], r[rec_fl(F - 1, F)]);
#pragma unroll
    for (int k = 0; k < DIM; ++k) {
        const double v = p.u[k][j];
        su[k][i] = v;
        split(v, r[rec_fh(1 + k, F)], r[rec_fl(1 + k, F)]);
    }
#pragma unroll
    for (int q = 0; q < REC_F4; ++q) rec[i * REC_F4 + q] = make_float4(r[4 * q], r[4 * q + 1], r[4 * q + 2], r[4 * q + 3]);
}

// cell tables: entry = start | end << 32 of the key-sorted particles in the cell
template <bool CLEAR>
__global__ void k_tables(TableArgs a)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < a.n) table_entries<CLEAR>(a, i);
}

__global__ void k_scatter_back(int dim, int64_t n, lp_particles p, const double* sx0, const double* sx1,
                               const double* sx2, const double* sV, const double* su0, const double* su1,
                               const double* su2, const double* sP, const double* sm, const uint32_t* sid)
{
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double* sx[3] = {sx0, sx1, sx2};
    const double* su[3] = {su0, su1, su2};
    for (int k = 0; k < dim; ++k) {
        p.x[k][i] = sx[k][i];
        p.u[k][i] = su[k][i];
    }
    p.V[i] = sV[i];
    p.P[i] = sP[i];
    p.m[i] = sm[i];
    p.id[i] = sid[i];
}

inline unsigned grid_for(int64_t n, int threads) { return (unsigned)((n + threads - 1) / threads); }

__global__ void k_sim_of(int64_t n, const int64_t* __restrict__ offsets, int nsim, uint32_t* __restrict__ sim_of)
{
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    int lo = 0, hi = nsim - 1;          // last simulation whose offset is <= i
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (offsets[mid] <= i) lo = mid; else hi = mid - 1;
    }
    sim_of[i] = (uint32_t)lo;
}

}  // namespace

cudaError_t sort_init()
{
    const cudaFuncAttribute at = cudaFuncAttributeMaxDynamicSharedMemorySize;
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(k_front_small<1>, at, (int)sizeof(FrontShared))) != cudaSuccess) return e;
    if ((e = cudaFuncSetAttribute(k_front_small<2>, at, (int)sizeof(FrontShared))) != cudaSuccess) return e;
    return cudaFuncSetAttribute(k_front_small<3>, at, (int)sizeof(FrontShared));
}

static TableArgs table_args(const lp_ctx* c, int64_t n)
{
    return TableArgs{c->dc.dim, c->dc.mbits, c->dc.dim == 1 ? 0 : n, c->keys_sorted, c->grange, c->level_off_dev, c->cells};
}

cudaError_t init_extent(lp_ctx* c, cudaStream_t s)
{
    const int ns = c->dc.nsim_max;
    k_init_extent<<<(unsigned)((8 * (int64_t)ns + 255) / 256), 256, 0, s>>>(c->ext, ns, c->tickets);
    return cudaGetLastError();
}

bool front_is_small(const lp_ctx* c, int64_t n) { return c->nsim == 1 && n <= FS_MAX; }

int front_launches(const lp_ctx* c, int64_t n)
{
    return front_is_small(c, n) ? 1 : 2 + (c->nsim > 1 ? 1 : 0);
}

// everything up to the sort; for small n the sort too (one kernel)
cudaError_t build_front(lp_ctx* c, const lp_particles* p, int64_t n_old, cudaStream_t s)
{
    const int64_t n = p->n;
    const int nsim = c->nsim, dim = c->dc.dim, mb = c->dc.mbits;
    const TableArgs old = table_args(c, n_old);
    const double* x1 = p->x[1] ? p->x[1] : p->x[0];
    const double* x2 = p->x[2] ? p->x[2] : p->x[0];
    if (front_is_small(c, n)) {
        // the buffers radix_sort ends in, so that a captured step finds the keys of
        // the one before it where the capture did.  (They may hold the last build's
        // keys: those are read before the block's barriers, the new ones written
        // after them.)
        const int out = radix_passes(c) & 1;
        c->keys_sorted = c->keys[out];
        c->perm_sorted = c->vals[out];
        return front_small(dim, (int)n, p->x[0], x1, x2, c->dc, c->grid, c->ext, old, c->sort_lo_bit, c->sort_hi_bit,
                           c->keys_sorted, c->perm_sorted, s);
    }
    const uint32_t* sim_of = nullptr;
    if (nsim > 1) {
        k_sim_of<<<grid_for(n, 256), 256, 0, s>>>(n, c->offsets, nsim, c->sim_of);
        sim_of = c->sim_of;
    }
    const int64_t nb_ = grid_for(n, 256);
    const unsigned blocks = nsim > 1 ? (unsigned)((n + 256 * EXT_ITEMS - 1) / (256 * EXT_ITEMS))
                                     : (unsigned)(nb_ < 152 * 8 ? nb_ : 152 * 8);
#define LP_BEGIN_ARGS n, p->x[0], x1, x2, sim_of, c->ext, c->dc, nsim, c->grid, c->tickets, old
    if (dim == 3) k_begin<3><<<blocks, 256, 0, s>>>(LP_BEGIN_ARGS);
    else if (dim == 2) k_begin<2><<<blocks, 256, 0, s>>>(LP_BEGIN_ARGS);
    else k_begin<1><<<blocks, 256, 0, s>>>(LP_BEGIN_ARGS);
#undef LP_BEGIN_ARGS
    const unsigned gb = grid_for(n, 256);
    if (dim == 3) k_keys<3><<<gb, 256, 0, s>>>(n, p->x[0], x1, x2, c->grid, sim_of, mb, c->keys[0], c->vals[0]);
    else if (dim == 2) k_keys<2><<<gb, 256, 0, s>>>(n, p->x[0], x1, x2, c->grid, sim_of, mb, c->keys[0], c->vals[0]);
    else k_keys<1><<<gb, 256, 0, s>>>(n, p->x[0], x1, x2, c->grid, sim_of, mb, c->keys[0], c->vals[0]);
    return cudaGetLastError();
}

// one pass of the sort; hist: RS_BINS x (tiles + 1) words
static void radix_pass(int64_t n, int shift, uint32_t* hist, const uint64_t* kin, const uint32_t* vin, uint64_t* kout,
                       uint32_t* vout, cudaStream_t s)
{
    const int64_t nblocks = (n + RS_TILE - 1) / RS_TILE;
    const unsigned nb = (unsigned)nblocks;
    uint32_t* const totals = hist + RS_BINS * nblocks;
    if (nblocks <= RS_FEW) {
        k_rs_upsweep<true><<<nb, RS_THREADS, 0, s>>>(n, kin, shift, hist, nblocks);
        k_rs_downsweep<true><<<nb, RS_THREADS, 0, s>>>(n, kin, vin, kout, vout, shift, hist, totals, nblocks);
        return;
    }
    k_rs_upsweep<false><<<nb, RS_THREADS, 0, s>>>(n, kin, shift, hist, nblocks);
    k_rs_scan<<<RS_BINS, 1024, 0, s>>>(hist, nblocks, totals);
    k_rs_downsweep<false><<<nb, RS_THREADS, 0, s>>>(n, kin, vin, kout, vout, shift, hist, totals, nblocks);
}

int radix_pass_launches(int64_t n) { return (n + RS_TILE - 1) / RS_TILE <= RS_FEW ? 2 : 3; }

int radix_passes(const lp_ctx* c) { return (c->sort_hi_bit - c->sort_lo_bit + RS_BITS - 1) / RS_BITS; }

cudaError_t radix_sort(lp_ctx* c, int64_t n, cudaStream_t s)
{
    int cur = 0;
    for (int sh = c->sort_lo_bit; sh < c->sort_hi_bit; sh += RS_BITS) {
        radix_pass(n, sh, c->hist, c->keys[cur], c->vals[cur], c->keys[cur ^ 1], c->vals[cur ^ 1], s);
        cur ^= 1;
    }
    c->keys_sorted = c->keys[cur];
    c->perm_sorted = c->vals[cur];
    return cudaGetLastError();
}

cudaError_t gather(lp_ctx* c, const lp_particles* p, cudaStream_t s)
{
    int64_t n = p->n;
    int dim = c->dc.dim;
    unsigned gb = grid_for(n, 256);
    const uint32_t* perm = c->perm_sorted;
    lp_particles q = *p;
    for (int k = dim; k < 3; ++k) { q.x[k] = p->x[0]; q.u[k] = p->u[0]; }
    const uint32_t* sim_of = c->nsim > 1 ? c->sim_of : nullptr;
#define LP_GATHER_ARGS n, perm, q, c->dc, c->sx[0], c->sx[1], c->sx[2], c->sV, c->su[0], c->su[1], c->su[2], \
        c->sP, c->sm, c->sid, c->rec, c->pos4, sim_of, c->ext
    if (dim == 3) k_gather<3><<<gb, 256, 0, s>>>(LP_GATHER_ARGS);
    else if (dim == 2) k_gather<2><<<gb, 256, 0, s>>>(LP_GATHER_ARGS);
    else k_gather<1><<<gb, 256, 0, s>>>(LP_GATHER_ARGS);
#undef LP_GATHER_ARGS
    // the cell levels need the m V extent the gather took
    k_finalize_levels<<<1, LEVEL_THREADS, 0, s>>>(c->dc, c->lmax_cap, c->nsim, c->ext, c->grid, c->grange, c->counters,
                                               c->tickets, c->dt_min);
    c->fresh_query = c->fresh_fit = 1;
    return cudaGetLastError();
}

cudaError_t gather_geometry(lp_ctx* c, const lp_particles* p, cudaStream_t s)
{
    int64_t n = p->n;
    int dim = c->dc.dim;
    unsigned gb = grid_for(n, 256);
    const uint32_t* perm = c->perm_sorted;
    lp_particles q = *p;
    for (int k = dim; k < 3; ++k) q.x[k] = p->x[0];
    const uint32_t* sim_of = c->nsim > 1 ? c->sim_of : nullptr;
#define LP_GATHER_ARGS n, perm, q, c->dc, c->sx[0], c->sx[1], c->sx[2], c->sV, c->sm, c->sid, c->pos4, sim_of, c->ext
    if (dim == 3) k_gather_geom<3><<<gb, 256, 0, s>>>(LP_GATHER_ARGS);
    else if (dim == 2) k_gather_geom<2><<<gb, 256, 0, s>>>(LP_GATHER_ARGS);
    else k_gather_geom<1><<<gb, 256, 0, s>>>(LP_GATHER_ARGS);
#undef LP_GATHER_ARGS
    k_finalize_levels<<<1, LEVEL_THREADS, 0, s>>>(c->dc, c->lmax_cap, c->nsim, c->ext, c->grid, c->grange, c->counters,
                                               c->tickets, c->dt_min);
    c->fresh_query = c->fresh_fit = 1;
    return cudaGetLastError();
}

cudaError_t gather_fields(lp_ctx* c, const lp_particles* p, cudaStream_t s)
{
    int64_t n = p->n;
    int dim = c->dc.dim;
    unsigned gb = grid_for(n, 256);
    const uint32_t* perm = c->perm_sorted;
    lp_particles q = *p;
    for (int k = dim; k < 3; ++k) q.u[k] = p->u[0];
    const double* sx1 = c->sx[dim > 1 ? 1 : 0];
    const double* sx2 = c->sx[dim > 2 ? 2 : 0];
    double* su1 = c->su[dim > 1 ? 1 : 0];
    double* su2 = c->su[dim > 2 ? 2 : 0];
#define LP_GATHER_ARGS n, perm, q, c->sx[0], sx1, sx2, c->sV, c->su[0], su1, su2, c->sP, c->rec
    if (dim == 3) k_gather_fields<3><<<gb, 256, 0, s>>>(LP_GATHER_ARGS);
    else if (dim == 2) k_gather_fields<2><<<gb, 256, 0, s>>>(LP_GATHER_ARGS);
    else k_gather_fields<1><<<gb, 256, 0, s>>>(LP_GATHER_ARGS);
#undef LP_GATHER_ARGS
    return cudaGetLastError();
}

cudaError_t fill_tables(lp_ctx* c, int64_t n, bool clear, cudaStream_t s)
{
    if (c->dc.dim == 1 || n == 0) return cudaSuccess;
    if (clear) k_tables<true><<<grid_for(n, 256), 256, 0, s>>>(table_args(c, n));
    else k_tables<false><<<grid_for(n, 256), 256, 0, s>>>(table_args(c, n));
    return cudaGetLastError();
}

cudaError_t scatter_back(lp_ctx* c, lp_particles* p, cudaStream_t s)
{
    int64_t n = p->n;
    if (n == 0) return cudaSuccess;
    lp_particles q = *p;
    for (int k = c->dc.dim; k < 3; ++k) { q.x[k] = p->x[0]; q.u[k] = p->u[0]; }
    k_scatter_back<<<grid_for(n, 256), 256, 0, s>>>(c->dc.dim, n, q, c->sx[0], c->sx[1], c->sx[2], c->sV, c->su[0],
                                                     c->su[1], c->su[2], c->sP, c->sm, c->sid);
    return cudaGetLastError();
}

}  // namespace lp

// ---------------------------------------------------------------------------
// Morton keys and sort order without any device allocation.
//
// Some callers cannot allocate device memory when they need the key order: a
// host application that owns every byte of device memory through its own pool
// and forbids other allocations, or a latency-critical loop where cudaMalloc's
// implicit device-wide synchronisation is not acceptable.  This entry point
// serves them: its scratch (key and index ping-pong buffers, digit histograms,
// the extent words and the cube) lives in one fixed file-scope device array,
// NOALLOC_MAX_N particles large, which every GPU that loads this library holds
// until the process exits.  It reuses the sort kernels above; nothing else in
// the library uses this array.
// ---------------------------------------------------------------------------
namespace lp {
namespace {

constexpr int64_t NOALLOC_MAX_N = LP_NOALLOC_MAX_N;
constexpr int64_t NA_BLOCKS = (NOALLOC_MAX_N + RS_TILE - 1) / RS_TILE;
// byte offsets inside the array (each 256-byte aligned)
constexpr size_t NA_KEYS0 = 0;
constexpr size_t NA_KEYS1 = NA_KEYS0 + 8 * NOALLOC_MAX_N;
constexpr size_t NA_VALS0 = NA_KEYS1 + 8 * NOALLOC_MAX_N;
constexpr size_t NA_VALS1 = NA_VALS0 + 4 * NOALLOC_MAX_N;
constexpr size_t NA_HIST = NA_VALS1 + 4 * NOALLOC_MAX_N;
constexpr size_t NA_EXT = NA_HIST + ((RS_BINS * (NA_BLOCKS + 1) * 4 + 255) / 256) * 256;   // counts + digit totals
constexpr size_t NA_GRID = NA_EXT + 256;
constexpr size_t NA_BYTES = NA_GRID + 256;

static __device__ __align__(256) unsigned char noalloc_scratch[NA_BYTES];

constexpr int NA_MAX_DEVICES = 64;
std::mutex na_mutex;
unsigned char* na_ptr[NA_MAX_DEVICES] = {};

// The device address of the array on the current device.  Outside stream
// capture it is looked up again on every call, so an address cached before a
// cudaDeviceReset (after which the runtime loads the module again, possibly at
// another address) is never used.  While `s` is capturing, no runtime call that
// could load the module is made: the address cached by the last call on this
// device outside capture is used, and a device never set up that way is an
// error.
cudaError_t noalloc_setup(cudaStream_t s, unsigned char** out)
{
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= NA_MAX_DEVICES) return cudaErrorInvalidDevice;
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    e = cudaStreamIsCapturing(s, &cs);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(na_mutex);
    if (cs == cudaStreamCaptureStatusNone) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, noalloc_scratch);
        if (e != cudaSuccess || (e = sort_init()) != cudaSuccess) return e;
        na_ptr[dev] = static_cast<unsigned char*>(p);
    } else if (!na_ptr[dev]) {
        return cudaErrorStreamCaptureUnsupported;
    }
    *out = na_ptr[dev];
    return cudaSuccess;
}

__global__ void k_copy_sorted(int64_t n, const uint64_t* __restrict__ ks, const uint32_t* __restrict__ vs,
                              uint64_t* __restrict__ ko, uint32_t* __restrict__ vo)
{
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) { ko[i] = ks[i]; vo[i] = vs[i]; }
}

}  // namespace
}  // namespace lp

extern "C" lp_status lp_sort_keys_noalloc(int32_t dim, int64_t n, const double* x0, const double* x1,
                                          const double* x2, uint64_t* keys_out, uint32_t* perm_out,
                                          lp_stream stream)
{
    using namespace lp;
    if (dim < 1 || dim > 3 || n < 0 || !keys_out || !perm_out) return LP_ERR_ARG;
    if (n > NOALLOC_MAX_N) return LP_ERR_CAPACITY;
    if (n == 0) return LP_OK;
    if (!x0 || (dim > 1 && !x1) || (dim > 2 && !x2)) return LP_ERR_ARG;
    unsigned char* base = nullptr;
    cudaStream_t s = (cudaStream_t)stream;
    if (noalloc_setup(s, &base) != cudaSuccess) return LP_ERR_CUDA;
    uint64_t* keys[2] = {reinterpret_cast<uint64_t*>(base + NA_KEYS0), reinterpret_cast<uint64_t*>(base + NA_KEYS1)};
    uint32_t* vals[2] = {reinterpret_cast<uint32_t*>(base + NA_VALS0), reinterpret_cast<uint32_t*>(base + NA_VALS1)};
    uint32_t* hist = reinterpret_cast<uint32_t*>(base + NA_HIST);
    unsigned long long* ext = reinterpret_cast<unsigned long long*>(base + NA_EXT);
    Grid* grid = reinterpret_cast<Grid*>(base + NA_GRID);
    const double* p1 = x1 ? x1 : x0;
    const double* p2 = x2 ? x2 : x0;
    // the cube: same kernels and parameters as a default context (fixed radius 1,
    // finest table level 9 in 3D, 13 in 2D); the radius only sets the level range
    DevCfg dc;
    memset(&dc, 0, sizeof(dc));
    dc.dim = dim;
    dc.radius_mode = LP_RADIUS_FIXED;
    dc.radius = 1.0;
    dc.mbits = MORTON_BITS;
    dc.nsim_max = 1;
    int lmax_cap = dim == 3 ? 9 : (dim == 2 ? 13 : 0);
    int lo_bit = 0, hi_bit = 64;
    sort_bit_range(dim, MORTON_BITS, lmax_cap, 0, lo_bit, hi_bit);
    const TableArgs none = {};
    if (n <= FS_MAX)
        return front_small(dim, (int)n, x0, p1, p2, dc, grid, ext, none, lo_bit, hi_bit, keys_out, perm_out, s) ==
                       cudaSuccess ? LP_OK : LP_ERR_CUDA;
    unsigned gb = grid_for(n, 256);
    int64_t nb_ = gb;
    unsigned rblocks = (unsigned)(nb_ < 152 * 8 ? nb_ : 152 * 8);
    unsigned int* ticket = reinterpret_cast<unsigned int*>(ext + 8);
    k_init_extent<<<1, 32, 0, s>>>(ext, 1, ticket);
    if (dim == 3) k_begin<3><<<rblocks, 256, 0, s>>>(n, x0, p1, p2, nullptr, ext, dc, 1, grid, ticket, none);
    else if (dim == 2) k_begin<2><<<rblocks, 256, 0, s>>>(n, x0, p1, p2, nullptr, ext, dc, 1, grid, ticket, none);
    else k_begin<1><<<rblocks, 256, 0, s>>>(n, x0, p1, p2, nullptr, ext, dc, 1, grid, ticket, none);
    if (dim == 3) k_keys<3><<<gb, 256, 0, s>>>(n, x0, p1, p2, grid, nullptr, MORTON_BITS, keys[0], vals[0]);
    else if (dim == 2) k_keys<2><<<gb, 256, 0, s>>>(n, x0, p1, p2, grid, nullptr, MORTON_BITS, keys[0], vals[0]);
    else k_keys<1><<<gb, 256, 0, s>>>(n, x0, p1, p2, grid, nullptr, MORTON_BITS, keys[0], vals[0]);
    int cur = 0;
    for (int sh = lo_bit; sh < hi_bit; sh += RS_BITS) {
        radix_pass(n, sh, hist, keys[cur], vals[cur], keys[cur ^ 1], vals[cur ^ 1], s);
        cur ^= 1;
    }
    k_copy_sorted<<<gb, 256, 0, s>>>(n, keys[cur], vals[cur], keys_out, perm_out);
    return cudaGetLastError() == cudaSuccess ? LP_OK : LP_ERR_CUDA;
}
