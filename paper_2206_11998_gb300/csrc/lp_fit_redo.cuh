// lp_fit_redo.cuh -- the FP64 redo of the stencils the FP32 pass listed, a
// block per particle.
//
// An FP64 warp instruction holds its scheduler's FP64 unit for 64 cycles
// whether one lane or all 32 take part, so a particle redone by one thread
// (k_step<double> and its like) is a chain of some 25,000 instructions, 0.7 to
// 1.3 ms, and a list of one particle takes as long as one of thousands.  The
// lists are short (a handful of the cloud's or the lattice's surface
// particles, some thousands on the 2D ensemble), so here the four warps of a
// block share one particle's fits:
//   - thread r forms row r of the stencil (offsets, differences, products);
//   - warp 0 runs the central fit's rotations as a systolic array: at beat b
//     stage k rotates row b - k, so all N columns advance at once, and an
//     element (k, l) of the factor belongs to one lane;
//   - warps 1..DIM run the one-sided fits of one axis each, a side per half
//     warp, a lane per column;
//   - the estimator and the blend take a lane per field.
// Every element goes through the operations of Givens::add, solve and
// solve_normal in their order, so the results are those of the thread-per-
// particle path bit for bit.  A particle costs more FP64 instructions in all
// this way (about 2,600 a block, against 29,600 a warp of 32 particles), so
// lists beyond REDO_BLOCK_MAX particles keep the thread-per-particle path: at
// 19 cycles an instruction and SM the two meet near 6,000 particles.
//
// Measured: 16 one-sided stencils of a 205k-particle lattice 699 -> 47 us, some
// 60 particles of the 1M jet 726 -> 53 us (most of them with a first-order
// fallback), 2,200 of the 2D ensemble 267 -> 185 us.
#pragma once

#include "lp_fit_kern.cuh"

namespace lp {

constexpr unsigned long long REDO_BLOCK_MAX = 4096;

template <int DIM, int F>
struct RedoShared {
    static constexpr int N = NU<DIM>::v;
    static constexpr int C = N + F;
    double A[KMAX][C];            // row r of the scaled second-order system, then its differences
    double R[KMAX][F];            // residuals of the correction pass
    double in[2][N + 1][C];       // values entering each stage, by beat parity
    double coef[N][3];            // a_k, c, s of the beat's rotations
    double U[N][C];               // the factor: U and Z
    double d[N];
    double x[N][F];
    double g[N][F];
    double os[DIM][2][F];
    double s1[F];
    double ssr, ratio;
    FitStats<double> st;
    float invS;
    int cnt;
    int state;                    // 0 ok, 1 first-order fallback, 2 no fit
    unsigned side[2 * DIM][4];    // rows on side q = 2 k + s, a word per warp
    int nsel[2 * DIM];
    unsigned char sel[2 * DIM][16];
    int ok[2 * DIM];
};

// one stage of Givens::add: the rotation that takes entry ak of weight w into a column with diagonal d
struct Rotation { double c, s; };
__device__ __forceinline__ Rotation rotate(double ak, double& w, double& d)
{
    using O = RN<double>;
    const double wa = O::mul(w, ak);
    const double dn = O::fma(wa, ak, d);
    const bool live = O::nonzero(wa) && O::positive(dn);
    const double inv = live ? O::rcp(dn) : 0.0;
    Rotation q;
    q.s = O::mul(wa, inv);
    q.c = live ? O::mul(d, inv) : 1.0;
    w = O::mul(w, q.c);
    d = live ? dn : d;
    return q;
}

// The rotations of rows [0, cnt) of the first NN columns and the differences,
// by one warp; leaves the factor in sm.U, sm.d and, with STATS, the residual
// sum of the last field in sm.ssr.  NN: N (second order) or DIM (first order).
template <int NN, bool STATS, int DIM, int F>
__device__ void systolic_givens(RedoShared<DIM, F>& sm, int cnt)
{
    using O = RN<double>;
    constexpr int N = NU<DIM>::v, C = NN + F, NE = NN * (NN - 1) / 2 + NN * F, S = (NE + 31) / 32;
    const int lane = (int)(threadIdx.x & 31u);
    auto col = [](int c) { return c < NN ? c : N + (c - NN); };     // column of sm.A
    int ek[S], el[S];
    double u[S];
#pragma unroll
    for (int s = 0; s < S; ++s) {
        int k = 0, rem = lane + 32 * s;
        while (k < NN && rem >= C - 1 - k) { rem -= C - 1 - k; ++k; }
        ek[s] = k;                                                  // NN: no element
        el[s] = k + 1 + rem;
        u[s] = 0.0;
    }
    double dk = 0.0, w = 0.0, ssr = 0.0;
    for (int b = 0; b < cnt + NN; ++b) {
        const int p = b & 1, r = b - lane;
        const double wup = __shfl_up_sync(0xffffffffu, w, 1);
        if (lane < NN && r >= 0 && r < cnt) {
            const double ak = lane == 0 ? sm.A[b][0] : sm.in[p][lane][lane];
            w = lane == 0 ? 1.0 : wup;
            const Rotation q = rotate(ak, w, dk);
            sm.coef[lane][0] = ak;
            sm.coef[lane][1] = q.c;
            sm.coef[lane][2] = q.s;
        }
        if (STATS && lane == NN && r >= 0 && r < cnt) {             // the row's weighted leftover
            const double bl = sm.in[p][NN][C - 1];
            ssr = O::fma(O::mul(wup, bl), bl, ssr);
        }
        __syncwarp();
#pragma unroll
        for (int s = 0; s < S; ++s) {
            const int k = ek[s], rr = b - k;
            if (k < NN && rr >= 0 && rr < cnt) {
                const double v = k == 0 ? sm.A[b][col(el[s])] : sm.in[p][k][el[s]];
                const double t = O::fma(-sm.coef[k][0], u[s], v);
                u[s] = O::fma(sm.coef[k][1], u[s], O::mul(sm.coef[k][2], v));
                sm.in[p ^ 1][k + 1][el[s]] = t;
            }
        }
        __syncwarp();
    }
#pragma unroll
    for (int s = 0; s < S; ++s)
        if (ek[s] < NN) sm.U[ek[s]][el[s]] = u[s];
    if (lane < NN) sm.d[lane] = dk;
    if (STATS && lane == NN) sm.ssr = ssr;
    __syncwarp();
}

// The ratio test's value, and x = U^{-1} Z of field f, from the factor in sm.
// Rolled loops over shared memory here and in the solves below: each runs once
// per particle, and unrolled they are code that is fetched for one use (the whole
// kernel 109 us with rolled loops, 113 unrolled, two particles at 131k).
template <int NN, int DIM, int F>
__device__ double factor_ratio(const RedoShared<DIM, F>& sm)
{
    double lo = sm.d[0], hi = sm.d[0];
#pragma unroll 1
    for (int k = 1; k < NN; ++k) {
        lo = sm.d[k] < lo ? sm.d[k] : lo;
        hi = sm.d[k] > hi ? sm.d[k] : hi;
    }
    return hi > 0.0 ? sqrt(RN<double>::div(lo, hi)) : 0.0;
}

template <int NN, int DIM, int F>
__device__ void back_solve(RedoShared<DIM, F>& sm, int f)
{
#pragma unroll 1
    for (int k = NN - 1; k >= 0; --k) {
        double s = sm.U[k][NN + f];
#pragma unroll 1
        for (int l = k + 1; l < NN; ++l) s = RN<double>::fma(-sm.U[k][l], sm.x[l][f], s);
        sm.x[k][f] = s;
    }
}

// The one-sided fits of axis k (one warp; half a warp per side, lane l of it
// column l of [offsets | differences]): component k into sm.os[k], sm.ok
template <int DIM, int F>
__device__ void onesided_axis(RedoShared<DIM, F>& sm, int k, double tau_rank)
{
    using O = RN<double>;
    constexpr int N = NU<DIM>::v, C = DIM + F;
    static_assert(C <= 16, "a side's columns fit half a warp");
    const int lane = (int)(threadIdx.x & 31u), s = lane >> 4, l = lane & 15, base = lane & 16;
    const int q = 2 * k + s, m = sm.nsel[q];
    const int mx = max(__shfl_sync(0xffffffffu, m, 0), __shfl_sync(0xffffffffu, m, 16));
    double d[DIM], u[DIM];
#pragma unroll
    for (int c = 0; c < DIM; ++c) { d[c] = 0.0; u[c] = 0.0; }
    const int ac = l < DIM ? l : N + (l - DIM);
    for (int r = 0; r < mx; ++r) {
        const bool on = r < m;
        double v = on && l < C ? sm.A[sm.sel[q][r]][ac] : 0.0, w = 1.0;
#pragma unroll
        for (int c = 0; c < DIM; ++c) {
            const double ak = __shfl_sync(0xffffffffu, v, base + c);
            if (on) {
                const Rotation g = rotate(ak, w, d[c]);
                const double t = O::fma(-ak, u[c], v);
                if (l > c) {
                    u[c] = O::fma(g.c, u[c], O::mul(g.s, v));
                    v = t;
                }
            }
        }
    }
    double lo = d[0], hi = d[0];
#pragma unroll
    for (int c = 1; c < DIM; ++c) {
        lo = d[c] < lo ? d[c] : lo;
        hi = d[c] > hi ? d[c] : hi;
    }
    const double rt = hi > 0.0 ? sqrt(O::div(lo, hi)) : 0.0;
    double x[DIM];
#pragma unroll
    for (int c = DIM - 1; c >= 0; --c) {
        double z = u[c];
#pragma unroll
        for (int e = c + 1; e < DIM; ++e) z = O::fma(-__shfl_sync(0xffffffffu, u[c], base + e), x[e], z);
        x[c] = z;
    }
    if (l >= DIM && l < C) {
        double v = x[0];
#pragma unroll
        for (int c = 1; c < DIM; ++c) v = k == c ? x[c] : v;
        sm.os[k][s][l - DIM] = v * (double)sm.invS;
    }
    if (l == 0) sm.ok[q] = m >= DIM && rt >= tau_rank;
}

// The fits of particle i by the block (FIT_THREADS threads): central
// derivatives in sm.x (scaled back; sm.state tells a fallback), statistics in
// sm.st with STATS, one-sided derivatives in sm.os / sm.ok with SIDES.
template <bool STATS, bool SIDES, int DIM, int F>
__device__ void redo_fits(const FitArgs& a, int64_t i, RedoShared<DIM, F>& sm)
{
    using O = RN<double>;
    constexpr int N = NU<DIM>::v;
    const int tid = (int)threadIdx.x, w = tid >> 5, lane = tid & 31;
    const unsigned lt = (1u << lane) - 1u;
    const DevCfg& c = a.c;
    Src<double, DIM, F> src(a, i);
    const int cnt = (int)a.count[i];
    const NbGlobal nb{a.idx + i * (int64_t)c.k_max};
    const double tau = c.tau64;
    __syncthreads();                                  // the shared buffers of the block's last particle
    if (tid == 0) {
        sm.invS = inv_scale(last_d2(src, nb, cnt));
        sm.cnt = cnt;
    }
    __syncthreads();
    const double invS = (double)sm.invS;
    int sg[DIM];
#pragma unroll
    for (int k = 0; k < DIM; ++k) sg[k] = 0;
    if (tid < cnt) {
        double d[DIM], b[F], row[N];
        src.fetch(nb[tid], d, b);
#pragma unroll
        for (int k = 0; k < DIM; ++k) {
            sg[k] = d[k] > 0.0 ? 1 : (d[k] < 0.0 ? -1 : 0);
            d[k] *= invS;
        }
        gfd_row<double, DIM>(d, row);
#pragma unroll
        for (int u = 0; u < N; ++u) sm.A[tid][u] = row[u];
#pragma unroll
        for (int f = 0; f < F; ++f) sm.A[tid][N + f] = b[f];
    }
    if (SIDES) {
        // the first k_side rows of each side, in list order
#pragma unroll
        for (int q = 0; q < 2 * DIM; ++q) {
            const unsigned m = __ballot_sync(0xffffffffu, sg[q >> 1] == ((q & 1) ? 1 : -1));
            if (lane == 0) sm.side[q][w] = m;
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 2 * DIM; ++q) {
            if (sg[q >> 1] == ((q & 1) ? 1 : -1)) {
                int rank = __popc(sm.side[q][w] & lt);
                for (int v = 0; v < w; ++v) rank += __popc(sm.side[q][v]);
                if (rank < c.k_side) sm.sel[q][rank] = (unsigned char)tid;
            }
            if (tid == q) {
                int n = 0;
                for (int v = 0; v < FIT_THREADS / 32; ++v) n += __popc(sm.side[q][v]);
                sm.nsel[q] = n < c.k_side ? n : c.k_side;
            }
        }
    }
    __syncthreads();
    if (w == 0) {
        systolic_givens<N, STATS>(sm, cnt);
        if (lane == 0) {
            sm.ratio = factor_ratio<N>(sm);
            sm.state = (!(sm.ratio >= tau) || cnt < N) ? 1 : 0;
        }
        __syncwarp();
        if (sm.state == 0 && lane < F) back_solve<N>(sm, lane);
    } else {
        if (SIDES && w <= DIM) onesided_axis(sm, w - 1, tau);
        if (STATS && w == 1) {                        // the statistics of the last field's differences
            double bmin = 0.0, bmax = 0.0, ssb = 0.0;
            for (int r = 0; r < cnt; ++r) {
                const double bl = sm.A[r][N + F - 1];
                bmin = bl < bmin ? bl : bmin;
                bmax = bl > bmax ? bl : bmax;
                ssb = O::fma(bl, bl, ssb);
            }
            if (lane == 0) { sm.st.bmin = bmin; sm.st.bmax = bmax; sm.st.ssb = ssb; }
        }
    }
    __syncthreads();
    if (STATS && tid == 0) sm.st.ssr = sm.ssr;
    if (sm.state == 0) {
        if (c.refine == LP_REFINE_ALWAYS || (c.refine == LP_REFINE_AUTO && sm.ratio < c.refine_ratio)) {
            // one correction step of the semi-normal equations: residuals (a
            // thread per row and field), their products (a thread per sum, rows in
            // list order), the two triangular solves (a lane per field)
            for (int e = tid; e < cnt * F; e += FIT_THREADS) {
                const int r = e / F, f = e - r * F;
                double res = sm.A[r][N + f];
#pragma unroll
                for (int u = 0; u < N; ++u) res = O::fma(-sm.A[r][u], sm.x[u][f], res);
                sm.R[r][f] = res;
            }
            __syncthreads();
            for (int e = tid; e < N * F; e += FIT_THREADS) {
                const int u = e / F, f = e - u * F;
                double g = 0.0;
                for (int r = 0; r < cnt; ++r) g = O::fma(sm.A[r][u], sm.R[r][f], g);
                sm.g[u][f] = g;
            }
            __syncthreads();
            if (tid < F) {
#pragma unroll 1
                for (int k = 0; k < N; ++k) {
                    double s = sm.g[k][tid];
#pragma unroll 1
                    for (int l = 0; l < k; ++l) s = O::fma(-sm.U[l][k], sm.g[l][tid], s);
                    sm.g[k][tid] = s;
                }
#pragma unroll 1
                for (int k = 0; k < N; ++k) sm.g[k][tid] = O::mul(sm.g[k][tid], O::rcp(sm.d[k]));
#pragma unroll 1
                for (int k = N - 1; k >= 0; --k) {
                    double s = sm.g[k][tid];
#pragma unroll 1
                    for (int l = k + 1; l < N; ++l) s = O::fma(-sm.U[k][l], sm.g[l][tid], s);
                    sm.g[k][tid] = s;
                }
#pragma unroll 1
                for (int k = 0; k < N; ++k) sm.x[k][tid] += sm.g[k][tid];
            }
        }
        __syncthreads();
        const double s2 = invS * invS;
        if (tid < N * F) sm.x[tid / F][tid % F] *= tid / F < DIM ? invS : s2;
    } else {
        // the first-order fit over the whole list; zero where that is deficient too
        if (w == 0) {
            systolic_givens<DIM, false>(sm, cnt);
            if (lane == 0 && (!(factor_ratio<DIM>(sm) >= tau) || cnt < DIM)) sm.state = 2;
            __syncwarp();
            if (lane < F) {
                if (sm.state == 1) back_solve<DIM>(sm, lane);
#pragma unroll
                for (int u = 0; u < N; ++u)
                    sm.x[u][lane] = sm.state == 1 && u < DIM ? sm.x[u][lane] * invS : 0.0;
            }
        }
    }
    __syncthreads();
}

// one step of particle i: the stages of step_one on the block's fits
template <int DIM, bool GATE>
__device__ void redo_step_block(const FitArgs& a, const StepOut& o, int64_t i, RedoShared<DIM, DIM + 2>& sm)
{
    constexpr int F = DIM + 2;
    constexpr int N = NU<DIM>::v;
    redo_fits<GATE, true>(a, i, sm);
    if (threadIdx.x >= 32) return;                    // (redo_fits starts with a barrier)
    const int lane = (int)threadIdx.x;
    const DevCfg& c = a.c;
    Loaded<DIM> L;
    step_load<double, DIM>(a, o, i, L);               // never frozen: frozen particles are not listed
    double cd[N][F], cdf[DIM][F], lw[F];
#pragma unroll
    for (int u = 0; u < N; ++u)
#pragma unroll
        for (int f = 0; f < F; ++f) cd[u][f] = sm.x[u][f];
    if (lane == 0) {
        if (sm.state) atomicAdd(a.counters + C_LINEAR, 1ull);
        if (sm.state == 2) atomicAdd(a.counters + C_NOFIT, 1ull);
    }
    bool mlp_skip = false;
    if (GATE && (o.features || c.estimator == LP_EST_MLP)) {
        // (central_gate's steps, the hidden units a lane each)
        float xf[MLP_IN];
        mlp_features<double, DIM>(cd, sm.st, sqrt(a.d2min[i]), L.s0[0], L.s0[F - 1], c.gamma, xf);
        if (o.features && lane < MLP_IN) {
            float v = xf[0];
#pragma unroll
            for (int k = 1; k < MLP_IN; ++k) v = lane == k ? xf[k] : v;
            o.features[i * MLP_IN + lane] = v;
        }
        if (c.estimator == LP_EST_MLP) {
            const float pg = mlp_prob_warp(xf, a.mlp_w);
            mlp_skip = pg < c.mlp_tau_lo;
            if (lane == 0) {
                if (o.gate_p) o.gate_p[i] = pg;
                atomicAdd(a.counters + (mlp_skip ? C_MLP_SKIP : C_MLP_UNCERTAIN), 1ull);
            }
        }
    }
    central_rates<double, DIM>(a, L, cd, cdf, lw);
    const bool plain = !mlp_skip || c.mlp_audit;
    double os[DIM][2][F];
#pragma unroll
    for (int k = 0; k < DIM; ++k)
#pragma unroll
        for (int s = 0; s < 2; ++s)
#pragma unroll
            for (int f = 0; f < F; ++f) os[k][s][f] = plain && sm.ok[2 * k + s] ? sm.os[k][s][f] : cdf[k][f];
    double uw[F];
    upwind_rates<double, DIM>((double)c.gamma, L.s0[0], L.s0[F - 1], os, uw);
    // lane f: the estimator, limiter and blend of field f
    const int f = lane < F ? lane : 0;
    double sl[DIM], sr[DIM], s0f = L.s0[0], uwf = uw[0], lwf = lw[0];
#pragma unroll
    for (int q = 1; q < F; ++q) {
        s0f = f == q ? L.s0[q] : s0f;
        uwf = f == q ? uw[q] : uwf;
        lwf = f == q ? lw[q] : lwf;
    }
#pragma unroll
    for (int k = 0; k < DIM; ++k) {
        sl[k] = os[k][0][0];
        sr[k] = os[k][1][0];
#pragma unroll
        for (int q = 1; q < F; ++q) {
            sl[k] = f == q ? os[k][0][q] : sl[k];
            sr[k] = f == q ? os[k][1][q] : sr[k];
        }
    }
    double rs = plain ? estimator_r<double, DIM>(sl, sr, sqrt(a.d2min[i]), s0f, c.s_ref[f], c.flat_eps, c.active_frac)
                      : 1.0;
    bool any = __any_sync(0xffffffffu, rs > 1.5);
    if (lane == 0 && mlp_skip && any) atomicAdd(a.counters + C_MLP_MISS, 1ull);
    if (mlp_skip) { any = false; rs = 1.0; }
    double p;
    const double s1 = blend_field<double>(c, L.dt, s0f, uwf, lwf, rs, any, p);
    if (lane < F) {
        if (o.phi) o.phi[i * F + f] = (float)p;
        if (o.r) o.r[i * F + f] = (float)rs;
        sm.s1[f] = s1;
    }
    __syncwarp();
    double s1v[F];
#pragma unroll
    for (int q = 0; q < F; ++q) s1v[q] = sm.s1[q];
    if (lane == 0) {
        store_state<DIM>(a, o, i, L, s1v, any);
        if (any) atomicAdd(a.counters + C_FLAGGED, 1ull);
    }
}

// The redo kernels: a block per particle for a short list, a thread per
// particle beyond REDO_BLOCK_MAX.
template <int DIM, bool GATE>
__global__ void __launch_bounds__(FIT_THREADS) k_step_redo(FitArgs a, StepOut o)
{
    __shared__ RedoShared<DIM, DIM + 2> sm;
    const unsigned long long len = *a.list_len;
    if (len <= REDO_BLOCK_MAX) {
        for (unsigned long long t = blockIdx.x; t < len; t += gridDim.x)
            redo_step_block<DIM, GATE>(a, o, a.list[t], sm);
        return;
    }
    for (unsigned long long t = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; t < len;
         t += (unsigned long long)gridDim.x * blockDim.x)
        step_one<double, DIM, GATE>(a, o, a.list[t]);
}

template <int DIM, int F>
__global__ void __launch_bounds__(FIT_THREADS) k_derivs_redo(FitArgs a, DerivOut o)
{
    __shared__ RedoShared<DIM, F> sm;
    constexpr int N = NU<DIM>::v;
    const unsigned long long len = *a.list_len;
    if (len <= REDO_BLOCK_MAX) {
        for (unsigned long long t = blockIdx.x; t < len; t += gridDim.x) {
            const int64_t i = a.list[t];
            redo_fits<false, false>(a, i, sm);
            const int state = sm.state;
            const int e = (int)threadIdx.x;
            if (e == 0) {
                if (state) atomicAdd(a.counters + (state == 2 ? C_NOFIT : C_LINEAR), 1ull);
                if (o.status && o.f_first == 0)
                    o.status[i] = FIT_FP64 | (state ? FIT_LINEAR : 0u) | (state == 2 ? FIT_NONE : 0u);
            }
            if (e < N * o.f_real) {
                const int f = e / N, u = e - f * N;
                const int64_t at = ((int64_t)(o.f_first + f) * a.n + i) * N + u;
                if (o.out_f64) static_cast<double*>(o.out)[at] = sm.x[u][f];
                else static_cast<float*>(o.out)[at] = (float)sm.x[u][f];
            }
        }
        return;
    }
    for (unsigned long long t = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; t < len;
         t += (unsigned long long)gridDim.x * blockDim.x)
        derivs_one<double, DIM, F>(a, o, a.list[t], NbGlobal{a.idx + (int64_t)a.list[t] * (int64_t)a.c.k_max});
}

template <int DIM, int F>
__global__ void __launch_bounds__(FIT_THREADS) k_onesided_redo(FitArgs a, double* out, int f_real)
{
    __shared__ RedoShared<DIM, F> sm;
    const unsigned long long len = *a.list_len;
    if (len <= REDO_BLOCK_MAX) {
        for (unsigned long long t = blockIdx.x; t < len; t += gridDim.x) {
            const int64_t i = a.list[t];
            redo_fits<false, true>(a, i, sm);
            const int e = (int)threadIdx.x;
            if (e < 2 * DIM * f_real) {
                const int q = e / f_real, f = e - q * f_real;
                out[(i * 2 * DIM + q) * f_real + f] = sm.ok[q] ? sm.os[q >> 1][q & 1][f] : sm.x[q >> 1][f];
            }
        }
        return;
    }
    for (unsigned long long t = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; t < len;
         t += (unsigned long long)gridDim.x * blockDim.x)
        onesided_one<double, DIM, F>(a, out, f_real, a.list[t]);
}

}  // namespace lp
