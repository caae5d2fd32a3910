// The FP64 duality gap of Sec. 3.3.3: per-pixel terms, their sums, the gap, the residual and the
// stopping test (device side; K's gap epilogue and the wavelet model use it).
#pragma once

#include <cuda_runtime.h>

#include "pat_internal.cuh"
#include "reduce.cuh"
#include "stencil.cuh"

namespace pat {

// ---------------------------------------------------------------------------------
// FP64 duality gap over pixels (Sec. 3.3.3, box-restricted reading)
// terms: {R1, R2, |K^T q - div r|_1, |E^T s - r|_1, |x - x_old|^2, |x_old|^2, dual residual}
// ---------------------------------------------------------------------------------
constexpr int GAP_PIX_TERMS = 7;   // sums over pixels
constexpr int GAP_TERMS = GAP_DATA_TERMS + GAP_PIX_TERMS;

// Distance of g from the normal cone of the radius-ball at p: the cone is {0} inside the
// ball and the ray through p on its sphere (the dual residual of a ball-constrained dual).
__device__ __forceinline__ float cone_distance2(float g0, float g1, float p0, float p1, float radius) {
    const float np = sqrtf(p0 * p0 + p1 * p1);
    const float lam = np >= radius * (1.f - 1e-6f) && np > 0.f ? fmaxf(0.f, (g0 * p0 + g1 * p1) / np) : 0.f;
    return sqrtf(fmaxf(g0 * g0 + g1 * g1 - lam * lam, 0.f));
}
__device__ __forceinline__ float cone_distance3(float g0, float g1, float g2, float p0, float p1, float p2,
                                                float radius) {
    const float np = sqrtf(p0 * p0 + p1 * p1 + p2 * p2);
    const float lam =
        np >= radius * (1.f - 1e-6f) && np > 0.f ? fmaxf(0.f, (g0 * p0 + g1 * p1 + g2 * p2) / np) : 0.f;
    return sqrtf(fmaxf(g0 * g0 + g1 * g1 + g2 * g2 - lam * lam, 0.f));
}

struct GapArgs {
    int n;
    float alpha, ab;      // ball radii of r and s
    double gamma;
    const float* xi;
    const float* x;       // x^{n+1}
    const float* x_old;   // x^n (NULL: residual terms are zero)
    const float* y;       // r, s at the same evaluation (y^{n+1})
    KtView kt;            // K^T q^{n+1} (fixed point)
    int reg;
};

// Adds the terms of pixels first, first + step, ... to acc: per-thread sums in FP32 (a thread
// covers few pixels, see gap_ctas; the block's sums are FP32 pairs per warp and FP64 across warps, since
// GB300's FP64 pipe runs at 1/64 of FP32).  The last term is the dual residual of the
// regulariser duals (distance of their argument from the normal cone of the ball at r and s),
// for the adaptive balance.
template <int REG>
__device__ __forceinline__ void gap_pixels(const GapArgs& a, const int first, const int step, float (&acc)[GAP_PIX_TERMS]) {
    const int N = a.n;
    const size_t NN = (size_t)N * N;
    const float gam = (float)a.gamma;
    const float alpha = a.alpha, ab = a.ab;
    auto X = [&](int c, int x, int y) -> float { return __ldg(a.x + c * NN + (size_t)y * N + x); };
    auto Yf = [&](int c, int x, int y) -> float { return __ldg(a.y + c * NN + (size_t)y * N + x); };
    // r masked for div (dTV: D_xi r), zero outside the grid
    auto rm = [&](int c, int x, int y) -> float {
        if (x < 0 || y < 0 || (c == 0 && x >= N - 1) || (c == 1 && y >= N - 1)) return 0.f;
        float r0 = Yf(0, x, y), r1 = Yf(1, x, y);
        if (REG == PAT_DTV) {
            float o0, o1;
            dxi_apply(__ldg(a.xi + (size_t)y * N + x), __ldg(a.xi + NN + (size_t)y * N + x), gam, r0, r1, o0, o1);
            r0 = o0;
            r1 = o1;
        }
        return c == 0 ? r0 : r1;
    };
    for (int p = first; p < N * N; p += step) {   // N <= 16384
        const int gy = p / N, gx = p - gy * N;
        const bool ax = gx < N - 1, by = gy < N - 1;
        const float u = X(0, gx, gy);
        float g0 = ax ? X(0, gx + 1, gy) - u : 0.f;
        float g1 = by ? X(0, gx, gy + 1) - u : 0.f;
        if (REG == PAT_DTV) {
            float o0, o1;
            dxi_apply(__ldg(a.xi + p), __ldg(a.xi + NN + p), gam, g0, g1, o0, o1);
            g0 = o0;
            g1 = o1;
        }
        if (REG == PAT_TGV) {
            g0 -= X(1, gx, gy);
            g1 -= X(2, gx, gy);
        }
        acc[0] += sqrtf(g0 * g0 + g1 * g1);
        acc[6] += cone_distance2(g0, g1, Yf(0, gx, gy), Yf(1, gx, gy), alpha);
        // box term of u: |K^T q - div r|; near convergence the two sides agree closely and
        // their FP32 difference is exact (Sterbenz), so FP32 keeps the term's precision
        const float divr = (rm(0, gx, gy) - rm(0, gx - 1, gy)) + (rm(1, gx, gy) - rm(1, gx, gy - 1));
        const float atu = a.kt.at(gx, gy, N) - divr;
        acc[2] += fabsf(atu);
        if (REG == PAT_TGV) {
            auto vm = [&](int c, int x, int y, bool mx) -> float {  // masked v for d^-
                if (x < 0 || y < 0 || (mx ? (x >= N - 1) : (y >= N - 1))) return 0.f;
                return X(1 + c, x, y);
            };
            const float e11 = vm(0, gx, gy, true) - vm(0, gx - 1, gy, true);
            const float e22 = vm(1, gx, gy, false) - vm(1, gx, gy - 1, false);
            const float e12 = ((vm(0, gx, gy, false) - vm(0, gx, gy - 1, false)) +
                               (vm(1, gx, gy, true) - vm(1, gx - 1, gy, true))) * kInvSqrt2f;
            acc[1] += sqrtf(e11 * e11 + e22 * e22 + e12 * e12);
            const float s11 = Yf(2, gx, gy), s22 = Yf(3, gx, gy), s12 = Yf(4, gx, gy);
            acc[6] += cone_distance3(e11, e22, e12, s11, s22, s12, ab);
            const float dx11 = ax ? Yf(2, gx + 1, gy) - s11 : 0.f;
            const float dy12 = by ? Yf(4, gx, gy + 1) - s12 : 0.f;
            const float dy22 = by ? Yf(3, gx, gy + 1) - s22 : 0.f;
            const float dx12 = ax ? Yf(4, gx + 1, gy) - s12 : 0.f;
            const float et1 = -dx11 - dy12 * kInvSqrt2f, et2 = -dy22 - dx12 * kInvSqrt2f;
            acc[3] += fabsf(et1 - Yf(0, gx, gy)) + fabsf(et2 - Yf(1, gx, gy));
        }
        if (a.x_old) {
            const int nc = REG == PAT_TGV ? 3 : 1;
            for (int c = 0; c < nc; ++c) {
                const float xn = X(c, gx, gy), xo = __ldg(a.x_old + c * NN + p);
                acc[4] += (xn - xo) * (xn - xo);
                acc[5] += xo * xo;
            }
        }
    }
}

struct InfoDev {
    double primal, dual, gap, rel_gap, residual;
    int iters_done, status, stop, iter;
    unsigned qmax_bits[2];  // max |q| of iterations of each parity (float bits)
    unsigned final_ticket;  // blocks of the pixel pass done (the last one resets it)
    float step_mul[2];      // {s, 1/s}: primal and dual step multipliers
    int n_adjust;           // adaptive-balance adjustments so far
};

struct FinalArgs {
    const double* data_part;   // term c of CTA b at [c * n_data + b]; pix_part alike
    int n_data;
    const double* pix_part;
    int n_pix;
    double alpha, beta, box_u, box_v, tol;
    int reg, adapt;
    InfoDev* info;
    int* batch_stopped;    // problems of the batch that have stopped (the host polls it)
};

// Adaptive primal-dual balance (residual balancing after Goldstein, Li, Yuan, Esser and
// Baraniuk 2015), in L1 norms at the evaluated state:
//  - primal residual |A^T y|_1 (G = 0, so A^T y = 0 at a solution);
//  - dual residual: |q - (Ku - f)|_1, plus the distance of grad u - v (dTV: D_xi grad u)
//    and of E v from the normal cones of the r- and s-balls.
// When one exceeds the other by more than BAL_DEAD, s (the primal step multiplier) moves
// toward balance by the square root of their ratio, clamped to a factor BAL_MAX_STEP.  The
// exponent decays by BAL_DECAY per adjustment, so s settles.
constexpr double BAL_DEAD = 2.0, BAL_MAX_STEP = 2.0, BAL_DECAY = 0.97, BAL_MIN = 1e-3, BAL_MAX = 1e3;

__device__ __forceinline__ void balance_update(InfoDev* in, double primal_res, double dual_res) {
    if (!(primal_res > 0 && dual_res > 0)) return;
    const double rho = primal_res / dual_res;
    if (rho >= 1.0 / BAL_DEAD && rho <= BAL_DEAD) return;
    const double f = fmin(fmax(sqrt(rho), 1.0 / BAL_MAX_STEP), BAL_MAX_STEP);
    double s = (double)in->step_mul[0] * pow(f, pow(BAL_DECAY, (double)in->n_adjust));
    s = fmin(fmax(s, BAL_MIN), BAL_MAX);
    in->step_mul[0] = (float)s;
    in->step_mul[1] = (float)(1.0 / s);
    in->n_adjust += 1;
}

// The summed terms of a problem from its partial sums, by one block (of at least 8 warps) in
// a fixed order: a warp takes whole terms, lane l of it the partials l, l + 32, ..., then a
// shuffle tree.  What bounds it is the FP64 pipe (16 clocks for a warp's addition) and the
// chain of dependent additions, so no warp repeats another's work and the terms of a warp
// overlap.
__device__ __forceinline__ void gap_sum_terms(const FinalArgs& f, double (&s_tot)[GAP_TERMS]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int NW = blockDim.x >> 5;
    constexpr int PER = (GAP_TERMS + 7) / 8;
    double v[PER];
#pragma unroll
    for (int e = 0; e < PER; ++e) {
        const int c = warp + e * NW;
        v[e] = 0.0;
        if (c >= GAP_TERMS) continue;
        const bool pix = c >= GAP_DATA_TERMS;
        const int n = pix ? f.n_pix : f.n_data;
        const double* part = pix ? f.pix_part + (size_t)(c - GAP_DATA_TERMS) * n : f.data_part + (size_t)c * n;
        for (int b0 = lane; b0 < n; b0 += 32 * 8) {   // eight loads in flight
            double x[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) x[k] = b0 + 32 * k < n ? __ldcg(part + b0 + 32 * k) : 0.0;
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (b0 + 32 * k < n) v[e] += x[k];
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int e = 0; e < PER; ++e) v[e] += __shfl_down_sync(0xffffffffu, v[e], o);
#pragma unroll
    for (int e = 0; e < PER; ++e)
        if (lane == 0 && warp + e * NW < GAP_TERMS) s_tot[warp + e * NW] = v[e];
    __syncthreads();
}

// The gap, the residual and the stopping test from the summed terms (thread 0; the residual,
// which nothing else needs, in a thread of another warp at the same time).
__device__ __forceinline__ void gap_evaluate(const FinalArgs& a, const double (&t)[GAP_TERMS]) {
    InfoDev* in = a.info;
    if (threadIdx.x == 32) {
        const double dx2 = t[8], x2 = t[9];
        in->residual = x2 > 0 ? sqrt(dx2 / x2) : (dx2 == 0 ? 0.0 : INFINITY);
    }
    if (threadIdx.x != 0) return;
    const double res2 = t[0], q2 = t[1], qf = t[2], dres_q = t[3];
    const double r1 = t[4], r2 = t[5], bu = t[6], bv = t[7], dres_rs = t[10];
    const double reg = a.reg == PAT_TGV ? r1 + a.beta * r2 : r1;
    const double primal = 0.5 * res2 + a.alpha * reg;
    const double dual = -(0.5 * q2 + qf) - a.box_u * bu - (a.reg == PAT_TGV ? a.box_v * bv : 0.0);
    const double gap = primal - dual;
    const double rel = primal > 0 ? gap / primal : (gap == 0 ? 0.0 : INFINITY);
    in->primal = primal;
    in->dual = dual;
    in->gap = gap;
    in->rel_gap = rel;
    in->iters_done = in->iter;
    if (!isfinite(gap) || !isfinite(primal)) {
        in->status = PAT_STATUS_DIVERGED;
        in->stop = 1;
        if (a.batch_stopped) atomicAdd(a.batch_stopped, 1);
    } else if (a.tol > 0 && rel <= a.tol) {
        in->status = PAT_STATUS_CONVERGED;
        in->stop = 1;
        if (a.batch_stopped) atomicAdd(a.batch_stopped, 1);
    } else if (a.adapt == PAT_ADAPT_BALANCE) {
        balance_update(in, bu + (a.reg == PAT_TGV ? bv : 0.0), dres_q + dres_rs);
    }
}

}  // namespace pat
