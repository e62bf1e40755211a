// Inverse evaluation of a mapped-Chebyshev expansion at arbitrary velocities:
//   u_N(v) = sum_k u~_k prod_l T~_{k_l}(v_l),  T~_k(v) = mu(xi)^4 T_k(xi) / sqrt(c_k),  xi = xi(v)
// (Eq. fN_Expansion with the trial functions of Eq. 1DCheby).  Given the weak-form
// coefficients Q_k of the collision operator it returns Q_N(v), the trial-space function whose
// coefficients they are (the trial and test functions are biorthonormal), so errors against a
// closed-form Q can be measured on a grid of velocities without leaving the device.
//
// One thread per point.  The sum over the last axis is cut into chunks of at most 32 coefficients
// whose T_k(x_l) a thread keeps in registers; for every row of coefficients (the leading axes' modes) a
// chunk is one FMA per coefficient -- every thread of a warp reads the same coefficient, a broadcast
// load -- and the rows go through a Clenshaw recurrence per leading axis.  Both run from the highest mode
// down, so that the small terms are added first: the error on smooth densities is that of a Clenshaw
// recurrence on every axis (2.8e-16 of the values at N = 48, logarithmic map, where sums from the lowest mode up
// left 4.4e-16).
//
// The FP64 pipe bounds it (two operations per SM and cycle on this GPU): Clenshaw recurrences
// on every axis take two operations per coefficient, this form one and two per row.  Blocks of one warp, so that
// the points spread evenly over the SMs, and registers for 12 of them per SM, so that a row's loads are all in
// flight at once (with the compiler's own choice few points were slower: N = 120, one point 0.68 ms instead of
// 0.61).  200 x 200 points at N = 48, 2D: 705 us with recurrences on every axis, 237 us so (one FMA per
// coefficient at the measured 5.3e11/s: 182 us).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "host.cuh"

#define PG_API extern "C" __attribute__((visibility("default")))

using namespace pgbh;

namespace {

constexpr double kSqrt2OverPi = 0.79788456080286535588;  // 1/sqrt(c_k), k >= 1
constexpr double kInvSqrtPi = 0.56418958354775628695;    // 1/sqrt(c_0)

// xi(v) and mu(xi)^4 = (1 - xi^2)^(1+r) / S^2 (Eq. 1D_mu_function), with 1 - xi^2 in a form
// without cancellation: sech^2(v/S) for the logarithmic map xi = tanh(v/S), S^2/(S^2 + v^2) for
// the algebraic map xi = v / sqrt(S^2 + v^2).
__device__ void map_point(double v, double S, int r, double &xi, double &mu4)
{
    double om;
    if (r == 0) {
        const double t = v / S;
        xi = tanh(t);
        const double ch = cosh(t);
        om = 1.0 / (ch * ch);
        mu4 = om / (S * S);
    } else {
        const double h = hypot(S, v);
        xi = v / h;
        om = S / h;
        om *= om;
        mu4 = om * om / (S * S);
    }
}

// sum_k a_k T_k(x) / sqrt(c_k), k = 0..N, of coefficients that next() gives from a_N down to a_0:
// sum_{k>=1} a_k T_k(x) = x b_1 - b_2 with b_k = a_k + 2 x b_{k+1} - b_{k+2}.
template <typename F>
__device__ __forceinline__ double clenshaw(int N, double x, F next)
{
    const double two_x = 2.0 * x;
    double b1 = 0.0, b2 = 0.0;
    for (int k = N; k > 0; --k) {
        const double t = fma(two_x, b1, next() - b2);
        b2 = b1;
        b1 = t;
    }
    const double a0 = next();
    return kSqrt2OverPi * fma(x, b1, -b2) + kInvSqrtPi * a0;
}

constexpr int kEvalThreads = 32;

// C: coefficients of the last axis per chunk.
template <int D, int C>
__global__ void __launch_bounds__(kEvalThreads, 12) k_evaluate(int N, double S, int r, const double *__restrict__ u,
                                                           long long npts, const double *__restrict__ pts,
                                                           double *__restrict__ out)
{
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < npts; p += stride) {
        double x[D];
        double w = 1.0;
        for (int l = 0; l < D; ++l) {
            double m4;
            map_point(pts[p * D + l], S, r, x[l], m4);
            w *= m4;
        }
        double total = 0.0;
        double ta = kInvSqrtPi, tb = kSqrt2OverPi * x[D - 1];  // the last axis' T_k/sqrt(c_k) and T_{k+1}/sqrt(c_{k+1})
        for (int done = 0; done <= N; done += C) {
            // the last chunk ends with the row: coefficients that were added before are multiplied by 0
            const int c0 = min(done, N + 1 - C);
            double T[C];
#pragma unroll
            for (int k = 0; k < C; ++k) {
                T[k] = 0.0;
                if (c0 + k < done) continue;
                T[k] = ta;
                // T_{k+2} = 2 x T_{k+1} - T_k, with T_0 in the scale of the others
                const double prev = (c0 + k == 0) ? kSqrt2OverPi : ta;
                ta = tb;
                tb = fma(2.0 * x[D - 1], tb, -prev);
            }
            auto row = [&](const double *q) {
                double s0 = 0.0, s1 = 0.0;
#pragma unroll
                for (int k = C - 1; k >= 0; --k) {
                    const double c = __ldg(q + k);
                    if (k & 1) s1 = fma(c, T[k], s1);
                    else s0 = fma(c, T[k], s0);
                }
                return s0 + s1;
            };
            // rows of the leading axes' modes, from the last one down
            const double *q = u + c0 + (D == 3 ? (size_t)(N + 1) * (N + 1) * (N + 1) : (size_t)(N + 1) * (N + 1));
            auto next_row = [&]() { return row(q -= N + 1); };
            if constexpr (D == 2) total += clenshaw(N, x[0], next_row);
            else total += clenshaw(N, x[0], [&]() { return clenshaw(N, x[1], next_row); });
        }
        out[p] = w * total;
    }
}

// Dispatch on the chunk size, 3 .. 32.
template <int D, int C>
void launch_evaluate(int c, int blocks, cudaStream_t s, int N, double S, int r, const double *u, long long npts,
                     const double *pts, double *out)
{
    if (c == C) k_evaluate<D, C><<<blocks, kEvalThreads, 0, s>>>(N, S, r, u, npts, pts, out);
    else if constexpr (C < 32) launch_evaluate<D, C + 1>(c, blocks, s, N, S, r, u, npts, pts, out);
}

}  // namespace

PG_API int pg_boltz_evaluate(pg_boltz_plan_t *p, const double *coef_dev, long long npts, const double *pts_dev,
                             double *out_dev)
{
    if (!p) return set_error(PG_ERR_ARG, "plan is NULL");
    if (p->batch) return set_error(PG_ERR_STATE, "evaluation is not available on batched plans");
    if (npts < 0) return set_error(PG_ERR_ARG, "npts must be >= 0");
    if (npts == 0) return PG_OK;
    if (!coef_dev || !pts_dev || !out_dev) return set_error(PG_ERR_ARG, "NULL device pointer");
    DeviceGuard guard(p->device);
    if (!guard.ok) return set_error(PG_ERR_CUDA, "cannot select the plan's device");
    // as few chunks of the last axis as 32 values in registers allow
    const int chunks = (p->N + 32) / 32, C = (p->N + chunks) / chunks;
    const int blocks = (int)std::min<long long>((npts + kEvalThreads - 1) / kEvalThreads, 1 << 20);
    if (p->d == 2)
        launch_evaluate<2, 3>(C, blocks, p->stream, p->N, p->S, p->r, coef_dev, npts, pts_dev, out_dev);
    else
        launch_evaluate<3, 3>(C, blocks, p->stream, p->N, p->S, p->r, coef_dev, npts, pts_dev, out_dev);
    return cuda_check(cudaGetLastError(), "evaluation kernel");
}
