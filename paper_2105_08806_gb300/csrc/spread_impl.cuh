// Spreading kernel templates shared by the FP32 and FP64 translation units.
//
// Fused post-collision point generation + exponential-of-semicircle spreading onto
// the folded cosine grid (Section 4.2, Eq. num_fast_k and Eq. nufft).
//
// One thread owns one class of node pairs (PairData: the pairs (i, j) that share their points) and walks the M sphere points sigma_m:
//   v'     = (v_i + v_j)/2 + |v_i - v_j| sigma_m / 2
//   z_l    = arccos(xi(v'_l))                     angle of the l-th mapped coordinate
//   q      = a_i a_j B(|v_i - v_j|) w_m prod_l mu(xi(v'_l))^-2
// and adds q prod_l psi(x_{g_l} - z_l) to the w^d cells of the folded grid around z.
// The gain coefficient is the cosine sum sum_p q_p prod_l cos(k_l z_pl); cos is even
// and 2 pi periodic, so the periodic grid of n cells folds onto its n/2 + 1 cells
// g = 0..n/2: every unfolded support index u is added at fold(u) = min(u mod n, n - u mod n).
//
// Stable forms of the angle and the weight from the map formulas of Section 2.1:
//   r = 1 (algebraic):   cos z = v/sqrt(S^2+v^2), sin z = S/sqrt(S^2+v^2)
//                        -> z = atan2(S, v),      mu^-2 = (S^2 + v^2)/S
//   r = 0 (logarithmic): cos z = tanh(v/S), sin z = sech(v/S)
//                        -> z = 2 atan(e^(-v/S)), mu^-2 = S cosh(v/S)
//                           (FP64: from e = e^-|v/S| <= 1, z = 2 atan(e) or pi - 2 atan(e))
// Kernel values: FP32 from ex2.approx / rsqrt.approx of the definition; FP64 from per-tap
// polynomials fitted on the host (kernel_weights_f64).
//
// Accumulation:
//  - the global folded grid holds int64 values in units of 2^-Eg, where B >= sum_p |q_p|
//    (an upper bound written by the loss kernel) and B 2^Eg <= 2^61: no cell can overflow,
//    and block partial sums add exactly and in any order;
//  - FP64 kernel: each block adds into a private copy of its slab of the grid in shared memory
//    that holds each cell as a 96-bit integer, 32 bits finer than the grid unit, in three 32-bit
//    words (WideTile: native 32-bit atomics, the next word's only when a carry or a high part
//    needs it).  The kernel weights are FP64; per point, a row factor R = round(q psi_a 2^(Eg+s))
//    with a per-point scale s that keeps R below 2^62 (3D: then round(R psi_b) in integers) is
//    formed once per row, and each contribution is round(R psi_c) from a 63-bit fixed-point psi_c
//    by four 32 x 32-bit integer products, so no FP64 operation runs per cell (the FP64 pipe of
//    this GPU runs at about 1/70 of the FP32 rate) and each contribution keeps about 2^-61 of its
//    size plus 2^-32 grid units.  At the end each cell rounds to the grid unit once per block.
//  - FP32 kernel: the private copy holds one signed 32-bit word per cell in units of 2^-Et,
//    Et = Eg - tile_bits(d), plus per-cell carry counters in a per-block global array (SplitTile):
//    the cell's value is word + 2^32 carry.  A contribution goes to its word with one native 32-bit
//    shared atomic, and only an addition that overflows the word's signed range (seen from the
//    returned old value) moves the cell's carry counter; the wraps of a run of w cells are
//    collected in a register mask and their carries added after the run.  (Floating-point shared atomics are
//    compare-and-swap loops and their rounding limits FP32 accuracy; 64-bit integer shared atomics
//    are several times slower than 32-bit ones.)  Points below 2^29 tile units -- nearly all of
//    them -- form their contributions in integers: the row factor 4 q psi_a (psi_b) and the column
//    factor 2^30 psi_c are rounded once per row and column, and a contribution is the rounded high
//    word of their 64-bit product (one integer multiply-add); larger points do the same on a coarser
//    unit of their own.  At the end each block adds
//    word + 2^32 carry (scaled by 2^tile_bits(d)) to the global grid.  Each contribution is rounded
//    to the tile unit (at most about one unit); all later additions are exact.
//
// Negligible classes: in the FP32 kernels a class whose strength bound keeps every one of its points
// below 0.1 tile unit adds exactly zero (every contribution rounds to zero), so it is skipped, and
// so are such points one by one; the FP64 kernels skip classes whose summed bounds stay below
// 2^-64 B (2^-3 grid units in all).  The FP32 kernels and the FP64 2D kernel queue the classes (items)
// that are not negligible per warp, so that its lanes spread together (with the node sets of the
// workloads here, up to 70% of all classes lie in the tails of f and are skipped).
#pragma once

#include <climits>
#include <cuda_runtime.h>

#include "pgb_internal.cuh"

namespace pgb {
namespace spread_detail {

template <typename T>
struct Fn;

template <>
struct Fn<float> {
    static __device__ __forceinline__ float sqrt_(float x) { return sqrtf(x); }
    static __device__ __forceinline__ float atan2_(float y, float x) { return atan2f(y, x); }
    static __device__ __forceinline__ float cosh_(float x) { return coshf(x); }
    static __device__ __forceinline__ float pow_(float x, float y) { return powf(x, y); }
    static __device__ __forceinline__ float floor_(float x) { return floorf(x); }
};

template <>
struct Fn<double> {
    static __device__ __forceinline__ double sqrt_(double x) { return sqrt(x); }
    static __device__ __forceinline__ double atan2_(double y, double x) { return atan2(y, x); }
    static __device__ __forceinline__ double cosh_(double x) { return cosh(x); }
    static __device__ __forceinline__ double pow_(double x, double y) { return pow(x, y); }
    static __device__ __forceinline__ double floor_(double x) { return floor(x); }
};

// Fold an unfolded periodic index u onto 0..n/2.
__device__ __forceinline__ int fold_index(int u, int n)
{
    int g = u % n;
    if (g < 0) g += n;
    return (g > (n >> 1)) ? n - g : g;
}

// 2^e as a float, 0 below the normal range (e <= 127).
__device__ __forceinline__ float exp2_int(int e) { return __int_as_float(max(e + 127, 0) << 23); }

// Unfolded index u of a point's support -> folded cell: min(|u|, |n - |u||), which is fold(u) for |u| <= 3n/2.
// A support reaches at most w/2 beyond [0, n/2], so |u| <= n/2 + w/2, and w <= 2n for every plan (n >= 8,
// w <= 16): no modulo and no branch (a general path here, never taken but for the smallest grids, was
// inlined at every tap row; with the guards of the inner taps, below, 1-4% of every FP32 evaluation).
__device__ __forceinline__ int fold_cell(int u, int n)
{
    u = abs(u);
    return min(u, abs(n - u));
}

// Kernel weights psi(x_u - z) of one axis, u = s..s+w-1, in units where one grid cell is 1 and
// x = z n / (2 pi): psi = exp(beta (sqrt(1 - t^2) - 1)), t = (u - x) 2/w.

// FP64: psi of tap a is a polynomial (kernel_poly_terms(w) terms) in the point's offset
// y = 2 (s - x) + w - 1 in (-1, 1] (t = (y + 1 + 2a - w)/w), fitted on the host.  Taps a and
// w-1-a mirror each other (t_{w-1-a}(-y) = -t_a(y) and psi is even), so one even part E_a(y^2)
// and one odd part y O_a(y^2) give both: about w + 2 FMAs per tap pair instead of an exp and a
// sqrt per tap.
// The coefficients sit in shared memory (s_kpoly, filled by load_kernel_poly at the start of each
// FP64 spreading kernel) and are read through an offset the compiler cannot see to be zero: read
// in place they cost one shared load each, whereas hoisted out of the point loops they would
// hold ~4 registers per tap and coefficient (spills at w >= 15).
__shared__ double s_kpoly[kPolyCoefF64];

__device__ __forceinline__ void load_kernel_poly(const double *kpoly)
{
    for (int k = threadIdx.x; k < kPolyCoefF64; k += blockDim.x) s_kpoly[k] = kpoly[k];
}

template <int W>
__device__ __forceinline__ int kernel_weights_f64(double x, double *wt)
{
    constexpr int P = kernel_poly_terms(W), NE = (P + 1) / 2, NO = P / 2;
    int zero;
    asm volatile("mov.b32 %0, 0;" : "=r"(zero));
    const double *cb = s_kpoly + zero;
    const int s = (int)floor(x - 0.5 * W) + 1;
    const double y = fma(2.0, double(s) - x, double(W - 1));
    const double u = y * y;
#pragma unroll
    for (int a = 0; a < (W + 1) / 2; ++a) {
        const double *c = cb + a * P;
        double e = c[NE - 1];
#pragma unroll
        for (int k = NE - 2; k >= 0; --k) e = fma(e, u, c[k]);
        if (2 * a + 1 == W) {  // middle tap of an odd width: even in y
            wt[a] = e;
        } else {
            double o = c[NE + NO - 1];
#pragma unroll
            for (int k = NO - 2; k >= 0; --k) o = fma(o, u, c[NE + k]);
            wt[a] = fma(y, o, e);
            wt[W - 1 - a] = fma(-y, o, e);
        }
    }
    return s;
}

__device__ __forceinline__ float ex2_approx(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rsqrt_approx(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float rcp_approx(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// atan(u) - u for |u| <= 1 as u^3 R(u^2): R is a degree-9 polynomial in u^2 fitted by
// fit_atan_f32.py (iteratively reweighted least squares towards the minimax error of atan; the
// fit's error is 1.7e-10, and evaluated in FP32 the correction carries at most 3e-8).  The
// leading term u stays exact, so atan(u) is carried as the two terms u + correction.
__device__ __forceinline__ float atan_correction_f32(float u)
{
    const float s = u * u;
    float r = 0.000990882766560405f;
    r = fmaf(r, s, -0.0066840073563619829f);
    r = fmaf(r, s, 0.021143804646584562f);
    r = fmaf(r, s, -0.042978293426904776f);
    r = fmaf(r, s, 0.066138929468158386f);
    r = fmaf(r, s, -0.087516064688656053f);
    r = fmaf(r, s, 0.1104117269740377f);
    r = fmaf(r, s, -0.14276990716236754f);
    r = fmaf(r, s, 0.19999428419267529f);
    r = fmaf(r, s, -0.33333319184448684f);
    return u * s * r;
}

// The factor mu^-2 of one mapped coordinate v in a point's strength (Section 2.1), FP32:
// (S^2 + v^2)/S (algebraic map) or S cosh(v/S) = S (e^-|v/S| + e^|v/S|)/2 (logarithmic map).
__device__ __forceinline__ float axis_m2_f32(const TypedConsts<float> &K, float v, bool alg)
{
    if (alg) return fmaf(v, v, K.SS) * K.invS;
    const float w = fmaf(v, K.invS, v * K.invS_lo);
    const float e = exp2f(-fabsf(w) * 1.4426950408889634f);
    return 0.5f * K.S * (__frcp_rn(e) + e);
}

// FP32 grid coordinate x = z n/(2 pi) of the angle z = arccos(xi(v)) of one mapped coordinate, as an
// integer cell X (an integer-valued float) and a fraction F in [0, 1) (Section 2.1).  With w = v/S:
//   r = 1: |w| <= 1: x = n/4 - gs atan(w);  w > 1: x = gs atan(S/v);  w < -1: x = n/2 + gs atan(S/v)
//          (z = pi/2 - atan(w) = atan(1/w) or pi + atan(1/w))
//   r = 0: x = 2 gs atan(e) (v >= 0) or n/2 - 2 gs atan(e) (v < 0), e = exp(-|v|/S)
// with gs = n/(2 pi), i.e. x = base - sg c atan(u) with |u| <= 1 and base in {0, n/4, n/2}.  The
// offsets are exact, c = gs (or 2 gs) is a two-term constant, atan(u) = u + correction is
// renormalised into two terms (Fast2Sum) and multiplied by c with its exact FMA residual, and
// base - sg c atan(u) is summed exactly (Fast2Sum), so the fraction F is accurate to about 1e-7
// of a cell: a grid coordinate rounded to FP32 as a whole (about 1e-6 of a cell at x ~ 100)
// shifts points that share a coordinate -- and many do, on a tensor grid of nodes -- coherently.
__device__ __forceinline__ void grid_coord_f32(const TypedConsts<float> &K, float v, bool alg, float &X, float &F)
{
    float base, sg, u, ch = K.gs, cl = K.gs_lo;
    if (alg) {
        const float w = fmaf(v, K.invS, v * K.invS_lo);  // v/S
        if (fabsf(w) <= 1.0f) {
            base = K.xq;
            sg = 1.0f;
            u = w;
        } else {  // u = S/v: the approximate reciprocal and one Newton step
            const float rv = rcp_approx(v);
            const float u0 = K.S * rv;
            u = fmaf(rv, fmaf(-v, u0, K.S), u0);
            base = v > 0.0f ? 0.0f : 2.0f * K.xq;
            sg = -1.0f;
        }
    } else {
        const float w = fmaf(v, K.invS, v * K.invS_lo);
        const float e = exp2f(-fabsf(w) * 1.4426950408889634f);  // exp(-|v|/S)
        u = e;
        base = v >= 0.0f ? 0.0f : 2.0f * K.xq;
        sg = v >= 0.0f ? -1.0f : 1.0f;
        ch = 2.0f * K.gs;
        cl = 2.0f * K.gs_lo;
    }
    const float corr = atan_correction_f32(u);
    const float ah = u + corr;                            // atan(u) = ah + al
    const float al = (u - ah) + corr;                     // exact (Fast2Sum: |u| >= |corr|)
    const float p1 = ch * ah;
    const float e1 = fmaf(ch, ah, -p1);                   // exact: p1 + e1 = ch ah
    const float pl = e1 + fmaf(ch, al, cl * ah);          // the rest of c atan(u): a few ulp of p1
    const float hi = base - sg * p1;
    const float err = (base - hi) - sg * p1;              // exact (|base| >= |p1| or base = 0)
    const float lo = err - sg * pl;
    X = floorf(hi);
    F = (hi - X) + lo;                                    // |lo| is far below one cell
    if (F < 0.0f) {
        F += 1.0f;
        X -= 1.0f;
        if (F >= 1.0f) {  // -F below half an ulp of 1: the point sits on the cell boundary
            F = 0.0f;
            X += 1.0f;
        }
    } else if (F >= 1.0f) {
        F -= 1.0f;
        X += 1.0f;
    }
}

// FP32 kernel value psi(t) 2^lsc = 2^(bl (sqrt(1 - t^2) - 1) + lsc) for |t| < 1 and 0 outside, with
// bl = beta log2(e) and bias = lsc - bl; the square root as (1 - t^2) rsqrt(1 - t^2).  Both
// approximations are good to a few 1e-7.
__device__ __forceinline__ float es_f32(float t, float bl, float bias)
{
    const float om = fmaf(-t, t, 1.0f);
    const float e = fmaf(bl, om * rsqrt_approx(om), bias);
    return om > 0.0f ? ex2_approx(e) : 0.0f;
}
// The same at tap a of W (known when the loop over taps is unrolled): only the first and the last tap
// can lie on the support's ends.
template <int W>
__device__ __forceinline__ float es_tap_f32(int a, float t0, float bl, float bias)
{
    const float t = fmaf((float)a, 2.0f / W, t0);
    if (a == 0 || a == W - 1) return es_f32(t, bl, bias);
    const float om = fmaf(-t, t, 1.0f);
    return ex2_approx(fmaf(bl, om * rsqrt_approx(om), bias));
}

// First tap s = X + c0 of a point at X + F for kernel width W (s = floor(x - W/2) + 1) and the tap
// offset t0 = (s - x) 2/W; tap a has t = t0 + a 2/W.
template <int W>
__device__ __forceinline__ int first_tap_f32(float X, float F, float &t0)
{
    int c0;
    if constexpr (W % 2 == 0) c0 = 1 - W / 2;
    else c0 = (F >= 0.5f ? 1 : 0) - (W - 1) / 2;
    t0 = ((float)c0 - F) * (2.0f / W);
    return (int)X + c0;
}

// FP32 weights psi(t_a) of one axis and the folded cells fold(s + a).
template <int W>
__device__ __forceinline__ void axis_weights_f32(const SpreadArgs &p, float X, float F, float *wt, int *idx)
{
    float t0;
    const int s = first_tap_f32<W>(X, F, t0);
    const float bl = p.cf.bl;
#pragma unroll
    for (int a = 0; a < W; ++a) {
        wt[a] = es_tap_f32<W>(a, t0, bl, -bl);
        idx[a] = fold_cell(s + a, p.n);
    }
}

// Row shear of the class numbering (PairCursor).
constexpr unsigned kPairShear = 1597u;

// Node pairs in classes.  A pair (i, j) adds M points around its centre (v_i + v_j)/2 at the radius
// |v_i - v_j|/2.  Exchanging the two nodes' components along any subset of axes changes neither --
// per axis the centre and the squared difference are symmetric -- so all 2^d ordered pairs of one
// class {i_0, j_0} x ... x {i_{d-1}, j_{d-1}} (an unordered pair of node indices per axis) add the
// same M points (for any sphere set), and each class is spread once with the sum of their strengths:
//   q = B(|v_i - v_j|) w_m prod mu^-2 . 2 prod_l (i_l == j_l ? 1/2 : 1) . sum_o a_{i(o)} a_{j(o)}
// over the 2^(d-1) ways o to exchange axes 0..d-2 (exchanging every axis swaps i and j: the factor
// 2; an axis with i_l == j_l would count its two equal ways twice: the factor 1/2).  That is N^4/4
// point sets in 2D and N^6/8 in 3D, where one per unordered pair {i, j} is N^4/2 and N^6/2: the
// spreading, which is all but a few percent of an evaluation, halves in 2D and quarters in 3D, and
// each strength is rounded once for the class instead of once per pair.
// Measured, one evaluation, one point set per unordered pair -> per class: 2D hard spheres N = 64,
// M = 32 FP32 2.39 -> 1.47 ms, FP64 223 -> 117 ms; 3D Maxwell N = 16, M = 32 FP32 21.6 -> 10.7 ms;
// 3D FP64 N = 11, M = 16 140 -> 46 ms.
template <typename T, int D>
struct PairData {
    T cen[D];            // (v_i + v_j)/2
    T rad;               // |v_i - v_j|/2
    T base;              // VHS: B sum_o a_{i(o)} a_{j(o)}; angular kernels: 1
    T sabs;              // B sum_o |a_{i(o)} a_{j(o)}|
    T mult;              // 2 prod_l (i_l == j_l ? 1/2 : 1)
    T x[1 << (D - 1)];   // angular kernels: B a_{i(o)} a_{j(o)}, bit l of o: axis l exchanged
    T dir[D];            // angular kernels: |v_i - v_j|^-1 (v_i - v_j), o = 0 (0 for i == j)
};

// Numbering: an axis has naxp = N (N + 1)/2 unordered pairs p = t N + u <-> {u, (u + t) mod N}
// (t = 0 the equal ones; for even N the row t = N/2 stops at u = N/2 - 1), and class pr is
// (row t, column u) with t = pr / naxp numbering the pairs of the leading axes and the last axis'
// pair i = (u + t K) mod naxp sheared by K = kPairShear per row.  The shear is a bijection of each
// row; it makes a lane that strides through the classes by a multiple of naxp visit every pair
// of the last axis, so the lanes of a warp meet the negligible classes of the tails of f at the
// same rate.

// A position in the numbering, advanced by a fixed stride without divisions: a stride of
// dt naxp + du moves i by di = (du + dt K) mod naxp, and by K mod naxp more when u wraps.
struct PairCursor {
    long long pr;
    int t, u, i;
};
struct PairStep {
    long long d;
    int dt, du, di, dk;
};

__device__ __forceinline__ PairCursor pair_cursor(int naxp, long long pr)
{
    PairCursor c;
    c.pr = pr;
    c.t = (int)(pr / naxp);
    c.u = (int)(pr - (long long)c.t * naxp);
    c.i = (int)(((long long)c.u + (long long)c.t * kPairShear) % naxp);
    return c;
}

__device__ __forceinline__ PairStep pair_step(int naxp, long long stride)
{
    PairStep s;
    s.d = stride;
    s.dt = (int)(stride / naxp);
    s.du = (int)(stride - (long long)s.dt * naxp);
    s.di = (int)(((long long)s.du + (long long)s.dt * kPairShear) % naxp);
    s.dk = (int)(kPairShear % naxp);
    return s;
}

__device__ __forceinline__ void pair_advance(int naxp, PairCursor &c, const PairStep &s)
{
    c.pr += s.d;
    c.t += s.dt;
    c.u += s.du;
    c.i += s.di;
    if (c.i >= naxp) c.i -= naxp;
    if (c.u >= naxp) {
        c.u -= naxp;
        c.t += 1;
        c.i += s.dk;
        if (c.i >= naxp) c.i -= naxp;
    }
}

// Row t = p / N of axis pair p = t N + u from a float quotient: (p + 1/2)/N lies at least 1/(2N)
// from an integer and its FP32 value within 2^-23 (p + 1/2)/N < 1/(4N) of it for p < 2^21 (every
// axis pair of a plan: N <= 512), so the truncation is the exact quotient.
__device__ __forceinline__ int axis_pair_row(int p, float invN) { return __float2int_rz(((float)p + 0.5f) * invN); }

// Load the class at cursor c; false when its strength is zero.  ANG: angular kernels.  FP32: strengths are
// formed times `pre` (product_scale).
template <typename T, int D, bool ANG = false>
__device__ __forceinline__ bool load_pair(const SpreadArgs &p, const PairCursor &c, T pre, PairData<T, D> &P)
{
    constexpr int NO = 1 << (D - 1);
    const int N = p.N;
    int ap[D];
    ap[D - 1] = c.i;
    if constexpr (D == 2) {
        ap[0] = c.t;
    } else {
        ap[0] = c.t / p.naxp;
        ap[1] = c.t - ap[0] * p.naxp;
    }
    const float invN = 1.0f / (float)N;
    int ni[D], nj[D];
    P.mult = T(2);
#pragma unroll
    for (int l = 0; l < D; ++l) {
        const int t = axis_pair_row(ap[l], invN);
        ni[l] = ap[l] - t * N;
        nj[l] = ni[l] + t;
        if (nj[l] >= N) nj[l] -= N;
        if (t == 0) P.mult *= T(0.5);
    }
    const T *vnode = static_cast<const T *>(p.vnode);
    const T *acoef = static_cast<const T *>(p.a);
    T x[NO], sum = T(0), sabs = T(0);
#pragma unroll
    for (int o = 0; o < NO; ++o) {
        int I = 0, J = 0;
#pragma unroll
        for (int l = 0; l < D; ++l) {
            const bool ex = (o >> l) & 1;
            I = I * N + (ex ? nj[l] : ni[l]);
            J = J * N + (ex ? ni[l] : nj[l]);
        }
        x[o] = (sizeof(T) == 4 ? acoef[I] * pre : acoef[I]) * acoef[J];
        sum += x[o];
        sabs += fabs(x[o]);
    }
    if (sabs == T(0)) return false;
    T g2 = T(0);
#pragma unroll
    for (int l = D - 1; l >= 0; --l) {
        const T vi = vnode[ni[l]], vj = vnode[nj[l]];
        T dl = vi - vj, sl = vi + vj;
        if constexpr (sizeof(T) == 4) {  // FP32 nodes carry their rounding in a second term
            const float li = p.vnode_lo[ni[l]], lj = p.vnode_lo[nj[l]];
            dl += li - lj;
            sl += li + lj;
        }
        g2 += dl * dl;
        P.cen[l] = T(0.5) * sl;
        if constexpr (ANG) P.dir[l] = dl;
    }
    const T g = Fn<T>::sqrt_(g2);
    if constexpr (ANG) {
        const T ginv = g > T(0) ? T(1) / g : T(0);
#pragma unroll
        for (int l = 0; l < D; ++l) P.dir[l] *= ginv;
    }
    const TypedConsts<T> &K = kconst<T>(p);
    T B;
    switch (p.fast_gamma) {
    case 0: B = K.Bconst; break;
    case 1: B = K.Bconst * g; break;
    case 2: B = K.Bconst * Fn<T>::sqrt_(g); break;
    default: B = K.Bconst * Fn<T>::pow_(g, K.gamma); break;
    }
    P.sabs = sabs * B;
    P.rad = T(0.5) * g;
    if constexpr (ANG) {
#pragma unroll
        for (int o = 0; o < NO; ++o) P.x[o] = x[o] * B;
        P.base = T(1);
        return P.sabs != T(0);
    } else {
        P.base = sum * B;
        return P.base != T(0);
    }
}

// sum_m |q_m| <= (strength) x this, for any share of the class' strength: W_sigma prod_l
// mu^-2(|c_l| + rad), since |v'_l| <= |c_l| + rad and mu^-2 grows with |v|.
template <typename T, int D>
__device__ __forceinline__ T pair_bound(const SpreadArgs &p, const PairData<T, D> &P)
{
    const TypedConsts<T> &K = kconst<T>(p);
    T U = K.Wang;
#pragma unroll
    for (int l = 0; l < D; ++l) {
        const T R = fabs(P.cen[l]) + P.rad;
        U *= (p.r == 1) ? (K.SS + R * R) * K.invS : K.S * Fn<T>::cosh_(R * K.invS);
    }
    return U;
}

// Global folded-grid cell of tile cell c (tile layout: see spread_point) in a tile whose first row is row_lo.
__device__ __forceinline__ int tile_to_grid_cell(int c, int D, int nf, int ncol, int cpad, int n, int row_lo)
{
    const int u = c % ncol - cpad;
    const int rest = c / ncol;  // row (2D) or row nf + j (3D), relative to row_lo
    return (row_lo * (D == 3 ? nf : 1) + rest) * nf + fold_index(u, n);
}

// Shared-memory accumulators of the block tile.
//
// FP32 path: one signed 32-bit fixed-point word per cell in shared memory, in units 2^-Et of the
// tile (Et = Eg - tile_bits(d)), plus a per-block carry array of the same layout in global memory.
// A contribution v in [-2^31, 2^31) goes to its word with one native 32-bit atomic; when that
// addition overflows the signed range (visible from the returned old value o and the result r:
// (o ^ r) & (v ^ r) < 0) the wrapped +-1 x 2^32 tile units go to the cell's carry counter; the
// direction is the addend's sign, which is that of the point's strength (every kernel weight is
// >= 0), so it is one value per point.  Atomic additions on a word are serialised, so every wrap
// is that of exactly one addition and word + 2^32 carry is the exact sum in any order.
// Contributions of larger points are scaled integers v 2^s: their low word goes to the word, the rest
// to the carry directly.  A block's partial sum in one cell stays below B 2^Et = 2^(61 - bits), so
// carries are rare (about B 2^Et / 2^32 in a whole evaluation) and a counter stays below
// 2^(29 - bits) in magnitude (bits = tile_bits(d)).

struct SplitTile {
    int *lo;     // tile words (shared memory)
    int *carry;  // this block's carry counters (global memory, same layout)
    // One addition of a run of consecutive cells: its wrap is shifted
    // into `mask` (one funnel shift) and the carries of the run are added afterwards, in
    // add_carries, where the mask is rarely non-zero.
    __device__ __forceinline__ unsigned add_int_run(int c, int v, unsigned mask) const
    {
        const int o = atomicAdd(lo + c, v);
        const int r = (int)((unsigned)o + (unsigned)v);
        return __funnelshift_l((unsigned)((o ^ r) & (v ^ r)), mask, 1);
    }
    // carries of a run of n additions to cells c0 .. c0+n-1 (bit n-1-k of mask: cell c0 + k)
    __device__ __forceinline__ void add_carries(int c0, int n, unsigned mask, int d) const
    {
        while (mask) {
            const int b = __ffs(mask) - 1;
            atomicAdd(carry + c0 + (n - 1 - b), d);
            mask &= mask - 1;
        }
    }
    // v 2^s for |v| < 2^31, 0 <= s < 32: its low word, signed, to the word, the rest to the carry counter
    __device__ __forceinline__ void add_scaled(int c, int v, int s) const
    {
        const int l = (int)((unsigned)v << s);
        const int h = (int)__funnelshift_l((unsigned)v, (unsigned)(v >> 31), s) - (l >> 31);
        const int o = atomicAdd(lo + c, l);
        const int r = (int)((unsigned)o + (unsigned)l);
        const int k = h + ((((o ^ r) & (l ^ r)) < 0) ? (l < 0 ? -1 : 1) : 0);
        if (k) atomicAdd(carry + c, k);
    }
    // the cell's sum in tile units
    __device__ __forceinline__ long long value(int c) const { return (long long)carry[c] * 4294967296LL + lo[c]; }
};
// FP64 path: one 96-bit two's-complement fixed-point value per cell in units 2^-(Eg+32), 32 bits
// finer than the global grid (B 2^Eg < 2^61), held as a fraction word, a low and a high 32-bit
// word in shared memory.  A contribution I + F 2^-32 (I an int64 in grid units, 0 <= F < 2^32)
// adds F to the fraction word and I plus the carry out of that addition to the low word, each with
// one native 32-bit atomic whose returned old value shows its carry; the high part of I plus the
// low word's carry goes to the high word by a third atomic when not zero (for positive
// contributions below 2^32 grid units, only on a carry).  The sum is exact in any order, and a
// partial sum stays below 2^63 grid units.  Shared-memory FP64 atomic adds, the other choice, run
// several times slower on this hardware (they spend the FP64 pipe).
struct WideTile {
    unsigned *fr;  // fraction words (shared memory)
    unsigned *lo;  // low words
    int *hi;       // high words
    // the cell's sum rounded to the grid unit
    __device__ __forceinline__ long long value(int c) const
    {
        const long long i = (long long)(((unsigned long long)(unsigned)hi[c] << 32) | lo[c]);
        return i + (fr[c] >= 0x80000000u ? 1 : 0);
    }
};

// Fixed-point kernel weight for the FP64 path: round(w 2^63) = h 2^32 + l (0 <= w <= 1 up to the
// polynomial's rounding; what rounds below 0 is 0).
struct FixW {
    unsigned h, l;
};
__device__ __forceinline__ FixW fix_weight(double w)
{
    const unsigned long long t = __double2ull_rn(w * 9223372036854775808.0);  // 2^63
    return FixW{(unsigned)(t >> 32), (unsigned)t};
}

// The fixed-point weights of one axis of a point at grid coordinate x, into local memory (rows are read
// one at a time, the last axis' weights loaded into registers once per point); returns the first
// tap.  One out-of-line copy serves every axis: inlined per axis the tap polynomials fill the
// registers that the rows need.
template <int W>
__device__ __noinline__ int axis_weights_f64(double x, FixW *out)
{
    double wt[W];
    const int s = kernel_weights_f64<W>(x, wt);
#pragma unroll
    for (int a = 0; a < W; ++a) out[a] = fix_weight(wt[a]);
    return s;
}

// round(R2 w / 2) for R2 < 2^63 and a fixed-point weight w: the high word of the 128-bit product
// R2 (w 2^63) plus 2^63, from four 32 x 32-bit products (the low half's low word is dropped after
// its carry: at most 2^-32 of a unit).
__device__ __forceinline__ unsigned long long fix_mul(unsigned long long R2, FixW w)
{
    const unsigned rh = (unsigned)(R2 >> 32), rl = (unsigned)R2;
    const unsigned long long t1 = (unsigned long long)rl * w.h + __umulhi(rl, w.l) + 0x80000000ull;
    const unsigned long long t2 = (unsigned long long)rh * w.l + (unsigned)t1;
    return (unsigned long long)rh * w.h + (t1 >> 32) + (t2 >> 32);
}

// The scale of a point of strength q (grid units 2^-Eg): its contributions are formed in units
// 2^-(Eg+s) with s = 60 - ilogb|q|, at most 32 (the fraction word's resolution) and at least 0, so that
// |q| 2^s < 2^61.  Points below 2^28 grid units thus have their row factors rounded to 2^-32 units, as their
// contributions are (at s = 94, 2^-61 of the point, the factors alone would be finer): an error that can at
// most double one that the sum of a cell, rounded to whole grid units per block, exceeds a millionfold.
struct WideScale {
    int s;
    unsigned long long q2;    // round(|q| 2^(s+1))
    unsigned long long neg;   // all ones for q < 0
};
__device__ __forceinline__ WideScale wide_scale(double q)
{
    const int e = ((__double2hiint(q) >> 20) & 0x7ff) - 1023;
    WideScale k;
    k.s = max(0, min(60 - e, 32));
    k.q2 = __double2ull_rn(fabs(q) * __hiloint2double((1023 + k.s + 1) << 20, 0));
    k.neg = q < 0.0 ? ~0ull : 0ull;
    return k;
}

// Add the W contributions of one row, round(R2 w_c / 2) in units 2^-(Eg+s) with the point's sign, to
// the cells at `base + idx[c]`.  A contribution splits into the cell's three words by three funnel
// shifts.  The fraction words of G taps are added before the first of their returned values is
// needed, then the low words, so that a warp waits for two atomics per group and not per tap.
template <int W>
__device__ __forceinline__ void wide_row(const WideTile &tile, int base, const int (&idx)[W], unsigned long long R2,
                                         const WideScale &k, const FixW (&fl)[W])
{
    constexpr int G = W <= 8 ? W : (W + 1) / 2;
#pragma unroll
    for (int g = 0; g < W; g += G) {
        unsigned F[G], of[G], jl[G], ol[G];
        int jh[G];
#pragma unroll
        for (int j = 0; j < G; ++j) {
            if (g + j >= W) break;
            const unsigned long long v = (fix_mul(R2, fl[g + j]) ^ k.neg) - k.neg;
            const unsigned vl = (unsigned)v, vh = (unsigned)(v >> 32);
            F[j] = __funnelshift_lc(0u, vl, 32 - k.s);  // v 2^(32-s), its low word
            jl[j] = __funnelshift_rc(vl, vh, k.s);      // v 2^-s
            jh[j] = (int)vh >> min(k.s, 31);
            of[j] = atomicAdd(tile.fr + base + idx[g + j], F[j]);
        }
#pragma unroll
        for (int j = 0; j < G; ++j) {
            if (g + j >= W) break;
            const unsigned long long J =
                (((unsigned long long)(unsigned)jh[j] << 32) | jl[j]) + (of[j] + F[j] < F[j] ? 1 : 0);
            jl[j] = (unsigned)J;
            jh[j] = (int)(J >> 32);
            ol[j] = atomicAdd(tile.lo + base + idx[g + j], jl[j]);
        }
#pragma unroll
        for (int j = 0; j < G; ++j) {
            if (g + j >= W) break;
            const int h = jh[j] + (ol[j] + jl[j] < jl[j] ? 1 : 0);
            if (h) atomicAdd(tile.hi + base + idx[g + j], h);
        }
    }
}

// One post-collision point: FP32 points carry each grid coordinate (one grid cell = 1,
// x = z n / (2 pi)) as an integer cell X (an integer-valued float) and a fraction F in [0, 1)
// (grid_coord_f32); FP64 points carry x itself.  q is the strength in tile units.
template <typename T, int D>
struct Point;
template <int D>
struct Point<float, D> {
    float X[D], F[D], q;
};
template <int D>
struct Point<double, D> {
    double x[D], q;
};

// Strength of point m of class P before the map factors: qbase w_m, for angular kernels times
// sum_o x_o b_e(cos theta_o) with the even part b_e of b (Horner in cos^2 theta) and the direction
// of the exchanged pair o (the components of its exchanged axes change sign).
template <typename T, int D, bool ANG>
__device__ __forceinline__ T point_base(const SpreadArgs &p, const PairData<T, D> &P, T qbase, int m)
{
    const T *sig = static_cast<const T *>(p.sig);
    const T *wsig = static_cast<const T *>(p.wsig);
    T q = qbase * wsig[m];
    if constexpr (ANG) {
        const TypedConsts<T> &K = kconst<T>(p);
        T s = T(0);
#pragma unroll
        for (int o = 0; o < (1 << (D - 1)); ++o) {
            T c = T(0);
#pragma unroll
            for (int l = 0; l < D; ++l) {
                const T t = P.dir[l] * sig[m * D + l];
                c += ((o >> l) & 1) ? -t : t;
            }
            const T c2 = c * c;
            T be = K.ang_even[p.nang_even - 1];
            for (int k = p.nang_even - 2; k >= 0; --k) be = be * c2 + K.ang_even[k];
            s += P.x[o] * be;
        }
        q *= s;
    }
    return q;
}

// FP32: the post-collision velocity v' = (v_i + v_j)/2 + |v_i - v_j| sigma_m / 2 of point m of
// pair P and its strength q (qbase = a_i a_j B x multiplicity x tile scale), without the grid
// coordinates.
template <int D, bool ANG>
__device__ __forceinline__ float point_velocity_f32(const SpreadArgs &p, const PairData<float, D> &P, float qbase,
                                                    int m, float (&vp)[D])
{
    const float *sig = static_cast<const float *>(p.sig);
    const TypedConsts<float> &K = kconst<float>(p);
    const bool alg = (p.r == 1);
    float q = point_base<float, D, ANG>(p, P, qbase, m);
#pragma unroll
    for (int l = 0; l < D; ++l) {
        vp[l] = fmaf(P.rad, sig[m * D + l], P.cen[l]);
        q *= axis_m2_f32(K, vp[l], alg);
    }
    return q;
}

// FP64 grid coordinate x = z n/(2 pi) of one mapped coordinate v, and its factor mu^-2.
__device__ __forceinline__ double grid_coord_f64(const TypedConsts<double> &K, double v, bool alg, double &m2)
{
    if (alg) {
        m2 = (K.SS + v * v) * K.invS;
        return atan2(K.S, v) * K.gs;
    }
    // z = 2 atan(e^-u) and mu^-2 = S cosh u with e = e^-|u| <= 1 (one exp and one atan
    // instead of sinh, cosh and atan2): for u < 0, 2 atan(e^|u|) = pi - 2 atan(e^-|u|)
    const double u = v * K.invS;
    const double e = exp(-fabs(u));
    const double at2 = 2.0 * atan(e);
    m2 = 0.5 * K.S * (e + 1.0 / e);
    return (u >= 0.0 ? at2 : 3.14159265358979323846 - at2) * K.gs;
}

// Point m of pair P (qbase = a_i a_j B x multiplicity x tile scale).
template <typename T, int D, bool ANG = false>
__device__ __forceinline__ void make_point(const SpreadArgs &p, const PairData<T, D> &P, T qbase, int m,
                                           Point<T, D> &pt)
{
    const TypedConsts<T> &K = kconst<T>(p);
    const bool alg = (p.r == 1);
    if constexpr (sizeof(T) == 4) {
        float vp[D];
        pt.q = point_velocity_f32<D, ANG>(p, P, qbase, m, vp);
#pragma unroll
        for (int l = 0; l < D; ++l) grid_coord_f32(K, vp[l], alg, pt.X[l], pt.F[l]);
    } else {
        const double *sig = static_cast<const double *>(p.sig);
        double q = point_base<double, D, ANG>(p, P, qbase, m);
#pragma unroll
        for (int l = 0; l < D; ++l) {
            double m2;
            pt.x[l] = grid_coord_f64(K, P.cen[l] + P.rad * sig[m * D + l], alg, m2);
            q *= m2;
        }
        pt.q = q;
    }
}

// Tile layout.  A block tile holds rows row_lo..row_lo+nrows-1 of axis 0 of the folded grid, and
// along the last axis (but for FP64 3D tiles, whose three words per cell leave no room for it: cpad = 0,
// ncol = nf, and a point's columns are folded once for its w^2 rows) it keeps the
// UNFOLDED columns that points reach, u at u + cpad (ncol cells, tile_cols): the w columns of a point are then consecutive, with no folding and no
// per-contribution index arithmetic.  The padding columns are folded onto their cells when the
// tile is added to the global grid (tile_to_grid_cell).  2D cell (row, u): row ncol + u + cpad;
// 3D cell (row, j, u): (row nf + j) ncol + u + cpad.

// ---- FP32 points
//
// Kinds of FP32 point: kInt -- |q| < 2^29 tile units; kLarge -- any q; kSmall -- |q| < trim_q
// (SpreadArgs): every contribution of a first or last tap of an axis rounds to zero, so only the inner
// (w-2)^d taps are added (the same bits).
constexpr int kInt = 0, kLarge = 1, kSmall = 2;
// Points below this many tile units take the integer products as they are; points below
// kNegligibleF32 add exactly zero (4 q psi rounds to 0 for every row) and are skipped, and so are
// pairs whose points all stay below it.
constexpr float kIntLimitF32 = 536870912.0f;  // 2^29
constexpr float kNegligibleF32 = 0.1f;

// round(a b / 2^32) for |a| < 2^31, 0 <= b <= 2^30: the high word of one 64-bit multiply-add
__device__ __forceinline__ int mulhi_rn(int a, int b)
{
    return (int)(((long long)a * (long long)b + 0x80000000LL) >> 32);
}

// Large points: the factor q4 of a point of strength q scaled by 2^-sc, which leaves |q| 2^-sc in [2^28, 2^29).
__device__ __forceinline__ float scale_large(float q4, float q, int &sc)
{
    sc = min(max(((__float_as_int(q) >> 23) & 255) - 127 - 28, 0), 31);
    return q4 * __int_as_float((127 - sc) << 23);
}

// Add the w^d contributions q psi_a psi_b psi_c of one FP32 point to the block tile: the column
// factors 2^30 psi_c and, per row, 4 q psi_a (psi_b) are rounded to integers, and a contribution is
// mulhi_rn of the two (at most about one tile unit of rounding).  kLarge: the same with q 2^-s in
// [2^28, 2^29) for the point's own s, i.e. rounded to 2^s tile units, 2^-28 of the point's strength
// (an FP32 product is rounded to 2^-24 of the contribution, which is more over a point's taps; and
// the float path that formed it took twice the instructions: 768 batched cells, where points of 2^29
// units are common, 43.9 -> 33.2 ms).  The tile holds every row of the grid.  3D points loop over their axis-0 rows (computing that
// row's kernel value in the loop) so that the unrolled code stays small.
template <int D, int W, int KIND>
__device__ __forceinline__ void spread_point_f32(const SpreadArgs &p, const Point<float, D> &pt,
                                                 const SplitTile &tile, int plane)
{
    const float q = pt.q;
    if (fabsf(q) < kNegligibleF32) return;  // every contribution rounds to zero
    const float bl = p.cf.bl;
    const float h2 = 2.0f / W;
    float t00, tl0;
    const int s0 = first_tap_f32<W>(pt.X[0], pt.F[0], t00);          // first row
    const int sl = first_tap_f32<W>(pt.X[D - 1], pt.F[D - 1], tl0);  // first column (unfolded)
    const int cb = min(max(sl + p.cpad, 0), p.ncol - W);            // clamped: x lies in [0, n/2]
    float w1[W];
    int c1[W];
    if constexpr (D == 3) {
        axis_weights_f32<W>(p, pt.X[1], pt.F[1], w1, c1);
#pragma unroll
        for (int b = 0; b < W; ++b) c1[b] = c1[b] * p.ncol + cb;
    }
    const int sg = q < 0.0f ? -1 : 1;  // the sign of every contribution (or zero)
    float q4 = 4.0f * q;
    int sc = 0;
    if constexpr (KIND == kLarge) q4 = scale_large(q4, q, sc);
    const float bias30 = 30.0f - bl;
    int wi[W];
#pragma unroll
    for (int c = 0; c < W; ++c) wi[c] = __float2int_rn(es_tap_f32<W>(c, tl0, bl, bias30));
    auto run = [&](int line, int rq) {
        if constexpr (KIND == kLarge) {
#pragma unroll
            for (int c = 0; c < W; ++c) tile.add_scaled(line + c, mulhi_rn(rq, wi[c]), sc);
        } else {
            unsigned wraps = 0u;
#pragma unroll
            for (int c = 0; c < W; ++c) wraps = tile.add_int_run(line + c, mulhi_rn(rq, wi[c]), wraps);
            if (wraps) tile.add_carries(line, W, wraps, sg);
        }
    };
    if constexpr (D == 2) {
#pragma unroll
        for (int a = 0; a < W; ++a) {
            const int r = fold_cell(s0 + a, p.n);
            run(r * plane + cb, __float2int_rn(q4 * es_f32(fmaf((float)a, h2, t00), bl, -bl)));
        }
    } else {
#pragma unroll 1
        for (int a = 0; a < W; ++a) {
            const int r = fold_cell(s0 + a, p.n);
            const float qa = q4 * es_f32(fmaf((float)a, h2, t00), bl, -bl);
            const int row = r * plane;
#pragma unroll
            for (int b = 0; b < W; ++b) run(row + c1[b], __float2int_rn(qa * w1[b]));
        }
    }
}

// Whether any of the w axis-0 rows of a point whose first tap is s lies in the slab.
template <int W>
__device__ __forceinline__ bool rows_hit_from(const SpreadArgs &p, int s, int row_lo, int nrows)
{
    bool hit = false;
#pragma unroll
    for (int a = 0; a < W; ++a) hit |= (unsigned)(fold_cell(s + a, p.n) - row_lo) < (unsigned)nrows;
    return hit;
}

// ---- FP64 points

// Add the w^d contributions of one FP64 point (q in grid units 2^-Eg) to the block tile.  SLAB:
// the tile holds a slab of the grid's rows and rows outside it are skipped; otherwise it holds
// every row (row_lo = 0, nrows = n/2 + 1).  The point works in units 2^-(Eg+s) (wide_scale) with FP64 kernel
// weights held in 63-bit fixed point: each row takes the integer R = round(q psi_a 2^s) (3D: then
// round(R psi_b)) and each cell round(R psi_c) -- integer products (fix_mul), about 2^-61 relative
// rounding -- which goes to the tile as grid units and 32 fraction bits (wide_row).
template <int D, int W, bool SLAB>
__device__ __forceinline__ void spread_point_f64(const SpreadArgs &p, const Point<double, D> &pt,
                                                 const WideTile &tile, int row_lo, int nrows, int plane)
{
    if (pt.q == 0.0) return;
    if constexpr (SLAB) {
        if (!rows_hit_from<W>(p, (int)floor(pt.x[0] - 0.5 * W) + 1, row_lo, nrows)) return;
    }
    const WideScale k = wide_scale(pt.q);
    FixW f0[W], fl[W];
    int cl[W];
    const int s0 = axis_weights_f64<W>(pt.x[0], f0);
    const int sl = axis_weights_f64<W>(pt.x[D - 1], fl);
    if constexpr (D == 2) {
        // consecutive padded columns (clamped: x lies in [0, n/2])
        const int cb = min(max(sl + p.cpad, 0), p.ncol - W);
#pragma unroll
        for (int c = 0; c < W; ++c) cl[c] = c;
#pragma unroll 1
        for (int a = 0; a < W; ++a) {
            const int r = fold_cell(s0 + a, p.n) - row_lo;
            if (SLAB && (unsigned)r >= (unsigned)nrows) continue;
            const unsigned long long R2 = fix_mul(k.q2, f0[a]) << 1;
            if (R2) wide_row<W>(tile, r * plane + cb, cl, R2, k, fl);
        }
    } else {
#pragma unroll
        for (int c = 0; c < W; ++c) cl[c] = fold_cell(sl + c, p.n);
        FixW f1[W];
        const int s1 = axis_weights_f64<W>(pt.x[1], f1);
#pragma unroll 1
        for (int a = 0; a < W; ++a) {
            const int r = fold_cell(s0 + a, p.n) - row_lo;
            if (SLAB && (unsigned)r >= (unsigned)nrows) continue;
            const unsigned long long Ra2 = fix_mul(k.q2, f0[a]) << 1;
            if (!Ra2) continue;
            const int row = r * plane;
#pragma unroll 1
            for (int b = 0; b < W; ++b) {
                const unsigned long long R2 = fix_mul(Ra2, f1[b]) << 1;
                if (R2) wide_row<W>(tile, row + fold_cell(s1 + b, p.n) * p.ncol, cl, R2, k, fl);
            }
        }
    }
}

// One point into a tile (every lane of the warp calls it, lanes without a pair with q = 0).  FP32:
// integer products for points below 2^29 tile units, chosen per lane (a point's contributions must
// not depend on its warp-mates: bitwise reproducibility across launch shapes; points of 2^29 tile
// units or more are rare); a lane whose point is below kNegligibleF32 idles.
template <typename T, int D, int W, typename Tile>
__device__ __forceinline__ void spread_point_body(const SpreadArgs &p, const Point<T, D> &pt, const Tile &tile,
                                                  int nrows, int plane)
{
    if constexpr (sizeof(T) == 4) {
        if (fabsf(pt.q) < kIntLimitF32) spread_point_f32<D, W, kInt>(p, pt, tile, plane);
        else spread_point_f32<D, W, kLarge>(p, pt, tile, plane);
    } else {
        spread_point_f64<D, W, false>(p, pt, tile, 0, nrows, plane);
    }
}

// Load the class at cursor c; whether it is not negligible: non-zero strength, not below the
// screening threshold tau (0: no screening; the sum of its pairs' bounds is compared, so every pair
// skipped is below tau), and a bound Ut >= floor_q on every point's |q| in tile units.  On success
// P.base is multiplied by the class' multiplicity.  sc: tile units per strength as load_pair forms it (so
// tau, too, is in those units).
template <typename T, int D, bool ANG>
__device__ __forceinline__ bool class_passes(const SpreadArgs &p, const PairCursor &c, T sc, T pre, T tau,
                                             T floor_q, PairData<T, D> &P)
{
    if (!load_pair<T, D, ANG>(p, c, pre, P)) return false;
    const T U = pair_bound<T, D>(p, P);
    if (tau > T(0) && P.sabs * U < tau) return false;
    if ((ANG ? P.sabs : fabs(P.base)) * U * P.mult * sc * kconst<T>(p).wmax < floor_q) return false;
    P.base *= P.mult;
    return true;
}

// Advance the cursor c (in steps of st, below `end`) to this lane's next class that is not
// negligible (class_passes); false when none is left.
template <typename T, int D, bool ANG>
__device__ __forceinline__ bool next_pair(const SpreadArgs &p, PairCursor &c, long long end, const PairStep &st, T sc,
                                          T pre, T tau, T floor_q, PairData<T, D> &P)
{
    for (; c.pr < end; pair_advance(p.naxp, c, st))
        if (class_passes<T, D, ANG>(p, c, sc, pre, tau, floor_q, P)) return true;
    return false;
}

// A pair of zero strength at the origin: its points add nothing (lanes whose pairs have run out).
template <typename T, int D>
__device__ __forceinline__ void zero_pair(PairData<T, D> &P)
{
#pragma unroll
    for (int l = 0; l < D; ++l) {
        P.cen[l] = T(0);
        P.dir[l] = T(0);
    }
#pragma unroll
    for (int o = 0; o < (1 << (D - 1)); ++o) P.x[o] = T(0);
    P.rad = T(0);
    P.base = T(0);
    P.sabs = T(0);
    P.mult = T(0);
}

// The pairs pr = first, first + stride, ... below end of one lane, spread into a tile that holds
// every row.  Every lane of the warp runs every point step (the loop conditions are uniform).
template <typename T, int D, int W, typename Tile, bool ANG>
__device__ __forceinline__ void spread_pairs(const SpreadArgs &p, long long first, long long end, long long stride,
                                             T sc, T pre, T tau, T floor_q, const Tile &tile, int nrows, int plane)
{
    PairCursor c = pair_cursor(p.naxp, first);
    const PairStep st = pair_step(p.naxp, stride);
    for (;;) {
        PairData<T, D> P;
        const bool ok = next_pair<T, D, ANG>(p, c, end, st, sc, pre, tau, floor_q, P);
        if (!__any_sync(0xffffffffu, ok)) break;
        if (!ok) zero_pair<T, D>(P);
        const T qbase = P.base * sc;
        for (int m = 0; m < p.M; ++m) {
            Point<T, D> pt;
            make_point<T, D, ANG>(p, P, qbase, m, pt);
            spread_point_body<T, D, W, Tile>(p, pt, tile, nrows, plane);
        }
        if (ok) pair_advance(p.naxp, c, st);
    }
}

// ---- slabbed FP64 grids: warp point queues
//
// When the folded grid is split into slabs along axis 0, a point adds to a block's slab only
// if one of its w axis-0 rows lies there, and with a few slabs most points of a warp miss it:
// spreading them where they are generated would leave most lanes idle while the others add.
// Instead each warp appends the points that hit its slab to a queue of 32 entries in shared
// memory (value k of slot j at buf[32 k + j]) and spreads a full queue with all 32 lanes, one point
// per lane.

// Spread queue slot `lane` (when valid) with the whole warp.
template <int D, int W>
__device__ __forceinline__ void queue_spread(const SpreadArgs &p, const double *buf, int lane, bool valid,
                                             const WideTile &tile, int row_lo, int nrows, int plane)
{
    if (!valid) return;
    Point<double, D> pt;
#pragma unroll
    for (int l = 0; l < D; ++l) pt.x[l] = buf[l * 32 + lane];
    pt.q = buf[D * 32 + lane];
    spread_point_f64<D, W, true>(p, pt, tile, row_lo, nrows, plane);
}

// The classes pr = first, first + nthr, ... below end of one thread, spread through the warp's
// queue `buf` (spread_queue_values x 32 values) into one slab.  Points below floor_q are not queued.
// Every loop condition is uniform over the warp.
template <int D, int W, bool ANG>
__device__ __forceinline__ void spread_pairs_queued(const SpreadArgs &p, long long first, long long end,
                                                    long long nthr, double sc, double tau, double floor_q,
                                                    const WideTile &tile, int row_lo, int nrows, int plane, double *buf)
{
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    int count = 0;  // queued points, the same in every lane
    PairCursor c = pair_cursor(p.naxp, first);
    const PairStep st = pair_step(p.naxp, nthr);
    for (;;) {
        PairData<double, D> P;
        const bool ok = next_pair<double, D, ANG>(p, c, end, st, sc, 1.0, tau, floor_q, P);
        if (!__any_sync(full, ok)) break;
        const double qbase = ok ? P.base * sc : 0.0;
        for (int m = 0; m < p.M; ++m) {
            Point<double, D> pt;
            bool hit = false;
            if (ok) {
                make_point<double, D, ANG>(p, P, qbase, m, pt);
                hit = fabs(pt.q) >= floor_q &&
                      rows_hit_from<W>(p, (int)floor(pt.x[0] - 0.5 * W) + 1, row_lo, nrows);
            }
            const unsigned mask = __ballot_sync(full, hit);
            const int n = __popc(mask), rank = __popc(mask & lt), room = 32 - count;
            auto put = [&](int slot) {
#pragma unroll
                for (int l = 0; l < D; ++l) buf[l * 32 + slot] = pt.x[l];
                buf[D * 32 + slot] = pt.q;
            };
            if (hit && rank < room) put(count + rank);
            if (n >= room) {  // full: spread 32 points, then queue the rest
                __syncwarp();
                queue_spread<D, W>(p, buf, lane, true, tile, row_lo, nrows, plane);
                __syncwarp();
                if (hit && rank >= room) put(rank - room);
                count = n - room;
            } else {
                count += n;
            }
        }
        if (ok) pair_advance(p.naxp, c, st);
    }
    __syncwarp();
    queue_spread<D, W>(p, buf, lane, lane < count, tile, row_lo, nrows, plane);
}

// ---- 2D FP32 grids in one tile: quads
//
// The M points of a class lie on a circle, sigma_m = (cos theta_m, sin theta_m) with theta_m =
// 2 pi m/M, and M is even, so the set is symmetric in both axes: the points of m = 0..M/4 and their
// mirror images (c_0 +- r cos theta_m, c_1 +- r sin theta_m) are all M points, four to a quad (two where
// the sine (m = 0) or the cosine (4m = M) is zero).  The four points take two coordinates per axis,
// so a quad evaluates four axes (coordinate, map factor, w kernel values) where four points alone
// would evaluate eight.  Nearly every quad of a class that is not negligible adds something (91% to
// 100% on the workloads' densities), so a lane spreads its own class' quads where it forms them, m in
// step with the warp's other lanes (their classes are unrelated); only quads with a point of 2^29
// tile units or more go through a queue, so that the slower large-point code runs with full
// warps (where such points are common -- 15% of them at N = 16 -- almost every warp had one and all
// its lanes waited).
// Measured against spreading point by point through a queue: the headline (N = 64, M = 32) 1.47 -> 1.21 ms,
// 2D angular N = 41 785 -> 706 us, 768 batched cells 40.3 -> 31.6 ms, RK4 at N = 32 11.9 -> 8.4 ms (with
// the scaled integers of the large points, below).  Bound by issue (70% active) and by bank
// conflicts of the tile's atomics (3.4 wavefronts each, the shared pipe 73% busy) about equally.

constexpr int kQuadValues = 6;  // a large quad: two coordinates per axis, two strengths

// Quad m of a class: the coordinates c +- r cos theta_m of axis 0 and c +- r sin theta_m of axis 1, their map
// factors mu^-2, and the strengths before them of the points (+,+), (-,-) and (+,-), (-,+).
struct Quad {
    float vr[2], vc[2], mr[2], mc[2], q1, q2;
};
template <bool ANG>
__device__ __forceinline__ Quad make_quad(const SpreadArgs &p, const PairData<float, 2> &P, float qbase, int m)
{
    const float *sig = static_cast<const float *>(p.sig);
    const TypedConsts<float> &K = p.cf;
    const bool alg = (p.r == 1);
    const float cs = sig[2 * m], sn = sig[2 * m + 1];
    Quad Q;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        Q.vr[k] = fmaf(P.rad, k ? -cs : cs, P.cen[0]);
        Q.vc[k] = fmaf(P.rad, k ? -sn : sn, P.cen[1]);
        Q.mr[k] = axis_m2_f32(K, Q.vr[k], alg);
        Q.mc[k] = axis_m2_f32(K, Q.vc[k], alg);
    }
    Q.q1 = Q.q2 = qbase * static_cast<const float *>(p.wsig)[m];
    if constexpr (ANG) {
        const float a0 = P.dir[0] * cs, a1 = P.dir[1] * sn;
        const float e0 = (a0 + a1) * (a0 + a1), e1 = (a0 - a1) * (a0 - a1);
        float b0 = K.ang_even[p.nang_even - 1], b1 = b0;
        for (int k = p.nang_even - 2; k >= 0; --k) {
            b0 = b0 * e0 + K.ang_even[k];
            b1 = b1 * e1 + K.ang_even[k];
        }
        Q.q2 = Q.q1 * (P.x[0] * b1 + P.x[1] * b0);
        Q.q1 = Q.q1 * (P.x[0] * b0 + P.x[1] * b1);
    }
    return Q;
}

// Column factors of one coordinate of axis 1: first padded column and round(2^30 psi_c).
template <int W>
struct QuadCols {
    int cb, wi[W];
};
template <int W>
__device__ __forceinline__ void quad_cols(const SpreadArgs &p, float v, QuadCols<W> &c)
{
    float X, F, t0;
    grid_coord_f32(p.cf, v, p.r == 1, X, F);
    const int s = first_tap_f32<W>(X, F, t0);
    c.cb = min(max(s + p.cpad, 0), p.ncol - W);  // clamped: x lies in [0, n/2]
    const float bias30 = 30.0f - p.cf.bl;
#pragma unroll
    for (int k = 0; k < W; ++k) c.wi[k] = __float2int_rn(es_tap_f32<W>(k, t0, p.cf.bl, bias30));
}

// The large quad in slot `lane` of the queue: its points one by one.
template <int W>
__device__ __noinline__ void spread_large_quad(const SpreadArgs &p, const float *buf, const SplitTile &tile, int plane)
{
    const int lane = threadIdx.x & 31;
    const bool alg = (p.r == 1);
#pragma unroll 1
    for (int k = 0; k < 4; ++k) {
        const float v0 = buf[(k & 1) * 32 + lane], v1 = buf[(2 + (k >> 1)) * 32 + lane];
        if (isinf(v0) || isinf(v1)) continue;  // a coordinate that has no mirror image
        Point<float, 2> pt;
        // points (+,+), (-,-) have the first strength, (+,-), (-,+) the second
        pt.q = buf[(4 + ((k == 1 || k == 2) ? 1 : 0)) * 32 + lane] * axis_m2_f32(p.cf, v0, alg) *
               axis_m2_f32(p.cf, v1, alg);
        grid_coord_f32(p.cf, v0, alg, pt.X[0], pt.F[0]);
        grid_coord_f32(p.cf, v1, alg, pt.X[1], pt.F[1]);
        spread_point_f32<2, W, kLarge>(p, pt, tile, plane);
    }
}

// One point of a quad, any strength, in little code: the rows in a loop and the taps as scaled integers
// (spread_point_f32's kLarge, the same bits for points below 2^29 tile units as kInt).  Small plans run
// every instruction a few times per warp, and what they wait for is mostly instruction fetch (2D Maxwell
// N = 16: 5.3 of 12 warps); one such loop serves all their points in place of the unrolled code for the four
// points of a quad and that of the large ones (spreading 33 -> 27 us).
template <int W>
__device__ __forceinline__ void spread_point_compact(const SpreadArgs &p, float v0, float v1, float q,
                                                     const SplitTile &tile, int plane)
{
    const TypedConsts<float> &K = p.cf;
    const bool alg = (p.r == 1);
    int first[2];
    float off[2];  // local memory
#pragma unroll 1
    for (int l = 0; l < 2; ++l) {
        float X, F, t0;
        grid_coord_f32(K, l ? v1 : v0, alg, X, F);
        first[l] = first_tap_f32<W>(X, F, t0);
        off[l] = t0;
    }
    const int cb = min(max(first[1] + p.cpad, 0), p.ncol - W);  // clamped: x lies in [0, n/2]
    int wi[W];
#pragma unroll
    for (int c = 0; c < W; ++c) wi[c] = __float2int_rn(es_tap_f32<W>(c, off[1], K.bl, 30.0f - K.bl));
    int sc;
    const float q4 = scale_large(4.0f * q, q, sc);
#pragma unroll 1
    for (int a = 0; a < W; ++a) {
        const int rq = __float2int_rn(q4 * es_f32(fmaf((float)a, 2.0f / W, off[0]), K.bl, -K.bl));
        const int line = fold_cell(first[0] + a, p.n) * plane + cb;
#pragma unroll
        for (int c = 0; c < W; ++c) tile.add_scaled(line + c, mulhi_rn(rq, wi[c]), sc);
    }
}

// SPLIT (small plans): classes are spread in p.nsplit shares of their quads; share g takes
// [share_start(g), share_start(g + 1)) of n.
__device__ __forceinline__ int share_start(const SpreadArgs &p, int g, int n)
{
    return (int)((long long)g * n / p.nsplit);
}

// Share g of the quads of one class per lane (every lane of the warp calls it; P.base = 0: none).  buf,
// count: the warp's queue of large quads, 32 slots of kQuadValues floats, and its fill.
template <int W, bool ANG, bool SPLIT>
__device__ __forceinline__ void spread_class_quads(const SpreadArgs &p, const PairData<float, 2> &P, float qbase, int g,
                                                   const SplitTile &tile, int plane, float *buf, int &count)
{
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const TypedConsts<float> &K = p.cf;
    const bool alg = (p.r == 1);
    int m0 = 0, m1 = p.M / 4 + 1, steps = m1;
    if constexpr (SPLIT) {
        steps = (m1 + p.nsplit - 1) / p.nsplit;  // the largest share, so that the lanes stay together
        m0 = share_start(p, g, m1);
        m1 = share_start(p, g + 1, m1);
    }
#pragma unroll 1
    for (int k = 0; k < steps; ++k) {
        const int m = SPLIT ? min(m0 + k, p.M / 4) : k;
        const bool one_row = (4 * m == p.M), one_col = (m == 0);  // no mirror image
        const Quad Q = make_quad<ANG>(p, P, (!SPLIT || m0 + k < m1) ? qbase : 0.0f, m);
        if constexpr (SPLIT) {
#pragma unroll 1
            for (int i = 0; i < 4; ++i) {
                const int t = i >> 1, r = i & 1;
                if ((t && one_col) || (r && one_row)) continue;
                const float q = (r == t ? Q.q1 : Q.q2) * (r ? Q.mr[1] : Q.mr[0]) * (t ? Q.mc[1] : Q.mc[0]);
                if (fabsf(q) >= kNegligibleF32)
                    spread_point_compact<W>(p, r ? Q.vr[1] : Q.vr[0], t ? Q.vc[1] : Q.vc[0], q, tile, plane);
            }
            continue;
        }
        const float qmax = fmaxf(fabsf(Q.q1), fabsf(Q.q2)) * fmaxf(Q.mr[0], Q.mr[1]) * fmaxf(Q.mc[0], Q.mc[1]);
        const bool large = qmax >= kIntLimitF32;
        const unsigned lmask = __ballot_sync(full, large);
        if (lmask) {
            const int n = __popc(lmask), rank = __popc(lmask & ((1u << lane) - 1u)), room = 32 - count;
            const float inf = __int_as_float(0x7f800000);
            auto put = [&](int slot) {
                buf[slot] = Q.vr[0];
                buf[32 + slot] = one_row ? inf : Q.vr[1];
                buf[64 + slot] = Q.vc[0];
                buf[96 + slot] = one_col ? inf : Q.vc[1];
                buf[128 + slot] = Q.q1;
                buf[160 + slot] = Q.q2;
            };
            if (large && rank < room) put(count + rank);
            if (n >= room) {
                __syncwarp();
                spread_large_quad<W>(p, buf, tile, plane);
                __syncwarp();
                if (large && rank >= room) put(rank - room);
                count = n - room;
            } else {
                count += n;
            }
        }
        if (large || !(qmax >= kNegligibleF32)) continue;
        QuadCols<W> col[2];
        quad_cols<W>(p, Q.vc[0], col[0]);
        if (!one_col) quad_cols<W>(p, Q.vc[1], col[1]);
#pragma unroll 1
        for (int s = 0; s < 2; ++s) {
            if (s && one_row) break;
            const float v = s ? Q.vr[1] : Q.vr[0];
            float X, F, t0;
            grid_coord_f32(K, v, alg, X, F);
            const int s0 = first_tap_f32<W>(X, F, t0);
            const float m4 = 4.0f * (s ? Q.mr[1] : Q.mr[0]);
            float pa[W];
            int ra[W];
#pragma unroll
            for (int k = 0; k < W; ++k) {
                pa[k] = es_tap_f32<W>(k, t0, K.bl, -K.bl);
                ra[k] = fold_cell(s0 + k, p.n) * plane;
            }
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                if (t && one_col) break;
                const float q4 = m4 * ((s != t) ? Q.q2 : Q.q1) * Q.mc[t];  // 4 q of the point
                const int sg = q4 < 0.0f ? -1 : 1;  // the sign of every contribution (or zero)
#pragma unroll
                for (int k = 0; k < W; ++k) {
                    const int rq = __float2int_rn(q4 * pa[k]);
                    const int row = ra[k] + col[t].cb;
                    unsigned wraps = 0u;
#pragma unroll
                    for (int j = 0; j < W; ++j) wraps = tile.add_int_run(row + j, mulhi_rn(rq, col[t].wi[j]), wraps);
                    if (wraps) tile.add_carries(row, W, wraps, sg);
                }
            }
        }
    }
}

// The velocities v' on axis 0 whose points may reach the rows row_lo .. row_lo+nrows-1: a point at x
// touches rows of [x - w/2, x + w/2] (and their mirror images beyond the grid's ends, which lie in the
// first and last slabs), and x falls with v'.  A thousandth of a cell is added at both ends for the
// rounding of x; a point that then misses the slab finds no row in it.  Two comparisons per point
// and slab, where forming x and folding w rows took 85 instructions (3D VHS N = 24, three slabs: 55.7 -> 52.4 ms).
struct SlabRange {
    float lo, hi;
};
template <int W>
__device__ __forceinline__ SlabRange slab_range(const SpreadArgs &p, int row_lo, int nrows)
{
    const double x0 = row_lo - 0.5 * W - 1e-3, x1 = row_lo + nrows - 1 + 0.5 * W + 1e-3;
    auto velocity = [&](double x) {
        const double z = x / p.grid_scale;
        return (float)(p.r == 1 ? p.S * cos(z) / sin(z) : -p.S * log(tan(0.5 * z)));
    };
    const float inf = __int_as_float(0x7f800000);
    return SlabRange{x1 >= 0.5 * p.n ? -inf : velocity(x1), x0 <= 0.0 ? inf : velocity(x0)};
}

// In a slabbed grid half of a quad's rows or more lie outside a block's slab, so there the quads are
// queued by halves (N = 120, M = 8: spreading 5.44 -> 4.58 ms against a queue of single points, 4.16 ms
// with the slab's velocity range): one coordinate of axis 0 whose rows may reach the slab, and the two of
// axis 1 with the strengths of their points (0: no such point), kQuadValues values.

// Add one point of a half quad: rows ra (-1: outside the slab) with factors pa, column factors col.
template <int W, int KIND>
__device__ __forceinline__ void half_quad_point(const SplitTile &tile, const int (&ra)[W], const float (&pa)[W],
                                                const QuadCols<W> &col, float q)
{
    const int sg = q < 0.0f ? -1 : 1;
    float q4 = 4.0f * q;
    int sc = 0;
    if constexpr (KIND == kLarge) q4 = scale_large(q4, q, sc);
#pragma unroll
    for (int k = 0; k < W; ++k) {
        if (ra[k] < 0) continue;
        const int rq = __float2int_rn(q4 * pa[k]);
        const int row = ra[k] + col.cb;
        if constexpr (KIND == kLarge) {
#pragma unroll 1
            for (int j = 0; j < W; ++j) tile.add_scaled(row + j, mulhi_rn(rq, col.wi[j]), sc);
        } else {
            unsigned wraps = 0u;
#pragma unroll
            for (int j = 0; j < W; ++j) wraps = tile.add_int_run(row + j, mulhi_rn(rq, col.wi[j]), wraps);
            if (wraps) tile.add_carries(row, W, wraps, sg);
        }
    }
}

// The half quad in slot `lane` of the queue (valid lanes).
template <int W>
__device__ __forceinline__ void spread_half_quad(const SpreadArgs &p, const float *buf, bool valid,
                                                 const SplitTile &tile, int row_lo, int nrows, int plane)
{
    if (!valid) return;
    const int lane = threadIdx.x & 31;
    const TypedConsts<float> &K = p.cf;
    float X, F, t0;
    grid_coord_f32(K, buf[lane], p.r == 1, X, F);
    const int s0 = first_tap_f32<W>(X, F, t0);
    float pa[W];
    int ra[W];
#pragma unroll
    for (int k = 0; k < W; ++k) {
        pa[k] = es_tap_f32<W>(k, t0, K.bl, -K.bl);
        const int r = fold_cell(s0 + k, p.n) - row_lo;
        ra[k] = (unsigned)r < (unsigned)nrows ? r * plane : -1;
    }
#pragma unroll 1
    for (int t = 0; t < 2; ++t) {
        const float q = buf[(3 + t) * 32 + lane];
        if (!(fabsf(q) >= kNegligibleF32)) continue;
        QuadCols<W> col;
        quad_cols<W>(p, buf[(1 + t) * 32 + lane], col);
        if (fabsf(q) < kIntLimitF32) half_quad_point<W, kInt>(tile, ra, pa, col, q);
        else half_quad_point<W, kLarge>(tile, ra, pa, col, q);  // rare in grids of this size
    }
}

// The points of one class per lane in a slab (every lane of the warp calls it; P.base = 0: none).
// buf, count: the warp's queue of half quads and its fill.
template <int W, bool ANG>
__device__ __forceinline__ void spread_class_halves(const SpreadArgs &p, const PairData<float, 2> &P, float qbase,
                                                    const SplitTile &tile, int row_lo, int nrows, int plane,
                                                    SlabRange range, float *buf, int &count)
{
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
#pragma unroll 1
    for (int m = 0; 4 * m <= p.M; ++m) {
        const Quad Q = make_quad<ANG>(p, P, qbase, m);
#pragma unroll 1
        for (int s = 0; s < 2; ++s) {
            if (s && 4 * m == p.M) break;  // no mirror image
            const float mr = s ? Q.mr[1] : Q.mr[0];
            const float qa = (s ? Q.q2 : Q.q1) * mr * Q.mc[0];
            const float qb = m ? (s ? Q.q1 : Q.q2) * mr * Q.mc[1] : 0.0f;
            const float vr = s ? Q.vr[1] : Q.vr[0];
            const bool hit = fmaxf(fabsf(qa), fabsf(qb)) >= kNegligibleF32 && vr >= range.lo && vr <= range.hi;
            const unsigned mask = __ballot_sync(full, hit);
            const int n = __popc(mask), rank = __popc(mask & ((1u << lane) - 1u)), room = 32 - count;
            auto put = [&](int slot) {
                buf[slot] = vr;
                buf[32 + slot] = Q.vc[0];
                buf[64 + slot] = Q.vc[1];
                buf[96 + slot] = qa;
                buf[128 + slot] = qb;
            };
            if (hit && rank < room) put(count + rank);
            if (n >= room) {
                __syncwarp();
                spread_half_quad<W>(p, buf, true, tile, row_lo, nrows, plane);
                __syncwarp();
                if (hit && rank >= room) put(rank - room);
                count = n - room;
            } else {
                count += n;
            }
        }
    }
}

// The classes pr = first, first + stride, ... below end of one lane, into a slab (SLAB) or a tile
// that holds every row.  The lanes test one class each per step; the ones that are not negligible go through a
// queue of 32, so that a warp always spreads 32 classes at once: of a lane's own classes, the share
// that is negligible varies from lane to lane, and with every lane spreading its own the warp
// waited for the lane with the most (about a third of the lanes' time on the headline workload).
// buf: the warp's queues, 32 slots of spread_queue_values(2, true, ANG) floats.
template <int W, bool ANG, bool SLAB, bool SPLIT>
__device__ __forceinline__ void spread_quads(const SpreadArgs &p, long long first, long long end, long long stride,
                                             float sc, float pre, float tau, const SplitTile &tile, int row_lo,
                                             int nrows, int plane, float *buf)
{
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    float *cbuf = buf + 32 * kQuadValues;  // the class queue
    SlabRange range{0.0f, 0.0f};
    if constexpr (SLAB) range = slab_range<W>(p, row_lo, nrows);
    int count = 0, nclass = 0;             // queued (large or half) quads and classes, the same in every lane
    PairCursor c = pair_cursor(p.naxp, first);
    const PairStep st = pair_step(p.naxp, stride);
    for (;;) {
        const bool more = __any_sync(full, c.pr < end);
        if (!more && nclass == 0) break;
        PairData<float, 2> P;
        bool hit = false;
        int share = 0;
        if (c.pr < end) {
            PairCursor cc = c;
            if constexpr (SPLIT) {  // the share is the slowest index
                share = c.t / p.naxp;
                cc.t = c.t - share * p.naxp;
            }
            hit = class_passes<float, 2, ANG>(p, cc, sc, pre, tau, kNegligibleF32, P);
            pair_advance(p.naxp, c, st);
        }
        auto put = [&](int slot) {
            cbuf[slot] = P.cen[0];
            cbuf[32 + slot] = P.cen[1];
            cbuf[64 + slot] = P.rad;
            cbuf[96 + slot] = P.base;
            if constexpr (ANG) {
                cbuf[128 + slot] = P.x[0];
                cbuf[160 + slot] = P.x[1];
                cbuf[192 + slot] = P.dir[0];
                cbuf[224 + slot] = P.dir[1];
            }
            if constexpr (SPLIT) cbuf[(ANG ? 256 : 128) + slot] = __int_as_float(share);
        };
        const unsigned mask = __ballot_sync(full, hit);
        const int n = __popc(mask), rank = __popc(mask & ((1u << lane) - 1u)), room = 32 - nclass;
        if (hit && rank < room) put(nclass + rank);
        __syncwarp();
        if (n >= room || !more) {  // a full queue, or what is left at the end
            const bool valid = lane < min(nclass + n, 32);
            PairData<float, 2> C;
            zero_pair<float, 2>(C);
            int mine = 0;
            if (valid) {
                C.cen[0] = cbuf[lane];
                C.cen[1] = cbuf[32 + lane];
                C.rad = cbuf[64 + lane];
                C.base = cbuf[96 + lane];
                if constexpr (ANG) {
                    C.x[0] = cbuf[128 + lane];
                    C.x[1] = cbuf[160 + lane];
                    C.dir[0] = cbuf[192 + lane];
                    C.dir[1] = cbuf[224 + lane];
                }
                if constexpr (SPLIT) mine = __float_as_int(cbuf[(ANG ? 256 : 128) + lane]);
            }
            __syncwarp();
            if (hit && rank >= room) put(rank - room);
            nclass = max(n - room, 0);
            if constexpr (SLAB) spread_class_halves<W, ANG>(p, C, C.base * sc, tile, row_lo, nrows, plane, range, buf, count);
            else spread_class_quads<W, ANG, SPLIT>(p, C, C.base * sc, mine, tile, plane, buf, count);
        } else {
            nclass += n;
        }
    }
    __syncwarp();
    if constexpr (SLAB) spread_half_quad<W>(p, buf, lane < count, tile, row_lo, nrows, plane);
    else if (!SPLIT && lane < count) spread_large_quad<W>(p, buf, tile, plane);
}

// ---- 3D FP32 grids
//
// As in 2D, classes that are not negligible go through a class queue.  Their points are formed 32 at
// a time and sorted by size into three queues (those that reach the block's slab, with slabs), each
// spread with full warps: small points, whose first and last taps on every axis add nothing ((w-2)^3
// of w^3 taps: 64 of 216), points of 2^29 tile units or more (scaled integers), and the others.
// Measured: 3D Maxwell N = 16, M = 32 9.55 -> 6.4 ms (one point queue, classes spread by the lane that
// found them -> this), 3D VHS N = 24 67 -> 56 ms.  Bound by the bank conflicts of the tile's atomics
// (shared pipe 77% busy at N = 16), issue 57%.
// Spread slot `lane` (valid lanes) of the queue of one kind of point (the same for the whole warp).  One
// copy of the coordinates and weights serves the three kinds, and only the tap loops differ: with a
// copy for each the loop outgrew the instruction cache (N = 24: 4.7 of 9.6 warps stalled on instruction fetch, 0.6 with one copy; 67 -> 57 ms).
template <int W, bool SLAB>
__device__ __forceinline__ void queue3_spread(const SpreadArgs &p, const float *buf, int kind, bool valid,
                                              const SplitTile &tile, int row_lo, int nrows, int plane)
{
    if (!valid) return;
    const int lane = threadIdx.x & 31;
    const bool alg = (p.r == 1);
    const float bl = p.cf.bl, h2 = 2.0f / W;
    float X, F, t0, tl0, t1;
    grid_coord_f32(p.cf, buf[64 + lane], alg, X, F);
    const int cb = min(max(first_tap_f32<W>(X, F, tl0) + p.cpad, 0), p.ncol - W);  // clamped: x lies in [0, n/2]
    grid_coord_f32(p.cf, buf[32 + lane], alg, X, F);
    const int s1 = first_tap_f32<W>(X, F, t1);
    grid_coord_f32(p.cf, buf[lane], alg, X, F);
    const int s0 = first_tap_f32<W>(X, F, t0);
    const float q = buf[96 + lane];
    int wi[W], c1[W];
    float w1[W];
#pragma unroll
    for (int k = 0; k < W; ++k) {
        wi[k] = __float2int_rn(es_tap_f32<W>(k, tl0, bl, 30.0f - bl));
        w1[k] = es_tap_f32<W>(k, t1, bl, -bl);
        c1[k] = fold_cell(s1 + k, p.n) * p.ncol + cb;
    }
    const int sg = q < 0.0f ? -1 : 1;  // the sign of every contribution (or zero)
    float q4 = 4.0f * q;
    int sc = 0;
    if (kind == kLarge) q4 = scale_large(q4, q, sc);
    const int a0 = (kind == kSmall) ? 1 : 0;
#pragma unroll 1
    for (int a = a0; a < W - a0; ++a) {
        int r = fold_cell(s0 + a, p.n);
        if constexpr (SLAB) {
            r -= row_lo;
            if ((unsigned)r >= (unsigned)nrows) continue;
        }
        const float qa = q4 * es_f32(fmaf((float)a, h2, t0), bl, -bl);
        const int row = r * plane;
        if (kind == kInt) {
#pragma unroll
            for (int b = 0; b < W; ++b) {
                const int rq = __float2int_rn(qa * w1[b]), line = row + c1[b];
                unsigned wraps = 0u;
#pragma unroll
                for (int c = 0; c < W; ++c) wraps = tile.add_int_run(line + c, mulhi_rn(rq, wi[c]), wraps);
                if (wraps) tile.add_carries(line, W, wraps, sg);
            }
        } else if (kind == kSmall) {
#pragma unroll
            for (int b = 1; b < W - 1; ++b) {
                const int rq = __float2int_rn(qa * w1[b]), line = row + c1[b];
                unsigned wraps = 0u;
#pragma unroll
                for (int c = 1; c < W - 1; ++c) wraps = tile.add_int_run(line + c, mulhi_rn(rq, wi[c]), wraps);
                if (wraps) tile.add_carries(line + 1, W - 2, wraps, sg);
            }
        } else {  // rare: small code
#pragma unroll 1
            for (int b = 0; b < W; ++b) {
                float wb = w1[0];
                int line = c1[0];
#pragma unroll
                for (int k = 1; k < W; ++k)
                    if (b == k) {
                        wb = w1[k];
                        line = c1[k];
                    }
                const int rq = __float2int_rn(qa * wb);
#pragma unroll
                for (int c = 0; c < W; ++c) tile.add_scaled(row + line + c, mulhi_rn(rq, wi[c]), sc);
            }
        }
    }
}

template <int W, bool ANG, bool SLAB>
__device__ __forceinline__ void spread_points3(const SpreadArgs &p, long long first, long long end, long long stride,
                                               float sc, float pre, float tau, const SplitTile &tile, int row_lo,
                                               int nrows, int plane, float *buf)
{
    constexpr int PV = 32 * 4;  // values of a point queue: velocity and strength
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    float *cbuf = buf + 3 * PV;  // the class queue
    SlabRange range{0.0f, 0.0f};
    if constexpr (SLAB) range = slab_range<W>(p, row_lo, nrows);
    int fill = 0;                // of the point queues kInt, kLarge, kSmall, 8 bits each; the same in every lane
    int nclass = 0;
    PairCursor c = pair_cursor(p.naxp, first);
    const PairStep st = pair_step(p.naxp, stride);
    for (;;) {
        const bool more = __any_sync(full, c.pr < end);
        const bool drain = !more && nclass == 0;  // no class left: spread what is queued, and end
        PairData<float, 3> C;
        zero_pair<float, 3>(C);
        if (!drain) {
            PairData<float, 3> P;
            bool hit = false;
            if (c.pr < end) {
                hit = class_passes<float, 3, ANG>(p, c, sc, pre, tau, kNegligibleF32, P);
                pair_advance(p.naxp, c, st);
            }
            auto put = [&](int slot) {
#pragma unroll
                for (int l = 0; l < 3; ++l) cbuf[l * 32 + slot] = P.cen[l];
                cbuf[96 + slot] = P.rad;
                cbuf[128 + slot] = P.base;
                if constexpr (ANG) {
#pragma unroll
                    for (int o = 0; o < 4; ++o) cbuf[(5 + o) * 32 + slot] = P.x[o];
#pragma unroll
                    for (int l = 0; l < 3; ++l) cbuf[(9 + l) * 32 + slot] = P.dir[l];
                }
            };
            const unsigned mask = __ballot_sync(full, hit);
            const int n = __popc(mask), rank = __popc(mask & lt), room = 32 - nclass;
            if (hit && rank < room) put(nclass + rank);
            __syncwarp();
            if (n < room && more) {
                nclass += n;
                continue;
            }
            // a full queue, or what is left at the end
            if (lane < min(nclass + n, 32)) {
#pragma unroll
                for (int l = 0; l < 3; ++l) C.cen[l] = cbuf[l * 32 + lane];
                C.rad = cbuf[96 + lane];
                C.base = cbuf[128 + lane];
                if constexpr (ANG) {
#pragma unroll
                    for (int o = 0; o < 4; ++o) C.x[o] = cbuf[(5 + o) * 32 + lane];
#pragma unroll
                    for (int l = 0; l < 3; ++l) C.dir[l] = cbuf[(9 + l) * 32 + lane];
                }
            }
            __syncwarp();
            if (hit && rank >= room) put(rank - room);
            nclass = max(n - room, 0);
        }
        const float qbase = C.base * sc;
#pragma unroll 1
        for (int m = 0; m < (drain ? 1 : p.M); ++m) {
            float v[3], q = 0.0f;
            int kind = -1;
            if (!drain) {
                q = point_velocity_f32<3, ANG>(p, C, qbase, m, v);
                const float qa = fabsf(q);
                if (qa >= kNegligibleF32) kind = qa >= kIntLimitF32 ? kLarge : qa < p.cf.trim_q ? kSmall : kInt;
                if constexpr (SLAB)
                    if (!(v[0] >= range.lo && v[0] <= range.hi)) kind = -1;
            }
#pragma unroll 1
            for (int k = 0; k < 3; ++k) {
                const unsigned km = __ballot_sync(full, kind == k);
                const int cnt = (fill >> (8 * k)) & 255;
                if (!km && !(drain && cnt)) continue;
                float *const pq = buf + k * PV;
                auto put = [&](int slot) {
#pragma unroll
                    for (int l = 0; l < 3; ++l) pq[l * 32 + slot] = v[l];
                    pq[96 + slot] = q;
                };
                const int kn = __popc(km), kr = __popc(km & lt), kroom = 32 - cnt;
                if (kind == k && kr < kroom) put(cnt + kr);
                int now = cnt + kn;
                if (kn >= kroom || drain) {
                    __syncwarp();
                    queue3_spread<W, SLAB>(p, pq, k, !drain || lane < cnt, tile, row_lo, nrows, plane);
                    __syncwarp();
                    if (kind == k && kr >= kroom) put(kr - kroom);
                    now = max(kn - kroom, 0);
                }
                fill += (now - cnt) << (8 * k);
            }
        }
        if (drain) break;
    }
}

// ---- 2D FP64 grids in one tile: quads of mirrored classes
//
// The nodes are symmetric about 0 on every axis, so reflecting an axis maps a class {i, j} of that axis to
// {N-1-i, N-1-j}, its centre to the opposite and its points to their mirror images, whose taps
// are the same weights at the mirrored cells (u -> n/2 - u).  The classes of an orbit under the two
// reflections therefore share their axis evaluations, as the four points of a quad do: four
// evaluations (angle, map factor, w tap polynomials -- all of the FP64 arithmetic) serve up to 16
// points, which leaves the spreading bound by its integer products and atomics instead of by the
// FP64 pipe (1.7 operations per SM per clock).
// Measured against points one by one: N = 64, M = 32, tol 1e-13 101 -> 44 ms, N = 40, M = 40, tol 1e-14
// (logarithmic map) 26.3 -> 11.2 ms.  Then issue is 57% active, the FP64 pipe 42% and the shared
// pipe 36% busy (N = 40, M = 8): latency of 16 warps, no single unit.
//
// An item is one quad m of one orbit (small plans: a share of it); p.orb lists the axis orbits'
// representatives i + j <= N-1 (the
// mirror image of i + j = N-1 is itself and its strength counts once).

// Grid coordinate and fixed-point weights of one axis, out of line (one copy); the first tap.
template <int W>
__device__ __noinline__ int axis_eval_f64(const SpreadArgs &p, double v, FixW *out, double *m2)
{
    double mm;
    const double x = grid_coord_f64(p.cd, v, p.r == 1, mm);
    *m2 = mm;
    double wt[W];
    const int s = kernel_weights_f64<W>(x, wt);
#pragma unroll
    for (int a = 0; a < W; ++a) out[a] = fix_weight(wt[a]);
    return s;
}

// One orbit: the geometry of its representative class, and per mirror image e (bit 0: axis 0 reflected,
// bit 1: axis 1) the strength B x multiplicity x sum_o a a in grid units, or (angular kernels) the two
// terms of the sum; 0 for mirror images that are negligible (class_passes).
template <bool ANG>
struct Orbit {
    double cen[2], rad, x0[4], x1[4], dir[2];
};

template <bool ANG>
__device__ __forceinline__ bool load_orbit(const SpreadArgs &p, int o0, int o1, double sc, double tau, double floor_q,
                                           Orbit<ANG> &O)
{
    const int N = p.N;
    const double *a = static_cast<const double *>(p.a), *vn = static_cast<const double *>(p.vnode);
    const unsigned w0 = p.orb[o0], w1 = p.orb[o1];
    const int i0 = w0 & 0xffffu, j0 = w0 >> 16, i1 = w1 & 0xffffu, j1 = w1 >> 16;
    const double vi0 = vn[i0], vj0 = vn[j0], vi1 = vn[i1], vj1 = vn[j1];
    const double d0 = vi0 - vj0, d1 = vi1 - vj1;
    const double g = sqrt(d0 * d0 + d1 * d1);
    const TypedConsts<double> &K = p.cd;
    double B;
    switch (p.fast_gamma) {
    case 0: B = K.Bconst; break;
    case 1: B = K.Bconst * g; break;
    case 2: B = K.Bconst * sqrt(g); break;
    default: B = K.Bconst * pow(g, K.gamma); break;
    }
    O.cen[0] = 0.5 * (vi0 + vj0);
    O.cen[1] = 0.5 * (vi1 + vj1);
    O.rad = 0.5 * g;
    double U = K.Wang;
#pragma unroll
    for (int l = 0; l < 2; ++l) {
        const double R = fabs(O.cen[l]) + O.rad;
        U *= (p.r == 1) ? (K.SS + R * R) * K.invS : K.S * cosh(R * K.invS);
    }
    if constexpr (ANG) {
        const double ginv = g > 0.0 ? 1.0 / g : 0.0;
        O.dir[0] = d0 * ginv;
        O.dir[1] = d1 * ginv;
    }
    const double Bm = B * 2.0 * (i0 == j0 ? 0.5 : 1.0) * (i1 == j1 ? 0.5 : 1.0) * sc;
    bool any = false;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int e0 = e & 1, e1 = e >> 1;
        const int x0 = e0 ? N - 1 - i0 : i0, y0 = e0 ? N - 1 - j0 : j0;
        const int x1 = e1 ? N - 1 - i1 : i1, y1 = e1 ? N - 1 - j1 : j1;
        const double s0 = a[x0 * N + x1] * a[y0 * N + y1], s1 = a[y0 * N + x1] * a[x0 * N + y1];
        const double sum = s0 + s1, sabs = fabs(s0) + fabs(s1);
        bool keep = !((e0 && i0 + j0 == N - 1) || (e1 && i1 + j1 == N - 1));
        // the screening threshold is in strengths, per pair sum B sabs
        if (tau > 0.0 && B * sabs * U < tau) keep = false;
        if ((ANG ? sabs : fabs(sum)) * Bm * U * K.wmax < floor_q) keep = false;
        O.x0[e] = keep ? Bm * (ANG ? s0 : sum) : 0.0;
        O.x1[e] = (ANG && keep) ? Bm * s1 : 0.0;
        any = any || (keep && (ANG ? sabs : fabs(sum)) * Bm > 0.0);
    }
    return any;
}

// The point sets of a quad: column sets h0 .. h1-1 (coordinate h >> 1, mirrored if h is odd) times row sets
// g0 .. g1-1.  Small plans cut the quads into shares (SpreadArgs::nsplit: 4, one column set each, or 16,
// one point set each), so that a thread adds 4 points or 1 in series instead of 16.
struct QuadShare {
    int h0, h1, g0, g1;
};
template <bool SPLIT>
__device__ __forceinline__ QuadShare quad_share(const SpreadArgs &p, int share)
{
    if (!SPLIT) return QuadShare{0, 4, 0, 4};
    if (p.nsplit == 4) return QuadShare{share, share + 1, 0, 4};
    return QuadShare{share >> 2, (share >> 2) + 1, share & 3, (share & 3) + 1};
}

// Whether share H of quad m of an orbit whose mirror images have strengths holds a point of one of them.
template <bool ANG>
__device__ __forceinline__ bool share_holds(const Orbit<ANG> &O, const QuadShare &H)
{
    bool any = false;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const bool in = (H.h1 - H.h0 > 1 || (H.h0 & 1) == (e >> 1)) && (H.g1 - H.g0 > 1 || (H.g0 & 1) == (e & 1));
        any = any || (in && (O.x0[e] != 0.0 || (ANG && O.x1[e] != 0.0)));
    }
    return any;
}

// Share H of quad m of an orbit.
template <int W, bool ANG, bool SPLIT>
__device__ __forceinline__ void spread_orbit_quad(const SpreadArgs &p, const Orbit<ANG> &O, int m, const QuadShare &H,
                                                  const WideTile &tile, int plane)
{
    const double *sig = static_cast<const double *>(p.sig);
    const int nrow = (4 * m == p.M) ? 1 : 2, ncolumn = (m == 0) ? 1 : 2;  // 1: no mirror image
    const double cs = sig[2 * m], sn = sig[2 * m + 1];
    FixW fr[2][W], fc[2][W];  // local memory
    double mr[2], mc[2];
    int sr[2], cc[2];
#pragma unroll 1
    for (int k = 0; k < 2; ++k) {
        if (k < nrow && 2 * k < H.g1 && 2 * k + 1 >= H.g0)
            sr[k] = axis_eval_f64<W>(p, O.cen[0] + (k ? -O.rad : O.rad) * cs, fr[k], &mr[k]);
        if (k < ncolumn && 2 * k < H.h1 && 2 * k + 1 >= H.h0) {
            const int s = axis_eval_f64<W>(p, O.cen[1] + (k ? -O.rad : O.rad) * sn, fc[k], &mc[k]);
            cc[k] = min(max(s + p.cpad, 0), p.ncol - W);  // clamped: x lies in [0, n/2]
        }
    }
    double b0 = 1.0, b1 = 1.0;  // b_e(cos theta) of the points (+,+), (-,-) and (+,-), (-,+), unexchanged pair
    if constexpr (ANG) {
        const double a0 = O.dir[0] * cs, a1 = O.dir[1] * sn;
        const double e0 = (a0 + a1) * (a0 + a1), e1 = (a0 - a1) * (a0 - a1);
        b0 = b1 = p.cd.ang_even[p.nang_even - 1];
        for (int k = p.nang_even - 2; k >= 0; --k) {
            b0 = b0 * e0 + p.cd.ang_even[k];
            b1 = b1 * e1 + p.cd.ang_even[k];
        }
    }
    const double wm = static_cast<const double *>(p.wsig)[m];
    int cl[W];
#pragma unroll
    for (int c = 0; c < W; ++c) cl[c] = c;
#pragma unroll 1
    for (int h = H.h0; h < H.h1; ++h) {  // column sets: coordinate t, mirrored (e1) or not
        const int t = h >> 1, e1 = h & 1;
        if (t >= ncolumn) break;
        FixW fl[W];
#pragma unroll
        for (int c = 0; c < W; ++c) fl[c] = fc[t][e1 ? W - 1 - c : c];
        const int cb = e1 ? p.ncol - W - cc[t] : cc[t];
#pragma unroll 1
        for (int g = H.g0; g < H.g1; ++g) {  // row sets: coordinate s, mirrored (e0) or not
            const int s = g >> 1, e0 = g & 1;
            if (s >= nrow) break;
            double q = O.x0[e0 + 2 * e1];
            if constexpr (ANG) q = (s == t) ? q * b0 + O.x1[e0 + 2 * e1] * b1 : q * b1 + O.x1[e0 + 2 * e1] * b0;
            q *= wm * mr[s] * mc[t];
            if (q == 0.0) continue;
            const WideScale k = wide_scale(q);
#pragma unroll 1
            for (int a = 0; a < W; ++a) {
                int r = fold_cell(sr[s] + a, p.n);
                if (e0) r = p.nf - 1 - r;
                const unsigned long long R2 = fix_mul(k.q2, fr[s][a]) << 1;
                if (R2) wide_row<W>(tile, r * plane + cb, cl, R2, k, fl);
            }
        }
    }
}

// The items it = first, first + stride, ... below end of one lane.  Items that are not negligible go
// through the warp's queue of 32 item numbers (ids), so that 32 lanes spread 32 items.
template <int W, bool ANG, bool SPLIT>
__device__ __forceinline__ void spread_orbits(const SpreadArgs &p, long long first, long long end, long long stride,
                                              double sc, double tau, double floor_q, const WideTile &tile, int plane,
                                              unsigned *ids)
{
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    int queued = 0;  // the same in every lane
    PairCursor c = pair_cursor(p.norb, first);
    const PairStep st = pair_step(p.norb, stride);
    for (;;) {
        const bool more = __any_sync(full, c.pr < end);
        if (!more && queued == 0) break;
        bool hit = false;
        // an item: quad and share, m nsplit + share = c.t / norb (slowest, so that a warp's lanes mostly share it),
        // orbits c.t % norb and c.i
        const unsigned id = (unsigned)c.t * (unsigned)p.norb + (unsigned)c.i;
        if (c.pr < end) {
            Orbit<ANG> O;
            if constexpr (SPLIT) {
                const int k = c.t / p.norb, m = k / p.nsplit;
                const QuadShare H = quad_share<true>(p, k % p.nsplit);
                // (no mirror image of a zero sine or cosine)
                hit = !(m == 0 && H.h0 > 1) && !(4 * m == p.M && H.g0 > 1) &&
                      load_orbit<ANG>(p, c.t % p.norb, c.i, sc, tau, floor_q, O) && share_holds<ANG>(O, H);
            } else {
                hit = load_orbit<ANG>(p, c.t % p.norb, c.i, sc, tau, floor_q, O);
            }
            pair_advance(p.norb, c, st);
        }
        const unsigned mask = __ballot_sync(full, hit);
        const int n = __popc(mask), rank = __popc(mask & ((1u << lane) - 1u)), room = 32 - queued;
        if (hit && rank < room) ids[queued + rank] = id;
        __syncwarp();
        if (n < room && more) {
            queued += n;
            continue;
        }
        const bool valid = lane < min(queued + n, 32);
        const unsigned mine = valid ? ids[lane] : 0u;
        __syncwarp();
        if (hit && rank >= room) ids[rank - room] = id;
        queued = max(n - room, 0);
        if (valid) {
            const int t = (int)(mine / (unsigned)p.norb);
            Orbit<ANG> O;
            load_orbit<ANG>(p, t % p.norb, (int)(mine - (unsigned)t * (unsigned)p.norb), sc, tau, floor_q, O);
            const int k = t / p.norb;
            if constexpr (SPLIT)
                spread_orbit_quad<W, ANG, true>(p, O, k / p.nsplit, quad_share<true>(p, k % p.nsplit), tile, plane);
            else
                spread_orbit_quad<W, ANG, false>(p, O, k, quad_share<false>(p, 0), tile, plane);
        }
        __syncwarp();
    }
}

struct SlabGeom {
    int row_lo, nrows, plane, ncell;
};

__device__ __forceinline__ SlabGeom slab_geometry(const SpreadArgs &p, int D)
{
    SlabGeom g;
    g.plane = (D == 3) ? p.nf * p.ncol : p.ncol;
    const int slab = blockIdx.x % p.nslab;
    g.row_lo = slab * p.rows_per_slab;
    const int row_hi = min(g.row_lo + p.rows_per_slab, p.nf);
    g.nrows = row_hi - g.row_lo;
    g.ncell = g.nrows * g.plane;
    return g;
}

// Pair numbering: the threads of one slab cover the pairs with stride `nthr`, thread r of the
// slab (r = 32 warp + lane) starting at (r A) mod nthr with A = 1000003, a prime above any
// thread count (at most SMs x 2048), so the starts are a permutation of 0..nthr-1.  Lanes of a
// warp then take pairs A apart modulo nthr: unrelated (t, i), whose 32 points rarely hit the
// same grid cells.  Neighbouring pairs produce neighbouring points and would serialise the
// shared-memory atomics; a plain lane stride of nwarps keeps the lanes on one node column
// whenever nwarps and N share a power of two.
__device__ __forceinline__ void pair_schedule(const SpreadArgs &p, long long &first, long long &nthr)
{
    const long long groups = gridDim.x / p.nslab;
    nthr = groups * blockDim.x;
    const long long r = (long long)(blockIdx.x / p.nslab) * blockDim.x + threadIdx.x;
    first = (r * 1000003LL) % nthr;
}

// The strength bound B, from its partial sums when the loss kernel left those (the same order in
// every block and for every block size; the factor covers FP32 rounding of the pair terms and of the
// strengths in the FP32 kernels).  Every thread of the block calls it.
__device__ __forceinline__ double strength_bound(const SpreadArgs &p)
{
    if (p.nub == 0) return *p.bound;
    __shared__ double s_bound;
    if (threadIdx.x < 32) {
        double v = 0.0;
        for (int k = threadIdx.x; k < p.nub; k += 32) v += p.ub[k];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
        if (threadIdx.x == 0) {
            v *= 1.0 + 1e-5;
            s_bound = v;
            if (blockIdx.x == 0) *p.bound_out = v;
        }
    }
    __syncthreads();
    return s_bound;
}

template <int D, int W, bool ANG, bool SPLIT>
__global__ void __launch_bounds__(kMaxThreadsF32) k_spread_f32(const __grid_constant__ SpreadArgs p)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    launch_dependents();
    const SlabGeom G = slab_geometry(p, D);
    if (G.nrows <= 0) return;  // uniform over the block: an empty trailing slab does nothing
    // (the tile and the carries are the block's own: no earlier kernel of this evaluation touches them)
    int *words = reinterpret_cast<int *>(smem_raw);
    int *carry = p.carry + (size_t)blockIdx.x * p.tile_cells;
    for (int c = threadIdx.x; c < G.ncell; c += blockDim.x) {
        words[c] = 0;
        carry[c] = 0;
    }
    grid_wait();
    const double Bnd = strength_bound(p);
    __syncthreads();
    const int Eg = global_exponent(Bnd);
    // Tile unit 2^-Et with Et = Eg - tile_bits(D) (2^-47 B or finer in 2D, 2^-53 B in 3D); a coarser
    // unit for inputs so small that sc would leave the float range.
    const int K = product_scale(Eg);
    const int Et = min(Eg - tile_bits(D), 120 + K);
    const int shift = Eg - Et;
    const SplitTile tile{words, carry};
    const float pre = exp2_int(K), sc = exp2_int(Et - K);
    const float tau = p.nub ? 0.0f : (float)ldexp(*p.tau, K);
    long long first, nthr;
    pair_schedule(p, first, nthr);
    if (p.nslab > 1) {
        float *buf = reinterpret_cast<float *>(smem_raw + tile_bytes((size_t)p.rows_per_slab * G.plane, true)) +
                     (threadIdx.x >> 5) * 32 * spread_queue_values(D, true, ANG);
        if constexpr (D == 2)
            spread_quads<W, ANG, true, false>(p, first, p.nclass, nthr, sc, pre, tau, tile, G.row_lo, G.nrows, G.plane, buf);
        else
            spread_points3<W, ANG, true>(p, first, p.nclass, nthr, sc, pre, tau, tile, G.row_lo, G.nrows, G.plane, buf);
    } else if (p.queued) {
        float *buf = reinterpret_cast<float *>(smem_raw + tile_bytes(G.ncell, true)) +
                     (threadIdx.x >> 5) * 32 * spread_queue_values(D, true, ANG);
        if constexpr (D == 2)
            spread_quads<W, ANG, false, SPLIT>(p, first, SPLIT ? p.nclass * p.nsplit : p.nclass, nthr, sc, pre, tau, tile, 0,
                                               G.nrows, G.plane, buf);
        else
            spread_points3<W, ANG, false>(p, first, p.nclass, nthr, sc, pre, tau, tile, 0, G.nrows, G.plane, buf);
    } else {
        spread_pairs<float, D, W, SplitTile, ANG>(p, first, p.nclass, nthr, sc, pre, tau, kNegligibleF32, tile, G.nrows,
                                                   G.plane);
    }
    __syncthreads();
    for (int c = threadIdx.x; c < G.ncell; c += blockDim.x) {
        const long long v = tile.value(c);
        // |v 2^shift| <= B 2^Eg <= 2^61
        if (v)
            atomicAdd(p.grid + tile_to_grid_cell(c, D, p.nf, p.ncol, p.cpad, p.n, G.row_lo),
                      (unsigned long long)(v * (1ll << shift)));
    }
}

template <int D, int W, bool ANG, bool SPLIT>
__global__ void __launch_bounds__(kMaxThreadsF64, 1) k_spread_f64(const __grid_constant__ SpreadArgs p)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    launch_dependents();
    const SlabGeom G = slab_geometry(p, D);
    if (G.nrows <= 0) return;  // uniform over the block
    // fraction, low and high words of rows_per_slab x plane cells each
    const size_t tile_cells = (size_t)p.rows_per_slab * G.plane;
    unsigned *words = reinterpret_cast<unsigned *>(smem_raw);
    const WideTile tile{words, words + tile_cells, reinterpret_cast<int *>(words + 2 * tile_cells)};
    for (int c = threadIdx.x; c < G.ncell; c += blockDim.x) {
        tile.fr[c] = 0u;
        tile.lo[c] = 0u;
        tile.hi[c] = 0;
    }
    load_kernel_poly(p.kpoly);
    grid_wait();
    const double Bnd = strength_bound(p);
    __syncthreads();
    const int Eg = global_exponent(Bnd);
    const double tau = p.nub ? 0.0 : *p.tau;
    const double sc = ldexp(1.0, Eg);  // strengths in grid units
    // classes whose summed strength bounds stay below 2^-64 B are skipped (per-point bound below
    // floor_q, and at most nclass classes): 2^-3 grid units at most in all
    const double floor_q = ldexp(Bnd, Eg - 64) * p.cd.wmax / (double)p.nclass;
    long long first, nthr;
    pair_schedule(p, first, nthr);
    if (p.nslab > 1) {
        double *buf = reinterpret_cast<double *>(smem_raw + tile_bytes(tile_cells, false)) +
                      (threadIdx.x >> 5) * 32 * spread_queue_values(D, false);
        spread_pairs_queued<D, W, ANG>(p, first, p.nclass, nthr, sc, tau, floor_q, tile, G.row_lo, G.nrows, G.plane,
                                       buf);
    } else if (D == 2 && p.queued) {
        if constexpr (D == 2) {
            unsigned *ids = reinterpret_cast<unsigned *>(smem_raw + tile_bytes(tile_cells, false)) +
                            (threadIdx.x >> 5) * 32;
            spread_orbits<W, ANG, SPLIT>(p, first, p.nitem, nthr, sc, tau, floor_q, tile, G.plane, ids);
        }
    } else {
        spread_pairs<double, D, W, WideTile, ANG>(p, first, p.nclass, nthr, sc, 1.0, tau, floor_q, tile, G.nrows,
                                                   G.plane);
    }
    __syncthreads();
    for (int c = threadIdx.x; c < G.ncell; c += blockDim.x) {
        const long long v = tile.value(c);
        if (v) atomicAdd(p.grid + tile_to_grid_cell(c, D, p.nf, p.ncol, p.cpad, p.n, G.row_lo), (unsigned long long)v);
    }
}

template <int D, int W, bool ANG>
cudaError_t launch_f32(const SpreadArgs &a, int blocks, int threads, size_t smem, cudaStream_t s)
{
    auto kern = k_spread_f32<D, W, ANG, false>;
    if constexpr (D == 2)
        if (a.nsplit > 1) kern = k_spread_f32<D, W, ANG, true>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return launch_dependent(kern, blocks, threads, smem, s, a);
}

template <int D, int W, bool ANG>
cudaError_t launch_f64(const SpreadArgs &a, int blocks, int threads, size_t smem, cudaStream_t s)
{
    auto kern = k_spread_f64<D, W, ANG, false>;
    if constexpr (D == 2)
        if (a.nsplit > 1) kern = k_spread_f64<D, W, ANG, true>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return launch_dependent(kern, blocks, threads, smem, s, a);
}

// Compile-time dispatch on the kernel width w in [W, WMAX].  ANG: the angular-kernel variant
// (instantiated in its own translation units).
template <bool F32, int D, int W, int WMAX, bool ANG>
struct WidthDispatch {
    static cudaError_t run(const SpreadArgs &a, int w, int blocks, int threads, size_t smem, cudaStream_t s)
    {
        if (w == W) {
            if constexpr (F32) return launch_f32<D, W, ANG>(a, blocks, threads, smem, s);
            else return launch_f64<D, W, ANG>(a, blocks, threads, smem, s);
        }
        if constexpr (W < WMAX) return WidthDispatch<F32, D, W + 1, WMAX, ANG>::run(a, w, blocks, threads, smem, s);
        return cudaErrorInvalidValue;
    }
};

}  // namespace spread_detail
}  // namespace pgb
