// Internal declarations of the sm_103a collision-operator library (not part of the ABI).
#pragma once

#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>

#include "pg_boltz.h"

namespace pgb {

// Everything the spreading kernel reads, passed by value.  The nodes, weights and
// coefficients are in the kernel's arithmetic type T (float or double).
// Angular factor of the collision kernel B(|g|, cos theta) = Bconst |g|^gamma b(cos theta)
// (Eq. collision_form), b(c) = sum_{p < n} c_p c^p; n = 0 is the VHS kernel (b = 1).
constexpr int kMaxAngular = 8;
// Coefficients of the FP64 spreading kernel's piecewise polynomial form (kernel_poly on the host):
// ceil(w/2) taps of kernel_poly_terms(w) each, for widths up to 16.  Degree w interpolates each tap
// to about the kernel's own truncation error exp(-beta) at the default oversampling 2 for w >= 7;
// narrower kernels take two more terms, which keeps oversampling up to 4 within a few times it.
__host__ __device__ constexpr int kernel_poly_terms(int w) { return w < 12 ? w + 3 : w + 1; }
constexpr int kPolyCoefF64 = 8 * 17;
struct Angular {
    int n;
    double c[kMaxAngular];
};

// Loop-invariant constants of the spreading kernels in their arithmetic type, filled once on the
// host (or by the batched kernel's cell switch) so the point loops convert nothing from double.
template <typename T>
struct TypedConsts {
    T S, invS, SS;      // map scale, 1/S, S^2
    T gs;               // grid_scale
    T Bconst, gamma;    // kernel constant and exponent
    T Wang;             // Wsig * angmax (pair bound factor)
    T wmax;             // wmax_frac
    T bl;               // beta log2(e): ES kernel values as powers of two
    T trim_q;
    T ang_even[kMaxAngular / 2];
    // FP32 point coordinates without systematic offsets or scale errors: a grid coordinate is
    // x = xq -+ atan(v/S) gs (r = 1) or 2 atan(exp(-v/S)) gs (r = 0) with xq = n/4 exact and the
    // products by 1/S and gs carried in two terms (hi + lo); zero in TypedConsts<double>
    T invS_lo, gs_lo, xq;
};

struct SpreadArgs {
    int d, N, M, r;
    int nnode;            // N^d interior nodes
    int naxp;             // unordered pairs of node indices per axis, unordered_pairs(N)
    long long nclass;     // classes of node pairs that share their points, naxp^d
    int nsplit;           // one-slab 2D grids, shares: FP32: of a class' quads; FP64: of a quad's points (1: all at once)
    int n, nf;            // periodic grid size, folded cells per axis (n/2 + 1)
    int rows_per_slab;    // folded-grid rows (axis 0) held in shared memory by one block
    int nslab;            // number of slabs covering axis 0
    int fast_gamma;       // 0: gamma = 0, 1: gamma = 1, 2: gamma = 1/2, 3: general pow
    double S, gamma, Bconst;
    double beta;          // exponential-of-semicircle shape
    double trim_q;        // FP32: below this many tile units the first and last taps of every axis add nothing
    double grid_scale;    // n / (2 pi): angle -> grid coordinate
    const void *vnode;    // N node velocities (same on every axis)
    const float *vnode_lo;  // FP32 plans: v - (double)vnode, so that hi + lo carries the node exactly
                            // to about 2^-48 (nullptr for FP64 plans)
    const void *a;        // nnode values a_i = W_i g_i
    const void *sig;      // M x d sphere points
    const void *wsig;     // M sphere weights
    double Wsig;          // sum_m w_m
    double wmax_frac;     // max_m w_m / sum_m w_m: one point's share of a pair's strength bound
    const double *bound;  // device scalar B >= sum_p |q_p| (written by the loss kernel)
    const double *ub;     // nub > 0: the partial sums of B / (1 + 1e-5) (LossArgs::ub); the kernel adds them up
    int nub;              // and block 0 writes *bound.  0: *bound and *tau were written before
    double *bound_out;    // = bound
    const double *tau;    // device scalar: node pairs whose strength bound is below it are skipped (0: none)
    unsigned long long *grid;  // nf^d folded grid, int64 fixed point in units of 2^-Eg
    int cpad;             // unfolded padding columns before the last axis' columns in block tiles
    int ncol;             // tile cells along the last axis (tile_cols)
    int tile_cells;       // cells of one block tile (rows_per_slab rows)
    int *carry;           // FP32: per-block carry counters, blocks x tile_cells (global memory)
    int queued;           // one-slab grids: 1 when the warps' queues follow the tile in shared memory (FP32:
                          // spread_queue_bytes of the launch's threads; FP64 2D: 32 item numbers per
                          // warp, and the fields below are set)
    const unsigned *orb;  // FP64 2D: the axis orbits' representative node pairs, i + 65536 j
    int norb;             // their number
    long long nitem;      // quads of all orbits, (M/4 + 1) norb^2, times nsplit
    // angular kernel: a spread pair stands for both orders, whose cos theta differ in sign, so
    // the gain needs the even part b_e(c) = (b(c) + b(-c))/2 = sum_k ang_even[k] c^(2k) only
    int nang_even;        // terms of ang_even; 0: VHS kernel (no angular factor)
    double ang_even[kMaxAngular / 2];
    double angmax;        // sum_k |ang_even[k]| >= |b_e(c)| on [-1, 1] (1 for VHS)
    // FP64 kernel weights: tap a (< ceil(w/2)) of a point at offset y in [-1, 1] within its cell is
    // E_a(y^2) + y O_a(y^2), and tap w-1-a is E_a(y^2) - y O_a(y^2); with P = kernel_poly_terms(w),
    // kpoly[a P + k] (device, kPolyCoefF64 doubles) holds the (P+1)/2 coefficients of E_a, then
    // the P/2 of O_a, lowest power first
    const double *kpoly;
    TypedConsts<float> cf;   // the double fields above as float (FP32 kernels)
    TypedConsts<double> cd;  // ... and as double (FP64 kernels)
};

// Fill a.cf and a.cd from the double fields (call after setting S, grid_scale, Bconst, gamma,
// Wsig, angmax, wmax_frac, beta, trim_q and ang_even).
template <typename T>
__host__ __device__ inline void fill_typed_consts(const SpreadArgs &a, TypedConsts<T> &c)
{
    c.S = T(a.S);
    c.invS = T(1.0 / a.S);
    c.SS = T(a.S * a.S);
    c.gs = T(a.grid_scale);
    c.Bconst = T(a.Bconst);
    c.gamma = T(a.gamma);
    c.Wang = T(a.Wsig * a.angmax);
    c.wmax = T(a.wmax_frac);
    c.bl = T(a.beta * 1.4426950408889634);
    c.trim_q = T(a.trim_q);
    for (int k = 0; k < kMaxAngular / 2; ++k) c.ang_even[k] = T(k < a.nang_even ? a.ang_even[k] : 0.0);
    c.invS_lo = T(1.0 / a.S - double(c.invS));
    c.gs_lo = T(a.grid_scale - double(c.gs));
    c.xq = T(0.25 * a.n);
}
__host__ __device__ inline void fill_spread_consts(SpreadArgs &a)
{
    fill_typed_consts<float>(a, a.cf);
    fill_typed_consts<double>(a, a.cd);
}
template <typename T>
__device__ __forceinline__ const TypedConsts<T> &kconst(const SpreadArgs &a)
{
    if constexpr (sizeof(T) == 4) return a.cf;
    else return a.cd;
}

// Programmatic dependent launch.  The kernels of one evaluation follow each other on the plan's stream,
// each a few microseconds but for the spreading.  A kernel launched by launch_dependent may start when
// every block of its predecessor has called launch_dependents() (or ended), so that its launch and
// set-up overlap the predecessor's run; grid_wait() then waits until the predecessor has completed and
// its writes are visible.  Every such kernel calls grid_wait() before it touches what an earlier
// kernel writes or reads; the first kernel of an evaluation is launched in the ordinary way.  In these
// kernels only the plan's constants may be const __restrict__: what an earlier kernel of the evaluation
// writes changes while they run, so the compiler must neither read it through the non-coherent path nor
// move its loads across grid_wait(), which orders only memory that other pointers may reach.  Without
// the launch attribute both calls do nothing.  2D Maxwell N = 16: 56.4 -> 49.5 us.
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
template <typename... P, typename... A>
cudaError_t launch_dependent(void (*kern)(P...), int blocks, int threads, size_t smem, cudaStream_t s, A &&...args)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    // captured kernels are launched in the ordinary way: as graph nodes with programmatic edges they ran
    // slower (RK4 at N = 32: 7.3 -> 7.7 ms)
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    const bool plain = cudaStreamIsCapturing(s, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone;
    cfg.attrs = &at;
    cfg.numAttrs = plain ? 0 : 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

// Unordered pairs of n things, equal ones included.
__host__ __device__ inline long long unordered_pairs(long long nnode) { return nnode * (nnode + 1) / 2; }

// Values per slot of the spreading kernels' warp queues.  FP32 2D: a large or half quad (6) and a class
// (5, angular kernels 9); 3D: three points by size (velocity and strength, 4 each) and a class (5,
// angular kernels 12).  FP64: a point, d coordinates and its strength.
__host__ __device__ constexpr int spread_queue_values(int d, bool f32, bool ang = false)
{
    return !f32 ? d + 1 : d == 2 ? (ang ? 15 : 11) : (ang ? 24 : 17);
}
// Shared memory of the warp queues of a spreading block of `threads` threads: 32 slots per warp.
__host__ __device__ constexpr size_t spread_queue_bytes(int threads, int d, bool f32, bool ang = false)
{
    return (size_t)(threads / 32) * 32 * spread_queue_values(d, f32, ang) * (f32 ? 4 : 8);
}
// Shared memory of a block tile of `cells` cells, rounded up to 16 bytes (the queues follow it):
// FP32 tiles hold one 32-bit word per cell, FP64 tiles three (fraction, low and high words).
__host__ __device__ inline size_t tile_bytes(size_t cells, bool f32)
{
    return (cells * (f32 ? 4 : 12) + 15) / 16 * 16;
}

// Padding columns of the block tiles' last axis for kernel width w, before the grid's columns and after
// them: the unfolded support of a point at grid coordinate x in [0, n/2] runs from floor(x - w/2) + 1 to
// floor(x - w/2) + w, i.e. from -((w-1)/2) to n/2 + w/2.  FP64 2D tiles are symmetric (their mirrored
// classes need it).  FP64 3D tiles have none (N = 11, w = 14: 24 instead of 38 cells per line of the
// grid, so that it fits one block instead of two slabs, both of which nearly every point reaches).
// (With one margin column more on each side FP32 3D tiles left room for 16 warps' queues instead of 20:
// N = 24 52 -> 44 ms, N = 16 6.4 -> 6.0 ms.)
__host__ __device__ inline int tile_col_pad(int w, int d, bool f32) { return f32 ? (w - 1) / 2 : d == 3 ? 0 : w / 2; }
__host__ __device__ inline int tile_cols(int nf, int w, int d, bool f32)
{
    return nf + tile_col_pad(w, d, f32) + ((d == 3 && !f32) ? 0 : w / 2);
}

// FP32 block tiles count in units 2^-(Eg - tile_bits(d)), about 2^-47 B (2D) or 2^-53 B (3D) for the
// strength bound B: each contribution is rounded to the tile unit once, and with w^3 contributions
// per point and the deconvolution's growth along three axes, 3D needs the finer unit for the FP32
// path's accuracy (with 2^-47 B the rounding was 3e-6 of the gain norm on the 3D gamma = 1/2
// workload, with 2^-53 B 4e-7); a coarser unit makes more node pairs negligible (skipped exactly)
// and more points fit the integer products, which is faster.
__host__ __device__ constexpr int tile_bits(int d) { return d == 3 ? 8 : 14; }

// Exponent Eg of the grid's fixed-point unit 2^-Eg: the largest E with B 2^E < 2^61 for the
// bound B >= sum_p |q_p| (0 when B is zero or not finite).
__host__ __device__ inline int global_exponent(double B)
{
    if (!(B > 0.0) || !(B < 1.0e300)) return 0;
    return 60 - ilogb(B);
}

// The FP32 kernels form the products a_i a_j of node values, and so the strengths, times 2^K with
// K = product_scale(Eg), about -log2 B: B bounds their sum, so they and the sums over a class stay away
// from both ends of FP32's range for every amplitude at which the node values themselves fit it (a power
// of two: no rounding changes).  K is kept within +-100, so that 2^K a_i does not leave the range in its turn.
// Without it the class sums overflowed from amplitudes of 1e19 on, and products underflowed below 1e-14.
__host__ __device__ inline int product_scale(int Eg)
{
    const int e = Eg - 60;
    return e > 100 ? 100 : e < -100 ? -100 : e;
}

// Screening of negligible node pairs: the loss kernel counts the pair bounds per binary
// exponent (kScreenBins bins, bin k holds bounds in [2^(k - kScreenOffset), 2^(k+1 - kScreenOffset)),
// the first and last bins also everything below / above).
constexpr int kScreenBins = 256;
constexpr int kScreenOffset = 200;
// Launch the spreading kernel for (precision, d, w); returns cudaSuccess or the launch error.
// One translation unit per (precision, d) keeps the parallel build short.
cudaError_t launch_spread_f32_d2(const SpreadArgs &a, int w, int blocks, int threads, size_t smem, cudaStream_t s);
cudaError_t launch_spread_f32_d3(const SpreadArgs &a, int w, int blocks, int threads, size_t smem, cudaStream_t s);
cudaError_t launch_spread_f64_d2(const SpreadArgs &a, int w, int blocks, int threads, size_t smem, cudaStream_t s);
cudaError_t launch_spread_f64_d3(const SpreadArgs &a, int w, int blocks, int threads, size_t smem, cudaStream_t s);
// The same with the angular factor of the collision kernel (a.nang_even > 0; called by the above).
cudaError_t launch_spread_f32_d2_ang(const SpreadArgs &a, int w, int blocks, int threads, size_t smem, cudaStream_t s);
cudaError_t launch_spread_f32_d3_ang(const SpreadArgs &a, int w, int blocks, int threads, size_t smem, cudaStream_t s);
cudaError_t launch_spread_f64_d2_ang(const SpreadArgs &a, int w, int blocks, int threads, size_t smem, cudaStream_t s);
cudaError_t launch_spread_f64_d3_ang(const SpreadArgs &a, int w, int blocks, int threads, size_t smem, cudaStream_t s);
// Highest kernel width with a compiled spreading kernel for each type.
constexpr int kMaxWidthF32 = 10;
constexpr int kMaxWidthF64 = 16;
static_assert(kPolyCoefF64 >= ((kMaxWidthF64 + 1) / 2) * kernel_poly_terms(kMaxWidthF64) &&
                  kPolyCoefF64 >= 6 * kernel_poly_terms(11),
              "kernel polynomial storage");
constexpr int kMinWidth = 2;
// Largest spreading block for each type (the kernels' launch bounds).  FP32: 640 threads with up to 96
// registers (the 2D quads keep their weights of both columns and a row set in registers; at 1024
// threads x 64 registers they spill: 768 batched cells 33.2 -> 31.6 ms, RK4 at N = 32 9.6 -> 8.4 ms, 2D
// Maxwell N = 16 88 -> 84 us, 3D VHS N = 24 63.7 -> 62.4 ms with 640).  Options may ask for up to
// kAcceptThreadsF32; a launch then has kMaxThreadsF32.
constexpr int kMaxThreadsF32 = 640;
constexpr int kAcceptThreadsF32 = 1024;
// FP64: 512 threads with 128 registers (the axis weights are formed out of line).  Options may ask for
// up to 512 in 3D and 256 in 2D.
constexpr int kMaxThreadsF64 = 512;
__host__ __device__ constexpr int accept_threads(int d, bool f32)
{
    return f32 ? kAcceptThreadsF32 : d == 3 ? 512 : 256;
}
// Largest block of the batched FP32 spreading kernel.
constexpr int kBatchThreadsF32 = kMaxThreadsF32;

// Three-axis shape of a C-order array; 2D arrays use e0 = 1.
struct Dims3 {
    int e[3];
};

// out = A contracted along axis `ax` (A is m x dims.e[ax], row-major) with `in`, or with the int64
// fixed-point array `fixed_in` (when not null).
struct AxisPass {
    const double *in;
    const unsigned long long *fixed_in;
    Dims3 dims;
    int ax, m;
    const double *A;
    double *out;
};
cudaError_t launch_axis_pass(const AxisPass &P, cudaStream_t s);
// Two independent passes in one launch; P0's fixed-point input is in units 2^-Eg (Eg from *B), times scale.
cudaError_t launch_axis_pass_pair(const AxisPass &P0, const AxisPass &P1, const double *B, double scale, cudaStream_t s);
// Last reconstruction pass along axis 2, then a_i = acc * prod_l scale[i_l];
// writes a (FP64) and, if af != nullptr, a float copy and, if alo != nullptr, what it leaves of a (a float);
// clears the nclear words at clear.
cudaError_t launch_recon_last(const double *in, Dims3 in_dims, const double *A, int m,
                              const double *scale, int d, double *a, float *af, float *alo, unsigned long long *clear,
                              long long nclear, cudaStream_t s);
// The loss sums h_i and the strength bound by mirror images of the nodes (VHS kernels, and angular ones
// in 2D, without screening; launch_loss otherwise).  f32: FP32 pair terms.
struct LossArgs {
    const double *a;        // N^d node values
    const float *a32, *a32lo;  // FP32 plans: a as a32 + a32lo (a32lo: 2D angular ones)
    const double *v64;      // N node velocities
    const float *v32, *v32lo;
    int N, M;
    int nloss;              // nodes with every index <= (N-1)/2, one block each
    int nbound;             // blocks of the bound, each writing one partial sum to ub
    const unsigned *orb;    // an axis' orbits of node pairs (SpreadArgs::orb)
    int norb;
    long long norbits;      // norb^d
    const double *sig64;    // sphere set (angular kernels)
    const float *sig32;
    Angular ang;
    double angmax, gamma;
    int fast_gamma;
    double Bw;
    const double *inv_mu2;
    double S;
    int r;
    double *h;              // N^d loss weights
    double *ub;             // nbound partial sums of the strength bound B / (1 + 1e-5)
};
cudaError_t launch_loss_mirror(const LossArgs &L, int d, bool f32, cudaStream_t s);
// Loss: h_i = a_i * Lsum_i * prod_l inv_mu2[i_l], Lsum_i = Bw * sum_j a_j B(|v_i - v_j|) A_ij,
// A_ij = (1/Wsig) sum_m w_m b(cos theta_ijm) for an angular kernel (ang.n > 0; the sum over the
// sphere set then runs per pair), 1 otherwise (Bw = Bconst Wsig);
// also ub_i = |a_i| Bw angmax sum_j |a_j| B_ij prod_l mu^-2(|c_l| + rad), an upper bound of the
// spreading strengths of the pairs (i, .).  FP32 pair terms (node differences with the nodes'
// rounding vnode32_lo added back, summed in FP64) carry a relative error near 1e-7 that differs
// from pair to pair; the bound gets a 1e-5 margin in k_bound_reduce.
// vnode32 != nullptr selects FP32 pair terms (the FP32 path).
// hist != nullptr: also count every pair bound |a_i| Bw |a_j| B_ij prod mu^-2 into the screening histogram.
cudaError_t launch_loss(const double *a, const float *a32, const double *vnode, const float *vnode32,
                        const float *vnode32_lo, int N,
                        int d, int M,
                        const double *sig, const double *wsig, const float *sig32, const float *wsig32,
                        const Angular &ang, double angmax, double Wsig, double gamma,
                        int fast_gamma, double Bw, const double *inv_mu2, double S, int r,
                        double *h, double *ub, unsigned long long *hist, cudaStream_t s);
// Screening bin of a pair bound u > 0.
__host__ __device__ inline int screen_bin(double u)
{
    int e = ilogb(u) + kScreenOffset;
    return e < 0 ? 0 : (e >= kScreenBins ? kScreenBins - 1 : e);
}
// B = sum_i ub_i (fixed summation order), written to *B.  When hist != nullptr also the screening
// threshold *tau = 2^(k - kScreenOffset) for the largest k with
//   sum_{bins j < k} count_j 2^(j+1 - kScreenOffset) <= eps * B
// (an upper bound of the total strength of the pairs below tau), else *tau = 0.
cudaError_t launch_bound_reduce(const double *ub, int n, const unsigned long long *hist, double eps, double *B,
                                double *tau, cudaStream_t s);
// Exact / FP32 value of the constant factors of an FP32 point strength: Bconst (the kernel's
// constant), the common sphere weight w and 1/S per axis enter every strength as rounded FP32
// constants, a common relative error that the transform of the FP32 grid divides out in FP64.
inline double fp32_strength_correction(double Bconst, double w, double S, int d)
{
    double c = (Bconst / (double)(float)Bconst) * (w / (double)(float)w);
    for (int l = 0; l < d; ++l) c *= (1.0 / S) / (double)(float)(1.0 / S);
    return c;
}
// Final pass along axis 2: Qp = D . G, Qm = E . H, Q = Qp - Qm (also copied to Qcopy).
cudaError_t launch_final(const double *G, Dims3 g_dims, const double *D, const double *H,
                         Dims3 h_dims, const double *E, int m, double *Q, double *Qplus,
                         double *Qcopy, cudaStream_t s);
// RK stage argument y = x + c k, and the RK4 update f += dt/6 (k1 + 2k2 + 2k3 + k4).
cudaError_t launch_axpy(const double *x, const double *k, double c, double *y, long long n, cudaStream_t s);
cudaError_t launch_rk4_update(double *f, const double *k1, const double *k2, const double *k3, const double *k4,
                              double dt, long long n, cudaStream_t s);
// Discrete weak-form functionals and scales for phi in {1, v_l, |v|^2}, added into out[2(d+2)].
cudaError_t launch_weak_moments(const double *a, const double *vnode, int N, int d, int M, const double *sig,
                                const double *wsig, const Angular &ang, double gamma, int fast_gamma, double Bconst,
                                double *out, cudaStream_t s);
// Diagnostics: mass/energy functionals of Q and Qplus and their L2 norms into out[6].
cudaError_t launch_moments(const double *Q, const double *Qplus, int d, int N, double S,
                           double *out, cudaStream_t s);

// Set the thread-local text returned by pg_boltz_last_error; returns code.
int record_error(int code, const char *msg);

}  // namespace pgb
