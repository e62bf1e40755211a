// Host-side internals shared by the plain and the batched plans: error state, device
// allocation with fault injection, and the quadrature / sphere / transform tables.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include "host.cuh"

#define PG_API extern "C" __attribute__((visibility("default")))

namespace {
thread_local std::string g_last_error;
std::atomic<int> g_fail_alloc_countdown{0};
}  // namespace

namespace pgbh {

int set_error(int code, const char *fmt, ...)
{
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof(buf), fmt, ap);
    va_end(ap);
    g_last_error = buf;
    return code;
}

int cuda_check(cudaError_t e, const char *what)
{
    if (e == cudaSuccess) return PG_OK;
    return set_error(PG_ERR_CUDA, "%s: %s", what, cudaGetErrorString(e));
}

// Gauss-Legendre nodes and weights on [-1, 1] (Newton iteration on P_n).
void gauss_legendre(int n, std::vector<double> &x, std::vector<double> &w)
{
    x.assign(n, 0.0);
    w.assign(n, 0.0);
    for (int i = 0; i < (n + 1) / 2; ++i) {
        double z = std::cos(kPi * (i + 0.75) / (n + 0.5));
        double dp = 0.0;
        for (int it = 0; it < 100; ++it) {
            double p0 = 1.0, p1 = z;
            for (int k = 2; k <= n; ++k) {
                double p2 = ((2.0 * k - 1.0) * z * p1 - (k - 1.0) * p0) / k;
                p0 = p1;
                p1 = p2;
            }
            dp = n * (z * p1 - p0) / (z * z - 1.0);
            double dz = p1 / dp;
            z -= dz;
            if (std::fabs(dz) < 1e-16) break;
        }
        double p0 = 1.0, p1 = z;
        for (int k = 2; k <= n; ++k) {
            double p2 = ((2.0 * k - 1.0) * z * p1 - (k - 1.0) * p0) / k;
            p0 = p1;
            p1 = p2;
        }
        dp = n * (z * p1 - p0) / (z * z - 1.0);
        x[i] = -z;
        x[n - 1 - i] = z;
        w[i] = w[n - 1 - i] = 2.0 / ((1.0 - z * z) * dp * dp);
    }
}


int grid_size(int N, double sigma)
{
    int n = (int)std::ceil(sigma * (2 * N + 1));
    return n + (n % 2);
}

double kernel_beta(int w, double sigma) { return 0.97 * kPi * (1.0 - 0.5 / sigma) * w; }

double trim_strength(int w, double beta)
{
    if (w < 4) return 0.0;
    const double t = 1.0 - 2.0 / w;
    return 0.37 / std::exp(beta * (std::sqrt(1.0 - t * t) - 1.0));
}

int width_for(double tol, double sigma)
{
    double per_w = 0.9 * std::sqrt(2.0 * (1.0 - 1.0 / sigma));
    int w = (int)std::ceil((-std::log10(tol) - 0.8) / per_w);
    return std::max(w, pgb::kMinWidth);
}

// Tap a of the kernel as a function of the offset y in [-1, 1]: t = (y + 1 + 2a - w)/w.
static long double kernel_tap(int w, double beta, int a, long double y)
{
    const long double t = (y + 1.0L + 2.0L * a - w) / w;
    const long double om = 1.0L - t * t;
    return om > 0.0L ? expl((long double)beta * (sqrtl(om) - 1.0L)) : 0.0L;
}

// Interpolate each tap at the P = kernel_poly_terms(w) Chebyshev points of [-1, 1] (coefficients
// of T_j by the discrete cosine sums, then expanded in powers of y through
// T_{j+1} = 2y T_j - T_{j-1}), all in long double; split into even and odd parts.
void kernel_poly(int w, double beta, double *c)
{
    const int P = pgb::kernel_poly_terms(w), NE = (P + 1) / 2, NO = P / 2;
    const long double pi = 3.141592653589793238462643383279502884L;
    std::vector<long double> g(P), cheb(P), mono(P), Tm(P), T0(P), T1(P);
    for (int a = 0; a < (w + 1) / 2; ++a) {
        for (int k = 0; k < P; ++k) g[k] = kernel_tap(w, beta, a, cosl(pi * (k + 0.5L) / P));
        for (int j = 0; j < P; ++j) {
            long double acc = 0.0L;
            for (int k = 0; k < P; ++k) acc += g[k] * cosl(pi * j * (k + 0.5L) / P);
            cheb[j] = acc * (j == 0 ? 1.0L : 2.0L) / P;
        }
        std::fill(mono.begin(), mono.end(), 0.0L);
        std::fill(T0.begin(), T0.end(), 0.0L);
        std::fill(T1.begin(), T1.end(), 0.0L);
        T0[0] = 1.0L;  // T_0
        if (P > 1) T1[1] = 1.0L;  // T_1
        for (int j = 0; j < P; ++j) {
            const std::vector<long double> &Tj = (j == 0) ? T0 : T1;
            for (int k = 0; k < P; ++k) mono[k] += cheb[j] * Tj[k];
            if (j >= 1) {  // T_{j+1} = 2 y T_j - T_{j-1} into Tm, then shift
                for (int k = 0; k < P; ++k) Tm[k] = (k > 0 ? 2.0L * T1[k - 1] : 0.0L) - T0[k];
                T0 = T1;
                T1 = Tm;
            }
        }
        for (int k = 0; k < NE; ++k) c[a * P + k] = (double)mono[2 * k];
        for (int k = 0; k < NO; ++k) c[a * P + NE + k] = (double)mono[2 * k + 1];
    }
}

// psi_hat(k) = int psi(x) cos(k x) dx with psi(x) = exp(beta (sqrt(1 - (x/alpha)^2) - 1)),
// |x| < alpha = w pi / n.  With x = alpha sin(theta) the integrand is smooth:
// alpha int_{-pi/2}^{pi/2} exp(beta (cos theta - 1)) cos(k alpha sin theta) cos theta dtheta.
std::vector<double> kernel_ft(int N, int w, double beta, int n)
{
    std::vector<double> gx, gw;
    gauss_legendre(256, gx, gw);
    const double alpha = w * kPi / n;
    std::vector<double> out(N + 1);
    for (int k = 0; k <= N; ++k) {
        double acc = 0.0;
        for (size_t t = 0; t < gx.size(); ++t) {
            double th = 0.5 * kPi * gx[t];
            acc += gw[t] * std::exp(beta * (std::cos(th) - 1.0)) * std::cos(k * alpha * std::sin(th)) *
                   std::cos(th);
        }
        out[k] = alpha * 0.5 * kPi * acc;
    }
    return out;
}

void sphere_points(int d, int M, int kind, std::vector<double> &pts, std::vector<double> &wts)
{
    pts.assign((size_t)M * d, 0.0);
    if (d == 2) {
        for (int m = 0; m < M; ++m) {
            double th = 2.0 * kPi * m / M;
            pts[2 * m] = std::cos(th);
            pts[2 * m + 1] = std::sin(th);
        }
        wts.assign(M, 2.0 * kPi / M);
        return;
    }
    const double golden = kPi * (3.0 - std::sqrt(5.0));
    if (kind == PG_SPHERE_FIBONACCI) {
        for (int m = 0; m < M; ++m) {
            double z = 1.0 - (2.0 * m + 1.0) / M;
            double rho = std::sqrt(1.0 - z * z);
            pts[3 * m] = rho * std::cos(m * golden);
            pts[3 * m + 1] = rho * std::sin(m * golden);
            pts[3 * m + 2] = z;
        }
    } else {
        const int h = M / 2;
        for (int m = 0; m < h; ++m) {
            double z = 1.0 - (2.0 * m + 1.0) / h;
            double rho = std::sqrt(1.0 - z * z);
            double x = rho * std::cos(m * golden), y = rho * std::sin(m * golden);
            pts[3 * m] = x;
            pts[3 * m + 1] = y;
            pts[3 * m + 2] = z;
            pts[3 * (m + h)] = -x;
            pts[3 * (m + h) + 1] = -y;
            pts[3 * (m + h) + 2] = -z;
        }
    }
    wts.assign(M, 4.0 * kPi / M);
}

std::vector<unsigned> axis_orbits(int N)
{
    std::vector<unsigned> t;
    for (int i = 0; 2 * i <= N - 1; ++i)
        for (int j = i; i + j <= N - 1; ++j) t.push_back((unsigned)i | (unsigned)j << 16);
    return t;
}

double map_v(double phi, double S, int r)
{
    // xi = -cos(phi); r = 1: v = S xi / sqrt(1 - xi^2) = -S cot(phi); r = 0: v = S atanh(xi) = S ln tan(phi/2)
    if (r == 1) return -S * std::cos(phi) / std::sin(phi);
    return S * std::log(std::tan(0.5 * phi));
}

NodeTables node_tables(int N, double S, int r)
{
    NodeTables t;
    t.R.assign((size_t)N * (N + 1), 0.0);
    t.E.assign((size_t)(N + 1) * N, 0.0);
    t.scale_a.assign(N, 0.0);
    t.inv_mu2.assign(N, 0.0);
    t.v.assign(N, 0.0);
    const double wnode = kPi / (N + 1);
    for (int i = 0; i < N; ++i) {
        const double phi = kPi * (i + 1) / (N + 1);
        // The nodes of the upper half are the exact mirror images of those of the lower half, which the
        // kernels' classes of mirrored node pairs rely on.  Evaluated at phi > pi/2 they would not be: the
        // rounding of phi moves sin(phi) by up to 1e-14 of itself near pi.
        const int low = std::min(i, N - 1 - i);
        const double phl = kPi * (low + 1) / (N + 1);
        const double mu2 = ipow(std::sin(phl), 1 + r) / S;
        t.scale_a[i] = wnode * mu2;
        t.inv_mu2[i] = 1.0 / mu2;
        t.v[i] = (2 * i == N - 1) ? 0.0 : (i == low) ? map_v(phl, S, r) : -map_v(phl, S, r);
        for (int k = 0; k <= N; ++k) {
            const double tk = std::cos(k * (kPi - phi)) / std::sqrt(k == 0 ? kPi : 0.5 * kPi);
            t.R[(size_t)i * (N + 1) + k] = tk;
            t.E[(size_t)k * N + i] = tk;
        }
    }
    return t;
}

std::vector<double> transform_matrix(int N, int n, int w, double beta)
{
    const int nf = n / 2 + 1;
    std::vector<double> ph = kernel_ft(N, w, beta, n);
    std::vector<double> D((size_t)(N + 1) * nf);
    for (int k = 0; k <= N; ++k) {
        const double ck = std::sqrt(k == 0 ? kPi : 0.5 * kPi);
        for (int g = 0; g < nf; ++g) {
            const long long kg = ((long long)k * g) % n;
            D[(size_t)k * nf + g] = (2.0 * kPi / n) * std::cos(2.0 * kPi * (double)kg / n) / (ck * ph[k]);
        }
    }
    return D;
}

pgb::Dims3 dims_of(int d, int a, int b, int c)
{
    pgb::Dims3 x;
    if (d == 2) {
        x.e[0] = 1;
        x.e[1] = b;
        x.e[2] = c;
    } else {
        x.e[0] = a;
        x.e[1] = b;
        x.e[2] = c;
    }
    return x;
}

int batch_block_threads(int d, bool f32, int ask, int automatic, size_t tile, size_t limit)
{
    const int max_threads = f32 ? pgb::kBatchThreadsF32 : pgb::kMaxThreadsF64;
    auto need = [&](int threads) { return tile + (f32 ? pgb::spread_queue_bytes(threads, d, true) : 0); };
    if (ask > 0 && f32 && tile + (size_t)ask * 4 * (2 * d + 1) > limit) return 0;
    int threads = ask > 0 ? std::min(ask, max_threads) : automatic;
    while (threads > 32 && need(threads) > limit) threads -= 32;
    return need(threads) <= limit ? threads : 0;
}

int spread_shape(const SpreadShapeIn &in, SpreadShape &out)
{
    const int d = in.d, N = in.N, nf = in.nf;
    const bool f32 = in.f32;
    const size_t elem = f32 ? 4 : 12;  // 32-bit words per cell: FP32 one, FP64 three
    // block tiles: rows of (nf^(d-2) x tile_cols) cells, the last axis padded with unfolded columns (FP64 3D: not)
    const size_t plane = (size_t)ipow(nf, d - 2) * pgb::tile_cols(nf, in.w, d, f32);
    // leave room for the kernels' static shared memory (FP64: the kernel polynomial)
    // (and 16 bytes for rounding the tile up to 16 bytes)
    const size_t max_smem = in.smem_block - 1024 - 16 - (f32 ? 0 : sizeof(double) * pgb::kPolyCoefF64);
    const int max_threads = f32 ? pgb::kMaxThreadsF32 : pgb::kMaxThreadsF64;
    const int accept_threads = pgb::accept_threads(d, f32);
    if (in.ask_threads > accept_threads || (in.ask_threads > 0 && in.ask_threads % 32))
        return set_error(PG_ERR_ARG, "spread_threads must be a multiple of 32 and <= %d", accept_threads);
    int ask_threads = std::min(in.ask_threads, max_threads);  // <= 0: chosen here
    const long long nclass = (long long)ipow((double)pgb::unordered_pairs(N), d);
    auto queue_bytes = [&](int threads) { return pgb::spread_queue_bytes(threads, d, f32, in.ang); };
    // threads whose queues fit beside a tile
    auto room = [&](size_t tile) { return tile < max_smem ? 32 * (int)((max_smem - tile) / queue_bytes(32)) : 0; };
    // small one-slab plans: blocks no larger than it takes for every SM to have one (each thread then owns
    // one item; 2D Maxwell N = 16 has one for each of 145 blocks of 384)
    auto small_block = [&](long long items) {
        const long long per_block = (items + in.sms - 1) / in.sms;
        return (int)std::min<long long>((std::max<long long>(per_block, 64) + 31) / 32 * 32, max_threads);
    };
    // FP32 2D: with fewer classes than threads, the classes' quads are cut into shares, so that there is
    // an item per thread (2D N = 16, M = 8: 18,496 classes of 3 quads, spreading 41 -> 31 us).  With
    // more classes (N = 32: 2.9 per thread) the repeated class tests cost what the fuller rounds gain.
    int nsplit = 1;
    if (f32 && d == 2)
        nsplit = (int)std::max<long long>(1, std::min<long long>(in.M / 4 + 1, (long long)in.sms * max_threads / nclass));

    int rows_fit = (int)std::min<size_t>(nf, max_smem / (plane * elem));
    const size_t whole = pgb::tile_bytes((size_t)nf * plane, f32);
    if (rows_fit == nf && f32 && ask_threads <= 0) {
        // A grid that nearly fills one block leaves room for the queues of a few warps only; two slabs, which
        // generate every point twice, are then faster.  One slab (its threads) against two, ms:
        //   2D w = 6, M = 8:   N = 114 (320) 3.28 / 3.54   N = 115 (256) 3.60 / 3.47   N = 116 (160) 5.22 / 3.52
        //   2D w = 6, M = 32:  N = 114 (320) 8.78 / 9.28   N = 115 (256) 9.29 / 8.96
        //   2D w = 8, M = 8:   N = 113 (384) 3.90 / 4.75   N = 114 (288) 4.73 / 4.51
        //   2D angular, M = 8: N = 112 (352) 3.45 / 3.91   N = 113 (288) 4.22 / 4.17
        //   3D w = 6:          N = 16 angular (512) 6.91 / 8.03   N = 17 (256) 3.04 / 2.36
        //   3D w = 8, sigma = 1.5: N = 22 (352) 11.1 / 11.0
        // (One slab spread point by point without queues, 640 threads: 3.15 at N = 115 and 3.79 at N = 117 where two
        // slabs take 3.47 and 3.78 ms, but N = 117 10.4 against 9.9 at M = 32, 9.98 against 8.84 angular, and 3D N = 17
        // 4.6 against 2.4.)
        if (room(whole) < std::min(small_block(nclass * nsplit), d == 3 ? 384 : 320)) rows_fit = nf - 1;
    }
    size_t qbytes = 0;
    if (rows_fit < nf) {
        // slabbed grid: the warps' queues (one block per SM) share the block's shared memory with the slab.
        // FP32: at least 384 threads, and as many as the fewest slabs that leave room for those allow
        // (a point is generated once per slab and its rows straddle two now and then)
        auto fit = [&](int thr) {
            qbytes = queue_bytes(thr);
            return (max_smem > qbytes) ? (int)std::min<size_t>(nf, (max_smem - qbytes) / (plane * elem)) : 0;
        };
        rows_fit = fit((ask_threads > 0) ? ask_threads : f32 ? 384 : max_threads);
        if (rows_fit < 1 && f32) {
            // a plane that leaves little room: the block that still fits, at worst one warp with half of the kilobyte
            // left for static shared memory (the FP32 kernels have 16 bytes)
            ask_threads = (ask_threads > 0) ? std::min(ask_threads, 128) : 128;
            while ((rows_fit = fit(ask_threads)) < 1 && ask_threads > 32) ask_threads -= 32;
            if (rows_fit < 1 && queue_bytes(32) + plane * elem <= max_smem + 512) rows_fit = 1;
        }
    }
    if (rows_fit < 1) return set_error(PG_ERR_ARG, "folded grid plane of %zu cells does not fit shared memory", plane);
    out.nslab = (nf + rows_fit - 1) / rows_fit;
    out.rows_per_slab = (nf + out.nslab - 1) / out.nslab;
    out.nslab = (nf + out.rows_per_slab - 1) / out.rows_per_slab;  // no empty trailing slab
    out.tile_cells = (long long)out.rows_per_slab * (long long)plane;
    const size_t tile = pgb::tile_bytes((size_t)out.tile_cells, f32);
    out.smem = tile;
    out.queued = 0;
    out.nsplit = 1;
    out.nitem = 0;
    long long items = nclass;
    // FP32: one block per SM (measured fastest; more, smaller blocks multiply the tile clears and flushes)
    int per_sm = 1;
    if (out.nslab > 1) {
        out.threads = ask_threads > 0 ? ask_threads : f32 ? std::min(max_threads, room(tile)) : max_threads;
        out.smem += queue_bytes(out.threads);
        if (ask_threads > 0 || !f32)
            per_sm = (int)(in.smem_sm / (out.smem + 1024 + in.smem_reserved));
    } else if (f32) {
        // the warps' queues follow the tile (2D: large quads; 3D: the points that add something)
        out.threads = ask_threads > 0 ? ask_threads : std::min(small_block(nclass * nsplit), room(whole));
        if (ask_threads > 0) per_sm = (int)(in.smem_sm / (tile + 1024 + in.smem_reserved));
        out.queued = room(whole) >= out.threads;  // (block sizes asked for may not fit: point by point, whole classes)
        if (out.queued) {
            out.smem += queue_bytes(out.threads);
            out.nsplit = nsplit;
            items = nclass * nsplit;
        }
    } else {
        // about 1024 resident threads per SM, small plans fewer
        per_sm = std::max(1, (int)(in.smem_sm / (tile + 1024 + in.smem_reserved)));
        out.threads = ask_threads > 0 ? ask_threads
                                      : std::min(std::max(128, std::min(max_threads, (1024 / per_sm) / 32 * 32)),
                                                 small_block(nclass));
        // 2D: quads of mirrored classes, numbered in 32 bits, 4 bytes of queue per thread
        const long long norb = (long long)axis_orbits(N).size();
        long long nitem = norb * norb * (in.M / 4 + 1);
        const long long all = (long long)in.sms * max_threads;
        // (two sphere points, and classes for two thirds of the threads at most: a class' two points at once are
        // faster, w = 14 N = 16 131 us, by quads 177; N = 20 197 / 332)
        if (d == 2 && nitem < (1ll << 32) && (in.M > 2 || nclass > all * 2 / 3)) {
            // With fewer items than threads the launch waits for the 16 points that a thread adds one after the
            // other: shares of 4 points, or of 1, which evaluate the axes 3 or 8 times as often.  us, whole / 4 / 16
            // shares: N = 8, M = 6, w = 14 276 / - / 84; N = 12, M = 8, w = 10 185 / 140 / 171; N = 14, M = 6, w = 14
            // 274 / 212 / 231; logarithmic map, w = 10: N = 15, M = 14 239 / 200, M = 22 (4 shares are 1.3 per
            // thread) 301 / 361.  (M = 4: 8 points in series; N = 14, w = 14 189 / 212 / 207.)
            const int share = 16 * nitem <= all * 3 / 4 ? 16 : (in.M > 4 && 4 * nitem <= all) ? 4 : 1;
            nitem *= share;
            int threads = ask_threads > 0 ? ask_threads : small_block(nitem);
            if (ask_threads <= 0)
                while (threads > 128 && tile + (size_t)threads * 4 > max_smem) threads -= 128;
            if (tile + (size_t)threads * 4 <= max_smem) {
                out.queued = 1;
                out.threads = threads;
                out.smem += (size_t)threads * 4;
                out.nitem = items = nitem;
                out.nsplit = share;
                if (ask_threads <= 0) per_sm = 1;
            }
        }
    }
    per_sm = std::min(per_sm, in.sm_threads / out.threads);
    if (in.ask_per_sm > 0) per_sm = std::min(per_sm, in.ask_per_sm);
    per_sm = std::max(per_sm, 1);
    long long blocks = (long long)in.sms * per_sm;
    blocks = std::max<long long>(blocks / out.nslab, 1) * out.nslab;
    blocks = std::min(blocks, ((items + out.threads - 1) / out.threads) * out.nslab);
    out.blocks = (int)blocks;
    // the pair schedule permutes thread starts by a multiplier prime to every smaller count
    if ((blocks / out.nslab) * out.threads >= 1000003)
        return set_error(PG_ERR_ARG, "spreading launch of %lld threads per slab exceeds the pair schedule's range",
                         (blocks / out.nslab) * out.threads);
    return PG_OK;
}

int dev_alloc(pg_boltz_plan_t *p, void **ptr, size_t bytes)
{
    *ptr = nullptr;
    int c = g_fail_alloc_countdown.load();
    if (c > 0) {
        if (g_fail_alloc_countdown.fetch_sub(1) == 1)
            return set_error(PG_ERR_NOMEM, "device allocation of %zu bytes failed (injected)", bytes);
    }
    cudaError_t e = cudaMalloc(ptr, bytes < 16 ? 16 : bytes);
    if (e != cudaSuccess) {
        *ptr = nullptr;
        cudaGetLastError();
        return set_error(e == cudaErrorMemoryAllocation ? PG_ERR_NOMEM : PG_ERR_CUDA,
                         "cudaMalloc(%zu) failed: %s", bytes, cudaGetErrorString(e));
    }
    p->allocs.push_back(*ptr);
    p->device_bytes += bytes;
    return PG_OK;
}

int upload_bytes(pg_boltz_plan_t *p, void **dst, const void *src, size_t bytes)
{
    int rc = dev_alloc(p, dst, bytes);
    if (rc) return rc;
    cudaError_t e = cudaMemcpy(*dst, src, bytes, cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return set_error(PG_ERR_CUDA, "upload failed: %s", cudaGetErrorString(e));
    return PG_OK;
}

void free_plan(pg_boltz_plan_t *p)
{
    if (!p) return;
    for (cudaEvent_t &e : p->ev)
        if (e) cudaEventDestroy(e);
    if (p->batch) pg_free_batch(p->batch);
    if (p->rk_exec) cudaGraphExecDestroy(p->rk_exec);
    if (p->rk_graph) cudaGraphDestroy(p->rk_graph);
    if (p->rk_cap_stream) cudaStreamDestroy(p->rk_cap_stream);
    for (void *q : p->allocs) cudaFree(q);
    p->allocs.clear();
    delete p;
}

}  // namespace pgbh

int pgb::record_error(int code, const char *msg) { return pgbh::set_error(code, "%s", msg); }

PG_API const char *pg_boltz_last_error(void) { return g_last_error.c_str(); }

PG_API void pg_boltz_debug_fail_alloc(int countdown) { g_fail_alloc_countdown.store(countdown > 0 ? countdown : 0); }
