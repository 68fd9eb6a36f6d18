// tbs_plan.cu -- plan-time tables: FFT twiddles and the spectrum of the
// cell-averaged free-space Green's function.
//
// The operator G of arxiv 2507.13754 (Section 2.2: G = F^-1 g~ F below
// Eq. 17) is realised with the free-space Green's function of Eq. 16 at
// epsilon -> 0, g(r) = (i/4) H0^(1)(k0 r) = (i/4) J0(k0 r) - (1/4) Y0(k0 r),
// averaged over each cell:
//     Gc[d] = (1/dx^2) * integral over cell d of g(|r|) d^2r.
// Everything here runs in FP64 (Bessel functions are CUDA's j0/j1/y0/y1);
// only the final spectrum is rounded to complex64.
//
//  * The self cell: subtract the logarithm.  Near r = 0,
//    Y0(z) = (2/pi)(ln(z/2) + gamma) J0(z) + O(z^2), so
//    g_s(r) = g(r) + ln(r)/(2 pi) is continuous; its mean is integrated in
//    polar coordinates over the 8 triangles of the square (24 x 24 points),
//    and the mean of ln r over a square of side h has the closed form
//    ln(h/2) + (ln 2 - 3 + pi/2)/2.
//  * 1 <= max(|a|,|b|) <= 3: 16 x 16 tensor Gauss-Legendre; up to 7 (and
//    everywhere when k0 dx > 2 or < 1e-9): 6 x 6.
//  * Farther cells: Graf's addition theorem about the cell's centre (r,
//    theta).  The square's symmetry leaves the orders m = 0, 4, 8, 12:
//        Gc = (i/4) [c_0 H_0(k0 r) + 2 sum c_m H_m(k0 r) cos(m theta)],
//        c_m = (1/h^2) * integral over the cell of J_m(k0 rho) cos(m phi).
//    For r >= 8 cells and k0 dx <= 2 the first order left out (16) is below
//    1e-15 of g.  The radial factors are interpolated: polynomials on
//    intervals of at most one cell and k0 * length <= 1, of degree 10, 10,
//    7 and 4, fitted at 12 Chebyshev nodes (H_m there by upward recurrence
//    from J0, J1, Y0, Y1: the error in J_m grows like Y_m, whose share of
//    the sum c_m bounds).  Emulated on the host against 30 digits, cells
//    from 8 to 2500 away are within 5e-15 for k0 dx from 1e-9 to 2; the
//    6 x 6 rule's worst there is 3.4e-14 (at k0 dx = 2).
//
// FP64 arithmetic bounds the build: this GPU issues about two FP64
// multiply-adds per SM and clock.  A direct 6 x 6 rule takes 36 pairs of
// Bessel functions per cell (41 ms at N = 2048), the modes about 110
// multiply-adds (measured figures at build_ghat).
//
// The table is even in both axes and symmetric under transposition, and so
// is its spectrum: the row transforms cover the N rows 0 .. N-1 (each
// mirrored into M points as it is read), the column transforms the columns
// kx = 0 .. M/2.  The result, scaled by dx^2/M^2, is the stored quadrant
// 0 <= kx, ky <= M/2.
#include "tbs_fft.cuh"
#include "tbs_internal.h"

#include <math.h>
#include <stdio.h>
#include <vector>

namespace tbs {

#define TBS_NQ_SELF 24
#define TBS_NQ_NEAR 16
#define TBS_NQ_FAR 6

constexpr int FIT_NODES = 12;             // Chebyshev nodes per interval
constexpr int NEAR_CELLS = 8;             // max(|a|, |b|) below: direct quadrature
// k0 dx for which the modes serve; below, Y_12 and the recurrence that forms it
// leave the range of FP64 (from 3e-26 on) and nobody samples that finely
constexpr double MODES_MIN_KH = 1e-9, MODES_MAX_KH = 2.0;
// polynomial degree of the radial factor of order 4 q, and the first of its
// coefficients (those of its real part, then of its imaginary part)
__host__ __device__ constexpr int fit_deg(int q) { return q < 2 ? 10 : q == 2 ? 7 : 4; }
__host__ __device__ constexpr int fit_off(int q) { return q == 0 ? 0 : q == 1 ? 22 : q == 2 ? 44 : 60; }
constexpr int FIT_COEFS = 70;
// first row of a degree's conversion in FitRule::mono
__host__ __device__ constexpr int fit_row(int q) { return q < 2 ? 0 : q == 2 ? 11 : 19; }
constexpr int FIT_ROWS = 24;

// The host-built rules, passed to the kernels by value.
struct NearRules {
    double xs[TBS_NQ_SELF], ws[TBS_NQ_SELF], xn[TBS_NQ_NEAR], wn[TBS_NQ_NEAR], xf[TBS_NQ_FAR], wf[TBS_NQ_FAR];
};
struct FitRule {
    double mono[FIT_ROWS][FIT_NODES];     // [fit_row + power][node]: values at the nodes -> monomial coefficients
    double node[FIT_NODES];               // in (0, 1), from the interval's start
    double c[4];                          // c_0, 2 c_4, 2 c_8, 2 c_12
};

// Gauss-Legendre rule on [-1, 1] by Newton's method on the Legendre
// polynomial, evaluated with Bonnet's recurrence; initial guesses from the
// asymptotic formula cos(pi (4i + 3) / (4n + 2)).
static void gauss_legendre_rule(int n, double *x, double *w) {
    for (int i = 0; i < n; i++) {
        double z = cos(M_PI * (4.0 * i + 3.0) / (4.0 * n + 2.0));
        double dp = 1.0;
        for (int it = 0; it < 100; it++) {
            double pkm1 = 1.0, pk = z;  // P_0, P_1
            for (int k = 1; k < n; k++) {
                const double pkp1 = ((2.0 * k + 1.0) * z * pk - k * pkm1) / (k + 1.0);
                pkm1 = pk;
                pk = pkp1;
            }
            if (n == 1) { pk = z; pkm1 = 1.0; }
            dp = n * (pkm1 - z * pk) / (1.0 - z * z);
            const double step = pk / dp;
            z -= step;
            if (fabs(step) < 1e-15) {
                // refresh the derivative at the final node
                double a = 1.0, b = z;
                for (int k = 1; k < n; k++) {
                    const double c = ((2.0 * k + 1.0) * z * b - k * a) / (k + 1.0);
                    a = b;
                    b = c;
                }
                if (n == 1) { b = z; a = 1.0; }
                dp = n * (a - z * b) / (1.0 - z * z);
                break;
            }
        }
        x[i] = z;
        w[i] = 2.0 / ((1.0 - z * z) * dp * dp);
    }
}

__device__ __forceinline__ double2 green_fp64(double k0, double r) {
    const double z = k0 * r;
    return make_double2(-0.25 * y0(z), 0.25 * j0(z));
}

// Sum of v over the block's 256 threads, valid in thread 0.
__device__ __forceinline__ double2 block_sum(double2 v, double2 *sh) {
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
        v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
        v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
    }
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0)
        for (int w = 1; w < 8; w++) {
            v.x += sh[w].x;
            v.y += sh[w].y;
        }
    return v;
}

// Cells by quadrature, one block per cell and one thread per point: the
// cells a, b < side (the self cell among them).  One thread per cell had
// left the self cell's 576 points to a single thread: 3.6 ms at any N.
__global__ void __launch_bounds__(256) green_near_kernel(int n, double k0, double dx,
                                                         const __grid_constant__ NearRules q,
                                                         double2 *__restrict__ gc) {
    __shared__ double2 sh[8];
    const int a = blockIdx.x, b = blockIdx.y;
    double2 s = make_double2(0.0, 0.0);
    if (a == 0 && b == 0) {
        for (int i = threadIdx.x; i < TBS_NQ_SELF * TBS_NQ_SELF; i += 256) {
            const int p = i / TBS_NQ_SELF, t = i % TBS_NQ_SELF;
            const double th = (q.xs[p] + 1.0) * (M_PI / 8.0);
            const double R = 0.5 * dx / cos(th);
            const double r = 0.5 * R * (q.xs[t] + 1.0);
            const double w = q.ws[p] * (M_PI / 8.0) * 0.5 * R * q.ws[t] * r;
            const double2 g = green_fp64(k0, r);
            s.x += w * (g.x + log(r) / (2.0 * M_PI));
            s.y += w * g.y;
        }
    } else {
        const bool near = (a <= 3 && b <= 3);
        const int nq = near ? TBS_NQ_NEAR : TBS_NQ_FAR;
        const double *gx = near ? q.xn : q.xf;
        const double *gw = near ? q.wn : q.wf;
        const int i = threadIdx.x / nq, j = threadIdx.x % nq;
        if (i < nq) {
            const double px = (a + 0.5 * gx[i]) * dx, py = (b + 0.5 * gx[j]) * dx;
            const double2 g = green_fp64(k0, sqrt(px * px + py * py));
            s.x = 0.25 * gw[i] * gw[j] * g.x;
            s.y = 0.25 * gw[i] * gw[j] * g.y;
        }
    }
    s = block_sum(s, sh);
    if (threadIdx.x == 0) {
        if (a == 0 && b == 0) {
            const double mean_ln = log(0.5 * dx) + 0.5 * (log(2.0) - 3.0 + 0.5 * M_PI);
            s.x = -mean_ln / (2.0 * M_PI) + 8.0 * s.x / (dx * dx);
            s.y = 8.0 * s.y / (dx * dx);
        }
        gc[(size_t)b * n + a] = s;
    }
}

// Cells outside the near square by the 6 x 6 rule, one thread per cell
// (k0 dx outside MODES_MIN_KH .. MODES_MAX_KH; above: fewer than about three
// points per wavelength).
__global__ void __launch_bounds__(128) green_direct_kernel(int n, double k0, double dx,
                                                           const __grid_constant__ NearRules q,
                                                           double2 *__restrict__ gc) {
    const int a = blockIdx.x * blockDim.x + threadIdx.x, b = blockIdx.y;
    if (a >= n || (a < NEAR_CELLS && b < NEAR_CELLS)) return;
    double2 s = make_double2(0.0, 0.0);
    for (int i = 0; i < TBS_NQ_FAR; i++) {
        const double px = (a + 0.5 * q.xf[i]) * dx;
        for (int j = 0; j < TBS_NQ_FAR; j++) {
            const double py = (b + 0.5 * q.xf[j]) * dx, w = 0.25 * q.wf[i] * q.wf[j];
            const double2 g = green_fp64(k0, sqrt(px * px + py * py));
            s.x = fma(w, g.x, s.x);
            s.y = fma(w, g.y, s.y);
        }
    }
    gc[(size_t)b * n + a] = s;
}

// Polynomials of the radial factors: block j fits the interval
// [NEAR + j / per_cell, NEAR + (j + 1) / per_cell) in cells of r; coefficient
// c of interval j at coef[c * count + j] (neighbouring cells of a row, whose
// intervals are neighbours, read neighbouring words).
__global__ void __launch_bounds__(96) green_fit_kernel(int count, int per_cell, double kh,
                                                       const __grid_constant__ FitRule f, double *__restrict__ coef) {
    __shared__ double v[8][FIT_NODES];
    const int j = blockIdx.x;
    if (threadIdx.x < FIT_NODES) {
        const double z = kh * (NEAR_CELLS + (j + f.node[threadIdx.x]) / per_cell);
        double jm = j0(z), j1m = j1(z), ym = y0(z), y1m = y1(z);
        const double iz = 1.0 / z;
#pragma unroll
        for (int m = 0; m <= 12; m++) {  // jm, ym: order m; j1m, y1m: order m + 1
            if (m % 4 == 0) {
                v[m / 2][threadIdx.x] = -0.25 * f.c[m / 4] * ym;
                v[m / 2 + 1][threadIdx.x] = 0.25 * f.c[m / 4] * jm;
            }
            const double jn = fma(2.0 * (m + 1) * iz, j1m, -jm), yn = fma(2.0 * (m + 1) * iz, y1m, -ym);
            jm = j1m;
            ym = y1m;
            j1m = jn;
            y1m = yn;
        }
    }
    __syncthreads();
    const int comp = threadIdx.x / FIT_NODES, p = threadIdx.x % FIT_NODES;
    const int q = comp / 2, deg = fit_deg(q);
    if (p > deg) return;
    double s = 0.0;
    for (int i = 0; i < FIT_NODES; i++) s = fma(f.mono[fit_row(q) + p][i], v[comp][i], s);
    coef[(size_t)(fit_off(q) + (comp & 1) * (deg + 1) + p) * count + j] = s;
}

// Far cells: tiles of 32 x 32 with bx >= by, each also written transposed.
__global__ void __launch_bounds__(256) green_far_kernel(int n, int count, int per_cell,
                                                        const double *__restrict__ coef, double2 *__restrict__ gc) {
    if (blockIdx.x < blockIdx.y) return;
    __shared__ double2 tile[32][33];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int a0 = blockIdx.x * 32, b0 = blockIdx.y * 32;
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const int a = a0 + tx, b = b0 + ty + 8 * k;
        if (a >= n || b >= n || (a < NEAR_CELLS && b < NEAR_CELLS)) continue;
        const double a2 = (double)a * a, b2 = (double)b * b, r2 = a2 + b2;
        const double u = (sqrt(r2) - NEAR_CELLS) * per_cell;
        int j = (int)u;
        if (j > count - 1) j = count - 1;
        const double x = fma(2.0, u - j, -1.0);
        const double *c = coef + j;
        double f[8];
        auto poly = [&](auto dc, int o) {  // degree D, coefficients from o on
            constexpr int D = decltype(dc)::value;
            double v = __ldg(c + (size_t)(o + D) * count);
#pragma unroll
            for (int p = D - 1; p >= 0; p--) v = fma(v, x, __ldg(c + (size_t)(o + p) * count));
            return v;
        };
        static_for<4>([&](auto qc) {
            constexpr int q = decltype(qc)::value;
            using D = std::integral_constant<int, fit_deg(q)>;
            f[2 * q] = poly(D{}, fit_off(q));
            f[2 * q + 1] = poly(D{}, fit_off(q) + fit_deg(q) + 1);
        });
        // cos 4 theta = (a^4 - 6 a^2 b^2 + b^4) / r^4, then cos 8 and 12 theta
        const double c4 = 1.0 - 8.0 * a2 * b2 / (r2 * r2), c8 = fma(2.0 * c4, c4, -1.0),
                     c12 = c4 * fma(4.0 * c4, c4, -3.0);
        const double2 g = make_double2(fma(c12, f[6], fma(c8, f[4], fma(c4, f[2], f[0]))),
                                       fma(c12, f[7], fma(c8, f[5], fma(c4, f[3], f[1]))));
        gc[(size_t)b * n + a] = g;
        tile[ty + 8 * k][tx] = g;
    }
    if (blockIdx.x == blockIdx.y) return;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const int a = a0 + ty + 8 * k, b = b0 + tx;  // element (a, b) of the transposed tile
        if (a < n && b < n) gc[(size_t)a * n + b] = tile[tx][ty + 8 * k];
    }
}

__global__ void twiddle64_kernel(int M, double2 *__restrict__ tw) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= M) return;
    double s, c;
    sincospi(2.0 * (double)k / (double)M, &s, &c);
    tw[k] = make_double2(c, -s);  // exp(-2 pi i k / M)
}

__global__ void twiddle32_kernel(int M, const double2 *__restrict__ tw64, float2 *__restrict__ tw) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= M) return;
    tw[k] = make_float2((float)tw64[k].x, (float)tw64[k].y);
}

// (p, q) <- (p + w q, p - w q) in six FP64 instructions
__device__ __forceinline__ void bfly64(double2 &p, double2 &q, double2 w) {
    const double sx = fma(w.x, q.x, fma(-w.y, q.y, p.x)), sy = fma(w.x, q.y, fma(w.y, q.x, p.y));
    q = make_double2(fma(2.0, p.x, -sx), fma(2.0, p.y, -sy));
    p = make_double2(sx, sy);
}
__device__ __forceinline__ void bfly64(double2 &p, double2 &q) {
    const double2 s = make_double2(p.x + q.x, p.y + q.y);
    q = make_double2(p.x - q.x, p.y - q.y);
    p = s;
}

// Forward FFT of one even line per block: the n stored values x[0 .. n-1] of
// line l are mirrored into M points (x[M - j] = x[j], zero between; M >= 2n - 1)
// as they are read.  Radix-4 Stockham stages (a radix-2 one first when log2 M
// is odd) between two buffers in shared memory, the stage twiddles folded into
// the two-point butterflies: 24 FP64 instructions per radix-4 butterfly and
// 16 in the first stage, against 32 for plain radix-2 stages (FP64 issue
// bounds the kernel).  The lines are even, so the outputs k = 0 .. M/2 are all:
// FINAL = false writes them transposed, out[k][l] (row M/2 to `last`);
// FINAL = true writes them scaled and rounded, ghq[l][k].
template <bool FINAL>
__global__ void __launch_bounds__(512) fft64_even_kernel(int n, int M, const double2 *__restrict__ in,
                                                         const double2 *__restrict__ in_last,
                                                         const double2 *__restrict__ tw, double scale,
                                                         double2 *__restrict__ out, double2 *__restrict__ last,
                                                         float2 *__restrict__ ghq) {
    extern __shared__ double2 sh64[];
    double2 *src = sh64, *dst = sh64 + M;
    const int l = blockIdx.x, half = M / 2;
    const double2 *row = (FINAL && l == half) ? in_last : in + (size_t)l * n;
    for (int i = threadIdx.x; i <= half; i += blockDim.x) {
        const double2 v = i < n ? row[i] : make_double2(0.0, 0.0);
        src[i] = v;
        if (i > 0 && i < half) src[M - i] = v;
    }
    __syncthreads();
    int Ns = 1;
    if (__popc(M - 1) & 1) {  // log2 M odd
        for (int j = threadIdx.x; j < half; j += blockDim.x) {
            double2 p = src[j], q = src[j + half];
            bfly64(p, q);
            dst[2 * j] = p;
            dst[2 * j + 1] = q;
        }
        __syncthreads();
        double2 *t = src;
        src = dst;
        dst = t;
        Ns = 2;
    }
    const int quarter = M / 4;
    for (; Ns < M; Ns <<= 2) {
        for (int j = threadIdx.x; j < quarter; j += blockDim.x) {
            const int k = j & (Ns - 1);
            double2 x0 = src[j], x1 = src[j + quarter], x2 = src[j + 2 * quarter], x3 = src[j + 3 * quarter];
            if (Ns == 1) {
                bfly64(x0, x2);
                bfly64(x1, x3);
                bfly64(x0, x1);
                x3 = make_double2(x3.y, -x3.x);  // times -i
                bfly64(x2, x3);
            } else {
                const int e = k * (M / (4 * Ns));
                const double2 w1 = __ldg(tw + e), w2 = __ldg(tw + 2 * e);
                bfly64(x0, x2, w2);
                bfly64(x1, x3, w2);
                bfly64(x0, x1, w1);
                bfly64(x2, x3, make_double2(w1.y, -w1.x));  // -i w1
            }
            double2 *d = dst + (j - k) * 4 + k;
            d[0] = x0;
            d[Ns] = x2;
            d[2 * Ns] = x1;
            d[3 * Ns] = x3;
        }
        __syncthreads();
        double2 *t = src;
        src = dst;
        dst = t;
    }
    if constexpr (FINAL) {
        const int qsp = ghat_stride(M);
        for (int i = threadIdx.x; i < qsp; i += blockDim.x)  // the padding column is zero
            ghq[(size_t)l * qsp + i] = i <= half ? make_float2((float)(src[i].x * scale), (float)(src[i].y * scale))
                                                 : make_float2(0.f, 0.f);
    } else {
        for (int i = threadIdx.x; i <= half; i += blockDim.x) (i < half ? out + (size_t)i * n : last)[l] = src[i];
    }
}

cudaError_t build_twiddles(int M, float2 *tw, cudaStream_t s) {
    double2 *tw64 = nullptr;
    cudaError_t e = cudaMalloc(&tw64, sizeof(double2) * M);
    if (e != cudaSuccess) return e;
    twiddle64_kernel<<<(M + 255) / 256, 256, 0, s>>>(M, tw64);
    twiddle32_kernel<<<(M + 255) / 256, 256, 0, s>>>(M, tw64, tw);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFree(tw64);
    return e;
}

// Coefficients c_m of the square cell (host): 16 x 16 Gauss-Legendre on a
// quarter of it (the integrand is even in both axes).
static double cell_mode(int m, double kh, const double *x, const double *w) {
    double s = 0.0;
    for (int i = 0; i < TBS_NQ_NEAR; i++)
        for (int j = 0; j < TBS_NQ_NEAR; j++) {
            const double px = 0.25 * (x[i] + 1.0), py = 0.25 * (x[j] + 1.0);
            s += 0.25 * w[i] * w[j] * jn(m, kh * sqrt(px * px + py * py)) * cos(m * atan2(py, px));
        }
    return s;
}

// Chebyshev nodes on (0, 1) and, for each degree, the conversion from values
// there to the monomial coefficients in x = 2 u - 1 of the Chebyshev series
// cut at that degree.
static void fit_rule(FitRule &f) {
    double t[FIT_NODES][FIT_NODES] = {};  // Chebyshev polynomials' coefficients
    t[0][0] = 1.0;
    t[1][1] = 1.0;
    for (int d = 2; d < FIT_NODES; d++)
        for (int p = 0; p <= d; p++) t[d][p] = (p > 0 ? 2.0 * t[d - 1][p - 1] : 0.0) - t[d - 2][p];
    for (int i = 0; i < FIT_NODES; i++) {
        const double th = M_PI * (i + 0.5) / FIT_NODES;
        f.node[i] = 0.5 * (cos(th) + 1.0);
        for (int q = 1; q < 4; q++)
            for (int p = 0; p <= fit_deg(q); p++) {
                double s = 0.0;
                for (int d = p; d <= fit_deg(q); d++) s += (d == 0 ? 1.0 : 2.0) / FIT_NODES * cos(d * th) * t[d][p];
                f.mono[fit_row(q) + p][i] = s;
            }
    }
}

// ghq: the quadrant; work / work2: n * M float2 of scratch each, work3: n
// double2 (the plan's intermediates and source field, idle here).
// Creating a plan takes 2.25 ms at N = 2048 and 0.86 ms at N = 1024; with the
// 6 x 6 rule everywhere, full transforms and transposes of allocated M x M
// arrays it took 46.0 and 12.3 ms.
cudaError_t build_ghat(int n, int M, double k0, double dx, float2 *ghq, float2 *work, float2 *work2, float2 *work3,
                       cudaStream_t s) {
    NearRules q;
    gauss_legendre_rule(TBS_NQ_SELF, q.xs, q.ws);
    gauss_legendre_rule(TBS_NQ_NEAR, q.xn, q.wn);
    gauss_legendre_rule(TBS_NQ_FAR, q.xf, q.wf);
    double2 *gc = reinterpret_cast<double2 *>(work), *mid = reinterpret_cast<double2 *>(work2);
    double2 *last = reinterpret_cast<double2 *>(work3);
    const double kh = k0 * dx;
    const bool modes = kh >= MODES_MIN_KH && kh <= MODES_MAX_KH && n > NEAR_CELLS;
    const int per_cell = kh > 1.0 ? 2 : 1;  // k0 * interval length <= 1
    const int count = modes ? (int)ceil((sqrt(2.0) * (n - 1) - NEAR_CELLS) * per_cell) + 1 : 0;
    double *scratch = nullptr;  // twiddles, then the radial fits
    cudaError_t e = cudaMalloc(&scratch, sizeof(double2) * M + sizeof(double) * FIT_COEFS * (size_t)count);
    if (e != cudaSuccess) return e;
    double2 *tw64 = reinterpret_cast<double2 *>(scratch);
    double *coef = scratch + 2 * (size_t)M;
    twiddle64_kernel<<<(M + 255) / 256, 256, 0, s>>>(M, tw64);
    const int side = n < NEAR_CELLS ? n : NEAR_CELLS;
    green_near_kernel<<<dim3(side, side), 256, 0, s>>>(n, k0, dx, q, gc);
    if (modes) {
        FitRule f;
        fit_rule(f);
        for (int i = 0; i < 4; i++) f.c[i] = (i ? 2.0 : 1.0) * cell_mode(4 * i, kh, q.xn, q.wn);
        green_fit_kernel<<<count, 96, 0, s>>>(count, per_cell, kh, f, coef);
        const int t = (n + 31) / 32;
        green_far_kernel<<<dim3(t, t), 256, 0, s>>>(n, count, per_cell, coef, gc);
    } else if (n > NEAR_CELLS) {
        green_direct_kernel<<<dim3((n + 127) / 128, n), 128, 0, s>>>(n, k0, dx, q, gc);
    }
    const size_t sh = 2 * (size_t)M * sizeof(double2);
    const int thr = M / 4 < 32 ? 32 : M / 4 > 512 ? 512 : M / 4;
    e = cudaFuncSetAttribute(fft64_even_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(fft64_even_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh);
    if (e == cudaSuccess) {
        fft64_even_kernel<false><<<n, thr, sh, s>>>(n, M, gc, nullptr, tw64, 1.0, mid, last, nullptr);
        fft64_even_kernel<true><<<M / 2 + 1, thr, sh, s>>>(n, M, mid, last, tw64,
                                                           dx * dx / ((double)M * (double)M), nullptr, nullptr, ghq);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFree(scratch);
    return e;
}

}  // namespace tbs
