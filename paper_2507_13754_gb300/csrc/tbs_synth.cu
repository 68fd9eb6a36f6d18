// tbs_synth.cu -- broadband synthesis: the time signal at a lattice of
// receivers from a set of single-frequency fields (one per frequency of a
// sweep, each on its own grid over the same physical domain):
//     s(X, t) = sum_k w_k psi_k(X) exp(-2 pi i f_k t)
// (e^{-i omega t} convention of the outgoing Green's function, Section 2.2).
//
// One block takes SY_RB receivers of one right-hand side and SY_THREADS time
// samples: it first gathers the weighted bilinear samples w_k psi_k(X_r) of
// its receivers into shared memory, then each thread produces its time
// sample, forming each phase factor once for all SY_RB receivers.  Phases f_k
// t_j are reduced modulo one cycle beyond FP32 (f t reaches thousands of
// cycles), the rest is FP32.  Frequencies go in chunks of SY_CHUNK per launch
// (the per-frequency table rides in the kernel parameters, so the call
// allocates nothing); later chunks add to the output.
#include "tbs.h"
#include "tbs_internal.h"

#include <math.h>
#include <stdio.h>
#include <string.h>

namespace {

constexpr int SY_CHUNK = 64;     // frequencies per launch
constexpr int SY_RB = 16;        // receivers per block
constexpr int SY_THREADS = 256;

struct SynthArgs {
    const float2 *field[SY_CHUNK];
    double inv_dx[SY_CHUNK];
    double f[SY_CHUNK];
    float w[SY_CHUNK];
    int n[SY_CHUNK];
    int count;       // frequencies in this chunk
    int accumulate;  // add to out (chunks after the first)
    int nx, ny, n_t;
    double x0, y0, sx, sy, t0, dt;
    float2 *out;
};
static_assert(sizeof(SynthArgs) <= 4000, "kernel parameter space");

// fractional cell index of coordinate p on a grid of n cell centres i * dx,
// clamped to [0, n - 1]; i0 <= n - 2 so that i0 + 1 is a cell too.  (Times
// 1/dx: the weights are continuous across cells, and an FP64 division is some
// thirty of the few FP64 instructions per cycle that the GPU has.)
__device__ __forceinline__ void cell_of(double p, double inv_dx, int n, int &i0, float &fr) {
    const double u = fmin(fmax(p * inv_dx, 0.0), (double)(n - 1));
    int i = (int)floor(u);
    if (i > n - 2) i = n - 2;
    i0 = i;
    fr = (float)(u - (double)i);
}

// One block: SY_RB receivers of one RHS, SY_THREADS times (one per thread);
// blockIdx = (receivers, RHS, times).  Per frequency a thread forms one phase
// and adds SY_RB products, so the phases' cost is spread over SY_RB receivers.
// FAST: every |f t| is below 2^16 cycles, and the phase is taken modulo one
// cycle in pairs of FP32 (f and t split in two) instead of three FP64
// instructions per (time, frequency), which bounded the kernel.  The part of
// the phase that FP32 drops is kept and turns the sine and cosine: with it the
// phase is within 6e-10 cycles over that range (rounded to FP32, as after the
// FP64 reduction: 1.5e-8), the factor within 8.2e-8 (1.35e-7).  A call with 512
// receivers, 4 RHS, 256 frequencies and 672 times: 492 us in FP64, 237 us here.
template <bool FAST>
__global__ void __launch_bounds__(SY_THREADS) synth_kernel(const __grid_constant__ SynthArgs a) {
    __shared__ float2 A[SY_CHUNK][SY_RB];
    __shared__ float2 fs[SY_CHUNK];  // FAST: f as an FP32 pair
    const int nr = a.nx * a.ny;
    const int r0 = blockIdx.x * SY_RB;
    const int rhs = blockIdx.y;
    for (int idx = threadIdx.x; idx < SY_RB * a.count; idx += SY_THREADS) {
        const int rr = idx % SY_RB, k = idx / SY_RB;
        const int r = r0 + rr;
        float2 s = make_float2(0.f, 0.f);
        if (r < nr) {
            const int n = a.n[k];
            int i0, j0;
            float fx, fy;
            cell_of(a.x0 + (double)(r % a.nx) * a.sx, a.inv_dx[k], n, i0, fx);
            cell_of(a.y0 + (double)(r / a.nx) * a.sy, a.inv_dx[k], n, j0, fy);
            const float2 *p = a.field[k] + ((size_t)rhs * n + j0) * n + i0;
            const float2 p00 = p[0], p01 = p[1], p10 = p[n], p11 = p[n + 1];
            const float ax = 1.f - fx, ay = 1.f - fy;
            const float re = ay * (ax * p00.x + fx * p01.x) + fy * (ax * p10.x + fx * p11.x);
            const float im = ay * (ax * p00.y + fx * p01.y) + fy * (ax * p10.y + fx * p11.y);
            s = make_float2(a.w[k] * re, a.w[k] * im);
        }
        A[k][rr] = s;
    }
    for (int k = threadIdx.x; FAST && k < a.count; k += SY_THREADS) {
        const float hi = (float)a.f[k];
        fs[k] = make_float2(hi, (float)(a.f[k] - (double)hi));
    }
    __syncthreads();
    for (long long jj = (long long)blockIdx.z * SY_THREADS + threadIdx.x; jj < a.n_t;
         jj += (long long)gridDim.z * SY_THREADS) {
        const int j = (int)jj;
        const double t = a.t0 + (double)j * a.dt;
        const float th = (float)t, tl = (float)(t - (double)th);
        float2 acc[SY_RB];
#pragma unroll
        for (int rr = 0; rr < SY_RB; rr++) acc[rr] = make_float2(0.f, 0.f);
        for (int k = 0; k < a.count; k++) {
            float sn, cs;  // exp(-2 pi i f t) = cs - i sn
            if constexpr (FAST) {
                const float2 f = fs[k];
                const float p = f.x * th;
                const float e = fmaf(f.x, th, -p) + fmaf(f.x, tl, f.y * th);  // f t - p
                const float r = p - rintf(p);                                 // exact
                const float q = r + e;
                sincospif(2.f * (q - rintf(q)), &sn, &cs);
                const float d = 6.2831853f * (e - (q - r));  // the angle that q dropped
                const float c0 = cs;
                cs = fmaf(-d, sn, cs);
                sn = fmaf(d, c0, sn);
            } else {
                const double cyc = a.f[k] * t;
                sincospif(2.f * (float)(cyc - rint(cyc)), &sn, &cs);
            }
#pragma unroll
            for (int rr = 0; rr < SY_RB; rr++) {
                const float2 v = A[k][rr];
                acc[rr].x = fmaf(v.x, cs, fmaf(v.y, sn, acc[rr].x));
                acc[rr].y = fmaf(v.y, cs, fmaf(-v.x, sn, acc[rr].y));
            }
        }
#pragma unroll
        for (int rr = 0; rr < SY_RB; rr++) {
            if (r0 + rr >= nr) break;
            float2 *o = a.out + ((size_t)rhs * nr + (r0 + rr)) * a.n_t + j;
            if (a.accumulate) {
                const float2 prev = *o;
                *o = make_float2(prev.x + acc[rr].x, prev.y + acc[rr].y);
            } else {
                *o = acc[rr];
            }
        }
    }
}

tbs_status sy_fail(tbs_status s, const char *msg) {
    tbs::set_last_error(msg);
    return s;
}

}  // namespace

extern "C" tbs_status tbs_synthesize(const tbs_synth_freq *freqs, int32_t n_freq, int32_t n_rhs, double x0,
                                     double y0, double sx, double sy, int32_t nx, int32_t ny, double t0, double dt,
                                     int32_t n_t, float *out, void *stream) {
    if (!freqs || !out) return sy_fail(TBS_ERR_INVALID_ARG, "tbs_synthesize: NULL pointer");
    if (n_freq < 1 || n_rhs < 1 || n_rhs > 65535 || nx < 1 || ny < 1 || n_t < 1)
        return sy_fail(TBS_ERR_INVALID_ARG, "tbs_synthesize: counts must be >= 1 (n_rhs <= 65535)");
    if ((long long)nx * ny > (1ll << 30))
        return sy_fail(TBS_ERR_INVALID_ARG, "tbs_synthesize: more than 2^30 receivers");
    if (!isfinite(x0) || !isfinite(y0) || !isfinite(sx) || !isfinite(sy) || !isfinite(t0) || !isfinite(dt))
        return sy_fail(TBS_ERR_INVALID_ARG, "tbs_synthesize: receiver lattice and times must be finite");
    for (int k = 0; k < n_freq; k++) {
        const tbs_synth_freq &q = freqs[k];
        if (!q.field || q.n < 2 || !(q.dx > 0) || !isfinite(q.dx) || !isfinite(q.freq_hz) || !isfinite(q.weight))
            return sy_fail(TBS_ERR_INVALID_ARG, "tbs_synthesize: bad frequency entry (field, n >= 2, dx > 0, finite)");
        if ((const void *)q.field == (const void *)out)
            return sy_fail(TBS_ERR_INVALID_ARG, "tbs_synthesize: out may not alias a field");
    }
    cudaStream_t s = (cudaStream_t)stream;
    const int nr = nx * ny;
    const int tz = (n_t - 1) / SY_THREADS + 1;
    const dim3 grid((nr + SY_RB - 1) / SY_RB, n_rhs, tz < 65535 ? tz : 65535);
    const double t_max = fmax(fabs(t0), fabs(t0 + (n_t - 1) * dt));
    for (int c = 0; c < n_freq; c += SY_CHUNK) {
        SynthArgs a;
        memset(&a, 0, sizeof(a));
        bool fast = t_max < 1e30;  // FP32 pairs hold t and every f
        a.count = n_freq - c < SY_CHUNK ? n_freq - c : SY_CHUNK;
        for (int k = 0; k < a.count; k++) {
            const tbs_synth_freq &q = freqs[c + k];
            a.field[k] = (const float2 *)q.field;
            a.inv_dx[k] = 1.0 / q.dx;
            fast = fast && fabs(q.freq_hz) < 1e30 && fabs(q.freq_hz) * t_max < 65536.0;
            a.f[k] = q.freq_hz;
            a.w[k] = (float)q.weight;
            a.n[k] = q.n;
        }
        a.accumulate = c > 0;
        a.nx = nx;
        a.ny = ny;
        a.n_t = n_t;
        a.x0 = x0;
        a.y0 = y0;
        a.sx = sx;
        a.sy = sy;
        a.t0 = t0;
        a.dt = dt;
        a.out = (float2 *)out;
        if (fast)
            synth_kernel<true><<<grid, SY_THREADS, 0, s>>>(a);
        else
            synth_kernel<false><<<grid, SY_THREADS, 0, s>>>(a);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) {
            char buf[256];
            snprintf(buf, sizeof(buf), "tbs_synthesize: launch failed: %s", cudaGetErrorString(e));
            return sy_fail(TBS_ERR_CUDA, buf);
        }
    }
    return TBS_OK;
}
