// Dynamical structure factor S(q, omega) from S(q, t) (Section 4): the windowed cosine
// transform of the even extension S(q, -t) = S(q, t) of the displacement series,
//   S(q, w_k) = dt * ( v_0 S(q, 0) + 2 sum_{t=1}^{n_t-1} v_t S(q, t) cos(w_k t dt) ),
// with v_t = 1 (no window), 0.5 (1 + cos(pi t / n_t)) (Hann) or exp(-(t / (width n_t))^2 / 2)
// (Gaussian).  The cosine advances by a rotation per step, re-seeded from sincos every 32
// steps, in FP64; a block (one frequency) makes its cosines once, a thread per run of 32, for
// all q-vectors.  The FP64 pipe bounds this kernel: two operations per (frequency, q,
// displacement) instead of six with a rotation in every thread (256 frequencies, 64 q, 128
// displacements: 65 -> 32 us).
#include <cuda_runtime.h>

#include "asd_internal.h"

namespace asd {
namespace {

constexpr int kMaxNt = 6000;  // window weights and cosines in shared memory (96 KB)

// SHORT: one run of displacements (n_t <= 32).  Every thread then rotates for itself beside its sum
// instead of waiting for the run (16 displacements, 16 q, 256 frequencies: 10.3 us, 12.3 with the
// run made first).
template <bool SHORT>
__global__ void sq_omega_kernel(const double *__restrict__ S, int n_t, int n_q, double dt,
                                int window, double width, const double *__restrict__ omega,
                                double *__restrict__ Sqw)
{
    extern __shared__ double v[];   // [n_t] window, then (not SHORT) [n_t] cosines
    double *ct = v + n_t;
    for (int t = threadIdx.x; t < n_t; t += blockDim.x) {
        double w = 1.0;
        if (window == 1) w = 0.5 * (1.0 + cospi((double)t / n_t));
        else if (window == 2) {
            const double x = (double)t / (width * n_t);
            w = exp(-0.5 * x * x);
        }
        v[t] = w;
    }
    const int k = blockIdx.x;
    const double th = omega[k] * dt;
    if (SHORT) __syncthreads();
    double sr, cr;
    sincos(th, &sr, &cr);  // rotation by one step
    if (!SHORT) {
        for (int t0 = 32 * threadIdx.x; t0 < n_t; t0 += 32 * blockDim.x) {
            double c = 1.0, s = 0.0;
            if (t0 > 0) sincos(th * t0, &s, &c);
            for (int t = t0; t < t0 + 32 && t < n_t; ++t) {
                ct[t] = c;
                const double c2 = c * cr - s * sr;
                s = s * cr + c * sr;
                c = c2;
            }
        }
        __syncthreads();
    }
    for (int q = threadIdx.x; q < n_q; q += blockDim.x) {
        double acc = 0.0;
        if (SHORT) {
            double c = 1.0, s = 0.0;
            for (int t = 1; t < n_t; ++t) {
                const double c2 = c * cr - s * sr;
                s = s * cr + c * sr;
                c = c2;
                acc = fma(v[t] * S[(int64_t)t * n_q + q], c, acc);
            }
        } else {
#pragma unroll 8
            for (int t = 1; t < n_t; ++t) acc = fma(v[t] * S[(int64_t)t * n_q + q], ct[t], acc);
        }
        Sqw[(int64_t)k * n_q + q] = dt * (v[0] * S[q] + 2.0 * acc);
    }
}

}  // namespace
}  // namespace asd

int asd_sq_omega(const double *S, int n_t, int n_q, double dt, int window, double width,
                 const double *omega, int n_w, double *Sqw, void *stream)
{
    using namespace asd;
    ASD_CHECK_ARG(S && omega && Sqw, "null argument");
    ASD_CHECK_ARG(n_t >= 1 && n_t <= kMaxNt, "n_t: 1..6000");
    ASD_CHECK_ARG(n_q >= 1 && n_w >= 1 && n_w <= 65535, "n_q >= 1, n_w in 1..65535");
    ASD_CHECK_ARG(dt > 0.0, "dt > 0");
    ASD_CHECK_ARG(window >= 0 && window <= 2, "window: 0 none, 1 Hann, 2 Gaussian");
    ASD_CHECK_ARG(window != 2 || width > 0.0, "Gaussian window needs width > 0");
    const bool one = n_t <= 32;
    const size_t smem = (one ? 1 : 2) * sizeof(double) * (size_t)n_t;   // 96 KB at most
    auto k = one ? sq_omega_kernel<true> : sq_omega_kernel<false>;
    if (smem > 48 * 1024) ASD_CUDA_TRY(allow_smem(k, 2 * sizeof(double) * kMaxNt));
    k<<<n_w, 128, smem, (cudaStream_t)stream>>>(S, n_t, n_q, dt, window, width, omega, Sqw);
    ASD_CUDA_TRY(cudaGetLastError());
    return ASD_OK;
}
