// Separable evaluation of the phase-weighted sum (the cosine part of Eq. 3 with the
// weights of Eq. 6).  cos(q.(r_i - r_j)) = cos(q.r_i) cos(q.r_j) + sin(q.r_i) sin(q.r_j)
// splits the pair sum into per-site transforms of every frame,
//   Fc(q; s, f, a) = sum_i cos(q.r_i) S_i(s, f, a),   Fs likewise with sin,
// and then
//   Sq_sum[t][q] = sum_{s, a, t0 < T0} Fc(s, t0 + t, a) Fc_B(s, t0, a) + Fs(...) Fs_B(...),
// where the B factors are the transforms of the (optionally centred) B operand: centring
// B per site subtracts its mean over (s, t0 < T0), which in the transform subtracts the
// same mean of Fc_B.  Cost O(N S F n_q) instead of O(N^2 S T0 n_t).
#include <cuda_runtime.h>

#include "asd_internal.h"

namespace asd {
namespace {

constexpr int kTS = 16;       // sites per pipeline stage
constexpr int kStages = 3;
constexpr int kSlice = 4096;  // sites per block; slices are combined with FP64 atomics

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, uint32_t bytes)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void cp_async4(uint32_t dst, const void *src, uint32_t bytes)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// Fb[m][k] += sum_{i in this block's slice} W[i][m] X[i][k]:  W = the (cos, sin) table seen
// as [N][ldw] floats (m = 2q: cos, 2q + 1: sin), X = the trajectory [N][K].  FP32 inside
// a slice (sites in ascending order), FP64 across slices.  Bound by the FP32 pipes: 8 x 8
// outputs per thread as packed FMAs on column pairs, both operands by site already, so they
// go to shared memory as they are (cp.async; 16 bytes where the trajectory's rows allow, the
// rows of an odd number of frames start anywhere).  TM = 128, 64 or 32 transform rows so that
// few q-vectors do not pay for padding, and 4 x 4 or 2 x 2 outputs per thread where the big
// tiles would leave SMs idle.  Measured, 40^3 sites, 64 q, 639 frames: 1.61 -> 0.77 ms (64 x 128
// tiles, 8 x 4 per thread, scalar loads, and a grid of 1.05 waves before; now the grid is 1.6
// blocks per SM of two that fit, which 104-column tiles did not better: 0.81); 20^3 sites, 16
// q, 263 frames: 550 -> 119 us.
template <int TM, int U>
__global__ void __launch_bounds__(256, U == 8 ? 2 : 4) nudft_kernel(const float *__restrict__ W, int ldw, int M,
                                                       const float *__restrict__ X, int64_t K,
                                                       int64_t N, int x16, double *__restrict__ Fb)
{
    // thread: U rows and U columns (8: in two groups of four)
    constexpr int NT = 256, TN = NT * U * U / TM, TX = TN / U, kFloats = kTS * (TM + TN);
    // 4-byte copies: a thread keeps its columns (kCols of them, NT apart) and walks the rows
    constexpr int kCols = TN > NT ? TN / NT : 1, kRows = TN > NT ? 1 : NT / TN;
    extern __shared__ __align__(16) float dyn[];
    const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
    const int m0 = blockIdx.y * TM;
    const int64_t k0 = (int64_t)blockIdx.x * TN;
    const int64_t i0 = (int64_t)blockIdx.z * kSlice;
    const int64_t i1 = i0 + kSlice < N ? i0 + kSlice : N;
    const int steps = (int)((i1 - i0 + kTS - 1) / kTS);
    // stage: kTS sites of TM table entries, then of TN trajectory columns; zeros past the ends
    auto load = [&](int st) {
        if (st < steps) {
            const uint32_t d = (uint32_t)__cvta_generic_to_shared(dyn + (st % kStages) * kFloats);
            const int64_t i = i0 + (int64_t)st * kTS;
#pragma unroll
            for (int e = tid; e < kTS * TM / 4; e += NT) {
                const int r = e / (TM / 4), c = e % (TM / 4) * 4;
                const bool ok = i + r < i1 && m0 + c < ldw;   // ldw is a multiple of 4
                cp_async16(d + (uint32_t)(r * TM + c) * 4, ok ? W + (i + r) * ldw + m0 + c : W,
                           ok ? 16u : 0u);
            }
            const uint32_t dx = d + kTS * TM * 4;
            if (x16) {
#pragma unroll
                for (int e = tid; e < kTS * TN / 4; e += NT) {
                    const int r = e / (TN / 4), c = e % (TN / 4) * 4;
                    const bool ok = i + r < i1 && k0 + c < K;   // K is a multiple of 4
                    cp_async16(dx + (uint32_t)(r * TN + c) * 4, ok ? X + (i + r) * K + k0 + c : X,
                               ok ? 16u : 0u);
                }
            } else {
                const int r0 = tid / TN, c0 = tid % TN;   // (kCols > 1: row 0, column tid)
                const float *src = X + (i + r0) * K + k0 + c0;
                const uint32_t dst = dx + (uint32_t)(r0 * TN + c0) * 4;
#pragma unroll
                for (int r = 0; r < kTS; r += kRows)
#pragma unroll
                    for (int u = 0; u < kCols; ++u) {
                        const bool ok = i + r0 + r < i1 && k0 + c0 + u * NT < K;
                        cp_async4(dst + (uint32_t)(r * TN + u * NT) * 4,
                                  ok ? src + (int64_t)r * K + u * NT : X, ok ? 4u : 0u);
                    }
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    uint64_t acc[U][U / 2];
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
        for (int v = 0; v < U / 2; ++v) acc[u][v] = 0ull;
    for (int st = 0; st < kStages - 1; ++st) load(st);
    for (int st = 0; st < steps; ++st) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
        __syncthreads();   // the stage is in, and every thread is done with the one before
        load(st + kStages - 1);
        const float *ws = dyn + (st % kStages) * kFloats, *xs = ws + kTS * TM;
#pragma unroll
        for (int r = 0; r < kTS; ++r) {
            float as[U];
            uint64_t a[U], b[U / 2];
            if (U == 2) {
                const float2 f = reinterpret_cast<const float2 *>(ws + r * TM)[ty];
                as[0] = f.x;
                as[1] = f.y;
                b[0] = reinterpret_cast<const uint64_t *>(xs + r * TN)[tx];
            } else {
#pragma unroll
                for (int h = 0; h < U / 4; ++h) {
                    const float4 f = reinterpret_cast<const float4 *>(ws + r * TM)[ty + h * (TM / 8)];
                    as[4 * h] = f.x;
                    as[4 * h + 1] = f.y;
                    as[4 * h + 2] = f.z;
                    as[4 * h + 3] = f.w;
                    const ulonglong2 v =
                        reinterpret_cast<const ulonglong2 *>(xs + r * TN)[tx + h * (TN / 8)];
                    b[2 * h] = v.x;
                    b[2 * h + 1] = v.y;
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) asm("mov.b64 %0, {%1, %1};" : "=l"(a[u]) : "f"(as[u]));
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int c = 0; c < U / 2; ++c) acc[u][c] = fma2(a[u], b[c], acc[u][c]);
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    constexpr int G = U < 4 ? U : 4;   // contiguous rows / columns of a group
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int m = m0 + u / G * (TM / 2) + ty * G + u % G;
        if (m >= M) continue;
#pragma unroll
        for (int c = 0; c < U / 2; ++c) {
            float lo, hi;
            asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(acc[u][c]));
            const int64_t k = k0 + 2 * c / G * (TN / 2) + tx * G + 2 * c % G;
            if (k < K) atomicAdd(&Fb[(int64_t)m * K + k], (double)lo);
            if (k + 1 < K) atomicAdd(&Fb[(int64_t)m * K + k + 1], (double)hi);
        }
    }
}

template <int TM, int U>
int launch_nudft(const float *W, int ldw, int M, const float *X, int64_t K, int64_t N, bool x16,
                 double *Fb, cudaStream_t s)
{
    constexpr int TN = 256 * U * U / TM;
    constexpr size_t smem = sizeof(float) * kStages * kTS * (TM + TN);
    ASD_CUDA_TRY(allow_smem(nudft_kernel<TM, U>, smem));
    dim3 g((unsigned)((K + TN - 1) / TN), (unsigned)((M + TM - 1) / TM),
           (unsigned)((N + kSlice - 1) / kSlice));
    nudft_kernel<TM, U><<<g, 256, smem, s>>>(W, ldw, M, X, K, N, x16, Fb);
    ASD_CUDA_TRY(cudaGetLastError());
    return ASD_OK;
}

__device__ __forceinline__ double block_sum(double v, double *red)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();
    if (l == 0) red[w] = v;
    __syncthreads();
    double s = 0.0;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) s += red[k];
    return s;
}

// Sq_sum[t][q] += sum_{s, a, t0 < T0} Fc(s, t0 + t, a) (Fc(s, t0, a) - mc_a)
//              + Fs(s, t0 + t, a) (Fs(s, t0, a) - ms_a),
// mc_a / ms_a = the mean over (s, t0 < T0) when centring, else 0.  Block (q, group of kTPB
// displacements, whose sums advance together: the origins are read once for all).  The FP64
// pipe bounds this kernel, so no centring subtractions without centring and no sine products
// unless asked for.  64 q, 128 displacements, T0 = 512: 194 -> 68 us.
constexpr int kTPB = 8;  // displacements per block

template <int PARTS>
__global__ void __launch_bounds__(256) sq_corr_kernel(const double *__restrict__ Fb, int64_t K,
                                                      int S, int F, int T0, int n_t, int center,
                                                      int n_q, double *__restrict__ Sq_sum)
{
    __shared__ double red[8], sums[8][PARTS * kTPB];
    const int q = blockIdx.x;
    const double *fc = Fb + (int64_t)(2 * q) * K;
    const double *fs = Fb + (int64_t)(2 * q + 1) * K;
    const int n_terms = S * T0 * 3;
    double mc[3] = {0.0, 0.0, 0.0}, ms[3] = {0.0, 0.0, 0.0};
    if (center) {
        for (int a = 0; a < 3; ++a) {
            double vc = 0.0, vs = 0.0;
            for (int e = threadIdx.x; e < S * T0; e += blockDim.x) {
                const int s = e / T0, t0 = e % T0;
                const int64_t k = ((int64_t)s * F + t0) * 3 + a;
                vc += fc[k];
                vs += fs[k];
            }
            mc[a] = block_sum(vc, red) / (double)(S * T0);
            ms[a] = block_sum(vs, red) / (double)(S * T0);
        }
    }
    // term e = 3 (s T0 + t0) + a lies at e + s skip of a transform row
    const int seg = 3 * T0, skip = 3 * (F - T0);
    const int tb = blockIdx.y * kTPB, tn = min(kTPB, n_t - tb);
    double v[kTPB] = {}, vs[kTPB] = {};
    for (int e = threadIdx.x; e < n_terms; e += blockDim.x) {
        const int64_t kb = e + (int64_t)(S > 1 ? e / seg : 0) * skip;
        double bc = fc[kb], bs = fs[kb];
        if (center) {
            const int a = e % 3;
            bc -= a == 0 ? mc[0] : a == 1 ? mc[1] : mc[2];
            bs -= a == 0 ? ms[0] : a == 1 ? ms[1] : ms[2];
        }
#pragma unroll
        for (int u = 0; u < kTPB; ++u) {
            if (u >= tn) break;
            const int64_t ka = kb + 3 * (int64_t)(tb + u);
            const double ac = fc[ka], as = fs[ka];
            v[u] = fma(ac, bc, v[u]);
            v[u] = fma(as, bs, v[u]);
            if (PARTS == 2) {   // sine part: sin(a - b) = sin a cos b - cos a sin b
                vs[u] = fma(as, bc, vs[u]);
                vs[u] = fma(-ac, bs, vs[u]);
            }
        }
    }
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
#pragma unroll
    for (int u = 0; u < kTPB; ++u) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            v[u] += __shfl_xor_sync(0xffffffffu, v[u], o);
            if (PARTS == 2) vs[u] += __shfl_xor_sync(0xffffffffu, vs[u], o);
        }
        if (l == 0) {
            sums[w][u * PARTS] = v[u];
            if (PARTS == 2) sums[w][u * PARTS + PARTS - 1] = vs[u];
        }
    }
    __syncthreads();
    if ((int)threadIdx.x < tn * PARTS) {
        double s = 0.0;
        for (int k = 0; k < 8; ++k) s += sums[k][threadIdx.x];
        const int u = threadIdx.x / PARTS, part = threadIdx.x % PARTS;
        Sq_sum[((int64_t)(tb + u) * n_q + q) * PARTS + part] += s;
    }
}

}  // namespace
}  // namespace asd

int asd_pair_corr_sq_separable(asd_corr_plan *p, const float *traj, double *Sq_sum, void *stream)
{
    using namespace asd;
    ASD_CHECK_ARG(p && traj && Sq_sum, "null argument");
    ASD_CHECK_ARG(p->n_q > 0 && p->sqF, "plan has no q-vectors");
    cudaStream_t s = (cudaStream_t)stream;
    const int64_t K = (int64_t)p->S * 3 * p->F;
    const int nqp = (p->n_q + kQChunk - 1) / kQChunk * kQChunk;
    const int M = 2 * p->n_q;
    ASD_CUDA_TRY(cudaMemsetAsync(p->sqF, 0, sizeof(double) * (size_t)M * K, s));
    ASD_CHECK_ARG((p->N + kSlice - 1) / kSlice <= 65535, "too many sites for the separable transform");
    const float *W = reinterpret_cast<const float *>(p->cs);
    // Tile choice.  The chain of sites in a slice is serial, so a launch takes (blocks per SM) x
    // (time of a block): big tiles for throughput, smaller ones where they leave SMs idle.
    // Estimated times in us for one slice, b blocks per SM, measured over 14^3 to 40^3 sites,
    // 150 to 639 frames and 16 to 100 q (16-byte / 4-byte trajectory copies):
    //   8 x 8 per thread    50 + 350 b /  90 + 360 b
    //   4 x 4               60 + 113 b /  75 + 145 b
    //   2 x 2               40 +  50 b /  60 +  60 b
    const bool x16 = K % 4 == 0 && (reinterpret_cast<uintptr_t>(traj) & 15) == 0;
    const auto rows = [&](int tm) { return (M + tm - 1) / tm * tm; };
    const int64_t slices = (p->N + kSlice - 1) / kSlice;
    const auto per_sm = [&](int tm, int tn) {
        const int64_t blocks = (K + tn - 1) / tn * (rows(tm) / tm) * slices;
        return (double)((blocks + p->sm_count - 1) / p->sm_count);
    };
    // (the tile height whose rows are least padded, the taller one on a tie)
    const int tm8 = rows(128) <= rows(64) && rows(128) <= rows(32) ? 128 : rows(64) <= rows(32) ? 64 : 32;
    const double u8 = per_sm(tm8, 16384 / tm8);
    const double t8 = x16 ? 50 + 350 * u8 : 90 + 360 * u8;
    const double t4 = x16 ? 60 + 113 * per_sm(32, 128) : 75 + 145 * per_sm(32, 128);
    const double t2 = x16 ? 40 + 50 * per_sm(32, 32) : 60 + 60 * per_sm(32, 32);
    auto k = t2 < t4 && t2 < t8 ? launch_nudft<32, 2>
             : t4 < t8          ? launch_nudft<32, 4>
             : tm8 == 64        ? launch_nudft<64, 8>
             : tm8 == 32        ? launch_nudft<32, 8>
                                : launch_nudft<128, 8>;
    const int rc = k(W, 2 * nqp, M, traj, K, p->N, x16, p->sqF, s);
    if (rc) return rc;
    dim3 g2((unsigned)p->n_q, (unsigned)((p->n_t + kTPB - 1) / kTPB), 1);
    auto corr = p->q_parts == 2 ? sq_corr_kernel<2> : sq_corr_kernel<1>;
    corr<<<g2, 256, 0, s>>>(p->sqF, K, p->S, p->F, p->T0, p->n_t, p->center, p->n_q, Sq_sum);
    ASD_CUDA_TRY(cudaGetLastError());
    return ASD_OK;
}
