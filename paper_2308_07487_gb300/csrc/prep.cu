// Operand preparation for the fused contraction (HBM-bound, once per call).
//
// The paper rebuilds its N x 3M GEMM operand from the trajectory at every time step
// and centres it while doing so (Section 3.2, Eq. 5).  Here the trajectory row of
// site i, traj[i][s][f][a], is already K-contiguous, so the operand for
// displacement t is the K-offset window that starts at element s*3F + 3t of that row.
// A TMA copy must start on a 16-byte boundary, so the row is stored in 16/elem_bytes
// shifted copies (copy c holds row[x + c] at x); the window then starts at
// x = s*3F + 3t - c in the copy with c = (s*3F + 3t) mod (16/elem_bytes).
//
// B (the t0 frames) is stored once, zero-padded per sample to Kseg = roundup(3*T0, BK)
// so that the extra columns of every A window meet zeros.  With center = 1, B is
// centred by the per-site mean over (s, t0 < T0); centring A as well would subtract a
// constant per (i, t) that multiplies sum_{s,t0}(B - mean B) = 0, so Eq. 5 and Eq. 4
// are reached with B alone.
//
// Precision forms: BF16 hi = RN(x); split-BF16 lo = RN(x - hi); TF32 = RNA to 10-bit
// mantissa (the tensor core would otherwise truncate); FP32: both operands by K (prep32_kernel).
#include <cuda_bf16.h>

#include "asd_internal.h"

namespace asd {
namespace {

__device__ __forceinline__ float tf32_round(float x)
{
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return __uint_as_float(r);
}

// mean over (s, t0 < T0) of each component, one warp per site
__global__ void means_kernel(const float *__restrict__ traj, int64_t N, int S, int F, int T0,
                             float *__restrict__ mean)
{
    const int64_t i = (int64_t)blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
    const int lane = threadIdx.x & 31;
    if (i >= N) return;
    double acc[3] = {0, 0, 0};
    for (int s = 0; s < S; ++s) {
        const float *row = traj + ((i * S + s) * (int64_t)F) * 3;
        for (int k = lane; k < 3 * T0; k += 32) acc[k % 3] += row[k];
    }
    // each lane holds partial sums per component; reduce each over the warp
    for (int a = 0; a < 3; ++a) {
        double v = acc[a];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        acc[a] = v;
    }
    if (lane == 0)
        for (int a = 0; a < 3; ++a) mean[3 * i + a] = (float)(acc[a] / ((double)S * T0));
}

// B operand: [N][S*Kseg], 8 consecutive k per thread; `block` of `blocks` takes a share
template <int FORM>
__device__ __forceinline__ void prep_b(const float *__restrict__ traj, int64_t N, int S, int F,
                                       int T0, int Kseg, const float *__restrict__ mean,
                                       int center, void *out0, void *out1, unsigned block,
                                       unsigned blocks)
{
    const int64_t chunks_per_row = (int64_t)S * Kseg / 8;
    const int64_t total = N * chunks_per_row;
    for (int64_t g = (int64_t)block * blockDim.x + threadIdx.x; g < total;
         g += (int64_t)blocks * blockDim.x) {
        const int64_t j = g / chunks_per_row;
        const int64_t kk = (g % chunks_per_row) * 8;
        const int s = (int)(kk / Kseg);
        const int k0 = (int)(kk % Kseg);
        const float *row = traj + ((j * S + s) * (int64_t)F) * 3;
        float v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int k = k0 + u;
            float x = 0.f;
            if (k < 3 * T0) {
                x = row[k];
                if (center) x -= mean[3 * j + k % 3];
            }
            v[u] = x;
        }
        const int64_t off = j * (int64_t)S * Kseg + kk;
        if (FORM == ASD_TF32) {
            float4 *o = reinterpret_cast<float4 *>(static_cast<float *>(out0) + off);
            for (int u = 0; u < 8; ++u) v[u] = tf32_round(v[u]);
            o[0] = make_float4(v[0], v[1], v[2], v[3]);
            o[1] = make_float4(v[4], v[5], v[6], v[7]);
        } else {
            __align__(16) __nv_bfloat16 hi[8], lo[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                hi[u] = __float2bfloat16_rn(v[u]);
                lo[u] = __float2bfloat16_rn(v[u] - __bfloat162float(hi[u]));
            }
            *reinterpret_cast<uint4 *>(static_cast<__nv_bfloat16 *>(out0) + off) =
                *reinterpret_cast<uint4 *>(hi);
            if (FORM == ASD_SPLIT_BF16)
                *reinterpret_cast<uint4 *>(static_cast<__nv_bfloat16 *>(out1) + off) =
                    *reinterpret_cast<uint4 *>(lo);
        }
    }
}

struct CopyPtrs {
    void *p[2][kMaxCopies];
};

// A operand copies: copy c, row i, elements x..x+V-1 (V = 16 / elem_bytes)
template <int FORM>
__device__ __forceinline__ void prep_a(const float *__restrict__ traj, int64_t row_begin,
                                       int64_t row_end, int64_t R, int64_t Rpad,
                                       const CopyPtrs &cp, unsigned block, unsigned blocks)
{
    constexpr int V = (FORM == ASD_TF32) ? 4 : 8;  // elements per 16-byte store = copies
    const int64_t chunks = Rpad / V;
    const int64_t total = (row_end - row_begin) * chunks;
    for (int64_t g = (int64_t)block * blockDim.x + threadIdx.x; g < total;
         g += (int64_t)blocks * blockDim.x) {
        const int64_t i = row_begin + g / chunks;
        const int64_t x0 = (g % chunks) * V;
        const float *row = traj + i * R;
        float w[2 * V];
#pragma unroll
        for (int u = 0; u < 2 * V - 1; ++u) {
            const int64_t x = x0 + u;
            w[u] = x < R ? __ldg(row + x) : 0.f;
        }
        const int64_t off = i * Rpad + x0;
#pragma unroll
        for (int c = 0; c < V; ++c) {
            if (FORM == ASD_TF32) {
                float4 o = make_float4(tf32_round(w[c]), tf32_round(w[c + 1]), tf32_round(w[c + 2]),
                                       tf32_round(w[c + 3]));
                *reinterpret_cast<float4 *>(static_cast<float *>(cp.p[0][c]) + off) = o;
            } else {
                __align__(16) __nv_bfloat16 hi[8], lo[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    hi[u] = __float2bfloat16_rn(w[c + u]);
                    lo[u] = __float2bfloat16_rn(w[c + u] - __bfloat162float(hi[u]));
                }
                *reinterpret_cast<uint4 *>(static_cast<__nv_bfloat16 *>(cp.p[0][c]) + off) =
                    *reinterpret_cast<uint4 *>(hi);
                if (FORM == ASD_SPLIT_BF16)
                    *reinterpret_cast<uint4 *>(static_cast<__nv_bfloat16 *>(cp.p[1][c]) + off) =
                        *reinterpret_cast<uint4 *>(lo);
            }
        }
    }
}

// FP32 form: operands by K.  32 x 32 tiles through shared memory, k along a trajectory row in,
// sites out: A[k][i] for rows [row_begin, row_end) and every k of the row, and
// B[s*Kseg + kl][j] = x (centred), zero for kl >= 3*T0 and for the padding sites.
struct Prep32Args {
    const float *traj;
    int64_t N, ld, R, row_begin, row_end;
    int S, F3, K3, Kseg;
    const float *mean;
    int center;
    float *A;
    float *B;
    int64_t tiles_a_k, tiles_a, tiles_b_k, tiles;   // along k, A in all; B along k; in all
};

__global__ void __launch_bounds__(256) prep32_kernel(const __grid_constant__ Prep32Args a)
{
    __shared__ float tile[32][33];
    const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
    for (int64_t blk = blockIdx.x; blk < a.tiles; blk += gridDim.x) {
        const bool is_a = blk < a.tiles_a;
        const int64_t b = is_a ? blk : blk - a.tiles_a;
        const int64_t tk = is_a ? a.tiles_a_k : a.tiles_b_k;
        const int64_t k0 = b % tk * 32, i0 = (is_a ? a.row_begin : 0) + b / tk * 32;
        const int64_t i1 = is_a ? a.row_end : a.N;
#pragma unroll
        for (int u = 0; u < 32; u += 8) {
            const int64_t i = i0 + y + u, k = k0 + x;
            float v = 0.f;
            if (i < i1) {
                if (is_a) {
                    if (k < a.R) v = __ldg(a.traj + i * a.R + k);
                } else {
                    const int s = (int)(k / a.Kseg), kl = (int)(k - (int64_t)s * a.Kseg);
                    if (s < a.S && kl < a.K3) {
                        v = __ldg(a.traj + i * a.R + (int64_t)s * a.F3 + kl);
                        if (a.center) v -= a.mean[3 * i + kl % 3];
                    }
                }
            }
            tile[y + u][x] = v;
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < 32; u += 8) {
            const int64_t k = k0 + y + u, i = i0 + x;
            const float v = tile[x][y + u];
            if (is_a) {
                if (k < a.R && i < i1) a.A[k * a.ld + i] = v;
            } else if (k < (int64_t)a.S * a.Kseg && i < a.ld) {
                a.B[k * a.ld + i] = v;
            }
        }
        __syncthreads();
    }
}

// Both operands in one launch, the first blocks_b blocks the B operand and the rest the A
// copies (a launch costs a call of a small problem 2 us, as much as its preparation:
// 16 x 16 sites, T0 = 64, preparation to normalisation 33.1 -> 30.8 us).
struct PrepArgs {
    const float *traj;
    int64_t N;
    int S, F, T0, Kseg;
    const float *mean;
    int center;
    void *b0, *b1;
    unsigned blocks_b;
    int64_t row_begin, row_end, R, Rpad;
    CopyPtrs cp;
};

template <int FORM>
__global__ void __launch_bounds__(256) prep_kernel(const __grid_constant__ PrepArgs a)
{
    if (blockIdx.x < a.blocks_b)
        prep_b<FORM>(a.traj, a.N, a.S, a.F, a.T0, a.Kseg, a.mean, a.center, a.b0, a.b1,
                     blockIdx.x, a.blocks_b);
    else
        prep_a<FORM>(a.traj, a.row_begin, a.row_end, a.R, a.Rpad, a.cp,
                     blockIdx.x - a.blocks_b, gridDim.x - a.blocks_b);
}

unsigned grid_for(int64_t work, int sm_count)
{
    int64_t b = (work + 255) / 256;
    int64_t cap = (int64_t)sm_count * 16;
    return (unsigned)(b < cap ? (b > 0 ? b : 1) : cap);
}

}  // namespace

int launch_prep(asd_corr_plan *p, const float *traj, int64_t row_begin, int64_t row_end,
                cudaStream_t s)
{
    const int T0 = p->T0, F = p->F, S = p->S;
    if (p->center) {
        means_kernel<<<(unsigned)((p->N + 7) / 8), 256, 0, s>>>(traj, p->N, S, F, T0, p->meanB);
        ASD_CUDA_TRY(cudaGetLastError());
    }
    if (!p->tc) {
        Prep32Args a{};
        a.traj = traj;
        a.N = p->N;
        a.ld = p->ldk;
        a.R = p->R;
        a.row_begin = row_begin;
        a.row_end = row_end;
        a.S = S;
        a.F3 = 3 * F;
        a.K3 = 3 * T0;
        a.Kseg = (int)p->Kseg;
        a.mean = p->meanB;
        a.center = p->center;
        a.A = p->Af32;
        a.B = p->Bf32;
        a.tiles_a_k = (p->R + 31) / 32;
        a.tiles_a = p->Af32 ? a.tiles_a_k * ((row_end - row_begin + 31) / 32) : 0;
        a.tiles_b_k = (p->Kb + 31) / 32;
        a.tiles = a.tiles_a + a.tiles_b_k * ((p->ldk + 31) / 32);
        const int64_t blocks = a.tiles < (1 << 20) ? a.tiles : 1 << 20;
        prep32_kernel<<<(unsigned)blocks, 256, 0, s>>>(a);
        ASD_CUDA_TRY(cudaGetLastError());
        return ASD_OK;
    }
    PrepArgs a{};
    a.traj = traj;
    a.N = p->N;
    a.S = S;
    a.F = F;
    a.T0 = T0;
    a.Kseg = (int)p->Kseg;
    a.mean = p->meanB;
    a.center = p->center;
    a.b0 = p->B[0];
    a.b1 = p->B[1];
    a.blocks_b = grid_for(p->N * p->Kb / 8, p->sm_count);
    a.row_begin = row_begin;
    a.row_end = row_end;
    a.R = p->R;
    a.Rpad = p->Rpad;
    for (int pl = 0; pl < p->n_planes; ++pl)
        for (int c = 0; c < p->n_copies; ++c) a.cp.p[pl][c] = p->A[pl][c];
    unsigned blocks = a.blocks_b;
    if (row_end > row_begin)
        blocks += grid_for((row_end - row_begin) * (p->Rpad / (p->prec == ASD_TF32 ? 4 : 8)),
                           p->sm_count);
    switch (p->prec) {
    case ASD_TF32: prep_kernel<ASD_TF32><<<blocks, 256, 0, s>>>(a); break;
    case ASD_BF16: prep_kernel<ASD_BF16><<<blocks, 256, 0, s>>>(a); break;
    default: prep_kernel<ASD_SPLIT_BF16><<<blocks, 256, 0, s>>>(a); break;
    }
    ASD_CUDA_TRY(cudaGetLastError());
    return ASD_OK;
}

}  // namespace asd
