// FP32 form: the fused contraction + epilogue on the CUDA cores (FFMA).
//
// It is the accuracy and speed baseline of the tensor-core forms.  Each CTA owns a
// 128 x 128 tile of G_t = A_t B^T for one displacement t (the paper's thread-block
// tile, Section 3.3), accumulates it in registers (8 x 8 per thread), and reduces the
// tile in place: distance bins through FP32 shared-memory atomics into one copy of the
// bins per warp (summed across the warps in FP64 at the end of the tile; FP64 shared
// atomics where the copies do not fit), phase weights
// through cos(a-b) = cos a cos b + sin a sin b with warp shuffles (Section 3.3, the
// shuffle + shared-memory + atomic reduction), then one FP64 global atomic per bin
// (and per q) per tile.  In the deterministic mode the same sums are 64-bit fixed point
// (integer atomics, the same bits in any order).
//
// Operands are prepared by K: A[k][site] of the whole trajectory row (the displacement's K
// window is a row offset, so no shifted copies) and B[k][site], zero padded.  Both go to shared
// memory as they are (cp.async, no registers, a three-stage pipeline of 16 k).  A thread's
// 8 x 8 outputs are 8 x 4 pairs of columns under packed FMAs: 32 instead of 64 issue slots
// per k, with which the FP32 pipes, which bound the kernel, stay 75 % busy.  Measured on the
// 24^3 glass, K = 1536, 96 bins and 32 q, 2 displacements: 37.8 -> 22.1 ms (31 -> 53 TFLOP/s;
// bins only 58, K = 6144 bins only 60); the steps: operands by K with cp.async and packed FMAs
// 28.1 (scalar FMAs 29.4; A stored twice per value to save packing 31.6), weights by q in the
// phase sums (whole lines instead of 16 per load) 24.6, 16 k per stage instead of 8 22.1.
// A plan without room for its copy of the trajectory by K (DIRECT) loads A from the trajectory
// row at the K-offset s*3F + 3t, four bytes at a time into the same stages, so with the same
// sums in the same order: 31.7 ms.
#include "asd_internal.h"
#include "geom.cuh"

namespace asd {
namespace {

constexpr int TM = 128, TN = 128, TK = 16;
constexpr int kStages = 3;
constexpr int kStageFloats = TK * (TM + TN);   // A, B
constexpr size_t kSumBytes = 48 * 1024;        // most that the bin and phase sums take

struct SimtParams {
    const float *A;   // [S*F3][ld]: the trajectory by K (DIRECT: the trajectory [N][R])
    const float *B;   // [S*Kseg][ld]
    int64_t ld;       // sites, padded to whole 16-byte words
    int64_t R;        // trajectory row length S*F3
    int F3;
    int K3;           // 3*T0
    int Kseg;         // B segment per sample
    int S;
    int N;
    int row_begin, row_end;
    int t_begin;      // displacement of grid slice blockIdx.z = 0
    int a16;          // A rows start on 16 bytes (a first row that is a multiple of four)
    int warp_bins;    // per-warp FP32 bin copies after the FP64 arrays
    EpiParams e;
    int *err;         // device error word (index checks of a checked build)
};

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

// (two CTAs per SM: at most 128 registers a thread)
template <bool DIRECT>
__global__ void __launch_bounds__(256, 2) simt_kernel(const __grid_constant__ SimtParams P)
{
    // pipeline stages, then [n_bins] and [n_q][q_parts] FP64, then [8][n_bins] FP32
    extern __shared__ __align__(16) float dyn[];
    double *red = reinterpret_cast<double *>(dyn + kStages * kStageFloats);
    double *sbins = red;
    double *sq = red + P.e.n_bins;
    float *wbins = reinterpret_cast<float *>(sq + P.e.n_q * P.e.q_parts);
    // deterministic mode: the same arrays as fixed point
    long long *sbins_i = reinterpret_cast<long long *>(sbins);
    long long *sq_i = reinterpret_cast<long long *>(sq);
    const double fscale = P.e.fix_scale ? *P.e.fix_scale : 0.0;

    const int tid = threadIdx.x;
    const int tx = tid & 15, ty = tid >> 4;
    const int t = P.t_begin + blockIdx.z;
    const int m0 = P.row_begin + blockIdx.x * TM;
    const int n0 = blockIdx.y * TN;
    for (int k = tid; k < P.e.n_bins + P.e.n_q * P.e.q_parts; k += 256) red[k] = 0.0;
    const bool wb_on = P.warp_bins && fscale == 0.0;
    if (wb_on)
        for (int k = tid; k < 8 * P.e.n_bins; k += 256) wbins[k] = 0.f;

    const int steps_per_seg = P.Kseg / TK;
    const int n_steps = P.S * steps_per_seg;
    // a stage: 16 k of 128 sites of each operand, [k][site] (512 16-byte words each, two per
    // thread, always the same four sites of it).  Rows past the range, columns past the last
    // site and k past 3*T0 read as zeros.
    const int four = (tid & 31) * 4;
    const uint32_t b_bytes = 4u * min(4, max(0, P.N - n0 - four));
    const int b_col = n0 + (b_bytes ? four : 0);   // (a column that exists where none is read)
    int ls = 0, lk = 0;   // sample and k of the next stage to load
    auto load = [&](int st) {
        if (st < n_steps) {
            float *buf = dyn + (st % kStages) * kStageFloats;
            const uint32_t da = (uint32_t)__cvta_generic_to_shared(buf);
            if (DIRECT) {
                const int k = tid & 15, r0 = tid >> 4;
                const float *A = P.A + (int64_t)(m0 + r0) * P.R + (int64_t)ls * P.F3 + 3 * t + lk + k;
#pragma unroll
                for (int u = 0; u < TM / 16; ++u) {
                    const bool ok = lk + k < P.K3 && m0 + r0 + 16 * u < P.row_end;
                    cp_async4(da + (uint32_t)(k * TM + r0 + 16 * u) * 4,
                              ok ? A + (int64_t)(16 * u) * P.R : P.A, ok ? 4u : 0u);
                }
            } else {
                const float *A = P.A + ((int64_t)ls * P.F3 + 3 * t + lk) * P.ld + m0 + four;
#pragma unroll
                for (int u = 0; u < TK / 8; ++u) {
                    const int k = (tid >> 5) + 8 * u;
                    const int left = lk + k < P.K3 ? min(4, max(0, P.row_end - m0 - four)) : 0;
                    const float *src = left ? A + k * P.ld : P.A;
                    const uint32_t dst = da + (uint32_t)(k * TM + four) * 4;
                    if (P.a16) {
                        cp_async16(dst, src, 4u * left);
                    } else {
                        for (int q = 0; q < 4; ++q)
                            cp_async4(dst + 4 * q, left > q ? src + q : P.A, left > q ? 4u : 0u);
                    }
                }
            }
            const float *B = P.B + ((int64_t)ls * P.Kseg + lk) * P.ld + b_col;
#pragma unroll
            for (int u = 0; u < TK / 8; ++u) {
                const int k = (tid >> 5) + 8 * u;
                cp_async16(da + (uint32_t)(TK * TM + k * TN + four) * 4, B + k * P.ld, b_bytes);
            }
            lk += TK;
            if (lk == P.Kseg) {
                lk = 0;
                ++ls;
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };

    uint64_t acc2[8][4];
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc2[r][c] = 0ull;

    for (int st = 0; st < kStages - 1; ++st) load(st);
    for (int st = 0; st < n_steps; ++st) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
        __syncthreads();   // the stage is in, and every thread is done with the one before
        load(st + kStages - 1);
        const float *As = dyn + (st % kStages) * kStageFloats;
        const float *Bs = As + TK * TM;
#pragma unroll
        for (int kk = 0; kk < TK; ++kk) {
            uint64_t a[8], b[4];
            const float4 *ap = reinterpret_cast<const float4 *>(As + kk * TM) + ty;
            const ulonglong2 *bp = reinterpret_cast<const ulonglong2 *>(Bs + kk * TN) + tx;
            ulonglong2 v;
            float4 f = ap[0], h = ap[16];
#define DUP(d, s) asm("mov.b64 %0, {%1, %1};" : "=l"(d) : "f"(s))
            DUP(a[0], f.x); DUP(a[1], f.y); DUP(a[2], f.z); DUP(a[3], f.w);
            DUP(a[4], h.x); DUP(a[5], h.y); DUP(a[6], h.z); DUP(a[7], h.w);
            v = bp[0];  b[0] = v.x; b[1] = v.y;
            v = bp[16]; b[2] = v.x; b[3] = v.y;
#pragma unroll
            for (int r = 0; r < 8; ++r)
#pragma unroll
                for (int c = 0; c < 4; ++c) acc2[r][c] = fma2(a[r], b[c], acc2[r][c]);
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    float acc[8][8];
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c)
            asm("mov.b64 {%0, %1}, %2;"
                : "=f"(acc[r][2 * c]), "=f"(acc[r][2 * c + 1])
                : "l"(acc2[r][c]));

    // ---------------- epilogue: reduce the tile ----------------
    int ri[8], cj[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        ri[u] = m0 + (u < 4 ? ty * 4 + u : 64 + ty * 4 + u - 4);
        cj[u] = n0 + (u < 4 ? tx * 4 + u : 64 + tx * 4 + u - 4);
    }
    const EpiParams &e = P.e;
    float *myb = wbins + (tid >> 5) * e.n_bins;
    if (e.n_bins > 0) {
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const bool rok = ri[r] < P.row_end;
            const int ir = rok ? ri[r] : P.row_begin;
            const int4 ci = e.coords[ir];
            const float4 pi = e.pos[ir];
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const bool ok = rok && cj[c] < P.N;
                const int jc = cj[c] < P.N ? cj[c] : 0;
                const float d2 = e.geom == ASD_GEOM_LATTICE
                                     ? lattice_d2(ci, e.coords[jc], e.Lx, e.Ly, e.Lz, e.periodic)
                                     : position_d2(pi, e.pos[jc]);
                const int b = bin_of_d2(d2, e.inv_w, e.n_bins, e.thr);
                if (ok && b < e.n_bins && ASD_INB(b >= 0, BND_SIMT_BIN, P.err)) {
                    if (fscale != 0.0) add_fixed(&sbins_i[b], to_fixed((double)acc[r][c], fscale));
                    else if (wb_on) atomicAdd(&myb[b], acc[r][c]);
                    else atomicAdd(&sbins[b], (double)acc[r][c]);
                }
            }
        }
    }
    if (e.n_q > 0) {
        const int lane = tid & 31;
        for (int q = 0; q < e.n_q; ++q) {
            float part = 0.f, part_s = 0.f;
            float2 wc[8];
            const float2 *csq = e.csT + (int64_t)q * e.cs_ld;   // a row per q: whole lines
#pragma unroll
            for (int c = 0; c < 8; c += 2) {   // two sites per 16-byte load (zeros past N)
                const float4 w = __ldg(reinterpret_cast<const float4 *>(csq + cj[c]));
                wc[c] = make_float2(w.x, w.y);
                wc[c + 1] = make_float2(w.z, w.w);
            }
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const float2 wr = ri[r] < P.row_end ? __ldg(csq + ri[r]) : make_float2(0.f, 0.f);
                float u = 0.f, v = 0.f;
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    u = fmaf(wc[c].x, acc[r][c], u);
                    v = fmaf(wc[c].y, acc[r][c], v);
                }
                part = fmaf(wr.x, u, fmaf(wr.y, v, part));        // cos(a - b)
                if (e.q_parts == 2) part_s = fmaf(wr.y, u, fmaf(-wr.x, v, part_s));  // sin(a - b)
            }
            // the warp's 32 partial sums (64 pairs each) in FP32, one FP64 add per warp
            // (FP64 arithmetic runs on a narrow pipe on this part)
            for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
            const bool qok = lane == 0 && ASD_INB(q < e.nq_pad, BND_SIMT_Q, P.err);
            if (qok) {
                if (fscale != 0.0) add_fixed(&sq_i[q * e.q_parts], to_fixed((double)part, fscale));
                else atomicAdd(&sq[q * e.q_parts], (double)part);
            }
            if (e.q_parts == 2) {
                for (int o = 16; o > 0; o >>= 1) part_s += __shfl_xor_sync(0xffffffffu, part_s, o);
                if (qok) {
                    if (fscale != 0.0) add_fixed(&sq_i[2 * q + 1], to_fixed((double)part_s, fscale));
                    else atomicAdd(&sq[2 * q + 1], (double)part_s);
                }
            }
        }
    }
    __syncthreads();
    if (fscale != 0.0) {
        for (int b = tid; b < e.n_bins; b += 256)
            if (sbins_i[b] != 0) add_fixed(&e.C_fix[(int64_t)t * e.n_bins + b], sbins_i[b]);
        for (int o = tid; o < e.n_q * e.q_parts; o += 256)
            if (sq_i[o] != 0) add_fixed(&e.Sq_fix[(int64_t)t * e.n_q * e.q_parts + o], sq_i[o]);
        return;
    }
    for (int b = tid; b < e.n_bins; b += 256) {
        double v = sbins[b];
        if (wb_on)
#pragma unroll
            for (int w = 0; w < 8; ++w) v += (double)wbins[w * e.n_bins + b];
        if (v != 0.0) atomicAdd(&e.C_sum[(int64_t)t * e.n_bins + b], v);
    }
    for (int o = tid; o < e.n_q * e.q_parts; o += 256)
        if (sq[o] != 0.0) atomicAdd(&e.Sq_sum[(int64_t)t * e.n_q * e.q_parts + o], sq[o]);
}

}  // namespace

int launch_simt(asd_corr_plan *p, int64_t row_begin, int64_t row_end, int t_begin, int t_end,
                double *C_sum, double *Sq_sum, cudaStream_t s)
{
    SimtParams P{};
    P.A = p->Af32 ? p->Af32 : p->prepared_traj;
    P.R = p->R;
    P.B = p->Bf32;
    P.ld = p->ldk;
    P.a16 = (row_begin & 3) == 0;
    P.F3 = 3 * p->F;
    P.K3 = 3 * p->T0;
    P.Kseg = (int)p->Kseg;
    P.S = p->S;
    P.N = (int)p->N;
    P.row_begin = (int)row_begin;
    P.row_end = (int)row_end;
    P.t_begin = t_begin;
    EpiParams &e = P.e;
    e.geom = p->d.geometry;
    e.Lx = p->d.L[0];
    e.Ly = p->d.L[1];
    e.Lz = p->d.L[2];
    e.periodic = p->d.periodic;
    e.inv_w = p->n_bins > 0 ? (float)(1.0 / p->d.bin_width) : 1.f;
    e.n_bins = p->n_bins;
    e.n_q = p->n_q;
    e.coords = p->coords;
    e.pos = p->pos;
    e.thr = p->thr;
    e.nq_pad = (p->n_q + kQChunk - 1) / kQChunk * kQChunk;
    e.q_parts = p->q_parts;
    e.csT = p->csT;
    e.cs_ld = p->ld32;
    e.C_sum = C_sum;
    e.Sq_sum = Sq_sum;
    e.C_fix = p->C_fix;
    e.Sq_fix = p->Sq_fix;
    e.fix_scale = p->d.deterministic ? p->fix_scale : nullptr;
    P.err = device_error_word();
    if (!P.err) return ASD_ECUDA;
    dim3 grid((unsigned)((row_end - row_begin + TM - 1) / TM), (unsigned)((p->N + TN - 1) / TN),
              (unsigned)(t_end - t_begin));
    if (grid.y > 65535u || grid.z > 65535u) {
        set_error_text("FP32 form: grid too large (N or n_t)");
        return ASD_EUNSUPPORTED;
    }
    size_t smem = sizeof(double) * (p->n_bins + p->n_q * p->q_parts);
    // per-warp FP32 bin copies where they and the FP64 sums fit
    P.warp_bins = !p->d.deterministic && smem + sizeof(float) * 8 * p->n_bins <= kSumBytes;
    if (P.warp_bins) smem += sizeof(float) * 8 * p->n_bins;
    smem += sizeof(float) * kStages * kStageFloats;
    auto k = p->Af32 ? simt_kernel<false> : simt_kernel<true>;
    ASD_CUDA_TRY(allow_smem(k, kSumBytes + sizeof(float) * kStages * kStageFloats));
    k<<<grid, 256, smem, s>>>(P);
    ASD_CUDA_TRY(cudaGetLastError());
    return ASD_OK;
}

}  // namespace asd
