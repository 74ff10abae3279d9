// Training of the learned von Mises-Fisher proposal (extension of the Monte Carlo of
// Section 2.1; the paper has no learned component).
//
// Model: x (neighbour spins, 3z) -> tanh(W1 x + b1) -> tanh(W2 h1 + b2)
// [-> tanh(Wm h2 + bm) with three hidden layers] -> o = W3 h_last + b3,
// mu = o[0:3]/|o[0:3]|, kappa = softplus(o[3]) + 1e-4.  Loss: the negative log-likelihood
// of the site spin y under vMF(mu, kappa):
//   NLL = -log kappa + log(2 pi) + kappa + log(1 - e^{-2 kappa}) - kappa mu.y
// (log of the normaliser 4 pi sinh(kappa) / kappa written to stay finite).
// Gradients: dNLL/dkappa = coth(kappa) - 1/kappa - mu.y (the Langevin function, with a
// series below kappa = 1e-2), dNLL/dv = -kappa (y - mu (mu.y)) / |v| for v = o[0:3],
// then back through the tanh layers.
//
// loss_grad: persistent blocks of 256 threads over tiles of 64 samples.  Every layer of a tile
// is a 64 x 64 product in registers (4 x 4 per thread) from shared memory: forward, deltas,
// and the weight gradients, whose sums stay in registers over a block's tiles, so the launch
// issues one global atomic per parameter per block.
#include <cuda_bf16.h>

#include "asd_internal.h"
#include "mlp.cuh"
#include "philox.cuh"

namespace asd {
namespace {

constexpr int H = kMlpHidden;
constexpr int kTile = 64;          // samples per tile
constexpr int kLG = 256;           // threads
constexpr int kAP = kTile + 4;     // row of activations, [feature][sample]: 16-byte aligned, and
                                   // 16 rows read together fall on different banks
constexpr int kWP = H + 4;         // row of a hidden layer's weights, likewise
// inputs padded to whole 16-byte words (zero weights and inputs add nothing)
__host__ __device__ constexpr int pad4(int n) { return (n + 3) / 4 * 4; }

// Packed parameters [W1 H*nin][b1 H] then, per further hidden layer, [W H*H][b H], then
// [W3 4*H][b3 4]; BF16 weights [W1]([W2][Wm])[W3].
__host__ __device__ inline int64_t n_params(int nin, int depth)
{
    return (int64_t)H * nin + H + (int64_t)(depth - 1) * (H * H + H) + 4 * H + 4;
}
__host__ __device__ inline int64_t n_weights(int nin, int depth)
{
    return (int64_t)H * nin + (int64_t)(depth - 1) * H * H + 4 * H;
}
inline bool shape_ok(int nin, int depth)
{
    return nin >= 3 && nin <= kMlpMaxIn && (depth == 2 || depth == 3);
}

__global__ void gather_kernel(int64_t N, int S, int z, const int *__restrict__ nbr,
                              const float *__restrict__ spins, float *__restrict__ x,
                              float *__restrict__ y)
{
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= N * S) return;
    const int64_t s = k / N, i = k % N;
    const float *Ys = spins + s * N * 3;
    for (int a = 0; a < z; ++a) {
        const int j = nbr[i * z + a];
        for (int c = 0; c < 3; ++c) x[k * 3 * z + 3 * a + c] = j >= 0 ? Ys[3 * (int64_t)j + c] : 0.f;
    }
    for (int c = 0; c < 3; ++c) y[3 * k + c] = Ys[3 * i + c];
}

__device__ __forceinline__ float langevin(float k)
{
    if (k < 1e-2f) return k * (1.f / 3.f) - k * k * k * (1.f / 45.f);
    return 1.f / tanhf(k) - 1.f / k;
}

// acc[i][j] (output k = 4 ty + i, samples 4 tx + j) += sum_c w[k][c] in[c][sample], c ascending
// (the order of the sampler's forward pass); w: rows of `ld` floats, in: [n][kAP], n a multiple
// of 4.
__device__ __forceinline__ void tile_forward(float (&acc)[4][4], const float *w, int ld,
                                             const float *in, int n, int ty, int tx)
{
#pragma unroll 2
    for (int c = 0; c < n; c += 4) {
        float4 wv[4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
            wv[i] = *reinterpret_cast<const float4 *>(w + (4 * ty + i) * ld + c);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const float4 v = *reinterpret_cast<const float4 *>(in + (c + u) * kAP + 4 * tx);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float wu = u == 0 ? wv[i].x : u == 1 ? wv[i].y : u == 2 ? wv[i].z : wv[i].w;
                acc[i][0] = fmaf(wu, v.x, acc[i][0]);
                acc[i][1] = fmaf(wu, v.y, acc[i][1]);
                acc[i][2] = fmaf(wu, v.z, acc[i][2]);
                acc[i][3] = fmaf(wu, v.w, acc[i][3]);
            }
        }
    }
}

// acc[i][j] (input c = 4 ty + i, samples 4 tx + j) += sum_k w[k][c] d[k][sample].
__device__ __forceinline__ void tile_backward(float (&acc)[4][4], const float *w, const float *d,
                                              int ty, int tx)
{
#pragma unroll 4
    for (int k = 0; k < H; ++k) {
        const float4 wk = *reinterpret_cast<const float4 *>(w + k * kWP + 4 * ty);
        const float4 v = *reinterpret_cast<const float4 *>(d + k * kAP + 4 * tx);
        const float ws[4] = {wk.x, wk.y, wk.z, wk.w}, vs[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(ws[i], vs[j], acc[i][j]);
    }
}

// A layer's BF16 weights [rows][cols] as FP32 rows of `ld` floats (zeros past a row's end), eight
// at a time where the caller's pointer is 16-byte aligned and no eight cross a gap between rows
// (rows * cols is a multiple of eight); else one by one, from any address.
__device__ __forceinline__ void load_weights(float *dst, int ld, const __nv_bfloat16 *src, int rows,
                                             int cols, int t, int nt)
{
    const bool dense = ld == cols;
    if ((dense || cols % 8 == 0) && (reinterpret_cast<uintptr_t>(src) & 15) == 0) {
        for (int e = t; e < rows * cols / 8; e += nt) {
            const uint4 v = __ldg(reinterpret_cast<const uint4 *>(src) + e);
            const int i = 8 * e;
            const uint32_t u[4] = {v.x, v.y, v.z, v.w};
            float4 f[2];
            float *fp = reinterpret_cast<float *>(f);
#pragma unroll
            for (int k = 0; k < 4; ++k) {   // BF16 is the high half of an FP32
                fp[2 * k] = __uint_as_float(u[k] << 16);
                fp[2 * k + 1] = __uint_as_float(u[k] & 0xffff0000u);
            }
            float4 *o = reinterpret_cast<float4 *>(dst + (dense ? i : i / cols * ld + i % cols));
            o[0] = f[0];
            o[1] = f[1];
        }
    } else {
        for (int e = t; e < rows * ld; e += nt) {
            const int r = e / ld, c = e - r * ld;
            dst[e] = c < cols ? __bfloat162float(src[r * cols + c]) : 0.f;
        }
    }
}

// g[i][j] += sum over the tile's samples of d[k_i] v[c_j], k_i = ty + 16 i, c_j = tx + 16 j
// (columns from n_c on are left out).  The tile's 64 terms are summed by themselves and added
// once: a running sum over all of a block's tiles would lose the small terms of later ones.
__device__ __forceinline__ void tile_grad(float (&g)[4][4], const float *d, const float *v, int n_c,
                                          int ty, int tx)
{
    float s[4][4] = {};
#pragma unroll 4
    for (int m = 0; m < kTile; m += 4) {
        float4 a[4], b[4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
            a[i] = *reinterpret_cast<const float4 *>(d + (ty + 16 * i) * kAP + m);
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (16 * j < n_c)
                b[j] = *reinterpret_cast<const float4 *>(v + min(tx + 16 * j, n_c - 1) * kAP + m);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (16 * j < n_c)
                    s[i][j] = fmaf(a[i].w, b[j].w,
                                   fmaf(a[i].z, b[j].z,
                                        fmaf(a[i].y, b[j].y, fmaf(a[i].x, b[j].x, s[i][j]))));
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) g[i][j] += s[i][j];
}

// Shared memory (floats) of the training kernel.
__host__ __device__ constexpr int lg_smem_floats(int nin, int depth)
{
    return H * pad4(nin) + (depth - 1) * H * kWP + 4 * H + (pad4(nin) + 2 * depth * H + 4) * kAP;
}

// Bound by shared-memory reads per FMA and, at the usual batch of 16384, by two short waves:
// a 4 x 4 register tile reads two 16-byte words per 16 FMAs.  One sample per thread before
// (64 threads per block, activations in registers, fully unrolled layers) ran one warp per
// scheduler from an instruction cache that did not hold its code.  Measured, a training step
// (two clears, this kernel, Adam) of 16384 pairs, two layers: 112 -> 34 us, of which this
// kernel 95 -> 24; of 1482 pairs 112 -> 30 us.
template <int DEPTH>
__global__ void __launch_bounds__(kLG) loss_grad_kernel(MlpView net, int64_t n,
                                                        const float *__restrict__ x,
                                                        const float *__restrict__ y,
                                                        float *__restrict__ grad,
                                                        double *__restrict__ loss)
{
    const int nin = net.n_in;
    extern __shared__ __align__(16) float sm[];
    const int ninp = pad4(nin);
    float *W1 = sm;                                 // [H][ninp]
    float *Wh = W1 + H * ninp;                      // [DEPTH - 1][H][kWP]
    float *W3 = Wh + (DEPTH - 1) * H * kWP;         // [4][H]
    float *Xs = W3 + 4 * H;                         // [ninp][kAP]
    float *Hs = Xs + ninp * kAP;                    // [DEPTH][H][kAP] activations
    float *Ds = Hs + DEPTH * H * kAP;               // [DEPTH][H][kAP] deltas
    float *DO = Ds + DEPTH * H * kAP;               // [4][kAP] outputs, then their deltas

    const int t = threadIdx.x, ty = t >> 4, tx = t & 15;
    load_weights(W1, ninp, net.W1, H, nin, t, kLG);
    for (int e = t; e < (ninp - nin) * kTile; e += kLG)   // the padding inputs
        Xs[(nin + e / kTile) * kAP + e % kTile] = 0.f;
    load_weights(Wh, kWP, net.W2, H, H, t, kLG);
    if (DEPTH == 3) load_weights(Wh + (DEPTH - 2) * H * kWP, kWP, net.Wm, H, H, t, kLG);
    load_weights(W3, H, net.W3, 4, H, t, kLG);
    // gradient sums of this block: weights as tile_grad lays them out; W3 and biases by thread
    float g1[4][4] = {}, gh[DEPTH - 1][4][4] = {}, g3 = 0.f, gb[2] = {0.f, 0.f};
    double my_loss = 0.0;

    for (int64_t base = (int64_t)blockIdx.x * kTile; base < n; base += (int64_t)gridDim.x * kTile) {
        __syncthreads();   // weights ready; the previous tile's gradients are summed
        for (int e = t; e < kTile * nin; e += kLG) {
            const int m = e / nin, c = e - m * nin;
            Xs[c * kAP + m] = base + m < n ? x[base * nin + e] : 0.f;
        }
        __syncthreads();
        // forward
#pragma unroll
        for (int l = 0; l < DEPTH; ++l) {
            const float *bl = l == 0 ? net.b1 : l == 1 ? net.b2 : net.bm;
            float acc[4][4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float b = __ldg(bl + 4 * ty + i);
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = b;
            }
            if (l == 0) tile_forward(acc, W1, ninp, Xs, ninp, ty, tx);
            else tile_forward(acc, Wh + (l - 1) * H * kWP, kWP, Hs + (l - 1) * H * kAP, H, ty, tx);
#pragma unroll
            for (int i = 0; i < 4; ++i)
                *reinterpret_cast<float4 *>(Hs + (l * H + 4 * ty + i) * kAP + 4 * tx) =
                    make_float4(tanhf(acc[i][0]), tanhf(acc[i][1]), tanhf(acc[i][2]),
                                tanhf(acc[i][3]));
            __syncthreads();
        }
        const float *Hl = Hs + (DEPTH - 1) * H * kAP;
        {
            const int q = t >> 6, m = t & 63;   // output q of sample m
            float a = __ldg(net.b3 + q);
#pragma unroll 16
            for (int c = 0; c < H; ++c) a = fmaf(W3[q * H + c], Hl[c * kAP + m], a);
            DO[q * kAP + m] = a;
        }
        __syncthreads();
        if (t < kTile) {
            const float o[4] = {DO[t], DO[kAP + t], DO[2 * kAP + t], DO[3 * kAP + t]};
            const int64_t s = base + t;
            float dO[4] = {0.f, 0.f, 0.f, 0.f};
            if (s < n) {
                const float yv[3] = {y[s * 3], y[s * 3 + 1], y[s * 3 + 2]};
                const float vn = sqrtf(fmaxf(o[0] * o[0] + o[1] * o[1] + o[2] * o[2], 1e-30f));
                const float mu[3] = {o[0] / vn, o[1] / vn, o[2] / vn};
                const float kap = softplus_f(o[3]) + 1e-4f;
                const float muy = mu[0] * yv[0] + mu[1] * yv[1] + mu[2] * yv[2];
                my_loss += (double)(-logf(kap) + 1.8378770664093453f + kap +
                                    log1pf(-expf(-2.f * kap)) - kap * muy);
                const float dk = langevin(kap) - muy;
                dO[3] = dk / (1.f + expf(-o[3]));  // d softplus / d o3 = sigmoid(o3)
                for (int c = 0; c < 3; ++c) dO[c] = -kap * (yv[c] - mu[c] * muy) / vn;
            }
            for (int q = 0; q < 4; ++q) DO[q * kAP + t] = dO[q];
        }
        __syncthreads();
        // deltas: the last hidden layer from the outputs, then down through the layers
        {
            float4 dv[4];
#pragma unroll
            for (int q = 0; q < 4; ++q)
                dv[q] = *reinterpret_cast<const float4 *>(DO + q * kAP + 4 * tx);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int k = 4 * ty + i;
                const float4 h = *reinterpret_cast<const float4 *>(Hl + k * kAP + 4 * tx);
                float4 g = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float w = W3[q * H + k];
                    g.x = fmaf(w, dv[q].x, g.x);
                    g.y = fmaf(w, dv[q].y, g.y);
                    g.z = fmaf(w, dv[q].z, g.z);
                    g.w = fmaf(w, dv[q].w, g.w);
                }
                *reinterpret_cast<float4 *>(Ds + ((DEPTH - 1) * H + k) * kAP + 4 * tx) =
                    make_float4(g.x * (1.f - h.x * h.x), g.y * (1.f - h.y * h.y),
                                g.z * (1.f - h.z * h.z), g.w * (1.f - h.w * h.w));
            }
        }
        __syncthreads();
#pragma unroll
        for (int l = DEPTH - 1; l >= 1; --l) {
            float acc[4][4] = {};
            tile_backward(acc, Wh + (l - 1) * H * kWP, Ds + l * H * kAP, ty, tx);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int c = 4 * ty + i;
                const float4 h =
                    *reinterpret_cast<const float4 *>(Hs + ((l - 1) * H + c) * kAP + 4 * tx);
                *reinterpret_cast<float4 *>(Ds + ((l - 1) * H + c) * kAP + 4 * tx) = make_float4(
                    acc[i][0] * (1.f - h.x * h.x), acc[i][1] * (1.f - h.y * h.y),
                    acc[i][2] * (1.f - h.z * h.z), acc[i][3] * (1.f - h.w * h.w));
            }
            // (this layer's weight gradients need no sync with the stores above)
            tile_grad(gh[l - 1], Ds + l * H * kAP, Hs + (l - 1) * H * kAP, H, ty, tx);
            __syncthreads();
        }
        tile_grad(g1, Ds, Xs, nin, ty, tx);
        {
            const int q = t >> 6, c = t & 63;   // W3[q][c]
            const float *dq = DO + q * kAP, *hc = Hl + c * kAP;
            float s = 0.f;
#pragma unroll 4
            for (int m = 0; m < kTile; m += 4) {
                const float4 d4 = *reinterpret_cast<const float4 *>(dq + m);
                const float4 h4 = *reinterpret_cast<const float4 *>(hc + m);
                s = fmaf(d4.w, h4.w, fmaf(d4.z, h4.z, fmaf(d4.y, h4.y, fmaf(d4.x, h4.x, s))));
            }
            g3 += s;
        }
        // biases: DEPTH x H hidden, then 4 outputs
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int r = t + u * kLG;
            if (r < DEPTH * H + 4) {
                const float *d = r < DEPTH * H ? Ds + r * kAP : DO + (r - DEPTH * H) * kAP;
                float g = 0.f;
                for (int m = 0; m < kTile; m += 4) {
                    const float4 d4 = *reinterpret_cast<const float4 *>(d + m);
                    g += (d4.x + d4.y) + (d4.z + d4.w);
                }
                gb[u] += g;
            }
        }
    }
    // packed layout [W1][b1] then per further hidden layer [W][b], then [W3][b3]
    auto put = [&](int e, float v) {
        if (v != 0.f) atomicAdd(&grad[e], v);
    };
    const int o2 = H * nin + H;   // start of the second hidden layer
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int k = ty + 16 * i, c = tx + 16 * j;
            if (c < nin) put(k * nin + c, g1[i][j]);
#pragma unroll
            for (int l = 1; l < DEPTH; ++l)
                put(o2 + (l - 1) * (H * H + H) + k * H + c, gh[l - 1][i][j]);
        }
    const int o3 = o2 + (DEPTH - 1) * (H * H + H);
    put(o3 + t, g3);
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int r = t + u * kLG;
        if (r < H) put(H * nin + r, gb[u]);
        else if (r < DEPTH * H) put(o2 + (r / H - 1) * (H * H + H) + H * H + r % H, gb[u]);
        else if (r < DEPTH * H + 4) put(o3 + 4 * H + r - DEPTH * H, gb[u]);
    }
    if (t < kTile) {
        for (int o = 16; o > 0; o >>= 1) my_loss += __shfl_xor_sync(0xffffffffu, my_loss, o);
        if ((t & 31) == 0) atomicAdd(loss, my_loss);
    }
}

// Position of parameter e of the packed vector in the packed BF16 weight buffer; -1 for
// biases.  *fan receives fan_in + fan_out of the weight's layer.
__device__ __forceinline__ int64_t weight_slot(int64_t e, int nin, int depth, int *fan)
{
    int64_t o = 0, w = 0;   // start of the layer in the parameters / in the BF16 buffer
    *fan = 0;
    if (e < o + (int64_t)H * nin) {
        *fan = nin + H;
        return w + (e - o);
    }
    o += (int64_t)H * nin + H;
    w += (int64_t)H * nin;
    if (e < o) return -1;   // b1
    for (int l = 1; l < depth; ++l) {
        if (e < o + H * H) {
            *fan = 2 * H;
            return w + (e - o);
        }
        o += H * H + H;
        w += H * H;
        if (e < o) return -1;
    }
    if (e < o + 4 * H) {
        *fan = H + 4;
        return w + (e - o);
    }
    return -1;              // b3
}

__global__ void adam_kernel(float *__restrict__ p, const float *__restrict__ g, float scale,
                            float *__restrict__ m, float *__restrict__ v, int64_t P, int nin,
                            int depth, float lr, float b1, float b2, float eps, float c1, float c2,
                            __nv_bfloat16 *__restrict__ wb)
{
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= P) return;
    const float gr = g[e] * scale;
    const float mm = b1 * m[e] + (1.f - b1) * gr;
    const float vv = b2 * v[e] + (1.f - b2) * gr * gr;
    m[e] = mm;
    v[e] = vv;
    const float np = p[e] - lr * (mm / c1) / (sqrtf(vv / c2) + eps);
    p[e] = np;
    int fan = 0;
    const int64_t w = weight_slot(e, nin, depth, &fan);
    if (w >= 0) wb[w] = __float2bfloat16_rn(np);
}

// Glorot-uniform weights (U(-a, a), a = sqrt(6 / (fan_in + fan_out))) from one Philox draw
// per parameter (counter = its index, key = the seed), zero biases; the BF16 copy beside.
__global__ void init_kernel(float *__restrict__ p, int64_t P, int nin, int depth, uint32_t k0,
                            uint32_t k1, __nv_bfloat16 *__restrict__ wb)
{
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= P) return;
    int fan = 0;
    const int64_t w = weight_slot(e, nin, depth, &fan);
    float v = 0.f;
    if (w >= 0) {
        const U4 r = philox4x32_10(U4{(uint32_t)e, (uint32_t)(e >> 32), 0x6D6C7069u, 0u}, k0, k1);
        const float a = sqrtf(6.f / (float)fan);
        v = a * (2.f * u01(r.x) - 1.f);
    }
    p[e] = v;
    if (w >= 0 && wb) wb[w] = __float2bfloat16_rn(v);
}

__global__ void bf16_kernel(const float *__restrict__ p, int64_t P, int nin, int depth,
                            __nv_bfloat16 *__restrict__ wb)
{
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= P) return;
    int fan = 0;
    const int64_t w = weight_slot(e, nin, depth, &fan);
    if (w >= 0) wb[w] = __float2bfloat16_rn(p[e]);
}

}  // namespace
}  // namespace asd

using namespace asd;

extern "C" {

int64_t asd_mlp_param_count(int n_in, int depth)
{
    return shape_ok(n_in, depth) ? n_params(n_in, depth) : 0;
}
int64_t asd_mlp_param_count_bf16(int n_in, int depth)
{
    return shape_ok(n_in, depth) ? n_weights(n_in, depth) : 0;
}

int asd_mlp_gather(const asd_system *sys, int n_samples, const float *spins, float *x, float *y,
                   void *stream)
{
    ASD_CHECK_ARG(sys && spins && x && y, "null argument");
    ASD_CHECK_ARG(sys->n_sites >= 1 && sys->z >= 1 && sys->z <= kMlpMaxIn / 3 && sys->nbr,
                  "bad system (z must be 1..8)");
    ASD_CHECK_ARG(n_samples >= 1, "bad n_samples");
    const int64_t n = sys->n_sites * n_samples;
    gather_kernel<<<(unsigned)((n + 255) / 256), 256, 0, (cudaStream_t)stream>>>(
        sys->n_sites, n_samples, sys->z, sys->nbr, spins, x, y);
    ASD_CUDA_TRY(cudaGetLastError());
    return ASD_OK;
}

int asd_mlp_loss_grad(const asd_mlp *net, int64_t n, const float *x, const float *y, float *grad,
                      double *loss, void *stream)
{
    ASD_CHECK_ARG(net && x && y && grad && loss, "null argument");
    const int depth = mlp_depth(*net);
    ASD_CHECK_ARG(net->n_hidden == kMlpHidden && shape_ok(net->n_in, depth),
                  "network shape must be [n_in <= 24 -> 64 (x2 or x3) -> 4]");
    ASD_CHECK_ARG(net->W1 && net->W2 && net->W3 && net->b1 && net->b2 && net->b3, "null weights");
    ASD_CHECK_ARG(depth == 2 || (net->Wm && net->bm), "null weights of the third layer");
    ASD_CHECK_ARG(n >= 0, "bad n");
    if (n == 0) return ASD_OK;
    const int nin = net->n_in;
    const size_t smem = sizeof(float) * (size_t)lg_smem_floats(nin, depth);
    auto k = depth == 2 ? loss_grad_kernel<2> : loss_grad_kernel<3>;
    ASD_CUDA_TRY(allow_smem(k, sizeof(float) * (size_t)lg_smem_floats(kMlpMaxIn, depth)));
    int dev = 0, sms = 0;
    ASD_CUDA_TRY(cudaGetDevice(&dev));
    ASD_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    // as many resident blocks per SM as shared memory allows (two of a two-layer network, one
    // of a three-layer network)
    int smem_sm = 0;
    ASD_CUDA_TRY(cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev));
    int per_sm = smem_sm / (int)(smem + 1024);
    per_sm = per_sm < 1 ? 1 : (per_sm > 2 ? 2 : per_sm);
    const int64_t tiles = (n + kTile - 1) / kTile;
    const int64_t blocks = tiles < (int64_t)sms * per_sm ? tiles : (int64_t)sms * per_sm;
    k<<<(unsigned)blocks, kLG, smem, (cudaStream_t)stream>>>(mlp_view(*net), n, x, y, grad, loss);
    ASD_CUDA_TRY(cudaGetLastError());
    return ASD_OK;
}

int asd_mlp_adam_step(float *params, const float *grad, float grad_scale, float *m, float *v,
                      int n_in, int depth, float lr, float beta1, float beta2, float eps,
                      int step, uint16_t *w_bf16, void *stream)
{
    ASD_CHECK_ARG(params && grad && m && v && w_bf16, "null argument");
    ASD_CHECK_ARG(shape_ok(n_in, depth) && step >= 1, "bad n_in, depth or step");
    const int64_t P = n_params(n_in, depth);
    const float c1 = 1.f - powf(beta1, (float)step), c2 = 1.f - powf(beta2, (float)step);
    adam_kernel<<<(unsigned)((P + 255) / 256), 256, 0, (cudaStream_t)stream>>>(
        params, grad, grad_scale, m, v, P, n_in, depth, lr, beta1, beta2, eps, c1, c2,
        reinterpret_cast<__nv_bfloat16 *>(w_bf16));
    ASD_CUDA_TRY(cudaGetLastError());
    return ASD_OK;
}

int asd_mlp_init(float *params, int n_in, int depth, uint64_t seed, uint16_t *w_bf16,
                 void *stream)
{
    ASD_CHECK_ARG(params, "null argument");
    ASD_CHECK_ARG(shape_ok(n_in, depth), "bad n_in (3..24) or depth (2, 3)");
    const int64_t P = n_params(n_in, depth);
    init_kernel<<<(unsigned)((P + 255) / 256), 256, 0, (cudaStream_t)stream>>>(
        params, P, n_in, depth, (uint32_t)seed, (uint32_t)(seed >> 32),
        reinterpret_cast<__nv_bfloat16 *>(w_bf16));
    ASD_CUDA_TRY(cudaGetLastError());
    return ASD_OK;
}

int asd_mlp_weights_bf16(const float *params, int n_in, int depth, uint16_t *w_bf16,
                         void *stream)
{
    ASD_CHECK_ARG(params && w_bf16, "null argument");
    ASD_CHECK_ARG(shape_ok(n_in, depth), "bad n_in (3..24) or depth (2, 3)");
    const int64_t P = n_params(n_in, depth);
    bf16_kernel<<<(unsigned)((P + 255) / 256), 256, 0, (cudaStream_t)stream>>>(
        params, P, n_in, depth, reinterpret_cast<__nv_bfloat16 *>(w_bf16));
    ASD_CUDA_TRY(cudaGetLastError());
    return ASD_OK;
}

}  // extern "C"
