// Learned von Mises-Fisher proposal network: the view the kernels read, and what its output
// means.
//
// x (the 3z neighbour spin components) -> h1 = tanh(W1 x + b1) -> h2 = tanh(W2 h1 + b2)
// [-> h3 = tanh(Wm h2 + bm) with three hidden layers] -> o = W3 h_last + b3;  mean
// direction mu = o[0:3] / |o[0:3]|,  kappa = softplus(o[3]).
// Weights are BF16 (row-major [out][in]), biases and all arithmetic FP32.
#pragma once

#include <cuda_bf16.h>

#include "../../include/asd.h"

namespace asd {

constexpr int kMlpHidden = 64;
constexpr int kMlpMaxIn = 24;
constexpr int kMlpMaxDepth = 3;   // hidden layers: 2 or 3

struct MlpView {
    int n_in;
    int depth;                       // hidden layers (2 or 3)
    const __nv_bfloat16 *W1, *W2, *Wm, *W3;
    const float *b1, *b2, *bm, *b3;
};

inline int mlp_depth(const asd_mlp &m) { return m.depth == 0 ? 2 : m.depth; }

inline MlpView mlp_view(const asd_mlp &m)
{
    MlpView v;
    v.n_in = m.n_in;
    v.depth = mlp_depth(m);
    v.W1 = reinterpret_cast<const __nv_bfloat16 *>(m.W1);
    v.W2 = reinterpret_cast<const __nv_bfloat16 *>(m.W2);
    v.Wm = reinterpret_cast<const __nv_bfloat16 *>(m.Wm);
    v.W3 = reinterpret_cast<const __nv_bfloat16 *>(m.W3);
    v.b1 = m.b1;
    v.b2 = m.b2;
    v.bm = m.bm;
    v.b3 = m.b3;
    return v;
}

__device__ __forceinline__ float softplus_f(float x) { return x > 20.f ? x : log1pf(expf(x)); }

// Mean direction and concentration of the proposal from the network's output.
__device__ __forceinline__ void mlp_vmf_of(const float *o, float *mu, float *kappa)
{
    const float inv = rsqrtf(fmaxf(o[0] * o[0] + o[1] * o[1] + o[2] * o[2], 1e-30f));
    mu[0] = o[0] * inv;
    mu[1] = o[1] * inv;
    mu[2] = o[2] * inv;
    *kappa = softplus_f(o[3]) + 1e-4f;
}

}  // namespace asd
