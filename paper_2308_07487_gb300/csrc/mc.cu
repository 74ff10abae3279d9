// Classical Monte Carlo for Heisenberg spins (Section 2.1), checkerboard-parallel.
//
// Metropolis: a trial spin is drawn uniformly on the sphere, or inside a cone about the
// current spin whose half-angle adapts between sweeps (the paper keeps the acceptance
// rate at least 20 %); it is accepted with probability min(1, exp(-beta dE)).
// Heat-bath: the new spin is drawn from the exact conditional of the terms linear in S,
// p(S) ~ exp(-beta S.h), a von Mises-Fisher law with mean -h/|h| and concentration
// beta|h|; with single-ion anisotropy the draw is a Metropolis-Hastings proposal accepted
// with min(1, exp(beta A (Sz_new^2 - Sz_old^2))), which keeps the chain exact.
// Energy change of a move: dE = (S' - S).h - A (S'z^2 - Sz^2), h = sum_j J_ij S_j +
// sum_j D_ij x S_j - Hz z^ (Eq. 1).
// Learned: a small MLP maps the neighbour spins to a vMF proposal; the
// Metropolis-Hastings ratio exp(-beta dE) q(S_old)/q(S_new) keeps the chain exact.
//
// Sites of one colour have no neighbours of that colour, so a colour is updated in
// parallel without races.  Randomness: Philox4x32-10 (Salmon et al., SC'11) keyed
// by the seed, counter (sweep, colour, sample, site); or caller-supplied uniforms.
#include <algorithm>

#include <cuda_bf16.h>

#include "asd_internal.h"
#include "grid_barrier.cuh"
#include "mlp.cuh"
#include "philox.cuh"

namespace asd {
namespace {

struct MCArgs {
    int64_t N;
    int S;
    int z;
    const int *nbr;
    const float *J;
    float Hz;
    const float *D;     // [N][z][3] DM vectors or null
    float A;            // single-ion anisotropy
    float beta;
    int proposal;
    const int *sites;   // this colour's sites
    int64_t n_sites_c;
    uint64_t seed;
    uint64_t ctr;       // counter + sweep
    int color;
    const float *uni;   // optional [S][N][4] uniforms of this sweep
    const float *cone;  // device cone half-angle
    unsigned long long *stats;  // [2]: proposed, accepted
    MlpView net;
};

__device__ __forceinline__ float3 f3(const float *p) { return make_float3(p[0], p[1], p[2]); }

// The arithmetic of a move is written out in rounded products, sums and FMAs: left to the
// compiler, which products it fuses depends on the shape of the surrounding code, and a chain
// follows the last bit of every spin (and of every decision).
__device__ __forceinline__ float dot3(float ax, float ay, float az, float bx, float by, float bz)
{
    return __fmaf_rn(az, bz, __fmaf_rn(ax, bx, __fmul_rn(ay, by)));
}
// a b - c d
__device__ __forceinline__ float det2(float a, float b, float c, float d)
{
    return __fmaf_rn(a, b, -__fmul_rn(c, d));
}

// unit vectors e1, e2 with (e1, e2, m) right-handed; the same rule as the oracle
__device__ __forceinline__ void frame_of(float3 m, float3 &e1, float3 &e2)
{
    // (0, 0, 1) x m, or (1, 0, 0) x m near the pole
    const float3 c = fabsf(m.z) < 0.9f ? make_float3(-m.y, m.x, 0.f) : make_float3(0.f, -m.z, m.y);
    const float inv = rsqrtf(dot3(c.x, c.y, c.z, c.x, c.y, c.z));
    e1 = make_float3(__fmul_rn(c.x, inv), __fmul_rn(c.y, inv), __fmul_rn(c.z, inv));
    e2 = make_float3(det2(m.y, e1.z, m.z, e1.y), det2(m.z, e1.x, m.x, e1.z),
                     det2(m.x, e1.y, m.y, e1.x));
}

// the unit vector at cos(angle) = c from m and azimuth phi
__device__ __forceinline__ float3 around(float3 m, float c, float phi)
{
    float3 e1, e2;
    frame_of(m, e1, e2);
    const float s = sqrtf(fmaxf(0.f, __fmaf_rn(-c, c, 1.f)));
    float sp, cp;
    sincosf(phi, &sp, &cp);
    auto comp = [&](float mm, float a, float b) {
        return __fmaf_rn(c, mm, __fmul_rn(s, __fmaf_rn(cp, a, __fmul_rn(sp, b))));
    };
    return make_float3(comp(m.x, e1.x, e2.x), comp(m.y, e1.y, e2.y), comp(m.z, e1.z, e2.z));
}

// cos of the angle to the mean for vMF(kappa) in 3D, from u in (0, 1]
__device__ __forceinline__ float vmf_w(float kappa, float u)
{
    if (kappa < 1e-6f) return __fmaf_rn(-2.f, u, 1.f);
    const float e = expf(__fmul_rn(-2.f, kappa));
    return fmaxf(-1.f, __fadd_rn(1.f, logf(__fmaf_rn(__fadd_rn(1.f, -u), e, u)) / kappa));
}

// Neighbour k's part of the local field: J S_j, and D_ij x S_j with DM vectors (d: the directed
// bond's, or null).
__device__ __forceinline__ void add_bond(float3 &h, float J, float3 sj, const float *__restrict__ d)
{
    h.x = __fmaf_rn(J, sj.x, h.x);
    h.y = __fmaf_rn(J, sj.y, h.y);
    h.z = __fmaf_rn(J, sj.z, h.z);
    if (d) {
        const float dx = __ldg(d), dy = __ldg(d + 1), dz = __ldg(d + 2);
        h.x = __fadd_rn(h.x, det2(dy, sj.z, dz, sj.y));
        h.y = __fadd_rn(h.y, det2(dz, sj.x, dx, sj.z));
        h.z = __fadd_rn(h.z, det2(dx, sj.y, dy, sj.x));
    }
}

// Local field of site i, the part linear in S_i, from a sample's spins; with nb also the
// neighbour spins (zeros for empty slots).
__device__ __forceinline__ float3 mc_field(const MCArgs &a, const float *Ys, int64_t i, float *nb)
{
    float3 h = make_float3(0.f, 0.f, -a.Hz);
    for (int k = 0; k < a.z; ++k) {
        const int j = __ldg(a.nbr + i * a.z + k);
        const float3 sj = j >= 0 ? f3(Ys + 3 * (int64_t)j) : make_float3(0.f, 0.f, 0.f);
        if (j >= 0)
            add_bond(h, __ldg(a.J + i * a.z + k), sj, a.D ? a.D + (i * a.z + k) * 3 : nullptr);
        if (nb) {
            nb[3 * k] = sj.x;
            nb[3 * k + 1] = sj.y;
            nb[3 * k + 2] = sj.z;
        }
    }
    return h;
}

// The four uniforms of site i of sample s in one sweep (ctr = counter + sweep; uni = the
// caller's numbers of the sweep, or null) and colour.
__device__ __forceinline__ void mc_uniforms(const MCArgs &a, const float *uni, uint64_t ctr,
                                            int color, int s, int64_t i, float (&u)[4])
{
    if (uni) {
        const float *up = uni + ((int64_t)s * a.N + i) * 4;
        u[0] = up[0]; u[1] = up[1]; u[2] = up[2]; u[3] = up[3];
    } else {
        const U4 r = philox4x32_10(U4{(uint32_t)i, (uint32_t)(i >> 32) ^ ((uint32_t)s << 8) ^
                                                       ((uint32_t)color << 28),
                                      (uint32_t)ctr, (uint32_t)(ctr >> 32)},
                                   (uint32_t)a.seed, (uint32_t)(a.seed >> 32));
        u[0] = u01(r.x); u[1] = u01(r.y); u[2] = u01(r.z); u[3] = u01(r.w);
    }
}

// Change of -A (S^z)^2 of a move, negated.
__device__ __forceinline__ float mc_daniso(const MCArgs &a, float3 old, float3 nw)
{
    return __fmul_rn(a.A, det2(nw.z, nw.z, old.z, old.z));
}

// Metropolis-Hastings decision on a move old -> nw with log q(old) - log q(new).
__device__ __forceinline__ bool mc_accept(const MCArgs &a, float3 h, float3 old, float3 nw,
                                          float logq_ratio, float u)
{
    const float dE =
        __fadd_rn(dot3(__fadd_rn(nw.y, -old.y), __fadd_rn(nw.x, -old.x), __fadd_rn(nw.z, -old.z),
                       h.y, h.x, h.z),
                  -mc_daniso(a, old, nw));
    const float la = __fmaf_rn(-a.beta, dE, logq_ratio);
    return la >= 0.f || u < expf(la);
}

constexpr float kTwoPi = 6.283185307179586f;

// One Metropolis (trial cone of half-angle acos(cmin)) or heat-bath move of a site in field h;
// true when accepted.
__device__ __forceinline__ bool mc_move(const MCArgs &a, float3 h, float3 old, const float (&u)[4],
                                        float cmin, float3 &nw)
{
    const float phi = __fmul_rn(kTwoPi, u[1]);
    if (a.proposal == ASD_HEATBATH) {
        const float hn = sqrtf(dot3(h.x, h.y, h.z, h.x, h.y, h.z));
        const float kappa = __fmul_rn(a.beta, hn);
        const float3 m = hn > 0.f ? make_float3(-h.x / hn, -h.y / hn, -h.z / hn)
                                  : make_float3(0.f, 0.f, 1.f);
        nw = around(m, vmf_w(kappa, u[0]), phi);
        const float la = __fmul_rn(a.beta, mc_daniso(a, old, nw));
        return la >= 0.f || u[2] < expf(la);
    }
    nw = around(old, __fadd_rn(1.f, -__fmul_rn(u[0], __fadd_rn(1.f, -cmin))), phi);
    return mc_accept(a, h, old, nw, 0.f, u[2]);
}

__device__ __forceinline__ float cone_cos(float cone)
{
    return cone <= 0.f || cone >= 3.14159265f ? -1.f : cosf(cone);
}

// cone <- cone * clamp(acceptance / 0.5, 0.5, 2), at most pi
__device__ __forceinline__ float next_cone(float cone, unsigned long long prop,
                                           unsigned long long acc)
{
    if (prop == 0) return cone;
    float r = (float)acc / (float)prop / 0.5f;
    r = fminf(2.f, fmaxf(0.5f, r));
    const float c = cone <= 0.f ? 3.14159265f : cone;
    return fminf(3.14159265f, c * r);
}

// Block totals of proposed / accepted moves into the sweep's counters.
__device__ __forceinline__ void mc_count(unsigned prop, unsigned acc, unsigned long long *stats)
{
    __shared__ unsigned int cnt[2];
    if (threadIdx.x < 2) cnt[threadIdx.x] = 0;
    __syncthreads();
    for (int o = 16; o > 0; o >>= 1) {
        prop += __shfl_xor_sync(0xffffffffu, prop, o);
        acc += __shfl_xor_sync(0xffffffffu, acc, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&cnt[0], prop);
        atomicAdd(&cnt[1], acc);
    }
    __syncthreads();
    if (threadIdx.x == 0 && cnt[0]) {
        atomicAdd(&stats[0], (unsigned long long)cnt[0]);
        atomicAdd(&stats[1], (unsigned long long)cnt[1]);
    }
}

// Metropolis and heat-bath: one thread per site of a colour.
__global__ void mc_color_kernel(MCArgs a, float *__restrict__ spins)
{
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    bool prop = false, acc = false;
    if (g < a.n_sites_c * a.S) {
        const int s = (int)(g / a.n_sites_c);
        const int64_t i = a.sites[g % a.n_sites_c];
        float *Ys = spins + (int64_t)s * a.N * 3;
        const float3 h = mc_field(a, Ys, i, nullptr);
        float u[4];
        mc_uniforms(a, a.uni, a.ctr, a.color, s, i, u);
        const float3 old = f3(Ys + 3 * i);
        float3 nw;
        prop = true;
        acc = mc_move(a, h, old, u, cone_cos(*a.cone), nw);
        if (acc) {
            Ys[3 * i] = nw.x;
            Ys[3 * i + 1] = nw.y;
            Ys[3 * i + 2] = nw.z;
        }
    }
    mc_count(prop, acc, a.stats);
}

// ---------------------------------------------------------------------------------------
// Persistent Metropolis / heat-bath sweeps
// ---------------------------------------------------------------------------------------
constexpr int kMcMaxColors = 16;
constexpr int kMcSweepsPerLaunch = 4096;   // other streams' work gets in between
constexpr int kMcLocalSites = 2048, kMcLocalMost = 4096;

struct MCRun {
    MCArgs a;                         // (per-colour fields unused)
    float *spins;
    int n_colors;
    int64_t off[kMcMaxColors + 1];    // colour offsets into a.sites
    int n_sweeps;
    int adapt;
    float *cone;                      // in and out
    unsigned long long *total;        // [2] proposed, accepted
    unsigned long long *slots;        // grid route, adapt: [4] accepted per sweep, zero at launch
    unsigned *bar;                    // grid route: barrier count, zero at launch
    int *err;
};

// All sweeps of a call in one launch.  A colour's update is a few hundred dependent
// instructions per site, so launches (5 us per colour for systems of some ten thousand sites,
// and one more per sweep for the counters) took most of the time.  LOCAL: a block per sample,
// spins in shared memory, a block barrier between colours.  Else a cooperative launch with a
// grid barrier between colours; what does not depend on the other colours' spins (site,
// bonds, uniforms, own spin) is fetched before the barrier.  Measured against a launch per
// colour and one per sweep: 40^3 sites, adaptive cone, 100 sweeps, 1.64 -> 0.77 ms (8.2 ->
// 3.9 us per colour, of which the barrier about 2); 36^2, 96 sweeps, 1157 -> 355 us; 13
// samples of 20^2, 49 sweeps, 748 -> 113 us.
template <int Z, bool LOCAL>
__global__ void __launch_bounds__(1024, 1) mc_persistent(const __grid_constant__ MCRun r)
{
    extern __shared__ __align__(16) uint8_t mc_smem[];
    __shared__ unsigned cnt;
    const MCArgs &a = r.a;
    const int tid = threadIdx.x, nt = blockDim.x;
    float4 *sm = reinterpret_cast<float4 *>(mc_smem);   // LOCAL: the sample's spins
    const int64_t N = a.N;
    if (LOCAL) {
        const float *src = r.spins + (int64_t)blockIdx.x * N * 3;
        for (int i = tid; i < (int)N; i += nt)
            sm[i] = make_float4(src[3 * i], src[3 * i + 1], src[3 * i + 2], 0.f);
        __syncthreads();
    }
    float cone = *r.cone;
    float cmin = cone_cos(cone);
    const int64_t first = LOCAL ? tid : (int64_t)blockIdx.x * nt + tid;
    const int64_t step = LOCAL ? nt : (int64_t)gridDim.x * nt;
    unsigned target = 0;
    unsigned long long accepted = 0;   // this thread's (adapt: block 0's totals over sweeps)

    // one site's bonds, own spin and uniforms
    constexpr int ZR = Z > 0 ? Z : 1;
    struct Site {
        int s;
        int64_t i;
        int nb[ZR];
        float J[ZR], u[4];
        float3 old;
        bool on;
    };
    auto spin = [&](int s, int64_t j) {
        if (LOCAL) {
            const float4 v = sm[j];
            return make_float3(v.x, v.y, v.z);
        }
        return f3(r.spins + ((int64_t)s * N + j) * 3);
    };
    auto fetch = [&](Site &q, int sw, int c, int64_t g) {
        const int64_t nc = r.off[c + 1] - r.off[c], n = LOCAL ? nc : nc * a.S;
        q.on = g < n;
        if (!q.on) return;
        q.s = LOCAL ? (int)blockIdx.x : (int)(g / nc);
        q.i = __ldg(a.sites + r.off[c] + (LOCAL ? g : g - (int64_t)q.s * nc));
        if (Z > 0)
#pragma unroll
            for (int k = 0; k < ZR; ++k) {
                q.nb[k] = __ldg(a.nbr + q.i * Z + k);
                q.J[k] = __ldg(a.J + q.i * Z + k);
            }
        mc_uniforms(a, a.uni ? a.uni + (size_t)sw * a.S * N * 4 : nullptr, a.ctr + (uint64_t)sw, c,
                    q.s, q.i, q.u);
        q.old = spin(q.s, q.i);
    };
    auto update = [&](const Site &q) -> unsigned {
        if (!q.on) return 0u;
        float3 h = make_float3(0.f, 0.f, -a.Hz);
        if (Z > 0) {
            float3 sj[ZR];
#pragma unroll
            for (int k = 0; k < ZR; ++k) sj[k] = spin(q.s, q.nb[k] < 0 ? q.i : q.nb[k]);
#pragma unroll
            for (int k = 0; k < ZR; ++k)
                if (q.nb[k] >= 0)
                    add_bond(h, q.J[k], sj[k], a.D ? a.D + (q.i * Z + k) * 3 : nullptr);
        } else {
            for (int k = 0; k < a.z; ++k) {
                const int j = __ldg(a.nbr + q.i * a.z + k);
                if (j >= 0)
                    add_bond(h, __ldg(a.J + q.i * a.z + k), spin(q.s, j),
                             a.D ? a.D + (q.i * a.z + k) * 3 : nullptr);
            }
        }
        float3 nw;
        if (!mc_move(a, h, q.old, q.u, cmin, nw)) return 0u;
        if (LOCAL) {
            sm[q.i] = make_float4(nw.x, nw.y, nw.z, 0.f);
        } else {
            float *y = r.spins + ((int64_t)q.s * N + q.i) * 3;
            y[0] = nw.x;
            y[1] = nw.y;
            y[2] = nw.z;
        }
        return 1u;
    };
    // accepted moves of the block, on every thread
    auto block_sum = [&](unsigned v) {
        if (tid == 0) cnt = 0;
        __syncthreads();
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if ((tid & 31) == 0 && v) atomicAdd(&cnt, v);
        __syncthreads();
        return cnt;
    };

    Site q;
    fetch(q, 0, 0, first);
    for (int sw = 0; sw < r.n_sweeps; ++sw) {
        unsigned acc = 0;
        for (int c = 0; c < r.n_colors; ++c) {
            acc += update(q);
            const int64_t nc = r.off[c + 1] - r.off[c], n = LOCAL ? nc : nc * a.S;
            for (int64_t g = first + step; g < n; g += step) {
                fetch(q, sw, c, g);
                acc += update(q);
            }
            // the next colour's first site (its own spin belongs to its colour: this one's
            // updates do not touch it)
            const bool more = c + 1 < r.n_colors || sw + 1 < r.n_sweeps;
            const int c2 = c + 1 < r.n_colors ? c + 1 : 0, sw2 = c2 ? sw : sw + 1;
            const bool own_ready = r.n_colors > 1;   // (one colour: its own sites come next)
            if (more && own_ready) fetch(q, sw2, c2, first);
            if (c == r.n_colors - 1 && r.adapt && !LOCAL) {
                const unsigned b = block_sum(acc);
                if (tid == 0 && b) atomicAdd(&r.slots[sw & 3], (unsigned long long)b);
            }
            if (LOCAL) {
                __syncthreads();
            } else if (more || r.adapt) {
                target += gridDim.x;
                if (!grid_barrier(r.bar, target, r.err)) return;
            }
            if (more && !own_ready) fetch(q, sw2, c2, first);
        }
        if (r.adapt) {
            // acceptance of the sweep over all samples, the same number in every block
            unsigned long long all;
            if (LOCAL) {
                all = block_sum(acc);
                __syncthreads();   // (cnt is reused)
            } else {
                all = *(volatile unsigned long long *)&r.slots[sw & 3];
                // the slot after next was last read before this sweep's barrier
                if (blockIdx.x == 0 && tid == 0) r.slots[(sw + 2) & 3] = 0;
            }
            accepted += all;
            cone = next_cone(cone, (unsigned long long)N * a.S, all);
            cmin = cone_cos(cone);
        } else {
            accepted += acc;
        }
    }
    if (!r.adapt) {
        for (int o = 16; o > 0; o >>= 1) accepted += __shfl_xor_sync(0xffffffffu, accepted, o);
        if ((tid & 31) == 0 && accepted) atomicAdd(&r.total[1], accepted);
    } else if (blockIdx.x == 0 && tid == 0) {
        r.total[1] += accepted;
        *r.cone = cone;
    }
    if (blockIdx.x == 0 && tid == 0) r.total[0] += (unsigned long long)N * a.S * r.n_sweeps;
    if (LOCAL) {
        float *dst = r.spins + (int64_t)blockIdx.x * N * 3;
        for (int i = tid; i < (int)N; i += nt) {
            const float4 v = sm[i];
            dst[3 * i] = v.x;
            dst[3 * i + 1] = v.y;
            dst[3 * i + 2] = v.z;
        }
    }
}

typedef void (*MCKernel)(MCRun);
struct MCRoute {
    MCKernel k = nullptr;   // null: one launch per colour
    bool local = false;
    unsigned grid = 0, block = 0;
    size_t smem = 0;
};

// Where the sweeps run: a block per sample (local), a cooperative launch over all samples (grid,
// at most one block per SM), or a launch per colour.  Adaptive runs of several samples share
// one cone, so they take the grid.
//
// One block is soon slower than the device, so local up to kMcLocalSites sites: 64^2, one chain,
// one sweep 21.7 us in a block, 13.4 by the grid, 17.1 by a launch per colour, ten sweeps 106, 69
// and 121; 44^2 15.7, 13.3 and 17.4, 56.6, 69.2 and 129; 16^3 with 26 bonds and DM vectors, ten
// sweeps, 1510, 744 and 965.  Twice as many where the grid's threads would each have several
// sites of a colour (but not many, where the grid's better balance pays): 152 chains of 64^2,
// ten sweeps, 110, 162 and 274.  Not local: one sweep of more sites than the device takes at
// once (300000 chains of 64 sites 392, 280 and 358), and samples of less than a warp per
// colour, more of them than there are blocks (300000 of one site, ten sweeps, 1147, 97 and 121).
//
// A launch per colour has more threads and so more loads in flight, which is what many bonds
// need on more sites than the grid has threads: 26 bonds, 400 chains of 16^3, one sweep, 285 us
// by the grid, 247 by launches; 1000 chains, ten sweeps, 5080 local, 4730; 12 bonds with DM
// vectors, 1000 chains, ten sweeps, 4930 local, 4650 and 4330.  And one pass over one colour has
// nothing to keep between launches.
int mc_route(const MCArgs &a, const int64_t *off, int n_colors, int n_sweeps, int adapt, int sms,
             MCRoute *out)
{
    *out = MCRoute();
    if (n_colors > kMcMaxColors || a.proposal == ASD_LEARNED) return ASD_OK;
    int64_t widest = 0, passes = 0;
    for (int c = 0; c < n_colors; ++c) {
        widest = std::max(widest, off[c + 1] - off[c]);
        if (off[c + 1] > off[c]) passes += n_sweeps;
    }
    const int64_t full = 1024 * (int64_t)sms, load = widest * a.S;
    const bool filled = load > full / 4 * 3;
    if (filled && (a.z > 8 || (a.D && a.z > 6))) return ASD_OK;
    MCRoute r;
    const bool local = (a.N <= kMcLocalSites ||
                        (a.N <= kMcLocalMost && filled && load <= 4 * full)) &&
                       !(filled && n_sweeps == 1) && !(widest < 32 && a.S > 32 * sms);
    if (local && (!adapt || a.S == 1)) {
        r.local = true;
        r.k = a.z == 4   ? mc_persistent<4, true>
              : a.z == 6 ? mc_persistent<6, true>
                         : mc_persistent<0, true>;
        r.grid = (unsigned)a.S;
        r.block = (unsigned)std::min<int64_t>(1024, (widest + 31) / 32 * 32);
        r.smem = sizeof(float4) * (size_t)a.N;
        ASD_CUDA_TRY(allow_smem(r.k, sizeof(float4) * kMcLocalMost));
        *out = r;
        return ASD_OK;
    }
    if (passes <= 1) return ASD_OK;
    int dev = 0, coop = 0, per_sm = 0;
    ASD_CUDA_TRY(cudaGetDevice(&dev));
    ASD_CUDA_TRY(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev));
    if (!coop) return ASD_OK;
    r.k = a.z == 4 ? mc_persistent<4, false> : a.z == 6 ? mc_persistent<6, false>
                                                        : mc_persistent<0, false>;
    // spread a colour over all SMs, whole warps per block, at most 1024 threads
    const int64_t n = widest * a.S, per = (n + sms - 1) / sms;
    r.block = (unsigned)std::min<int64_t>(1024, std::max<int64_t>(128, (per + 31) / 32 * 32));
    r.grid = (unsigned)std::min<int64_t>(sms, (n + r.block - 1) / r.block);
    ASD_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, r.k, (int)r.block, 0));
    if ((int64_t)per_sm * sms >= r.grid) *out = r;
    return ASD_OK;
}

// Learned proposal: T sites per thread, the network's weights in shared memory as FP32.
// Bound by the instruction issue of the forward pass (5.1 thousand FMAs and 128 tanh per site
// and two layers) and by the weight reads: one 16-byte word serves 4 T FMAs of a thread, and
// a warp's broadcast read takes as long as four FMAs, so T = 2 where there are sites enough
// to fill the chip with it.  Activations stay in registers for the layer that reads them and
// pass through the thread's own column of shared memory between layers (so the loop over
// outputs is a loop and the code fits the instruction cache).  Every sum runs over its
// inputs in ascending order from the bias.  Measured against a thread per site with its
// activations in local memory and weights from global memory: eight 128^2 chains, 10 sweeps
// (65536 sites per colour), 3.24 -> 0.68 ms; 28 samples of 16^2, three layers, 5 sweeps,
// 1.81 -> 0.26 ms.
constexpr int kMlBlock = 128;
template <int NIN>
constexpr int ml_row() { return (NIN + 3) / 4 * 4; }   // floats per first-layer row
template <int NIN, int T>
constexpr size_t ml_smem(int depth)
{
    return sizeof(float) * ((size_t)kMlpHidden * ml_row<NIN>() +
                            (size_t)(depth - 1) * kMlpHidden * kMlpHidden + 4 * kMlpHidden +
                            (size_t)depth * kMlpHidden + 4 + (size_t)T * kMlpHidden * kMlBlock);
}

template <int NIN, int T>
__global__ void __launch_bounds__(kMlBlock, 2) mc_learned_kernel(MCArgs a, float *__restrict__ spins)
{
    constexpr int H = kMlpHidden, RW = ml_row<NIN>();
    extern __shared__ __align__(16) float ml_sm[];
    const MlpView &net = a.net;
    const int depth = net.depth, nin = net.n_in, tid = threadIdx.x;
    float *W1 = ml_sm;                            // [H][RW], zero padded
    float *Wh = W1 + H * RW;                      // [depth - 1][H][H]
    float *W3T = Wh + (depth - 1) * H * H;        // [H][4]
    float *bias = W3T + 4 * H;                    // [depth][H]
    float *b3 = bias + depth * H;                 // [4]
    float *act = b3 + 4;                          // [H][T][block]: this thread's column
    for (int e = tid; e < H * RW; e += kMlBlock) {
        const int k = e / RW, c = e - k * RW;
        W1[e] = c < nin ? __bfloat162float(net.W1[k * nin + c]) : 0.f;
    }
    for (int e = tid; e < H * H; e += kMlBlock) {
        Wh[e] = __bfloat162float(net.W2[e]);
        if (depth == 3) Wh[H * H + e] = __bfloat162float(net.Wm[e]);
    }
    for (int e = tid; e < 4 * H; e += kMlBlock)
        W3T[e] = __bfloat162float(net.W3[(e & 3) * H + (e >> 2)]);
    for (int e = tid; e < H; e += kMlBlock) {
        bias[e] = net.b1[e];
        bias[H + e] = net.b2[e];
        if (depth == 3) bias[2 * H + e] = net.bm[e];
    }
    if (tid < 4) b3[tid] = net.b3[tid];
    __syncthreads();

    unsigned prop = 0, acc = 0;
    const int64_t n = a.n_sites_c * a.S, groups = (n + T - 1) / T;
    for (int64_t g0 = (int64_t)blockIdx.x * kMlBlock + tid; g0 < groups;
         g0 += (int64_t)gridDim.x * kMlBlock) {
        int s[T];
        int64_t site[T];
        bool on[T];
        float3 h[T];
        float o[T][4];
        {
            float x[T][RW];
#pragma unroll
            for (int u = 0; u < T; ++u) {
                const int64_t g = g0 + u * groups;   // a warp's sites stay consecutive
                on[u] = g < n;
                const int64_t gc = on[u] ? g : g0;
                s[u] = (int)(gc / a.n_sites_c);
                site[u] = a.sites[gc % a.n_sites_c];
                float nb[kMlpMaxIn];
                h[u] = mc_field(a, spins + (int64_t)s[u] * a.N * 3, site[u], nb);
#pragma unroll
                for (int c = 0; c < RW; ++c) x[u][c] = c < nin ? nb[c] : 0.f;
            }
#pragma unroll 2
            for (int k = 0; k < H; ++k) {
                float v[T];
#pragma unroll
                for (int u = 0; u < T; ++u) v[u] = bias[k];
#pragma unroll
                for (int c = 0; c < RW; c += 4) {
                    const float4 w = *reinterpret_cast<const float4 *>(W1 + k * RW + c);
#pragma unroll
                    for (int u = 0; u < T; ++u) {
                        v[u] = fmaf(w.x, x[u][c], v[u]);
                        v[u] = fmaf(w.y, x[u][c + 1], v[u]);
                        v[u] = fmaf(w.z, x[u][c + 2], v[u]);
                        v[u] = fmaf(w.w, x[u][c + 3], v[u]);
                    }
                }
#pragma unroll
                for (int u = 0; u < T; ++u) act[(k * T + u) * kMlBlock + tid] = tanhf(v[u]);
            }
        }
#pragma unroll
        for (int u = 0; u < T; ++u)
#pragma unroll
            for (int q = 0; q < 4; ++q) o[u][q] = b3[q];
        for (int l = 1; l < depth; ++l) {
            float hv[T][H];
#pragma unroll
            for (int c = 0; c < H; ++c)
#pragma unroll
                for (int u = 0; u < T; ++u) hv[u][c] = act[(c * T + u) * kMlBlock + tid];
            const float *W = Wh + (l - 1) * H * H, *bl = bias + l * H;
            const bool out = l == depth - 1;
#pragma unroll 1
            for (int k = 0; k < H; k += 4) {
                float v[T][4];
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int u = 0; u < T; ++u) v[u][i] = bl[k + i];
#pragma unroll
                for (int c = 0; c < H; c += 4)
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float4 w = *reinterpret_cast<const float4 *>(W + (k + i) * H + c);
#pragma unroll
                        for (int u = 0; u < T; ++u) {
                            v[u][i] = fmaf(w.x, hv[u][c], v[u][i]);
                            v[u][i] = fmaf(w.y, hv[u][c + 1], v[u][i]);
                            v[u][i] = fmaf(w.z, hv[u][c + 2], v[u][i]);
                            v[u][i] = fmaf(w.w, hv[u][c + 3], v[u][i]);
                        }
                    }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float4 w3 = *reinterpret_cast<const float4 *>(W3T + 4 * (k + i));
#pragma unroll
                    for (int u = 0; u < T; ++u) {
                        const float t = tanhf(v[u][i]);
                        if (out) {
                            o[u][0] = fmaf(w3.x, t, o[u][0]);
                            o[u][1] = fmaf(w3.y, t, o[u][1]);
                            o[u][2] = fmaf(w3.z, t, o[u][2]);
                            o[u][3] = fmaf(w3.w, t, o[u][3]);
                        } else {
                            act[((k + i) * T + u) * kMlBlock + tid] = t;
                        }
                    }
                }
            }
        }
#pragma unroll
        for (int u = 0; u < T; ++u) {
            if (!on[u]) continue;
            float mu[3], kappa, un[4];
            mlp_vmf_of(o[u], mu, &kappa);
            mc_uniforms(a, a.uni, a.ctr, a.color, s[u], site[u], un);
            float *y = spins + ((int64_t)s[u] * a.N + site[u]) * 3;
            const float3 old = f3(y), m = make_float3(mu[0], mu[1], mu[2]);
            const float3 nw = around(m, vmf_w(kappa, un[0]), __fmul_rn(kTwoPi, un[1]));
            const float logq_ratio = __fmul_rn(
                kappa, dot3(__fadd_rn(old.x, -nw.x), __fadd_rn(old.y, -nw.y),
                            __fadd_rn(old.z, -nw.z), m.x, m.y, m.z));
            ++prop;
            if (mc_accept(a, h[u], old, nw, logq_ratio, un[2])) {
                ++acc;
                y[0] = nw.x;
                y[1] = nw.y;
                y[2] = nw.z;
            }
        }
    }
    mc_count(prop, acc, a.stats);
}

template <int NIN, int T>
int launch_learned_t(const MCArgs &a, float *spins, int sms, cudaStream_t s)
{
    auto k = mc_learned_kernel<NIN, T>;
    const size_t smem = ml_smem<NIN, T>(a.net.depth);
    ASD_CUDA_TRY(allow_smem(k, ml_smem<NIN, T>(3)));
    const int64_t groups = (a.n_sites_c * a.S + T - 1) / T;
    const int64_t blocks = (groups + kMlBlock - 1) / kMlBlock;
    const int64_t most = 2 * (int64_t)sms;
    k<<<(unsigned)(blocks < most ? blocks : most), kMlBlock, smem, s>>>(a, spins);
    ASD_CUDA_TRY(cudaGetLastError());
    return ASD_OK;
}

// Two sites per thread when even so every SM gets a block; one otherwise (half the latency of
// a thread's forward pass).
template <int NIN>
int launch_learned(const MCArgs &a, float *spins, int sms, cudaStream_t s)
{
    if (a.n_sites_c * a.S >= 2 * (int64_t)kMlBlock * sms) return launch_learned_t<NIN, 2>(a, spins, sms, s);
    return launch_learned_t<NIN, 1>(a, spins, sms, s);
}

// next cone from the sweep's acceptance; counters of the sweep reset
__global__ void adapt_cone(unsigned long long *sweep_stats, unsigned long long *total, float *cone)
{
    const unsigned long long p = sweep_stats[0], a = sweep_stats[1];
    total[0] += p;
    total[1] += a;
    sweep_stats[0] = sweep_stats[1] = 0;
    *cone = next_cone(*cone, p, a);
}

// counters to zero and the first cone (a kernel parameter: a copy from this host variable
// could not be captured)
__global__ void set_mc_state(unsigned long long *cnt, float *d_cone, float cone)
{
    if (threadIdx.x < 9) cnt[threadIdx.x] = 0;
    if (threadIdx.x == 9) *d_cone = cone;
}

__global__ void accumulate_stats(unsigned long long *sweep_stats, unsigned long long *total)
{
    total[0] += sweep_stats[0];
    total[1] += sweep_stats[1];
    sweep_stats[0] = sweep_stats[1] = 0;
}

}  // namespace
}  // namespace asd

using namespace asd;

extern "C" int asd_thermalize(const asd_system *sys, int n_samples, float *spins, float T,
                              int n_sweeps, int proposal, const asd_mlp *net, float cone,
                              int adapt, uint64_t seed, uint64_t counter, const float *uniforms,
                              asd_mc_stats *stats, void *stream)
{
    ASD_CHECK_ARG(sys && spins, "null argument");
    ASD_CHECK_ARG(sys->n_sites >= 1 && sys->z >= 0 && sys->z <= 32, "bad system");
    ASD_CHECK_ARG(sys->z == 0 || (sys->nbr && sys->J), "neighbour table required");
    ASD_CHECK_ARG(sys->n_colors >= 1 && sys->color_sites && sys->color_offsets, "colouring required");
    ASD_CHECK_ARG(sys->color_offsets[0] == 0 && sys->color_offsets[sys->n_colors] == sys->n_sites,
                  "colour offsets must cover every site once");
    ASD_CHECK_ARG(n_samples >= 1 && n_sweeps >= 0 && T > 0.f, "bad n_samples/n_sweeps/T");
    ASD_CHECK_ARG(proposal >= ASD_METROPOLIS && proposal <= ASD_LEARNED, "bad proposal");
    MlpView view{};
    if (proposal == ASD_LEARNED) {
        ASD_CHECK_ARG(net && net->W1 && net->W2 && net->W3 && net->b1 && net->b2 && net->b3,
                      "learned proposal needs a network");
        ASD_CHECK_ARG(net->n_in == 3 * sys->z && net->n_in <= kMlpMaxIn &&
                          net->n_hidden == kMlpHidden,
                      "network shape must be [3z -> 64 (x2 or x3) -> 4]");
        ASD_CHECK_ARG(mlp_depth(*net) == 2 || (mlp_depth(*net) == 3 && net->Wm && net->bm),
                      "network depth must be 2, or 3 with the third layer's weights");
        view = mlp_view(*net);
    }
    cudaStream_t s = (cudaStream_t)stream;
    int dev = 0, sms = 0;
    ASD_CUDA_TRY(cudaGetDevice(&dev));
    ASD_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    unsigned long long *cnt = nullptr;
    // sweep counters [2], totals [2], acceptance slots [4], grid barrier, cone
    ASD_CUDA_TRY(cudaMallocAsync(&cnt, 10 * sizeof(unsigned long long), s));
    unsigned *bar = reinterpret_cast<unsigned *>(cnt + 8);
    float *d_cone = reinterpret_cast<float *>(cnt + 9);
    int rc = ASD_OK;
    do {
        set_mc_state<<<1, 16, 0, s>>>(cnt, d_cone, cone);
        MCArgs a{};
        a.N = sys->n_sites;
        a.S = n_samples;
        a.z = sys->z;
        a.nbr = sys->nbr;
        a.J = sys->J;
        a.Hz = sys->Hz;
        a.D = sys->D;
        a.A = sys->A;
        a.beta = 1.f / T;
        a.proposal = proposal;
        a.seed = seed;
        a.cone = d_cone;
        a.stats = cnt;
        a.net = view;
        MCRoute rt;
        if ((rc = mc_route(a, sys->color_offsets, sys->n_colors, n_sweeps,
                           adapt && proposal == ASD_METROPOLIS, sms, &rt)))
            break;
        if (rt.k) {
            MCRun r{};
            r.a = a;
            r.a.sites = sys->color_sites;
            r.spins = spins;
            r.n_colors = sys->n_colors;
            for (int c = 0; c <= sys->n_colors; ++c) r.off[c] = sys->color_offsets[c];
            r.adapt = adapt && proposal == ASD_METROPOLIS;
            r.cone = d_cone;
            r.total = cnt + 2;
            r.slots = cnt + 4;
            r.bar = bar;
            r.err = device_error_word();
            if (!r.err) {
                rc = ASD_ECUDA;
                break;
            }
            for (int sw = 0; sw < n_sweeps; sw += kMcSweepsPerLaunch) {
                r.n_sweeps = std::min(kMcSweepsPerLaunch, n_sweeps - sw);
                r.a.ctr = counter + (uint64_t)sw;
                r.a.uni = uniforms ? uniforms + (size_t)sw * n_samples * sys->n_sites * 4 : nullptr;
                if (rt.local) {
                    rt.k<<<rt.grid, rt.block, rt.smem, s>>>(r);
                    continue;
                }
                if (sw > 0)   // barrier and slots start at zero
                    cudaMemsetAsync(cnt + 4, 0, 5 * sizeof(unsigned long long), s);
                void *args[] = {&r};
                const cudaError_t e = cudaLaunchCooperativeKernel(
                    (const void *)rt.k, dim3(rt.grid), dim3(rt.block), args, rt.smem, s);
                if (e != cudaSuccess) {
                    set_cuda_error(e, "asd_thermalize: cooperative launch");
                    rc = ASD_ECUDA;
                    break;
                }
            }
        } else {
            for (int sw = 0; sw < n_sweeps; ++sw) {
                a.ctr = counter + (uint64_t)sw;
                a.uni = uniforms ? uniforms + (size_t)sw * n_samples * sys->n_sites * 4 : nullptr;
                for (int c = 0; c < sys->n_colors; ++c) {
                    a.color = c;
                    a.sites = sys->color_sites + sys->color_offsets[c];
                    a.n_sites_c = sys->color_offsets[c + 1] - sys->color_offsets[c];
                    const int64_t n = a.n_sites_c * n_samples;
                    if (n == 0) continue;
                    if (proposal == ASD_LEARNED) {
                        rc = view.n_in == 12   ? launch_learned<12>(a, spins, sms, s)
                             : view.n_in == 18 ? launch_learned<18>(a, spins, sms, s)
                                               : launch_learned<kMlpMaxIn>(a, spins, sms, s);
                        if (rc) break;
                    } else {
                        mc_color_kernel<<<(unsigned)((n + 127) / 128), 128, 0, s>>>(a, spins);
                    }
                }
                if (rc) break;
                if (adapt && proposal == ASD_METROPOLIS) adapt_cone<<<1, 1, 0, s>>>(cnt, cnt + 2, d_cone);
                else accumulate_stats<<<1, 1, 0, s>>>(cnt, cnt + 2);
            }
        }
        if (rc) break;
        if (cudaGetLastError() != cudaSuccess) {
            rc = ASD_ECUDA;
            break;
        }
        if (stats) {
            unsigned long long h[2];
            float hc;
            if (cudaMemcpyAsync(h, cnt + 2, sizeof h, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
                cudaMemcpyAsync(&hc, d_cone, sizeof hc, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
                cudaStreamSynchronize(s) != cudaSuccess) {
                rc = ASD_ECUDA;
                break;
            }
            stats->proposed = (int64_t)h[0];
            stats->accepted = (int64_t)h[1];
            stats->cone = hc;
        }
    } while (0);
    cudaFreeAsync(cnt, s);
    if (rc == ASD_ECUDA) set_error_text("asd_thermalize: CUDA call failed");
    return rc;
}
