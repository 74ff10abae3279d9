// Landau-Lifshitz dynamics (Eq. 2): dS_i/dt = (dH/dS_i) x S_i, classic RK4.
//
// H of Eq. 1 (exchange, DM, single-ion anisotropy, field), so the local field is
// h_i = sum_j J_ij S_j + sum_j D_ij x S_j - 2 A S^z_i z^ - Hz z^ (D_ij the DM vector of the
// directed bond, D_ji = -D_ij: Algorithm 1's exchange, DMI, anisotropy and field
// contributions).  As in Algorithm 1, one thread handles
// one site and the S samples are processed by the same launch (the paper passes its
// M configurations to one kernel, Section 3.1); the RK4 stages keep their derivative
// in separate arrays so sites never race (Section 3.1).  No renormalisation: the paper
// notes its RK4 evolution is not norm preserving.
//
// A stage needs every neighbour's previous stage.  Routes, by size (ll_run):
//   ll_persistent<LOCAL>   one block per sample, or per several small ones, the state in shared
//                          memory, a block barrier between stages: samples of up to 2048 sites;
//   ll_tagged              a cooperative launch over every (sample, site), one site per thread;
//                          blocks exchange stage inputs as words that carry their stage number;
//   ll_persistent<global>  a cooperative launch, the state in L2, a grid barrier between stages:
//                          up to two sites per thread;
//   rk4_stage              one launch per stage: larger systems.
// The last stage writes the new state and, every `stride` steps, the trajectory frame in the
// site-major layout traj[i][s][f][a] consumed by asd_pair_corr.  All routes do the same
// arithmetic in the same order.
#include <algorithm>

#include "asd_internal.h"
#include "grid_barrier.cuh"

namespace asd {
namespace {

struct LLArgs {
    int64_t N;
    int S;
    int z;
    const int *nbr;
    const float *J;
    float Hz;
    const float *D;  // [N][z][3] or null
    float A;
};

// One neighbour's part of the local field: J S_j, and D_ij x S_j with DM vectors (d: the
// directed bond's, or null).
__device__ __forceinline__ void add_bond(float3 &h, float J, float sx, float sy, float sz,
                                         const float *__restrict__ d)
{
    h.x = fmaf(J, sx, h.x);
    h.y = fmaf(J, sy, h.y);
    h.z = fmaf(J, sz, h.z);
    if (d) {
        const float dx = __ldg(d), dy = __ldg(d + 1), dz = __ldg(d + 2);
        h.x += dy * sz - dz * sy;
        h.y += dz * sx - dx * sz;
        h.z += dx * sy - dy * sx;
    }
}

__device__ __forceinline__ float3 field(const LLArgs &a, const float *__restrict__ Y, int s,
                                        int64_t i)
{
    const float *Ys = Y + (int64_t)s * a.N * 3;
    float3 h = make_float3(0.f, 0.f, -a.Hz);
    for (int k = 0; k < a.z; ++k) {
        const int j = __ldg(a.nbr + i * a.z + k);
        if (j < 0) continue;
        // (add_bond's sums, written out: through the call a stage of 70^3 sites took 3 to 8 %
        // longer, at 32 instead of 40 registers and a nearly empty second wave of blocks)
        const float Jij = __ldg(a.J + i * a.z + k);
        h.x = fmaf(Jij, Ys[3 * (int64_t)j + 0], h.x);
        h.y = fmaf(Jij, Ys[3 * (int64_t)j + 1], h.y);
        h.z = fmaf(Jij, Ys[3 * (int64_t)j + 2], h.z);
        if (a.D) {
            const float *d = a.D + (i * a.z + k) * 3;
            const float dx = __ldg(d), dy = __ldg(d + 1), dz = __ldg(d + 2);
            const float sx = Ys[3 * (int64_t)j], sy = Ys[3 * (int64_t)j + 1],
                        sz = Ys[3 * (int64_t)j + 2];
            h.x += dy * sz - dz * sy;
            h.y += dz * sx - dx * sz;
            h.z += dx * sy - dy * sx;
        }
    }
    h.z = fmaf(-2.f * a.A, Ys[3 * i + 2], h.z);
    return h;
}

__device__ __forceinline__ float3 cross(float3 a, float3 b)
{
    return make_float3(a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x);
}

// stage k (1..4): reads Yin (the stage input), writes the next stage input and the
// running combination acc = k1 + 2 k2 + 2 k3.
template <int STAGE>
__global__ void rk4_stage(LLArgs a, float *__restrict__ Y, const float *__restrict__ Yin,
                          float *__restrict__ Yout, float *__restrict__ acc, float dt, float *traj,
                          int F, int frame)
{
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= a.N * a.S) return;
    const int s = (int)(g / a.N);
    const int64_t i = g % a.N;
    const int64_t o = (int64_t)s * a.N * 3 + 3 * i;
    const float3 h = field(a, Yin, s, i);
    const float3 x = make_float3(Yin[o], Yin[o + 1], Yin[o + 2]);
    const float3 k = cross(h, x);
    const float3 y = make_float3(Y[o], Y[o + 1], Y[o + 2]);
    if (STAGE == 1) {
        acc[o] = k.x; acc[o + 1] = k.y; acc[o + 2] = k.z;
    } else if (STAGE < 4) {
        acc[o] += 2.f * k.x; acc[o + 1] += 2.f * k.y; acc[o + 2] += 2.f * k.z;
    }
    if (STAGE < 4) {
        const float c = STAGE == 3 ? dt : 0.5f * dt;
        Yout[o] = fmaf(c, k.x, y.x);
        Yout[o + 1] = fmaf(c, k.y, y.y);
        Yout[o + 2] = fmaf(c, k.z, y.z);
    } else {
        const float c = dt / 6.f;
        const float3 n = make_float3(fmaf(c, acc[o] + k.x, y.x), fmaf(c, acc[o + 1] + k.y, y.y),
                                     fmaf(c, acc[o + 2] + k.z, y.z));
        Y[o] = n.x; Y[o + 1] = n.y; Y[o + 2] = n.z;
        if (frame >= 0) {
            float *dst = traj + ((i * a.S + s) * (int64_t)F + frame) * 3;
            dst[0] = n.x; dst[1] = n.y; dst[2] = n.z;
        }
    }
}

__global__ void write_frame0(const float *__restrict__ Y, int64_t N, int S, float *traj, int F)
{
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= N * S) return;
    const int s = (int)(g / N);
    const int64_t i = g % N;
    const float *src = Y + (int64_t)s * N * 3 + 3 * i;
    float *dst = traj + ((i * S + s) * (int64_t)F) * 3;
    dst[0] = src[0]; dst[1] = src[1]; dst[2] = src[2];
}

// ---------------------------------------------------------------------------------------
// Persistent routes
// ---------------------------------------------------------------------------------------
constexpr int kLLThreads = 1024;
constexpr int kLLMaxSpt = 2;                       // sites per thread
constexpr int64_t kLLPackSites = 256;              // sites of small samples per block
constexpr size_t kLLMaxSmem = 220 * 1024;
constexpr int kLLStepsPerLaunch = 4096;            // other streams' work gets in between

struct LLRun {
    LLArgs a;
    const float *in;     // [S][N][3] state at the first step
    float *out;          // [S][N][3] state after the last step, or null
    float4 *Y, *T1, *T2; // global route: state and stage inputs [S][N]
    int n_buf;           // ll_tagged: stage inputs from Y on, 2 .. kLLMaxBufs
    int per_block;       // samples per block (PACK)
    unsigned *bar;       // cooperative routes: grid barrier count (zero at launch)
    float *traj;
    int F;
    int64_t step0, step1;  // steps [step0, step1) of the run
    int stride;
    float dt;
    int stage_frames;    // 1: frames go out through shared memory, kLLFrames at a time
    int *err;
};
constexpr int kLLGroup = 4;                         // bonds loaded together (Z = 0)
constexpr int kLLMaxBufs = 9;                       // stage inputs of ll_tagged
constexpr int kLLFrames = 4;
constexpr int kLLFramePitch = 3 * kLLFrames + 1;   // words per site (odd: no bank conflicts)

// All steps of a launch.  Bound by the latency of a stage (380 to 640 dependent stages, each
// a few hundred cycles of loads and arithmetic), not by bandwidth, so the work is to take the
// launches, the index loads and the global round trips out of a stage: bonds (neighbour,
// coupling) are read once, into registers for Z = 4 or 6 bonds and one site a thread, else
// into shared memory (Z = 0: any number of bonds); state and derivative sum of the own sites stay in
// registers; neighbours are read as one 16-byte word from shared memory (LOCAL) or L2.
// Measured against a launch per stage: 50 samples of 16^2 sites, 95 steps, 1572 -> 121 us
// (4.1 -> 0.32 us per stage); 64^3, 159 steps, 6.14 -> 3.36 ms (9.6 -> 5.3 us per stage, of
// which the barrier about 2); frames stored by each site as they come instead of gathered:
// 130 us and 3.78 ms.  36^2 sites and two samples, 90 steps: 1.58 -> 0.53 ms, though only
// two blocks run.
template <int SPT, int Z, bool LOCAL, bool PACK = false>
__global__ void __launch_bounds__(kLLThreads, 1) ll_persistent(const __grid_constant__ LLRun r)
{
    extern __shared__ __align__(16) uint8_t ll_smem[];
    constexpr bool kReg = Z > 0 && SPT == 1;   // bonds in registers
    const LLArgs &a = r.a;
    const int N = (int)a.N, nt = blockDim.x, tid = threadIdx.x;
    const int64_t n = (int64_t)N * a.S;
    // contiguous runs of the flattened (sample, site) list per block: LOCAL a sample (PACK:
    // per_block of them), else SPT nt sites.  Slot = site index within the block, tid + k nt.
    const int slots = LOCAL ? (PACK ? r.per_block * N : N) : SPT * nt;
    const int64_t g0 = (int64_t)blockIdx.x * slots;
    // state arrays indexed by the flattened site minus `base`
    const int64_t base = LOCAL ? g0 : 0;
    float4 *Y = LOCAL ? reinterpret_cast<float4 *>(ll_smem) : r.Y;
    float4 *T1 = LOCAL ? Y + slots : r.T1;
    float4 *T2 = LOCAL ? T1 + slots : r.T2;
    // bonds in shared memory: [k][slot]
    int *sm_nbr = reinterpret_cast<int *>(ll_smem + (LOCAL ? (size_t)48 * slots : 0));
    float *sm_J = reinterpret_cast<float *>(sm_nbr + (kReg ? 0 : (size_t)a.z * slots));
    float *sm_frames = sm_J + (kReg ? 0 : (size_t)a.z * slots);

    constexpr int ZR = Z > 0 ? Z : 1, ZB = kReg ? Z : 1;
    int nb[ZB];
    float Jr[ZB];
    float3 y[SPT], acc[SPT], x[SPT];
    bool on[SPT];
    int own[SPT];                      // index of the own site in the state arrays
    int site[SPT];                     // site in its sample
    float *dst[SPT];                   // its last trajectory frame
#pragma unroll
    for (int u = 0; u < SPT; ++u) {
        const int slot = u * nt + tid;
        const int64_t g = g0 + slot;
        on[u] = LOCAL && !PACK ? slot < N : slot < slots && g < n;
        const int64_t gc = on[u] ? g : g0;
        const int s = LOCAL && !PACK ? (int)blockIdx.x : (int)(gc / N);
        site[u] = (int)(gc - (int64_t)s * N);
        const int off = (int)((int64_t)s * N - base);   // the sample's first index
        own[u] = (int)(gc - base);
        if (kReg) {
#pragma unroll
            for (int k = 0; k < ZB; ++k) {
                const int j = on[u] ? __ldg(a.nbr + (int64_t)site[u] * Z + k) : -1;
                nb[k] = j < 0 ? -1 : j + off;
                Jr[k] = on[u] ? __ldg(a.J + (int64_t)site[u] * Z + k) : 0.f;
            }
        } else if (on[u]) {
            for (int k = 0; k < a.z; ++k) {
                const int j = __ldg(a.nbr + (int64_t)site[u] * a.z + k);
                sm_nbr[k * slots + slot] = j < 0 ? -1 : j + off;
                sm_J[k * slots + slot] = __ldg(a.J + (int64_t)site[u] * a.z + k);
            }
        }
        const float *src = r.in + 3 * gc;
        y[u] = make_float3(src[0], src[1], src[2]);
        x[u] = y[u];
        dst[u] = r.traj + (((int64_t)site[u] * a.S + s) * r.F + r.step0 / r.stride) * 3;
        if (on[u]) {
            Y[own[u]] = make_float4(y[u].x, y[u].y, y[u].z, 0.f);
            if (r.step0 == 0) {
                dst[u][0] = y[u].x; dst[u][1] = y[u].y; dst[u][2] = y[u].z;
            }
        }
    }
    int in_frame = (int)(r.step0 % r.stride);   // steps since the last frame
    // Frames.  A frame's 12 bytes per site lie a trajectory row apart, so a warp storing one
    // touches 32 lines per instruction; kLLFrames frames gathered in shared memory go out
    // with consecutive lanes on consecutive words of a site's row.
    int n_held = 0;
    int64_t f_held = r.step0 / r.stride + 1;    // first frame held
    auto put_frames = [&]() {
        __syncthreads();   // every site's frames are in
        const int words = 3 * n_held,
                  left = LOCAL && !PACK ? N : (int)min((int64_t)slots, n - g0);
        for (int e = tid; e < left * words; e += nt) {
            const int slot = e / words, c = e - slot * words;
            const int64_t g = g0 + slot;
            const int64_t s = LOCAL && !PACK ? blockIdx.x : g / N, i = g - s * N;
            r.traj[((i * a.S + s) * r.F + f_held) * 3 + c] = sm_frames[slot * kLLFramePitch + c];
        }
        f_held += n_held;
        n_held = 0;
        __syncthreads();   // the buffer may be filled again
    };
    unsigned target = 0;
    auto barrier = [&]() {
        if (LOCAL) {
            __syncthreads();
            return true;
        }
        target += gridDim.x;
        return grid_barrier(r.bar, target, r.err);
    };
    if (!barrier()) return;

    // derivative of own site u from the stage input V (own value x[u])
    auto deriv = [&](int u, const float4 *V) {
        float3 h = make_float3(0.f, 0.f, -a.Hz);
        const int slot = u * nt + tid;
        if (Z > 0) {
            // all neighbours' loads in flight, then the sums in bond order
            float4 sj[ZR];
            int j[ZR];
#pragma unroll
            for (int k = 0; k < ZR; ++k) {
                j[k] = kReg ? nb[kReg ? k : 0] : sm_nbr[k * slots + slot];
                sj[k] = V[j[k] < 0 ? own[u] : j[k]];
            }
#pragma unroll
            for (int k = 0; k < ZR; ++k)
                if (j[k] >= 0)
                    add_bond(h, kReg ? Jr[kReg ? k : 0] : sm_J[k * slots + slot], sj[k].x,
                             sj[k].y, sj[k].z,
                             a.D ? a.D + ((int64_t)site[u] * Z + k) * 3 : nullptr);
        } else if (LOCAL) {
            for (int k = 0; k < a.z; ++k) {
                const int j = sm_nbr[k * slots + slot];
                if (j < 0) continue;
                const float4 sj = V[j];
                add_bond(h, sm_J[k * slots + slot], sj.x, sj.y, sj.z,
                         a.D ? a.D + ((int64_t)site[u] * a.z + k) * 3 : nullptr);
            }
        } else {
            // from L2: a group's loads in flight together (one after the other, the 26 bonds of a
            // stage took 9 us, more than a launch per stage: 12^3 sites, 40 stages, 379 -> 204 us;
            // from shared memory, above, groups gain nothing and cost 10 % with DM vectors)
            for (int k0 = 0; k0 < a.z; k0 += kLLGroup) {
                float4 sj[kLLGroup];
                int j[kLLGroup];
#pragma unroll
                for (int q = 0; q < kLLGroup; ++q) {
                    j[q] = k0 + q < a.z ? sm_nbr[(k0 + q) * slots + slot] : -1;
                    sj[q] = V[j[q] < 0 ? own[u] : j[q]];
                }
#pragma unroll
                for (int q = 0; q < kLLGroup; ++q)
                    if (j[q] >= 0)
                        add_bond(h, sm_J[(k0 + q) * slots + slot], sj[q].x, sj[q].y, sj[q].z,
                                 a.D ? a.D + ((int64_t)site[u] * a.z + k0 + q) * 3 : nullptr);
            }
        }
        h.z = fmaf(-2.f * a.A, x[u].z, h.z);
        return cross(h, x[u]);
    };
    for (int64_t st = r.step0; st < r.step1; ++st) {
#pragma unroll
        for (int stage = 1; stage <= 4; ++stage) {
            const float4 *in = stage == 1 ? Y : stage == 3 ? T2 : T1;
            float4 *out = stage == 4 ? Y : stage == 2 ? T2 : T1;
#pragma unroll
            for (int u = 0; u < SPT; ++u) {
                if (!on[u]) continue;
                const float3 k = deriv(u, in);
                if (stage == 1) {
                    acc[u] = k;
                } else if (stage < 4) {
                    acc[u].x += 2.f * k.x;
                    acc[u].y += 2.f * k.y;
                    acc[u].z += 2.f * k.z;
                }
                if (stage < 4) {
                    const float c = stage == 3 ? r.dt : 0.5f * r.dt;
                    x[u] = make_float3(fmaf(c, k.x, y[u].x), fmaf(c, k.y, y[u].y),
                                       fmaf(c, k.z, y[u].z));
                } else {
                    const float c = r.dt / 6.f;
                    y[u] = make_float3(fmaf(c, acc[u].x + k.x, y[u].x),
                                       fmaf(c, acc[u].y + k.y, y[u].y),
                                       fmaf(c, acc[u].z + k.z, y[u].z));
                    x[u] = y[u];
                }
                out[own[u]] = make_float4(x[u].x, x[u].y, x[u].z, 0.f);
            }
            // (the frame's stores are in flight while the barrier runs)
            if (stage == 4 && ++in_frame == r.stride) {
                in_frame = 0;
#pragma unroll
                for (int u = 0; u < SPT; ++u) {
                    dst[u] += 3;
                    float *d = r.stage_frames
                                   ? sm_frames + (u * nt + tid) * kLLFramePitch + 3 * n_held
                                   : dst[u];
                    if (on[u]) {
                        d[0] = y[u].x; d[1] = y[u].y; d[2] = y[u].z;
                    }
                }
                if (r.stage_frames && ++n_held == kLLFrames) put_frames();
            }
            if (!barrier()) return;
        }
    }
    if (n_held > 0) put_frames();
    if (r.out)
#pragma unroll
        for (int u = 0; u < SPT; ++u)
            if (on[u]) {
                float *o = r.out + 3 * (own[u] + base);
                o[0] = y[u].x; o[1] = y[u].y; o[2] = y[u].z;
            }
}

// 16-byte loads and stores of one access at GPU scope: a value and its stage number together.
__device__ __forceinline__ float4 ld_tagged(const float4 *p)
{
    uint64_t lo, hi;
    asm volatile("{\n\t.reg .b128 t;\n\tld.relaxed.gpu.global.b128 t, [%2];\n\t"
                 "mov.b128 {%0, %1}, t;\n}\n"
                 : "=l"(lo), "=l"(hi)
                 : "l"(p)
                 : "memory");
    return make_float4(__uint_as_float((uint32_t)lo), __uint_as_float((uint32_t)(lo >> 32)),
                       __uint_as_float((uint32_t)hi), __uint_as_float((uint32_t)(hi >> 32)));
}
__device__ __forceinline__ void st_tagged(float4 *p, float3 v, int tag)
{
    const uint64_t lo = (uint64_t)__float_as_uint(v.x) | (uint64_t)__float_as_uint(v.y) << 32;
    const uint64_t hi = (uint64_t)__float_as_uint(v.z) | (uint64_t)(uint32_t)tag << 32;
    asm volatile("{\n\t.reg .b128 t;\n\tmov.b128 t, {%1, %2};\n\t"
                 "st.relaxed.gpu.global.b128 [%0], t;\n}\n" ::"l"(p), "l"(lo), "l"(hi)
                 : "memory");
}

// The same run, one site per thread, without a grid barrier in every stage (which was about 2
// of the 2.5 to 2.8 us of a stage at these sizes).  The block's own stage inputs are in shared
// memory; other blocks' come from global memory as 16-byte words that carry their stage number,
// and a reader waits for the number it needs, so a stage costs one store and one load through
// L2.  Stage g's inputs are in buffer g mod n_buf; a grid barrier every n_buf - 1 stages keeps a
// block from overwriting a buffer that another still reads, whatever the bond table.  A block
// waits only for what others wrote in the stage before, so every wait ends; all are bounded.
// Measured against a barrier per stage: 48^3 sites, 67 steps, 738 -> 566 us; 8 samples of 18^3, 105
// steps, 1022 -> 736 us (2.1 and 1.75 us per stage).  With two sites per thread it is slower (64^3,
// 159 steps, 3.35 -> 4.17 ms: a stage is bound by issue slots there, and the tests of the
// numbers add to them), so ll_persistent keeps those.
template <int Z>
__global__ void __launch_bounds__(kLLThreads, 1) ll_tagged(const __grid_constant__ LLRun r)
{
    extern __shared__ __align__(16) uint8_t ll_smem[];
    constexpr bool kReg = Z > 0;   // bonds in registers
    const LLArgs &a = r.a;
    const int N = (int)a.N, nt = blockDim.x, tid = threadIdx.x;
    const int64_t n = (int64_t)N * a.S;
    const int64_t g0 = (int64_t)blockIdx.x * nt;
    // two stages' inputs of the block's sites, bonds [k][slot], held frames
    float4 *sm = reinterpret_cast<float4 *>(ll_smem);
    int *sm_nbr = reinterpret_cast<int *>(sm + 2 * nt);
    float *sm_J = reinterpret_cast<float *>(sm_nbr + (kReg ? 0 : a.z * nt));
    float *sm_frames = sm_J + (kReg ? 0 : a.z * nt);

    constexpr int ZB = kReg ? Z : 1;
    int nb[ZB];
    float Jr[ZB];
    const bool on = g0 + tid < n;
    const int64_t gc = on ? g0 + tid : g0;
    const int s = (int)(gc / N), site = (int)(gc - (int64_t)s * N);
    // a neighbour as its slot, or -2 - its flattened index when another block has it (-1: none)
    const int off = (int)((int64_t)s * N);
    auto place = [&](int j) {
        if (j < 0) return -1;
        const int64_t slot = (int64_t)j + off - g0;
        return slot >= 0 && slot < nt ? (int)slot : -2 - (j + off);
    };
    if (kReg) {
#pragma unroll
        for (int k = 0; k < ZB; ++k) {
            nb[k] = on ? place(__ldg(a.nbr + (int64_t)site * Z + k)) : -1;
            Jr[k] = on ? __ldg(a.J + (int64_t)site * Z + k) : 0.f;
        }
    } else if (on) {
        for (int k = 0; k < a.z; ++k) {
            sm_nbr[k * nt + tid] = place(__ldg(a.nbr + (int64_t)site * a.z + k));
            sm_J[k * nt + tid] = __ldg(a.J + (int64_t)site * a.z + k);
        }
    }
    const float *src = r.in + 3 * gc;
    float3 y = make_float3(src[0], src[1], src[2]), x = y, acc;
    float *dst = r.traj + (((int64_t)site * a.S + s) * r.F + r.step0 / r.stride) * 3;
    if (on) {
        sm[tid] = make_float4(y.x, y.y, y.z, 0.f);
        st_tagged(r.Y + gc, y, 0);
        for (int b = 1; b < r.n_buf; ++b) st_tagged(r.Y + b * n + gc, y, -1);
        if (r.step0 == 0) {
            dst[0] = y.x; dst[1] = y.y; dst[2] = y.z;
        }
    }
    int in_frame = (int)(r.step0 % r.stride);   // steps since the last frame
    int n_held = 0;                             // frames held (as in ll_persistent)
    int64_t f_held = r.step0 / r.stride + 1;
    auto put_frames = [&]() {
        __syncthreads();
        const int words = 3 * n_held, left = (int)min((int64_t)nt, n - g0);
        for (int e = tid; e < left * words; e += nt) {
            const int slot = e / words, c = e - slot * words;
            const int64_t g = g0 + slot, sl = g / N, i = g - sl * N;
            r.traj[((i * a.S + sl) * r.F + f_held) * 3 + c] = sm_frames[slot * kLLFramePitch + c];
        }
        f_held += n_held;
        n_held = 0;
        __syncthreads();
    };
    unsigned target = gridDim.x;
    if (!grid_barrier(r.bar, target, r.err)) return;

    bool alive = true;   // no wait of this thread has given up
    // the value of stage g of another block's site, once it is there
    auto wait_tagged = [&](const float4 *p, int g) {
        float4 v = ld_tagged(p);
        unsigned long long t0 = 0;
        for (unsigned it = 1; __float_as_int(v.w) != g; ++it) {
            if ((it & 1023u) == 0) {
                unsigned long long now;
                asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
                if (t0 == 0) t0 = now;
                else if (now - t0 > kGridTimeoutNs) {
                    atomicCAS(r.err, 0, (int)DEV_TIMEOUT_GRID);
                    alive = false;
                    break;
                }
            }
            v = ld_tagged(p);
        }
        return v;
    };
    // derivative of the own site from the inputs of stage g (V: the block's, G: everyone's)
    auto deriv = [&](int g, const float4 *V, const float4 *G) {
        float3 h = make_float3(0.f, 0.f, -a.Hz);
        if (kReg) {
            // all neighbours' loads in flight, then the late ones again, then the sums in bond
            // order
            float4 sj[ZB];
#pragma unroll
            for (int k = 0; k < ZB; ++k) {
                if (nb[k] >= -1) sj[k] = V[nb[k] < 0 ? tid : nb[k]];
                else sj[k] = ld_tagged(G - (nb[k] + 2));
            }
#pragma unroll
            for (int k = 0; k < ZB; ++k)
                if (nb[k] < -1 && __float_as_int(sj[k].w) != g)
                    sj[k] = wait_tagged(G - (nb[k] + 2), g);
#pragma unroll
            for (int k = 0; k < ZB; ++k)
                if (nb[k] != -1)
                    add_bond(h, Jr[k], sj[k].x, sj[k].y, sj[k].z,
                             a.D ? a.D + ((int64_t)site * Z + k) * 3 : nullptr);
        } else {
            for (int k0 = 0; k0 < a.z; k0 += kLLGroup) {   // (as above, a group at a time)
                float4 sj[kLLGroup];
                int j[kLLGroup];
#pragma unroll
                for (int q = 0; q < kLLGroup; ++q) {
                    j[q] = k0 + q < a.z ? sm_nbr[(k0 + q) * nt + tid] : -1;
                    if (j[q] >= -1) sj[q] = V[j[q] < 0 ? tid : j[q]];
                    else sj[q] = ld_tagged(G - (j[q] + 2));
                }
#pragma unroll
                for (int q = 0; q < kLLGroup; ++q)
                    if (j[q] < -1 && __float_as_int(sj[q].w) != g)
                        sj[q] = wait_tagged(G - (j[q] + 2), g);
#pragma unroll
                for (int q = 0; q < kLLGroup; ++q)
                    if (j[q] != -1)
                        add_bond(h, sm_J[(k0 + q) * nt + tid], sj[q].x, sj[q].y, sj[q].z,
                                 a.D ? a.D + ((int64_t)site * a.z + k0 + q) * 3 : nullptr);
            }
        }
        h.z = fmaf(-2.f * a.A, x.z, h.z);
        return cross(h, x);
    };
    int g = 0, b_in = 0, since = 0;   // stage, its buffer, stages since the last grid barrier
    for (int64_t st = r.step0; st < r.step1; ++st) {
#pragma unroll
        for (int stage = 1; stage <= 4; ++stage) {
            const float4 *V = sm + (stage & 1 ? 0 : nt), *G = r.Y + (int64_t)b_in * n;
            float4 *out = sm + (stage & 1 ? nt : 0);
            if (++b_in == r.n_buf) b_in = 0;
            if (on) {
                const float3 k = deriv(g, V, G);
                if (stage == 1) {
                    acc = k;
                } else if (stage < 4) {
                    acc.x += 2.f * k.x;
                    acc.y += 2.f * k.y;
                    acc.z += 2.f * k.z;
                }
                if (stage < 4) {
                    const float c = stage == 3 ? r.dt : 0.5f * r.dt;
                    x = make_float3(fmaf(c, k.x, y.x), fmaf(c, k.y, y.y), fmaf(c, k.z, y.z));
                } else {
                    const float c = r.dt / 6.f;
                    y = make_float3(fmaf(c, acc.x + k.x, y.x), fmaf(c, acc.y + k.y, y.y),
                                    fmaf(c, acc.z + k.z, y.z));
                    x = y;
                }
                st_tagged(r.Y + (int64_t)b_in * n + gc, x, g + 1);
                out[tid] = make_float4(x.x, x.y, x.z, 0.f);
            }
            ++g;
            if (stage == 4 && ++in_frame == r.stride) {
                in_frame = 0;
                dst += 3;
                float *d = r.stage_frames ? sm_frames + tid * kLLFramePitch + 3 * n_held : dst;
                if (on) {
                    d[0] = y.x; d[1] = y.y; d[2] = y.z;
                }
                if (r.stage_frames && ++n_held == kLLFrames) put_frames();
            }
            if (!__syncthreads_and(alive)) return;
            if (++since == r.n_buf - 1) {
                since = 0;
                target += gridDim.x;
                if (!grid_barrier(r.bar, target, r.err)) return;
            }
        }
    }
    if (n_held > 0) put_frames();
    if (r.out && on) {
        float *o = r.out + 3 * gc;
        o[0] = y.x; o[1] = y.y; o[2] = y.z;
    }
}

typedef void (*LLKernel)(LLRun);

template <int SPT, bool LOCAL>
LLKernel ll_kernel_z(int z)
{
    if (z == 4) return ll_persistent<SPT, 4, LOCAL>;
    if (z == 6) return ll_persistent<SPT, 6, LOCAL>;
    return ll_persistent<SPT, 0, LOCAL>;
}

// A persistent route for the run: kernel, grid, block, shared memory; kernel = null when
// the system is too large for one.
struct LLRoute {
    LLKernel k = nullptr;
    bool local = false, tagged = false;
    unsigned grid = 0, block = 0;
    size_t smem = 0;
    int per_block = 1;   // local: samples per block
    bool stage_frames = false;
};

// One block per sample up to 2048 sites (two per thread; the state and any table must fit
// shared memory; samples of up to 48 sites share blocks where there are more than the
// device holds at once (32 blocks per SM): 300000 samples of one site, one step, 213 us in a warp
// each, 12.4 shared, 37 by a launch per stage; of 4 sites 262, 45 and 77; of 64 sites 50 us for
// 20000 in blocks of their own, 57 shared).  Otherwise a cooperative launch, one block per SM, one or two sites per
// thread.  Beyond that (more than 2048 sites per SM) a launch per stage: with four sites per
// thread, their bonds in shared memory, the cooperative kernel took 54.8 -> 64.6 us (80^3
// glass, one step), 385 -> 450 us (68^3, 10 steps), and gained 4 to 17 % only on lattices of
// four bonds (700^2, 10 steps, 506 -> 434 us).
int ll_route(const LLArgs &a, LLRoute *out)
{
    *out = LLRoute();
    int dev = 0, sms = 0, coop = 0;
    ASD_CUDA_TRY(cudaGetDevice(&dev));
    ASD_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    ASD_CUDA_TRY(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev));
    const int64_t n = a.N * a.S;
    LLRoute r;
    // (int indices of the state arrays)
    if (n > (int64_t)1 << 30) return ASD_OK;
    const auto bonds = [&](int spt, int64_t slots) -> size_t {
        return spt == 1 && (a.z == 4 || a.z == 6) ? 0 : (size_t)a.z * slots * 8;
    };
    // frames gathered in shared memory where it has room
    const auto add_frames = [](LLRoute &r, size_t smem, int64_t slots) {
        const size_t more = sizeof(float) * kLLFramePitch * (size_t)slots;
        r.stage_frames = smem + more <= kLLMaxSmem;
        r.smem = smem + (r.stage_frames ? more : 0);
    };
    if (a.N <= 2 * kLLThreads) {
        const int spt = a.N <= kLLThreads ? 1 : 2;
        const size_t smem = (size_t)48 * a.N + bonds(spt, a.N);
        if (smem <= kLLMaxSmem) {
            r.local = true;
            r.k = spt == 1 ? ll_kernel_z<1, true>(a.z) : ll_kernel_z<2, true>(a.z);
            // more samples than blocks fit the device at once (32 per SM): several per block
            if (a.S > 32 * sms && a.N <= 48) {
                r.per_block = (int)(kLLPackSites / a.N);
                r.k = a.z == 4   ? ll_persistent<1, 4, true, true>
                      : a.z == 6 ? ll_persistent<1, 6, true, true>
                                 : ll_persistent<1, 0, true, true>;
            }
            const int64_t slots = r.per_block * a.N;
            r.grid = (unsigned)((a.S + r.per_block - 1) / r.per_block);
            r.block = (unsigned)(((slots + spt - 1) / spt + 31) / 32 * 32);
            add_frames(r, (size_t)48 * slots + bonds(spt, slots), slots);
            ASD_CUDA_TRY(allow_smem(r.k, kLLMaxSmem));
            *out = r;
            return ASD_OK;
        }
    }
    if (!coop) return ASD_OK;
    for (int spt = 1; spt <= kLLMaxSpt; spt *= 2) {
        if ((int64_t)sms * kLLThreads * spt < n) continue;
        // spread the sites over all SMs, whole warps per block
        const int64_t per = (n + (int64_t)sms * spt - 1) / ((int64_t)sms * spt);
        r.block = (unsigned)((per + 31) / 32 * 32);
        r.grid = (unsigned)((n + (int64_t)r.block * spt - 1) / ((int64_t)r.block * spt));
        r.smem = bonds(spt, (int64_t)spt * r.block);
        if (r.smem > kLLMaxSmem) return ASD_OK;
        // one site per thread: ll_tagged, unless many bonds leave no room for its inputs
        const size_t own = 2 * sizeof(float4) * (size_t)r.block;
        r.tagged = spt == 1 && r.smem + own <= kLLMaxSmem;
        add_frames(r, r.smem + (r.tagged ? own : 0), (int64_t)spt * r.block);
        r.k = r.tagged ? (a.z == 4 ? ll_tagged<4> : a.z == 6 ? ll_tagged<6> : ll_tagged<0>)
              : spt == 1 ? ll_persistent<1, 0, false> : ll_kernel_z<2, false>(a.z);
        ASD_CUDA_TRY(allow_smem(r.k, kLLMaxSmem));
        int per_sm = 0;
        ASD_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, r.k, (int)r.block,
                                                                   r.smem));
        if ((int64_t)per_sm * sms >= r.grid) *out = r;
        return ASD_OK;
    }
    return ASD_OK;
}

// The whole run with the work buffers at ws (16-byte aligned, ws_bytes >= 48 per site-sample)
// and the barrier count at bar.
int ll_run(const LLArgs &a, const LLRoute &rt, const float *spins0, float dt, int n_frames,
           int stride, float *traj, float *spins_out, void *ws, size_t ws_bytes, unsigned *bar,
           cudaStream_t s)
{
    const int64_t n = a.N * a.S;
    const int64_t steps = (int64_t)(n_frames - 1) * stride;
    if (rt.k) {
        LLRun r{};
        r.a = a;
        r.Y = static_cast<float4 *>(ws);
        r.T1 = r.Y + n;
        r.T2 = r.T1 + n;
        // (the state between launches goes through the first 12 bytes per site of T1, or of a
        // part of the work area that ll_tagged does not use)
        float *mid = reinterpret_cast<float *>(r.T1);
        if (rt.tagged) {
            const int keep = steps > kLLStepsPerLaunch ? 1 : 0;
            r.n_buf = (int)std::min<size_t>(kLLMaxBufs, ws_bytes / (sizeof(float4) * n) - keep);
            mid = reinterpret_cast<float *>(r.Y + (int64_t)r.n_buf * n);
        }
        r.bar = bar;
        r.traj = traj;
        r.F = n_frames;
        r.stride = stride;
        r.dt = dt;
        r.stage_frames = rt.stage_frames;
        r.per_block = rt.per_block;
        r.err = device_error_word();
        if (!r.err) return ASD_ECUDA;
        const float *in = spins0;
        int64_t st = 0;
        do {
            r.step0 = st;
            r.step1 = std::min<int64_t>(steps, st + kLLStepsPerLaunch);
            r.in = in;
            r.out = r.step1 == steps ? spins_out : mid;
            if (rt.local) {
                rt.k<<<rt.grid, rt.block, rt.smem, s>>>(r);
                ASD_CUDA_TRY(cudaGetLastError());
            } else {
                ASD_CUDA_TRY(cudaMemsetAsync(bar, 0, sizeof(unsigned), s));
                void *args[] = {&r};
                ASD_CUDA_TRY(cudaLaunchCooperativeKernel((const void *)rt.k, dim3(rt.grid),
                                                         dim3(rt.block), args, rt.smem, s));
            }
            in = r.out;
            st = r.step1;
        } while (st < steps);
        return ASD_OK;
    }
    const size_t bytes = sizeof(float) * 3 * (size_t)n;
    // every buffer is written before it is read: Y by the copy, acc by stage 1, T1 / T2
    // by the stage that produces them, so no clearing is needed
    float *Y = static_cast<float *>(ws), *T1 = Y + 3 * n, *T2 = Y + 6 * n, *acc = Y + 9 * n;
    const unsigned blocks = (unsigned)((n + 255) / 256);
    ASD_CUDA_TRY(cudaMemcpyAsync(Y, spins0, bytes, cudaMemcpyDeviceToDevice, s));
    write_frame0<<<blocks, 256, 0, s>>>(Y, a.N, a.S, traj, n_frames);
    for (int f = 1; f < n_frames; ++f) {
        for (int k = 0; k < stride; ++k) {
            const int frame = k == stride - 1 ? f : -1;
            rk4_stage<1><<<blocks, 256, 0, s>>>(a, Y, Y, T1, acc, dt, traj, n_frames, -1);
            rk4_stage<2><<<blocks, 256, 0, s>>>(a, Y, T1, T2, acc, dt, traj, n_frames, -1);
            rk4_stage<3><<<blocks, 256, 0, s>>>(a, Y, T2, T1, acc, dt, traj, n_frames, -1);
            rk4_stage<4><<<blocks, 256, 0, s>>>(a, Y, T1, nullptr, acc, dt, traj, n_frames, frame);
        }
    }
    ASD_CUDA_TRY(cudaGetLastError());
    if (spins_out)
        ASD_CUDA_TRY(cudaMemcpyAsync(spins_out, Y, bytes, cudaMemcpyDeviceToDevice, s));
    return ASD_OK;
}

}  // namespace
}  // namespace asd

using namespace asd;

extern "C" int asd_ll_integrate(const asd_system *sys, int n_samples, const float *spins0,
                                float dt, int n_frames, int stride, float *traj, float *spins_out,
                                void *stream)
{
    ASD_CHECK_ARG(sys && spins0 && traj, "null argument");
    ASD_CHECK_ARG(sys->n_sites >= 1 && sys->z >= 0 && sys->z <= 32, "bad system");
    ASD_CHECK_ARG(sys->z == 0 || (sys->nbr && sys->J), "neighbour table required");
    ASD_CHECK_ARG(n_samples >= 1 && n_frames >= 1 && stride >= 1, "bad n_samples/n_frames/stride");
    cudaStream_t s = (cudaStream_t)stream;
    LLArgs a{sys->n_sites, n_samples, sys->z, sys->nbr, sys->J, sys->Hz, sys->D, sys->A};
    LLRoute rt;
    int rc = ll_route(a, &rt);
    if (rc) return rc;
    const int64_t n = sys->n_sites * n_samples;
    char *ws = nullptr;
    // (a block per sample in one launch keeps everything on chip)
    const bool need = !rt.local || (int64_t)(n_frames - 1) * stride > kLLStepsPerLaunch;
    const size_t bytes = (rt.tagged ? 16 * (kLLMaxBufs + 1) : 48) * (size_t)n;
    if (need) ASD_CUDA_TRY(cudaMallocAsync(&ws, bytes + 16, s));
    rc = ll_run(a, rt, spins0, dt, n_frames, stride, traj, spins_out, ws, bytes,
                reinterpret_cast<unsigned *>(ws + bytes), s);
    if (need) cudaFreeAsync(ws, s);
    return rc;
}

// ---------------------------------------------------------------------------------------
// No-allocation variant: the same RK4 launches with their four work buffers (state,
// two stage inputs, derivative sum) carved from one fixed device array reserved with the
// library, for callers that cannot allocate device memory (see include/asd.h).
// ---------------------------------------------------------------------------------------
#include <mutex>

namespace asd {
namespace {

constexpr int64_t kLLStaticMaxSiteSamples = 1 << 18;  // n_sites * n_samples limit
constexpr int kLLStaticMaxDevices = 64;

// 48 B x 262144 site-samples = 12 MiB per device (three 16-byte state buffers, or four 12-byte
// ones), then the grid barrier's count
static __device__ __align__(256) float g_ll_scratch[4 * 3 * kLLStaticMaxSiteSamples + 64];

std::mutex g_ll_scratch_mu;
struct ScratchSlot {
    unsigned long long ctx_id;  // context the address belongs to (0: not looked up)
    float *addr;
};
ScratchSlot g_ll_scratch_slot[kLLStaticMaxDevices] = {};

// Unique ID of the calling thread's current context (cuCtxGetId through the runtime's
// driver entry point; no link against libcuda), or 0 when the query is unavailable.
typedef CUresult (*PFN_ctxGetCurrent)(CUcontext *);
typedef CUresult (*PFN_ctxGetId)(CUcontext, unsigned long long *);
unsigned long long current_context_id()
{
    static PFN_ctxGetCurrent get_cur = nullptr;
    static PFN_ctxGetId get_id = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *a = nullptr, *b = nullptr;
        cudaDriverEntryPointQueryResult qa, qb;
        if (cudaGetDriverEntryPoint("cuCtxGetCurrent", &a, cudaEnableDefault, &qa) == cudaSuccess &&
            qa == cudaDriverEntryPointSuccess &&
            cudaGetDriverEntryPoint("cuCtxGetId", &b, cudaEnableDefault, &qb) == cudaSuccess &&
            qb == cudaDriverEntryPointSuccess) {
            get_cur = reinterpret_cast<PFN_ctxGetCurrent>(a);
            get_id = reinterpret_cast<PFN_ctxGetId>(b);
        }
    });
    if (!get_cur || !get_id) return 0;
    CUcontext c = nullptr;
    unsigned long long id = 0;
    if (get_cur(&c) != CUDA_SUCCESS || !c || get_id(c, &id) != CUDA_SUCCESS) return 0;
    return id;
}

// Device address of g_ll_scratch in the current context.  In host code the symbol itself
// is only a host-side stand-in; kernels must be given this address.  It is looked up
// once per device and again whenever the device's context has changed (after
// cudaDeviceReset the module, and with it the array, lives at a new address).
int ll_scratch_address(float **out)
{
    int dev = 0;
    ASD_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kLLStaticMaxDevices) {
        set_error_text("asd_ll_integrate_noalloc: device index out of range");
        return ASD_EUNSUPPORTED;
    }
    // (cudaGetDevice above leaves the device's primary context current for this thread
    // once the runtime has initialised it; with no context to identify, id is 0 and the
    // address is looked up on every call)
    const unsigned long long id = current_context_id();
    std::lock_guard<std::mutex> lock(g_ll_scratch_mu);
    ScratchSlot &sl = g_ll_scratch_slot[dev];
    if (!sl.addr || id == 0 || sl.ctx_id != id) {
        void *p = nullptr;
        ASD_CUDA_TRY(cudaGetSymbolAddress(&p, g_ll_scratch));
        sl.addr = static_cast<float *>(p);
        sl.ctx_id = id;
    }
    *out = sl.addr;
    return ASD_OK;
}

}  // namespace
}  // namespace asd

extern "C" int asd_ll_integrate_noalloc(const asd_system *sys, int n_samples, const float *spins0,
                                        float dt, int n_frames, int stride, float *traj,
                                        float *spins_out, void *stream)
{
    ASD_CHECK_ARG(sys && spins0 && traj, "null argument");
    ASD_CHECK_ARG(sys->n_sites >= 1 && sys->z >= 0 && sys->z <= 32, "bad system");
    ASD_CHECK_ARG(sys->z == 0 || (sys->nbr && sys->J), "neighbour table required");
    ASD_CHECK_ARG(n_samples >= 1 && n_frames >= 1 && stride >= 1, "bad n_samples/n_frames/stride");
    ASD_CHECK_ARG(sys->n_sites * (int64_t)n_samples <= kLLStaticMaxSiteSamples,
                  "asd_ll_integrate_noalloc: n_sites * n_samples exceeds the fixed work area "
                  "(262144 site-samples); use asd_ll_integrate");
    float *ws = nullptr;
    int rc = ll_scratch_address(&ws);
    if (rc) return rc;
    LLArgs a{sys->n_sites, n_samples, sys->z, sys->nbr, sys->J, sys->Hz, sys->D, sys->A};
    LLRoute rt;
    rc = ll_route(a, &rt);
    if (rc) return rc;
    return ll_run(a, rt, spins0, dt, n_frames, stride, traj, spins_out, ws,
                  sizeof(float) * 4 * 3 * (size_t)kLLStaticMaxSiteSamples,
                  reinterpret_cast<unsigned *>(ws + 4 * 3 * kLLStaticMaxSiteSamples),
                  (cudaStream_t)stream);
}
