// Tensor-core forms (TF32, BF16, split-BF16): fused contraction + reduction epilogue.
//
// The method casts the pair sum of Eq. 4 / Eq. 5 for one time displacement as a GEMM
// G_t = A_t B^T (Section 3.2) and fuses the element-wise reduction that follows it --
// the bin sums or the phase-weighted inner product of Eq. 3 / Eq. 6 -- into the GEMM
// epilogue so that G_t never reaches memory (Sections 3.3-3.4).  On sm_103a this is:
//
//   warp 0      TMA producer: streams 128-row A tiles (K-offset windows of the
//               trajectory copies) and BN-row B tiles into a shared-memory ring;
//   warp 1      allocates TMEM and, from one thread, issues tcgen05.mma into one of two
//               128 x BN FP32 accumulators in tensor memory (double buffered), committing
//               each stage back to the ring and each finished work item to the epilogue;
//   then one    geometry: one tile ahead of the epilogue, loads the tile's column geometry
//               into one of two shared-memory buffers and finds its bin window(s);
//   then four   (tiles of at most 192 columns) read the phase product out of TMEM, one warp
//               per lane quarter;
//   warps 2..   epilogue (EW = 4 or 8 warps): reads the accumulator from TMEM and
//               reduces it -- per-thread private FP32 bins in shared memory
//               (conflict-free [bin][row] layout), phase weights from per-site cos/sin
//               tables -- then FP64 per-CTA sums and FP64 atomics into the outputs.
//
// The accumulator living in TMEM plays the role of the paper's OTF_SM shared-memory
// staging of the C tile (Section 3.4): the epilogue never holds the tile in registers.
// The per-pair phase factor uses cos(a - b) = cos a cos b + sin a sin b (and
// sin(a - b) = sin a cos b - cos a sin b for the sine part) on tables made once per
// plan, so no transcendental is evaluated per pair (the register-spill problem of the
// paper's OTF_REG variant).
//
// Persistent: one CTA per SM (or one CTA pair per two SMs) takes (problem, t, row tile,
// column tile) work items in grouped raster order (raster_m row tiles per group, 16 by
// default) so concurrently running CTAs share A and B panels in L2; the TMA thread claims
// each item from a global counter (or, static, takes every n-th) and passes its K chunks,
// one sub-item each, to the other roles.  Several problems (a batched ensemble) share the
// list.  Every wait is bounded: after kTimeoutNs a role records an error in the device
// error word and stops; the CTA then drains its own in-flight copies and MMAs, frees TMEM
// and exits.
#pragma once

#include <cuda_bf16.h>

#include "asd_internal.h"
#include "geom.cuh"

namespace asd {
namespace {

// Epilogue warps EW (template parameter): 4 (one per TMEM lane quarter, all columns) or
// 8 (two per quarter, half the columns each).  Threads = TMA warp + MMA warp + EW warps +
// geometry warp + phase read-out warps.
constexpr int kMaxEpiWarps = 8;
constexpr unsigned long long kTimeoutNs = 4000000000ull;
// TMEM: 512 columns per CTA (one CTA per SM): two BN-column accumulators, then (phase
// workloads, BN <= 192) the 128-column phase product P of one pass of 64 q-vectors.
constexpr uint32_t kTmemAlloc = 512;
constexpr int kPCols = 2 * kPhaseQ;           // u (cosine weights) and v (sine weights)
constexpr uint32_t kWBytes = 128u * 128u;     // one plane of a W stage: 128 rows x 64 BF16
// Work items are handed from the TMA thread to the MMA thread and the epilogue warps
// through a ring of kWQ slots in shared memory.  With the dynamic schedule the TMA thread
// claims each item from a global counter, so the items in flight across the grid stay
// together whatever each item costs (L2 reuse of A / B panels, no drift, balanced tail);
// the static schedule takes, in round k of n CTAs, item k n + (cid + k) mod n.
//
// A slot holds the decoded sub-item, so only the TMA thread decodes (its 64-bit divisions
// and descriptor reads cost every epilogue thread 0.7 to 2.1 thousand cycles per sub-item
// before), and it decodes the next item in the middle of the current one's K blocks, its
// claim from the counter made an item earlier still.
constexpr int kWQ = 4;
struct __align__(16) WorkSlot {
    int p;          // problem, -1: no work left
    int t, m0, n0;  // displacement, first row and column of the tile
    int row_end;
    int kci;        // K chunk of the tile, 0: first
    int last;       // 1: the tile's last chunk
    int nk;         // K blocks of the chunk
};
// Private bins are a [bin][128 * EW/4] array: epilogue thread (row r, column half h)
// only ever touches column r + 128 h, i.e. bank r mod 32, so the per-pair accumulation
// is free of bank conflicts whatever the bins of the 32 lanes are (with an odd stride,
// bins that fall as the row index rises put a whole warp on one bank).  The per-tile
// flush reads whole bin rows warp-cooperatively (bin_stride, asd_internal.h).

// ------------------------------------------------------------------------------------
// PTX wrappers
// ------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t saddr(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ unsigned long long gtimer()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait for the phase with the given parity; false after kTimeoutNs (the error
// word then holds `code`).  (A CTA pair's waits on barriers the other CTA signals use the
// same test: the tcgen05 fences around the arrive and the wait order the tensor-memory
// accesses, and TMA and MMA completions are counted by the barrier itself; a cluster-scope
// acquire in every wait measured 30 % slower.)  Inlined: as a call its saved registers were
// spilled around every wait of every role; 48^3 glass BF16 94.0 -> 84.1 ms (86.0 since the phase
// product has a conversion barrier per accumulator), 32^3 glass
// split-BF16 19.3 -> 18.8 ms.
__device__ __forceinline__ bool mbar_wait_for(uint32_t bar, uint32_t parity, int *err, int code,
                                          unsigned long long limit_ns)
{
    if (mbar_test(bar, parity)) return true;
    const unsigned long long t0 = gtimer();
    for (uint32_t it = 1;; ++it) {
        if (mbar_test(bar, parity)) return true;
        if ((it & 1023u) == 0 && gtimer() - t0 > limit_ns) {
            atomicCAS(err, 0, code);
            return false;
        }
    }
}

__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, int *err, int code)
{
    return mbar_wait_for(bar, parity, err, code, kTimeoutNs);
}

// ---- CTA pairs (tcgen05 cta_group::2): two CTAs of a cluster share one 256-row MMA ----
__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

// Shared-memory address of the same variable in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t mapa(uint32_t addr, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}

__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Arrive on a barrier of any CTA of the cluster (release at cluster scope).
__device__ __forceinline__ void mbar_arrive_cl(uint32_t cl_addr)
{
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cl_addr)
                 : "memory");
}

// TMA tile load into this CTA's shared memory whose completion is counted on a barrier
// of the pair's first CTA (cl_bar: a cluster address).
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap *map,
                                                 uint32_t cl_bar, int x, int y)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile"
        ".mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(cl_bar), "r"(x), "r"(y)
        : "memory");
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, uint32_t bar,
                                            int x, int y)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4}], [%2];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(x), "r"(y)
        : "memory");
}

// TMEM allocation by one warp; with CG = 2 one warp of each CTA of the pair performs it
// together (the same columns in both CTAs).
template <int CG>
__device__ __forceinline__ void tmem_alloc(uint32_t dst_slot, uint32_t ncols)
{
    if constexpr (CG == 2) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         dst_slot),
                     "r"(ncols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         dst_slot),
                     "r"(ncols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
}

template <int CG>
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols)
{
    if constexpr (CG == 2)
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr),
                     "r"(ncols)
                     : "memory");
    else
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr),
                     "r"(ncols)
                     : "memory");
}

__device__ __forceinline__ void tc_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Arrive on `bar` (a cluster address with CG = 2: this CTA's or the peer's) once the
// MMAs this thread issued so far have completed.
template <int CG = 1>
__device__ __forceinline__ void tc_commit(uint32_t bar)
{
    if constexpr (CG == 2)
        asm volatile(
            "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
            : "memory");
    else
        asm volatile(
            "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
            : "memory");
}

// D (TMEM) = / += A B^T with A and B in shared memory.  CG = 2: a 256-row MMA over the
// pair, A rows 0-127 and B columns 0-N/2 from this CTA, the rest from the peer at the
// same addresses, D rows split between the two CTAs' TMEM.
template <bool TF32, int CG = 1>
__device__ __forceinline__ void tc_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc,
                                       uint32_t acc)
{
    if constexpr (CG == 2) {
        if (TF32)
            asm volatile(
                "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                "tcgen05.mma.cta_group::2.kind::tf32 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
                "l"(a), "l"(b), "r"(idesc), "r"(acc));
        else
            asm volatile(
                "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
                "l"(a), "l"(b), "r"(idesc), "r"(acc));
    } else {
        if (TF32)
            asm volatile(
                "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
                "l"(a), "l"(b), "r"(idesc), "r"(acc));
        else
            asm volatile(
                "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
                "l"(a), "l"(b), "r"(idesc), "r"(acc));
    }
}

// MMA with the A operand in tensor memory (128 lanes = rows, K along the columns, two
// BF16 elements per 32-bit column, the even element in the low half) and B in shared
// memory: the phase product P = G W of the epilogue.
template <int CG = 1>
__device__ __forceinline__ void tc_mma_ts(uint32_t d, uint32_t a_tmem, uint64_t b, uint32_t idesc,
                                          uint32_t acc)
{
    if constexpr (CG == 2)
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::2.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d),
            "r"(a_tmem), "l"(b), "r"(idesc), "r"(acc));
    else
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d),
            "r"(a_tmem), "l"(b), "r"(idesc), "r"(acc));
}

// 32 lanes x 8 consecutive 32-bit columns (this thread's lane), and its wait, tied to the
// registers.
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                   "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait8x2(uint32_t (&a)[8], uint32_t (&b)[8])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(a[4]), "+r"(a[5]),
                   "+r"(a[6]), "+r"(a[7]), "+r"(b[0]), "+r"(b[1]), "+r"(b[2]), "+r"(b[3]),
                   "+r"(b[4]), "+r"(b[5]), "+r"(b[6]), "+r"(b[7])
                 :
                 : "memory");
}

// Store 16 consecutive 32-bit columns of this thread's lane; complete after tmem_wait_st.
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
        "%11, %12, %13, %14, %15, %16};" ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]),
        "r"(r[15])
        : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Issue half of tmem_ld32: the registers are valid only after tmem_wait32 on them.
__device__ __forceinline__ void tmem_ld32_issue(uint32_t taddr, uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
        "%11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, "
        "%28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
          "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
          "=r"(r[31])
        : "r"(taddr));
}

// Wait for the TMEM loads of this thread; tied to the registers so no use of them can be
// scheduled before it.
__device__ __forceinline__ void tmem_wait32(uint32_t (&r)[32])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]),
                   "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]),
                   "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]), "+r"(r[16]), "+r"(r[17]),
                   "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]),
                   "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]),
                   "+r"(r[30]), "+r"(r[31])
                 :
                 : "memory");
}

// 32 lanes x 32 consecutive 32-bit columns; the wait is tied to the registers so no
// use of them can be scheduled before it.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
        "%11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, "
        "%28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
          "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
          "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]),
                   "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]),
                   "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]), "+r"(r[16]), "+r"(r[17]),
                   "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]),
                   "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]),
                   "+r"(r[30]), "+r"(r[31])
                 :
                 : "memory");
}

__device__ __forceinline__ void epi_sync(int nthreads)
{
    __syncwarp();
    asm volatile("bar.sync 1, %0;" ::"r"(nthreads) : "memory");
}

// Epilogue barrier that also ANDs a flag over the epilogue threads (128 or 256), so that every
// thread takes the same branch after a bounded wait.
__device__ __forceinline__ bool epi_sync_and(bool v, int nthreads)
{
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\t"
        "bar.red.and.pred q, 1, %2, p;\n\tselp.u32 %0, 1, 0, q;\n}\n"
        : "=r"(r)
        : "r"((uint32_t)v), "r"(nthreads)
        : "memory");
    return r != 0;
}

// Shared-memory matrix descriptor, K-major, swizzled (128B: mode 2, 64B: mode 4).
// SBO = 8 rows x swizzle span; LBO unused for swizzled K-major; version 1 (sm_100).
__device__ __forceinline__ uint64_t sdesc(uint32_t addr, int swb)
{
    uint64_t d = (uint64_t)((addr & 0x3FFFFu) >> 4);
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)((8u * swb) >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)(swb == 128 ? 2 : 4) << 61;
    return d;
}

// Instruction descriptor: FP32 accumulate, A/B = BF16 (1) or TF32 (2), both K-major,
// N columns, M rows (128, or 256 for a CTA pair).
__host__ __device__ constexpr uint32_t idesc(bool tf32, int N, int M = kBM)
{
    return (1u << 4) | ((tf32 ? 2u : 1u) << 7) | ((tf32 ? 2u : 1u) << 10) |
           ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// ------------------------------------------------------------------------------------
// shared-memory layout of the epilogue region
// ------------------------------------------------------------------------------------
// Bin window(s) of a tile.  One window: private row k holds bin blo + k.  Positions whose
// columns join two far-apart groups of sites may take two: rows [0, n1) for bins blo + k
// (column chunks before `split`), rows [n1, nwp) for bins blo2 + k - n1.
struct TileWindow {
    int blo, blo2, n1, nwp, split;
    int bhi;       // largest bin the tile can keep (positions)
    int fit;       // positions: every kept bin of the tile is in the window(s)
    int pad;
};

struct EpiLayout {
    uint32_t cacc, qacc, fb, geo, win, par, var, total;
};

__host__ __device__ inline uint32_t take(uint32_t &o, uint32_t bytes)
{
    o = (o + 15u) & ~15u;
    uint32_t r = o;
    o += bytes;
    return r;
}

// The per-problem part of the epilogue's shared memory: the private bins (NW + 1 rows,
// the last one the trash row of dropped pairs) followed by the bin threshold pairs (FP32)
// or, for lattices, the d2 -> bin table (uint16).  A batched launch sizes it for the
// largest problem and lays it out again whenever the problem changes.
__host__ __device__ inline uint32_t var_bins_bytes(int NW, int ew)
{
    return (4u * (NW + 1) * bin_stride(ew) + 15u) & ~15u;
}
__host__ __device__ inline uint32_t var_bytes(int NW, int nb, int nlut, int ew)
{
    const uint32_t tb = 8u * (nb + 1), lb = 2u * nlut;
    return var_bins_bytes(NW, ew) + (((tb > lb ? tb : lb) + 15u) & ~15u);
}

// Epilogue shared memory: the fixed arrays (sized for the largest n_bins / n_q of the
// launch) and the per-problem region of `vb` bytes.
__host__ __device__ inline EpiLayout epi_layout(uint32_t vb, int nb, int nq, int BN, int ew,
                                                int det)
{
    EpiLayout L;
    uint32_t o = 0;
    // per-CTA bin sums (FP64, or 64-bit fixed point in the deterministic mode)
    L.cacc = take(o, 8u * (nb > 0 ? nb : 1));
    // phase sums per TMEM lane quarter and (q, part), nq = n_q * parts (FP64 or fixed point);
    // each quarter's sums belong to its read-out warp
    L.qacc = take(o, 8u * 4 * (nq > 0 ? nq : 1));
    // fallback bins of pairs outside the private window (FP32, or fixed point)
    L.fb = take(o, (det ? 8u : 4u) * (nb > 0 ? nb : 1));
    // two tiles' column geometry (x, y, z arrays, or one array of packed coordinates) and bin
    // windows, filled by the geometry warp
    L.geo = take(o, 2u * 12u * BN);
    L.win = take(o, 2u * (uint32_t)sizeof(TileWindow));
    // the current problem's parameters (global memory is several hundred cycles away while
    // the operand streams run)
    L.par = take(o, (uint32_t)sizeof(EpiParams) + 16u);
    L.var = take(o, vb);
    L.total = (o + 1023u) & ~1023u;
    return L;
}

// Per-role walk over the work list: the fields that decoding needs stay in registers until
// the problem changes (a batched launch would otherwise search the descriptors per item).
struct WorkCursor {
    int p = -1;
    int64_t begin = 0, end = 0;  // flattened work items [begin, end) belong to problem p
    int tiles_m, tiles_n, kch, G, nk, row_begin, row_end, t_begin;
    int nkb, F3, n_copies, Kseg, npass;
    int64_t per_t;
};

// a / b of non-negative numbers, in 32 bits where they fit (a 64-bit division takes about
// a hundred instructions).
__device__ __forceinline__ int64_t div_small(int64_t a, int64_t b)
{
    if (((a | b) >> 32) == 0) return (int64_t)((uint32_t)a / (uint32_t)b);
    return a / b;
}

// A tile of the work list.
struct TileInfo {
    int t, m0, n0;
};

// Work item tau = one (problem, displacement, row tile, column tile) in grouped raster order;
// its K chunks are consecutive sub-items on the same CTA (they share the tile's geometry and
// private bins).  Row tiles are row_step rows (256 for a CTA pair, whose second CTA takes
// rows row_off = 128 on).
__device__ __forceinline__ TileInfo decode(WorkCursor &cu, const TcProblem *__restrict__ probs,
                                           int n_probs, const TcDims &one, const TcOverride &ov,
                                           int64_t tau, int BN, int row_step, int row_off)
{
    if (cu.p < 0 || tau >= cu.end) {
        int p = cu.p < 0 ? 0 : cu.p;
        while (p + 1 < n_probs && probs[p + 1].tile_begin <= tau) ++p;
        const TcDims P = n_probs == 1 ? one : probs[p].dims;
        cu.p = p;
        const int tiles_m = ov.active ? ov.tiles_m : P.tiles_m;
        cu.begin = ov.active ? 0 : probs[p].tile_begin;
        cu.end = cu.begin + (ov.active ? ov.n_tiles : probs[p].n_tiles);
        cu.tiles_m = tiles_m;
        cu.tiles_n = P.tiles_n;
        cu.kch = P.k_chunks;
        cu.G = max(1, P.group_m);
        cu.nkb = P.nkb;
        cu.nk = P.S * P.nkb;
        cu.F3 = P.F3;
        cu.n_copies = P.n_copies;
        cu.Kseg = P.Kseg;
        cu.npass = P.npass;
        cu.row_begin = ov.active ? ov.row_begin : P.row_begin;
        cu.row_end = ov.active ? ov.row_end : P.row_end;
        cu.t_begin = ov.active ? ov.t_begin : 0;
        cu.per_t = (int64_t)cu.tiles_m * cu.tiles_n;
    }
    const int64_t l = tau - cu.begin;
    const int64_t t = div_small(l, cu.per_t), rem = l - t * cu.per_t;
    const int64_t gspan = (int64_t)cu.G * cu.tiles_n;
    const int64_t grp = div_small(rem, gspan), r2 = rem - grp * gspan;
    const int first_m = (int)grp * cu.G;
    const int gsz = min(cu.G, cu.tiles_m - first_m);
    const int64_t col = div_small(r2, gsz);
    TileInfo ti;
    ti.t = cu.t_begin + (int)t;
    ti.m0 = cu.row_begin + (first_m + (int)(r2 - col * gsz)) * row_step + row_off;
    ti.n0 = (int)col * BN;
    return ti;
}

// Exact bin of an FP32 d2 from a table of threshold pairs thr2[k] = (thr[k], thr[k+1]),
// thr[k] = (k w)^2 rounded up to FP32: a first guess from the square root, then one
// 8-byte load corrects it by one either way (the same result as two dependent fix-ups,
// since the guess is within one bin).  Returns 0 .. n_bins + 1 (>= n_bins: dropped).
__device__ __forceinline__ int bin_of_d2_pair(float d2, float inv_w, int nb,
                                              const float2 *__restrict__ thr2, int *err)
{
    const float r = d2 * rsqrtf(fmaxf(d2, 1e-30f));
    const int k = min((int)(r * inv_w), nb);
    if (!ASD_INB(k >= 0, BND_THR, err)) return nb;  // dropped
    (void)err;
    const float2 t = thr2[k];
    return k + (d2 >= t.y ? 1 : 0) - (d2 < t.x ? 1 : 0);
}

// Per-tile constants of the binning epilogue, held in registers.
struct BinArgs {
    int Lx, Ly, Lz, periodic;
    float inv_w;
    int nb, blo, nwp, trash;
    int NB;                  // fallback bins of the launch
    int n_lut;
    double fscale;           // fixed-point scale (deterministic mode), else 0
    int *err;
};

enum { BIN_LUT = 0, BIN_THR = 1, BIN_POS = 2 };

// The values of N pairs (of a chunk, from column k0 on) into this thread's private bins (slot >= 0)
// or the shared fallback bins (slot -1 - bin), in column order.
template <int STRIDE, int N>
__device__ __forceinline__ void add_slots(const uint32_t (&g)[32], int k0, const int (&slot)[N],
                                          bool row_ok,
                                          float *__restrict__ myb, void *__restrict__ fbv,
                                          const BinArgs &ba)
{
    const bool det = ba.fscale != 0.0;
#pragma unroll
    for (int k = 0; k < N; ++k) {
        // rows past the range: their accumulator rows may come from A rows that were
        // never prepared, so the value is replaced (a product with 0 would keep a NaN)
        const float val = row_ok ? __uint_as_float(g[k0 + k]) : 0.f;
        if (slot[k] < 0) {
            const int b = -1 - slot[k];
            if (!ASD_INB(b < ba.NB, BND_FALLBACK, ba.err)) continue;
            // deterministic mode: fixed-point sums (integer adds in any order)
            if (det) add_fixed(static_cast<long long *>(fbv) + b, to_fixed(val, ba.fscale));
            else atomicAdd(static_cast<float *>(fbv) + b, val);
        } else if (ASD_INB(slot[k] <= ba.trash, BND_PRIV, ba.err)) {
            myb[slot[k] * STRIDE] += val;
        }
    }
}

// Bin 32 consecutive columns of one accumulator row.  Phase 1 computes the exact bin
// slot of every pair (loads of geometry and tables only, so the 32 independent chains
// overlap); phase 2 adds the 32 values into this thread's private bins (its column of
// the [bin][STRIDE] array) or, for bins outside the window, into the shared fallback
// bins.  Without a window, blo = 0 and nwp = nb, so every kept bin is private.
// MODE: BIN_LUT (lattice, d2 -> bin table), BIN_THR (lattice, thresholds), BIN_POS
// (FP32 positions, thresholds).
template <int MODE, int STRIDE>
__device__ __forceinline__ void bin_chunk(const uint32_t (&g)[32], bool row_ok, int4 ri, float4 rp,
                                          const float *__restrict__ cg, int BN,
                                          const float *__restrict__ thr,
                                          float *__restrict__ myb, void *__restrict__ fbv,
                                          const BinArgs ba)
{
    int slot[32];
#pragma unroll
    for (int k = 0; k < 32; ++k) {
        const float4 cj4 = make_float4(cg[k], cg[BN + k], cg[2 * BN + k], 0.f);
        int b;
        if (MODE == BIN_POS) {
            b = bin_of_d2_pair(position_d2(rp, cj4), ba.inv_w, ba.nb,
                               reinterpret_cast<const float2 *>(thr), ba.err);
        } else {
            const int4 cj = make_int4(__float_as_int(cj4.x), __float_as_int(cj4.y),
                                      __float_as_int(cj4.z), 0);
            const int d2 = lattice_d2i(ri, cj, ba.Lx, ba.Ly, ba.Lz, ba.periodic);
            if (MODE == BIN_LUT)
                b = ASD_INB((unsigned)d2 < (unsigned)ba.n_lut, BND_LUT, ba.err)
                        ? reinterpret_cast<const uint16_t *>(thr)[d2]
                        : ba.nb;
            else
                b = bin_of_d2_pair((float)d2, ba.inv_w, ba.nb,
                                   reinterpret_cast<const float2 *>(thr), ba.err);
        }
        const int lb = b - ba.blo;
        slot[k] = (unsigned)lb < (unsigned)ba.nwp ? lb : (b < ba.nb ? -1 - b : ba.trash);
    }
    add_slots<STRIDE>(g, 0, slot, row_ok, myb, fbv, ba);
}

// ---- branch-free binning: packed FP32 pairs, two columns per instruction ----
// Issue slots bound this part of the epilogue (two warps per scheduler share the slots of
// a column's ~50 instructions), so the distance, the guess and the threshold of two
// columns go through the packed add / mul / fma (one issue for two FP32 results, each
// rounded as the scalar instruction rounds it).  Measured with the grouped adds below
// against scalar instructions, two-sided thresholds and one add after the other (64 q in
// all): 48^3 glass BF16, 2 displacements 139.8 -> 118.3 ms, 32^3 glass split-BF16 22.6 ->
// 22.0 ms (its other epilogue parts bound it); lattices with the shorter distance below
// and the grouped adds: 24-sample ensemble 33.7 -> 30.6 ms, 34^3 with K = 444 35.2 -> 26.9.
__device__ __forceinline__ uint64_t pack2(float a, float b)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float &a, float &b)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ float sqrt_guess(float x)
{
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Constants of the branch-free rule for one tile: 1 / w and w in both halves, the word
// offset rule off = bin * STRIDE + c0 (c0 takes out the window start and the 2^23 bias of
// a bin's float form), n_bins, and the trash row of dropped pairs.
struct FastBin {
    uint64_t inv2, w2;
    const float2 *thr2;
    int nb;
    uint32_t c0, trash_off;
};
constexpr float kBinBase = 8388608.f;          // 2^23: its float holds an integer below
constexpr uint32_t kBinBaseBits = 0x4B000000u; // 2^23 in the low bits

// Private-bin word offsets of two columns from their squared distances.  The guess is
// sqrt(d2) / w rounded to nearest, k or k + 1 for an exact bin k (the square root is good
// to 2^-22, a bin to n_bins <= 4096, so the error is below 1e-2 of a bin), so one threshold
// decides: bin = guess - (d2 < thr[guess]).  Adding 2^23 rounds without a conversion (like
// the square root those run on the quarter-rate unit).  EXACT: thr[k] = RN(RN(k w)^2) for
// every k (the host checks the table), computed; else loaded.  DROP: pairs at n_bins and
// beyond exist and go to the trash row; otherwise every bin is below n_bins.  Finite
// coordinates only (the plan checks them; others take the general rule).
template <bool EXACT, bool DROP, int STRIDE>
__device__ __forceinline__ void bin2(uint32_t &o0, uint32_t &o1, uint64_t d2, const FastBin &fb)
{
    float s0, s1, r0, r1, l0, l1;
    unpack2(d2, s0, s1);
    uint64_t x = mul2(pack2(sqrt_guess(s0), sqrt_guess(s1)), fb.inv2);
    if (DROP) {
        unpack2(x, r0, r1);
        x = pack2(fminf(r0, (float)fb.nb), fminf(r1, (float)fb.nb));
    }
    const uint64_t g = add2(x, pack2(kBinBase, kBinBase));
    unpack2(g, r0, r1);
    if (EXACT) {
        const uint64_t kw = mul2(add2(g, pack2(-kBinBase, -kBinBase)), fb.w2);
        unpack2(mul2(kw, kw), l0, l1);
    } else {
        l0 = fb.thr2[__float_as_uint(r0) - kBinBaseBits].x;
        l1 = fb.thr2[__float_as_uint(r1) - kBinBaseBits].x;
    }
    const uint32_t b0 = __float_as_uint(r0) - (s0 < l0 ? 1u : 0u);
    const uint32_t b1 = __float_as_uint(r1) - (s1 < l1 ? 1u : 0u);
    o0 = b0 * STRIDE + fb.c0;
    o1 = b1 * STRIDE + fb.c0;
    if (DROP) {
        const uint32_t lim = kBinBaseBits + (uint32_t)fb.nb;
        o0 = b0 < lim ? o0 : fb.trash_off;
        o1 = b1 < lim ? o1 : fb.trash_off;
    }
}

// FP32 positions: the squared distance is position_d2's, fma(dz, dz, fma(dy, dy, dx dx))
// of FP32 differences, for the row at minus (nx, ny, nz) and columns stored by component.
template <bool EXACT, bool DROP, int STRIDE, int N>
__device__ __forceinline__ void pos_offsets(uint32_t (&off)[N], uint64_t nx, uint64_t ny,
                                            uint64_t nz, const float *__restrict__ cg, int BN,
                                            const FastBin &fb)
{
#pragma unroll
    for (int k = 0; k < N; k += 4) {
        const float4 X = *reinterpret_cast<const float4 *>(cg + k);
        const float4 Y = *reinterpret_cast<const float4 *>(cg + BN + k);
        const float4 Z = *reinterpret_cast<const float4 *>(cg + 2 * BN + k);
        uint64_t d = add2(pack2(X.x, X.y), nx), s = mul2(d, d);
        d = add2(pack2(Y.x, Y.y), ny);
        s = fma2(d, d, s);
        d = add2(pack2(Z.x, Z.y), nz);
        s = fma2(d, d, s);
        bin2<EXACT, DROP, STRIDE>(off[k], off[k + 1], s, fb);
        d = add2(pack2(X.z, X.w), nx);
        s = mul2(d, d);
        d = add2(pack2(Y.z, Y.w), ny);
        s = fma2(d, d, s);
        d = add2(pack2(Z.z, Z.w), nz);
        s = fma2(d, d, s);
        bin2<EXACT, DROP, STRIDE>(off[k + 2], off[k + 3], s, fb);
    }
}

// bin_chunk for FP32 positions under the branch-free rule: tiles whose bins do not fit the private
// window.  24^3 glass in row order, 256 bins of 0.17, K = 192, 16 displacements, split-BF16: 37.2 ms
// before the binning above took registers from bin_chunk, 38.6 with it, 34.9 here.
template <int STRIDE>
__device__ __forceinline__ void pos_chunk(const uint32_t (&g)[32], bool row_ok, float4 rp,
                                          const float *__restrict__ cg, int BN,
                                          const float *__restrict__ thr, float *__restrict__ myb,
                                          void *__restrict__ fbv, const BinArgs ba)
{
    const FastBin fb = {pack2(ba.inv_w, ba.inv_w), 0ull, reinterpret_cast<const float2 *>(thr),
                        ba.nb, 0u - kBinBaseBits, (uint32_t)ba.nb};
    // (eight columns at a time: the registers of a whole chunk would be taken from the usual
    // path, 48^3 glass BF16 85.4 -> 86.7 ms; now 86.0)
#pragma unroll
    for (int h = 0; h < 32; h += 8) {
        uint32_t bin[8];
        pos_offsets<false, true, 1>(bin, pack2(-rp.x, -rp.x), pack2(-rp.y, -rp.y),
                                    pack2(-rp.z, -rp.z), cg + h, BN, fb);
        int slot[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int b = (int)bin[k], lb = b - ba.blo;
            slot[k] = (unsigned)lb < (unsigned)ba.nwp ? lb : (b < ba.nb ? -1 - b : ba.trash);
        }
        add_slots<STRIDE>(g, h, slot, row_ok, myb, fbv, ba);
    }
}

// Lattices with byte-sized extents (EpiParams::fast): coordinates packed one per byte
// (x | y<<8 | z<<16).  Per axis d = |a - b|, e = |L - 2 d| = |d - (L - d)| and the minimum
// image min(d, L - d) = (L - e) / 2, so one byte dot product of L - e gives 4 d2 (no byte
// borrows: d < L and e <= L).
__device__ __forceinline__ uint32_t pk_4d2(uint32_t c, uint32_t rpk, uint32_t Lpk)
{
    const uint32_t d = __vabsdiffu4(c, rpk);
    const uint32_t m = Lpk - __vabsdiffu4(d, Lpk - d);
    return __dp4a(m, m, 0u);
}

// Offsets from the d2 -> bin table (entries pre-scaled by the bin stride, the trash row
// for dropped pairs), or from table thresholds.
template <bool LUT, int STRIDE>
__device__ __forceinline__ void pk_offsets(uint32_t (&off)[32], uint32_t rpk, uint32_t Lpk,
                                           const uint4 *__restrict__ cpk,
                                           const void *__restrict__ tab, float inv_w, int nb,
                                           uint32_t trash_off, int n_lut, int *err)
{
    (void)n_lut;
    (void)err;
#pragma unroll
    for (int k4 = 0; k4 < 8; ++k4) {
        const uint4 c4 = cpk[k4];
        const uint32_t cc[4] = {c4.x, c4.y, c4.z, c4.w};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const uint32_t d2 = pk_4d2(cc[u], rpk, Lpk) >> 2;
            if (LUT) {
                off[4 * k4 + u] = ASD_INB(d2 < (uint32_t)n_lut, BND_LUT, err)
                                      ? reinterpret_cast<const uint16_t *>(tab)[d2]
                                      : trash_off;
            } else {
                const int b = bin_of_d2_pair((float)d2, inv_w, nb,
                                             reinterpret_cast<const float2 *>(tab), err);
                off[4 * k4 + u] = b < nb ? (uint32_t)(b * STRIDE) : trash_off;
            }
        }
    }
}

// Add 32 values to this thread's private bins, in column order.  One read-modify-write
// after the other is a chain of shared-memory latencies (the compiler may not move a load
// above a store that could be to the same bin), so four bins are loaded together and a
// value whose bin came up earlier in its group takes that sum instead of the loaded one:
// the same additions in the same order, a quarter of the chain.
__device__ __forceinline__ void add_private(float *__restrict__ mb, const uint32_t (&off)[32],
                                            const uint32_t (&g)[32], uint32_t trash_off, int *err)
{
    (void)trash_off;
    (void)err;
#pragma unroll
    for (int k = 0; k < 32; k += 4) {
        const uint32_t o0 = off[k], o1 = off[k + 1], o2 = off[k + 2], o3 = off[k + 3];
        if (!ASD_INB(max(max(o0, o1), max(o2, o3)) <= trash_off, BND_PRIV, err)) continue;
        float v0 = mb[o0], v1 = mb[o1], v2 = mb[o2], v3 = mb[o3];
        v0 += __uint_as_float(g[k]);
        v1 = (o1 == o0 ? v0 : v1) + __uint_as_float(g[k + 1]);
        v2 = (o2 == o1 ? v1 : o2 == o0 ? v0 : v2) + __uint_as_float(g[k + 2]);
        v3 = (o3 == o2 ? v2 : o3 == o1 ? v1 : o3 == o0 ? v0 : v3) + __uint_as_float(g[k + 3]);
        mb[o0] = v0;
        mb[o1] = v1;
        mb[o2] = v2;
        mb[o3] = v3;
    }
}

using LaunchArgs = TcLaunchArgs;

// Sum of 8 per-lane values over the warp's 32 lanes by recursive halving: each exchange
// sends the half of the values this lane does not keep; after three steps lanes
// 4m .. 4m + 3 hold partial sums of value m (bits 4, 3, 2 of the lane, highest first), which
// the last two exchanges add.
__device__ __forceinline__ float warp_sum8(float (&z)[8], int lane)
{
#pragma unroll
    for (int hh = 4, o = 16; hh >= 1; hh >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int k = 0; k < hh; ++k) {
            const float send = up ? z[k] : z[k + hh];
            const float keep = up ? z[k + hh] : z[k];
            z[k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    const float w = z[0] + __shfl_xor_sync(0xffffffffu, z[0], 2);
    return w + __shfl_xor_sync(0xffffffffu, w, 1);
}

__device__ __forceinline__ float warp_min(float x)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x = fminf(x, __shfl_xor_sync(0xffffffffu, x, o));
    return x;
}
__device__ __forceinline__ float warp_max(float x)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, o));
    return x;
}

// ------------------------------------------------------------------------------------
// the kernel
// ------------------------------------------------------------------------------------
// CG = 2: CTA pairs (clusters of two).  The pair computes a 256-row tile with one MMA
// thread (in the first CTA) issuing tcgen05 cta_group::2 MMAs: each CTA loads its own
// 128 A rows and half of the B columns, so per SM the operand traffic of a 256 x BN
// tile is that of a 128 x (128 + BN/2) one; each CTA's TMEM holds its 128 rows and its
// epilogue bins them.  Both CTAs walk the same fixed order of work items; the second
// CTA's epilogue warps release accumulators and phase products on the first CTA's
// barriers.
__host__ __device__ constexpr bool phase_ok(int BN) { return 2 * BN + kPCols <= (int)kTmemAlloc; }
__host__ __device__ constexpr int readout_warps(int BN) { return phase_ok(BN) ? 4 : 0; }
__host__ __device__ constexpr int tc_threads(int BN, int EW)
{
    return 32 * (3 + EW + readout_warps(BN));
}

template <int FORM, int BN, int SWB, int EW, int CG>
__global__ void __launch_bounds__(tc_threads(BN, EW), 1) pc_tc_kernel(const __grid_constant__ LaunchArgs args)
{
    constexpr int kEpiWarps = EW;
    constexpr int kEpiThreads = 32 * EW;
    constexpr int kBinStride = bin_stride(EW);
    constexpr int kHalves = EW / 4;
    constexpr int kChunks = BN / 32;                                 // 32-column chunks
    static_assert(kChunks <= 8, "one lane per column chunk");
    constexpr bool kTF32 = FORM == ASD_TF32;
    constexpr int kPlanes = FORM == ASD_SPLIT_BF16 ? 2 : 1;
    constexpr uint32_t kABytes = kBM * SWB;
    constexpr uint32_t kBBytes = (BN / CG) * SWB;   // this CTA's B columns
    constexpr uint32_t kStageBytes = kPlanes * (kABytes + kBBytes);
    constexpr int kKSteps = SWB / 32;          // one MMA k-step covers 32 bytes of K
    constexpr int kBK = SWB / (kTF32 ? 4 : 2); // K elements per stage
    constexpr uint32_t kIdesc = idesc(kTF32, BN, kBM * CG);
    // Phase weights on the tensor core (problems with n_q > 0; the plan picks BN <= 192):
    // after the epilogue has binned a K chunk of a tile it stores the chunk's G, split
    // into BF16 hi + lo, back over the accumulator's own columns (chunk of 32 columns ->
    // 16 columns of hi, then 16 of lo), and one pass of kPhaseQ q-vectors is the
    // 128 x 128 x BN product P = G W with W[c][o] = cos / sin(q_o . r_c) of the tile's
    // columns, streamed through the operand ring (64 columns c per stage).  Split-BF16 and
    // TF32 issue hi*hi + hi*lo + lo*hi (the FP32-accurate sum); BF16 issues hi*hi.
    constexpr bool kPhaseOK = phase_ok(BN);
    constexpr int kRoWarps = readout_warps(BN);
    constexpr int kWPlanes = FORM == ASD_BF16 ? 1 : 2;
    constexpr int kWStages = BN / 64;          // W stages per pass (64 columns c each)
    constexpr uint32_t kWB = kWBytes / CG;     // one W plane of this CTA (its output half)
    constexpr uint32_t kIdescP = idesc(false, kPCols, kBM * CG);
    static_assert(!kPhaseOK || (kStageBytes >= kWPlanes * kWB && BN % 64 == 0),
                  "a W stage fits a ring stage");
    static_assert(CG == 1 || CG == 2, "CTA groups of one or two");

    extern __shared__ __align__(1024) uint8_t smem_raw[];
    // 1024-byte aligned base for the swizzled tiles
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                ~(uintptr_t)1023);
    const int stages = args.stages;
    uint8_t *tiles = smem;
    uint8_t *epi = tiles + (size_t)stages * kStageBytes;
    const EpiLayout EL = epi_layout(args.VB, args.NB, args.NQ, BN, EW, args.det);
    uint64_t *bars = reinterpret_cast<uint64_t *>(epi + EL.total);
    // bars: full[stages], empty[stages], tfull[2], tempty[2], drain, wqfull[kWQ],
    // wqempty[kWQ], conv[2], pfull, pempty, tmm[2], gfull[2], gempty[2]; then the work ring
    // wq[kWQ] and the TMEM address slot
    const uint32_t wqfull0 = saddr(bars + 2 * stages + 5);
    const uint32_t wqempty0 = saddr(bars + 2 * stages + 5 + kWQ);
    // conv[a]: the epilogue has stored the G of the chunk in accumulator a as BF16 hi / lo (one
    // arrival per warp).  One barrier per accumulator: the MMA thread hands out the next item's
    // accumulator before it waits for this item's conversion, so the epilogue may convert two
    // items before the first wait; on one barrier the second phase would complete unseen and
    // the wait for the first (by parity) never end.  A second arrival on conv[a] needs the
    // accumulator again, which the MMA thread hands out only after tmm[a], issued after its
    // wait on conv[a];
    // pfull: the phase product to be read out is complete; pempty: the read-out warps have
    // read it; tmm[a]: the phase product of the chunk in accumulator a is complete, so the
    // buffer is free (for phase work the MMA thread releases the accumulator, not the
    // epilogue); gfull / gempty: a tile's geometry buffer is filled / has been used
    const uint32_t conv0 = saddr(bars + 2 * stages + 5 + 2 * kWQ);
    const uint32_t pfull = conv0 + 16, pempty = conv0 + 24, tmm0 = conv0 + 32;
    const uint32_t gfull0 = conv0 + 48, gempty0 = conv0 + 64;
    volatile WorkSlot *wq = reinterpret_cast<volatile WorkSlot *>(
        (reinterpret_cast<uintptr_t>(bars + 2 * stages + 15 + 2 * kWQ) + 15) & ~(uintptr_t)15);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(const_cast<WorkSlot *>(wq + kWQ));
    const uint32_t full0 = saddr(bars), empty0 = saddr(bars + stages);
    const uint32_t tfull0 = saddr(bars + 2 * stages), tempty0 = saddr(bars + 2 * stages + 2);
    const uint32_t drain = saddr(bars + 2 * stages + 4);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // CTA pair: rank in the pair; the first CTA (rank 0) issues the MMAs.  lead(a) is the
    // cluster address of barrier a in the first CTA, peer(a) in the other one.
    const uint32_t rank = CG == 2 ? cluster_rank() : 0u;
    const bool leader = rank == 0;
    auto lead = [&](uint32_t a) { return CG == 2 ? mapa(a, 0) : a; };
    auto peer = [&](uint32_t a) { return CG == 2 ? mapa(a, 1) : a; };
    if (threadIdx.x == 0) {
        for (int s = 0; s < stages; ++s) {
            mbar_init(full0 + 8 * s, 1);
            // a stage is free again once the MMAs that read it have completed
            mbar_init(empty0 + 8 * s, 1);
        }
        // (a pair's epilogue barriers count the warps of both CTAs)
        for (int a = 0; a < 2; ++a) {
            mbar_init(tfull0 + 8 * a, 1);
            mbar_init(tempty0 + 8 * a, kEpiWarps * CG);
        }
        mbar_init(drain, 1);
        for (int k = 0; k < kWQ; ++k) {
            mbar_init(wqfull0 + 8 * k, 1);
            // released by the MMA thread (the first CTA of a pair only), one lane of every
            // epilogue and read-out warp and the geometry warp
            mbar_init(wqempty0 + 8 * k, (leader ? 1 : 0) + kEpiWarps + 1 + kRoWarps);
        }
        mbar_init(pfull, 1);
        mbar_init(pempty, 4 * CG);
        for (int a = 0; a < 2; ++a) {
            mbar_init(conv0 + 8 * a, kEpiWarps * CG);
            mbar_init(tmm0 + 8 * a, 1);
            mbar_init(gfull0 + 8 * a, 1);
            mbar_init(gempty0 + 8 * a, kEpiWarps);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // descriptors of the first problem (a batch's other problems fetch theirs when they come)
    if (warp == 0) {
        const CUtensorMap *maps = &args.probs->mapA[0][0];
        constexpr int kMaps = 2 * kMaxCopies + 4;   // mapA, mapB, mapW
        const int n_copies = args.one.n_copies;
        if (lane < kMaps && (lane >= 2 * kMaxCopies || lane % kMaxCopies < n_copies) &&
            (lane < 2 * kMaxCopies + 2 || args.one.npass > 0) &&
            !(kPlanes == 1 && ((lane >= kMaxCopies && lane < 2 * kMaxCopies) ||
                               lane == 2 * kMaxCopies + 1)))
            asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(maps + lane))
                         : "memory");
    }
    if (warp == 1) tmem_alloc<CG>(saddr(tmem_slot), kTmemAlloc);
    tc_before();
    __syncthreads();
    // a pair's barriers are initialised in both CTAs before either signals the other
    if constexpr (CG == 2) cluster_sync();
    tc_after();
    const uint32_t tmem = *tmem_slot;
    const TcProblem *__restrict__ probs = args.probs;
    // work units: CTAs, or pairs
    const int64_t cid = blockIdx.x / CG, n_ctas = gridDim.x / CG;
    const int row_step = kBM * CG, row_off = kBM * (int)rank;

    if (warp == 0) {
        // ======================= TMA producer =======================
        if (lane == 0) {
            int stage = 0;
            uint32_t phase = 0;
            bool ok = true;
            WorkCursor cu;
            // the previous work item, while its phase sub-passes are still to be loaded: they
            // follow this item's K blocks
            int pend_p = -1, pend_n0 = 0, pend_G = 0;
            int64_t n_claimed = 0;  // work items claimed (static schedule)
            auto next_stage = [&]() {
                if (++stage == stages) {
                    stage = 0;
                    phase ^= 1;
                }
            };
            // W stage j of pass pp (sub-pass g = pp kWStages + j)
            // (a pair: each CTA loads its half of the outputs; the first CTA's full barrier
            // counts the bytes of both)
            auto load_sub = [&](int g) {
                const TcProblem &Q = probs[pend_p];
                const int pp = g / kWStages, j = g % kWStages;
                if (!mbar_wait(empty0 + 8 * stage, phase ^ 1, args.err, DEV_TIMEOUT_TMA))
                    return false;
                const uint32_t fb = full0 + 8 * stage;
                if (leader) mbar_expect_tx(fb, CG * kWPlanes * kWB);
                uint8_t *st = tiles + (size_t)stage * kStageBytes;
#pragma unroll
                for (int pl = 0; pl < kWPlanes; ++pl) {
                    const int y = pp * kPCols + (int)rank * (kPCols / CG);
                    if constexpr (CG == 2)
                        tma_load_2d_pair(saddr(st + pl * kWB), &Q.mapW[pl], lead(fb),
                                         pend_n0 + 64 * j, y);
                    else
                        tma_load_2d(saddr(st + pl * kWB), &Q.mapW[pl], fb, pend_n0 + 64 * j, y);
                }
                next_stage();
                return true;
            };
            // Sub-items (a work item's K chunks) in this CTA's work ring.  A lone CTA claims
            // work items from the counter (dynamic schedule) or in a fixed order; both CTAs
            // of a pair walk the same fixed order (measured against handing each item from
            // the first CTA to the second: 542 against 506 TFLOP/s on the 26^3 lattice).
            // The fixed order: in round k of n CTAs (pairs), CTA c takes item
            // k n + (c + k) mod n.  Without the rotation a raster group of a multiple of n
            // items would put every CTA on the same columns in every group, so the costly
            // column tiles would always land on the same CTAs.
            auto claim = [&]() -> int64_t {
                if (args.counter && CG == 1)
                    return n_ctas + (int64_t)atomicAdd(args.counter, 1ull);
                const int64_t r = n_claimed * n_ctas + (cid + n_claimed) % n_ctas;
                ++n_claimed;
                return r;
            };
            // (the first items are the CTAs' numbers: no claim to wait for)
            int64_t tau_next = args.counter && CG == 1 ? cid : claim();
            // the next item, once decoded (p = -1: none left), and the current one
            int p_next = -2, p_cur = -1, kci = 0, kch = 0;
            TileInfo t_next = {}, ti = {};
            auto take = [&]() {
                const int64_t tau = tau_next;
                if (tau >= args.total_tiles) {
                    p_next = -1;
                    return;
                }
                tau_next = claim();   // its reply is not waited for until the next call
                t_next = decode(cu, probs, args.n_probs, args.one, args.ov, tau, BN, row_step,
                                row_off);
                p_next = cu.p;
            };
            take();
            WorkCursor wc;   // the current item's problem (cu may be one item ahead)
            for (int64_t v = 0; ok; ++v) {
                const int qs = (int)(v % kWQ);
                // the next chunk of the current item, or the first of a new one
                if (++kci >= kch) {
                    if (p_next == -2) take();
                    if (p_next >= 0 && p_next != p_cur) wc = cu;
                    p_cur = p_next;
                    ti = t_next;
                    p_next = -2;
                    kci = 0;
                    kch = p_cur < 0 ? 1 : wc.kch;
                }
                const int kg0 = p_cur < 0 ? 0 : (int)div_small((int64_t)kci * wc.nk, kch);
                const int kg1 = p_cur < 0 ? 0 : (int)div_small((int64_t)(kci + 1) * wc.nk, kch);
                // publish the sub-item once its ring slot is free
                if (!mbar_wait(wqempty0 + 8 * qs, (uint32_t)((v / kWQ) & 1) ^ 1u, args.err,
                               DEV_TIMEOUT_TMA)) {
                    ok = false;
                    break;
                }
                volatile WorkSlot &w = wq[qs];
                w.p = p_cur;
                w.t = ti.t;
                w.m0 = ti.m0;
                w.n0 = ti.n0;
                w.row_end = wc.row_end;
                w.kci = kci;
                w.last = kci == kch - 1;
                w.nk = kg1 - kg0;
                mbar_arrive(wqfull0 + 8 * qs);  // release: the slot is visible to the waiters
                if (p_cur < 0) break;
                const TcProblem &P = probs[p_cur];
                const int nk = kg1 - kg0;
                // decode the next item in the middle of this one's last chunk
                const int kg_take = kci == kch - 1 ? kg0 + nk / 2 : -1;
                // sample and K block inside it, and the operand window of that sample
                int s = kg0 / wc.nkb, kb = kg0 - s * wc.nkb;
                int xw = s * wc.F3 + 3 * ti.t, c = xw % wc.n_copies;
                for (int kg = kg0; kg < kg1 && ok; ++kg) {
                    if (!mbar_wait(empty0 + 8 * stage, phase ^ 1, args.err, DEV_TIMEOUT_TMA)) {
                        ok = false;
                        break;
                    }
                    const uint32_t fb = full0 + 8 * stage;
                    if (leader) mbar_expect_tx(fb, CG * kStageBytes);
                    uint8_t *st = tiles + (size_t)stage * kStageBytes;
                    // this CTA's B columns (a pair splits the tile's columns)
                    const int nb0 = ti.n0 + (int)rank * (BN / CG);
#pragma unroll
                    for (int pl = 0; pl < kPlanes; ++pl) {
                        if constexpr (CG == 2) {
                            tma_load_2d_pair(saddr(st + pl * kABytes), &P.mapA[pl][c],
                                             lead(fb), xw - c + kb * kBK, ti.m0);
                            tma_load_2d_pair(saddr(st + kPlanes * kABytes + pl * kBBytes),
                                             &P.mapB[pl], lead(fb), s * wc.Kseg + kb * kBK,
                                             nb0);
                        } else {
                            tma_load_2d(saddr(st + pl * kABytes), &P.mapA[pl][c], fb,
                                        xw - c + kb * kBK, ti.m0);
                            tma_load_2d(saddr(st + kPlanes * kABytes + pl * kBBytes),
                                        &P.mapB[pl], fb, s * wc.Kseg + kb * kBK, nb0);
                        }
                    }
                    next_stage();
                    if (++kb == wc.nkb) {
                        kb = 0;
                        ++s;
                        xw += wc.F3;
                        c = xw % wc.n_copies;
                    }
                    if (kg == kg_take) take();
                }
                // the previous item's phase sub-passes, in the order the MMA thread issues them
                if constexpr (kPhaseOK)
                    if (pend_p >= 0)
                        for (int g = 0; g < pend_G && ok; ++g) ok = load_sub(g);
                pend_p = -1;
                if (kPhaseOK && wc.npass > 0) {
                    pend_p = p_cur;
                    pend_n0 = ti.n0;
                    pend_G = wc.npass * kWStages;
                }
            }
            // the last item's phase sub-passes
            if (kPhaseOK && ok && pend_p >= 0)
                for (int g = 0; g < pend_G && ok; ++g) ok = load_sub(g);
            // drain: wait until the last fill of every stage has landed
            for (int k = 0; k < stages; ++k) {
                if (--stage < 0) {
                    stage = stages - 1;
                    phase ^= 1;
                }
                // the most recent fill of `stage` used parity `phase`; if that stage was never
                // filled, its barrier is still in phase 0 and parity 1 reads as complete (a
                // pair's fills all complete on the first CTA's barriers: it waits for both)
                if (leader) mbar_wait(full0 + 8 * stage, phase, args.err, DEV_TIMEOUT_TMA);
            }
        }
    } else if (warp == 1) {
        // ======================= MMA issuer =======================
        // (a pair's MMAs are issued by the first CTA; its commits release the stages and
        // hand the accumulators to the epilogues of both CTAs)
        auto commit_both = [&](uint32_t a) {
            if constexpr (CG == 2) {
                tc_commit<2>(a);
                tc_commit<2>(peer(a));
            } else {
                tc_commit(a);
            }
        };
        if (lane == 0 && leader) {
            int stage = 0;
            uint32_t phase = 0;
            uint32_t v = 0;
            bool ok = true;
            int p_cur = -1, npass = 0;
            // previous sub-item with phase sub-passes still to issue: its accumulator
            // buffer and sub-pass count; whether its product adds to P (a later K chunk of
            // a tile with one pass: P sums the chunks and is read out once) and whether it
            // completes P for the read-out
            int pend_acc = -1, pend_G = 0;
            bool pend_add = false, pend_done = false;
            // parity of the next conversion to wait for, one bit per accumulator; passes that
            // started P afresh (one read-out each)
            uint32_t conv_par = 0, n_own = 0;
            // how each accumulator was last released (0: not used yet, 1: by the epilogue
            // on tempty, 2: by this thread's commit on tmm after the chunk's phase product)
            // and the waits taken on each barrier
            int rel[2] = {0, 0};
            uint32_t n_te[2] = {0, 0}, n_tm[2] = {0, 0};
            const uint32_t ptm = tmem + 2 * BN;  // phase product P
            // sub-pass g of the previous item's phase product: pass pp = g / kWStages adds
            // G[:, c] W[c, :] for the 64 columns c of W stage j = g % kWStages to P, A = the
            // BF16 hi / lo copy of G in its accumulator columns
            auto issue_sub = [&](int g) {
                const int pp = g / kWStages, j = g % kWStages;
                const uint32_t g0 = tmem + (uint32_t)pend_acc * BN;
                if (!mbar_wait(full0 + 8 * stage, phase, args.err, DEV_TIMEOUT_MMA))
                    return false;
                if (j == 0) {
                    // G stored as BF16 by the epilogue (once per chunk); a pass that starts
                    // P afresh waits until the previous P has been read out
                    if (pp == 0) {
                        if (!mbar_wait(conv0 + 8 * pend_acc, (conv_par >> pend_acc) & 1,
                                       args.err, DEV_TIMEOUT_MMA))
                            return false;
                        conv_par ^= 1u << pend_acc;
                    }
                    if (!pend_add) {
                        if (!mbar_wait(pempty, (n_own & 1) ^ 1, args.err, DEV_TIMEOUT_MMA))
                            return false;
                        ++n_own;
                    }
                }
                tc_after();
                uint8_t *st = tiles + (size_t)stage * kStageBytes;
                const uint64_t w0 = sdesc(saddr(st), 128);
                const uint64_t w1 = sdesc(saddr(st + kWB), 128);
#pragma unroll
                for (int ks = 0; ks < 4; ++ks) {
                    // columns c = 64 j + 16 ks: chunk c / 32 holds hi in its first 16 TMEM
                    // columns and lo in the next 16
                    const int c = 64 * j + 16 * ks;
                    const uint32_t ahi = g0 + 32 * (c >> 5) + 8 * ((c >> 4) & 1);
                    const uint64_t off = (uint64_t)(ks * 32) >> 4;
                    const uint32_t accum = pend_add || (j | ks) != 0;
                    tc_mma_ts<CG>(ptm, ahi, w0 + off, kIdescP, accum);           // hi*hi
                    if (kWPlanes == 2) {
                        tc_mma_ts<CG>(ptm, ahi, w1 + off, kIdescP, 1u);          // hi*lo
                        tc_mma_ts<CG>(ptm, ahi + 16, w0 + off, kIdescP, 1u);     // lo*hi
                    }
                }
                commit_both(empty0 + 8 * stage);
                if (++stage == stages) {
                    stage = 0;
                    phase ^= 1;
                }
                if (j == kWStages - 1 && pend_done) commit_both(pfull);
                // the chunk's accumulator is free once its phase product has completed
                if (g == pend_G - 1) tc_commit<CG>(tmm0 + 8 * pend_acc);
                return true;
            };
            for (;; ++v) {
                const int qs = (int)(v % kWQ);
                if (!mbar_wait(wqfull0 + 8 * qs, (v / kWQ) & 1, args.err, DEV_TIMEOUT_MMA)) {
                    ok = false;
                    break;
                }
                const int p = wq[qs].p, kci = wq[qs].kci, last = wq[qs].last, nk = wq[qs].nk;
                mbar_arrive(wqempty0 + 8 * qs);
                if (p < 0) break;
                if (p != p_cur) {
                    p_cur = p;
                    npass = args.n_probs == 1 ? args.one.npass : probs[p].dims.npass;
                }
                const bool phs = kPhaseOK && npass > 0;
                const uint32_t acc = v & 1;
                // wait until the accumulator's previous chunk has released it
                if (rel[acc] == 1 && !mbar_wait(tempty0 + 8 * acc, n_te[acc]++ & 1, args.err,
                                                DEV_TIMEOUT_MMA)) {
                    ok = false;
                    break;
                }
                if (rel[acc] == 2 && !mbar_wait(tmm0 + 8 * acc, n_tm[acc]++ & 1, args.err,
                                                DEV_TIMEOUT_MMA)) {
                    ok = false;
                    break;
                }
                rel[acc] = phs ? 2 : 1;
                tc_after();
                const uint32_t d = tmem + acc * BN;
                for (int kb = 0; kb < nk; ++kb) {  // 0: the first block of this chunk
                    if (!mbar_wait(full0 + 8 * stage, phase, args.err, DEV_TIMEOUT_MMA)) {
                        ok = false;
                        break;
                    }
                    tc_after();
                    uint8_t *st = tiles + (size_t)stage * kStageBytes;
                    const uint64_t a0 = sdesc(saddr(st), SWB);
                    const uint64_t b0 = sdesc(saddr(st + kPlanes * kABytes), SWB);
#pragma unroll
                    for (int ks = 0; ks < kKSteps; ++ks) {
                        const uint64_t off = (uint64_t)(ks * 32) >> 4;
                        const uint32_t first = (kb | ks) != 0;
                        if (kPlanes == 1) {
                            tc_mma<kTF32, CG>(d, a0 + off, b0 + off, kIdesc, first);
                        } else {
                            const uint64_t a1 = sdesc(saddr(st + kABytes), SWB);
                            const uint64_t b1 = sdesc(saddr(st + 2 * kABytes + kBBytes), SWB);
                            tc_mma<false, CG>(d, a0 + off, b0 + off, kIdesc, first);  // hi*hi
                            tc_mma<false, CG>(d, a0 + off, b1 + off, kIdesc, 1u);     // hi*lo
                            tc_mma<false, CG>(d, a1 + off, b0 + off, kIdesc, 1u);     // lo*hi
                        }
                    }
                    commit_both(empty0 + 8 * stage);
                    if (++stage == stages) {
                        stage = 0;
                        phase ^= 1;
                    }
                }
                if (!ok) break;
                commit_both(tfull0 + 8 * acc);
                // The previous item's phase product, after this item's accumulator is handed
                // over: its wait for the epilogue's BF16 copy then holds nobody up, where two
                // thirds into the K blocks it stalled the rest of them (and so the epilogue's
                // next tile) whenever the binning was the slower side.  48^3 glass BF16 at
                // 2/3, 5/6 and the end: 103.0, 96.9, 94.0 ms; 32^3 glass split-BF16 the same.
                if constexpr (kPhaseOK)
                    if (pend_acc >= 0)
                        for (int g = 0; g < pend_G && ok; ++g) ok = issue_sub(g);
                if (!ok) break;
                pend_acc = -1;
                if (phs) {
                    // one pass: P sums the tile's chunks and is read out after the last
                    const bool across = npass == 1;
                    pend_acc = (int)acc;
                    pend_G = npass * kWStages;
                    pend_add = across && kci > 0;
                    pend_done = !across || last;
                }
            }
            // the last item's phase sub-passes
            if (kPhaseOK && ok && pend_acc >= 0)
                for (int g = 0; g < pend_G && ok; ++g) ok = issue_sub(g);
            // drain every MMA this thread issued before TMEM is released
            tc_commit<CG>(drain);
            mbar_wait(drain, 0, args.err, DEV_TIMEOUT_MMA);
        }
    } else if (warp == 2 + kEpiWarps) {
        // ======================= geometry =======================
        // (on the epilogue warps, behind two barriers and several dependent global loads,
        // this took 5 to 10 thousand cycles of each tile; the epilogue now waits for it less
        // than 1 thousand)
        uint32_t item = 0;  // tiles prepared
        for (uint32_t v = 0;; ++v) {
            const int qs = (int)(v % kWQ);
            bool ok = mbar_wait(wqfull0 + 8 * qs, (v / kWQ) & 1, args.err, DEV_TIMEOUT_EPI);
            if (!__all_sync(0xffffffffu, ok)) break;
            const int p = wq[qs].p, m0 = wq[qs].m0, n0 = wq[qs].n0, row_end = wq[qs].row_end;
            const bool first = wq[qs].kci == 0;
            __syncwarp();
            if (lane == 0) mbar_arrive(wqempty0 + 8 * qs);
            if (p < 0) break;
            if (!first || probs[p].epi.n_bins == 0) continue;   // (phase sums need no geometry)
            const uint32_t gb = item & 1;
            ok = mbar_wait(gempty0 + 8 * gb, ((item >> 1) & 1) ^ 1u, args.err, DEV_TIMEOUT_EPI);
            if (!__all_sync(0xffffffffu, ok)) break;
            ++item;
            const EpiParams &E = probs[p].epi;
            const int N = probs[p].dims.N;
            float *cg = reinterpret_cast<float *>(epi + EL.geo) + gb * 3 * BN;
            const bool lattice = E.geom == ASD_GEOM_LATTICE;
            // columns (past the last site: its geometry, with zero products), one per lane
            // and 32-column chunk
            float cx[kChunks][3];
#pragma unroll
            for (int m = 0; m < kChunks; ++m) {
                const int c = 32 * m + lane, j = min(n0 + c, N - 1);
                if (lattice) {
                    const int4 g = E.coords[j];
                    if (E.fast && (E.NW + 1) * kBinStride <= 65536) {
                        reinterpret_cast<uint32_t *>(cg)[c] =
                            (uint32_t)g.x | ((uint32_t)g.y << 8) | ((uint32_t)g.z << 16);
                    } else {
                        cg[c] = __int_as_float(g.x);
                        cg[BN + c] = __int_as_float(g.y);
                        cg[2 * BN + c] = __int_as_float(g.z);
                    }
                    cx[m][0] = (float)g.x;
                    cx[m][1] = (float)g.y;
                    cx[m][2] = (float)g.z;
                } else {
                    const float4 g = E.pos[j];
                    cg[c] = cx[m][0] = g.x;
                    cg[BN + c] = cx[m][1] = g.y;
                    cg[2 * BN + c] = cx[m][2] = g.z;
                }
            }
            TileWindow tw = {0, 0, E.NW, E.n_bins, kChunks, E.n_bins - 1,
                             !E.use_window && E.pos_ok, 0};
            if (E.use_window) {
                // boxes of the rows inside the range and of each column chunk
                float rl[3] = {3e38f, 3e38f, 3e38f}, rh[3] = {-3e38f, -3e38f, -3e38f};
                for (int m = 0; m < kBM / 32; ++m) {
                    const int i = m0 + 32 * m + lane;
                    if (i < row_end) {
                        float r[3];
                        if (lattice) {
                            const int4 g = E.coords[i];
                            r[0] = (float)g.x;
                            r[1] = (float)g.y;
                            r[2] = (float)g.z;
                        } else {
                            const float4 g = E.pos[i];
                            r[0] = g.x;
                            r[1] = g.y;
                            r[2] = g.z;
                        }
#pragma unroll
                        for (int a = 0; a < 3; ++a) {
                            rl[a] = fminf(rl[a], r[a]);
                            rh[a] = fmaxf(rh[a], r[a]);
                        }
                    }
                }
                // (lane m keeps the box of chunk m)
                float bl[3], bh[3], cl[3], ch[3];
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    rl[a] = warp_min(rl[a]);
                    rh[a] = warp_max(rh[a]);
                    bl[a] = cl[a] = 3e38f;
                    bh[a] = ch[a] = -3e38f;
#pragma unroll
                    for (int m = 0; m < kChunks; ++m) {
                        const float lo = warp_min(cx[m][a]), hi = warp_max(cx[m][a]);
                        if (lane == m) {
                            bl[a] = lo;
                            bh[a] = hi;
                        }
                        cl[a] = fminf(cl[a], lo);
                        ch[a] = fmaxf(ch[a], hi);
                    }
                }
                auto box_d2 = [&](const float (&lo)[3], const float (&hi)[3], float &dmin,
                                  float &dmax) {
                    dmin = dmax = 0.f;
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        float gap = fmaxf(0.f, fmaxf(lo[a] - rh[a], rl[a] - hi[a]));
                        if (lattice && E.periodic) {
                            const float L = a == 0 ? E.Lx : a == 1 ? E.Ly : E.Lz;
                            gap = fminf(gap, fmaxf(0.f, fmaxf(lo[a] + L - rh[a], rl[a] - (hi[a] + L))));
                            gap = fminf(gap, fmaxf(0.f, fmaxf(lo[a] - L - rh[a], rl[a] - (hi[a] - L))));
                        }
                        const float far = fmaxf(hi[a] - rl[a], rh[a] - lo[a]);
                        dmin += gap * gap;
                        dmax += far * far;
                    }
                };
                auto lo_bin = [&](float d2) {
                    return max(0, bin_of_d2(d2 * 0.999f, E.inv_w, E.n_bins, E.thr) - 1);
                };
                auto hi_bin = [&](float d2) {
                    return min(E.n_bins - 1,
                               bin_of_d2(d2 * 1.001f + 1e-30f, E.inv_w, E.n_bins, E.thr) + 1);
                };
                float dmin, dmax;
                box_d2(cl, ch, dmin, dmax);
                tw.blo = lo_bin(dmin);
                if (!lattice) {
                    tw.bhi = hi_bin(dmax);
                    tw.nwp = tw.bhi - tw.blo + 1;
                    tw.fit = E.pos_ok && tw.nwp <= E.NW;
                    if (!tw.fit && E.pos_ok) {
                        // bins of each 32-column chunk (lane c computes chunk c), then the
                        // first split of the chunks into two windows that together fit
                        box_d2(bl, bh, dmin, dmax);
                        const int lo_c = lane < kChunks ? lo_bin(dmin) : 0;
                        const int hi_c = lane < kChunks ? hi_bin(dmax) : 0;
                        int lo[kChunks], hi[kChunks];
#pragma unroll
                        for (int c = 0; c < kChunks; ++c) {
                            lo[c] = __shfl_sync(0xffffffffu, lo_c, c);
                            hi[c] = __shfl_sync(0xffffffffu, hi_c, c);
                        }
                        // one window over the chunks' bins (narrower than the tile's
                        // box); only when that does not fit, two windows, which are then
                        // disjoint (two overlapping ones would span no more than their
                        // sum), so no bin has two private rows
                        int l0 = 1 << 30, h0 = -1;
#pragma unroll
                        for (int c = 0; c < kChunks; ++c) {
                            l0 = min(l0, lo[c]);
                            h0 = max(h0, hi[c]);
                        }
                        int best = E.NW + 1, b1 = 0, b2 = 0, bn = 0, bs = kChunks;
                        if (h0 - l0 + 1 <= E.NW) {
                            best = h0 - l0 + 1;
                            b1 = l0;
                            bn = E.NW;
                        }
#pragma unroll
                        for (int sp = 1; sp < kChunks && best > E.NW; ++sp) {
                            int l1 = 1 << 30, h1 = -1, l2 = 1 << 30, h2 = -1;
#pragma unroll
                            for (int c = 0; c < kChunks; ++c) {
                                if (c < sp) { l1 = min(l1, lo[c]); h1 = max(h1, hi[c]); }
                                else { l2 = min(l2, lo[c]); h2 = max(h2, hi[c]); }
                            }
                            const int need = (h1 - l1 + 1) + (h2 - l2 + 1);
                            if (need < best) {
                                best = need;
                                b1 = l1;
                                bn = h1 - l1 + 1;
                                b2 = l2;
                                bs = sp;
                            }
                        }
                        if (best <= E.NW) {
                            tw.fit = 1;
                            tw.nwp = best;
                            tw.blo = b1;
                            tw.blo2 = b2;
                            tw.n1 = bn;
                            tw.split = bs;
                        }
                    }
                }
            }
            if (lane == 0) reinterpret_cast<TileWindow *>(epi + EL.win)[gb] = tw;
            __syncwarp();   // (every lane's stores before the arrive's release)
            if (lane == 0) mbar_arrive(gfull0 + 8 * gb);
        }
    } else if (kPhaseOK && warp > 2 + kEpiWarps) {
        // ======================= phase read-out =======================
        // Phase product of each pass: P[r][o] = sum_c G_rc W_co, u = P[.][0:64) (cosine column
        // weights), v = P[.][64:128) (sine).  Row r adds cos(q.r_i) u + sin(q.r_i) v (cosine
        // part) and sin(q.r_i) u - cos(q.r_i) v (sine part), the angle-difference identities
        // of Eq. 6's weight; a warp sums its 32 rows by recursive halving and adds them to
        // its FP64 sums.  Warps of their own: the 64 row weights of a row come from L2 behind
        // the operand streams, and the read-out on the epilogue warps, between the binning
        // of two tiles, took 8 to 12 thousand cycles of each tile (48^3 glass BF16, the
        // epilogue's other parts as now: 122 -> 100 ms, 32^3 glass split-BF16 21.3 -> 19.3); here the weights of the next read-out load
        // while its product is still to come, and the binning does not wait.  One pass:
        // P sums the tile's K chunks and is read out after the last; several passes: each is
        // read out per chunk.
        const int q4 = warp & 3;   // TMEM lane quarter of this warp
        double *qa = reinterpret_cast<double *>(epi + EL.qacc) + q4 * args.NQ;
        long long *qai = reinterpret_cast<long long *>(qa);   // deterministic mode
        for (int k = lane; k < args.NQ; k += 32) qa[k] = 0.0;
        __syncwarp();
        const uint32_t pt = tmem + ((uint32_t)(q4 * 32) << 16) + 2 * BN;
        int cur_p = -1, cur_t = -1, N = 0, n_q = 0, npass = 0, parts = 1, n_t = 0;
        int64_t ld = 0;
        const float2 *csT = nullptr;
        double fscale = 0.0, *Qs = nullptr;
        long long *Qf = nullptr;
        bool det = false;
        uint32_t n_pass = 0;   // passes read out (parity of pfull)
        // the sums of the current (problem, t), added to the outputs when it changes
        auto flush_q = [&]() {
            if (cur_p < 0 || n_q == 0) return;
            const bool t_ok = ASD_INB((unsigned)cur_t < (unsigned)n_t, BND_WORK, args.err);
            for (int k = lane; k < n_q * parts; k += 32) {
                const int64_t o = (int64_t)cur_t * n_q * parts + k;
                if (det) {
                    if (qai[k] != 0 && t_ok) add_fixed(&Qf[o], qai[k]);
                } else if (qa[k] != 0.0 && t_ok) {
                    atomicAdd(&Qs[o], qa[k]);
                }
                qa[k] = 0.0;
            }
            __syncwarp();
        };
        bool ok = true;
        for (uint32_t v = 0; ok; ++v) {
            const int qs = (int)(v % kWQ);
            ok = __all_sync(0xffffffffu, mbar_wait(wqfull0 + 8 * qs, (v / kWQ) & 1, args.err,
                                                   DEV_TIMEOUT_EPI));
            if (!ok) break;
            const int p = wq[qs].p, t = wq[qs].t, i = wq[qs].m0 + q4 * 32 + lane;
            const bool row_ok = i < wq[qs].row_end, last = wq[qs].last != 0;
            __syncwarp();
            if (lane == 0) mbar_arrive(wqempty0 + 8 * qs);
            if (p < 0) break;
            if (p != cur_p || t != cur_t) flush_q();
            if (p != cur_p) {
                const EpiParams &E = probs[p].epi;
                N = probs[p].dims.N;
                n_t = probs[p].dims.n_t;
                n_q = E.n_q;
                npass = E.npass;
                parts = E.q_parts;
                csT = E.csT;
                ld = E.cs_ld;
                det = E.fix_scale != nullptr;
                fscale = det ? *E.fix_scale : 0.0;
                Qs = args.ov.active ? args.ov.Sq_sum : E.Sq_sum;
                Qf = E.Sq_fix;
            }
            cur_p = p;
            cur_t = t;
            if (n_q == 0 || (npass == 1 && !last)) continue;
            // (rows past the range hold zeros in P)
            const float2 *cs = csT + (row_ok ? i : N - 1);
            for (int q0 = 0; ok && q0 < npass * kPhaseQ; q0 += 32) {
                // 32 q-vectors (half a pass) at a time; the table has a row per q, so a
                // warp's 32 consecutive sites read two or three lines per q.  Rows past n_q
                // up to the padding are zero.
                float2 cw[32];
#pragma unroll
                for (int k = 0; k < 32; ++k)
                    if (q0 + (k & 24) < n_q) cw[k] = cs[(int64_t)(q0 + k) * ld];
                    else cw[k] = make_float2(0.f, 0.f);
                const int h = q0 & 32;   // second half of the pass
                if (h == 0) {
                    ok = __all_sync(0xffffffffu,
                                    mbar_wait(pfull, n_pass & 1, args.err, DEV_TIMEOUT_EPI));
                    if (!ok) break;
                    ++n_pass;
                    tc_after();
                }
                float xs = 0.f, ys = 0.f;   // this lane's q of the 32
#pragma unroll
                for (int j = 0; j < 32; j += 8) {
                    if (q0 + j >= n_q) break;   // (few q-vectors: 8 at a time, not 64)
                    uint32_t u[8], w[8];
                    tmem_ld8(pt + h + j, u);
                    tmem_ld8(pt + kPhaseQ + h + j, w);
                    tmem_wait8x2(u, w);
                    float x[8];
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        x[k] = fmaf(cw[j + k].x, __uint_as_float(u[k]),
                                    cw[j + k].y * __uint_as_float(w[k]));
                    const float xj = warp_sum8(x, lane);
                    // (every fourth lane group holds one of the eight; lane & 3 picks j, so
                    // one FP64 conversion and add serves all 32)
                    if ((lane & 3) == (j >> 3)) xs = xj;
                    if (parts == 2) {
#pragma unroll
                        for (int k = 0; k < 8; ++k)
                            x[k] = fmaf(cw[j + k].y, __uint_as_float(u[k]),
                                        -cw[j + k].x * __uint_as_float(w[k]));
                        const float yj = warp_sum8(x, lane);
                        if ((lane & 3) == (j >> 3)) ys = yj;
                    }
                }
                const int qme = q0 + (lane & 3) * 8 + ((lane >> 4) & 1) * 4 +
                                ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1);
                if (qme < n_q && ASD_INB((qme + 1) * parts <= args.NQ, BND_Q, args.err)) {
                    if (det) qai[qme * parts] += to_fixed((double)xs, fscale);
                    else qa[qme * parts] += (double)xs;
                    if (parts == 2) {
                        if (det) qai[qme * 2 + 1] += to_fixed((double)ys, fscale);
                        else qa[qme * 2 + 1] += (double)ys;
                    }
                }
                // P read: the next pass (or item) may overwrite it
                if (h == 32) {
                    tc_before();
                    __syncwarp();
                    if (lane == 0) {
                        if constexpr (CG == 2) mbar_arrive_cl(lead(pempty));
                        else mbar_arrive(pempty);
                    }
                }
            }
        }
        __syncwarp();
        if (ok) flush_q();
    } else {
        // ======================= epilogue =======================
        const int et = threadIdx.x - 64;          // 0 .. kEpiThreads - 1
        const int q4 = warp & 3;                  // TMEM lane quarter of this warp
        const int r = q4 * 32 + lane;             // accumulator row = tile row
        const int ew = warp - 2;                  // epilogue warp 0..7
        const int half = ew >> 2;                 // which part of the columns (EW = 8)
        const int ch0 = half * (BN / 32 / kHalves), ch1 = ch0 + BN / 32 / kHalves;
        // private bins and bin table of the current problem (set when the problem changes)
        float *bins = reinterpret_cast<float *>(epi + EL.var);
        float *fb = reinterpret_cast<float *>(epi + EL.fb);
        double *cacc = reinterpret_cast<double *>(epi + EL.cacc);
        // the same arrays as 64-bit fixed point (problems in the deterministic mode)
        long long *fbi = reinterpret_cast<long long *>(epi + EL.fb);
        long long *cacci = reinterpret_cast<long long *>(epi + EL.cacc);
        // the current problem's parameters and fixed-point scale (0: FP sums)
        const EpiParams &E = *reinterpret_cast<const EpiParams *>(epi + EL.par);
        double fscale = 0.0;
        bool det = false;
        float *thr_s = bins;
        for (int k = et; k < args.NB; k += kEpiThreads) {
            if (args.det) fbi[k] = 0;
            else fb[k] = 0.f;
            cacc[k] = 0.0;  // (all-zero bits: also fixed-point zero)
        }

        int cur_p = -1, cur_t = -1, N = 0;
        // fast lattice binning also needs the private-bin offsets of this launch (the
        // largest window of a batch, plus its trash row) to fit the 16-bit table entries
        auto fast_ok = [&]() { return E.fast && (E.NW + 1) * kBinStride <= 65536; };
        // Store a 32-column chunk of this thread's accumulator row back as BF16 hi / lo
        // (16 columns each, two values per column, the even column in the low half):
        // the A operand of the phase product.  Rows past the range store zeros.
        auto to_bf16 = [&](const uint32_t (&g)[32], uint32_t tcol, bool keep) {
            uint32_t hi[16], lo[16];
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                const float a = keep ? __uint_as_float(g[2 * k]) : 0.f;
                const float b = keep ? __uint_as_float(g[2 * k + 1]) : 0.f;
                const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
                const float2 hf = __bfloat1622float2(h);
                const __nv_bfloat162 l = __floats2bfloat162_rn(a - hf.x, b - hf.y);
                hi[k] = *reinterpret_cast<const uint32_t *>(&h);
                lo[k] = *reinterpret_cast<const uint32_t *>(&l);
            }
            tmem_st16(tcol, hi);
            tmem_st16(tcol + 16, lo);
        };
        uint32_t v = 0;
        bool ok = true;
        // the current tile: this thread's row site and its geometry, whether the row is in the
        // range, the tile's columns and bin window(s)
        int4 ri = make_int4(0, 0, 0, 0);
        float4 rp = make_float4(0.f, 0.f, 0.f, 0.f);
        int ic = 0;
        bool row_ok = false;
        uint32_t item = 0;   // tiles begun
        const float *colgeo = nullptr;
        TileWindow tw = {};
        // per-CTA FP64 sums of the current (problem, t), added to the outputs when it changes
        // (deterministic mode: fixed-point sums into the problem's fixed-point arrays)
        auto flush_acc = [&](int p, int t) {
            double *Cs = args.ov.active ? args.ov.C_sum : E.C_sum;
            const bool t_ok = ASD_INB((unsigned)t < (unsigned)probs[p].dims.n_t, BND_WORK, args.err);
            for (int b = et; b < E.n_bins; b += kEpiThreads) {
                const int64_t o = (int64_t)t * E.n_bins + b;
                if (det) {
                    if (cacci[b] != 0 && t_ok) add_fixed(&E.C_fix[o], cacci[b]);
                } else if (cacc[b] != 0.0 && t_ok) {
                    atomicAdd(&Cs[o], cacc[b]);
                }
                cacc[b] = 0.0;
            }
        };
        bool bins_on = false;
        // row geometry of the current tile (the load is in flight while the waits run)
        auto load_row = [&]() {
            // rows past the range (ragged tiles) read the geometry of a valid site and
            // contribute zeros
            if (E.geom == ASD_GEOM_LATTICE) ri = E.coords[ic];
            else rp = E.pos[ic];
        };
        for (;; ++v) {
            const int qs = (int)(v % kWQ);
            const uint32_t acc = v & 1, use = v >> 1;
            // the sub-item, its tile's geometry and its accumulator; every thread waits by
            // itself, then all agree (a wait that gave up in one stops all)
            bool got = mbar_wait(wqfull0 + 8 * qs, (v / kWQ) & 1, args.err, DEV_TIMEOUT_EPI);
            int p = -1, t = 0, kci = 0, lst = 0;
            bool new_t = false;
            if (got) {
                p = wq[qs].p;
                t = wq[qs].t;
                kci = wq[qs].kci;
                lst = wq[qs].last;
                if (kci == 0 && p >= 0) {
                    const int i = wq[qs].m0 + r;
                    row_ok = i < wq[qs].row_end;
                    if (p == cur_p) {
                        ic = row_ok ? i : N - 1;
                        load_row();
                    } else {
                        ic = i;   // (N is read at the problem switch below)
                    }
                }
            }
            __syncwarp();
            if (lane == 0 && got) mbar_arrive(wqempty0 + 8 * qs);
            const bool end = got && p < 0;
            const bool first = kci == 0, last = lst != 0;
            if (got && !end && p != cur_p) {
                // (a thread whose wait gave up meets the others at this barrier from the one
                // below: it is the same barrier, and all stop)
                ok = epi_sync_and(true, kEpiThreads);
                if (!ok) break;
                // another problem: finish the previous one, then load its parameters and
                // lay out the per-problem region (every bin was zeroed at its flush)
                if (cur_p >= 0) flush_acc(cur_p, cur_t);
                epi_sync(kEpiThreads);
                const uint32_t *src = reinterpret_cast<const uint32_t *>(&probs[p].epi);
                uint32_t *dst = reinterpret_cast<uint32_t *>(epi + EL.par);
                for (int k = et; k < (int)(sizeof(EpiParams) / 4); k += kEpiThreads)
                    dst[k] = src[k];
                epi_sync(kEpiThreads);
                cur_p = p;
                cur_t = t;
                N = probs[p].dims.N;
                det = E.fix_scale != nullptr;
                fscale = det ? *E.fix_scale : 0.0;
                if (!row_ok) ic = N - 1;
                load_row();
                bins = reinterpret_cast<float *>(epi + EL.var);
                thr_s = reinterpret_cast<float *>(epi + EL.var + var_bins_bytes(E.NW, EW));
                // (a checked build also tests that the problem's bins and table fit the
                // launch's per-problem region; if not, the problem is not binned)
                bins_on = E.n_bins > 0 &&
                          ASD_INB(var_bytes(E.NW, E.n_bins, E.n_lut, EW) <= args.VB,
                                  BND_REGION, args.err);
                if (bins_on) {
                    for (int k = et; k < (E.NW + 1) * kBinStride; k += kEpiThreads)
                        bins[k] = 0.f;
                    if (E.n_lut > 0) {
                        // fast form: entries become private-bin word offsets (the host
                        // checked that (n_bins + 1) * stride fits 16 bits); dropped
                        // pairs: the trash row E.NW, which no flush reads
                        uint16_t *lut_s = reinterpret_cast<uint16_t *>(thr_s);
                        for (int k = et; k < E.n_lut; k += kEpiThreads) {
                            const int b = E.lut[k];
                            lut_s[k] = (uint16_t)(fast_ok()
                                                      ? (b < E.n_bins ? b : E.NW) * kBinStride
                                                      : b);
                        }
                    } else {
                        float2 *thr2 = reinterpret_cast<float2 *>(thr_s);
                        for (int k = et; k <= E.n_bins; k += kEpiThreads)
                            thr2[k] = make_float2(E.thr[k], E.thr[k + 1]);
                    }
                }
                epi_sync(kEpiThreads);
            } else if (got && !end && first && t != cur_t) {
                new_t = true;
            }
            if (got && !end) {
                if (first && E.n_bins > 0)
                    got = mbar_wait(gfull0 + 8 * (item & 1), (item >> 1) & 1, args.err,
                                    DEV_TIMEOUT_EPI);
                got = got && mbar_wait(tfull0 + 8 * acc, use & 1, args.err, DEV_TIMEOUT_EPI);
            }
            // (also orders the flush of the previous tile's private bins before new adds)
            ok = epi_sync_and(got, kEpiThreads);
            if (!ok || end) break;
            tc_after();
            if (first && new_t) {
                flush_acc(cur_p, cur_t);
                cur_t = t;
            }
            if (first && E.n_bins > 0) {
                const uint32_t gb = item & 1;
                colgeo = reinterpret_cast<const float *>(epi + EL.geo) + gb * 3 * BN;
                tw = reinterpret_cast<const TileWindow *>(epi + EL.win)[gb];
                ++item;
            }
            const bool lattice = E.geom == ASD_GEOM_LATTICE;
            // phase weights of this item go through the tensor core (see kPhaseOK)
            const bool ph = kPhaseOK && E.n_q > 0;
            const uint32_t tbase = tmem + ((uint32_t)(q4 * 32) << 16) + acc * BN;

            if (bins_on) {
                BinArgs ba;
                ba.Lx = E.Lx;
                ba.Ly = E.Ly;
                ba.Lz = E.Lz;
                ba.periodic = E.periodic;
                ba.inv_w = E.inv_w;
                ba.nb = E.n_bins;
                ba.blo = E.use_window ? tw.blo : 0;
                ba.nwp = E.use_window ? E.NW : E.n_bins;
                ba.trash = E.NW;
                ba.NB = args.NB;
                ba.n_lut = E.n_lut;
                ba.fscale = fscale;
                ba.err = args.err;
                const int mode = !lattice ? BIN_POS : (E.n_lut > 0 ? BIN_LUT : BIN_THR);
                if (fast_ok()) {
                    // rows past the range skip the pairs (the TMEM loads stay warp-wide)
                    const uint32_t rpk =
                        (uint32_t)ri.x | ((uint32_t)ri.y << 8) | ((uint32_t)ri.z << 16);
                    float *mb = bins + r + kBM * half;
                    const bool lut = E.n_lut > 0;
                    const uint32_t trash_off = (uint32_t)E.NW * kBinStride;
                    for (int ch = ch0; ch < ch1; ++ch) {
                        // the TMEM load runs while the bin offsets are computed
                        uint32_t g[32], off[32];
                        tmem_ld32_issue(tbase + ch * 32, g);
                        const uint4 *cp = reinterpret_cast<const uint4 *>(colgeo) + ch * 8;
                        if (lut)
                            pk_offsets<true, kBinStride>(off, rpk, E.Lpk, cp, thr_s, E.inv_w,
                                                         E.n_bins, trash_off, E.n_lut, args.err);
                        else
                            pk_offsets<false, kBinStride>(off, rpk, E.Lpk, cp, thr_s, E.inv_w,
                                                          E.n_bins, trash_off, E.n_lut, args.err);
                        tmem_wait32(g);
                        if (row_ok) add_private(mb, off, g, trash_off, args.err);
                        if (ph) to_bf16(g, tbase + ch * 32, row_ok);
                    }
                } else if (mode == BIN_POS && tw.fit) {
                    // rows past the range skip the pairs (the TMEM loads stay warp-wide)
                    float *mb = bins + r + kBM * half;
                    const uint32_t trash_off = (uint32_t)E.NW * kBinStride;
                    FastBin fbin = {pack2(E.inv_w, E.inv_w), pack2(E.w, E.w),
                                    reinterpret_cast<const float2 *>(thr_s), E.n_bins, 0u,
                                    trash_off};
                    const uint64_t nx = pack2(-rp.x, -rp.x), ny = pack2(-rp.y, -rp.y),
                                   nz = pack2(-rp.z, -rp.z);
                    // whether some pair of the tile may lie at n_bins or beyond
                    const bool drop = !E.no_drop && (!E.use_window || tw.bhi == E.n_bins - 1);
                    for (int ch = ch0; ch < ch1; ++ch) {
                        // (private row of bin b: b - blo, or b - blo2 + n1 in a second window)
                        const int b0 = !E.use_window ? 0 : ch < tw.split ? tw.blo : tw.blo2 - tw.n1;
                        uint32_t g[32], off[32];
                        tmem_ld32_issue(tbase + ch * 32, g);
                        const float *cg = colgeo + ch * 32;
                        fbin.c0 = 0u - (kBinBaseBits + (uint32_t)b0) * (uint32_t)kBinStride;
                        if (E.thr_exact && !drop)
                            pos_offsets<true, false, kBinStride>(off, nx, ny, nz, cg, BN, fbin);
                        else if (E.thr_exact)
                            pos_offsets<true, true, kBinStride>(off, nx, ny, nz, cg, BN, fbin);
                        else if (!drop)
                            pos_offsets<false, false, kBinStride>(off, nx, ny, nz, cg, BN, fbin);
                        else
                            pos_offsets<false, true, kBinStride>(off, nx, ny, nz, cg, BN, fbin);
                        tmem_wait32(g);
                        if (row_ok) add_private(mb, off, g, trash_off, args.err);
                        if (ph) to_bf16(g, tbase + ch * 32, row_ok);
                    }
                } else
                for (int ch = ch0; ch < ch1; ++ch) {
                    uint32_t g[32];
                    tmem_ld32(tbase + ch * 32, g);
                    const float *cg = colgeo + ch * 32;
                    float *mb = bins + r + kBM * half;
                    void *fbv = det ? static_cast<void *>(fbi) : static_cast<void *>(fb);
                    if (mode == BIN_LUT)
                        bin_chunk<BIN_LUT, kBinStride>(g, row_ok, ri, rp, cg, BN, thr_s, mb, fbv,
                                                      ba);
                    else if (mode == BIN_THR)
                        bin_chunk<BIN_THR, kBinStride>(g, row_ok, ri, rp, cg, BN, thr_s, mb, fbv,
                                                      ba);
                    else if (E.pos_ok)
                        pos_chunk<kBinStride>(g, row_ok, rp, cg, BN, thr_s, mb, fbv, ba);
                    else
                        bin_chunk<BIN_POS, kBinStride>(g, row_ok, ri, rp, cg, BN, thr_s, mb, fbv,
                                                      ba);
                    if (ph) to_bf16(g, tbase + ch * 32, row_ok);
                }
            } else if (ph) {
                for (int ch = ch0; ch < ch1; ++ch) {
                    uint32_t g[32];
                    tmem_ld32(tbase + ch * 32, g);
                    to_bf16(g, tbase + ch * 32, row_ok);
                }
            }
            // without phase weights the accumulator buffer is free for the MMA warp now;
            // with them the BF16 copy of G is in place and the MMA thread may start the
            // phase product (the accumulator stays taken until that product is complete)
            if (ph) tmem_wait_st();
            tc_before();
            __syncwarp();
            // (a pair's epilogue warps arrive on the first CTA's barriers)
            if (lane == 0) {
                const uint32_t a = (ph ? conv0 : tempty0) + 8 * acc;
                if constexpr (CG == 2) mbar_arrive_cl(lead(a));
                else mbar_arrive(a);
            }
            // the tile's geometry buffer may be filled again
            if (last && E.n_bins > 0 && lane == 0) mbar_arrive(gempty0 + 8 * ((item - 1) & 1));
            if (last) epi_sync(kEpiThreads);  // all private bins written
            if (bins_on && last) {
                // private rows this tile may have written: with the branch-free position
                // path only the tile's own bin range, else the whole window / bin set
                const int NWp = !E.use_window ? E.n_bins
                                : (!lattice && tw.fit ? min(E.NW, tw.nwp) : E.NW);
                // epilogue warp ew reduces eight bins at a time: conflict-free loads, then the
                // FP32 tree of the warp by recursive halving (each exchange sends the half
                // of the bins this lane does not keep: 9 shuffles for 8 bins), after which
                // every fourth lane holds one of the bins.  Lane & 3 picks the round, so one
                // FP64 conversion and add serves up to four rounds, 32 bins (the FP64 pipe
                // is narrow on this part; one lane adding bin after bin took most of this
                // part's time: 8.2 -> 2.7 thousand cycles per tile on a 34^3 lattice, 6.3 -> 3.5
                // on the 32^3 glass).
                for (int b0 = 8 * ew; b0 < NWp; b0 += 32 * kEpiWarps) {
                    float sum = 0.f;
                    int k = NWp;
#pragma unroll 1
                    for (int rd = 0; rd < 4; ++rd) {
                        const int b1 = b0 + rd * 8 * kEpiWarps;
                        if (b1 >= NWp) break;
                        float v8[8];
#pragma unroll
                        for (int u = 0; u < 8; ++u) {
                            // (past the last row: that row again, a value no lane keeps)
                            const float *row = bins + min(b1 + u, NWp - 1) * kBinStride;
                            v8[u] = 0.f;
#pragma unroll
                            for (int m = 0; m < kBinStride / 32; ++m) v8[u] += row[lane + 32 * m];
                        }
                        __syncwarp();
#pragma unroll
                        for (int u = 0; u < 8; ++u) {
                            float4 *row = reinterpret_cast<float4 *>(bins + (b1 + u) * kBinStride);
                            if (b1 + u < NWp)
#pragma unroll
                                for (int m = 0; m < kBinStride / 128; ++m)
                                    row[lane + 32 * m] = make_float4(0.f, 0.f, 0.f, 0.f);
                        }
                        const float sr = warp_sum8(v8, lane);
                        if ((lane & 3) == rd) {
                            sum = sr;
                            k = b1 + ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 +
                                ((lane >> 2) & 1);
                        }
                    }
                    const int b = k < tw.n1 ? tw.blo + k : tw.blo2 + (k - tw.n1);
                    if (k < NWp && b < E.n_bins && ASD_INB(b < args.NB, BND_CACC, args.err)) {
                        if (det) cacci[b] += to_fixed((double)sum, fscale);
                        else cacc[b] += (double)sum;
                    }
                }
                // (tiles whose bins all fit the window put nothing into the fallback bins)
                if (E.use_window && (lattice || !tw.fit)) {
                    epi_sync(kEpiThreads);  // the fallback bins update the same accumulators
                    for (int b = et; b < E.n_bins; b += kEpiThreads) {
                        if (det) {
                            cacci[b] += fbi[b];
                            fbi[b] = 0;
                        } else if (fb[b] != 0.f) {
                            cacc[b] += (double)fb[b];
                            fb[b] = 0.f;
                        }
                    }
                }
            }
        }
        epi_sync(kEpiThreads);
        if (ok && cur_p >= 0) flush_acc(cur_p, cur_t);
    }
    __syncwarp();
    __syncthreads();
    // a pair: neither CTA leaves (or frees TMEM) while the other may still signal it or
    // the first CTA's MMAs may still write its accumulators
    if constexpr (CG == 2) cluster_sync();
    if (warp == 1) {
        tc_after();
        tmem_dealloc<CG>(tmem, kTmemAlloc);
    }
    // the last CTA to finish leaves the work-item counter at zero for the next launch (a
    // memset before every launch cost a small call 1.5 us); every claim was made before
    if (CG == 1 && args.counter && threadIdx.x == 0 &&
        atomicAdd(args.counter + 1, 1ull) == gridDim.x - 1) {
        args.counter[0] = 0;
        args.counter[1] = 0;
    }
}

template <int FORM, int BN, int SWB, int EW, int CG>
int launch_one(const LaunchArgs &a, size_t smem, int sm_count, cudaStream_t s)
{
    auto k = pc_tc_kernel<FORM, BN, SWB, EW, CG>;
    constexpr int kThreads = tc_threads(BN, EW);
    ASD_CUDA_TRY(allow_smem(k, kMaxSmem));
    if constexpr (CG == 1) {
        // persistent: one CTA per SM, no more CTAs than work items
        const int grid = (int)(a.total_tiles < sm_count ? a.total_tiles : sm_count);
        k<<<grid, kThreads, smem, s>>>(a);
    } else {
        // persistent pairs: clusters of two CTAs, as many as can be resident at once (one
        // CTA per SM), no more than work items
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = 2;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3((unsigned)sm_count, 1, 1);
        cfg.blockDim = dim3(kThreads, 1, 1);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = s;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int clusters = 0;
        ASD_CUDA_TRY(cudaOccupancyMaxActiveClusters(&clusters, k, &cfg));
        if (clusters < 1) {
            set_error_text("no CTA pair fits on the device");
            return ASD_EUNSUPPORTED;
        }
        const int64_t pairs = a.total_tiles < clusters ? a.total_tiles : clusters;
        cfg.gridDim = dim3((unsigned)(2 * pairs), 1, 1);
        ASD_CUDA_TRY(cudaLaunchKernelEx(&cfg, k, a));
    }
    ASD_CUDA_TRY(cudaGetLastError());
    return ASD_OK;
}

}  // namespace

// Launch one precision form with CTA pairs (tile widths 256 and 192, 4 or 8 epilogue
// warps); instantiated in its own translation unit per form (pc_tc_*_pair.cu).
template <int FORM>
int tc_launch_pair(const TcLaunchArgs &a, size_t smem, int BN, int ew, int sm_count,
                   cudaStream_t s)
{
    constexpr int SWB = FORM == ASD_SPLIT_BF16 ? 64 : 128;
    if (BN == 256 && ew == 4) return launch_one<FORM, 256, SWB, 4, 2>(a, smem, sm_count, s);
    if (BN == 256 && ew == 8) return launch_one<FORM, 256, SWB, 8, 2>(a, smem, sm_count, s);
    if (BN == 192 && ew == 4) return launch_one<FORM, 192, SWB, 4, 2>(a, smem, sm_count, s);
    if (BN == 192 && ew == 8) return launch_one<FORM, 192, SWB, 8, 2>(a, smem, sm_count, s);
    set_error_text("tensor-core kernel: CTA pairs need 192- or 256-wide tiles");
    return ASD_EUNSUPPORTED;
}

// Launch one precision form.  Instantiated combinations (the rest are rejected):
//   BN = 256 and BN = 192 with 4 or 8 epilogue warps; BN = 128 with 4 warps (192 and 128
//   are the tile widths that leave TMEM room for the phase product); cg = 2 goes to the
//   CTA-pair kernels.
template <int FORM>
int tc_launch_form(const TcLaunchArgs &a, size_t smem, int BN, int ew, int cg, int sm_count,
                   cudaStream_t s)
{
    constexpr int SWB = FORM == ASD_SPLIT_BF16 ? 64 : 128;
    if (cg == 2) return tc_launch_pair<FORM>(a, smem, BN, ew, sm_count, s);
    if (BN == 256 && ew == 4) return launch_one<FORM, 256, SWB, 4, 1>(a, smem, sm_count, s);
    if (BN == 256 && ew == 8) return launch_one<FORM, 256, SWB, 8, 1>(a, smem, sm_count, s);
    if (BN == 192 && ew == 4) return launch_one<FORM, 192, SWB, 4, 1>(a, smem, sm_count, s);
    if (BN == 192 && ew == 8) return launch_one<FORM, 192, SWB, 8, 1>(a, smem, sm_count, s);
    if (BN == 128 && ew == 4) return launch_one<FORM, 128, SWB, 4, 1>(a, smem, sm_count, s);
    set_error_text("tensor-core kernel: unsupported (tile width, epilogue warps)");
    return ASD_EUNSUPPORTED;
}

}  // namespace asd
