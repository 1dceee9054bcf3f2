// Thin inline-PTX wrappers for the sm_100a features the kernels use:
// mbarrier, TMA tiled loads (each CTA fetches its own tiles), tcgen05 MMA / TMEM, proxy fences.
// Every wait is bounded: after TIK_WAIT_LIMIT_NS the waiter raises a flag in the
// device status word and in a CTA-local abort word, and every later wait of that
// CTA returns at once, so a scheduling bug ends the kernel instead of hanging it.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <stdint.h>

namespace tik {

constexpr unsigned long long TIK_WAIT_LIMIT_NS = 2000000000ull;  // 2 s per wait
constexpr int TIK_DEV_BAD_BLOCK = 1;      // block-table entry outside [0, num_pages)
constexpr int TIK_DEV_BAD_TARGET = 2;     // target id outside [0, V)
constexpr int TIK_DEV_WAIT_EXPIRED = 4;   // a bounded wait ran out
constexpr int TIK_DEV_BAD_POSITION = 8;   // token position outside the cos/sin table
constexpr int TIK_DEV_BAD_CONTEXT = 16;   // decode: ctx_lens[b] above the host's max_ctx_len

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ unsigned long long globaltimer_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

// ---------------------------------------------------------------- mbarrier
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_barrier_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// Bounded wait.  `abort_word` lives in shared memory (one per CTA).
__device__ __forceinline__ void mbar_wait(uint32_t bar, uint32_t parity,
                                          volatile int* abort_word, int* dev_status) {
    if (mbar_try_wait(bar, parity)) return;
    const unsigned long long t0 = globaltimer_ns();
    for (uint32_t it = 1;; ++it) {
        if (mbar_try_wait(bar, parity)) return;
        if ((it & 63u) == 0u) {
            if (*abort_word) return;
            if (globaltimer_ns() - t0 > TIK_WAIT_LIMIT_NS) {
                *abort_word = 1;
                atomicOr(dev_status, TIK_DEV_WAIT_EXPIRED);
                return;
            }
        }
    }
}

// The same for a converged warp (the issuing warps): every lane waits, all leave together.
__device__ __forceinline__ void mbar_wait_warp(uint32_t bar, uint32_t parity,
                                               volatile int* abort_word, int* dev_status) {
    mbar_wait(bar, parity, abort_word, dev_status);
    __syncwarp();
}
// A value that is the same in all lanes, in a form the compiler knows to be (uniform registers).
__device__ __forceinline__ int warp_uniform(int v) { return __shfl_sync(0xffffffffu, v, 0); }
__device__ __forceinline__ uint32_t warp_uniform(uint32_t v) { return __shfl_sync(0xffffffffu, v, 0); }

// The sequence s with cu[s] <= token < cu[s + 1] (empty sequences skipped), found by a whole warp: 32 probes
// per round, so one or two rounds of global latency instead of the log2(S) dependent loads of a binary
// search.  0 <= token; S >= 1.
__device__ __forceinline__ int warp_find_sequence(const int32_t* cu, int S, long long token, int lane) {
    int lo = 0, hi = S;                  // cu[lo] <= token, and cu[hi] > token if the token exists
    while (hi - lo > 1) {
        const int step = (hi - lo + 31) / 32, probe = lo + step * (lane + 1);
        const unsigned below = __ballot_sync(0xffffffffu, probe < hi && cu[probe] <= token);
        const int n = __popc(below);     // cu is ascending: the first n probes
        lo += step * n;
        hi = min(hi, lo + step);
    }
    return lo;
}

// ---------------------------------------------------------------- programmatic dependent launch
// A kernel launched with the programmatic-stream-serialization attribute may start while its
// predecessor in the stream still runs: its CTAs are scheduled once every CTA of the predecessor
// has executed launch_dependents (or exited), and pdl_wait() blocks until the predecessor has
// completed and its writes are visible.  Every kernel of the library is launched this way
// (launch_pdl in tik_internal.h): block scheduling, barrier set-up and tensor-memory allocation of a
// call run under the tail of the call before it.  The rules that keep a chain of such kernels
// ordered like a plain stream:
//   * before pdl_wait() a CTA touches no global memory except kernel parameters and L2 prefetches
//     (writes land in L2, so a prefetched line cannot go stale);
//   * every CTA executes pdl_wait() on every path, early exits included, so a grid completes after
//     its predecessor.  Two grids overlap their predecessor on purpose, which writes nothing that they read: the dQ
//     grid of the backward and the persistent grid behind the single-tile grid.  They wait at their end (one
//     block of dQ, every CTA of the other), never release dependents early, and read what earlier calls may have
//     left in L1 around it (__ldcg);
//   * pdl_launch_dependents() comes after pdl_wait(): when a kernel starts, everything before its
//     immediate predecessor has completed;
//   * ... and after the CTA's tensor memory is allocated (behind the barrier that publishes its address): a dependent
//     CTA that shares the SM allocates before it waits, and must not hold columns that an earlier CTA, which it
//     waits for, has yet to get;
//   * a call of many small CTAs per SM releases its dependents at its end when the next kernel may be of that kind
//     too (calls of few CTAs and those before a decode step at the start): early dependents take the slots that happen to be free and the next call runs with its CTAs spread
//     unevenly (pre-attention step of 5 x 450 tokens, 64 + 8 heads, call after call: 20.6 us in plain stream order, 29.4
//     released at the start, 20.9 at the end; cache write of 5 x 600 tokens 3.9 and 3.6; backward of one sequence of 2048
//     tokens, whose delta kernel comes first, 120.8 and 117.3).  RMSNorm and SwiGLU, which a GEMM follows, release at
//     the start: its weight prefetch runs under them (RMSNorm, GEMM, SwiGLU, GEMM of 64 rows 86.1 us, 89.6 otherwise);
//   * no kernel parameter is __restrict__ and nothing is loaded through the read-only path (__ldg): a kernel's
//     lifetime overlaps the one that writes its inputs, and either would let the compiler take them for constant
//     throughout and move a load above the wait.
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// ---------------------------------------------------------------- fences
__device__ __forceinline__ void fence_proxy_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// ---------------------------------------------------------------- TMA (tiled loads, one destination CTA each)
__device__ __forceinline__ void tma_prefetch_desc(const CUtensorMap* m) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(m)) : "memory");
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* m, uint32_t bar,
                                            int c0, int c1) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4}], [%2];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(m)), "r"(bar), "r"(c0), "r"(c1)
        : "memory");
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* m, uint32_t bar,
                                            int c0, int c1, int c2) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(m)), "r"(bar), "r"(c0), "r"(c1), "r"(c2)
        : "memory");
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* m, uint32_t bar,
                                            int c0, int c1, int c2, int c3) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4, %5, %6}], [%2];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(m)), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
        : "memory");
}

// L2 prefetch of a tile (no shared-memory destination, no barrier).
__device__ __forceinline__ void tma_prefetch_l2_3d(const CUtensorMap* m, int c0, int c1, int c2) {
    asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];" ::"l"(
                     reinterpret_cast<uint64_t>(m)),
                 "r"(c0), "r"(c1), "r"(c2)
                 : "memory");
}
__device__ __forceinline__ void tma_prefetch_l2_4d(const CUtensorMap* m, int c0, int c1, int c2, int c3) {
    asm volatile("cp.async.bulk.prefetch.tensor.4d.L2.global.tile [%0, {%1, %2, %3, %4}];" ::"l"(
                     reinterpret_cast<uint64_t>(m)),
                 "r"(c0), "r"(c1), "r"(c2), "r"(c3)
                 : "memory");
}
__device__ __forceinline__ void tma_prefetch_l2_2d(const CUtensorMap* m, int c0, int c1) {
    asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];" ::"l"(
                     reinterpret_cast<uint64_t>(m)),
                 "r"(c0), "r"(c1)
                 : "memory");
}
// Tiled store shared -> global (bulk async group); never started at a negative coordinate.
__device__ __forceinline__ void tma_store_3d(const CUtensorMap* m, uint32_t src, int c0, int c1, int c2) {
    asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.tile.bulk_group [%0, {%2, %3, %4}], [%1];" ::"l"(
                     reinterpret_cast<uint64_t>(m)),
                 "r"(src), "r"(c0), "r"(c1), "r"(c2)
                 : "memory");
}
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* m, uint32_t src, int c0, int c1) {
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%2, %3}], [%1];" ::"l"(
                     reinterpret_cast<uint64_t>(m)),
                 "r"(src), "r"(c0), "r"(c1)
                 : "memory");
}
// at most one bulk store group of this thread is still reading its shared-memory source
__device__ __forceinline__ void tma_store_wait_read1() {
    asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
}
__device__ __forceinline__ void tma_store_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// waits until the committed stores have finished reading shared memory
__device__ __forceinline__ void tma_store_wait_read() {
    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}
__device__ __forceinline__ void tma_store_wait_all() {
    asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

// ---------------------------------------------------------------- TMEM
// One full warp allocates `ncols` (power of two, >= 32) columns; the base address lands in smem.
__device__ __forceinline__ void tmem_alloc(uint32_t smem_dst, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_dst),
                 "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols)
                 : "memory");
}

// 32 lanes x 32 columns of 32-bit: thread i of the warp gets lane (base+i), registers = columns.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
          "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]),
          "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]),
          "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%32], "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31};" ::"r"(r[0]),
        "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
        "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]),
        "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]),
        "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]),
        "r"(r[30]), "r"(r[31]), "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%16], "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15};" ::"r"(r[0]),
        "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
        "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() {
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_wait_st() {
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// ---------------------------------------------------------------- tcgen05.mma (bf16 x bf16 -> fp32)
// Shared-memory matrix descriptor, 128-byte swizzle.  `lbo`/`sbo` in bytes.
//  K-major operand (rows of 64 bf16 = 128 B, 8-row atoms of 1 KiB): sbo = 1024, lbo unused.
//  MN-major operand (64 contiguous MN elements per row, 8 K-rows per atom): lbo = bytes between
//  64-element MN groups, sbo = bytes between 8-row K groups.
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    uint64_t d = 0;
    d |= static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);
    d |= static_cast<uint64_t>((lbo >> 4) & 0x3FFFu) << 16;
    d |= static_cast<uint64_t>((sbo >> 4) & 0x3FFFu) << 32;
    d |= 1ull << 46;   // descriptor version for sm_100
    d |= 2ull << 61;   // SWIZZLE_128B
    return d;
}
// Instruction descriptor: D fp32, A/B bf16, A K-major; B K-major or MN-major.
__host__ __device__ constexpr uint32_t mma_idesc_bf16(int M, int N, bool b_mn_major) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((b_mn_major ? 1u : 0u) << 16) |
           (static_cast<uint32_t>(N >> 3) << 17) | (static_cast<uint32_t>(M >> 4) << 24);
}
// Named barriers (ids 1..15; 0 is __syncthreads): producer side arrives, consumer side syncs.
__device__ __forceinline__ void named_bar_arrive(uint32_t id, uint32_t nthreads) {
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}
__device__ __forceinline__ void named_bar_sync(uint32_t id, uint32_t nthreads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}
// ---- MMA chains issued from one asm block.  The issuing warp's own instruction stream limits how fast
// MMAs enter the tensor pipe.  tcgen05 instructions take their operands from the warp's uniform
// registers, so the WHOLE warp, converged, executes the issue path -- waits (mbar_wait_warp), descriptor
// arithmetic on warp-uniform values, chains, commits -- and one elected lane issues.  With the path
// inside `if (lane == 0)` every operand of every MMA was moved over from per-thread registers:
// stand-alone, a chain of eight M128 x N128 x K16 with two barrier waits and two commits took 1485 clk of
// issue that way and takes 824 this way (512 clk of MMAs); a chain alone 798 -> 627.
// Offsets are in descriptor units (16 bytes).
#define TIK_MMA_SS_STEP(OFFA, OFFB)                                   \
    "add.u64 da, %1, " #OFFA ";\n\t"                                  \
    "add.u64 db, %2, " #OFFB ";\n\t"                                  \
    "@e tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %3, pt;\n\t"

// K-major A and B, 64-wide K slice inside one 128B-swizzle atom: 4 steps of 32 bytes.
// first_accumulate == 0 makes the first MMA overwrite D.
__device__ __forceinline__ void mma_ss_chain4(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc,
                                              uint32_t idesc, uint32_t first_accumulate) {
    asm volatile(
        "{\n\t.reg .pred p0, pt, e;\n\telect.sync _|e, 0xffffffff;\n\t.reg .b64 da, db;\n\t"
        "setp.ne.b32 p0, %4, 0;\n\tsetp.eq.b32 pt, 0, 0;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p0;\n\t"
        TIK_MMA_SS_STEP(2, 2) TIK_MMA_SS_STEP(4, 4) TIK_MMA_SS_STEP(6, 6)
        "}" ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(first_accumulate)
        : "memory");
}
// Same for a 128-wide K (two atoms 16 KiB = 1024 units apart): 8 steps, first one overwrites D.
__device__ __forceinline__ void mma_ss_chain8_fresh(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc,
                                                    uint32_t idesc) {
    asm volatile(
        "{\n\t.reg .pred p0, pt, e;\n\telect.sync _|e, 0xffffffff;\n\t.reg .b64 da, db;\n\t"
        "setp.ne.b32 p0, 0, 0;\n\tsetp.eq.b32 pt, 0, 0;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p0;\n\t"
        TIK_MMA_SS_STEP(2, 2) TIK_MMA_SS_STEP(4, 4) TIK_MMA_SS_STEP(6, 6)
        TIK_MMA_SS_STEP(1024, 1024) TIK_MMA_SS_STEP(1026, 1026) TIK_MMA_SS_STEP(1028, 1028)
        TIK_MMA_SS_STEP(1030, 1030)
        "}" ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc)
        : "memory");
}
__device__ __forceinline__ void mma_ss_chain4_fresh(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc,
                                                    uint32_t idesc) {
    mma_ss_chain4(d_tmem, a_desc, b_desc, idesc, 0u);
}

// A from TMEM (8 columns per step), B = MN-major tile whose 16-key steps are 2 KiB = 128 units
// apart: the 8 steps of one 128-key tile.  first_accumulate == 0 overwrites D on the first step.
#define TIK_MMA_TS_STEP(OFFA, OFFB)                                   \
    "add.u32 ta, %1, " #OFFA ";\n\t"                                  \
    "add.u64 db, %2, " #OFFB ";\n\t"                                  \
    "@e tcgen05.mma.cta_group::1.kind::f16 [%0], [ta], db, %3, pt;\n\t"
__device__ __forceinline__ void mma_ts_chain8(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc,
                                              uint32_t idesc, uint32_t first_accumulate) {
    asm volatile(
        "{\n\t.reg .pred p0, pt, e;\n\telect.sync _|e, 0xffffffff;\n\t.reg .b64 db;\n\t.reg .b32 ta;\n\t"
        "setp.ne.b32 p0, %4, 0;\n\tsetp.eq.b32 pt, 0, 0;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p0;\n\t"
        TIK_MMA_TS_STEP(8, 128) TIK_MMA_TS_STEP(16, 256) TIK_MMA_TS_STEP(24, 384)
        TIK_MMA_TS_STEP(32, 512) TIK_MMA_TS_STEP(40, 640) TIK_MMA_TS_STEP(48, 768)
        TIK_MMA_TS_STEP(56, 896)
        "}" ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(first_accumulate)
        : "memory");
}

// All eight steps with A laid out as four 32-column blocks whose first 16 columns hold the two
// steps of that block (a thread that owns 32 fp32 columns of a tile leaves the bf16 pairs of its
// 32 contraction rows in the first 16 of them).
__device__ __forceinline__ void mma_ts_chain8_blocks(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc,
                                                     uint32_t idesc, uint32_t first_accumulate) {
    asm volatile(
        "{\n\t.reg .pred p0, pt, e;\n\telect.sync _|e, 0xffffffff;\n\t.reg .b64 db;\n\t.reg .b32 ta;\n\t"
        "setp.ne.b32 p0, %4, 0;\n\tsetp.eq.b32 pt, 0, 0;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p0;\n\t"
        TIK_MMA_TS_STEP(8, 128) TIK_MMA_TS_STEP(32, 256) TIK_MMA_TS_STEP(40, 384)
        TIK_MMA_TS_STEP(64, 512) TIK_MMA_TS_STEP(72, 640) TIK_MMA_TS_STEP(96, 768)
        TIK_MMA_TS_STEP(104, 896)
        "}" ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(first_accumulate)
        : "memory");
}

// ---------------------------------------------------------------- CTA pairs (cta_group::2)
// Two CTAs of a cluster of two, on neighbouring SMs, execute one MMA of M = 256: each holds its
// own 128 rows of A and half of the B tile in its shared memory and its own 128 accumulator rows
// in its tensor memory.  The MMA is issued by an elected lane of the leader CTA's (cluster rank 0) issuing warp.
__device__ __forceinline__ uint32_t cluster_ctarank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// shared::cluster address of the location `saddr` (a shared::cta address) in the CTA of rank `rank`
__device__ __forceinline__ uint32_t mapa_cluster(uint32_t saddr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// arrive on an mbarrier of any CTA of the cluster
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// TMA tile load into this CTA's shared memory whose bytes are counted on a barrier that may live
// in the peer CTA (every CTA fetches its own tile)
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* m, uint32_t bar_cluster_addr,
                                                 int c0, int c1) {
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4}], [%2];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(m)), "r"(bar_cluster_addr), "r"(c0), "r"(c1)
        : "memory");
}
// Tensor-memory allocation for a CTA pair: one warp of EACH CTA (the same warp index, the same
// shared-memory slot offset) executes these.
__device__ __forceinline__ void tmem_alloc_pair(uint32_t smem_dst, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_dst), "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tmem_relinquish_pair() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
// Pair MMA chain over a 64-wide K slice (4 steps of 32 bytes), K-major A and B, as mma_ss_chain4.
__device__ __forceinline__ void mma_ss_chain4_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc,
                                                   uint32_t idesc, uint32_t first_accumulate) {
    asm volatile(
        "{\n\t.reg .pred p0, pt, e;\n\telect.sync _|e, 0xffffffff;\n\t.reg .b64 da, db;\n\t"
        "setp.ne.b32 p0, %4, 0;\n\tsetp.eq.b32 pt, 0, 0;\n\t"
        "@e tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p0;\n\t"
        "add.u64 da, %1, 2;\n\tadd.u64 db, %2, 2;\n\t"
        "@e tcgen05.mma.cta_group::2.kind::f16 [%0], da, db, %3, pt;\n\t"
        "add.u64 da, %1, 4;\n\tadd.u64 db, %2, 4;\n\t"
        "@e tcgen05.mma.cta_group::2.kind::f16 [%0], da, db, %3, pt;\n\t"
        "add.u64 da, %1, 6;\n\tadd.u64 db, %2, 6;\n\t"
        "@e tcgen05.mma.cta_group::2.kind::f16 [%0], da, db, %3, pt;\n\t"
        "}" ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(first_accumulate)
        : "memory");
}
// Arrives on one mbarrier (of either CTA: a shared::cluster address) once all pair MMAs issued so
// far by this warp have completed.
__device__ __forceinline__ void mma_commit_pair(uint32_t bar_cluster_addr) {
    asm volatile(
        "{\n\t.reg .pred e;\n\telect.sync _|e, 0xffffffff;\n\t"
        "@e tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(bar_cluster_addr)
        : "memory");
}

// Arrives on the mbarrier once all MMAs issued so far by this warp (its elected lane) have completed.
__device__ __forceinline__ void mma_commit(uint32_t bar) {
    asm volatile(
        "{\n\t.reg .pred e;\n\telect.sync _|e, 0xffffffff;\n\t"
        "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(bar)
        : "memory");
}

}  // namespace tik
