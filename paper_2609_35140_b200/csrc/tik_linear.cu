// Dense linear layer y = x W^T (bf16 in, fp32 accumulation in TMEM, bf16 out) for sm_100a: the
// FFN projections of the unified operator set.  An output element is one fixed chain of K16 MMAs in
// ascending K into one fp32 accumulator (no split-K), so it depends on its x row and its W row only: a
// row gives the same bits whether it is computed alone (decode) or inside a long batch (prefill, policy
// update), and whichever of the three kernels below computes it:
//   linear_kernel         CTA pairs (two-SM M256 MMAs), for calls that fill the chip: band raster, or
//                         persistent over (column step, pair of row tiles) units
//   linear_unit_kernel    persistent single CTAs over (column unit, row tile) units, for calls of few rows or
//                         narrow outputs that pairs of 256 x 256 would leave idle SMs
//   linear_narrow_kernel  one unit of few weight rows per CTA, for narrow outputs
// linear_narrow_choose and linear_choose (tik_internal.h) pick.
#include "tik_core.cuh"
#include "tik_internal.h"
#include "tik_ptx.cuh"

namespace tik {

namespace lin {
constexpr int NB = 256;                      // output columns per MMA
constexpr uint32_t A_BYTES = 128 * 128;      // 128 rows x 64 bf16
constexpr uint32_t STG_BYTES = 128 * 128;    // output staging: 128 rows x 64 bf16, two buffers
constexpr int BAND = 32;                     // row tiles per L2 band (even: CTA pairs stay inside a band)
constexpr int THREADS = 192;                 // warp 0 TMA, warp 1 MMA, warps 2..5 epilogue
// Two CTAs on neighbouring SMs share every MMA (M = 256 rows); each stages its own 128 rows of
// x and half of a step's weight rows, as in the log-probability kernel.
constexpr int STAGES = 6;
constexpr uint32_t STAGE_BYTES = A_BYTES + (NB / 2) * 128;
constexpr uint32_t OFF_STG = STAGES * STAGE_BYTES;
constexpr uint32_t OFF_BAR = OFF_STG + 2 * STG_BYTES;
constexpr uint32_t BYTES = OFF_BAR + 256;
constexpr uint32_t ALLOC = BYTES + 1024;
}  // namespace lin

// A TMA warp streams 64-wide K slices of x and W through a shared-memory ring, an MMA warp accumulates the
// whole K range into one of two 256-column TMEM accumulators, and four epilogue warps (one thread per row)
// round the accumulator to bf16 and send it out through shared memory and tiled TMA stores while the next
// step is being accumulated.
__global__ void __launch_bounds__(lin::THREADS, 1)
linear_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
              const __grid_constant__ CUtensorMap tmY, const LinearParams p) {
    using namespace lin;
    constexpr uint32_t TMEM_COLS = 512;      // two 256-column accumulators
    constexpr uint32_t IDESC = mma_idesc_bf16(256, NB, false);
    const int tid = threadIdx.x, warp = warp_uniform(tid >> 5), lane = tid & 31;
    const uint32_t rank = cluster_ctarank();     // 0 = the CTA that issues the pair's MMAs

    // raster: bands of BAND row tiles; within a band the row tile varies fastest so the CTAs in
    // flight share one super-chunk of W in L2 and W is streamed from HBM once per band
    const int ntile = static_cast<int>((p.T + 127) / 128);
    const long long per_band = static_cast<long long>(BAND) * p.nsuper;
    const int band = static_cast<int>(blockIdx.x / per_band);
    const int band_tiles = min(BAND, ntile - band * BAND);
    const long long rem = blockIdx.x - band * per_band;
    const int sup = static_cast<int>(rem / BAND);
    const int tile_in_band = static_cast<int>(rem % BAND);
    // unit mode (up to 16 row tiles): one persistent pair per two SMs walks the
    // units q = pair index, + number of pairs, ...; unit q = (column step q / ntp, pair of row
    // tiles q % ntp): the pairs running at one time share a few steps of W in L2, and x (at most
    // 2048 rows) stays there throughout.  Same MMA chain per element.
    const bool unit_mode = p.unit_mode != 0;
    const int u_first = static_cast<int>(blockIdx.x >> 1), u_stride = static_cast<int>(gridDim.x >> 1);
    if (!unit_mode && (tile_in_band & ~1) >= band_tiles) {   // a pair leaves only together
        pdl_wait();
        return;
    }
    const int row_fixed = (band * BAND + tile_in_band) * 128;
    const int col_base = sup * p.super_cols;
    const int ntp = unit_mode ? p.ntp : 1;
    auto row_of = [&](int nt) {
        return unit_mode ? (2 * ((u_first + nt * u_stride) % ntp) + static_cast<int>(rank)) * 128 : row_fixed;
    };
    auto col_of = [&](int nt) { return unit_mode ? ((u_first + nt * u_stride) / ntp) * NB : col_base + nt * NB; };
    const int n_nt = unit_mode ? (p.nunit - u_first + u_stride - 1) / u_stride
                               : min(p.super_cols / NB, (p.N - col_base + NB - 1) / NB);   // 256-column steps
    const int n_kb = p.K / 64;

    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw_addr = smem_u32(smem_raw);
    const uint32_t pad = (1024u - (raw_addr & 1023u)) & 1023u;
    uint8_t* smem = smem_raw + pad;
    const uint32_t sbase = raw_addr + pad;
    const uint32_t bar_full = sbase + OFF_BAR;               // STAGES barriers
    const uint32_t bar_empty = bar_full + 8 * STAGES;        // STAGES barriers
    const uint32_t bar_acc_full = bar_empty + 8 * STAGES;    // 2
    const uint32_t bar_acc_empty = bar_acc_full + 16;        // 2
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem + OFF_BAR + 8 * (2 * STAGES + 4));
    volatile int* abort_word = reinterpret_cast<volatile int*>(smem + OFF_BAR + 8 * (2 * STAGES + 4) + 4);

    if (tid == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(bar_full + 8 * s, 1);
            mbar_init(bar_empty + 8 * s, 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(bar_acc_full + 8 * b, 1);
            mbar_init(bar_acc_empty + 8 * b, 256);
        }
        fence_barrier_init();
        tma_prefetch_desc(&tmA);
        tma_prefetch_desc(&tmB);
        tma_prefetch_desc(&tmY);
        // this CTA's first weight tiles on their way to L2 while the kernel before this one drains
        const int first_col = col_of(0) + (NB / 2) * static_cast<int>(rank);
        if (static_cast<int>(blockIdx.x) < p.sm_count && first_col < p.N)
            for (int kb = 0; kb < min(n_kb, STAGES); ++kb) tma_prefetch_l2_2d(&tmB, kb * 64, first_col);
    }
    if (warp == 1) {
        tmem_alloc_pair(smem_u32(const_cast<uint32_t*>(tmem_slot)), TMEM_COLS);
        tmem_relinquish_pair();
    }
    pdl_wait();
    if (tid == 0) *abort_word = (*reinterpret_cast<volatile int*>(p.dev_status) & TIK_DEV_WAIT_EXPIRED) ? 1 : 0;
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();            // the peer's barriers exist before anything signals them
    tc_fence_after();
    pdl_launch_dependents();
    const uint32_t tmem = *tmem_slot;
    const uint32_t lead_full = mapa_cluster(bar_full, 0);
    const uint32_t lead_acc_empty = mapa_cluster(bar_acc_empty, 0);
    const uint32_t peer_empty = mapa_cluster(bar_empty, 1);
    const uint32_t peer_acc_full = mapa_cluster(bar_acc_full, 1);

    if (warp == 0) {
        // ------------------------------------------------------------ TMA producer
        if (lane == 0) {
            uint32_t it = 0;
            for (int nt = 0; nt < n_nt; ++nt) {
                const int col0 = col_of(nt), row0 = row_of(nt);
                for (int kb = 0; kb < n_kb; ++kb, ++it) {
                    if (*abort_word) break;      // a wait expired somewhere: stop issuing copies
                    const int s = it % STAGES;
                    const uint32_t use = it / STAGES;
                    if (use > 0) mbar_wait(bar_empty + 8 * s, (use - 1) & 1, abort_word, p.dev_status);
                    // rows past T and W rows past N are outside the tensor maps and arrive as zeros
                    if (rank == 0) mbar_expect_tx(bar_full + 8 * s, 2 * STAGE_BYTES);   // both CTAs' bytes
                    tma_load_2d_pair(sbase + s * STAGE_BYTES, &tmA, lead_full + 8 * s, kb * 64, row0);
                    tma_load_2d_pair(sbase + s * STAGE_BYTES + A_BYTES, &tmB, lead_full + 8 * s, kb * 64,
                                     col0 + (NB / 2) * static_cast<int>(rank));
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer
        if (rank == 0) {
            const uint32_t tmem = warp_uniform(*tmem_slot);
            uint32_t it = 0;
            for (int nt = 0; nt < n_nt; ++nt) {
                const int buf = nt & 1;
                const uint32_t use = nt >> 1;
                if (use > 0) mbar_wait_warp(bar_acc_empty + 8 * buf, (use - 1) & 1, abort_word, p.dev_status);
                tc_fence_after();
                for (int kb = 0; kb < n_kb; ++kb, ++it) {
                    if (*abort_word) break;
                    const int s = it % STAGES;
                    mbar_wait_warp(bar_full + 8 * s, (it / STAGES) & 1, abort_word, p.dev_status);
                    tc_fence_after();
                    const uint32_t a0 = sbase + s * STAGE_BYTES, b0 = a0 + A_BYTES;
                    mma_ss_chain4_pair(tmem + buf * NB, smem_desc_sw128(a0, 0, 1024), smem_desc_sw128(b0, 0, 1024), IDESC, kb ? 1u : 0u);
                    mma_commit_pair(bar_empty + 8 * s);
                    mma_commit_pair(peer_empty + 8 * s);
                }
                mma_commit_pair(bar_acc_full + 8 * buf);
                mma_commit_pair(peer_acc_full + 8 * buf);
            }
        }
    } else {
        // ------------------------------------------------------------ epilogue (warps 2..5)
        // Thread per row: 64 columns at a time go from TMEM to a 128B-swizzled staging tile in
        // shared memory and leave as one tiled TMA store of 128 rows x 128 bytes (row-by-row
        // 16-byte stores from 128 threads cost a third of the kernel on wide outputs).  The store
        // clips at the tensor's bounds, so rows past T and columns past N need no guard.  Two
        // staging tiles alternate; the storing thread lets at most one store group read behind it.
        const int quarter = warp & 3;                      // TMEM lane quarter of this warp
        const int row = quarter * 32 + lane;
        uint32_t piece = 0;
        for (int nt = 0; nt < n_nt; ++nt) {
            const int buf = nt & 1;
            mbar_wait(bar_acc_full + 8 * buf, (nt >> 1) & 1, abort_word, p.dev_status);
            tc_fence_after();
            const int col0 = col_of(nt), row0 = row_of(nt);
            const uint32_t taddr = tmem + (static_cast<uint32_t>(quarter * 32) << 16) + buf * NB;
#pragma unroll 1
            for (int q = 0; q < NB / 64; ++q, ++piece) {
                if (col0 + 64 * q >= p.N) break;               // uniform: columns past N
                uint32_t v[64];
                tmem_ld32(taddr + 64 * q, *reinterpret_cast<uint32_t(*)[32]>(&v[0]));
                tmem_ld32(taddr + 64 * q + 32, *reinterpret_cast<uint32_t(*)[32]>(&v[32]));
                tmem_wait_ld();
                uint8_t* stg = smem + OFF_STG + (piece & 1) * STG_BYTES;
                // the store that last read this staging tile (two pieces ago) has finished reading
                if (warp == 2 && lane == 0) tma_store_wait_read1();
                named_bar_sync(1, 128);
#pragma unroll
                for (int c16 = 0; c16 < 8; ++c16) {
                    const uint4 val = make_uint4(
                        pack_bf16x2(__uint_as_float(v[8 * c16]), __uint_as_float(v[8 * c16 + 1])),
                        pack_bf16x2(__uint_as_float(v[8 * c16 + 2]), __uint_as_float(v[8 * c16 + 3])),
                        pack_bf16x2(__uint_as_float(v[8 * c16 + 4]), __uint_as_float(v[8 * c16 + 5])),
                        pack_bf16x2(__uint_as_float(v[8 * c16 + 6]), __uint_as_float(v[8 * c16 + 7])));
                    *reinterpret_cast<uint4*>(stg + row * 128 + ((c16 ^ (row & 7)) << 4)) = val;
                }
                fence_proxy_async_smem();
                named_bar_sync(1, 128);
                if (warp == 2 && lane == 0) {
                    tma_store_2d(&tmY, smem_u32(stg), col0 + 64 * q, row0);
                    tma_store_commit();
                }
            }
            // all TMEM reads of this accumulator are done: hand it back to the MMA warp
            tc_fence_before();
            mbar_arrive_cluster(lead_acc_empty + 8 * buf);
        }
        if (warp == 2 && lane == 0) tma_store_wait_read();     // shared memory stays valid until the last read
    }

    if (*abort_word) {   // let copies and MMAs in flight finish before shared memory and TMEM are released
        const unsigned long long t0 = globaltimer_ns();
        while (globaltimer_ns() - t0 < 1000000ull) {
        }
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();            // neither CTA leaves while the other may still touch it
    if (warp == 1) tmem_dealloc_pair(tmem, TMEM_COLS);
}

// ---------------------------------------------------------------------------------------------
// Calls of few rows (one row tile: a decode step) and of up to 16 row tiles whose output is too narrow for
// the pair kernel's 256 x 256 units to occupy the SMs.  A call of one row tile is one pass over W at HBM
// rate, so the schedule is built for bytes in flight and even SM load: the grid is one persistent
// CTA per SM walking units u = blockIdx.x, + gridDim.x, ...; a unit is `nu` = 64, 128 or 256 output columns of
// one row tile (row tile fastest: the CTAs running at one time share W columns in L2);
// only `a_rows` = 8, 16, 32, 64 or 128 rows of x are staged per K slice (the MMA spans 64 or 128 rows: rows
// past a_rows read whatever the stage holds, their accumulator rows are never stored); the ring
// has as many stages as fit in 192 KiB (3 .. 12) of one, two or four K slices each, and the producer runs ahead
// into the next unit while the epilogue of the last one drains.
namespace linu {
constexpr uint32_t RING_BYTES = 192 * 1024;
constexpr int MAX_STAGES = 12;
constexpr uint32_t OFF_STG = RING_BYTES;
constexpr uint32_t OFF_BAR = OFF_STG + 2 * lin::STG_BYTES;
constexpr uint32_t BYTES = OFF_BAR + 512;
constexpr uint32_t ALLOC = BYTES + 1024;
}  // namespace linu

__global__ void __launch_bounds__(lin::THREADS, 1)
linear_unit_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                   const __grid_constant__ CUtensorMap tmY, const LinearParams p) {
    using namespace linu;
    constexpr uint32_t TMEM_COLS = 512;      // two accumulators, 256 columns apart
    const int tid = threadIdx.x, warp = warp_uniform(tid >> 5), lane = tid & 31;
    const int nu = p.nu;
    const uint32_t a_bytes = static_cast<uint32_t>(p.a_rows) * 128u;
    const uint32_t slice_bytes = a_bytes + static_cast<uint32_t>(nu) * 128u;      // a multiple of 1 KiB
    // K slices per stage: the issuing warp spends ~300 cycles per stage on its barrier wait, fence,
    // descriptors and commit, more than four narrow MMAs run (N = 128: 256 cycles, N = 64: ~190);
    // 256 / nu slices per stage (as long as three stages fit) bring that share down (N = 256 MMAs run
    // 512 cycles per slice and hide it)
    int kps = 256 / nu;
    while (kps > 1 && RING_BYTES / (slice_bytes * static_cast<uint32_t>(kps)) < 3u) kps >>= 1;
    const uint32_t stage_bytes = slice_bytes * static_cast<uint32_t>(kps);
    const int nst = min(MAX_STAGES, static_cast<int>(RING_BYTES / stage_bytes));
    const int n_my = (p.nunit - static_cast<int>(blockIdx.x) + static_cast<int>(gridDim.x) - 1) / static_cast<int>(gridDim.x);
    const int n_kb = p.K / 64;
    // At most 64 rows: M64, half the tensor work of M128 (16 rows, K 1536, N 17920, in a graph: 14 -> 11.3 us);
    // accumulator row i then sits on lane i % 16 of lane quarter i / 16.
    const bool m64 = p.a_rows <= 64;
    const uint32_t idesc = mma_idesc_bf16(m64 ? 64 : 128, nu, false);
    // (the divisions, for calls of one row tile, cost 0.2 us of 6)
    auto unit_of = [&](int i) { return static_cast<int>(blockIdx.x) + i * static_cast<int>(gridDim.x); };
    auto unit_col = [&](int i) { return (p.ntp == 1 ? unit_of(i) : unit_of(i) / p.ntp) * nu; };
    auto unit_row = [&](int i) { return p.ntp == 1 ? 0 : unit_of(i) % p.ntp * 128; };

    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw_addr = smem_u32(smem_raw);
    const uint32_t pad = (1024u - (raw_addr & 1023u)) & 1023u;
    uint8_t* smem = smem_raw + pad;
    const uint32_t sbase = raw_addr + pad;
    const uint32_t bar_full = sbase + OFF_BAR;                   // MAX_STAGES barriers
    const uint32_t bar_empty = bar_full + 8 * MAX_STAGES;        // MAX_STAGES barriers
    const uint32_t bar_acc_full = bar_empty + 8 * MAX_STAGES;    // 2
    const uint32_t bar_acc_empty = bar_acc_full + 16;            // 2
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem + OFF_BAR + 8 * (2 * MAX_STAGES + 4));
    volatile int* abort_word = reinterpret_cast<volatile int*>(smem + OFF_BAR + 8 * (2 * MAX_STAGES + 4) + 4);

    if (tid == 0) {
        for (int s = 0; s < MAX_STAGES; ++s) {
            mbar_init(bar_full + 8 * s, 1);
            mbar_init(bar_empty + 8 * s, 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(bar_acc_full + 8 * b, 1);
            mbar_init(bar_acc_empty + 8 * b, 128);
        }
        fence_barrier_init();
        tma_prefetch_desc(&tmA);
        tma_prefetch_desc(&tmB);
        tma_prefetch_desc(&tmY);
        // the first 256 KiB of this CTA's weights are requested into L2 while the kernel before this
        // one drains (an HBM-bound call whose x is a few KiB has nothing else to wait for)
        const int ahead = min(n_kb, static_cast<int>((256u * 1024u) / (static_cast<uint32_t>(nu) * 128u)));
        const int first_col = unit_col(0);
        for (int kb = 0; kb < ahead; ++kb) tma_prefetch_l2_2d(&tmB, kb * 64, first_col);
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(const_cast<uint32_t*>(tmem_slot)), TMEM_COLS);
        tmem_relinquish();
    }
    pdl_wait();
    if (tid == 0) *abort_word = (*reinterpret_cast<volatile int*>(p.dev_status) & TIK_DEV_WAIT_EXPIRED) ? 1 : 0;
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_launch_dependents();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        // ------------------------------------------------------------ TMA producer
        if (lane == 0) {
            int s = 0;
            uint32_t use = 0;                    // how often stage s has been filled before
            for (int i = 0; i < n_my; ++i) {
                const int col0 = unit_col(i), row0 = unit_row(i);
                for (int kb = 0; kb < n_kb; kb += kps) {
                    if (*abort_word) break;
                    if (use > 0) mbar_wait(bar_empty + 8 * s, (use - 1) & 1, abort_word, p.dev_status);
                    const int ns = min(kps, n_kb - kb);
                    mbar_expect_tx(bar_full + 8 * s, slice_bytes * static_cast<uint32_t>(ns));
                    for (int sl = 0; sl < ns; ++sl) {
                        const uint32_t dst = sbase + s * stage_bytes + sl * slice_bytes;
                        tma_load_2d(dst + a_bytes, &tmB, bar_full + 8 * s, (kb + sl) * 64, col0);   // W rows past N: zeros
                        tma_load_2d(dst, &tmA, bar_full + 8 * s, (kb + sl) * 64, row0);             // x rows past T: zeros
                    }
                    if (++s == nst) {
                        s = 0;
                        ++use;
                    }
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer
        {
            const uint32_t tmem = warp_uniform(*tmem_slot);
            int s = 0;
            uint32_t use = 0;
            for (int i = 0; i < n_my; ++i) {
                const int buf = i & 1;
                const uint32_t acc_use = i >> 1;
                if (acc_use > 0) mbar_wait_warp(bar_acc_empty + 8 * buf, (acc_use - 1) & 1, abort_word, p.dev_status);
                tc_fence_after();
                for (int kb = 0; kb < n_kb; kb += kps) {
                    if (*abort_word) break;
                    mbar_wait_warp(bar_full + 8 * s, use & 1, abort_word, p.dev_status);
                    tc_fence_after();
                    const uint32_t a0 = sbase + s * stage_bytes, b0 = a0 + a_bytes;
                    const int ns = min(kps, n_kb - kb);
                    for (int sl = 0; sl < ns; ++sl)
                        mma_ss_chain4(tmem + buf * 256, smem_desc_sw128(a0 + sl * slice_bytes, 0, 1024),
                                      smem_desc_sw128(b0 + sl * slice_bytes, 0, 1024), idesc, (kb + sl) ? 1u : 0u);
                    mma_commit(bar_empty + 8 * s);
                    if (++s == nst) {
                        s = 0;
                        ++use;
                    }
                }
                mma_commit(bar_acc_full + 8 * buf);
            }
        }
    } else {
        // ------------------------------------------------------------ epilogue (warps 2..5)
        // As in the batched kernel: a thread per accumulator row, 64 columns at a time through a
        // swizzled staging tile and one tiled TMA store, which clips rows past T and columns past N.
        const int quarter = warp & 3;
        const int row = m64 ? quarter * 16 + (lane & 15) : quarter * 32 + lane;
        uint32_t piece = 0;
        for (int i = 0; i < n_my; ++i) {
            const int buf = i & 1;
            mbar_wait(bar_acc_full + 8 * buf, (i >> 1) & 1, abort_word, p.dev_status);
            tc_fence_after();
            const int col0 = unit_col(i), row0 = unit_row(i);
            const uint32_t taddr = tmem + (static_cast<uint32_t>(quarter * 32) << 16) + buf * 256;
#pragma unroll 1
            for (int q = 0; q < nu / 64; ++q, ++piece) {
                if (col0 + 64 * q >= p.N) break;
                uint32_t v[64];
                tmem_ld32(taddr + 64 * q, *reinterpret_cast<uint32_t(*)[32]>(&v[0]));
                tmem_ld32(taddr + 64 * q + 32, *reinterpret_cast<uint32_t(*)[32]>(&v[32]));
                tmem_wait_ld();
                uint8_t* stg = smem + OFF_STG + (piece & 1) * lin::STG_BYTES;
                if (warp == 2 && lane == 0) tma_store_wait_read1();
                named_bar_sync(1, 128);
                if (!m64 || lane < 16)
#pragma unroll
                for (int c16 = 0; c16 < 8; ++c16) {
                    const uint4 val = make_uint4(
                        pack_bf16x2(__uint_as_float(v[8 * c16]), __uint_as_float(v[8 * c16 + 1])),
                        pack_bf16x2(__uint_as_float(v[8 * c16 + 2]), __uint_as_float(v[8 * c16 + 3])),
                        pack_bf16x2(__uint_as_float(v[8 * c16 + 4]), __uint_as_float(v[8 * c16 + 5])),
                        pack_bf16x2(__uint_as_float(v[8 * c16 + 6]), __uint_as_float(v[8 * c16 + 7])));
                    *reinterpret_cast<uint4*>(stg + row * 128 + ((c16 ^ (row & 7)) << 4)) = val;
                }
                fence_proxy_async_smem();
                named_bar_sync(1, 128);
                if (warp == 2 && lane == 0) {
                    tma_store_2d(&tmY, smem_u32(stg), col0 + 64 * q, row0);
                    tma_store_commit();
                }
            }
            tc_fence_before();
            mbar_arrive(bar_acc_empty + 8 * buf);
        }
        if (warp == 2 && lane == 0) tma_store_wait_read();
    }

    if (*abort_word) {   // let copies and MMAs in flight finish before shared memory and TMEM are released
        const unsigned long long t0 = globaltimer_ns();
        while (globaltimer_ns() - t0 < 1000000ull) {
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem, TMEM_COLS);
}

static cudaError_t launch_linear_unit(const CUtensorMap& tmA, const CUtensorMap& tmB, const CUtensorMap& tmY,
                                      const LinearParams& p, cudaStream_t stream) {
    static DeviceOnce configured;
    cudaError_t e = configured.run([&]() {
        return cudaFuncSetAttribute(linear_unit_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    static_cast<int>(linu::ALLOC));
    });
    if (e != cudaSuccess) return e;
    const int grid = p.nunit < p.sm_count ? p.nunit : p.sm_count;
    return launch_pdl(linear_unit_kernel, dim3(grid), lin::THREADS, linu::ALLOC, stream, 1, tmA, tmB, tmY, p);
}

// ---------------------------------------------------------------------------------------------
// Calls with a narrow output (the down, q, k, v and output projections of a rollout step, and calls of some row
// tiles whose N is smaller still).  linear_unit_kernel gives such a call at most N / 64 CTAs per row tile; K is not
// split (an element is one chain), so the way to shorten the call is fewer weight rows per CTA on more SMs: r = 8,
// 16, .. 64 of them, as few as spread the call over all SMs, times one row tile.
// What bounds it is the chain of K / 16 MMAs, which is a CTA's whatever its share of the work is: ~17 clk + one
// per 128 bytes of the operands' rows in shared memory (K 18944, N 3584, 64 rows: 36.9 us, 32.9 with no copies at
// all, 16.9 with a quarter of the MMAs).  So the operand that is M (64 or 128 rows are read, whatever is staged) is
// the one whose choice reads fewer rows: the weights (M64) for few rows of x, x (M64, M128) for more.  The
// products of an element and the order of its sums are the same either way, so are the bits.
// Ring: stages of kps K slices; one TMA copy per operand and stage through a [K / 64][rows][64] view.
// linear_unit_kernel -> weights as M, W out of HBM, in a graph: T = 16: K 8960, N 1536 26.3 -> 12.2 us; K 18944, N 3584
// 52 -> 27.4; K 27648, N 5120 75 -> 46.  Weights as M -> x as M: T = 64: K 1536, N 256 5.2 -> 4.4; K 8960,
// N 1536 18.3 -> 13.4; K 3584, N 4608 10.4 -> 9.0; K 18944, N 3584 37.7 -> 34.5.  linear_unit_kernel -> x as M,
// T = 100: K 8960, N 1536 24.6 -> 19.6; K 18944, N 3584 52.8 -> 44.9; T = 300: K 1536, N 256 6.5 -> 5.3.
namespace linn {
constexpr uint32_t RING_BYTES = LINEAR_NARROW_RING;
constexpr int MAX_STAGES = 12;
constexpr uint32_t OFF_BAR = RING_BYTES + 64 * 128;      // (the M operand's read may run past its staged rows: never past this)
constexpr uint32_t BYTES = OFF_BAR + 512;
constexpr uint32_t ALLOC = BYTES + 1024;
}  // namespace linn

template <bool XM>     // the M operand: x (or its 128-row tiles), else the weights
__global__ void __launch_bounds__(lin::THREADS, 1)
linear_narrow_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX, const LinearParams p) {
    using namespace linn;
    constexpr uint32_t TMEM_COLS = 128;
    const int tid = threadIdx.x, warp = warp_uniform(tid >> 5), lane = tid & 31;
    const int r = p.nu, kps = p.kps, n_kb = p.K / 64;
    const int cu = !XM || p.ntp == 1 ? static_cast<int>(blockIdx.x) : static_cast<int>(blockIdx.x) / p.ntp;
    const int n0 = cu * r, row0 = XM ? (static_cast<int>(blockIdx.x) - cu * p.ntp) * 128 : 0;
    const int m = XM ? p.m : 64;                 // rows of the M operand
    const uint32_t w_slice = static_cast<uint32_t>(r) * 128u, x_slice = static_cast<uint32_t>(p.a_rows) * 128u;
    const uint32_t w_bytes = w_slice * static_cast<uint32_t>(kps);
    const uint32_t stage_bytes = w_bytes + x_slice * static_cast<uint32_t>(kps);
    const int nst = p.nst;
    const uint32_t idesc = mma_idesc_bf16(m, XM ? r : p.a_rows, false);

    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw_addr = smem_u32(smem_raw);
    const uint32_t pad = (1024u - (raw_addr & 1023u)) & 1023u;
    uint8_t* smem = smem_raw + pad;
    const uint32_t sbase = raw_addr + pad;
    const uint32_t bar_full = sbase + OFF_BAR;                   // MAX_STAGES barriers
    const uint32_t bar_empty = bar_full + 8 * MAX_STAGES;        // MAX_STAGES barriers
    const uint32_t bar_acc = bar_empty + 8 * MAX_STAGES;
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem + OFF_BAR + 8 * (2 * MAX_STAGES + 1));
    volatile int* abort_word = reinterpret_cast<volatile int*>(smem + OFF_BAR + 8 * (2 * MAX_STAGES + 1) + 4);

    if (tid == 0) {
        for (int s = 0; s < MAX_STAGES; ++s) {
            mbar_init(bar_full + 8 * s, 1);
            mbar_init(bar_empty + 8 * s, 1);
        }
        mbar_init(bar_acc, 1);
        fence_barrier_init();
        tma_prefetch_desc(&tmW);
        tma_prefetch_desc(&tmX);
        // the first 256 KiB of this CTA's weights on their way to L2 while the kernel before this one drains
        const int ahead = min(n_kb, static_cast<int>((256u * 1024u) / w_slice));
        for (int kb = 0; kb < ahead; kb += kps) tma_prefetch_l2_3d(&tmW, 0, n0, kb);
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(const_cast<uint32_t*>(tmem_slot)), TMEM_COLS);
        tmem_relinquish();
    }
    pdl_wait();
    if (tid == 0) *abort_word = (*reinterpret_cast<volatile int*>(p.dev_status) & TIK_DEV_WAIT_EXPIRED) ? 1 : 0;
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_launch_dependents();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        // ------------------------------------------------------------ TMA producer
        if (lane == 0) {
            int s = 0;
            uint32_t use = 0;                    // how often stage s has been filled before
            for (int kb = 0; kb < n_kb; kb += kps) {
                if (*abort_word) break;
                if (use > 0) mbar_wait(bar_empty + 8 * s, (use - 1) & 1, abort_word, p.dev_status);
                const uint32_t dst = sbase + s * stage_bytes;
                // W rows past N, x rows past T and slices past K arrive as zeros
                mbar_expect_tx(bar_full + 8 * s, stage_bytes);
                tma_load_3d(dst, &tmW, bar_full + 8 * s, 0, n0, kb);
                tma_load_3d(dst + w_bytes, &tmX, bar_full + 8 * s, 0, row0, kb);
                if (++s == nst) {
                    s = 0;
                    ++use;
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer
        {
            const uint32_t tmem = warp_uniform(*tmem_slot);
            int s = 0;
            uint32_t use = 0;
            for (int kb = 0; kb < n_kb; kb += kps) {
                if (*abort_word) break;
                mbar_wait_warp(bar_full + 8 * s, use & 1, abort_word, p.dev_status);
                tc_fence_after();
                const uint32_t w0 = sbase + s * stage_bytes, x0 = w0 + w_bytes;
                const uint32_t a0 = XM ? x0 : w0, b0 = XM ? w0 : x0, a_step = XM ? x_slice : w_slice, b_step = XM ? w_slice : x_slice;
                const int ns = min(kps, n_kb - kb);
                for (int sl = 0; sl < ns; ++sl)
                    mma_ss_chain4(tmem, smem_desc_sw128(a0 + sl * a_step, 0, 1024), smem_desc_sw128(b0 + sl * b_step, 0, 1024),
                                  idesc, (kb + sl) ? 1u : 0u);
                mma_commit(bar_empty + 8 * s);
                if (++s == nst) {
                    s = 0;
                    ++use;
                }
            }
            mma_commit(bar_acc);
        }
    } else {
        // ------------------------------------------------------------ epilogue (warps 2..5)
        // An M64 accumulator has 16 rows in each lane quarter, an M128 one 32.
        const int quarter = warp & 3;
        const uint32_t taddr = tmem + (static_cast<uint32_t>(quarter * 32) << 16);
        const int i0 = (m == 64 ? 16 : 32) * quarter, i_m = i0 + lane;      // row of the M operand
        const bool mine = m == 128 || lane < 16;
        mbar_wait(bar_acc, 0, abort_word, p.dev_status);
        tc_fence_after();
        if (XM) {                                // thread per row of x, r columns of it
            const long long row = row0 + i_m;
            const bool valid = mine && i_m < p.a_rows && row < p.T;
            __nv_bfloat16* const y = p.y + row * p.N + n0;
            if (row0 + i0 < p.T)
                for (int c0 = 0; c0 < r; c0 += 32) {
                    uint32_t v[32];
                    tmem_ld32(taddr + c0, v);
                    tmem_wait_ld();
#pragma unroll
                    for (int c = 0; c < 32; c += 8) {
                        const uint4 val = make_uint4(pack_bf16x2(__uint_as_float(v[c]), __uint_as_float(v[c + 1])),
                                                     pack_bf16x2(__uint_as_float(v[c + 2]), __uint_as_float(v[c + 3])),
                                                     pack_bf16x2(__uint_as_float(v[c + 4]), __uint_as_float(v[c + 5])),
                                                     pack_bf16x2(__uint_as_float(v[c + 6]), __uint_as_float(v[c + 7])));
                        if (valid && c0 + c < r && n0 + c0 + c < p.N) *reinterpret_cast<uint4*>(y + c0 + c) = val;
                    }
                }
        } else if (i0 < r) {                     // thread per output column, a column of the accumulator is a row of x
            const bool valid = mine && i_m < r && n0 + i_m < p.N;
            for (int c0 = 0; c0 < static_cast<int>(p.T); c0 += 32) {
                uint32_t v[32];
                tmem_ld32(taddr + c0, v);
                tmem_wait_ld();
                __nv_bfloat16* const y = p.y + static_cast<long long>(c0) * p.N + n0 + i_m;
                const int nt = min(32, static_cast<int>(p.T) - c0);
#pragma unroll
                for (int i = 0; i < 32; ++i)
                    if (valid && i < nt) y[static_cast<long long>(i) * p.N] = __float2bfloat16_rn(__uint_as_float(v[i]));
            }
        }
    }

    if (*abort_word) {   // let copies and MMAs in flight finish before shared memory and TMEM are released
        const unsigned long long t0 = globaltimer_ns();
        while (globaltimer_ns() - t0 < 1000000ull) {
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem, TMEM_COLS);
}

cudaError_t launch_linear_narrow(const CUtensorMap& tmW, const CUtensorMap& tmX, const LinearParams& p, cudaStream_t stream) {
    static DeviceOnce configured;
    cudaError_t e = configured.run([&]() {
        for (auto k : {linear_narrow_kernel<false>, linear_narrow_kernel<true>}) {
            const cudaError_t err = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(linn::ALLOC));
            if (err != cudaSuccess) return err;
        }
        return cudaSuccess;
    });
    if (e != cudaSuccess) return e;
    return launch_pdl(p.m ? linear_narrow_kernel<true> : linear_narrow_kernel<false>, dim3(static_cast<unsigned>(p.nunit)),
                      lin::THREADS, linn::ALLOC, stream, 1, tmW, tmX, p);
}

// pair = true: tmB must have a box of 128 rows (each CTA of a pair stages half of a step's)
cudaError_t launch_linear(const CUtensorMap& tmA, const CUtensorMap& tmB, const CUtensorMap& tmY,
                          const LinearParams& p, bool pair, cudaStream_t stream) {
    if (p.T <= 0) return cudaSuccess;
    if (!pair) return launch_linear_unit(tmA, tmB, tmY, p, stream);
    static DeviceOnce configured;     // the opt-in belongs to the (function, device) pair
    cudaError_t e = configured.run([&]() {
        return cudaFuncSetAttribute(linear_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(lin::ALLOC));
    });
    if (e != cudaSuccess) return e;
    const long long ntile = (p.T + 127) / 128;
    const long long nband = (ntile + lin::BAND - 1) / lin::BAND;
    long long grid = nband * lin::BAND * p.nsuper;               // even: BAND is
    if (p.unit_mode) {
        const int slots = p.sm_count / 2;
        grid = 2ll * (slots < p.nunit ? slots : p.nunit);
    }
    return launch_pdl(linear_kernel, dim3(static_cast<unsigned>(grid)), lin::THREADS, lin::ALLOC, stream, 2, tmA, tmB, tmY, p);
}

}  // namespace tik
