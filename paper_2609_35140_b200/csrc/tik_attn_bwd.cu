// Backward of the packed causal GQA attention (policy-update backward) for sm_100a.
//
// Deterministic by construction: no atomics and no split accumulation.  Two launches of one
// kernel body recompute the score tiles and differ in which side stays resident:
//   DQ  mode: a CTA owns one 128-row query tile of one (sequence, head) and walks the KV tiles
//             0..i:      S = Q_i K_j^T, dP = dO_i V_j^T, dS = P o (dP - delta),
//             dQ_i += dS K_j                                     (accumulator in TMEM)
//             and then the same for the CTA's next query head of that KV head: its loads start with the last
//             score products, its first steps run under the epilogue of the head before
//   DKV mode: a CTA owns one 128-row KV tile of one (sequence, KV head) and walks the query
//             tiles i >= j of the G query heads of that KV head, one after the other:
//             S^T = K_j Q_i^T, dP^T = V_j dO_i^T, dV_j += P^T dO_i, dK_j += dS^T Q_i
// with P = exp2(S c - lse log2 e) from the forward's log-sum-exp and delta = rowsum(dO o O)
// (a small kernel of its own).  All products run on tcgen05 at full width (128 streamed rows): the two
// score products with both operands in shared memory (TMA, 128B swizzle), the gradient products with
// the bf16 weights P / dS read from TMEM, written there in place of the fp32 scores they came from.
// One TMA warp, one MMA-issuing warp (DQ: two), and sixteen element-wise warps, four threads per tile row
// with 32 columns each, all on the same step.  A thread writes its 32 weights over the first 16 of its own
// 32 score columns, so no other thread's columns are touched.
//
// DKV: S and dP are one TMEM tile each (with the two accumulators TMEM is full), and what overlaps
// is the two halves of the element-wise work: P needs S only, so while dV += P^T dO and the next S run, dP
// turns into dS, and while dK += dS^T Q and the next dP run, the next P is computed.  Issue order of a step:
// dV(t), S(t+1), dK(t), dP(t+1).  (Before, a step was two halves of 64 streamed rows whose score
// products are bound by shared-memory reads of the 128-row operand: a chain of eight took 554 clk
// where the full-width one takes 627.)  dK/dV pass of 9001 + 16384 tokens (32/8 heads) 5.8 -> 4.35 ms at full
// clocks; whole backward of 2 x 4000 tokens 816 -> 775 us, 10 x 1200 532 -> 510, 4 x 8000 (4/1 heads, d 64) 538
// -> 522; two sequences of 128 tokens (d 64), a chain of single steps, 13.6 -> 14.0.
// Every wait is bounded and raises TIK_DEV_WAIT_EXPIRED instead of hanging.
#include "tik_core.cuh"
#include "tik_internal.h"
#include "tik_ptx.cuh"

namespace tik {

enum { BWD_DQ = 0, BWD_DKV = 1 };
// warp 0 TMA, warp 1 MMA (DQ: the score products), warps 2-17 element-wise (four threads per tile
// row), warp 18 DQ: the gradient products
constexpr int BWD_THREADS = 608;
// Streamed tiles: three stages of c1 (DQ: K tiles, DKV: Q tiles, in use until the second gradient
// product of their step) and two of c2 (DQ: V, DKV: dO).
constexpr int C1_STAGES = 3, C2_STAGES = 2;

template <int D, int MODE>
struct BwdSmem {
    static constexpr uint32_t ATOM = 128 * 128;           // 128 rows x 64 bf16
    static constexpr uint32_t TILE = (D / 64) * ATOM;
    static constexpr uint32_t OFF_R = 0;                  // two resident row-side tiles
    static constexpr uint32_t OFF_C1 = 2 * TILE;
    static constexpr uint32_t OFF_C2 = OFF_C1 + C1_STAGES * TILE;
    static constexpr uint32_t OFF_BAR = OFF_C2 + C2_STAGES * TILE;
    static constexpr uint32_t OFF_SC = OFF_BAR + 160;     // DKV: [2 buffers][-l2 x 128 | -delta x 128] floats of the columns
    static constexpr uint32_t BYTES = OFF_SC + ((MODE == 0) ? 0 : 2 * 2 * 128 * 4);      // base must be 1 KiB aligned
};

template <int D, int MODE>
__global__ void __launch_bounds__(BWD_THREADS, 1)
attn_bwd_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmDO,
                const BwdParams p) {
    using L = BwdSmem<D, MODE>;
    constexpr int NATOM = D / 64;
    constexpr uint32_t TMEM_COLS = 512;
    // TMEM columns.  DKV: S, dP, two accumulators.  DQ: S, two dP tiles used alternately, one accumulator.
    constexpr uint32_t COL_T1 = 0, COL_T2 = 128;
    constexpr uint32_t COL_T2B = 256;                                   // DQ only
    constexpr uint32_t COL_A1 = (MODE == BWD_DQ) ? 384 : 256, COL_A2 = 256 + D;
    constexpr uint32_t IDESC_SC = mma_idesc_bf16(128, 128, false);
    constexpr uint32_t IDESC_OUT = mma_idesc_bf16(128, D, true);
    const int tid = threadIdx.x, warp = warp_uniform(tid >> 5), lane = tid & 31;

    // Launch order and dependencies: delta kernel, dK/dV grid, dQ grid, each with a programmatic
    // dependency.  The dK/dV grid waits for the delta kernel here.  The dQ grid starts once every CTA
    // of the dK/dV grid has passed that wait and holds its tensor memory (so everything it reads is complete) and must not wait
    // for that grid: its CTAs fill the SMs that the dK/dV grid's last CTAs leave idle.  Only its last
    // block waits for the dK/dV grid, at its end, so that the dQ grid completes after it (and no dQ CTA
    // releases its dependents early).  Two sequences of 96 and 160 tokens (4/1 heads, d 64), forward and
    // backward: 32.2 -> 27.6 us.
    if (MODE == BWD_DKV) pdl_wait();
    const bool last_block = MODE == BWD_DQ && blockIdx.x == gridDim.x - 1 && blockIdx.y == gridDim.y - 1 &&
                            blockIdx.z == gridDim.z - 1;

    // ---------------------------------------------------------------- work item
    const int seq = blockIdx.z;
    // (around L1 in the dQ grid, here and for lse and delta below: no wait of its own precedes the reads, and these
    // buffers are rewritten from call to call)
    auto cu = [&](int i) { return MODE == BWD_DQ ? __ldcg(&p.cu_seqlens[i]) : p.cu_seqlens[i]; };
    const int tok0 = cu(seq);
    const int len = cu(seq + 1) - tok0;
    if (len <= 0) {
        if (last_block) pdl_wait();
        return;
    }
    const int nq = (len + 127) / 128;                      // tiles of the sequence (query and KV alike)
    int own, head = 0, kvh, n_steps, n_heads = 1;
    if (MODE == BWD_DQ) {
        // query tiles from the heaviest down; heads fastest or one after the other: bwd_dq_choose.  (The dK/dV grid with
        // its heads fastest is no faster.)
        const int group = p.dq_tiles_first ? blockIdx.y : blockIdx.x;
        own = p.dq_tiles_first ? gridDim.x - 1 - blockIdx.x : gridDim.y - 1 - blockIdx.y;
        if (own >= nq) return;                             // (never the last block: its tile is 0)
        kvh = group / p.dq_groups;
        const int g0 = (group - kvh * p.dq_groups) * p.dq_heads;
        head = kvh * p.G + g0;                             // the first of the CTA's heads, taken one after the other
        n_heads = min(p.dq_heads, p.G - g0);
        n_steps = own + 1;                                 // KV tiles 0..own, for each of them
    } else {
        own = blockIdx.x;                                  // KV tile, heaviest first
        if (own >= nq) return;
        kvh = blockIdx.y;
        n_steps = p.G * (nq - own);                        // (g, query tile i >= own), g outermost
    }
    const int n_steps_v = n_steps;       // (the issuing warps shadow it with a warp-uniform copy)
    // DKV: tile and query head of a step, walked one step at a time
    struct Walk {
        int tile, head;
    };
    auto walk_on = [&](Walk& w) {
        if (++w.tile == nq) {
            w.tile = own;
            ++w.head;
        }
    };
    const Walk walk_start = {own, kvh * p.G};

    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = smem_raw;
    const uint32_t sbase = smem_u32(smem_raw);
    if (sbase & 1023u) {     // the swizzled tiles need a 1 KiB aligned base: refuse to run otherwise
        if (tid == 0) atomicOr(p.dev_status, TIK_DEV_WAIT_EXPIRED);
        if (last_block) pdl_wait();
        return;
    }
    const uint32_t sR1 = sbase + L::OFF_R, sR2 = sR1 + L::TILE;
    const uint32_t bar0 = sbase + L::OFF_BAR;
    const uint32_t bar_r = bar0;                 // row-side tiles landed
    const uint32_t bar_c1full = bar0 + 8;        // [3] c1 tile landed
    const uint32_t bar_c1empty = bar0 + 32;      // [3] the gradient product that read it is done
    const uint32_t bar_c2full = bar0 + 56;       // [2] c2 tile landed
    const uint32_t bar_c2empty = bar0 + 72;      // [2] its last product (DQ: dP, DKV: dV) is done
    const uint32_t bar_s = bar0 + 88;            // S of a step ready (DQ: S and dP)
    const uint32_t bar_aux = bar0 + 96;          // DQ: S is in registers (16 warps); DKV: dP of a step ready
    const uint32_t bar_p = bar0 + 104;           // DQ: dS of a step written (16 warps); DKV: P written (16 warps)
    const uint32_t bar_ds = bar0 + 112;          // DKV: dS written (16 warps)
    const uint32_t bar_acc = bar0 + 120;         // all MMAs done
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem + L::OFF_BAR + 128);
    volatile int* abort_word = reinterpret_cast<volatile int*>(smem + L::OFF_BAR + 132);
    const uint32_t bar_gdone = bar0 + 136;       // [2] DQ: the gradient product that read a dS tile is done
    const uint32_t bar_rempty = bar0 + 152;      // DQ: a head's last score products have read the row-side tiles
    float* sc_base = reinterpret_cast<float*>(smem + L::OFF_SC);

    if (tid == 0) {
        mbar_init(bar_r, 1);
        for (int i = 0; i < C1_STAGES; ++i) {
            mbar_init(bar_c1full + 8 * i, 1);
            mbar_init(bar_c1empty + 8 * i, 1);
        }
        for (int i = 0; i < C2_STAGES; ++i) {
            mbar_init(bar_c2full + 8 * i, 1);
            mbar_init(bar_c2empty + 8 * i, 1);
        }
        mbar_init(bar_s, 1);
        mbar_init(bar_aux, MODE == BWD_DQ ? 16 : 1);
        mbar_init(bar_p, 16);
        mbar_init(bar_ds, 16);
        mbar_init(bar_acc, 1);
        mbar_init(bar_gdone, 1);
        mbar_init(bar_gdone + 8, 1);
        mbar_init(bar_rempty, 1);
        *abort_word = (*reinterpret_cast<volatile int*>(p.dev_status) & TIK_DEV_WAIT_EXPIRED) ? 1 : 0;
        fence_barrier_init();
        tma_prefetch_desc(&tmQ);
        tma_prefetch_desc(&tmK);
        tma_prefetch_desc(&tmV);
        tma_prefetch_desc(&tmDO);
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(const_cast<uint32_t*>(tmem_slot)), TMEM_COLS);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (MODE == BWD_DKV) pdl_launch_dependents();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        // ------------------------------------------------------------ TMA producer
        if (lane == 0) {
            const int row_own = tok0 + 128 * own;
            auto load_rows = [&](int h) {
                mbar_expect_tx(bar_r, 2 * L::TILE);
                for (int a = 0; a < NATOM; ++a) {
                    tma_load_3d(sR1 + a * L::ATOM, MODE == BWD_DQ ? &tmQ : &tmK, bar_r, a * 64, h, row_own);
                    tma_load_3d(sR2 + a * L::ATOM, MODE == BWD_DQ ? &tmDO : &tmV, bar_r, a * 64, h, row_own);
                }
            };
            load_rows(MODE == BWD_DQ ? head : kvh);
            const CUtensorMap* tm1 = MODE == BWD_DQ ? &tmK : &tmQ;
            const CUtensorMap* tm2 = MODE == BWD_DQ ? &tmV : &tmDO;
            Walk w = walk_start;
            const int n_all = n_steps * n_heads;
            int tile = 0, hl = 0;                // DQ: KV tile and head of the CTA
            for (int t = 0; t < n_all; ++t) {
                if (*abort_word) break;          // a wait expired somewhere: stop issuing copies
                const int row = tok0 + 128 * (MODE == BWD_DQ ? tile : w.tile), h = MODE == BWD_DQ ? kvh : w.head;
                walk_on(w);
                const int s1 = t % C1_STAGES, s2 = t % C2_STAGES;
                if (t >= C1_STAGES) mbar_wait(bar_c1empty + 8 * s1, (t / C1_STAGES - 1) & 1, abort_word, p.dev_status);
                mbar_expect_tx(bar_c1full + 8 * s1, L::TILE);
                for (int a = 0; a < NATOM; ++a)
                    tma_load_3d(sbase + L::OFF_C1 + s1 * L::TILE + a * L::ATOM, tm1, bar_c1full + 8 * s1, a * 64, h, row);
                if (t >= C2_STAGES) mbar_wait(bar_c2empty + 8 * s2, (t / C2_STAGES - 1) & 1, abort_word, p.dev_status);
                mbar_expect_tx(bar_c2full + 8 * s2, L::TILE);
                for (int a = 0; a < NATOM; ++a)
                    tma_load_3d(sbase + L::OFF_C2 + s2 * L::TILE + a * L::ATOM, tm2, bar_c2full + 8 * s2, a * 64, h, row);
                // the next head's rows, behind its first KV tile (whose stages are free before the rows are)
                if (MODE == BWD_DQ) {
                    if (tile == 0 && hl > 0) {
                        mbar_wait(bar_rempty, (hl - 1) & 1, abort_word, p.dev_status);
                        if (*abort_word) break;
                        load_rows(head + hl);
                    }
                    if (++tile == n_steps) {
                        tile = 0;
                        ++hl;
                    }
                }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer
        const uint32_t tmem = warp_uniform(*tmem_slot);
        const int n_steps = warp_uniform(n_steps_v);
        if (MODE == BWD_DKV) mbar_wait_warp(bar_r, 0, abort_word, p.dev_status);
        const uint64_t dr1 = smem_desc_sw128(sR1, 0, 1024), dr2 = smem_desc_sw128(sR2, 0, 1024);
        auto c1_addr = [&](int t) { return sbase + L::OFF_C1 + (t % C1_STAGES) * L::TILE; };
        auto c2_addr = [&](int t) { return sbase + L::OFF_C2 + (t % C2_STAGES) * L::TILE; };
        auto wait_c1 = [&](int t) {
            mbar_wait_warp(bar_c1full + 8 * (t % C1_STAGES), (t / C1_STAGES) & 1, abort_word, p.dev_status);
        };
        auto wait_c2 = [&](int t) {
            mbar_wait_warp(bar_c2full + 8 * (t % C2_STAGES), (t / C2_STAGES) & 1, abort_word, p.dev_status);
        };
        auto score = [&](uint32_t col, uint64_t dr, uint32_t c) {      // [col ...] = R C^T
            if (D == 128) mma_ss_chain8_fresh(tmem + col, dr, smem_desc_sw128(c, 0, 1024), IDESC_SC);
            else mma_ss_chain4_fresh(tmem + col, dr, smem_desc_sw128(c, 0, 1024), IDESC_SC);
        };
        if (MODE == BWD_DQ) {
            // only dS feeds a gradient product, so the score tile S is free again as soon as the
            // element-wise threads hold it in registers, and dP / dS alternate between two tiles.  Both
            // score products of step t+1 are issued while the element-wise work of step t runs, the
            // gradient product of step t right behind them.
            const int n_all = n_steps * warp_uniform(n_heads);
            for (int t = 0, tile = 0, hl = 0; t < n_all; ++t) {
                if (*abort_word) break;
                if (tile == 0) mbar_wait_warp(bar_r, hl & 1, abort_word, p.dev_status);
                wait_c1(t);
                wait_c2(t);
                if (t > 0) mbar_wait_warp(bar_aux, (t - 1) & 1, abort_word, p.dev_status);   // S of step t-1 is in registers
                // the dP tile of this parity held dS of step t-2 (the two issuing warps have no
                // common program order, so its gradient product is waited for)
                if (t > 1) mbar_wait_warp(bar_gdone + 8 * (t & 1), ((t - 2) >> 1) & 1, abort_word, p.dev_status);
                tc_fence_after();
                score(COL_T1, dr1, c1_addr(t));
                score((t & 1) ? COL_T2B : COL_T2, dr2, c2_addr(t));
                mma_commit(bar_s);
                mma_commit(bar_c2empty + 8 * (t % C2_STAGES));      // the V stage is done with
                if (++tile == n_steps) {
                    tile = 0;
                    if (++hl < n_heads) mma_commit(bar_rempty);
                }
            }
        } else {
            // MMAs issued by one warp execute in order: S(t+1) overwrites P(t) only after dV(t) has read it,
            // dP(t+1) overwrites dS(t) only after dK(t)
            wait_c1(0);
            tc_fence_after();
            score(COL_T1, dr1, c1_addr(0));
            mma_commit(bar_s);
            wait_c2(0);
            score(COL_T2, dr2, c2_addr(0));
            mma_commit(bar_aux);
            for (int t = 0; t < n_steps; ++t) {
                if (*abort_word) break;
                const bool more = t + 1 < n_steps;
                mbar_wait_warp(bar_p, t & 1, abort_word, p.dev_status);
                tc_fence_after();
                mma_ts_chain8_blocks(tmem + COL_A2, tmem + COL_T1, smem_desc_sw128(c2_addr(t), L::ATOM, 1024), IDESC_OUT, t > 0 ? 1u : 0u);
                mma_commit(bar_c2empty + 8 * (t % C2_STAGES));
                if (more) {
                    wait_c1(t + 1);
                    score(COL_T1, dr1, c1_addr(t + 1));
                    mma_commit(bar_s);
                }
                mbar_wait_warp(bar_ds, t & 1, abort_word, p.dev_status);
                tc_fence_after();
                mma_ts_chain8_blocks(tmem + COL_A1, tmem + COL_T2, smem_desc_sw128(c1_addr(t), L::ATOM, 1024), IDESC_OUT, t > 0 ? 1u : 0u);
                mma_commit(bar_c1empty + 8 * (t % C1_STAGES));
                if (more) {
                    wait_c2(t + 1);
                    score(COL_T2, dr2, c2_addr(t + 1));
                    mma_commit(bar_aux);
                }
            }
            mma_commit(bar_acc);
        }
        __syncwarp();
    } else if (warp == 18) {
        // ------------------------------------------------------------ DQ: gradient-product issuer
        // A warp of its own, so that its waits and commits do not stand between two score products.
        if (MODE == BWD_DQ) {
            const uint32_t tmem = warp_uniform(*tmem_slot);
            const int n_steps = warp_uniform(n_steps_v);
            const int n_all = n_steps * warp_uniform(n_heads);
            for (int t = 0, tile = 0; t < n_all; ++t) {
                if (*abort_word) break;
                // (a head's first dS is there only after every warp has read the previous head's accumulator)
                mbar_wait_warp(bar_p, t & 1, abort_word, p.dev_status);
                tc_fence_after();
                // A = dS: every thread left its 32 columns' bf16 pairs in the first 16 columns of
                // its own 32-column block, so the eight 16-key steps sit at 0, 8, 32, 40, ...
                mma_ts_chain8_blocks(tmem + COL_A1, tmem + ((t & 1) ? COL_T2B : COL_T2),
                                     smem_desc_sw128(sbase + L::OFF_C1 + (t % C1_STAGES) * L::TILE, L::ATOM, 1024),
                                     IDESC_OUT, tile > 0 ? 1u : 0u);
                mma_commit(bar_c1empty + 8 * (t % C1_STAGES));
                mma_commit(bar_gdone + 8 * (t & 1));
                if (++tile == n_steps) {
                    tile = 0;
                    mma_commit(bar_acc);
                }
            }
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------------ element-wise warps
        const int quarter = warp & 3;                      // TMEM lane quarter of this warp
        const int r = quarter * 32 + lane;                 // tile row == TMEM lane
        const int cq = (warp - 2) >> 2;                    // which 32 of the tile's 128 columns this thread works on
        const int et = (warp - 2) * 32 + lane;             // 0..511
        const uint32_t tlane = tmem + (static_cast<uint32_t>(quarter * 32) << 16);
        const int row_abs = 128 * own + r;                 // position of this row in the sequence
        const float c = p.c;                               // scale * log2(e)
        auto fetch_row = [&](int h, float& l2, float& dl) {
            l2 = 0.0f;
            dl = 0.0f;
            if (row_abs < len) {
                const long long idx = (static_cast<long long>(tok0) + row_abs) * p.Hq + h;
                l2 = __fmul_rn(__ldcg(&p.lse[idx]), LOG2E_F);
                dl = __ldcg(&p.delta[idx]);
            }
        };
        // DKV: the scalars belong to the columns (query rows of the streamed tile).  Threads 0..127 fetch
        // those of the next step's columns; they reach the others through shared memory
        // (double-buffered, stored negated and as two arrays, so that neighbouring columns' values load
        // as 16-byte vectors, ready for the two-wide arithmetic).
        auto fetch_col = [&](const Walk& w, bool any, float& l2, float& dl) {
            l2 = 0.0f;
            dl = 0.0f;
            const int qa = 128 * w.tile + et;
            if (any && et < 128 && qa < len) {
                const long long idx = (static_cast<long long>(tok0) + qa) * p.Hq + w.head;
                l2 = __fmul_rn(p.lse[idx], LOG2E_F);
                dl = __ldcg(&p.delta[idx]);
            }
        };
        auto pass_col = [&](int t, float l2, float dl) {
            if (et < 128) {
                sc_base[(t & 1) * 256 + et] = -l2;
                sc_base[(t & 1) * 256 + 128 + et] = -dl;
            }
            named_bar_sync(1, 512);
        };
        // fp32 accumulators -> bf16 rows
        auto epilogue = [&](int hd, uint32_t phase) {
            mbar_wait(bar_acc, phase, abort_word, p.dev_status);
            tc_fence_after();
            const bool valid = row_abs < len;
            const long long tok = static_cast<long long>(tok0) + row_abs;
            __nv_bfloat16* out1 = (MODE == BWD_DQ) ? p.dq + (tok * p.Hq + hd) * D : p.dk + (tok * p.Hkv + kvh) * D;
            __nv_bfloat16* out2 = p.dv + (tok * p.Hkv + kvh) * D;
            // blocks of 32 columns of dQ (DKV: of dK, then dV) over the four threads of a row
#pragma unroll 1
            for (int u = cq; u < (MODE == BWD_DKV ? 2 : 1) * (D / 32); u += 4) {
                const bool second = u >= D / 32;
                const int col = 32 * (second ? u - D / 32 : u);
                __nv_bfloat16* out = (second ? out2 : out1) + col;
                const float osc = second ? 1.0f : p.scale;             // dQ, dK carry the softmax scale; dV does not
                uint32_t v[32];
                tmem_ld32(tlane + (second ? COL_A2 : COL_A1) + col, v);
                tmem_wait_ld();
                if (valid) {
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        reinterpret_cast<uint4*>(out)[i] = make_uint4(
                            pack_bf16x2(__fmul_rn(__uint_as_float(v[8 * i]), osc), __fmul_rn(__uint_as_float(v[8 * i + 1]), osc)),
                            pack_bf16x2(__fmul_rn(__uint_as_float(v[8 * i + 2]), osc), __fmul_rn(__uint_as_float(v[8 * i + 3]), osc)),
                            pack_bf16x2(__fmul_rn(__uint_as_float(v[8 * i + 4]), osc), __fmul_rn(__uint_as_float(v[8 * i + 5]), osc)),
                            pack_bf16x2(__fmul_rn(__uint_as_float(v[8 * i + 6]), osc), __fmul_rn(__uint_as_float(v[8 * i + 7]), osc)));
                }
            }
        };
        if (MODE == BWD_DQ) {
            float row_l2, row_dl, next_l2 = 0.0f, next_dl = 0.0f;
            fetch_row(head, row_l2, row_dl);
            int t = 0;                           // steps so far, of all heads
            for (int hl = 0; hl < n_heads; ++hl) {
                if (hl + 1 < n_heads) fetch_row(head + hl + 1, next_l2, next_dl);
                const float nl2 = -row_l2, ndl = -row_dl;
                for (int tile = 0; tile < n_steps; ++tile, ++t) {
                    mbar_wait(bar_s, t & 1, abort_word, p.dev_status);
                    tc_fence_after();
                    const uint32_t t2 = tlane + ((t & 1) ? COL_T2B : COL_T2) + 32 * cq;
                    uint32_t s_[32], d_[32];
                    tmem_ld32(tlane + COL_T1 + 32 * cq, s_);
                    tmem_ld32(t2, d_);
                    tmem_wait_ld();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar_aux);            // S is in registers: the next QK^T may overwrite it
                    uint32_t dk_[16];
                    if (tile != own) {               // off the diagonal nothing is masked: two-wide, no compares
#pragma unroll
                        for (int i = 0; i < 32; i += 2) {
                            float p0, p1, ds0, ds1;
                            bwd_pds_x2(__uint_as_float(s_[i]), __uint_as_float(s_[i + 1]), __uint_as_float(d_[i]),
                                       __uint_as_float(d_[i + 1]), c, nl2, nl2, ndl, ndl, p0, p1, ds0, ds1);
                            dk_[i >> 1] = pack_bf16x2(ds0, ds1);
                        }
                    } else {
                        const int col0_abs = 128 * tile + 32 * cq;
#pragma unroll
                        for (int i = 0; i < 32; i += 2) {
                            float dsv[2];
#pragma unroll
                            for (int e = 0; e < 2; ++e) {
                                const bool masked = col0_abs + i + e > row_abs;      // key after query
                                const float pe = bwd_p(__uint_as_float(s_[i + e]), c, row_l2);
                                dsv[e] = masked ? 0.0f : bwd_ds(pe, __uint_as_float(d_[i + e]), row_dl);
                            }
                            dk_[i >> 1] = pack_bf16x2(dsv[0], dsv[1]);
                        }
                    }
                    // dS goes over the first 16 of this thread's own 32 dP columns: no other thread reads them
                    tmem_st16(t2, dk_);
                    tmem_wait_st();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar_p);
                }
                epilogue(head + hl, hl & 1);
                row_l2 = next_l2;
                row_dl = next_dl;
            }
        } else {
            float l2, dl;
            Walk here = walk_start, next = walk_start;
            fetch_col(here, true, l2, dl);
            pass_col(0, l2, dl);
            for (int t = 0; t < n_steps; ++t, here = next) {
                walk_on(next);
                fetch_col(next, t + 1 < n_steps, l2, dl);                  // in flight during this step
                const float* csc = sc_base + (t & 1) * 256 + 32 * cq;      // -l2 of this thread's 32 columns; -delta at + 128
                // column cc is masked for this row when it lies in the row's past (query before key) or past
                // the end of the sequence: the diagonal tile and the sequence's last query tile only;
                // everywhere else the two-wide path runs without compares and selects
                const int col0_abs = 128 * here.tile + 32 * cq;
                const bool any_mask = here.tile == own || col0_abs + 32 > len;
                const uint32_t t1 = tlane + COL_T1 + 32 * cq, t2 = tlane + COL_T2 + 32 * cq;
                float pv[32];
                uint32_t w[16];
                mbar_wait(bar_s, t & 1, abort_word, p.dev_status);
                tc_fence_after();
                {
                    uint32_t s_[32];
                    tmem_ld32(t1, s_);
                    tmem_wait_ld();
                    if (!any_mask) {
#pragma unroll
                        for (int i = 0; i < 32; i += 4) {
                            const float4 nl = *reinterpret_cast<const float4*>(&csc[i]);
                            bwd_p_x2(__uint_as_float(s_[i]), __uint_as_float(s_[i + 1]), c, nl.x, nl.y, pv[i], pv[i + 1]);
                            bwd_p_x2(__uint_as_float(s_[i + 2]), __uint_as_float(s_[i + 3]), c, nl.z, nl.w, pv[i + 2], pv[i + 3]);
                        }
                    } else {
#pragma unroll
                        for (int i = 0; i < 32; ++i) {
                            const bool masked = (row_abs > col0_abs + i) || (col0_abs + i >= len);
                            pv[i] = masked ? 0.0f : bwd_p(__uint_as_float(s_[i]), c, -csc[i]);
                        }
                    }
                }
#pragma unroll
                for (int i = 0; i < 16; ++i) w[i] = pack_bf16x2(pv[2 * i], pv[2 * i + 1]);
                tmem_st16(t1, w);
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_p);
                mbar_wait(bar_aux, t & 1, abort_word, p.dev_status);
                tc_fence_after();
                {
                    uint32_t d_[32];
                    tmem_ld32(t2, d_);
                    tmem_wait_ld();
#pragma unroll
                    for (int i = 0; i < 32; i += 4) {
                        const float4 nd = *reinterpret_cast<const float4*>(&csc[128 + i]);
                        float ds[4];
                        bwd_ds_x2(pv[i], pv[i + 1], __uint_as_float(d_[i]), __uint_as_float(d_[i + 1]), nd.x, nd.y, ds[0], ds[1]);
                        bwd_ds_x2(pv[i + 2], pv[i + 3], __uint_as_float(d_[i + 2]), __uint_as_float(d_[i + 3]), nd.z, nd.w, ds[2], ds[3]);
                        if (any_mask) {      // (a masked column's dP may hold anything finite times zero, or not finite: select)
#pragma unroll
                            for (int e = 0; e < 4; ++e)
                                if (row_abs > col0_abs + i + e || col0_abs + i + e >= len) ds[e] = 0.0f;
                        }
                        w[i >> 1] = pack_bf16x2(ds[0], ds[1]);
                        w[(i >> 1) + 1] = pack_bf16x2(ds[2], ds[3]);
                    }
                }
                tmem_st16(t2, w);
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_ds);
                pass_col(t + 1, l2, dl);       // (the buffer was last read a step ago, before the previous barrier)
            }
            epilogue(0, 0);
        }
    }

    if (*abort_word) {   // let copies and MMAs in flight finish before shared memory and TMEM are released
        const unsigned long long t0 = globaltimer_ns();
        while (globaltimer_ns() - t0 < 1000000ull) {
        }
    }
    if (last_block) pdl_wait();
    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem, TMEM_COLS);
}

// delta[token][head] = sum_c dO * O in fp32: a warp per (token, head), lane chain then butterfly.
// HBM-bound: a warp takes eight vectors, all sixteen loads issued before the first sum (53 000 tokens x
// 28 heads x 128: 180 -> 118 us = 4.3 -> 6.5 TB/s, one vector per warp before).
constexpr int DELTA_VPW = 8;
template <int D>
__global__ void __launch_bounds__(256) bwd_delta_kernel(const __nv_bfloat16* o, const __nv_bfloat16* dout,
                                                       float* delta, long long n_vec) {
    pdl_wait();
    const long long v0 = ((static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5) * DELTA_VPW;
    const int lane = threadIdx.x & 31;
    constexpr int W = D / 64;                               // 32-bit words per lane (4 or 2 elements)
    uint32_t ow[DELTA_VPW][W], dw[DELTA_VPW][W];
#pragma unroll
    for (int j = 0; j < DELTA_VPW; ++j) {
        if (v0 + j < n_vec) {
            const __nv_bfloat16* op = o + (v0 + j) * D + 2 * W * lane;
            const __nv_bfloat16* dp = dout + (v0 + j) * D + 2 * W * lane;
            if (W == 2) {
                const uint2 a = *reinterpret_cast<const uint2*>(op), b = *reinterpret_cast<const uint2*>(dp);
                ow[j][0] = a.x, ow[j][W - 1] = a.y, dw[j][0] = b.x, dw[j][W - 1] = b.y;
            } else {
                ow[j][0] = *reinterpret_cast<const uint32_t*>(op);
                dw[j][0] = *reinterpret_cast<const uint32_t*>(dp);
            }
        } else {
#pragma unroll
            for (int e = 0; e < W; ++e) ow[j][e] = dw[j][e] = 0;
        }
    }
    float mine = 0.0f;                                      // lane j keeps vector j's sum
#pragma unroll
    for (int j = 0; j < DELTA_VPW; ++j) {
        float part = 0.0f;
#pragma unroll
        for (int e = 0; e < W; ++e) {                       // bf16 -> fp32 is exact
            part = __fmaf_rn(__uint_as_float(dw[j][e] << 16), __uint_as_float(ow[j][e] << 16), part);
            part = __fmaf_rn(__uint_as_float(dw[j][e] & 0xffff0000u), __uint_as_float(ow[j][e] & 0xffff0000u), part);
        }
        part = hn_warp_total(part);
        if (lane == j) mine = part;
    }
    if (lane < DELTA_VPW && v0 + lane < n_vec) delta[v0 + lane] = mine;
    pdl_launch_dependents();       // (at the end: the rule in tik_ptx.cuh)
}

template <int D, int MODE>
static cudaError_t launch_bwd_t(dim3 grid, const CUtensorMap& tmQ, const CUtensorMap& tmK, const CUtensorMap& tmV,
                                const CUtensorMap& tmDO, const BwdParams& p, cudaStream_t stream) {
    auto kern = attn_bwd_kernel<D, MODE>;
    static DeviceOnce configured;     // the opt-in belongs to the (function, device) pair
    {
        cudaError_t e = configured.run([&]() {
            return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        static_cast<int>(BwdSmem<D, MODE>::BYTES));
        });
        if (e != cudaSuccess) return e;
    }
    return launch_pdl(kern, grid, BWD_THREADS, BwdSmem<D, MODE>::BYTES, stream, 1, tmQ, tmK, tmV, tmDO, p);
}

cudaError_t launch_attn_bwd(int d, int max_tiles, int S, const CUtensorMap& tmQ, const CUtensorMap& tmK,
                            const CUtensorMap& tmV, const CUtensorMap& tmDO, const BwdParams& p,
                            const void* o, const void* dout, long long n_vec, cudaStream_t stream) {
    const unsigned dgrid = static_cast<unsigned>((n_vec + 8 * DELTA_VPW - 1) / (8 * DELTA_VPW));
    cudaError_t e = launch_pdl(d == 128 ? bwd_delta_kernel<128> : bwd_delta_kernel<64>, dim3(dgrid), 256, 0, stream, 1,
                               static_cast<const __nv_bfloat16*>(o), static_cast<const __nv_bfloat16*>(dout), p.delta, n_vec);
    if (e != cudaSuccess) return e;
    const dim3 gkv(max_tiles, p.Hkv, S);
    const dim3 gq = p.dq_tiles_first ? dim3(max_tiles, p.Hkv * p.dq_groups, S) : dim3(p.Hkv * p.dq_groups, max_tiles, S);
    if (d == 128) {
        e = launch_bwd_t<128, BWD_DKV>(gkv, tmQ, tmK, tmV, tmDO, p, stream);
        if (e == cudaSuccess) e = launch_bwd_t<128, BWD_DQ>(gq, tmQ, tmK, tmV, tmDO, p, stream);
    } else {
        e = launch_bwd_t<64, BWD_DKV>(gkv, tmQ, tmK, tmV, tmDO, p, stream);
        if (e == cudaSuccess) e = launch_bwd_t<64, BWD_DQ>(gq, tmQ, tmK, tmV, tmDO, p, stream);
    }
    return e;
}

}  // namespace tik
