// Decode attention for calls that leave most SMs idle: a cluster of CTAs per 2048-key chunk.
//
// With few (sequence, KV head, chunk) items the other decode kernels take as long as one CTA needs for
// one chunk: 64 KiB of keys and values per 128-key tile through one SM (~0.8 us per tile, ~14 us for a
// chunk) whatever the memory system could deliver.  Here C = 4 CTAs share a chunk.  What may be
// split without touching the contract: score columns (a key's scores are one MMA chain of their own)
// and output columns (a column of O is one chain over the keys of its own).  What may not: the chain of an
// output element over the chunk's tiles, and the order of the row sums.  So, tile by tile and pipelined:
//   1. scores: CTA r computes S = Q K^T of the tiles r, r + C, ...; four transfer warps put every score row
//      into the shared memory of all C CTAs (distributed shared memory, a remote mbarrier per tile);
//   2. softmax: a warp takes two tiles, a thread one row's half tile: 64 exponentials, its half row
//      sum, its bf16 weights.  Serial across tiles is only the recurrence of the reference maximum, over tile
//      maxima that the warps publish.  Every CTA does all of it;
//   3. values: CTA r accumulates O over all tiles in ascending order for its own D / C columns, so a CTA
//      loads a C-th of V; weights come from shared memory, and the rare rescale of O between
//      two tiles is known when the tile's weights are.
// Every chunk leaves its partial for combine_kernel, or its rows when it is the only one.
// Same tiles, same MMA chains over d and keys, same row-sum shape, same rescales, so same bits as
// every other regime.  Query rows and weights are 8-row atoms read with a zero stride between row
// groups (see tik_decode.cu); M64 MMAs suffice for G <= 8 rows.  Head size 128 only.
// Measured in a CUDA graph of back-to-back calls, keys out of HBM (one CTA per chunk -> this): one sequence, 4 KV
// heads x 7, 2000 keys 15.3 -> 13.4 us, 4321 16.9 -> 15.0, 16000 19.1 -> 17.7.
#include "tik_core.cuh"
#include "tik_internal.h"
#include "tik_ptx.cuh"

namespace tik {

// warps 0-7 softmax, 8-11 transfer, 12 TMA, 13 MMA
constexpr int DX_THREADS = 32 * 14;

constexpr int DX_D = 128;                                       // head size

struct DXSmem {
    static constexpr int D = DX_D;
    static constexpr uint32_t ATOM = 128 * 128;                  // 128 keys x 64 bf16
    static constexpr uint32_t UNIT = (D / 64) * ATOM;            // one K tile, or four tiles' V columns of this CTA
    static constexpr uint32_t NU = 4;                              // ring units (128 KiB)
    static constexpr uint32_t OFF_RING = 0;
    static constexpr uint32_t OFF_Q = NU * UNIT;                 // D / 64 atoms of 8 rows x 128 bytes
    // scores of a tile: 8 rows of 128 fp32, the row pitch 16 bytes longer so that eight rows' 16-byte
    // reads meet all banks; the tile's weights (2 atoms of 8 rows x 128 bytes) overlay them
    static constexpr uint32_t S_PITCH = 128 * 4 + 16;
    static constexpr uint32_t S_TILE = 5 * 1024;
    static constexpr uint32_t OFF_S = OFF_Q + (D / 64) * 1024;
    static constexpr uint32_t OFF_TM = OFF_S + TILES_PER_CHUNK * S_TILE;     // [16 tiles][8 rows] tile maxima
    static constexpr uint32_t OFF_AL = OFF_TM + 16 * 8 * 4;      // [16][8] rescale factors
    static constexpr uint32_t OFF_RS = OFF_AL + 16 * 8 * 4;      // [16][2][8] half row sums
    static constexpr uint32_t OFF_M = OFF_RS + 2 * 16 * 8 * 4;   // [8] last reference maximum
    static constexpr uint32_t OFF_FLAG = OFF_M + 8 * 4;          // [16] tiles before which O is rescaled
    static constexpr uint32_t OFF_TAB = OFF_FLAG + 16 * 4;       // [128] physical pages of the chunk
    static constexpr uint32_t OFF_BAR = OFF_TAB + 128 * 4;
    static constexpr uint32_t BYTES = OFF_BAR + 512;
};

__device__ __forceinline__ void st_cluster_f4(uint32_t addr, float a, float b, float c, float d) {
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}
// Bounded wait on a barrier that other CTAs of the cluster arrive on: their writes before the arrival
// are visible after it.
__device__ __forceinline__ void mbar_wait_cluster(uint32_t bar, uint32_t parity, volatile int* abort_word, int* dev_status) {
    const unsigned long long t0 = globaltimer_ns();
    for (uint32_t it = 1;; ++it) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
        if (ok) return;
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
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// A chain over 128 contraction steps of 16: A = compact 8-row atoms (64 descriptor units per 64
// columns).  QK: B atoms 16 KiB apart; PV: B rows of 64 bytes.
__device__ __forceinline__ void mma_ss_chain8_compact_k(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc) {
    asm volatile(
        "{\n\t.reg .pred p0, pt, e;\n\telect.sync _|e, 0xffffffff;\n\t.reg .b64 da, db;\n\t"
        "setp.ne.b32 p0, 0, 0;\n\tsetp.eq.b32 pt, 0, 0;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p0;\n\t"
        TIK_MMA_SS_STEP(2, 2) TIK_MMA_SS_STEP(4, 4) TIK_MMA_SS_STEP(6, 6)
        TIK_MMA_SS_STEP(64, 1024) TIK_MMA_SS_STEP(66, 1026) TIK_MMA_SS_STEP(68, 1028)
        TIK_MMA_SS_STEP(70, 1030)
        "}" ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc)
        : "memory");
}
__device__ __forceinline__ void mma_ss_chain8_compact_v32(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                                          uint32_t first_accumulate) {
    asm volatile(
        "{\n\t.reg .pred p0, pt, e;\n\telect.sync _|e, 0xffffffff;\n\t.reg .b64 da, db;\n\t"
        "setp.ne.b32 p0, %4, 0;\n\tsetp.eq.b32 pt, 0, 0;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p0;\n\t"
        TIK_MMA_SS_STEP(2, 64) TIK_MMA_SS_STEP(4, 128) TIK_MMA_SS_STEP(6, 192)
        TIK_MMA_SS_STEP(64, 256) TIK_MMA_SS_STEP(66, 320) TIK_MMA_SS_STEP(68, 384)
        TIK_MMA_SS_STEP(70, 448)
        "}" ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(first_accumulate)
        : "memory");
}
// 64-byte swizzle (rows of 32 bf16, 8-row groups of 512 bytes): the V columns of one of four CTAs
__device__ __forceinline__ uint64_t smem_desc_sw64(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    uint64_t d = 0;
    d |= static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);
    d |= static_cast<uint64_t>((lbo >> 4) & 0x3FFFu) << 16;
    d |= static_cast<uint64_t>((sbo >> 4) & 0x3FFFu) << 32;
    d |= 1ull << 46;
    d |= 4ull << 61;   // SWIZZLE_64B
    return d;
}

__global__ void __launch_bounds__(DX_THREADS, 1)
decode_cluster_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                      const __grid_constant__ CUtensorMap tmV, const __grid_constant__ AttnParams p) {
    using L = DXSmem;
    constexpr int D = DX_D, C = DECODE_CLUSTER;
    constexpr int NATOM = D / 64;
    constexpr int VC = D / C;                                  // output columns of this CTA
    constexpr uint32_t VBYTES = 128 * VC * 2;                  // one tile's V columns: a C-th of a unit
    constexpr int NU = static_cast<int>(L::NU);
    constexpr uint32_t TMEM_COLS = 512;
    constexpr int NSB = 3;                                     // score buffers of 128 columns
    constexpr uint32_t COL_O = 384;
    constexpr uint32_t IDESC_QK = mma_idesc_bf16(64, 128, false);
    constexpr uint32_t IDESC_PV = mma_idesc_bf16(64, VC, true);
    static_assert(VC == 32, "rows of 64 bytes: mma_ss_chain8_compact_v32, the 64-byte swizzle of tmV");

    const int tid = threadIdx.x, warp = warp_uniform(tid >> 5), lane = tid & 31;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = smem_raw;
    const uint32_t sbase = smem_u32(smem_raw);
    const uint32_t sRing = sbase + L::OFF_RING, sQ = sbase + L::OFF_Q, sS = sbase + L::OFF_S;
    const uint32_t bar0 = sbase + L::OFF_BAR;
    const uint32_t bar_full = bar0;              // [8] ring unit landed
    const uint32_t bar_empty = bar0 + 64;        // [8] ring unit read
    const uint32_t bar_q = bar0 + 128;
    const uint32_t bar_sfull = bar0 + 136;       // [3] scores of an own tile in a score buffer
    const uint32_t bar_sfree = bar0 + 160;       // [3] ... and read from it (4 warps)
    const uint32_t bar_tile = bar0 + 184;        // [16] score rows of a tile are in this CTA's shared memory (4 warps)
    const uint32_t bar_tm = bar0 + 312;          // [8] maxima of a softmax warp's two tiles published
    const uint32_t bar_p = bar0 + 376;           // [8] weights of a softmax warp's two tiles written
    const uint32_t bar_pv = bar0 + 440;          // PV up to a rescale, or the last one, done
    const uint32_t bar_resc = bar0 + 448;        // O rescaled
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem + L::OFF_BAR + 456);
    volatile int* abort_word = reinterpret_cast<volatile int*>(smem + L::OFF_BAR + 460);
    int* const tab = reinterpret_cast<int*>(smem + L::OFF_TAB);

    // ---------------------------------------------------------------- set-up that needs no input
    if (warp == 12) {
        if (lane == 0) {
            tma_prefetch_desc(&tmQ);
            tma_prefetch_desc(&tmK);
            tma_prefetch_desc(&tmV);
        }
        for (int i = lane; i < 57; i += 32) {
            const bool four = (i >= 20 && i < 23) || (i >= 23 && i < 39);     // sfree, tile: four warps
            mbar_init(bar0 + 8 * i, four ? 4 : 1);
        }
        fence_barrier_init();
        // rows >= G of the query atoms are never loaded
        for (uint32_t i = lane; i < NATOM * 1024 / 16; i += 32)
            reinterpret_cast<uint4*>(smem + L::OFF_Q)[i] = make_uint4(0, 0, 0, 0);
        fence_proxy_async_smem();
        __syncwarp();
    } else if (warp == 13) {
        tmem_alloc(smem_u32(const_cast<uint32_t*>(tmem_slot)), TMEM_COLS);
        tmem_relinquish();
    }
    pdl_wait();
    if (tid == 0) *abort_word = (*reinterpret_cast<volatile int*>(p.dev_status) & TIK_DEV_WAIT_EXPIRED) ? 1 : 0;

    const int seq = blockIdx.z, kvh = blockIdx.y, chunk = static_cast<int>(blockIdx.x) / C;
    const int rank = static_cast<int>(cluster_ctarank());
    const int head = kvh * p.G;
    const int tile0 = chunk * TILES_PER_CHUNK;
    if (warp == 12) {
        // the query rows and the chunk's block-table entries do not wait for the context length
        if (lane == 0) {
            mbar_expect_tx(bar_q, static_cast<uint32_t>(p.G) * 128u * NATOM);
            for (int a = 0; a < NATOM; ++a) tma_load_3d(sQ + a * 1024, &tmQ, bar_q, a * 64, head, seq);
        }
        for (int i = lane; i < (CHUNK >> p.page_shift); i += 32) {
            const int lp = ((128 * tile0) >> p.page_shift) + i;
            tab[i] = (lp < p.max_blocks) ? p.block_table[static_cast<long long>(seq) * p.max_blocks + lp] : -1;
        }
        __syncwarp();
    }
    int ctx = warp_uniform(p.ctx_lens[seq]);
    if (ctx > p.max_ctx) {
        if (tid == 0 && blockIdx.x == 0 && blockIdx.y == 0) atomicOr(p.dev_status, TIK_DEV_BAD_CONTEXT);
        ctx = p.max_ctx;
    }
    const bool idle = ctx <= 0 || chunk * CHUNK >= ctx || (sbase & 1023u) != 0;     // (the same in all CTAs of a cluster)
    if (idle) {
        if ((sbase & 1023u) != 0 && tid == 0) atomicOr(p.dev_status, TIK_DEV_WAIT_EXPIRED);
        __syncthreads();
        if (warp == 12) {
            mbar_wait(bar_q, 0, abort_word, p.dev_status);     // its copy is in flight
            if (*abort_word) {
                const unsigned long long t0 = globaltimer_ns();
                while (globaltimer_ns() - t0 < 1000000ull) {
                }
            }
        }
        __syncthreads();
        if (warp == 13) tmem_dealloc(*tmem_slot, TMEM_COLS);
        return;
    }
    const int n_tiles = min(TILES_PER_CHUNK, (ctx - 1) / 128 - tile0 + 1);
    const int nk = (n_tiles - rank + C - 1) / C;               // own score tiles rank, rank + C, ... (0 when n_tiles <= rank)
    const int nv = (n_tiles + C - 1) / C;                      // V units of C tiles
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_launch_dependents();       // the combine kernel may be scheduled behind this grid
    // Two cluster barriers: the first says that every CTA's mbarriers exist, the second that nobody
    // writes to another CTA any more (a thread arrives there after its last remote write, all wait at the end).
    cluster_arrive();
    const uint32_t tmem = warp_uniform(*tmem_slot);

    if (warp == 12) {
        // ------------------------------------------------------------ TMA: K tiles, V columns
        for (int i = lane; i < (CHUNK >> p.page_shift); i += 32) {
            int ph = tab[i];
            if ((((128 * tile0) >> p.page_shift) + i) << p.page_shift >= ctx) {
                ph = p.num_pages;       // out of range: the box is filled with zeros
            } else if (ph < 0 || ph >= p.num_pages) {
                atomicOr(p.dev_status, TIK_DEV_BAD_BLOCK);
                ph = p.num_pages;
            }
            tab[i] = ph;
        }
        __syncwarp();
        const int my = lane & (p.pages_per_tile - 1);
        const uint32_t page_row = static_cast<uint32_t>(my << p.page_shift);
        for (int n = 0; n < nk + nv; ++n) {
            if (*abort_word) break;
            const int u = n % NU;
            if (n >= NU) mbar_wait_warp(bar_empty + 8 * u, (n / NU - 1) & 1, abort_word, p.dev_status);
            const uint32_t full = bar_full + 8 * u, dst = sRing + u * L::UNIT;
            if (n < nk) {
                if (lane == 0) mbar_expect_tx(full, L::UNIT);
                __syncwarp();
                if (lane < p.pages_per_tile) {
                    const int ph = tab[((rank + n * C) << p.ppt_shift) + my];
                    for (int a = 0; a < NATOM; ++a)
                        tma_load_4d(dst + a * L::ATOM + page_row * 128u, &tmK, full, a * 64, 0, kvh, ph);
                }
            } else {
                const int t0 = (n - nk) * C, nt = min(C, n_tiles - t0);
                if (lane == 0) mbar_expect_tx(full, static_cast<uint32_t>(nt) * VBYTES);
                __syncwarp();
                if (lane < p.pages_per_tile)
                    for (int t = 0; t < nt; ++t)
                        tma_load_4d(dst + t * VBYTES + page_row * (VC * 2), &tmV, full, rank * VC, 0, kvh,
                                    tab[((t0 + t) << p.ppt_shift) + my]);
            }
        }
        __syncwarp();
        cluster_wait();
        cluster_arrive();
    } else if (warp == 13) {
        // ------------------------------------------------------------ MMA issuer (whole warp)
        cluster_wait();
        cluster_arrive();
        mbar_wait_warp(bar_q, 0, abort_word, p.dev_status);
        const uint64_t dq = smem_desc_sw128(sQ, 0, 0);      // stride 0 between 8-row groups: every group reads rows 0..7
        for (int i = 0; i < nk; ++i) {
            if (*abort_word) break;
            const int u = i % NU, b = i % NSB;
            mbar_wait_warp(bar_full + 8 * u, (i / NU) & 1, abort_word, p.dev_status);
            if (i >= NSB) mbar_wait_warp(bar_sfree + 8 * b, (i / NSB - 1) & 1, abort_word, p.dev_status);
            tc_fence_after();
            const uint64_t dk = smem_desc_sw128(sRing + u * L::UNIT, 0, 1024);
            mma_ss_chain8_compact_k(tmem + 128 * b, dq, dk, IDESC_QK);
            mma_commit(bar_sfull + 8 * b);
            mma_commit(bar_empty + 8 * u);
        }
        const volatile int* flag = reinterpret_cast<const volatile int*>(smem + L::OFF_FLAG);
        int resc = 0;
        for (int t = 0; t < n_tiles; ++t) {
            if (*abort_word) break;
            const int n = nk + t / C, u = n % NU;
            if (t % C == 0) mbar_wait_warp(bar_full + 8 * u, (n / NU) & 1, abort_word, p.dev_status);
            if (t % 2 == 0) mbar_wait_warp(bar_p + 8 * (t / 2), 0, abort_word, p.dev_status);
            if (warp_uniform(flag[t]) != 0) {
                // O of the tiles before this one is complete, then rescaled by warp 0
                mma_commit(bar_pv);
                mbar_wait_warp(bar_resc, resc & 1, abort_word, p.dev_status);
                ++resc;
            }
            tc_fence_after();
            const uint64_t dp = smem_desc_sw128(sS + t * L::S_TILE, 0, 0);
            const uint32_t v = sRing + u * L::UNIT + (t % C) * VBYTES;
            mma_ss_chain8_compact_v32(tmem + COL_O, dp, smem_desc_sw64(v, 8192, 512), IDESC_PV, t > 0 ? 1u : 0u);
            if (t % C == C - 1 || t == n_tiles - 1) mma_commit(bar_empty + 8 * u);
        }
        mma_commit(bar_pv);
    } else if (warp >= 8) {
        // ------------------------------------------------------------ transfer: scores of the own tiles to all CTAs
        // M64 accumulator: row i of the query group on lanes i and i + 8 of every quarter (row groups
        // repeat).  Warp `quarter` reads 32 columns; lanes 0-7 write columns 0..15 of them, lanes 8-15
        // columns 16..31, to the same place in every CTA.
        const int quarter = warp & 3;
        const uint32_t tlane = tmem + (static_cast<uint32_t>(quarter * 32) << 16);
        const int row = lane & 7, hi = (lane >> 3) & 1;
        const bool writer = lane < 16 && row < p.G;
        uint32_t dst[C];
#pragma unroll
        for (int k = 0; k < C; ++k)
            dst[k] = mapa_cluster(sS, static_cast<uint32_t>(k)) + row * L::S_PITCH + quarter * 128u + hi * 64u;
        const uint32_t my_bar = mapa_cluster(bar_tile, static_cast<uint32_t>(lane < C ? lane : 0));
        cluster_wait();                                        // the other CTAs' barriers exist
        for (int i = 0; i < nk; ++i) {
            const int b = i % NSB, t = rank + i * C;
            mbar_wait_warp(bar_sfull + 8 * b, (i / NSB) & 1, abort_word, p.dev_status);
            tc_fence_after();
            uint32_t sc[32];
            tmem_ld32(tlane + 128 * b + 32 * quarter, sc);
            tmem_wait_ld();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_sfree + 8 * b);
            if (writer) {
                float x[16];
                const int kmax = (ctx - 1) - 128 * (tile0 + t) - 32 * quarter - 16 * hi;     // own columns > kmax are masked
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    x[j] = __uint_as_float(hi ? sc[16 + j] : sc[j]);
                    if (j > kmax) x[j] = -CUDART_INF_F;
                }
#pragma unroll
                for (int k = 0; k < C; ++k)
#pragma unroll
                    for (int j = 0; j < 16; j += 4)
                        st_cluster_f4(dst[k] + t * L::S_TILE + 4u * j, x[j], x[j + 1], x[j + 2], x[j + 3]);
            }
            __syncwarp();
            if (lane < C) mbar_arrive_cluster(my_bar + 8 * t);
        }
        __syncwarp();
        cluster_arrive();
    } else {
        // ------------------------------------------------------------ softmax: two tiles per warp
        const int row = lane & 7, half = (lane >> 3) & 1, t = 2 * warp + (lane >> 4);
        float* const tmax = reinterpret_cast<float*>(smem + L::OFF_TM);
        float* const alphas = reinterpret_cast<float*>(smem + L::OFF_AL);
        float* const sums = reinterpret_cast<float*>(smem + L::OFF_RS);
        float* const m_last = reinterpret_cast<float*>(smem + L::OFF_M);
        volatile int* const flag = reinterpret_cast<volatile int*>(smem + L::OFF_FLAG);
        const float c = p.c;
        cluster_wait();
        if (2 * warp < n_tiles) {
            const bool live = t < n_tiles && row < p.G;
            mbar_wait_cluster(bar_tile + 8 * (2 * warp), 0, abort_word, p.dev_status);
            if (2 * warp + 1 < n_tiles) mbar_wait_cluster(bar_tile + 8 * (2 * warp + 1), 0, abort_word, p.dev_status);
            __syncwarp();
            uint32_t s[64];
            float mt = -CUDART_INF_F;
            if (live) {
                const float4* src = reinterpret_cast<const float4*>(smem + L::OFF_S + t * L::S_TILE + row * L::S_PITCH + half * 256);
                float mx[4];
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    const float4 v = src[i];
                    s[4 * i] = __float_as_uint(v.x), s[4 * i + 1] = __float_as_uint(v.y);
                    s[4 * i + 2] = __float_as_uint(v.z), s[4 * i + 3] = __float_as_uint(v.w);
                    const float m2 = fmaxf(fmaxf(v.x, v.y), fmaxf(v.z, v.w));
                    mx[i & 3] = i < 4 ? m2 : fmaxf(mx[i & 3], m2);
                }
                mt = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
            }
            mt = fmaxf(mt, __shfl_xor_sync(0xffffffffu, mt, 8));   // the other half of the row's tile
            if (half == 0) tmax[t * 8 + row] = mt;
            __syncwarp();                                          // (all scores of the two tiles are in registers)
            if (lane == 0) mbar_arrive(bar_tm + 8 * warp);
            float m_old = -CUDART_INF_F, m_new = -CUDART_INF_F;
            for (int w = 0; w <= warp; ++w) {
                if (w < warp) mbar_wait_warp(bar_tm + 8 * w, 0, abort_word, p.dev_status);
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const float mj = tmax[(2 * w + j) * 8 + row];
                    if (2 * w + j <= t) {
                        m_old = m_new;
                        m_new = softmax_next_max(m_old, mj, c);
                    }
                }
            }
            const float alpha = softmax_alpha(m_old, m_new, c);    // 0 on the chunk's first tile
            const unsigned moved = __ballot_sync(0xffffffffu, live && t > 0 && alpha != 1.0f);
            if (live) {
                const float neg_mc = -__fmul_rn(m_new, c);
                RowSum4 rs;
                rs.reset();
#pragma unroll
                for (int i = 0; i < 64; i += 8) softmax_p8(&s[i], c, neg_mc, rs, &s[i >> 1]);
                uint8_t* const atom = smem + L::OFF_S + t * L::S_TILE + half * 1024 + row * 128;
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    *reinterpret_cast<uint4*>(atom + ((i ^ row) << 4)) = make_uint4(s[4 * i], s[4 * i + 1], s[4 * i + 2], s[4 * i + 3]);
                sums[(2 * t + half) * 8 + row] = rs.total();
                if (half == 0) {
                    alphas[t * 8 + row] = alpha;
                    if (t == n_tiles - 1) m_last[row] = m_new;
                }
            }
            if ((lane & 15) == 0) flag[t] = (moved & (0xffffu << (lane & 16))) ? 1 : 0;
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_p + 8 * warp);
        }
        if (warp == 0) {
            // -------------------------------------------------------- rescales of O, then the chunk's result
            const uint32_t tlane = tmem;                           // lane quarter 0: rows 0 .. 7 on lanes 0 .. 7
            int phase = 0;
            float l_lo = 0.0f, l_hi = 0.0f;
            for (int j = 0; j < n_tiles; ++j) {
                if (j % 2 == 0) mbar_wait_warp(bar_p + 8 * (j / 2), 0, abort_word, p.dev_status);
                const float a = row < p.G ? alphas[j * 8 + row] : 1.0f;
                l_lo = __fmaf_rn(l_lo, a, row < p.G ? sums[(2 * j) * 8 + row] : 0.0f);
                l_hi = __fmaf_rn(l_hi, a, row < p.G ? sums[(2 * j + 1) * 8 + row] : 0.0f);
                if (warp_uniform(flag[j]) != 0) {
                    mbar_wait_warp(bar_pv, phase & 1, abort_word, p.dev_status);
                    ++phase;
                    tc_fence_after();
#pragma unroll 1
                    for (int cc = 0; cc < VC / 32; ++cc) {
                        uint32_t v[32];
                        tmem_ld32(tlane + COL_O + 32 * cc, v);
                        tmem_wait_ld();
#pragma unroll
                        for (int i = 0; i < 32; ++i) v[i] = __float_as_uint(rescale_o(__uint_as_float(v[i]), a));
                        tmem_st32(tlane + COL_O + 32 * cc, v);
                    }
                    tmem_wait_st();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar_resc);
                }
            }
            mbar_wait_warp(bar_pv, phase & 1, abort_word, p.dev_status);
            tc_fence_after();
            const float m = row < p.G ? m_last[row] : 0.0f;
            const float Ltot = finalize_l(l_lo, l_hi), inv = finalize_inv(Ltot);
            const long long orow = static_cast<long long>(seq) * p.Hq + head + lane;
            const long long slot = orow * p.nchunk_max + chunk;
            const bool store = lane < p.G && !*abort_word;         // (lanes 0 .. 7: G <= 8)
            if (store && rank == 0) {
                if (p.direct_out) {
                    if (p.lse) p.lse[orow] = finalize_lse(m, Ltot, c);
                } else {
                    p.part_ml[4 * slot] = m;
                    p.part_ml[4 * slot + 1] = l_lo;
                    p.part_ml[4 * slot + 2] = l_hi;
                }
            }
#pragma unroll 1
            for (int cc = 0; cc < VC / 32; ++cc) {
                uint32_t v[32];
                tmem_ld32(tlane + COL_O + 32 * cc, v);
                tmem_wait_ld();
                if (!store) continue;
                if (p.direct_out) {
                    // one chunk per sequence: the partial is the result (see the decode mode of attn_kernel)
                    uint4* d4 = reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(p.o) + orow * D + rank * VC + 32 * cc);
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        d4[i] = make_uint4(
                            pack_bf16x2(finalize_o(__uint_as_float(v[8 * i]), inv), finalize_o(__uint_as_float(v[8 * i + 1]), inv)),
                            pack_bf16x2(finalize_o(__uint_as_float(v[8 * i + 2]), inv), finalize_o(__uint_as_float(v[8 * i + 3]), inv)),
                            pack_bf16x2(finalize_o(__uint_as_float(v[8 * i + 4]), inv), finalize_o(__uint_as_float(v[8 * i + 5]), inv)),
                            pack_bf16x2(finalize_o(__uint_as_float(v[8 * i + 6]), inv), finalize_o(__uint_as_float(v[8 * i + 7]), inv)));
                } else {
                    float4* d4 = reinterpret_cast<float4*>(p.part_o + slot * D + rank * VC + 32 * cc);
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        d4[i] = make_float4(__uint_as_float(v[4 * i]), __uint_as_float(v[4 * i + 1]),
                                            __uint_as_float(v[4 * i + 2]), __uint_as_float(v[4 * i + 3]));
                }
            }
        }
        __syncwarp();
        cluster_arrive();
    }

    // ---------------------------------------------------------------- teardown
    if (*abort_word) {   // let copies and MMAs in flight finish before shared memory and TMEM are released
        const unsigned long long t0 = globaltimer_ns();
        while (globaltimer_ns() - t0 < 1000000ull) {
        }
    }
    __syncwarp();
    cluster_wait();
    tc_fence_before();
    __syncthreads();
    if (warp == 13) tmem_dealloc(tmem, TMEM_COLS);
}

static cudaError_t configure() {
    static DeviceOnce configured;     // the shared-memory opt-in belongs to the (function, device) pair
    return configured.run([&]() {
        return cudaFuncSetAttribute(decode_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    static_cast<int>(DXSmem::BYTES));
    });
}

cudaError_t decode_cluster_max_active(int* clusters) {
    const cudaError_t e = configure();
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = DECODE_CLUSTER;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(DECODE_CLUSTER);
    cfg.blockDim = dim3(DX_THREADS);
    cfg.dynamicSmemBytes = DXSmem::BYTES;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaOccupancyMaxActiveClusters(clusters, decode_cluster_kernel, &cfg);
}

cudaError_t launch_decode_cluster(int nchunk, int Hkv, int B, const CUtensorMap& tmQ, const CUtensorMap& tmK,
                                  const CUtensorMap& tmV, const AttnParams& p, cudaStream_t stream) {
    const cudaError_t e = configure();
    if (e != cudaSuccess) return e;
    return launch_pdl(decode_cluster_kernel, dim3(static_cast<unsigned>(nchunk) * DECODE_CLUSTER, static_cast<unsigned>(Hkv), static_cast<unsigned>(B)),
                      DX_THREADS, DXSmem::BYTES, stream, DECODE_CLUSTER, tmQ, tmK, tmV, p);
}

}  // namespace tik
