// Host-side declarations shared by the translation units of libtik (not part of the ABI).
#pragma once
#include <cuda_bf16.h>
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <atomic>
#include <string>

struct tik_ctx {
    int device = 0;
    int sm_count = 0;
    int max_clusters = 0;               // clusters of the cluster decode kernel that run at one time
    int* dev_status = nullptr;          // one int of device flags (TIK_DEV_*)
    void* encode_tiled = nullptr;       // cuTensorMapEncodeTiled from the driver
    std::string last_error;
};

namespace tik {

// Kernel launches issued by the library in this process (every launch site counts itself): what
// tik_kernel_launches() reports, so that a caller can state how many kernels a region launched.
extern std::atomic<unsigned long long> g_kernel_launches;
inline void count_launch() { g_kernel_launches.fetch_add(1, std::memory_order_relaxed); }


// Launch with programmatic stream serialization (see tik_ptx.cuh); clusters of `cluster` CTAs when > 1.
// Every call was preceded by a full drain, launch latency and CTA set-up (~5 us between kernels of 3 to
// 20 us): a 16-row decoder layer of 12 launches (H 1536) 116 -> 99 us, two short sequences forward +
// backward 36.9 -> 31.8 us, a 1000-token prompt (28/4 heads) 24.9 -> 23.5 us.
template <class... P, class... A>
cudaError_t launch_pdl(void (*kern)(P...), dim3 grid, unsigned threads, size_t smem, cudaStream_t stream, unsigned cluster,
                       A&&... args) {
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    count_launch();
    return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

// Runs a per-device set-up step (typically cudaFuncSetAttribute, whose effect belongs to the
// current device's context) once for every device that reaches it.  One flag per device ordinal;
// a failed step is retried by the next call.  Two threads racing on a device's first call may
// both run the step, which is harmless for idempotent set-up.
struct DeviceOnce {
    static constexpr int MAX_DEVICES = 64;
    std::atomic<bool> done[MAX_DEVICES] = {};
    bool is_done(int device) const {
        return device >= 0 && device < MAX_DEVICES && done[device].load(std::memory_order_acquire);
    }
    void mark(int device) {
        if (device >= 0 && device < MAX_DEVICES) done[device].store(true, std::memory_order_release);
    }
    // `device` < 0: use the current CUDA device.  Ordinals beyond the table run the step every time.
    template <class F>
    cudaError_t run(F&& step, int device = -1) {
        if (device < 0) {
            cudaError_t e = cudaGetDevice(&device);
            if (e != cudaSuccess) return e;
        }
        if (is_done(device)) return cudaSuccess;
        cudaError_t e = step();
        if (e == cudaSuccess) mark(device);
        return e;
    }
};

// Builds a bf16 tiled tensor map with 128-byte swizzle; dims/box innermost first, strides
// in bytes for dims 1..rank-1.  Returns false (and fills err) on failure.  swizzle64: 64-byte swizzle instead.
bool make_tmap_bf16(tik_ctx* ctx, CUtensorMap* out, const void* base, int rank,
                    const uint64_t* dims, const uint64_t* strides_bytes, const uint32_t* box,
                    std::string* err, bool swizzle64 = false);

struct AttnParams {
    alignas(64) CUtensorMap tmO; // train / prefill: tiled map of the output (same shape and box as Q)
    alignas(64) CUtensorMap tmO32;   // the same tensor with a box of 32 rows (persistent kernel: one warp's rows)
    void* o;                     // bf16 output rows
    float* lse;                  // optional
    const int32_t* cu_seqlens;   // train: per sequence; prefill: per sequence, query tokens
    const int32_t* ctx_lens;     // prefill / decode
    const int32_t* block_table;  // prefill / decode
    int max_blocks;
    int Hq, Hkv, G;
    int page_size, pages_per_tile, num_pages;
    float c;                     // softmax_scale * log2(e)
    float* part_o;               // decode: [B][Hq][nchunk_max][d]
    float* part_ml;              // decode: [B][Hq][nchunk_max][4] = m, l_lo, l_hi, unused
    int page_shift, ppt_shift;   // log2(page_size), log2(pages_per_tile)
    int nchunk_max;
    int max_ctx;                 // decode: the host's bound on ctx_lens (sized the grid and the scratch)
    int cpc;                     // decode: consecutive chunks streamed by one CTA
    int direct_out;              // decode: one chunk per sequence by the host's bound -- the chunk's partial is
                                 // the result, normalised and stored by the decode kernel itself (no combine)
    int* dev_status;
    int lookahead;               // train / prefill: block distance of the query-tile L2 prefetch
    int npair;                   // train / prefill, one CTA per item: the first 2 npair query tiles go in pairs (<= 8)
    int x_base;                  // train / prefill, one CTA per item: candidate index of the grid's last block (0, or 8: single tiles only)
    int wait_at_end;             // persistent kernel: 1 = launched behind the single-tile grid (see launch_attn_persist)
};

// mode: 0 train (packed K/V), 1 prefill (paged K/V), 2 decode (paged K/V, chunk partials)
cudaError_t launch_attn(int d, int mode, dim3 grid, const CUtensorMap& tmQ, const CUtensorMap& tmK,
                        const CUtensorMap& tmV, const AttnParams& p, cudaStream_t stream);
cudaError_t launch_combine(int d, const AttnParams& p, int B, cudaStream_t stream);
// Decode for query groups of at most DECODE2_MAX_G heads (tik_decode.cu): two small CTAs per SM,
// same grid, scratch layout and output bits as launch_attn in decode mode.
constexpr int DECODE2_MAX_G = 8;
cudaError_t launch_decode2(int d, dim3 grid, const CUtensorMap& tmQ, const CUtensorMap& tmK, const CUtensorMap& tmV,
                           const AttnParams& p, cudaStream_t stream);

// Decode of small calls (tik_decode_cluster.cu), d = 128: clusters of four CTAs per chunk.  tmV has a box of
// 32 columns, with the 64-byte swizzle.  Same scratch layout and output bits.
constexpr int DECODE_CLUSTER = 4;
cudaError_t decode_cluster_max_active(int* clusters);     // of the current device; launches nothing
cudaError_t launch_decode_cluster(int nchunk, int Hkv, int B, const CUtensorMap& tmQ, const CUtensorMap& tmK,
                                  const CUtensorMap& tmV, const AttnParams& p, cudaStream_t stream);

// Persistent full-sequence attention (tik_attn_persist.cu): a planning kernel writes the list of
// work items of the call into `plan` (attn_plan_bytes bytes, 16-byte aligned), then one CTA per SM
// walks it.  X = candidate items per sequence for the host's length bound (as the grid's x extent
// of the one-CTA-per-item kernel).  Same output bits as launch_attn.
size_t attn_plan_bytes(int64_t S, int64_t max_positions);
bool attn_persist_supported(int64_t S, int64_t max_positions);
cudaError_t launch_attn_persist(int d, bool paged, int sm_count, int S, int X, const CUtensorMap& tmQ,
                                const CUtensorMap& tmK, const CUtensorMap& tmV, const AttnParams& p, void* plan,
                                cudaStream_t stream);

struct PrepParams {
    __nv_bfloat16* q;            // [total_new][Hq][d], in place
    __nv_bfloat16* k;            // [total_new][Hkv][d], in place
    const __nv_bfloat16* v;      // [total_new][Hkv][d] or null
    const __nv_bfloat16* q_weight;   // [d] or null (no Q norm)
    const __nv_bfloat16* k_weight;   // [d] or null (no K norm)
    float eps;
    const float* cos_sin;        // [max_pos][d]: cos | sin
    int max_pos;
    const int32_t* cu_new;       // [S+1]
    const int32_t* ctx_lens;     // [S] context after the write, or null (positions start at 0)
    __nv_bfloat16* k_cache;      // [num_pages][Hkv][page_size][d] or null (no cache write)
    __nv_bfloat16* v_cache;
    const int32_t* block_table;
    int max_blocks, S, Hq, Hkv, page_size, num_pages;
    long long total_new;
    int* dev_status;
};
cudaError_t launch_prep(int d, const PrepParams& p, int64_t total_new, cudaStream_t stream);

// Decode with one CTA per SM: how many consecutive chunks a CTA streams.  A CTA's set-up and drain cost about
// a third of one chunk's streaming time, so several chunks per CTA pay as long as the grid still covers
// the SMs four times.  Chunk partials do not depend on this choice.
inline int decode_chunks_per_cta(long long B, int Hkv, int nchunk, int sm_count) {
    const long long slots = sm_count > 0 ? sm_count : 148;
    for (int c = 4; c > 1; --c)
        if (c <= nchunk && B * Hkv * ((nchunk + c - 1) / c) >= 4 * slots) return c;
    return 1;
}
cudaError_t launch_kv_write(const void* k_new, const void* v_new, const int32_t* cu_new,
                            const int32_t* ctx_lens, void* k_cache, void* v_cache,
                            const int32_t* block_table, int max_blocks, int S, int64_t total_new,
                            int Hkv, int d, int page_size, int num_pages, int* dev_status,
                            cudaStream_t stream);

struct LogprobParams {
    const int32_t* target;
    float* logprob;
    float* lse;                  // optional
    float* part_ml;              // [T][nsuper][2]
    float* z_target;             // [T]
    int64_t T;
    int H, V, nsuper;
    int spc;                     // consecutive 1024-column super-chunks walked by one CTA
    int unit_mode;               // 1: T <= LP_UNIT_MODE_ROWS: persistent CTAs over 256-column steps, one (max, sum) pair per 128-column tile
    int nunit, ntile128;         // units = ceil(V / 256) x ntp, ceil(V / 128)
    int ntp;                     // unit mode: pairs of token tiles (single CTAs: 1)
    int sm_count;
    float inv_temperature;
    int* dev_status;
};
cudaError_t launch_logprob(const CUtensorMap& tmA, const CUtensorMap& tmB, const LogprobParams& p, bool pair,
                           cudaStream_t stream);

struct NormParams {
    const __nv_bfloat16* x;      // [T][H]
    __nv_bfloat16* residual;     // [T][H] in/out, or null (plain RMSNorm)
    const __nv_bfloat16* weight; // [H]
    __nv_bfloat16* y;            // [T][H] (may be x)
    float eps;
    long long T;
    int H;
};
cudaError_t launch_rmsnorm(const NormParams& p, cudaStream_t stream);
cudaError_t launch_swiglu(const void* gate_up, void* out, long long T, int I, cudaStream_t stream);

struct LinearParams {
    __nv_bfloat16* y;            // [T][N]
    int64_t T;
    int K, N, nsuper;
    int super_cols;              // pairs, band raster: output columns per CTA, a multiple of 256, at most 4096
    int unit_mode;               // persistent CTAs (pairs) over nunit units
    int ntp;                     // units per column step: row tiles (pairs: pairs of row tiles)
    int nu, nunit, a_rows;       // columns per unit 64 / 128 / 256 (pairs: 256), units, staged x rows 8 / 16 / 32 / 64 / 128
                                 // (narrow outputs: weight rows per CTA 8 .. 64, CTAs, x rows 8 .. 128)
    int kps, nst;                // narrow outputs: K slices per ring stage, stages (12 at most)
    int m;                       // narrow outputs: rows of the M operand if that is x: 64 or 128; 0: the weights
    int sm_count;
    int* dev_status;
};
// Schedule of a call of at most 16 row tiles, from a cost model: rounds of units x K slices x the time of one
// 64-wide K slice, as measured on a B200 with W out of HBM.  A single CTA takes in x and W rows at ~130 GB/s
// (128 rows: N = 64 190 ns, 128 235 ns, 256 370 ns); a pair's slice (256 x 256) is its MMAs, ~300 ns, and a
// pair costs ~2 us more to set up and to drain.  Ties go to pairs and the wider unit (fewer bytes out of L2), but with
// one row tile of more than 64 rows to the narrower one: such a call is one pass over W, and three rounds of 128
// columns keep more SMs at it than two of 256 whose second is not full.  256 columns -> 128, us: 65 / 128 rows of K
// 5120, N 55296 96.2 / 98.4 -> 91.6 / 94.6; K 3584, N 40960 63.9 / 65.6 -> 58.9 / 60.3; K 1536, N 46080 31.6 / 33.1 ->
// 29.1 / 30.3.
// Before, every call of 129 .. 2048 rows ran as pairs; us, pairs -> the choice, W out of HBM:
//   K 8960,  N 1536:   129 rows 44.2 -> 29.8 (64 columns), 1024 rows 44.6 -> 34.3 (128), 2000 rows 47 (pairs)
//   K 18944, N 3584:   129 rows 88.5 -> 61.0 (64), 512 rows 89.1 -> 73.6 (128), 741 rows 91.1 (pairs; 128: 140)
//   K 3584,  N 3584:   129 rows 21.0 -> 14.6 (64), 512 rows 21.2 -> 16.1 (128)
//   K 1536,  N 256:    129 .. 2000 rows 11.7 -> 7.5 (64)
//   K 3584,  N 37888:  278 rows 89.1 -> 82.6 (256), 512 rows 98 (pairs; 256: 109)
struct LinearChoice {
    bool pair;
    int nu;
    bool units;                  // persistent over units, else the band raster (pairs)
};
// Rows of x that a K slice of a call of one row tile stages.  What lies past T arrives as zeros, but not for free: with 32
// rows for calls of 1 .. 7 the x copies of all CTAs were late (K 8960, N 10240, 1 row 43.6 us, 33.9 with 8; N 12288 43.8,
// 37.4; 16 rows, N 10240 35.8, 34.3 with 16).
inline int linear_staged_rows(long long T) { return T <= 8 ? 8 : T <= 16 ? 16 : T <= 32 ? 32 : T <= 64 ? 64 : 128; }
inline LinearChoice linear_choose(long long T, int K, int N, int a_rows, int sm_count) {
    const long long ntile = (T + 127) / 128;
    LinearChoice best = {false, 256, true};
    double best_us = -1.0;
    const double tie = ntile == 1 && a_rows == 128 ? 1.02 : 0.98;
    auto consider = [&](bool pair, int nu) {
        const long long slots = pair ? sm_count / 2 : sm_count;
        const long long units = static_cast<long long>((N + nu - 1) / nu) * (pair ? (ntile + 1) / 2 : ntile);
        const long long rounds = (units + slots - 1) / slots;
        const double slice_ns = pair ? 300.0 : (a_rows + nu) * 128.0 / 130.0;
        const double us = rounds * (K / 64) * slice_ns * 1e-3 + (pair ? 2.0 : 0.0);
        if (best_us < 0.0 || us < best_us * tie) {
            best_us = us;
            best = {pair, nu, true};
        }
    };
    if (ntile > 1) consider(true, 256);
    for (int nu = 256; nu >= 64; nu /= 2) consider(false, nu);
    return best;
}
// The kernel of a call that the narrow schedule does not take.  More than 16 row tiles: the band raster (x no longer
// fits L2).
inline LinearChoice linear_wide_choose(const LinearParams& p) {
    if (p.T > 16 * 128) return {true, 256, false};
    return linear_choose(p.T, p.K, p.N, std::max(32, linear_staged_rows(p.T)), p.sm_count);
}
// The narrow schedule: one unit of nu weight rows x one row tile per CTA, nu as few as need no more CTAs than SMs
// (whole 8-row swizzle atoms; an MMA of 128 rows takes N = 16 i), or one CTA per row tile when there are more of those.
// A second wave repeats the whole chain over K: 768 rows x N 1184, K 8960, in 150 CTAs 49.7 us, by the unit kernel 26.4;
// 8192 x 104, K 3584, in 192 CTAs 27.0, by pairs 20.8.  One CTA per row tile reads x once (K 3584, N 8, pairs -> this:
// 20000 rows 45.6 -> 32.4, 100000 rows 156 -> 108).  In one wave, K 3584, pairs -> this: 2304 x 256 22.0 -> 12.1, 5000 x 128
// 22.1 -> 13.4.  Its time is the MMAs' shared-memory reads,
// 64 or 128 rows of the M operand + the N operand's, and what TMA writes there: the operand whose choice as M
// reads fewer rows is M (x must be for more than 80 rows).  Above 48 weight rows and 80 x rows the unit
// kernel is as fast or faster (K 18944, N 3584, 256 rows: 53.1 us, 54.5 here; K 1536, N 8960, 128 rows: 8.3, 8.5).
inline bool linear_narrow_choose(LinearParams& p) {
    const long long ntile = (p.T + 127) / 128;
    const int rows = static_cast<int>(p.T < 128 ? p.T : 128), t16 = (rows + 15) / 16 * 16, m = rows > 64 ? 128 : 64;
    const long long ctas = ntile < p.sm_count ? p.sm_count / ntile : 1;      // that a row tile may take
    auto weight_rows = [&](int atom) {
        const long long per = atom * ctas;
        return atom * ((p.N + per - 1) / per);
    };
    const long long nw = weight_rows(8), nx = weight_rows(m == 128 ? 16 : 8);
    const bool x_is_m = t16 > 80 || (m == 128 ? m + nx <= 64 + t16 : nx < t16);
    const int most = t16 > 80 ? 48 : 64;
    if ((x_is_m ? nx : nw) > most || p.N * ntile > static_cast<long long>(most) * p.sm_count) return false;
    p.m = x_is_m ? m : 0;
    p.nu = static_cast<int>(x_is_m ? nx : nw);
    p.a_rows = x_is_m ? (rows + 7) / 8 * 8 : t16;
    p.ntp = static_cast<int>(ntile);
    p.nunit = (p.N + p.nu - 1) / p.nu * p.ntp;
    return true;
}
// tmW / tmX: [K / 64][rows][64] views with boxes of 64 x nu x kps and 64 x a_rows x kps
constexpr uint32_t LINEAR_NARROW_RING = 216 * 1024;
cudaError_t launch_linear_narrow(const CUtensorMap& tmW, const CUtensorMap& tmX, const LinearParams& p, cudaStream_t stream);
cudaError_t launch_linear(const CUtensorMap& tmA, const CUtensorMap& tmB, const CUtensorMap& tmY,
                          const LinearParams& p, bool pair, cudaStream_t stream);

struct BwdParams {
    const int32_t* cu_seqlens;   // [S+1]
    const float* lse;            // [total][Hq], natural log, from the forward
    float* delta;                // [total][Hq] scratch: rowsum(dO o O)
    __nv_bfloat16* dq;           // [total][Hq][d]
    __nv_bfloat16* dk;           // [total][Hkv][d]
    __nv_bfloat16* dv;           // [total][Hkv][d]
    int Hq, Hkv, G;
    float c;                     // softmax_scale * log2(e)
    float scale;
    int dq_heads, dq_groups;     // query heads per dQ CTA, CTAs per KV head: ceil(G / dq_heads)
    int dq_tiles_first;          // dQ grid: query tiles fastest, one head after the other; 0: heads fastest
    int* dev_status;
};
// The dQ grid of a backward call: heads per CTA and order.
//
// Query heads per CTA: a head's set-up, first loads and epilogue run under its neighbour's steps, but longer
// CTAs leave a longer tail.  Backward, us, 1 / 2 / 4 heads per CTA in the order below, with items (tile, head) per SM:
//   (d 128, 64/8 heads) 47 x 45..238 tokens, 41: 381 / 321 / 306;  21 x 77..681, 35: 542 / 468 / 456;  16 x 500..3000, 107:
//   4280 / 4132 / 4102
//   (32/8) 10 x 385..2369, 27: 934 / 860 / 844;  8 x 100..400, 4.8: 60.3 / 53.8 / 56.9;  2048, 3.5: 130 / 130 / 130
//   (28/4) 16 x 1280..5120, 71: 3983 / 3888 / 3855;  32 x 60..128, 6.1: 62.0 / 56.4 / 56.2
//   (12/2) 16 x 1000..3000, 21: 820 / 774 / 795;  (8/1) 8 x 2000, 6.9: 254 / 258 / 264
//   (d 64, 4/1) 9 x 3440..7743, 11: 713 / 731 / 765;  40 x 100..500, 3.5: 34.2 / 33.9 / 35.9
//
// Order: heads fastest runs the heavy query tiles of all heads first and leaves the light ones for the end of the grid, a
// tail shorter by ~0.6 us per tile of the longest sequence and head of a CTA.  Tiles fastest where that costs more.
// Backward, us, tiles fastest / heads fastest:
//   shorter tail    (8/8) 3 x 1500 66.4 / 60.1;  (32/8) 2 x 4096 918 / 886;  (12/2) 8 x 4096 1355 / 1309;  (16/16) 10240, K and V
//                   84 MB, 1350 / 1297
//   K and V of all the heads are in use at a time, and beyond two thirds of L2 are read again
//                   (32/32) 16384 6475 / 6860;  (64/64) 8192 3469 / 3859;  (32/8) 24576, 101 MB, 13862 / 14146;  65536 96531 /
//                   100267;  ((16/16) 12288, 101 MB, 1885 / 1845)
//   many KV heads   (64/64) 4 x 2048 1216 / 1354;  (32/32) 2 x 4096 983 / 997 and 997 / 969;  8 x 1024 433 / 436
//   empty tiles, of sequences shorter than max_seqlen: a CTA starts every ~10 ns, which hides while other heads' tiles are at
//   work; all heads' empty tiles in one run do not.  By empty CTAs per tile of max_seqlen and head of a CTA (60: the two even)
//                   475 (64/8) 32 x 200..1000 under 8192 1370 / 1468;  236 (64/8) 32 x 200..2000 3545 / 3577;  118 (28/4) 32 x
//                   200..2000 1577 / 1603;  60.1 (32/8) 8 x 1000 under 16384 410 / 430;  56 (28/4) 16 x 1433..5120 3920 / 3904;
//                   53 (28/4) 2 x 1000 under 16384 121 / 118;  44 (12/2) 32 x 200..2000 692 / 682;  24 (28/4) 4 x 1000 under 4096
//                   152 / 146;  6 (32/8) 4000 under 16384 492 / 448
inline void bwd_dq_choose(BwdParams& p, int64_t S, int64_t total_tokens, int64_t max_seqlen, int d, int sm_count) {
    const int64_t max_tiles = (max_seqlen + 127) / 128, most = total_tokens / 128 + S;
    const int64_t items = (most < max_tiles * S ? most : max_tiles * S) * p.Hq;
    p.dq_heads = items < 5ll * sm_count ? 1 : items < 12ll * sm_count || max_tiles > 12 ? 2 : 4;
    p.dq_heads = p.dq_heads < p.G ? p.dq_heads : p.G;
    p.dq_groups = (p.G + p.dq_heads - 1) / p.dq_heads;
    const int64_t kv_bytes = (max_seqlen < total_tokens ? max_seqlen : total_tokens) * p.Hkv * d * 4;
    const bool hidden = (S * max_seqlen - total_tokens) * p.Hkv * p.dq_groups <= 60 * max_seqlen * p.dq_heads;
    p.dq_tiles_first = max_tiles > 65535 || p.Hkv > 32 || kv_bytes > 80ll << 20 || !hidden;   // (65535: a grid's second axis)
}
cudaError_t launch_attn_bwd(int d, int max_tiles, int S, const CUtensorMap& tmQ, const CUtensorMap& tmK,
                            const CUtensorMap& tmV, const CUtensorMap& tmDO, const BwdParams& p,
                            const void* o, const void* dout, long long n_vec, cudaStream_t stream);

}  // namespace tik
