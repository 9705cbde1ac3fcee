// Layer-by-layer implicit-GEMM convolution on the tensor cores (sm_100a): one launch per convolution over a batch of
// noisy samples, for the networks whose activations do not fit in shared memory (the 224 x 224 bottleneck network of
// the paper's second workload, Sec. 4.1).  Activations are the layer-by-layer engine's: int8, global memory,
// [sample][y][x][channel padded to 16].
//
//   D[pixel, cout] = sum over (tap, cin) of A[pixel, (tap, cin)] * W[cout, (tap, cin)]
//
// A tile is 128 output pixels x N output channels (N a multiple of 16, at most 256) whose int32 accumulators live in tensor
// memory.  The kernel is persistent (one CTA per SM, tiles dealt round-robin) and its warps have fixed roles that
// meet only at mbarriers:
//   * four warps gather operand rows: per reduction block (four columns of 16 input channels of a filter tap) a lane issues four
//     asynchronous 16-byte copies (through L1) into the K-major core-matrix layout (four lanes read one pixel's 64 bytes) whose
//     completion arrives on the stage's barrier; a pixel outside the image is copied from a run of the input
//     zero-point kept behind the repacked weights;
//   * one thread streams the matching slices of the repacked weights with bulk copies into the same stages; for a
//     1 x 1 stride-1 layer it also brings the operand rows, one tensor copy (cp.async.bulk.tensor) per block, and
//     the gather warps idle;
//   * one thread issues two tcgen05.mma (kind::i8, K = 32) per stage and commits the stage back to the loaders;
//     accumulators take two column ranges of tensor memory in turn (four in whole tiles of 64 channels by tensor copy), so a
//     tile's reduction runs under the previous ones' epilogue;
//   * the others requantise (fixed-point multiplier, shift, zero-points, residual add, clamp): in whole tiles (channels in
//     multiples of 64) as fragments (epilogue_whole), sixteen warps where the operands come by tensor copy and eight
//     where they are gathered; in the general form eight, one tile row per thread (epilogue_rows).
// 1 x 1 layers that expand the channels, which the epilogue bounds, take tiles of 256 pixels x 128 channels (kPair): a
// thread then reads a channel's constants once for two operands.
// Every wait is bounded; on expiry a role raises the CTA's abort flag and the error word, the others leave their
// loops, and the CTA frees its tensor memory and returns.
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "isc_conv.cuh"
#include "isc_epilogue.cuh"
#include "isc_internal.h"
#include "isc_tc.cuh"

namespace isc {

using namespace tc;
using namespace conv;

namespace {

constexpr int kTileM = 128;
constexpr int kBlockK = 64;                  // bytes of K per stage: two MMA K-steps
constexpr int kMaxStages = 16;
constexpr int kPairN = 128;                  // channels of a paired tile: two operands of 128 rows, two tiles in tensor memory
constexpr int kStemEpi = 8, kStemThreads = 32 * (kStemEpi + 1);        // k_stem: two threads per tile row and the MMA warp; two CTAs per SM
constexpr size_t kStemSmemPair = 108 * 1024, kStemSmemLimit = 220 * 1024;       // dynamic shared memory of k_stem: for two CTAs per SM; at most
constexpr size_t kStemSmemOwn = 5248;        // its static shared memory and what the system takes of a CTA's
constexpr int kRowTeams = 2, kRowWarps = 4 * kRowTeams;                // epilogue_rows: a team of four warps takes every other tile
// Warps of k_igemm by role: epilogue, gather, and one each for MMAs and weights.  Whole tiles whose operands come by tensor copy
// need no gather warps and have sixteen epilogue warps; beside four gather warps sixteen would leave a thread 80 registers,
// and two gather warps were too few (3 x 3 stride 2, 128 channels at 56 x 56: 156 -> 202 us).
__host__ __device__ constexpr int igemm_epi_warps(bool whole, bool copy) { return whole && copy ? 16 : kRowWarps; }
__host__ __device__ constexpr int igemm_gather_warps(bool whole, bool copy) { return whole && copy ? 0 : 4; }
__host__ __device__ constexpr int igemm_threads(bool whole, bool copy) { return 32 * (igemm_epi_warps(whole, copy) + igemm_gather_warps(whole, copy) + 2); }

struct IgemmParams {
    alignas(64) CUtensorMap tmap_a;          // the input as (16 bytes, pixel, 16-byte column of the channels): see tma_a
    alignas(64) CUtensorMap tmap_res;        // the residual operand as (channel, pixel), boxes of a tile: prefetched into L2
    GLayer L;
    int prefetch_res;
    int tma_a;                               // 1 x 1 stride 1: the operand rows arrive by one tensor copy per block, the gather warps idle
    int batch, n_tile, tiles_n, n_acc, acc_stride, tmem_cols, stages;     // accumulators in tensor memory; columns from one to the next
    int units, n_blocks;                     // 16-byte columns of the reduction (filter tap, 16 input channels); blocks of four of them
    uint32_t scratch_off;                    // epilogue_rows: the warps' row scratch within the dynamic shared memory
    uint32_t m_total, tiles_m;               // batch * hout * wout (< 2^31); tiles of 128 of them
    const int8_t *in, *res;
    int8_t *out;
    const int8_t *wpack;                     // [cout tile][block][4 K columns][n_tile rows][16 bytes]
    const int8_t *zp_run;                    // 64 bytes of the input zero-point: the operand row of a pixel outside the image
    const int4 *cst;                         // per output channel: folded bias, multiplier, rounding addend, shift - 1
    int fast_requant, fast_residual, lo;     // the layer has the 32-bit form; residual rescale by 2^-31 or 2^-32; lower clamp
    uint32_t res_m2, res_k8;                 // residual multiplier in the 2^-32 form, or as a single-precision number; that form's offset
    int res_short;                           // the residual term is a single-precision product (see requant16_fast)
    int debug_stall;                         // test hook: the weights are never sent, so every wait of the kernel runs out
    long long res_r2;
    int32_t *err;
};

// What an epilogue warp needs from the kernel's prologue.
struct EpiCtx {
    uint32_t sbase, tmem, n_tiles, grid_n;
    int tiles_n, warp, lane;
    uint32_t cst_s, acc_full, acc_free;       // shared-memory addresses: constants, the accumulators' barriers
    const volatile int *abort_flag;
};

// The epilogue of the general form.  Warp w owns lanes 32 (w mod 4) .. +31 of an accumulator (= 32 tile rows) and all N
// columns; team w / 4 takes every other tile of the CTA (accumulator `team`).  A thread requantises its own row in
// place in a per-warp scratch area in shared memory (row stride N + 16 bytes: conflict-free for the row-wise and
// for the coalesced access).  After every 64 columns the warp writes those columns of its 32 rows out as runs of
// 64 contiguous bytes per row and requests the same columns of the residual rows of its next tile into the
// space that has just been read, so memory traffic runs under the arithmetic of the following columns.
// kMode 0: 64-bit requantisation (any shift), 1: 32-bit form, 2 / 3: 32-bit form with the residual add (3: its
// single-precision form).
template <int kMode>
__device__ __forceinline__ bool epilogue_rows(const IgemmParams &p, const EpiCtx &c)
{
    const GLayer &L = p.L;
    const int warp = c.warp, lane = c.lane, n_tile = p.n_tile, tiles_n = c.tiles_n;
    const int q = warp & 3, team = warp >> 2;
    const uint32_t lane_base = (uint32_t)(q * 32) << 16;
    const uint32_t row_stride = epi_row_stride(n_tile);
    const uint32_t scr0 = c.sbase + p.scratch_off + (uint32_t)warp * 32u * row_stride;
    const uint32_t scr_row = scr0 + (uint32_t)lane * row_stride;
    // coalesced access to 64 columns of the 32 rows: four lanes per row, eight rows per instruction
    const int crow = lane >> 2, cchunk = lane & 3;
    const uint32_t scr_co = scr0 + (uint32_t)crow * row_stride + (uint32_t)cchunk * 16u;
    const size_t co_step = (size_t)8 * L.coutp;
    // where tile t's rows start in the output / residual tensors, for this lane's coalesced position; null when the
    // row is beyond the last pixel (the rows of a warp that are valid are its first ones)
    auto tile_ptr = [&](const int8_t *base, uint32_t t, uint32_t &rows) {
        const uint32_t m_idx = t / (uint32_t)tiles_n;
        const uint32_t m0 = m_idx * kTileM + (uint32_t)q * 32u;
        rows = m0 < p.m_total ? min(32u, p.m_total - m0) : 0u;
        return base + (size_t)(m0 + (uint32_t)crow) * L.coutp + (int)(t - m_idx * tiles_n) * n_tile + cchunk * 16;
    };
    auto tile_cols = [&](uint32_t t) { return min(n_tile, L.coutp - (int)(t % (uint32_t)tiles_n) * n_tile); };       // a multiple of 16
    auto residual_fetch = [&](const int8_t *src, uint32_t rows, int c0, int n_cols) {
        if (c0 + cchunk * 16 >= n_cols) return;
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if ((uint32_t)(8 * k + crow) < rows) cp_async16(scr_co + (uint32_t)(8 * k) * row_stride + (uint32_t)c0, src + (size_t)k * co_step + c0);
    };
    // the team's tiles: every kRowTeams-th of the CTA's
    const uint32_t t_step = (uint32_t)kRowTeams * c.grid_n;
    uint32_t t = blockIdx.x + (uint32_t)team * c.grid_n;
    if (kMode >= 2 && t < c.n_tiles) {
        uint32_t rows;
        const int8_t *src = tile_ptr(p.res, t, rows);
        for (int c0 = 0; c0 < n_tile; c0 += 64) residual_fetch(src, rows, c0, tile_cols(t));
    }
    for (int au = 0; t < c.n_tiles; t += t_step, ++au) {
        const uint32_t m_idx = t / (uint32_t)tiles_n;
        const int n0 = (int)(t - m_idx * tiles_n) * n_tile;
        const uint32_t m = m_idx * kTileM + (uint32_t)q * 32u + (uint32_t)lane;
        const int8_t *res_px = (kMode == 0 && p.res && m < p.m_total) ? p.res + (size_t)m * L.coutp : nullptr;
        uint32_t rows, rows_next = 0;
        int8_t *dst = const_cast<int8_t *>(tile_ptr(p.out, t, rows));
        const int8_t *res_next = (kMode >= 2 && t + t_step < c.n_tiles) ? tile_ptr(p.res, t + t_step, rows_next) : nullptr;
        cp_async_wait_all();                                        // the tile's residual rows, requested during the previous tile
        __syncwarp();
        if (!wait_bar<kHintEpi>(c.acc_full + 8u * (uint32_t)team, (uint32_t)au & 1u, c.abort_flag)) {
            cp_async_wait_all();                                    // the next tile's residual rows may still be landing
            return false;
        }
        tc_fence_after();
        const int n_cols = tile_cols(t), n_cols_next = res_next ? tile_cols(t + t_step) : 0;
        const uint32_t acc_base = c.tmem + lane_base + (uint32_t)(team * p.acc_stride);
        const uint32_t cst0 = c.cst_s + (uint32_t)n0 * 16u;
        // 32 columns per step, the accumulators of the next step requested before this step's arithmetic
        auto step = [&](int (&acc)[2][16], int c0) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int cc = c0 + 16 * h;
                if (h == 1 && cc >= n_cols) break;
                uint4 v;
                if (kMode == 3) {
                    v = requant16_fast<2>(acc[h], cst0 + (uint32_t)cc * 16u, ld_shared_v4(scr_row + (uint32_t)cc), p.res_m2, 0ll, p.res_k8, p.lo);
                } else if (kMode == 2) {
                    v = requant16_fast<1>(acc[h], cst0 + (uint32_t)cc * 16u, ld_shared_v4(scr_row + (uint32_t)cc), p.res_m2, p.res_r2, 0u, p.lo);
                } else if (kMode == 1) {
                    v = requant16_fast<0>(acc[h], cst0 + (uint32_t)cc * 16u, make_uint4(0, 0, 0, 0), 0u, 0ll, 0u, p.lo);
                } else {
#pragma unroll
                    for (int o = 0; o < 16; ++o) acc[h][o] += __ldg(L.bias + n0 + cc + o);
                    v = epilogue16(acc[h], L, n0 + cc, res_px);
                }
                st_shared_v4(scr_row + (uint32_t)cc, v);
            }
        };
        int acc_a[2][16], acc_b[2][16];
        tmem_ld32_issue(acc_base, acc_a);
#pragma unroll 1
        for (int c0 = 0; c0 < n_cols; c0 += 64) {
            const bool second = c0 + 32 < n_cols, more = c0 + 64 < n_cols;
            tmem_ld32_wait(acc_a);
            if (second) tmem_ld32_issue(acc_base + (uint32_t)c0 + 32u, acc_b);
            step(acc_a, c0);
            if (second) tmem_ld32_wait(acc_b);
            if (more) {
                tmem_ld32_issue(acc_base + (uint32_t)c0 + 64u, acc_a);
            } else {
                tc_fence_before();
                mbar_arrive(c.acc_free + 8u * (uint32_t)team);      // the accumulator is in registers: the next tile may overwrite it
            }
            if (second) step(acc_b, c0 + 32);
            __syncwarp();
            const bool mine = c0 + cchunk * 16 < n_cols;            // a row holds the tile's columns and no more
            uint4 v[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) v[k] = ld_shared_v4(mine ? scr_co + (uint32_t)(8 * k) * row_stride + (uint32_t)c0 : scr0);
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (mine && (uint32_t)(8 * k + crow) < rows) *reinterpret_cast<uint4 *>(dst + (size_t)k * co_step + c0) = v[k];
            __syncwarp();
            if (res_next) residual_fetch(res_next, rows_next, c0, n_cols_next);
        }
        for (int c0 = (n_cols + 63) & ~63; c0 < n_cols_next; c0 += 64) residual_fetch(res_next, rows_next, c0, n_cols_next);
    }
    cp_async_wait_all();
    return true;
}

// The epilogue of whole tiles (every column valid, a multiple of 64 of them).  Accumulators are read as fragments: of 16
// columns a thread holds four in each of four rows per operand (lane / 4 + 8 i), and the columns of the weights are ordered
// so that its columns of four such chunks are 16 consecutive channels (igemm_channel).  A thread's four constants of a chunk
// serve eight outputs each in a paired tile, residual rows are read and results written straight from registers (four lanes
// make 64 contiguous bytes of a pixel), nothing passes through shared memory, and sixteen warps have registers enough.  (One row
// per thread took a 16-byte constant per one or two outputs, a scratch row in shared memory both ways, and eight warps, two
// per scheduler, which left its latency exposed: 64 -> 256 channels with a residual operand at 56 x 56, 512 samples: 280 us in all, now 253.)
// n_acc accumulators are in flight.  A quarter's four warps (operands by tensor copy) share two: two take every other tile, and
// in it every other unit; with four accumulators (64 columns) each takes every fourth tile.  Of a quarter's two warps
// (gathered operands) each takes every other tile, all of it.
// kMode 0: 64-bit requantisation (any shift), 1: 32-bit form, 2 / 3: 32-bit form with the residual add (3: its
// single-precision form).  kClamp: the lower clamp is above -128.
template <int kMode, bool kPair, bool kClamp, int kWarps>
__device__ __forceinline__ bool epilogue_whole(const IgemmParams &p, const EpiCtx &c)
{
    constexpr uint32_t kMT = kPair ? 2 : 1;
    const GLayer &L = p.L;
    const uint32_t word = (uint32_t)c.lane & 3u, q = (uint32_t)c.warp & 3u, w4 = (uint32_t)c.warp >> 2;
    const uint32_t n_acc = (uint32_t)p.n_acc, team = w4 & (n_acc - 1u), split = (uint32_t)(kWarps / 4) / n_acc, part = w4 / n_acc;
    const uint32_t n_units = kMT * ((uint32_t)p.n_tile >> 6), coutp = (uint32_t)L.coutp;       // a unit: 128 rows x 64 columns
    const uint32_t acc0 = c.tmem + (q * 32u << 16) + team * (uint32_t)p.acc_stride, bar_full = c.acc_full + 8u * team, bar_free = c.acc_free + 8u * team;
    const bool has_res = kMode >= 2 || (kMode == 0 && p.res);
    uint32_t use = 0;
    for (uint32_t t = blockIdx.x + team * c.grid_n; t < c.n_tiles; t += n_acc * c.grid_n, ++use) {
        const uint32_t m_idx = t / (uint32_t)c.tiles_n, n0 = (t - m_idx * (uint32_t)c.tiles_n) * (uint32_t)p.n_tile + word * 16u;
        bool ready = false;
#pragma unroll 1
        for (uint32_t unit = part; unit < n_units; unit += split) {
            const uint32_t mt = kPair ? unit & 1u : 0u, col = (kPair ? unit >> 1 : unit) * 64u;
            const uint32_t row = (m_idx * kMT + mt) * (uint32_t)kTileM + q * 32u + ((uint32_t)c.lane >> 2);
            const uint32_t rem = row < p.m_total ? p.m_total - row : 0u;                 // valid rows are this thread's first ones
            const size_t at = (size_t)row * coutp + n0 + col;
            uint32_t io[4][4];                                                          // residual bytes, then results
#pragma unroll
            for (int i = 0; i < 4; ++i) {
#pragma unroll
                for (int k = 0; k < 4; ++k) io[i][k] = 0;
                if (has_res && (uint32_t)(8 * i) < rem) ld_global_v4(p.res + at + (size_t)(8 * i) * coutp, io[i]);
            }
            if (!ready) {
                ready = __all_sync(0xffffffffu, wait_bar<kHintEpi>(bar_full, use & 1u, c.abort_flag));
                if (!ready) return false;
                tc_fence_after();
            }
            const uint32_t acc = acc0 + mt * kPairN + col, cst = c.cst_s + (n0 + col) * 16u - word * 240u;       // n0 has the thread's 16 channels
            int a[2][8];
            tmem_ld_frag(acc, a[0]);
#pragma unroll
            for (int ch = 0; ch < 4; ++ch) {
                int4 k4[4];
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(k4[k].x), "=r"(k4[k].y), "=r"(k4[k].z), "=r"(k4[k].w) : "r"(cst + (uint32_t)(ch * 256 + k * 64)));
#pragma unroll
                for (int hf = 0; hf < 2; ++hf) {
                    tmem_ld_frag_wait(a[hf]);
                    // the next accumulators, before this step's arithmetic
                    if (hf == 0) tmem_ld_frag(acc + (uint32_t)(ch * 16) + (16u << 16), a[1]);
                    else if (ch < 3) tmem_ld_frag(acc + (uint32_t)(ch * 16 + 16), a[0]);
                    else if (unit + split >= n_units) {
                        tc_fence_before();
                        mbar_arrive(bar_free);                  // the accumulators are in registers: the next tile may overwrite them
                    }
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        uint32_t &w = io[2 * hf + j][ch];
                        const uint32_t rw = w ^ 0x80808080u;
                        int y[4];
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const int v = a[hf][2 * j + (k & 1) + 4 * (k >> 1)];
                            if (kMode == 0) {
                                const int o = (int)(n0 + col) + 4 * ch + k;
                                const long long rt = has_res ? residual_term(byte_of(w, k), L.zp_res, L.res_mult, L.res_shift) : 0ll;
                                y[k] = o < L.cout ? requant_clamp(v + __ldg(L.bias + o), __ldg(L.mult + o), __ldg(L.shift + o), rt, L.zp_out, p.lo) : 0;
                            } else {
                                y[k] = requant1<kMode == 3 ? 2 : kMode == 2 ? 1 : 0, kClamp>(v, k4[k], rw, k, p.res_m2, p.res_r2, p.res_k8, p.lo);
                            }
                        }
                        w = pack4_sat(y[0], y[1], y[2], y[3]);
                    }
                }
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if ((uint32_t)(8 * i) < rem) st_global_v4(p.out + at + (size_t)(8 * i) * coutp, io[i]);
        }
        if (!ready) {                                                                   // fewer units than parts: let the tile go
            if (!__all_sync(0xffffffffu, wait_bar<kHintEpi>(bar_full, use & 1u, c.abort_flag))) return false;
            tc_fence_before();
            mbar_arrive(bar_free);
        }
    }
    return true;
}

// kWhole: input channels and output tiles are multiples of 64 (what the wide bottleneck networks consist of); the other
// form takes any layer.  Two kernels, because the general form's masks cost registers and a tenth of the speed.
// kPair: tiles of 256 pixels x 128 channels (see igemm_paired).  kCopy: operand rows by tensor copy (the general form
// looks at tma_a instead).
template <bool kWhole, bool kPair, bool kCopy>
__global__ void __launch_bounds__(igemm_threads(kWhole, kCopy), 1) k_igemm(const __grid_constant__ IgemmParams p)
{
    extern __shared__ __align__(128) uint8_t smem[];            // operand stages | requantisation constants | scratch of the general form's epilogue
    constexpr int kEpi = igemm_epi_warps(kWhole, kCopy), kGatherWarps = igemm_gather_warps(kWhole, kCopy), kGemmThreads = igemm_threads(kWhole, kCopy);
    constexpr int kGatherRows = kGatherWarps ? kTileM / kGatherWarps : 8;          // tile rows of a gather warp
    const bool copied = kWhole ? kCopy : p.tma_a != 0;
    __shared__ unsigned long long bar_full[kMaxStages], bar_free[kMaxStages], bar_acc_full[4], bar_acc_free[4];
    __shared__ uint32_t tmem_base_s;
    __shared__ volatile int abort_s;
    const GLayer &L = p.L;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t sbase = smem_u32(smem);
    const int n_tile = p.n_tile, stages = p.stages;
    constexpr uint32_t a_half = kTileM * kBlockK, a_bytes = kPair ? 2 * a_half : a_half;
    const uint32_t b_bytes = (uint32_t)n_tile * kBlockK, stage_bytes = a_bytes + b_bytes;
    int4 *cst_s = reinterpret_cast<int4 *>(smem + (size_t)stages * stage_bytes);
    if (tid == 0) {
        for (int s = 0; s < stages; ++s) { mbar_init(smem_u32(&bar_full[s]), copied ? 1 : kGatherWarps * 32 + 1); mbar_init(smem_u32(&bar_free[s]), 1); }
        for (int i = 0; i < p.n_acc; ++i) { mbar_init(smem_u32(&bar_acc_full[i]), 1); mbar_init(smem_u32(&bar_acc_free[i]), kEpi * 32 / p.n_acc); }
        abort_s = 0;
    }
    if (warp == 0) tmem_alloc(smem_u32(&tmem_base_s), (uint32_t)p.tmem_cols);
    for (int i = tid; i < p.tiles_n * n_tile; i += kGemmThreads) cst_s[i] = __ldg(p.cst + i);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_proxy_async();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    chain_start();
    const uint32_t tmem = tmem_base_s;
    chain_wait();

    // tiles in m-major order (the CTAs of one wave share operand rows in L2), dealt round-robin to the CTAs
    const int tiles_n = p.tiles_n;
    const uint32_t n_tiles = p.tiles_m * (uint32_t)tiles_n, grid_n = gridDim.x;
    const int cblocks = L.cinp / kBlockK, nkb = p.n_blocks;
    bool ok = true;

    if (warp < kEpi) {
        EpiCtx c;
        c.sbase = sbase; c.tmem = tmem; c.n_tiles = n_tiles; c.grid_n = grid_n; c.tiles_n = tiles_n; c.warp = warp; c.lane = lane;
        c.cst_s = smem_u32(cst_s);
        c.acc_full = smem_u32(&bar_acc_full[0]); c.acc_free = smem_u32(&bar_acc_free[0]);
        c.abort_flag = &abort_s;
        const bool fast = p.fast_requant && (!p.res || p.fast_residual), clamp = p.lo > -128;
        if constexpr (kWhole) {
            if (!kPair && !fast) ok = epilogue_whole<0, kPair, true, kEpi>(p, c);              // paired tiles take the 32-bit form only
            else if (p.res && p.res_short) ok = clamp ? epilogue_whole<3, kPair, true, kEpi>(p, c) : epilogue_whole<3, kPair, false, kEpi>(p, c);
            else if (p.res) ok = epilogue_whole<2, kPair, true, kEpi>(p, c);
            else ok = clamp ? epilogue_whole<1, kPair, true, kEpi>(p, c) : epilogue_whole<1, kPair, false, kEpi>(p, c);
        } else {
            if (fast && p.res && p.res_short) ok = epilogue_rows<3>(p, c);
            else if (fast && p.res) ok = epilogue_rows<2>(p, c);
            else if (fast) ok = epilogue_rows<1>(p, c);
            else ok = epilogue_rows<0>(p, c);
        }
    } else if (warp < kEpi + kGatherWarps) {
        // ---- operand rows: per reduction block a warp copies its tile rows x 64 bytes with asynchronous 16-byte
        // copies (lane = 16-byte column x row within a group of eight, so that an instruction reads whole
        // 64-byte rows) whose completion arrives on the stage's barrier.  A row outside the image is copied from a
        // 64-byte run of the input zero-point that follows the repacked weights, so every row takes the same path.
        const int gw = warp - kEpi, chunk = lane & 3, rsub = lane >> 2;
        const int8_t *zp_src = p.zp_run + chunk * 16;
        const int8_t *in_c = p.in + chunk * 16;
        // K-major core matrices: 16-byte column j of row r at j * (128 rows * 16) + r * 16
        const uint32_t dst0 = sbase + (uint32_t)chunk * 2048u + (uint32_t)(kGatherRows * gw + rsub) * 16u;
        Ring ring;
        const uint32_t px_per_sample = (uint32_t)(L.hout * L.wout);
        for (uint32_t t = blockIdx.x; t < n_tiles && ok && !copied; t += grid_n) {
            const uint32_t m0 = (t / (uint32_t)tiles_n) * kTileM + (uint32_t)(kGatherRows * gw + rsub);
            constexpr int kRows = kGatherRows / 8;
            int iy0[kRows], ix0[kRows], off[kRows];             // this lane's rows: 8 apart
#pragma unroll
            for (int i = 0; i < kRows; ++i) {
                const uint32_t m = m0 + 8u * (uint32_t)i;
                const bool valid = m < p.m_total;
                const uint32_t mm = valid ? m : 0u;
                const uint32_t b = mm / px_per_sample, pp = mm - b * px_per_sample;
                const int oy = (int)(pp / (uint32_t)L.wout), ox = (int)pp - oy * L.wout;
                iy0[i] = valid ? oy * L.stride - L.pad : -0x100000;             // an invalid row is outside for every tap
                ix0[i] = ox * L.stride - L.pad;
                off[i] = (((int)b * L.hin + oy * L.stride - L.pad) * L.win + ix0[i]) * L.cinp;    // the tensor is < 2^31 bytes
            }
            if (!kWhole) {
                // channels no multiple of 64: this lane's column of a block is a tap and 16 channels of its own; columns
                // beyond the last one meet zero weights
                const int c16s = L.cinp >> 4;
                int u = chunk, c16 = chunk % c16s, r = (chunk / c16s) / L.kw, sx = (chunk / c16s) % L.kw;
                for (int kb = 0; kb < nkb; ++kb, ring.advance(stages)) {
                    if (ring.use >= 1) {
                        ok = wait_bar<kHintLoad>(smem_u32(&bar_free[ring.s]), (uint32_t)(ring.use - 1) & 1u, &abort_s);
                        if (!ok) break;
                    }
                    const uint32_t dst = dst0 + (uint32_t)ring.s * stage_bytes;
                    const int add = (r * L.win + sx) * L.cinp + c16 * 16;
#pragma unroll
                    for (int i = 0; i < kRows; ++i) {
                        const bool inside = (unsigned)(iy0[i] + r) < (unsigned)L.hin && (unsigned)(ix0[i] + sx) < (unsigned)L.win && u < p.units;
                        cp_async16_cached(dst + (uint32_t)i * 128u, inside ? p.in + (off[i] + add) : zp_src);
                    }
                    cp_async_arrive(smem_u32(&bar_full[ring.s]));
                    u += 4; c16 += 4;
                    while (c16 >= c16s) {
                        c16 -= c16s;
                        if (++sx == L.kw) { sx = 0; ++r; }
                    }
                }
                continue;
            }
            for (int tap = 0, r = 0, sx = 0; tap < L.kh * L.kw && ok; ++tap, sx = (sx + 1 == L.kw) ? 0 : sx + 1, r += (sx == 0)) {
                const int tap_off = (r * L.win + sx) * L.cinp;
                bool inside[kRows];
#pragma unroll
                for (int i = 0; i < kRows; ++i) inside[i] = (unsigned)(iy0[i] + r) < (unsigned)L.hin && (unsigned)(ix0[i] + sx) < (unsigned)L.win;
                for (int cb = 0; cb < cblocks; ++cb, ring.advance(stages)) {
                    if (ring.use >= 1) {
                        ok = wait_bar<kHintLoad>(smem_u32(&bar_free[ring.s]), (uint32_t)(ring.use - 1) & 1u, &abort_s);
                        if (!ok) break;
                    }
                    const uint32_t dst = dst0 + (uint32_t)ring.s * stage_bytes;
#pragma unroll
                    for (int i = 0; i < kRows; ++i) {
                        cp_async16_cached(dst + (uint32_t)i * 128u, inside[i] ? in_c + (off[i] + tap_off + cb * kBlockK) : zp_src);
                    }
                    cp_async_arrive(smem_u32(&bar_full[ring.s]));
                }
            }
        }
        cp_async_wait_all();
    } else if (warp == kEpi + kGatherWarps) {
        // ---- one thread issues the MMAs: two K-steps per stage, accumulators alternate between two column ranges
        if (lane == 0) {
            const uint32_t idesc = (2u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n_tile >> 3) << 17) | ((uint32_t)(kTileM >> 4) << 24);
            Ring ring;
            int j = 0;
            for (uint32_t t = blockIdx.x; t < n_tiles && ok; t += grid_n, ++j) {
                const int buf = j & (p.n_acc - 1), au = p.n_acc == 4 ? j >> 2 : j >> 1;
                if (au >= 1) {
                    ok = wait_bar<kHintMma>(smem_u32(&bar_acc_free[buf]), (uint32_t)(au - 1) & 1u, &abort_s);
                    if (!ok) break;
                }
                for (int kb = 0; kb < nkb; ++kb, ring.advance(stages)) {
                    ok = wait_bar<kHintMma>(smem_u32(&bar_full[ring.s]), (uint32_t)ring.use & 1u, &abort_s);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t stage = sbase + (uint32_t)ring.s * stage_bytes;
#pragma unroll
                    for (int k2 = 0; k2 < 2; ++k2) {
                        if (!kWhole && k2 == 1 && 4 * kb + 2 >= p.units) break;            // the last block's second half is padding
                        const uint64_t ad = make_desc(stage + (uint32_t)k2 * 4096u, 2048u, 128u);
                        const uint64_t bd = make_desc(stage + a_bytes + (uint32_t)k2 * 2u * (uint32_t)n_tile * 16u, (uint32_t)n_tile * 16u, 128u);
                        mma_i8(tmem + (uint32_t)(buf * p.acc_stride), ad, bd, idesc, (kb > 0 || k2 > 0) ? 1u : 0u);
                        if (kPair) mma_i8(tmem + (uint32_t)(buf * p.acc_stride + kPairN), ad + (uint64_t)(a_half >> 4), bd, idesc, (kb > 0 || k2 > 0) ? 1u : 0u);
                    }
                    commit_to(smem_u32(&bar_free[ring.s]));
                }
                if (ok) commit_to(smem_u32(&bar_acc_full[buf]));
            }
        }
        __syncwarp();
    } else {
        // ---- one thread streams the repacked weights: one bulk copy per block into the stage's second part
        if (lane == 0 && !p.debug_stall) {
            Ring ring;
            for (uint32_t t = blockIdx.x; t < n_tiles && ok; t += grid_n) {
                // the tile's residual bytes, about a tile ahead of their use (258 -> 253 us)
                if (kWhole && p.prefetch_res)
                    asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];"
                                 ::"l"(reinterpret_cast<uint64_t>(&p.tmap_res)), "r"((int)(t % (uint32_t)tiles_n) * n_tile), "r"((int)(t / (uint32_t)tiles_n) * (kPair ? 2 * kTileM : kTileM)) : "memory");
                const int8_t *wtile = p.wpack + (size_t)(t % tiles_n) * (size_t)nkb * b_bytes;
                for (int kb = 0; kb < nkb; ++kb, ring.advance(stages)) {
                    if (ring.use >= 1) {
                        ok = wait_bar<kHintLoad>(smem_u32(&bar_free[ring.s]), (uint32_t)(ring.use - 1) & 1u, &abort_s);
                        if (!ok) break;
                    }
                    mbar_expect_tx(smem_u32(&bar_full[ring.s]), copied ? a_bytes + b_bytes : b_bytes);
                    if (copied) {
                        // box {16 bytes, 128 pixels, 4 columns} of the 3-D view lands as [column][pixel][16 bytes], which is
                        // the K-major core-matrix layout; pixels beyond the last one are filled with zeros and never stored
#pragma unroll
                        for (int mt = 0; mt < (kPair ? 2 : 1); ++mt)
                            asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
                                         ::"r"(sbase + (uint32_t)ring.s * stage_bytes + (uint32_t)mt * a_half), "l"(reinterpret_cast<uint64_t>(&p.tmap_a)), "r"(0),
                                           "r"((int)((t / (uint32_t)tiles_n) * (kPair ? 2 * kTileM : kTileM)) + mt * kTileM), "r"(kb * 4),
                                           "r"(smem_u32(&bar_full[ring.s])) : "memory");
                    }
                    bulk_g2s(sbase + (uint32_t)ring.s * stage_bytes + a_bytes, wtile + (size_t)kb * b_bytes, b_bytes, smem_u32(&bar_full[ring.s]));
                }
            }
            if (!ok) {
                // copies already issued may still be landing in this CTA's shared memory: give them time before the exit
                const unsigned long long t0 = globaltimer();
                while (globaltimer() - t0 < 50000ull) __nanosleep(1000);
            }
        }
        __syncwarp();
    }
    if (!ok) {
        if (!abort_s) atomicCAS(p.err, 0, 1 + (int)blockIdx.x);
        abort_s = 1;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    __syncwarp();                                         // lanes that gave up a wait on their own meet again
    if (warp == 0) tmem_dealloc(tmem, (uint32_t)p.tmem_cols);
}


// ------------------------------------------------------------------ first convolution on the tensor cores
//
// The stem of a network whose input is the noisy image (Def. 3.4): a k x k convolution over <= 4 input channels.
// A piece of work is one sample x one band of output rows; a CTA takes every grid-th (with a CTA for each, the set-up, the
// weights and the noise tables' copy were a sixth of a small image's time: 3 x 3 on 32 x 32, 5,100 samples: 388 -> 330 us).  The band's input rows are drawn (Philox -> inverse-CDF table ->
// add -> saturate to 0..255, Def. 3.3 / Eq. 2) into a shared-memory patch as 4 bytes per pixel, padded with the input
// zero-point, and never written to memory.  The GEMM takes one filter row per K-step: eight horizontally adjacent
// pixels x 4 bytes = 32 bytes of K (pixels beyond the filter width meet zero weights), so 128 output pixels are `kh`
// MMAs.  The patch is spread once into positions of 16 bytes, position i of a row being the four pixels from i * stride
// on, with the rows ordered by (row mod stride, row / stride): output pixel (y, x) then reads filter row r at position
// r's first + y * pitch + x, and a filter row is an address offset of the operand descriptor (the second 16 bytes of K
// lie 4 / stride positions on, or in a second plane when that is no whole number).  Copying each output pixel's kh
// windows into an operand stage moved five times as many bytes and put a CTA barrier before every tile.  A tile is
// 256 positions (two M operands), so that a thread requantises two rows and reads a channel's constants once for both;
// the positions behind a row's last pixel are computed and not stored.  A ninth warp issues the MMAs.  7 x 7 stride 2 on
// 224 x 224, 512 samples: 833 -> 640 us with the table of bins (the search by guide and bisection took 260 of them: two loads
// and two for each step, of 32 lanes from as many places, which is bank conflicts); of what is left the Philox rounds take
// some 70, the search as much, the epilogue 95 and the copy to positions 47, the rest is the patch and the barriers.
struct StemParams {
    GLayer L;
    int in_c, band_rows, n_bands, tmem_cols;
    uint32_t n_items;                        // samples * bands
    int pitch, rows_class, planes;           // positions of a row; rows of one (row mod stride) class; planes of positions
    uint32_t plane_pos, k_step;              // positions of a plane; bytes from the first to the second 16 bytes of K
    uint32_t w_bytes, pos_off, patch_off;
    int slots;                               // pairs of accumulators in tensor memory
    uint32_t tab_off;                        // the noise tables' copy in shared memory (after the patch), 0: searched in global memory
    int tab_words, bin_bits;                 // of the copy; bits of the bins if they are what is copied, else 0
    const uint8_t *x;                        // clean images, CHW, one after the other
    NoiseStream ns;                          // the counter's words come from `run`
    const int8_t *wpack;                     // [filter row][2 K columns][coutp rows][16 bytes]
    const int4 *cst;
    int fast_requant, lo;
    int debug_stall;                         // test hook: the weights are never sent, so that the kernel's waits run out
    int8_t *out;
    int32_t *err;
    SampleRun run;
};

// Rows 32 (warp mod 4) .. + 31 of both operands of every tile, half of the channels.
template <bool kFast, bool kClamp>
__device__ __forceinline__ bool stem_epilogue(const StemParams &p, uint32_t tmem, uint32_t cst, uint32_t bar_full, uint32_t bar_free, uint32_t first_tile, int n_tiles,
                                              int band_rows, size_t first_px, const volatile int *abort_flag)
{
    const GLayer &L = p.L;
    const int N = L.coutp, row = (int)threadIdx.x & (kTileM - 1), half = (N / 16 + 1) / 2 * 16;
    const int c_begin = threadIdx.x >= kTileM ? half : 0, c_end = threadIdx.x >= kTileM ? N : half;
    const uint32_t lanes = tmem + ((uint32_t)(row & ~31) << 16);
    for (int t = 0; t < n_tiles; ++t) {
        const uint32_t tile = first_tile + (uint32_t)t, slot = p.slots == 2 ? tile & 1u : 0u, use = p.slots == 2 ? tile >> 1 : tile;
        int8_t *dst[2];
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) {
            const int f = t * 2 * kTileM + mt * kTileM + row, y = f / p.pitch, x = f - y * p.pitch;
            dst[mt] = y < band_rows && x < L.wout ? p.out + (first_px + (size_t)(y * L.wout + x)) * L.coutp : nullptr;
        }
        if (!wait_bar<kHintEpi>(bar_full + 8u * slot, use & 1u, abort_flag)) return false;
        tc_fence_after();
        const uint32_t acc = lanes + slot * (uint32_t)(2 * N);
#pragma unroll 1
        for (int c0 = c_begin; c0 < c_end; c0 += 16) {
            int a[2][16];
            tmem_ld16_issue(acc + (uint32_t)c0, a[0]);
            tmem_ld16_issue(acc + (uint32_t)(N + c0), a[1]);
            tmem_ld32_wait(a);
            uint4 o[2];
            if (kFast) {
                const uint32_t none[4] = {0, 0, 0, 0};
                requant16x2<0, kClamp>(a, cst + (uint32_t)c0 * 16u, none, none, 0u, 0ll, 0u, p.lo, o);
            } else {
#pragma unroll
                for (int mt = 0; mt < 2; ++mt) {
#pragma unroll
                    for (int k = 0; k < 16; ++k) a[mt][k] += __ldg(L.bias + c0 + k);
                    o[mt] = epilogue16(a[mt], L, c0, nullptr);
                }
            }
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
                if (dst[mt]) *reinterpret_cast<uint4 *>(dst[mt] + c0) = o[mt];
        }
        tc_fence_before();
        mbar_arrive(bar_free + 8u * slot);
    }
    return true;
}

__global__ void __launch_bounds__(kStemThreads, 2) k_stem(const __grid_constant__ StemParams p)
{
    extern __shared__ __align__(128) uint8_t smem[];        // weights | positions | patch | noise tables
    __shared__ unsigned long long bar_w, bar_full[2], bar_free[2];
    __shared__ uint32_t tmem_base_s;
    __shared__ volatile int abort_s;
    __shared__ __align__(16) int4 cst_s[256];
    const GLayer &L = p.L;
    const int tid = threadIdx.x, warp = (int)warp_uniform((uint32_t)tid >> 5);
    const uint32_t sbase = smem_u32(smem);
    const int N = L.coutp, kh = L.kh;
    if (tid == 0) {
        mbar_init(smem_u32(&bar_w), 1);
        for (int i = 0; i < 2; ++i) { mbar_init(smem_u32(&bar_full[i]), 1); mbar_init(smem_u32(&bar_free[i]), 2 * kTileM); }
        abort_s = 0;
    }
    if (warp == 0) tmem_alloc(smem_u32(&tmem_base_s), (uint32_t)p.tmem_cols);
    for (int i = tid; i < N; i += kStemThreads) cst_s[i] = __ldg(p.cst + i);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_proxy_async();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    chain_start();
    const uint32_t tmem = tmem_base_s;
    if (tid == 0 && !p.debug_stall) {
        mbar_expect_tx(smem_u32(&bar_w), p.w_bytes);
        bulk_g2s(sbase, p.wpack, p.w_bytes, smem_u32(&bar_w));
    }

    uint32_t *patch = reinterpret_cast<uint32_t *>(smem + p.patch_off);
    const uint32_t zp_fill = (uint32_t)(L.zp_in & 0xFF) * (0x01010101u >> (8 * (4 - p.in_c)));
    if (p.tab_off) {
        // the bins, or the cumulative table and the guide table that follows it in memory
        const uint32_t *from = p.bin_bits ? reinterpret_cast<const uint32_t *>(p.ns.bins) : p.ns.cum;
        uint32_t *tab = reinterpret_cast<uint32_t *>(smem + p.tab_off);
        for (int i = tid; i < p.tab_words; i += kStemThreads) tab[i] = __ldg(from + i);
    }
    // the levels of a Philox block's four uniforms
    auto levels4 = [&](uint4 r, int (&z)[4]) {
        if (p.bin_bits) {
            if (noise_levels4_bins(r, sbase + p.tab_off, nullptr, p.bin_bits, z)) return;
        } else if (p.tab_off) {
            return noise_levels4_shared(r, sbase + p.tab_off, sbase + p.tab_off + 4u * (uint32_t)(2 * p.ns.T + 1), p.ns.T, p.ns.guide_steps, z);
        }
        noise_levels4(r, p.ns.cum, p.ns.guide, p.ns.T, p.ns.guide_steps, z);
    };
    bool ok = true;
    uint32_t first_tile = 0;                                    // of the item, counted over the CTA's items
    for (uint32_t item = blockIdx.x; item < p.n_items; item += gridDim.x) {
        // ---- the band's noisy input rows
        const uint32_t b = item / (uint32_t)p.n_bands, band = item - b * (uint32_t)p.n_bands;
        const SampleRun::Sample sample = p.run.at(b);
        const int64_t j = (int64_t)sample.number;
        const uint64_t image_id = p.run.image_id0 + sample.image;
        const uint32_t ctr2 = (uint32_t)image_id;
        const uint8_t *x = p.x + sample.image * (size_t)(p.in_c * L.hin * L.win);
        const int oy0 = (int)band * p.band_rows, oy1 = min(L.hout, oy0 + p.band_rows);
        const int wpad = L.win + 2 * L.pad + 8;                     // 8 more pixels: the windows of the last columns stay inside
        const int iy0 = oy0 * L.stride - L.pad;
        const int rows_in = (oy1 - oy0 - 1) * L.stride + kh;
        for (int i = tid; i < rows_in * wpad; i += kStemThreads) patch[i] = zp_fill;
        __syncthreads();
        const int vy0 = max(0, iy0), vy1 = min(L.hin, iy0 + rows_in);
        if (vy1 > vy0) {
            uint8_t *pb = reinterpret_cast<uint8_t *>(patch);
            const uint32_t ctr3 = sample.phase | ((uint32_t)(image_id >> 32) & 0xFFFFu) << 16 | (uint32_t)(((j >> 32) & 0xFF) << 8);
            const uint32_t ctr1 = (uint32_t)(j & 0xFFFFFFFFll);
            if ((L.win & 3) == 0 && p.ns.guide) {
                // every Philox block (four consecutive elements of the CHW order) lies within one image row: a thread
                // takes whole blocks, all channels of the band's rows as one index space, the four searches interleaved
                const int qpr = L.win >> 2, qpc = (vy1 - vy0) * qpr;
                for (int i = tid; i < p.in_c * qpc; i += kStemThreads) {
                    const int c = i / qpc, ic = i - c * qpc;
                    const int hr = ic / qpr, wq = ic - hr * qpr;
                    const int h = vy0 + hr;
                    const uint32_t e = (uint32_t)((c * L.hin + h) * L.win) + 4u * (uint32_t)wq;
                    const uint4 r = philox4x32_10(make_uint4(e >> 2, ctr1, ctr2, ctr3), p.ns.key0, p.ns.key1);
                    const uint32_t clean = __ldg(reinterpret_cast<const uint32_t *>(x + e));
                    int z[4];
                    levels4(r, z);
                    uint8_t *dst = pb + ((h - iy0) * wpad + (4 * wq + L.pad)) * 4 + c;
#pragma unroll
                    for (int k = 0; k < 4; ++k) dst[4 * k] = (uint8_t)min(255, max(0, (int)((clean >> (8 * k)) & 0xFFu) + z[k]));
                }
            } else {
                // any width: a block's elements may lie in two rows, and its first and last in another band or channel
                const int rows = vy1 - vy0, blocks = (rows * L.win + 3) / 4 + 1;                  // of a channel, at most
                for (int i = tid; i < p.in_c * blocks; i += kStemThreads) {
                    const int c = i / blocks;
                    const int64_t e_begin = ((int64_t)c * L.hin + vy0) * L.win, q = (e_begin >> 2) + (i - c * blocks);
                    int at = (int)(4 * q - e_begin);                                             // of the block's first element among the band's
                    if (at >= rows * L.win) continue;
                    const uint4 r = philox4x32_10(make_uint4((uint32_t)q, ctr1, ctr2, ctr3), p.ns.key0, p.ns.key1);
                    int z[4];
                    if (p.ns.guide) {
                        levels4(r, z);
                    } else {
                        const uint32_t u[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
                        for (int k = 0; k < 4; ++k) z[k] = noise_level(u[k], p.ns.cum, p.ns.T);
                    }
                    int h = at < 0 ? 0 : at / L.win, w = at - h * L.win;                          // (negative before the band's first element)
#pragma unroll
                    for (int k = 0; k < 4; ++k, ++at, ++w) {
                        if (w == L.win) { w = 0; ++h; }
                        if (at < 0 || at >= rows * L.win) continue;
                        const int v = min(255, max(0, (int)__ldg(x + e_begin + at) + z[k]));
                        pb[((vy0 + h - iy0) * wpad + (w + L.pad)) * 4 + c] = (uint8_t)v;
                    }
                }
            }
        }
        __syncthreads();

        // ---- the patch as positions (see above)
        const uint32_t pos = sbase + p.pos_off;
        for (int i = tid; i < p.planes * rows_in * p.pitch; i += kStemThreads) {
            int y = i / p.pitch;
            const int x = i - y * p.pitch, plane = y >= rows_in ? 1 : 0;
            y -= plane * rows_in;
            const uint32_t *src = patch + y * wpad + x * L.stride + 4 * plane;
            const int at = (y % L.stride * p.rows_class + y / L.stride) * p.pitch + x;
            st_shared_v4(pos + ((uint32_t)plane * p.plane_pos + (uint32_t)at) * 16u, make_uint4(src[0], src[1], src[2], src[3]));
        }
        fence_proxy_async();
        __syncthreads();

        if (first_tile == 0) chain_wait();                    // the noise needed nothing of the launch before; the output buffer does
        const int band_rows = oy1 - oy0, n_tiles = (band_rows * p.pitch + 2 * kTileM - 1) / (2 * kTileM);
        if (warp < kStemEpi) {
            const size_t first_px = ((size_t)b * L.hout + oy0) * L.wout;
            const uint32_t cst = smem_u32(cst_s), full = smem_u32(&bar_full[0]), free_ = smem_u32(&bar_free[0]);
            if (!p.fast_requant) ok = stem_epilogue<false, true>(p, tmem, cst, full, free_, first_tile, n_tiles, band_rows, first_px, &abort_s);
            else if (p.lo > -128) ok = stem_epilogue<true, true>(p, tmem, cst, full, free_, first_tile, n_tiles, band_rows, first_px, &abort_s);
            else ok = stem_epilogue<true, false>(p, tmem, cst, full, free_, first_tile, n_tiles, band_rows, first_px, &abort_s);
        } else {
            const uint32_t lane0 = elect_one() ? 1u : 0u;
            const uint32_t idesc = (2u << 4) | (0u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(kTileM >> 4) << 24);
            if (first_tile == 0) ok = wait_warp(smem_u32(&bar_w), 0u, &abort_s);
            tc_fence_after();
            for (int t = 0; t < n_tiles && ok; ++t) {
                const uint32_t tile = first_tile + (uint32_t)t, slot = p.slots == 2 ? tile & 1u : 0u, use = p.slots == 2 ? tile >> 1 : tile;
                if (use >= 1) {
                    ok = wait_warp(smem_u32(&bar_free[slot]), (use - 1u) & 1u, &abort_s);
                    if (!ok) break;
                    tc_fence_after();
                }
                for (int mt = 0; mt < 2; ++mt)
                    for (int r = 0; r < kh; ++r) {
                        const int at = (r % L.stride * p.rows_class + r / L.stride) * p.pitch + t * 2 * kTileM + mt * kTileM;
                        const uint64_t ad = make_desc(pos + (uint32_t)at * 16u, p.k_step, 128u);
                        const uint64_t bd = make_desc(sbase + (uint32_t)r * 2u * (uint32_t)N * 16u, (uint32_t)N * 16u, 128u);
                        mma_i8_if(lane0, tmem + (slot * 2u + (uint32_t)mt) * (uint32_t)N, ad, bd, idesc, r > 0 ? 1u : 0u);
                    }
                commit_if(lane0, smem_u32(&bar_full[slot]));
            }
        }
        first_tile += (uint32_t)n_tiles;
        if (!ok) abort_s = 1;
        // the item's MMAs are complete (their accumulators have been read): the next one may overwrite positions and patch
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        if (abort_s) break;
    }
    if (!ok) abort_s = 1;
    if (!ok) atomicCAS(p.err, 0, 1 + (int)blockIdx.x);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    __syncwarp();                                         // lanes that gave up a wait on their own meet again
    if (warp == 0) tmem_dealloc(tmem, (uint32_t)p.tmem_cols);
}

}  // namespace

// ------------------------------------------------------------------ host side

namespace {

// Paired tiles are 128 channels wide, and an MMA of that width reads its operands at the shared memory's full bandwidth.
// That pays where there are no more than 128 channels (the tile is as wide anyway) and in short reductions, where the
// epilogue's constants weigh more (512 -> 256 channels at 28 x 28 became 84 -> 121 us, 512 -> 2048 at 7 x 7 57 -> 76 us).
bool igemm_pairable(const GLayer &G)
{
    return G.kh == 1 && G.kw == 1 && G.stride == 1 && G.pad == 0 && G.cinp % kBlockK == 0 && G.coutp % kPairN == 0 &&
           (G.coutp == kPairN || G.cinp <= 128);
}

// Whether a launch of `tiles_m` x `tiles_n` single tiles, which the CTAs take in rounds, pairs them: unless the coarser
// rounds would cost more than the cheaper epilogue saves (a fifth).
bool igemm_paired(uint32_t tiles_m, uint32_t tiles_n, uint32_t n_sms)
{
    const uint32_t single = (tiles_m * tiles_n + n_sms - 1) / n_sms, pairs = ((tiles_m + 1) / 2 * tiles_n + n_sms - 1) / n_sms;
    return 8 * pairs <= 5 * single;
}

}  // namespace

// Output channels in as few tiles of at most 256 as possible, all of the same width (a multiple of 16; the last one may
// be partly padding).
// A 1 x 1 stride-1 layer for which paired tiles pay has tiles of 128, whether a launch pairs them or not.
int igemm_tile_n(const GLayer &G)
{
    if (igemm_pairable(G)) return kPairN;
    const int tiles = (G.coutp + 255) / 256;
    return ((G.coutp + tiles - 1) / tiles + 15) & ~15;
}

namespace {

// Whole tiles: input channels and the output channels' tiles are multiples of 64.
bool igemm_whole(const GLayer &G) { return G.cinp % kBlockK == 0 && igemm_tile_n(G) % 64 == 0 && G.coutp % igemm_tile_n(G) == 0; }

// The output channel of a column of the accumulators: in whole tiles, column 16 t + 8 h + 2 c + e of 64 is channel
// 16 c + 4 t + 2 h + e (see epilogue_whole).
int igemm_channel(const GLayer &G, int col)
{
    if (!igemm_whole(G)) return col;
    return (col & ~63) | ((col & 6) << 3) | ((col & 48) >> 2) | ((col & 8) >> 2) | (col & 1);
}

int igemm_tiles(const GLayer &G) { return igemm_pairable(G) ? G.coutp / kPairN : (G.coutp + 255) / 256; }
int igemm_units(const GLayer &G) { return G.kh * G.kw * (G.cinp / 16); }
int igemm_blocks(const GLayer &G) { return (igemm_units(G) + 3) / 4; }

// Dynamic shared memory of a launch: the constants of every output channel, the epilogue warps' scratch, and operand
// stages, of which two are needed at least.
constexpr size_t kSmemLimit = 226 * 1024;
struct IgemmSmem {
    size_t cst, scratch, stage;
    bool fits() const { return cst + scratch + 2 * stage <= kSmemLimit; }
};
IgemmSmem igemm_smem(const GLayer &G, bool paired)
{
    const size_t n_tile = (size_t)igemm_tile_n(G), rows = paired ? 2 : 1;
    return IgemmSmem{(size_t)igemm_tiles(G) * n_tile * 16, (size_t)kRowWarps * 32 * rows * epi_row_stride((int)n_tile),
                     (size_t)kTileM * kBlockK * rows + n_tile * kBlockK};
}

}  // namespace

// Convolutions and FC layers whose constants leave room for the operands: up to 6,912 output channels in tiles of 256,
// 10,112 in tiles of 128.  Wider ones stay on the plain kernel.
bool igemm_takes(const GLayer &G) { return (G.op == ISC_CONV2D || G.op == ISC_FC) && igemm_smem(G, false).fits(); }

// constants of that many channels: the last tile's padding included
int igemm_padded_cout(const GLayer &G) { return igemm_tiles(G) * igemm_tile_n(G); }

// the repacked weights, then 64 bytes of the input zero-point (the operand row of a pixel outside the image)
size_t igemm_pack_bytes(const GLayer &G)
{
    return (size_t)igemm_padded_cout(G) * (size_t)igemm_blocks(G) * kBlockK + kBlockK;
}

// w: [cout][cin][kh][kw] as the model gives it -> [cout tile][block][4 columns][n_tile rows][16]; column u of the
// reduction is 16 input channels of one filter tap, tap-major
void igemm_pack_weights(const GLayer &G, const int8_t *w, int8_t *out)
{
    const int n_tile = igemm_tile_n(G), taps = G.kh * G.kw, c16s = G.cinp / 16, units = igemm_units(G), columns = 4 * igemm_blocks(G);
    std::vector<int> channel((size_t)n_tile);                   // (worked out for each byte, ResNet-50 took twice as long to load)
    for (int n = 0; n < n_tile; ++n) channel[(size_t)n] = igemm_channel(G, n);
    size_t at = 0;
    for (int t = 0; t < igemm_tiles(G); ++t)
        for (int u = 0; u < columns; ++u) {
            const int tap = u / c16s, c0 = (u - tap * c16s) * 16;
            for (int n = 0; n < n_tile; ++n)
                for (int e = 0; e < 16; ++e, ++at) {
                    const int oc = t * n_tile + channel[(size_t)n], ci = c0 + e;
                    out[at] = (u < units && oc < G.cout && ci < G.cin) ? w[((size_t)oc * G.cin + ci) * taps + tap] : (int8_t)0;
                }
        }
    for (int e = 0; e < kBlockK; ++e) out[at + e] = (int8_t)G.zp_in;
}

// The constants of igemm_constants in the order in which the kernel reads them: the four of channels 16 c + 4 t + k, c = 0 to 3, of
// 64 lie side by side.
void igemm_order_constants(const GLayer &G, int32_t *out4, int n_out)
{
    if (!igemm_whole(G)) return;
    const std::vector<int32_t> in(out4, out4 + 4 * (size_t)n_out);
    for (int o = 0; o < n_out; ++o) {
        const int at = (o & ~63) | (o & 15) << 2 | ((o >> 4) & 3);
        memcpy(out4 + 4 * (size_t)at, &in[4 * (size_t)o], 16);
    }
}

// 32-bit row and byte offsets inside the tensor-core kernels
bool conv_offsets_fit(const GLayer &G, int64_t batch)
{
    return batch * G.hout * G.wout * ((G.coutp + 255) / 256) < (1ll << 31) - 512 && batch * G.hin * G.win * G.cinp < (1ll << 31);
}

// The residual term F(u) = floor((u * m2 + R2) / 2^32), u = r + 128 in 0..255 (see requant16_fast), as
// hi32((256 k + u) * m2) - c: the smallest k < 4096 for which the two agree on all 256 inputs, or false.
ResidualForm residual_form(int res_mult, int res_shift, int zp_res, int32_t *c_out)
{
    ResidualForm f;
    const int n = 31 - res_shift;
    if ((n != 31 && n != 32) || res_mult < (1 << 30)) return f;
    // res_mult / 2^n = mant * 2^-e with a mantissa of 24 bits, and the numbers next to it
    const int64_t nearest = ((int64_t)res_mult + 64) >> 7;                     // 2^23 .. 2^24
    const int e = n - 7;
    for (int64_t mant : {nearest, nearest + 1, nearest - 1}) {
        if (mant < (1 << 23) || mant > (1 << 24)) continue;
        for (uint32_t k = 0; k < 4096; ++k) {
            int64_t c = 0;
            bool same = true;
            for (int u = 0; u < 256 && same; ++u) {
                const int64_t want = ((int64_t)(u - 128 - zp_res) * res_mult + (1ll << (n - 1))) >> n;      // arithmetic shift: floor
                const int64_t x = (int64_t)(256u * k + (uint32_t)u) * mant, q = x >> e, r = x & ((1ll << e) - 1), half = 1ll << (e - 1);
                const int64_t got = q + (r > half || (r == half && (q & 1)) ? 1 : 0);
                if (u == 0) c = got - want;
                same = got - want == c;
            }
            if (!same) continue;
            const float m = (float)ldexp((double)mant, -e);
            f.k8 = k << 8;
            memcpy(&f.m_bits, &m, sizeof(m));
            *c_out = (int32_t)c;
            return f;
        }
    }
    return f;
}

// Per output channel {folded bias, multiplier, rounding addend, shift - 1}; returns whether the layer has the 32-bit form:
// every shift is >= 2 and every addend leaves room for the product (shifts up to 24 whatever the zero-point).  `bias_folded`, `mult`, `shift` are the layer's host arrays padded to coutp.  For a
// layer with a residual operand whose term is a single-precision product, that product's constant is folded into the
// rounding addends.
bool igemm_constants(const GLayer &G, const int32_t *bias_folded, const int32_t *mult, const int32_t *shift, int32_t *out4, int n_out,
                     bool has_residual, ResidualForm *form)
{
    // channels beyond the layer's own (padding of the tensor and of the last tile) come out as zero
    auto addend = [&](int o, int32_t c) { return (1ll << (shift[o] - 2)) + ((long long)G.zp_out - c) * (1ll << (shift[o] - 1)); };
    bool fast = true;
    for (int o = 0; o < G.cout; ++o) fast = fast && shift[o] >= 2 && requant_addend_fits(addend(o, 0));
    int32_t c_res = 0;
    ResidualForm f;
    if (fast && has_residual) f = residual_form(G.res_mult, G.res_shift, G.zp_res, &c_res);
    bool short_form = f.exists();
    for (int o = 0; o < G.cout && short_form; ++o) short_form = requant_addend_fits(addend(o, c_res));
    if (!short_form) c_res = 0;
    if (form) *form = short_form ? f : ResidualForm();
    memset(out4, 0, sizeof(int32_t) * 4 * (size_t)n_out);
    for (int o = 0; o < G.cout && fast; ++o) {                  // (the 64-bit form does not read them)
        out4[4 * o + 0] = bias_folded[o];
        out4[4 * o + 1] = mult[o];
        out4[4 * o + 2] = (int32_t)addend(o, c_res);
        out4[4 * o + 3] = shift[o] - 1;
    }
    return fast;
}

typedef CUresult (*EncodeFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                             const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

cudaError_t tc_prepare(TcDevice *dev, int ordinal)
{
    TcDevice d;
    d.ordinal = ordinal;
    int major = 0;
    d.chained = cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, ordinal) == cudaSuccess && major >= 9;
    cudaError_t e = cudaDeviceGetAttribute(&d.n_sms, cudaDevAttrMultiProcessorCount, ordinal);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_igemm<true, true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemLimit);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_igemm<true, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemLimit);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_igemm<true, false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemLimit);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_igemm<false, false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemLimit);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_stem, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kStemSmemLimit);
    if (e == cudaSuccess) e = halo_prepare();
    if (e != cudaSuccess) { cudaGetLastError(); return e; }
    void *fn = nullptr;
    cudaDriverEntryPointQueryResult qr;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qr) == cudaSuccess && qr == cudaDriverEntryPointSuccess) d.encode = fn;
    else cudaGetLastError();
    *dev = d;
    return cudaSuccess;
}

cudaError_t launch_igemm_conv(const TcDevice &dev, const GLayer &G, const int8_t *wpack, const int32_t *cst, bool fast, const ResidualForm &form, int batch, const int8_t *in,
                              const int8_t *res, int8_t *out, int32_t *err, cudaStream_t st, bool debug_stall, bool tensor_copy)
{
    IgemmParams p;
    p.L = G;
    p.cst = reinterpret_cast<const int4 *>(cst);
    p.fast_requant = fast ? 1 : 0;
    p.lo = G.relu ? (G.zp_out > -128 ? G.zp_out : -128) : -128;
    const int res_n = 31 - G.res_shift;
    p.fast_residual = (res_n == 31 || res_n == 32) ? 1 : 0;
    p.debug_stall = debug_stall ? 1 : 0;
    // A 1 x 1 stride-1 layer reads its input as the matrix [pixel][channel]: the tile's operand rows are a box of the
    // view (16 bytes, pixel, 16-byte column) and come by tensor copy.  Without the driver's encoder (or if it refuses the
    // view) the gather warps do the work.
    p.tma_a = 0;
    memset(&p.tmap_a, 0, sizeof(p.tmap_a));
    if (tensor_copy && G.kh == 1 && G.kw == 1 && G.stride == 1 && G.pad == 0) {
        if (const EncodeFn encode = (EncodeFn)dev.encode) {
            const cuuint64_t dims[3] = {16, (cuuint64_t)batch * G.hin * G.win, (cuuint64_t)(G.cinp / 16)};
            const cuuint64_t strides[2] = {(cuuint64_t)G.cinp, 16};
            const cuuint32_t box[3] = {16, (cuuint32_t)kTileM, (cuuint32_t)(kBlockK / 16)}, estr[3] = {1, 1, 1};
            const CUresult r = encode(&p.tmap_a, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, const_cast<int8_t *>(in), dims, strides, box, estr,
                                      CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                                      CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
            if (r == CUDA_SUCCESS) p.tma_a = 1;
            else if (getenv("ISC_DEBUG_CUDA")) fprintf(stderr, "isc: cuTensorMapEncodeTiled: %d\n", (int)r);
        }
    }
    p.res_m2 = 0; p.res_r2 = 0;
    p.res_short = res && form.exists() ? 1 : 0;
    p.res_k8 = p.res_short ? form.k8 : 0u;
    if (p.res_short) {
        p.res_m2 = form.m_bits;
    } else if (res && p.fast_residual) {
        p.res_m2 = (uint32_t)((unsigned long long)(uint32_t)G.res_mult << (32 - res_n));
        p.res_r2 = ((1ll << (res_n - 1)) - (128ll + G.zp_res) * (long long)G.res_mult) * (1ll << (32 - res_n));
    }
    p.batch = batch;
    if (!igemm_takes(G) || !conv_offsets_fit(G, batch)) return cudaErrorInvalidValue;
    p.n_tile = igemm_tile_n(G);
    p.tiles_n = igemm_tiles(G);
    p.units = igemm_units(G);
    p.n_blocks = igemm_blocks(G);
    p.zp_run = wpack + igemm_pack_bytes(G) - kBlockK;
    p.m_total = (uint32_t)((long long)batch * G.hout * G.wout);
    p.tiles_m = (p.m_total + kTileM - 1) / kTileM;
    p.in = in; p.res = res; p.out = out; p.wpack = wpack; p.err = err;
    if (p.tiles_m == 0) return cudaSuccess;
    const bool paired = igemm_pairable(G) && igemm_smem(G, true).fits() && p.tma_a && p.fast_requant && (!res || p.fast_residual) &&
                        igemm_paired(p.tiles_m, (uint32_t)p.tiles_n, (uint32_t)dev.n_sms);
    if (paired) p.tiles_m = (p.tiles_m + 1) / 2;
    const bool whole = igemm_whole(G);
    p.acc_stride = paired ? 2 * kPairN : (p.n_tile + 31) & ~31;          // epilogue_rows loads 32 columns at a time
    // the same view's encoder for the residual operand (its rows are a multiple of 16 bytes, its boxes at most 256 x 256)
    p.prefetch_res = 0;
    memset(&p.tmap_res, 0, sizeof(p.tmap_res));
    if (const EncodeFn encode = whole && res && p.tma_a ? (EncodeFn)dev.encode : nullptr) {
        const cuuint64_t dims[2] = {(cuuint64_t)G.coutp, (cuuint64_t)p.m_total}, strides[1] = {(cuuint64_t)G.coutp};
        const cuuint32_t box[2] = {(cuuint32_t)p.n_tile, (cuuint32_t)(paired ? 2 * kTileM : kTileM)}, estr[2] = {1, 1};
        p.prefetch_res = encode(&p.tmap_res, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<int8_t *>(res), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                                CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    }
    p.n_acc = whole && p.tma_a && p.acc_stride <= 64 ? 4 : 2;
    p.tmem_cols = 64;
    while (p.tmem_cols < p.n_acc * p.acc_stride) p.tmem_cols <<= 1;
    // as many operand stages as fit beside the constants, at most kMaxStages
    IgemmSmem s = igemm_smem(G, paired);
    if (whole) s.scratch = 0;
    p.stages = (int)std::min<size_t>(kMaxStages, (kSmemLimit - s.cst - s.scratch) / s.stage);
    p.scratch_off = (uint32_t)((size_t)p.stages * s.stage + s.cst);
    const size_t smem = (size_t)p.stages * s.stage + s.cst + s.scratch;
    // persistent: one CTA per SM (shared memory and the 512 tensor-memory columns allow no second one at N = 256)
    const uint32_t n_tiles = p.tiles_m * (uint32_t)p.tiles_n;
    const unsigned grid = std::min<uint32_t>(n_tiles, (uint32_t)dev.n_sms);
    return launch_chained(dev.chained, paired ? k_igemm<true, true, true> : !whole ? k_igemm<false, false, false> : p.tma_a ? k_igemm<true, false, true> : k_igemm<true, false, false>,
                          dim3(grid), igemm_threads(whole, p.tma_a != 0), smem, st, p);
}

// ---- the stem

size_t stem_pack_bytes(const GLayer &G) { return (size_t)G.kh * G.coutp * 32; }

namespace {

struct StemConfig {
    int band_rows, pitch, rows_class, planes;
    uint32_t plane_pos, k_step, w_bytes, pos_bytes, patch_bytes;
    size_t smem() const { return (size_t)w_bytes + pos_bytes + patch_bytes; }
};

// Bands of `rows` output rows, if two CTAs per SM and some noise tables fit then (one row: if one CTA does).
bool stem_config(const GLayer &G, int in_c, int rows, StemConfig *c)
{
    if (G.op != ISC_CONV2D || in_c > 4 || G.kw > 8 || G.kh > 8 || G.coutp % 16 != 0 || G.coutp > 256) return false;
    const bool second = G.kw > 4, whole = 4 % G.stride == 0;
    c->planes = second && !whole ? 2 : 1;
    c->pitch = G.wout + (second && whole ? 4 / G.stride : 0);
    c->w_bytes = (uint32_t)stem_pack_bytes(G);
    const int rows_in = (rows - 1) * G.stride + G.kh;
    const size_t patch = ((size_t)rows_in * (G.win + 2 * G.pad + 8) * 4 + 15) & ~(size_t)15;
    c->band_rows = rows;
    c->rows_class = (rows_in + G.stride - 1) / G.stride;
    const size_t plane_pos = (size_t)G.stride * c->rows_class * c->pitch + 2 * kTileM + 8;        // the last tile reads beyond the last row
    const size_t total = c->w_bytes + plane_pos * c->planes * 16 + patch;
    if (total > (rows > 1 ? 94 : 214) * (size_t)1024) return false;
    c->plane_pos = (uint32_t)plane_pos;
    c->pos_bytes = (uint32_t)(plane_pos * c->planes * 16);
    c->patch_bytes = (uint32_t)patch;
    c->k_step = !second ? 16u : whole ? 16u * (uint32_t)(4 / G.stride) : c->plane_pos * 16u;
    return c->k_step < (1u << 18);
}

// Bands of eight rows, or of fewer if that does not fit.
bool stem_config_any(const GLayer &G, int in_c, StemConfig *c)
{
    for (int rows = 8; rows >= 1; rows >>= 1)
        if (stem_config(G, in_c, rows, c)) return true;
    return false;
}

// Where a launch finds its noise levels: the bins in shared memory, the guide and cumulative tables there, or those in global memory.
enum class StemTables { kBins, kFront, kGlobal };

// Bands of at most 32 rows and tables for `batch` samples on `ctas` CTAs, two per SM: such that the CTA with the most work has
// the least.  An item costs its input rows and some six rows' worth of barriers and phases (3 x 3 on 32 x 32, 5,100 samples:
// 330 us in bands of 8 rows, 220 in one of 32); short bands share out more evenly.  A row drawn by search costs 1.8 times one
// drawn by bins with the tables in shared memory, whose copy costs the item too, and twice with them in global memory, or more
// where the two CTAs' shared memory passes the split of 196 KB and leaves the L1 next to nothing.  So tables take their room from
// the bands: 7 x 7 stride 2 on 224 x 224, 700 samples with sigma = 1 (41 KB of bins), took 1,404 us in bands of 8 rows with the
// search in shared memory, 1,540 in bands of 11 without any table there, and takes 1,213 in bands of 6 with the bins; with
// sigma = 4.6 (70 KB of tables, no bins) 2,330 us in bands of 11 and 1,787 in bands of 10.
void stem_bands(const GLayer &G, int in_c, int64_t batch, int64_t ctas, size_t bins, size_t front, StemConfig *c, StemTables *tables)
{
    int64_t best = INT64_MAX;
    for (int want = 32, last = 0; want >= 1; --want) {
        const int bands = (G.hout + want - 1) / want, rows = (G.hout + bands - 1) / bands;
        StemConfig t;
        if (rows == last || !stem_config(G, in_c, rows, &t) || t.smem() > kStemSmemPair) continue;
        last = rows;
        StemTables at = StemTables::kGlobal;
        int row = 2 * (t.smem() + kStemSmemOwn) <= 196 * 1024 ? 20 : 26, item = 60;
        if (bins && t.smem() + bins <= kStemSmemPair) { at = StemTables::kBins; row = 10; }
        else if (front && t.smem() + front <= kStemSmemPair) { at = StemTables::kFront; row = 18; item += (int)(front / 1024); }
        const int64_t cost = (batch * bands + ctas - 1) / ctas * (((rows - 1) * G.stride + G.kh) * row + item);
        if (cost < best) { best = cost; *c = t; *tables = at; }
    }
}

}  // namespace

bool stem_fits(const GLayer &G, int in_c)
{
    StemConfig c;
    return stem_config_any(G, in_c, &c);
}

// w: [cout][cin][kh][kw] -> [filter row][2 columns of 16 bytes][coutp rows][16]: byte pix * 4 + ch of a row's 32
void stem_pack_weights(const GLayer &G, const int8_t *w, int8_t *out)
{
    size_t at = 0;
    for (int r = 0; r < G.kh; ++r)
        for (int j = 0; j < 2; ++j)
            for (int n = 0; n < G.coutp; ++n)
                for (int e = 0; e < 16; ++e, ++at) {
                    const int c32 = j * 16 + e, pix = c32 >> 2, ch = c32 & 3;
                    out[at] = (n < G.cout && pix < G.kw && ch < G.cin) ? w[(((size_t)n * G.cin + ch) * G.kh + r) * G.kw + pix] : (int8_t)0;
                }
}

cudaError_t launch_stem_conv(const TcDevice &dev, const GLayer &G, const int8_t *wpack, const int32_t *cst, bool fast, const uint8_t *x_chw, int in_c,
                             const NoiseStream &ns, const SampleRun &run, int batch, int8_t *out, int32_t *err, cudaStream_t st, bool debug_stall, bool chained)
{
    StemParams p;
    p.L = G;
    p.in_c = in_c;
    StemConfig c;
    if (!stem_config_any(G, in_c, &c)) return cudaErrorInvalidValue;
    // the guide table has to follow the cumulative one
    const size_t bins = ns.bins && ns.guide ? (size_t)noise_bins_side(ns.bin_bits) * 16 : 0;
    const size_t front = ns.guide && ns.guide == ns.cum + (2 * ns.T + 1) ? ((size_t)(2 * ns.T + 1 + kNoiseGuide + 1) * 4 + 15) & ~(size_t)15 : 0;
    StemTables tables = StemTables::kGlobal;
    if (c.smem() <= kStemSmemPair) stem_bands(G, in_c, batch, 2ll * dev.n_sms, bins, front, &c, &tables);
    else if (bins && c.smem() + bins <= kStemSmemLimit) tables = StemTables::kBins;
    else if (front && c.smem() + front <= kStemSmemLimit) tables = StemTables::kFront;
    p.band_rows = c.band_rows;
    p.n_bands = (G.hout + p.band_rows - 1) / p.band_rows;
    p.pitch = c.pitch; p.rows_class = c.rows_class; p.planes = c.planes;
    p.plane_pos = c.plane_pos; p.k_step = c.k_step;
    p.w_bytes = c.w_bytes; p.pos_off = c.w_bytes; p.patch_off = c.w_bytes + c.pos_bytes;
    p.slots = G.coutp <= 64 ? 2 : 1;                             // two CTAs share the 512 columns of an SM
    int cols = 32;
    while (cols < p.slots * 2 * G.coutp) cols <<= 1;
    p.tmem_cols = cols;
    p.x = x_chw; p.ns = ns; p.run = run; p.wpack = wpack;
    p.cst = reinterpret_cast<const int4 *>(cst);
    p.fast_requant = fast ? 1 : 0;
    p.lo = G.relu ? (G.zp_out > -128 ? G.zp_out : -128) : -128;
    p.out = out; p.err = err;
    p.debug_stall = debug_stall ? 1 : 0;
    size_t smem = c.smem();
    const size_t tab = tables == StemTables::kBins ? bins : tables == StemTables::kFront ? front : 0;
    p.tab_off = tab ? (uint32_t)smem : 0;
    p.tab_words = tables == StemTables::kFront ? 2 * ns.T + 1 + kNoiseGuide + 1 : (int)(tab / 4);
    p.bin_bits = tables == StemTables::kBins ? ns.bin_bits : 0;
    smem += tab;
    if (batch <= 0) return cudaSuccess;
    p.n_items = (uint32_t)p.n_bands * (uint32_t)batch;
    // A CTA takes one item after the other; where levels are searched in bands of many pixels, an item (7 x 7 stride 2 on
    // 300 x 300, 700 samples with sigma = 1: 3,128 and 2,940 us; 32 x 32, 6,000 samples with sigma = 2: 482 and 509; equal with bins).
    const bool search_long = !p.bin_bits && ((p.band_rows - 1) * G.stride + G.kh) * G.win >= 3000;
    const uint32_t ctas = search_long ? p.n_items : (uint32_t)dev.n_sms * (smem <= kStemSmemPair ? 2u : 1u);
    return launch_chained(chained && dev.chained, k_stem, dim3(std::min(p.n_items, ctas)), kStemThreads, smem, st, p);
}

}  // namespace isc

