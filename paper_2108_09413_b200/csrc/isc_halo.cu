// Stride-1 "same" convolutions of the layer-by-layer engine on the tensor cores with the input tile resident in shared
// memory (sm_100a): one launch per convolution over a batch of noisy samples, activations as in isc_generic.cu.
//
// Layout.  The batch's pixels lie on a line of positions f = (image * (H + p) + y) * (W + p) + x, p = (k - 1) / 2, with p
// padding columns behind every row and p padding rows behind every image, which are the neighbours' left and upper
// padding too.  The neighbour (dr, ds) of position f is f + dr * (W + p) + ds, for every f.  A tile is 256 consecutive
// positions (two M = 128 operands); it and the halo before and behind it are copied to shared memory once, per plane of
// 16 channels as [position][16 bytes] (padding positions take the input zero-point), and every filter tap reads it there:
// a tap is an address offset of the operand descriptor.  The gathering kernel (isc_igemm.cu) copies each of a 3 x 3
// filter's nine operands from the caches instead, 8 KB per 64 bytes of K, which bounds it at about 20 bytes a clock
// and SM.  Positions that are padding are computed and not stored (3 % of a 56 x 56 map's, 23 % of a 7 x 7 map's).
//
// Reduction: two rings of stages.  An A stage holds one or two pairs of planes of the tile; a B block the weights of one
// filter row of a pair (K = 32 per tap, the planes' distance is the descriptor's leading-dimension offset; an odd last
// plane takes its taps in pairs instead, distance one position).  All B blocks stay in shared memory when they fit.
//
// Roles (warps), which meet at mbarriers: four gather warps; two MMA warps, one per M operand, which run converged on
// warp-uniform values and predicate the instruction itself on one lane (a lone lane that builds descriptors in ordinary
// registers took 450 cycles per MMA beside the other roles); one weights warp; sixteen epilogue warps in four teams of
// four.  An output tile is 256 positions x at most 128 channels; up to 64 channels four of them fit into tensor memory
// and each team takes every fourth, else two fit and two teams halve the channels of every second.  With eight warps
// in two teams the epilogue's latency (a few hundred instructions at ten cycles each) was twice the MMAs' time.  A
// thread requantises one row of both M operands, so that a channel's constants are read once for two outputs: reading
// them once for each saturates the shared-memory pipe at 6 outputs a clock and SM.  Results leave, and residual rows
// arrive, as runs of up to 64 bytes through a scratch area.
// Every wait is bounded; on expiry a role raises the CTA's abort flag and the error word, the others leave their loops,
// and the CTA frees its tensor memory and returns.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cstring>

#include "isc_conv.cuh"
#include "isc_epilogue.cuh"
#include "isc_internal.h"
#include "isc_tc.cuh"

namespace isc {

using namespace tc;
using namespace conv;

namespace {

constexpr int kM = 128, kMT = 2, kTile = kM * kMT;      // rows of one MMA, MMAs side by side, positions of a tile
constexpr int kTeams = 4, kEpi = 4 * kTeams, kGather = 4;
constexpr int kThreads = 32 * (kEpi + kGather + kMT + 1);
constexpr int kMaxRing = 8;
constexpr int kFlat = 12;                               // positions of a tile that a gather lane keeps the addresses of
constexpr int kMaxN = 128;                              // output channels of a tile: two of them, times kMT, fill tensor memory
constexpr size_t kSmemMax = 226 * 1024;

struct HaloParams {
    GLayer L;
    int wp, hp, halo;                        // row pitch and rows per image on the line of positions; halo positions on either side
    int batch, c16s;                         // planes
    int stage_planes, lpp_log;               // planes of an A stage (2 or 4); log2 of the gather lanes that share a position
    int n_stages;                            // A stages of a tile
    int flat_steps;                          // positions per gather lane if at most kFlat, else 0
    uint32_t positions, tile_pos, plane_bytes, a_bytes;     // of the batch; copied per tile; of a plane; of an A stage
    int ring_a, ring_b, resident;            // stages; B blocks (one tile's after the other when resident)
    int n_tile, tiles_n, n_blocks, tmem_cols;               // B blocks of an output tile: kh for each pair of planes
    int slots_log, col_split;                // log2 of the accumulators in tensor memory (4 or 2); channels per team when two share a tile, else 0
    uint32_t n_items;                        // tiles * tiles_n
    int lpr_log;                             // log2 of the lanes that share a row in the coalesced accesses
    uint32_t b_off, cst_off, scratch_off, rowtab_off;
    FastDiv by_image, by_wp, by_hp, by_tiles_n;     // positions of an image, of a row; rows of an image; output tiles of a tile
    const int8_t *in, *res;
    int8_t *out;
    const int8_t *wpack;                     // [cout tile][block][kh steps][2 columns][n_tile rows][16 bytes]
    const int8_t *zp_run;
    const int4 *cst;
    int fast, lo, res_short;
    uint32_t res_m2, res_k8;
    long long res_r2;
    int debug_stall;                         // test hook: the weights are never sent, so that the kernel's waits run out
    int32_t *err;
};

struct RoleCtx {
    uint32_t sbase, tmem, acc_full, acc_free;
    int warp, lane;
    const volatile int *abort_flag;
};

// The epilogue of one warp: rows 32 q .. + 31 of both M operands of its team's output tiles, at most 64 channels.
// kMode 0: 64-bit requantisation (any shift), 1: 32-bit form, 2 / 3: 32-bit form with the residual add (3: its
// single-precision form).  kClamp: the lower clamp is above -128.
template <int kMode, bool kClamp>
__device__ __forceinline__ bool halo_epilogue(const HaloParams &p, const RoleCtx &c)
{
    const GLayer &L = p.L;
    const int lane = c.lane, q = c.warp & 3, team = c.warp >> 2;
    constexpr bool kHasRes = kMode >= 2;
    const uint32_t slot = (uint32_t)team & ((1u << p.slots_log) - 1u);
    const int c_first = (team >> p.slots_log) * p.col_split;        // of the output tile: this team's channels
    const int lpr = 1 << p.lpr_log, rpi = 32 >> p.lpr_log;           // lanes per row, rows per instruction
    const int crow = lane >> p.lpr_log, cchunk = lane & (lpr - 1);
    // Scratch: per M operand 32 rows without padding; the 16-byte columns of a row are permuted by the row's number so
    // that neither the row-wise nor the coalesced access has bank conflicts.  (rpi is a multiple of the period.)
    const uint32_t row_bytes = 16u << p.lpr_log, mt_step = 32u * row_bytes;
    const uint32_t scr0 = c.sbase + p.scratch_off + (uint32_t)c.warp * (kMT * mt_step);
    auto permuted = [&](int row, uint32_t col) { return col ^ (p.lpr_log == 2 ? ((uint32_t)row >> 1) & 3u : ((uint32_t)row >> 2) & 1u); };
    const uint32_t scr_row = scr0 + (uint32_t)lane * row_bytes;
    const uint32_t scr_co = scr0 + (uint32_t)crow * row_bytes + permuted(crow, (uint32_t)cchunk) * 16u;
    const uint32_t rowtab = c.sbase + p.rowtab_off + (uint32_t)c.warp * (uint32_t)(2 * 32 * kMT * 4);
    const uint32_t i_step = gridDim.x << p.slots_log;
    // an output tile: item = tile * tiles_n + n.  Its rows' byte offsets in the output go to the warp's table (-1: padding).
    auto open_item = [&](uint32_t item, uint32_t tab, int &n0, int &n_cols) {
        uint32_t n;
        const uint32_t tile = p.by_tiles_n.divmod(item, n);
        n0 = (int)n * p.n_tile + c_first;
        n_cols = min(p.n_tile, L.coutp - (int)n * p.n_tile) - c_first;
        if (p.col_split && c_first == 0) n_cols = min(n_cols, p.col_split);
#pragma unroll
        for (int mt = 0; mt < kMT; ++mt) {
            const uint32_t f = tile * kTile + (uint32_t)(mt * kM + q * 32 + lane);
            uint32_t r, x;
            const uint32_t img = p.by_image.divmod(f, r), y = p.by_wp.divmod(r, x);
            const bool valid = f < p.positions && y < (uint32_t)L.hout && x < (uint32_t)L.wout;
            const int off = valid ? (int)(((img * (uint32_t)L.hout + y) * (uint32_t)L.wout + x) * (uint32_t)L.coutp) : -1;
            asm volatile("st.shared.u32 [%0], %1;" ::"r"(tab + (uint32_t)(mt * 32 + lane) * 4u), "r"(off) : "memory");
        }
        __syncwarp();
    };
    auto row_off = [&](uint32_t tab, int mt, int k) { return (int)lds32(tab + (uint32_t)(mt * 32 + k * rpi + crow) * 4u); };
    auto fetch_residual = [&](uint32_t tab, int n0, int n_cols) {
        if (cchunk * 16 >= n_cols) return;
#pragma unroll
        for (int mt = 0; mt < kMT; ++mt)
            for (int k = 0; k < lpr; ++k) {
                const int off = row_off(tab, mt, k);
                if (off >= 0) cp_async16(scr_co + (uint32_t)mt * mt_step + (uint32_t)(k * rpi) * row_bytes, p.res + off + n0 + cchunk * 16);
            }
    };
    const uint32_t acc0 = c.tmem + ((uint32_t)(q * 32) << 16) + slot * (uint32_t)(kMT * p.n_tile) + (uint32_t)c_first, acc1 = acc0 + (uint32_t)p.n_tile;
    const uint32_t bar_full = c.acc_full + 8u * slot, bar_free = c.acc_free + 8u * slot;
    uint32_t item = blockIdx.x + slot * gridDim.x, tab = rowtab;
    int n0 = 0, n_cols = 0;
    if (item < p.n_items) {
        open_item(item, tab, n0, n_cols);
        if (kHasRes) fetch_residual(tab, n0, n_cols);
    }
    for (uint32_t use = 0; item < p.n_items; item += i_step, ++use) {
        const uint32_t tab_next = 2u * rowtab + (uint32_t)(32 * kMT * 4) - tab;          // the other table
        int n0_next = 0, cols_next = 0;
        if (item + i_step < p.n_items) open_item(item + i_step, tab_next, n0_next, cols_next);
        if (kHasRes) cp_async_wait_all();                               // this tile's residual rows, requested during the previous one
        __syncwarp();
        if (!wait_bar<kHintEpi>(bar_full, use & 1u, c.abort_flag)) {
            cp_async_wait_all();
            return false;
        }
        tc_fence_after();
        if (n_cols <= 0) {                                              // the second team of a partial tile
            tc_fence_before();
            mbar_arrive(bar_free);
        }
        const uint32_t cst0 = c.sbase + p.cst_off + (uint32_t)n0 * 16u;
#pragma unroll 1
        for (int cc = 0; cc < n_cols; cc += 16) {
            int a[2][16];
            tmem_ld16_issue(acc0 + (uint32_t)cc, a[0]);
            tmem_ld16_issue(acc1 + (uint32_t)cc, a[1]);
            const uint32_t scr = scr_row + permuted(lane, (uint32_t)cc >> 4) * 16u;
            uint32_t r0[4] = {0, 0, 0, 0}, r1[4] = {0, 0, 0, 0};
            if (kHasRes) {
                const uint4 u = ld_shared_v4(scr), v = ld_shared_v4(scr + mt_step);
                r0[0] = u.x ^ 0x80808080u; r0[1] = u.y ^ 0x80808080u; r0[2] = u.z ^ 0x80808080u; r0[3] = u.w ^ 0x80808080u;
                r1[0] = v.x ^ 0x80808080u; r1[1] = v.y ^ 0x80808080u; r1[2] = v.z ^ 0x80808080u; r1[3] = v.w ^ 0x80808080u;
            }
            tmem_ld32_wait(a);
            if (cc + 16 >= n_cols) {
                tc_fence_before();
                mbar_arrive(bar_free);                                  // the accumulators are in registers: the next tile may overwrite them
            }
            uint4 o[2];
            if (kMode == 0) {
#pragma unroll
                for (int mt = 0; mt < 2; ++mt) {
                    const int off = (int)lds32(tab + (uint32_t)(mt * 32 + lane) * 4u);
#pragma unroll
                    for (int k = 0; k < 16; ++k) a[mt][k] += __ldg(L.bias + n0 + cc + k);
                    o[mt] = epilogue16(a[mt], L, n0 + cc, p.res && off >= 0 ? p.res + off : nullptr);
                }
            } else {
                constexpr int kRes = kMode == 3 ? 2 : kMode == 2 ? 1 : 0;
                requant16x2<kRes, kClamp>(a, cst0 + (uint32_t)cc * 16u, r0, r1, p.res_m2, p.res_r2, p.res_k8, p.lo, o);
            }
            st_shared_v4(scr, o[0]);
            st_shared_v4(scr + mt_step, o[1]);
        }
        __syncwarp();
        if (cchunk * 16 < n_cols) {
            int8_t *dst = p.out + n0 + cchunk * 16;
#pragma unroll
            for (int mt = 0; mt < kMT; ++mt)
                for (int k = 0; k < lpr; ++k) {
                    const int off = row_off(tab, mt, k);
                    if (off >= 0) *reinterpret_cast<uint4 *>(dst + off) = ld_shared_v4(scr_co + (uint32_t)mt * mt_step + (uint32_t)(k * rpi) * row_bytes);
                }
        }
        __syncwarp();
        if (kHasRes && cols_next > 0) fetch_residual(tab_next, n0_next, cols_next);
        tab = tab_next; n0 = n0_next; n_cols = cols_next;
    }
    cp_async_wait_all();
    return true;
}

// The MMAs of one M operand (mt), by a converged warp.  Barrier pairs: x = full, y = free.  KH: filter side, 0 = any.
template <int KH>
__device__ __forceinline__ bool issue_role(const HaloParams &p, uint32_t sbase, uint32_t tmem, int mt, uint2 a_bars, uint2 b_bars, uint2 acc_bars, const volatile int *abort_flag)
{
    const int k = KH ? KH : p.L.kh;
    const uint32_t lane0 = elect_one() ? 1u : 0u;
    const int pairs = p.c16s >> 1, pairs_stage = p.stage_planes >> 1;
    const uint32_t idesc = (2u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(p.n_tile >> 3) << 17) | ((uint32_t)(kM >> 4) << 24);
    const uint32_t plane16 = p.plane_bytes >> 4, stage16 = p.a_bytes >> 4, step16 = (uint32_t)p.n_tile * 2u, block16 = step16 * (uint32_t)k;
    const uint64_t a_desc = make_desc(sbase + (uint32_t)(mt * kM) * 16u, p.plane_bytes, 128u), a_desc_odd = make_desc(sbase + (uint32_t)(mt * kM) * 16u, 16u, 128u);
    const uint64_t b_desc = make_desc(sbase + p.b_off, (uint32_t)p.n_tile * 16u, 128u);
    uint32_t a_s = 0, a_use = 0, b_s = 0, b_use = 0, i = 0;
    for (uint32_t item = blockIdx.x; item < p.n_items; item += gridDim.x, ++i) {
        const uint32_t slot = i & ((1u << p.slots_log) - 1u), use = i >> p.slots_log;
        if (use >= 1 && !wait_warp(acc_bars.y + 8u * slot, (use - 1) & 1u, abort_flag)) return false;
        if (p.resident) {
            if (i == 0 && !wait_warp(b_bars.x, 0u, abort_flag)) return false;
            uint32_t n;
            p.by_tiles_n.divmod(item, n);
            b_s = n * (uint32_t)p.n_blocks;
        }
        const uint32_t d = tmem + (slot * kMT + (uint32_t)mt) * (uint32_t)p.n_tile;
        uint32_t acc = 0;
        // a filter row of a pair of planes (of the odd last plane): k (half as many) MMAs
        auto row = [&](uint64_t ad, int steps, uint32_t a_step) {
            if (!p.resident) {
                if (!wait_warp(b_bars.x + 8u * b_s, b_use & 1u, abort_flag)) return false;
                tc_fence_after();
            }
            const uint64_t bd = b_desc + (uint64_t)(b_s * block16);
            if (KH) {
#pragma unroll
                for (int s = 0; s < KH; ++s)
                    if (s < steps) mma_i8_if(lane0, d, ad + (uint64_t)((uint32_t)s * a_step), bd + (uint64_t)((uint32_t)s * step16), idesc, s ? 1u : acc);
            } else {
                for (int s = 0; s < steps; ++s) mma_i8_if(lane0, d, ad + (uint64_t)((uint32_t)s * a_step), bd + (uint64_t)((uint32_t)s * step16), idesc, s ? 1u : acc);
            }
            acc = 1;
            if (!p.resident) commit_if(lane0, b_bars.y + 8u * b_s);
            ++b_s;
            if (!p.resident && b_s == (uint32_t)p.ring_b) { b_s = 0; ++b_use; }
            return true;
        };
        for (int st = 0; st < p.n_stages; ++st) {
            if (!wait_warp(a_bars.x + 8u * a_s, a_use & 1u, abort_flag)) return false;
            tc_fence_after();
            const uint32_t a0 = a_s * stage16;
            for (int j = 0; j < pairs_stage; ++j) {
                const int pair = st * pairs_stage + j;
                const uint32_t a_off = a0 + (uint32_t)(2 * j) * plane16;
                if (pair < pairs) {
                    for (int r = 0; r < k; ++r)
                        if (!row(a_desc + (uint64_t)(a_off + (uint32_t)(r * p.wp)), k, 1u)) return false;
                } else if (2 * pair < p.c16s) {
                    for (int r = 0; r < k; ++r)
                        if (!row(a_desc_odd + (uint64_t)(a_off + (uint32_t)(r * p.wp)), (k + 1) >> 1, 2u)) return false;
                }
            }
            commit_if(lane0, a_bars.y + 8u * a_s);
            if (++a_s == (uint32_t)p.ring_a) { a_s = 0; ++a_use; }
        }
        commit_if(lane0, acc_bars.x + 8u * slot);
    }
    return true;
}

__global__ void __launch_bounds__(kThreads, 1) k_halo(const __grid_constant__ HaloParams p)
{
    extern __shared__ __align__(128) uint8_t smem[];      // A stages | B blocks | constants | epilogue scratch | row tables
    __shared__ unsigned long long bar_a_full[kMaxRing], bar_a_free[kMaxRing], bar_b_full[kMaxRing], bar_b_free[kMaxRing], bar_acc_full[4], bar_acc_free[4];
    __shared__ uint32_t tmem_base_s;
    __shared__ volatile int abort_s;
    chain_start();
    const GLayer &L = p.L;
    const int tid = threadIdx.x, warp = (int)warp_uniform((uint32_t)tid >> 5), lane = tid & 31;
    const uint32_t sbase = smem_u32(smem);
    if (tid == 0) {
        for (int s = 0; s < kMaxRing; ++s) { mbar_init(smem_u32(&bar_a_full[s]), kGather * 32); mbar_init(smem_u32(&bar_a_free[s]), kMT); }
        for (int s = 0; s < kMaxRing; ++s) { mbar_init(smem_u32(&bar_b_full[s]), 1); mbar_init(smem_u32(&bar_b_free[s]), kMT); }
        for (int s = 0; s < 4; ++s) { mbar_init(smem_u32(&bar_acc_full[s]), kMT); mbar_init(smem_u32(&bar_acc_free[s]), (4 * 32 * kTeams) >> p.slots_log); }
        abort_s = 0;
    }
    if (warp == 0) tmem_alloc(smem_u32(&tmem_base_s), (uint32_t)p.tmem_cols);
    {
        int4 *cst_s = reinterpret_cast<int4 *>(smem + p.cst_off);
        for (int i = tid; i < p.tiles_n * p.n_tile; i += kThreads) cst_s[i] = __ldg(p.cst + i);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_proxy_async();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base_s;
    chain_wait();
    const uint32_t block_bytes = (uint32_t)(p.n_tile * L.kh) * 32u;
    const uint2 a_bars = make_uint2(smem_u32(&bar_a_full[0]), smem_u32(&bar_a_free[0])), b_bars = make_uint2(smem_u32(&bar_b_full[0]), smem_u32(&bar_b_free[0])),
                acc_bars = make_uint2(smem_u32(&bar_acc_full[0]), smem_u32(&bar_acc_free[0]));
    bool ok = true;

    if (warp < kEpi) {
        RoleCtx c{sbase, tmem, acc_bars.x, acc_bars.y, warp, lane, &abort_s};
        const bool clamp = p.lo > -128;
        if (!p.fast) ok = halo_epilogue<0, true>(p, c);
        else if (!p.res) ok = clamp ? halo_epilogue<1, true>(p, c) : halo_epilogue<1, false>(p, c);
        else if (!p.res_short) ok = halo_epilogue<2, true>(p, c);
        else ok = clamp ? halo_epilogue<3, true>(p, c) : halo_epilogue<3, false>(p, c);
    } else if (warp < kEpi + kGather && p.flat_steps > 0) {
        // ---- A stages, position by position: lanes share a position's planes (16 bytes each).  Where a lane's positions lie
        // is worked out once per tile, independently of each other, and kept for the tile's stages.  The form below walks
        // the rows of the images one after the other, a chain of dependent instructions that a short tile does not hide
        // (4096 samples of a network of 32 to 128 channels on 32 x 32 to 8 x 8 maps: 2.27 -> 2.18 ms); it stays for
        // tiles with more than kFlat positions per lane (64 channels: maps of more than 56 columns).
        const int lpp = 1 << p.lpp_log, per_warp = 32 >> p.lpp_log, chunk = lane & (lpp - 1);
        const uint32_t first_pos = (uint32_t)((warp - kEpi) * per_warp + (lane >> p.lpp_log)), step_pos = (uint32_t)(kGather * per_warp);
        Ring ring;
        for (uint32_t item = blockIdx.x; item < p.n_items && ok; item += gridDim.x) {
            // one image further on, so that the halo before the first tile is no negative number
            const uint32_t first = p.by_tiles_n.div(item) * kTile + (uint32_t)(p.wp * p.hp) - (uint32_t)p.halo + first_pos;
            int off[kFlat];                                             // of the pixel's first byte in the input; -1: padding
#pragma unroll
            for (int i = 0; i < kFlat; ++i) {
                uint32_t x, y;
                const uint32_t img = p.by_hp.divmod(p.by_wp.divmod(first + (uint32_t)i * step_pos, x), y) - 1u;
                const bool inside = x < (uint32_t)L.win && y < (uint32_t)L.hin && img < (uint32_t)p.batch;
                off[i] = inside ? (int)(((img * (uint32_t)L.hin + y) * (uint32_t)L.win + x) * (uint32_t)L.cinp) : -1;
            }
            for (int plane = chunk, st = 0; st < p.n_stages; ++st, plane += p.stage_planes, ring.advance(p.ring_a)) {
                if (ring.use >= 1) {
                    ok = wait_bar<kHintLoad>(a_bars.y + 8u * (uint32_t)ring.s, (uint32_t)(ring.use - 1) & 1u, &abort_s);
                    if (!ok) break;
                }
                if (plane < p.c16s) {
                    const uint32_t dst = sbase + (uint32_t)ring.s * p.a_bytes + (uint32_t)chunk * p.plane_bytes + first_pos * 16u;
                    const int8_t *src = p.in + plane * 16;
#pragma unroll
                    for (int i = 0; i < kFlat; ++i)
                        if (first_pos + (uint32_t)i * step_pos < p.tile_pos) cp_async16_cached(dst + (uint32_t)i * step_pos * 16u, off[i] >= 0 ? src + off[i] : p.zp_run);
                }
                cp_async_arrive(a_bars.x + 8u * (uint32_t)ring.s);
            }
        }
        cp_async_wait_all();
    } else if (warp < kEpi + kGather) {
        // ---- A stages, row by row of the images: rows go round the warps, lanes share a position's planes (16 bytes
        // each), so that a copy costs a handful of instructions
        const int lpp = 1 << p.lpp_log, per_warp = 32 >> p.lpp_log, chunk = lane & (lpp - 1), sub = lane >> p.lpp_log;
        const int wp = p.wp, hp = p.hp, tile_pos = (int)p.tile_pos;
        const uint32_t src_step = (uint32_t)(per_warp * L.cinp), dst_step = (uint32_t)per_warp * 16u;
        Ring ring;
        for (uint32_t item = blockIdx.x; item < p.n_items && ok; item += gridDim.x) {
            // the tile's first position, one image further on so that the halo before the first tile is no negative number
            const uint32_t first = p.by_tiles_n.div(item) * kTile + (uint32_t)(wp * hp) - (uint32_t)p.halo;
            const uint32_t row0 = p.by_wp.div(first);
            const int at0 = (int)(row0 * (uint32_t)wp) - (int)first + (warp - kEpi) * wp;          // tile position of the row's first one
            const uint32_t row = row0 + (uint32_t)(warp - kEpi), img = p.by_hp.div(row);
            const int y0 = (int)(row - img * (uint32_t)hp), b0 = (int)img - 1;
            for (int plane = chunk, st = 0; st < p.n_stages; ++st, plane += p.stage_planes, ring.advance(p.ring_a)) {
                if (ring.use >= 1) {
                    ok = wait_bar<kHintLoad>(a_bars.y + 8u * (uint32_t)ring.s, (uint32_t)(ring.use - 1) & 1u, &abort_s);
                    if (!ok) break;
                }
                if (plane < p.c16s) {
                    const uint32_t a_base = sbase + (uint32_t)ring.s * p.a_bytes + (uint32_t)chunk * p.plane_bytes;
                    int y = y0, b = b0;
                    for (int at = at0; at < tile_pos; at += kGather * wp) {
                        int x = max(-at, 0) + sub;
                        const int x_end = min(wp, tile_pos - at);
                        const int w_in = (y < L.hin && b >= 0 && b < p.batch) ? L.win : 0;         // pixels of the row; the rest is padding
                        const int8_t *src = p.in + ((uint32_t)(b * L.hin + y) * (uint32_t)L.win + (uint32_t)x) * (uint32_t)L.cinp + (uint32_t)plane * 16u;
                        uint32_t dst = a_base + (uint32_t)(at + x) * 16u;
                        for (; x < x_end; x += per_warp, src += src_step, dst += dst_step) cp_async16_cached(dst, x < w_in ? src : p.zp_run);
                        y += kGather;
                        while (y >= hp) { y -= hp; ++b; }
                    }
                }
                cp_async_arrive(a_bars.x + 8u * (uint32_t)ring.s);
            }
        }
        cp_async_wait_all();
    } else if (warp < kEpi + kGather + kMT) {
        // ---- one warp per M operand issues its MMAs
        const int mt = warp - kEpi - kGather;
        ok = L.kh == 3 ? issue_role<3>(p, sbase, tmem, mt, a_bars, b_bars, acc_bars, &abort_s) : issue_role<0>(p, sbase, tmem, mt, a_bars, b_bars, acc_bars, &abort_s);
    } else {
        // ---- one thread streams the repacked weights
        if (lane == 0 && !p.debug_stall) {
            if (p.resident) {
                const uint32_t blocks = (uint32_t)(p.tiles_n * p.n_blocks);
                mbar_expect_tx(b_bars.x, blocks * block_bytes);
                for (uint32_t b = 0; b < blocks; ++b) bulk_g2s(sbase + p.b_off + b * block_bytes, p.wpack + (size_t)b * block_bytes, block_bytes, b_bars.x);
            } else {
                Ring ring;
                for (uint32_t item = blockIdx.x; item < p.n_items && ok; item += gridDim.x) {
                    uint32_t n;
                    p.by_tiles_n.divmod(item, n);
                    const int8_t *w = p.wpack + (size_t)n * (size_t)p.n_blocks * block_bytes;
                    for (int b = 0; b < p.n_blocks; ++b, w += block_bytes, ring.advance(p.ring_b)) {
                        if (ring.use >= 1) {
                            ok = wait_bar<kHintLoad>(b_bars.y + 8u * (uint32_t)ring.s, (uint32_t)(ring.use - 1) & 1u, &abort_s);
                            if (!ok) break;
                        }
                        mbar_expect_tx(b_bars.x + 8u * (uint32_t)ring.s, block_bytes);
                        bulk_g2s(sbase + p.b_off + (uint32_t)ring.s * block_bytes, w, block_bytes, b_bars.x + 8u * (uint32_t)ring.s);
                    }
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

}  // namespace

// ------------------------------------------------------------------ host side

namespace {

struct HaloConfig {
    int halo, wp, hp, c16s, tiles_n, n_tile, n_blocks, stage_planes, n_stages, ring_a, ring_b, resident, lpr_log, slots_log, col_split;
    uint32_t positions_tile, plane_positions, plane_bytes, a_bytes;
    size_t b_off, cst_off, scratch_off, rowtab_off, smem;
};

bool halo_config(const GLayer &G, HaloConfig *c)
{
    if (G.op != ISC_CONV2D || G.stride != 1 || G.kh != G.kw || !(G.kh & 1) || G.kh < 3 || G.pad != (G.kh - 1) / 2) return false;
    c->wp = G.win + G.pad; c->hp = G.hin + G.pad;
    c->halo = G.pad * c->wp + G.pad;
    c->c16s = G.cinp / 16;
    c->tiles_n = (G.coutp + kMaxN - 1) / kMaxN;
    c->n_tile = ((G.coutp + c->tiles_n - 1) / c->tiles_n + 15) & ~15;
    c->n_blocks = (c->c16s + 1) / 2 * G.kh;
    c->slots_log = c->n_tile <= 64 ? 2 : 1;
    c->col_split = c->n_tile <= 64 ? 0 : (c->n_tile / 2 + 15) & ~15;
    c->lpr_log = c->n_tile <= 32 ? 1 : 2;
    c->positions_tile = (uint32_t)(kTile + 2 * c->halo);
    c->plane_positions = (c->positions_tile + 1u) | 1u;          // an odd number of 16-byte rows: planes start in different banks; one to spare
    c->plane_bytes = c->plane_positions * 16u;
    const size_t scratch = (size_t)kEpi * 32 * kMT * (16u << c->lpr_log), rowtab = (size_t)kEpi * 2 * 32 * kMT * 4;
    const size_t cst = (size_t)c->tiles_n * c->n_tile * 16;
    const size_t block = (size_t)c->n_tile * G.kh * 32, all = block * (size_t)c->n_blocks * (size_t)c->tiles_n;
    // A stages of two pairs of planes where the channels are multiples of 64, else (or when three do not fit) of one;
    // the weights resident if they fit beside three stages, else a ring of at least three blocks
    for (int planes = c->c16s % 4 == 0 ? 4 : 2; planes >= 2; planes -= 2) {
        c->stage_planes = planes;
        c->n_stages = (c->c16s + planes - 1) / planes;
        c->a_bytes = (c->plane_bytes * (uint32_t)planes + 127u) & ~127u;
        const size_t fixed = cst + scratch + rowtab;
        if (fixed + 3 * (size_t)c->a_bytes + std::min(all, 3 * block) > kSmemMax) continue;
        c->resident = fixed + 3 * (size_t)c->a_bytes + all <= kSmemMax;
        size_t room = kSmemMax - fixed;
        if (c->resident) {
            c->ring_b = 1;
            c->ring_a = (int)std::min<size_t>(kMaxRing, (room - all) / c->a_bytes);
            c->b_off = (size_t)c->ring_a * c->a_bytes;
            c->cst_off = c->b_off + all;
        } else {
            // what is left beyond three of each goes to the weights first: they come from further away
            c->ring_b = (int)std::min<size_t>(kMaxRing - 2, (room - 3 * (size_t)c->a_bytes) / block);
            c->ring_a = (int)std::min<size_t>(kMaxRing, (room - (size_t)c->ring_b * block) / c->a_bytes);
            c->b_off = (size_t)c->ring_a * c->a_bytes;
            c->cst_off = c->b_off + (size_t)c->ring_b * block;
        }
        c->scratch_off = c->cst_off + cst;
        c->rowtab_off = c->scratch_off + scratch;
        c->smem = c->rowtab_off + rowtab;
        return true;
    }
    return false;
}

}  // namespace

bool halo_fits(const GLayer &G)
{
    HaloConfig c;
    return halo_config(G, &c);
}

// Besides the tensors' offsets: positions, those of one more image and a halo included, are divided as numbers below 2^31.
bool halo_offsets_fit(const GLayer &G, int64_t batch)
{
    HaloConfig c;
    return halo_config(G, &c) && conv_offsets_fit(G, batch) &&
           (batch + 1) * (int64_t)c.hp * c.wp + c.positions_tile + 2 * kTile < (1ll << 31);
}

size_t halo_pack_bytes(const GLayer &G)
{
    HaloConfig c;
    if (!halo_config(G, &c)) return 0;
    return (size_t)c.tiles_n * c.n_blocks * c.n_tile * G.kh * 32 + 64;
}

int halo_padded_cout(const GLayer &G)
{
    const int tiles = (G.coutp + kMaxN - 1) / kMaxN;
    return tiles * (((G.coutp + tiles - 1) / tiles + 15) & ~15);
}

// w: [cout][cin][kh][kw] -> [cout tile][block][kh steps][2 columns][n_tile rows][16]; then 64 bytes of the input
// zero-point.  Block (plane pair, filter row): step s = tap (row, s), columns = the two planes; of the odd last plane:
// columns = taps (row, 2 s) and (row, 2 s + 1).
void halo_pack(const GLayer &G, const int8_t *w, int8_t *out)
{
    HaloConfig c;
    halo_config(G, &c);
    const int k = G.kh;
    size_t at = 0;
    for (int t = 0; t < c.tiles_n; ++t)
        for (int b = 0; b < c.n_blocks; ++b)
            for (int s = 0; s < k; ++s)
                for (int col = 0; col < 2; ++col) {
                    const int pair = b / k, r = b % k;
                    const bool odd = 2 * pair + 1 == c.c16s;
                    const int plane = odd ? 2 * pair : 2 * pair + col, tap_x = odd ? 2 * s + col : s;
                    for (int n = 0; n < c.n_tile; ++n)
                        for (int e = 0; e < 16; ++e, ++at) {
                            const int oc = t * c.n_tile + n, ci = plane * 16 + e;
                            out[at] = (tap_x < k && oc < G.cout && ci < G.cin) ? w[(((size_t)oc * G.cin + ci) * k + r) * k + tap_x] : (int8_t)0;
                        }
                }
    for (int e = 0; e < 64; ++e) out[at + e] = (int8_t)G.zp_in;
}

cudaError_t halo_prepare() { return cudaFuncSetAttribute(k_halo, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax); }

cudaError_t launch_halo_conv(const TcDevice &dev, const GLayer &G, const int8_t *wpack, const int32_t *cst, bool fast, const ResidualForm &form, int batch,
                             const int8_t *in, const int8_t *res, int8_t *out, int32_t *err, cudaStream_t st, bool debug_stall)
{
    HaloConfig c;
    if (!halo_config(G, &c) || !halo_offsets_fit(G, batch)) return cudaErrorInvalidValue;
    const long long positions = (long long)batch * c.hp * c.wp;
    if (batch <= 0) return cudaSuccess;
    HaloParams p;
    memset(&p, 0, sizeof(p));
    p.L = G;
    p.wp = c.wp; p.hp = c.hp; p.halo = c.halo;
    p.batch = batch; p.c16s = c.c16s;
    p.stage_planes = c.stage_planes; p.n_stages = c.n_stages;
    p.lpp_log = c.c16s == 1 ? 0 : c.stage_planes == 4 ? 2 : 1;
    const uint32_t lane_pos = (uint32_t)kGather * (32u >> p.lpp_log);
    p.flat_steps = (int)((c.positions_tile + lane_pos - 1) / lane_pos);
    if (p.flat_steps > kFlat) p.flat_steps = 0;
    p.positions = (uint32_t)positions;
    p.tile_pos = c.positions_tile; p.plane_bytes = c.plane_bytes; p.a_bytes = c.a_bytes;
    p.ring_a = c.ring_a; p.ring_b = c.ring_b; p.resident = c.resident;
    p.n_tile = c.n_tile; p.tiles_n = c.tiles_n; p.n_blocks = c.n_blocks;
    p.slots_log = c.slots_log; p.col_split = c.col_split;
    p.tmem_cols = 64;
    while (p.tmem_cols < (kMT * p.n_tile) << p.slots_log) p.tmem_cols <<= 1;
    p.n_items = (uint32_t)((positions + kTile - 1) / kTile) * (uint32_t)c.tiles_n;
    p.by_image = FastDiv::make((uint32_t)(c.wp * c.hp));
    p.by_wp = FastDiv::make((uint32_t)c.wp);
    p.by_hp = FastDiv::make((uint32_t)c.hp);
    p.by_tiles_n = FastDiv::make((uint32_t)c.tiles_n);
    p.lpr_log = c.lpr_log;
    p.b_off = (uint32_t)c.b_off; p.cst_off = (uint32_t)c.cst_off;
    p.scratch_off = (uint32_t)c.scratch_off; p.rowtab_off = (uint32_t)c.rowtab_off;
    p.in = in; p.res = res; p.out = out; p.wpack = wpack;
    p.zp_run = wpack + halo_pack_bytes(G) - 64;
    p.cst = reinterpret_cast<const int4 *>(cst);
    p.lo = G.relu ? (G.zp_out > -128 ? G.zp_out : -128) : -128;
    const int res_n = 31 - G.res_shift;
    p.fast = fast && (!res || res_n == 31 || res_n == 32);
    p.res_short = res && form.exists();
    p.res_k8 = p.res_short ? form.k8 : 0u;
    if (p.res_short) {
        p.res_m2 = form.m_bits;
    } else if (res && p.fast) {
        p.res_m2 = (uint32_t)((unsigned long long)(uint32_t)G.res_mult << (32 - res_n));
        p.res_r2 = ((1ll << (res_n - 1)) - (128ll + G.zp_res) * (long long)G.res_mult) * (1ll << (32 - res_n));
    }
    p.debug_stall = debug_stall ? 1 : 0;
    p.err = err;
    return launch_chained(dev.chained, k_halo, dim3(std::min<uint32_t>(p.n_items, (uint32_t)dev.n_sms)), kThreads, c.smem, st, p);
}

}  // namespace isc
