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
// in two teams the epilogue's latency (a few hundred instructions at ten cycles each) was twice the MMAs' time.
// Accumulators are read as fragments: a thread holds four rows and up to sixteen consecutive channels (the columns of the
// weights are ordered for that, halo_channel), a constant in registers serves four outputs, and residual rows are read and
// results written straight from registers.  (With a row per thread, rows' offsets and bytes went through shared memory and
// a 32-channel layer took 18 instructions per output.)  This and gather_flat, 32 -> 32 channels at 32 x 32, 5,100 samples:
// 187 -> 166 us, with a residual operand 207 -> 194; what is left is shared memory's bandwidth: the MMAs' operands, the
// copies and the epilogue's constants keep it busy for 97 % of a 64-channel layer's time.
// Every wait is bounded; on expiry a role raises the CTA's abort flag and the error word, the others leave their loops,
// and the CTA frees its tensor memory and returns.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
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

constexpr int kM = 128, kMT = 2, kTile = kM * kMT;      // rows of one MMA, MMAs side by side, positions of a tile
constexpr int kTeams = 4, kEpi = 4 * kTeams, kGather = 4;
constexpr int kThreads = 32 * (kEpi + kGather + kMT + 1);
constexpr int kMaxRing = 8;
constexpr int kFlat = 10;                               // positions of a tile that a gather lane keeps the addresses of
constexpr int kMaxN = 128;                              // output channels of a tile: two of them, times kMT, fill tensor memory
constexpr size_t kSmemMax = 226 * 1024;

struct HaloParams {
    GLayer L;
    int wp, hp, halo;                        // row pitch and rows per image on the line of positions; halo positions on either side
    int batch, c16s;                         // planes
    int stage_planes, lpp_log;               // planes of an A stage (2 or 4); log2 of the gather lanes that share a position
    int n_stages;                            // A stages of a tile
    int flat_steps;                          // positions per gather lane, at most kFlat; 0: copied by rows
    uint32_t positions, tile_pos, plane_bytes, a_bytes;     // of the batch; copied per tile; of a plane; of an A stage
    int ring_a, ring_b, resident;            // stages; B blocks (one tile's after the other when resident)
    int n_tile, tiles_n, n_blocks, tmem_cols;               // B blocks of an output tile: kh for each pair of planes
    int slots_log, col_split;                // log2 of the accumulators in tensor memory (4 or 2); channels per team when two share a tile, else 0
    uint32_t n_items;                        // tiles * tiles_n
    uint32_t b_off, cst_off;
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
    const int q = c.warp & 3, team = c.warp >> 2;
    const bool has_res = kMode >= 2 || (kMode == 0 && p.res);
    const uint32_t slot = (uint32_t)team & ((1u << p.slots_log) - 1u), word = (uint32_t)c.lane & 3u;
    const int c_first = (team >> p.slots_log) * p.col_split;        // of the output tile: this team's channels
    const uint32_t acc0 = c.tmem + ((uint32_t)(q * 32) << 16) + slot * (uint32_t)(kMT * p.n_tile) + (uint32_t)c_first;
    const uint32_t bar_full = c.acc_full + 8u * slot, bar_free = c.acc_free + 8u * slot;
    uint32_t use = 0;
    for (uint32_t item = blockIdx.x + slot * gridDim.x; item < p.n_items; item += gridDim.x << p.slots_log, ++use) {
        // an output tile: item = tile * tiles_n + n
        uint32_t n;
        const uint32_t tile = p.by_tiles_n.divmod(item, n);
        int n_cols = min(p.n_tile, L.coutp - (int)n * p.n_tile) - c_first;
        if (p.col_split && c_first == 0) n_cols = min(n_cols, p.col_split);
        const int chunks = n_cols >> 4;                             // of 16 channels; a thread's are 4 * chunks consecutive ones
        const uint32_t n0 = n * (uint32_t)p.n_tile + (uint32_t)c_first, ch0 = n0 + word * 4u * (uint32_t)chunks;
        bool ready = false;
#pragma unroll 1
        for (int mt = 0; mt < kMT && chunks > 0; ++mt) {
            // byte offset of the output row whose number is this lane's (-1: padding), and of this thread's four rows
            int off[4];
            {
                const uint32_t f = tile * kTile + (uint32_t)(mt * kM + q * 32 + c.lane);
                uint32_t r, x;
                const uint32_t img = p.by_image.divmod(f, r), y = p.by_wp.divmod(r, x);
                const bool valid = f < p.positions && y < (uint32_t)L.hout && x < (uint32_t)L.wout;
                const int mine = valid ? (int)(((img * (uint32_t)L.hout + y) * (uint32_t)L.wout + x) * (uint32_t)L.coutp) : -1;
#pragma unroll
                for (int i = 0; i < 4; ++i) off[i] = __shfl_sync(0xffffffffu, mine, (c.lane >> 2) + 8 * i);
            }
            uint32_t io[4][4];                                      // residual bytes, then results
#pragma unroll
            for (int i = 0; i < 4; ++i) {
#pragma unroll
                for (int k = 0; k < 4; ++k) io[i][k] = 0;
                if (has_res && off[i] >= 0) {
                    const int8_t *src = p.res + (uint32_t)off[i] + ch0;
                    if (chunks == 4) ld_global_v4(src, io[i]);
                    else {
#pragma unroll
                        for (int k = 0; k < 3; ++k)
                            if (k < chunks) io[i][k] = ld_global_u32(src + 4 * k);
                    }
                }
            }
            if (!ready) {
                ready = __all_sync(0xffffffffu, wait_bar<kHintEpi>(bar_full, use & 1u, c.abort_flag));
                if (!ready) return false;
                tc_fence_after();
            }
            const uint32_t acc = acc0 + (uint32_t)(mt * p.n_tile), cst = c.sbase + p.cst_off + n0 * 16u + word * 16u;
            int a[2][8];
            tmem_ld_frag(acc, a[0]);
#pragma unroll
            for (int ch = 0; ch < 4; ++ch) {
                if (ch >= chunks) break;
                int4 k4[4];
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(k4[k].x), "=r"(k4[k].y), "=r"(k4[k].z), "=r"(k4[k].w) : "r"(cst + (uint32_t)(ch * 256 + k * 64)));
#pragma unroll
                for (int hf = 0; hf < 2; ++hf) {
                    tmem_ld_frag_wait(a[hf]);
                    // the next accumulators, before this step's arithmetic
                    if (hf == 0) tmem_ld_frag(acc + (uint32_t)(ch * 16) + (16u << 16), a[1]);
                    else if (ch + 1 < chunks) tmem_ld_frag(acc + (uint32_t)(ch * 16 + 16), a[0]);
                    else if (mt == kMT - 1) {
                        tc_fence_before();
                        mbar_arrive(bar_free);                      // the accumulators are in registers: the next tile may overwrite them
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
                                const int o = (int)ch0 + 4 * ch + k;
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
            for (int i = 0; i < 4; ++i) {
                if (off[i] < 0) continue;
                int8_t *dst = p.out + (uint32_t)off[i] + ch0;
                if (chunks == 4) st_global_v4(dst, io[i]);
                else if (chunks == 2) st_global_v2(dst, io[i][0], io[i][1]);
                else {
#pragma unroll
                    for (int k = 0; k < 3; ++k)
                        if (k < chunks) st_global_u32(dst + 4 * k, io[i][k]);
                }
            }
        }
        if (!ready) {                                               // the second team of a partial tile
            if (!__all_sync(0xffffffffu, wait_bar<kHintEpi>(bar_full, use & 1u, c.abort_flag))) return false;
            tc_fence_before();
            mbar_arrive(bar_free);
        }
    }
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

// A stages, position by position: lanes share a position's planes (16 bytes each).  Where a lane's N positions lie is worked out
// per tile and kept for the tile's stages: once by division, then by adding the distance from one tile of the CTA to the
// next, row by row and image by image.  (By division for each tile, and for twelve positions whatever the tile had, four
// gather warps took as long for a tile as everything else.)
template <int N>
__device__ __forceinline__ bool gather_flat(const HaloParams &p, uint32_t sbase, int gw, int lane, uint2 a_bars, const volatile int *abort_flag)
{
    const GLayer &L = p.L;
    const int lpp = 1 << p.lpp_log, per_warp = 32 >> p.lpp_log, chunk = lane & (lpp - 1);
    const uint32_t first_pos = (uint32_t)(gw * per_warp + (lane >> p.lpp_log)), step_pos = (uint32_t)(kGather * per_warp);
    const uint32_t win = (uint32_t)L.win, hin = (uint32_t)L.hin, wp = (uint32_t)p.wp, hp = (uint32_t)p.hp, image = wp * hp;
    Ring ring;
    uint32_t have = 0;                                              // positions that the tile has
#pragma unroll
    for (int i = 0; i < N; ++i) have |= first_pos + (uint32_t)i * step_pos < p.tile_pos ? 1u << i : 0u;
    // of each position, counted from one image before the first (so that the halo before the first tile is no negative
    // number): column, row, and byte offset of its pixel in the input, whether it has one or not
    uint32_t x[N], y[N], at[N], tile = 0;
    for (uint32_t item = blockIdx.x; item < p.n_items; item += gridDim.x) {
        const uint32_t next = p.by_tiles_n.div(item);
        if (item == blockIdx.x) {
            const uint32_t first = next * kTile + image - (uint32_t)p.halo + first_pos;
#pragma unroll
            for (int i = 0; i < N; ++i) {
                const uint32_t img = p.by_hp.divmod(p.by_wp.divmod(first + (uint32_t)i * step_pos, x[i]), y[i]);
                at[i] = ((img - 1u) * hin + y[i]) * win * (uint32_t)L.cinp + x[i] * (uint32_t)L.cinp;
            }
        } else {
            uint32_t dx, dy;
            const uint32_t di = p.by_hp.divmod(p.by_wp.divmod((next - tile) * kTile, dx), dy);
            const uint32_t d = ((di * hin + dy) * win + dx) * (uint32_t)L.cinp;
            const uint32_t wrap_x = (wp - win) * (uint32_t)L.cinp, wrap_y = (hp - hin) * win * (uint32_t)L.cinp;
#pragma unroll
            for (int i = 0; i < N; ++i) {
                x[i] += dx;
                y[i] += dy;
                at[i] += d;
                if (x[i] >= wp) { x[i] -= wp; y[i] += 1u; at[i] -= wrap_x; }
                if (y[i] >= hp) { y[i] -= hp; at[i] -= wrap_y; }
            }
        }
        tile = next;
        // positions of the tile that lie in no image: before the first, from the end of the last on
        const uint32_t first = tile * kTile + first_pos, begin = (uint32_t)p.halo, end = p.positions + begin;
        uint32_t inside = 0;
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const uint32_t f = first + (uint32_t)i * step_pos;
            inside |= x[i] < win && y[i] < hin && f >= begin && f < end ? 1u << i : 0u;
        }
        for (int plane = chunk, st = 0; st < p.n_stages; ++st, plane += p.stage_planes, ring.advance(p.ring_a)) {
            if (ring.use >= 1 && !wait_bar<kHintLoad>(a_bars.y + 8u * (uint32_t)ring.s, (uint32_t)(ring.use - 1) & 1u, abort_flag)) {
                cp_async_wait_all();
                return false;
            }
            if (plane < p.c16s) {
                const uint32_t dst = sbase + (uint32_t)ring.s * p.a_bytes + (uint32_t)chunk * p.plane_bytes + first_pos * 16u;
                const int8_t *src = p.in + plane * 16;
#pragma unroll
                for (int i = 0; i < N; ++i)
                    if ((have >> i) & 1u) cp_async16_cached(dst + (uint32_t)i * step_pos * 16u, (inside >> i) & 1u ? src + at[i] : p.zp_run);
            }
            cp_async_arrive(a_bars.x + 8u * (uint32_t)ring.s);
        }
    }
    cp_async_wait_all();
    return true;
}

__global__ void __launch_bounds__(kThreads, 1) k_halo(const __grid_constant__ HaloParams p)
{
    extern __shared__ __align__(128) uint8_t smem[];      // A stages | B blocks | constants
    __shared__ unsigned long long bar_a_full[kMaxRing], bar_a_free[kMaxRing], bar_b_full[kMaxRing], bar_b_free[kMaxRing], bar_acc_full[4], bar_acc_free[4];
    __shared__ uint32_t tmem_base_s;
    __shared__ volatile int abort_s;
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
    chain_start();
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
        const int gw = warp - kEpi;
        ok = p.flat_steps <= 6 ? gather_flat<6>(p, sbase, gw, lane, a_bars, &abort_s) : gather_flat<kFlat>(p, sbase, gw, lane, a_bars, &abort_s);
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
    int halo, wp, hp, c16s, tiles_n, n_tile, n_blocks, stage_planes, n_stages, ring_a, ring_b, resident, slots_log, col_split;
    uint32_t positions_tile, plane_positions, plane_bytes, a_bytes;
    size_t b_off, cst_off, smem;
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
    c->positions_tile = (uint32_t)(kTile + 2 * c->halo);
    c->plane_positions = (c->positions_tile + 1u) | 1u;          // an odd number of 16-byte rows: planes start in different banks; one to spare
    c->plane_bytes = c->plane_positions * 16u;
    const size_t cst = (size_t)c->tiles_n * c->n_tile * 16;
    const size_t block = (size_t)c->n_tile * G.kh * 32, all = block * (size_t)c->n_blocks * (size_t)c->tiles_n;
    // A stages of two pairs of planes where the channels are multiples of 64, else (or when three do not fit) of one;
    // the weights resident if they fit beside three stages, else a ring of at least three blocks
    for (int planes = c->c16s % 4 == 0 ? 4 : 2; planes >= 2; planes -= 2) {
        c->stage_planes = planes;
        c->n_stages = (c->c16s + planes - 1) / planes;
        c->a_bytes = (c->plane_bytes * (uint32_t)planes + 127u) & ~127u;
        const size_t fixed = cst;
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
        c->smem = c->cst_off + cst;
        return true;
    }
    return false;
}

// The team's block of an output tile that column `col` (of the padded output channels) lies in: its first column and width.
void halo_block(const GLayer &G, const HaloConfig &c, int col, int *first, int *width)
{
    const int tile = col / c.n_tile * c.n_tile, valid = std::min(c.n_tile, G.coutp - tile), in_tile = col - tile;
    const int split = c.col_split && valid > c.col_split ? c.col_split : valid;
    *first = tile + (in_tile < split ? 0 : split);
    *width = in_tile < split ? split : valid - split;
    if (in_tile >= valid) { *first = tile + valid; *width = 0; }          // padding
}

// The output channel of a column of the accumulators: column 16 t + 8 h + 2 c + e of a block of 16 u is channel
// 4 u c + 4 t + 2 h + e of it (see halo_epilogue).
int halo_channel(const GLayer &G, const HaloConfig &c, int col)
{
    int first, width;
    halo_block(G, c, col, &first, &width);
    if (!width) return col;
    const int b = col - first;
    return first + width / 4 * ((b >> 1) & 3) + 4 * (b >> 4) + ((b >> 2) & 2) + (b & 1);
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
    std::vector<int> channel((size_t)c.tiles_n * c.n_tile);
    for (size_t col = 0; col < channel.size(); ++col) channel[col] = halo_channel(G, c, (int)col);
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
                            const int oc = channel[(size_t)(t * c.n_tile + n)], ci = plane * 16 + e;
                            out[at] = (tap_x < k && oc < G.cout && ci < G.cin) ? w[(((size_t)oc * G.cin + ci) * k + r) * k + tap_x] : (int8_t)0;
                        }
                }
    for (int e = 0; e < 64; ++e) out[at + e] = (int8_t)G.zp_in;
}

// The constants of igemm_constants in the order in which the kernel reads them: the four of channels 4 u c + 4 t + k, c = 0 to 3, of
// a block lie side by side.
void halo_order_constants(const GLayer &G, int32_t *out4, int n_out)
{
    HaloConfig c;
    if (!halo_config(G, &c)) return;
    const std::vector<int32_t> in(out4, out4 + 4 * (size_t)n_out);
    for (int col = 0; col < n_out; ++col) {
        int first, width;
        halo_block(G, c, col, &first, &width);
        if (!width) continue;
        const int b = col - first;                       // position: t * 16 + k * 4 + c
        const int channel = first + width / 4 * (b & 3) + 4 * (b >> 4) + ((b >> 2) & 3);
        memcpy(out4 + 4 * (size_t)col, &in[4 * (size_t)channel], 16);
    }
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
    // By rows where a row's last step leaves at most an eighth of its lanes idle, or where there are more positions than a
    // lane keeps.  A layer of 512 samples by rows and by positions: 64 channels at 56 x 56 (rows of 57, steps of 8) 86 and 98
    // us, 128 at 28 x 28 (29) 51 and 53, 256 at 14 x 14 (15) 57 and 60; rows of one step, 512 at 7 x 7, 67 and 64.  A network of
    // 32, 64 and 128 channels at 32 x 32 to 8 x 8 (rows of 33 in steps of 16, of 17 and 9 in steps of 8): 2,394 and 2,200.
    const int step = 32 >> p.lpp_log, full = (c.wp + step - 1) / step * step;
    if (p.flat_steps > kFlat || (c.wp > step && 8 * (full - c.wp) <= full)) p.flat_steps = 0;
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
    p.b_off = (uint32_t)c.b_off; p.cst_off = (uint32_t)c.cst_off;
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
