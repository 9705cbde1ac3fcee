// Layer-by-layer engine: one kernel launch per layer over a batch of noisy samples, int8
// activations in global memory as [sample][y][x][channel padded to 16].  It runs every layer
// type of the ABI and any shape; the shared-memory-resident tensor-core engine
// (isc_line.cu) takes over for the CIFAR-shaped residual networks it is specialised for.
//
// The noisy copies of the image (Def. 3.4: x + delta, delta ~ discrete Gaussian of Eq. 2)
// are produced inside the first convolution's input staging and never written to memory.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "isc_conv.cuh"
#include "isc_epilogue.cuh"
#include "isc_internal.h"

namespace isc {

namespace {

// ------------------------------------------------------------------ random stream

// Philox4x32-10 (Salmon et al., SC'11): ten rounds of two 32x32->64 multiplies and xors,
// the key advanced by the Weyl constants between rounds.
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint32_t k0, uint32_t k1)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint32_t hi0 = __umulhi(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
        c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    return c;
}

// Smallest table index k in [0, 2T] with u < cum[k]; 2T when there is none.
__device__ __forceinline__ int dgauss_index(uint32_t u, const uint32_t *__restrict__ cum, int T)
{
    int lo = 0, hi = 2 * T;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (u < __ldg(cum + mid)) hi = mid; else lo = mid + 1;
    }
    return lo;
}

__device__ __forceinline__ uint4 sample_counter(const NoiseStream &ns, int64_t j, uint32_t block)
{
    return make_uint4(block, (uint32_t)(j & 0xFFFFFFFFll), ns.ctr2,
                      ns.ctr3_fixed | (uint32_t)(((j >> 32) & 0xFF) << 8));
}

__device__ __forceinline__ uint32_t word_of(const uint4 &v, int i)
{
    return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w;
}

// ------------------------------------------------------------------ dot products

__device__ __forceinline__ int dp4a_ss(int a, int b, int c) { return __dp4a(a, b, c); }

__device__ __forceinline__ int dp4a_us(uint32_t a, int b, int c)
{
    int d;
    asm("dp4a.u32.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}

// ------------------------------------------------------------------ first convolution

// One block = one sample x one band of output rows.  The band's input rows are drawn
// (Philox -> table search -> add -> saturate to 0..255) into shared memory as [row][col][4]
// bytes, then every thread computes output pixels x 16 output channels from that patch.
__global__ void __launch_bounds__(128)
k_first_conv(GLayer L, const uint8_t *__restrict__ images, int in_c, NoiseStream ns, SampleRun run, int band_rows,
             int8_t *__restrict__ out)
{
    extern __shared__ uint32_t patch[];   // [rows_in][wpad] packed 4 channels
    const int b = blockIdx.y;
    const SampleRun::Sample sample = run.at((uint32_t)b);
    const uint64_t image_id = run.image_id0 + sample.image;
    const uint8_t *__restrict__ x = images + sample.image * (size_t)(in_c * L.hin * L.win);
    const int64_t j = (int64_t)sample.number;
    ns.ctr2 = (uint32_t)image_id;
    ns.ctr3_fixed = sample.phase | ((uint32_t)(image_id >> 32) & 0xFFFFu) << 16;
    const int oy0 = blockIdx.x * band_rows;
    const int oy1 = min(L.hout, oy0 + band_rows);
    const int wpad = L.win + 2 * L.pad;
    const int iy0 = oy0 * L.stride - L.pad;                       // first input row of the patch
    const int rows_in = (oy1 - oy0 - 1) * L.stride + L.kh;
    const uint32_t zp_fill = (uint32_t)(L.zp_in & 0xFF) * (0x01010101u >> (8 * (4 - in_c)));   // padding value = zp_in

    for (int i = threadIdx.x; i < rows_in * wpad; i += blockDim.x) patch[i] = zp_fill;
    __syncthreads();

    // valid input rows of this band
    const int vy0 = max(0, iy0), vy1 = min(L.hin, iy0 + rows_in);
    if (vy1 > vy0) {
        uint8_t *pb = reinterpret_cast<uint8_t *>(patch);
        for (int c = 0; c < in_c; ++c) {
            const int64_t e_begin = ((int64_t)c * L.hin + vy0) * L.win;
            const int64_t e_end = ((int64_t)c * L.hin + vy1) * L.win;
            const int64_t q_begin = e_begin >> 2, q_end = (e_end + 3) >> 2;
            for (int64_t q = q_begin + threadIdx.x; q < q_end; q += blockDim.x) {
                const uint4 r = philox4x32_10(sample_counter(ns, j, (uint32_t)q), ns.key0, ns.key1);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int64_t e = q * 4 + k;
                    if (e < e_begin || e >= e_end) continue;
                    const int rem = (int)(e - (int64_t)c * L.hin * L.win);
                    const int h = rem / L.win, w = rem - h * L.win;
                    const int delta = dgauss_index(word_of(r, k), ns.cum, ns.T) - ns.T;
                    int v = (int)__ldg(x + e) + delta;
                    v = min(255, max(0, v));
                    pb[((h - iy0) * wpad + (w + L.pad)) * 4 + c] = (uint8_t)v;
                }
            }
        }
    }
    __syncthreads();

    const int groups = L.coutp >> 4;
    const int items = (oy1 - oy0) * L.wout * groups;
    const int taps = L.kh * L.kw;
    const int32_t *w32 = reinterpret_cast<const int32_t *>(L.w);
    for (int it = threadIdx.x; it < items; it += blockDim.x) {
        const int g = it / ((oy1 - oy0) * L.wout);
        const int p = it - g * ((oy1 - oy0) * L.wout);
        const int oyl = p / L.wout, ox = p - oyl * L.wout;
        int acc[16];
#pragma unroll
        for (int o = 0; o < 16; ++o) acc[o] = __ldg(L.bias + g * 16 + o);
        for (int r = 0; r < L.kh; ++r)
            for (int s = 0; s < L.kw; ++s) {
                const uint32_t a = patch[(oyl * L.stride + r) * wpad + ox * L.stride + s];
                const int32_t *wp = w32 + (size_t)(g * 16) * taps + r * L.kw + s;
#pragma unroll
                for (int o = 0; o < 16; ++o) acc[o] = dp4a_us(a, __ldg(wp + (size_t)o * taps), acc[o]);
            }
        const uint4 v = epilogue16(acc, L, g * 16, nullptr);
        const size_t px = ((size_t)b * L.hout + (oy0 + oyl)) * L.wout + ox;
        *reinterpret_cast<uint4 *>(out + px * L.coutp + g * 16) = v;
    }
}

// Debug aid: the noisy, saturated input of each sample as [sample][C][H][W] int32.
__global__ void k_noisy_input(const uint8_t *__restrict__ x, int d, NoiseStream ns, int batch,
                              int32_t *__restrict__ out)
{
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t nq = ((int64_t)d + 3) >> 2;
    if (idx >= nq * batch) return;
    const int b = (int)(idx / nq);
    const int64_t q = idx - (int64_t)b * nq;
    const uint4 r = philox4x32_10(sample_counter(ns, ns.first_sample + b, (uint32_t)q), ns.key0, ns.key1);
    for (int k = 0; k < 4; ++k) {
        const int64_t e = q * 4 + k;
        if (e >= d) break;
        const int delta = dgauss_index(word_of(r, k), ns.cum, ns.T) - ns.T;
        out[(int64_t)b * d + e] = min(255, max(0, (int)x[e] + delta));
    }
}

// ------------------------------------------------------------------ generic convolution / FC

// thread = one output pixel x 16 output channels; int8 x int8 dot products four at a time.
__global__ void __launch_bounds__(128)
k_conv(GLayer L, int batch, const int8_t *__restrict__ in, const int8_t *__restrict__ res,
       int8_t *__restrict__ out)
{
    const int64_t npx = (int64_t)batch * L.hout * L.wout;
    const int64_t px = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (px >= npx) return;
    const int g = blockIdx.y;
    const int ox = (int)(px % L.wout);
    const int oy = (int)((px / L.wout) % L.hout);
    const int b = (int)(px / ((int64_t)L.wout * L.hout));
    const int c16s = L.cinp >> 4;
    const int taps = L.kh * L.kw;
    const uint32_t zp4 = (uint32_t)(L.zp_in & 0xFF) * 0x01010101u;

    int acc[16];
#pragma unroll
    for (int o = 0; o < 16; ++o) acc[o] = __ldg(L.bias + g * 16 + o);

    for (int r = 0; r < L.kh; ++r) {
        const int iy = oy * L.stride + r - L.pad;
        for (int s = 0; s < L.kw; ++s) {
            const int ix = ox * L.stride + s - L.pad;
            const bool inside = iy >= 0 && iy < L.hin && ix >= 0 && ix < L.win;
            const uint4 *ap = reinterpret_cast<const uint4 *>(
                in + (((size_t)b * L.hin + (inside ? iy : 0)) * L.win + (inside ? ix : 0)) * L.cinp);
            const uint4 *wp = reinterpret_cast<const uint4 *>(L.w) +
                              ((size_t)(g * taps + r * L.kw + s) * c16s) * 16;
            for (int c = 0; c < c16s; ++c) {
                const uint4 a = inside ? __ldg(ap + c) : make_uint4(zp4, zp4, zp4, zp4);
#pragma unroll
                for (int o = 0; o < 16; ++o) {
                    const uint4 wv = __ldg(wp + c * 16 + o);
                    int t = acc[o];
                    t = dp4a_ss((int)a.x, (int)wv.x, t);
                    t = dp4a_ss((int)a.y, (int)wv.y, t);
                    t = dp4a_ss((int)a.z, (int)wv.z, t);
                    t = dp4a_ss((int)a.w, (int)wv.w, t);
                    acc[o] = t;
                }
            }
        }
    }
    const int8_t *res_px = res ? res + (size_t)px * L.coutp : nullptr;
    const uint4 v = epilogue16(acc, L, g * 16, res_px);
    *reinterpret_cast<uint4 *>(out + (size_t)px * L.coutp + g * 16) = v;
}

// ------------------------------------------------------------------ pools

// A warp takes 32 channels of one sample, four at a time per lane (the layout pads channels to 16), every fourth pixel per group
// of eight lanes.
__global__ void k_gavgpool(GLayer L, int batch, const int8_t *in, int8_t *out)
{
    conv::chain_start();
    conv::chain_wait();
    const int warp = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31, words = L.cinp >> 2, groups = (words + 7) >> 3;
    if (warp >= batch * groups) return;
    const int b = warp / groups, word = (warp - b * groups) * 8 + (lane & 7), hw = L.hin * L.win;
    const bool live = word < words;
    const int *p = reinterpret_cast<const int *>(in + (size_t)b * hw * L.cinp) + (live ? word : 0);
    long long total[4] = {0, 0, 0, 0};
    for (int i0 = 0; i0 < hw; i0 += 1 << 20) {                 // 32-bit sums of 2^20 bytes
        int sum[4] = {0, 0, 0, 0};
        for (int i = i0 + (lane >> 3); i < min(hw, i0 + (1 << 20)); i += 4) {
            const int v = p[(size_t)i * words];
            sum[0] = __dp4a(v, 1, sum[0]);
            sum[1] = __dp4a(v, 1 << 8, sum[1]);
            sum[2] = __dp4a(v, 1 << 16, sum[2]);
            sum[3] = __dp4a(v, 1 << 24, sum[3]);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            sum[k] += __shfl_xor_sync(0xffffffffu, sum[k], 8);
            sum[k] += __shfl_xor_sync(0xffffffffu, sum[k], 16);
            total[k] += sum[k];
        }
    }
    if (!live || lane >= 8) return;
    const int n = 31 + __ldg(L.shift), lo = L.relu ? max(-128, L.zp_out) : -128;
    uint32_t packed = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (4 * word + k >= L.cin) continue;
        long long v = ((total[k] - (long long)hw * L.zp_in) * (long long)__ldg(L.mult) + (1ll << (n - 1))) >> n;
        v += L.zp_out;
        v = v < lo ? lo : v;
        v = v > 127 ? 127 : v;
        packed |= (uint32_t)((int)v & 0xFF) << (8 * k);
    }
    reinterpret_cast<uint32_t *>(out)[b * words + word] = packed;
}

// Thread = one output pixel x 16 channels.  A tap outside the image repeats one inside the window, which changes no
// maximum, so that all taps of a 3 x 3 window (K = 3) are loaded without branches and together; the maximum of signed
// bytes is that of the 16-bit halves whose high byte they are (two packed maxima and a shift per four channels instead
// of an emulated four-byte one).  With 64-bit index arithmetic and a branch per tap the 3 x 3 stride-2 pool of a 112 x 112
// x 64 map took 146 us for 512 samples, now 84 us (6.1 TB/s of the measured 6.5).  K = 0: any window.
template <int K>
__global__ void k_maxpool(GLayer L, conv::FastDiv by_c16, conv::FastDiv by_w, uint32_t n, const int8_t *__restrict__ in, int8_t *__restrict__ out)
{
    conv::chain_start();
    conv::chain_wait();
    const uint32_t idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= n) return;
    uint32_t g, ox;
    const uint32_t px = by_c16.divmod(idx, g), oy = by_w.divmod(px, ox);
    const int kh = K ? K : L.kh, kw = K ? K : L.kw, y0 = (int)oy * L.stride - L.pad, x0 = (int)ox * L.stride - L.pad;
    const int8_t *src = in + (size_t)blockIdx.y * L.hin * L.win * L.cinp + g * 16;
    uint32_t odd[4], even[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) odd[k] = even[k] = 0x80008000u;
    if (y0 + kh > 0 && y0 < L.hin && x0 + kw > 0 && x0 < L.win) {
        auto tap = [&](int r, int c) {
            const int iy = min(max(y0 + r, 0), L.hin - 1), ix = min(max(x0 + c, 0), L.win - 1);
            uint4 v;                                             // not through the read-only path: the layer before may still have been running when this one started
            asm volatile("ld.global.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(src + (size_t)(iy * L.win + ix) * L.cinp));
            return v;
        };
        auto take = [&](const uint4 &a) {
            const uint32_t w[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                odd[k] = __vmaxs2(odd[k], w[k]);
                even[k] = __vmaxs2(even[k], w[k] << 8);
            }
        };
        if (K) {
            uint4 a[K ? K * K : 1];
#pragma unroll
            for (int i = 0; i < K * K; ++i) a[i] = tap(i / (K ? K : 1), i % (K ? K : 1));
#pragma unroll
            for (int i = 0; i < K * K; ++i) take(a[i]);
        } else {
            for (int r = 0; r < kh; ++r)
                for (int c = 0; c < kw; ++c) take(tap(r, c));
        }
    }
    uint32_t m[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) m[k] = __byte_perm(even[k], odd[k], 0x7351u);
    *reinterpret_cast<uint4 *>(out + ((size_t)blockIdx.y * L.hout * L.wout + px) * L.cinp + g * 16) = make_uint4(m[0], m[1], m[2], m[3]);
}

// ------------------------------------------------------------------ votes

// Argmax over the logits (lowest index wins ties; rows are 16-byte aligned) and one vote per sample; a warp's equal votes are one
// addition.  2^log_lanes lanes share a sample, a lane for 16 to 31 classes of up to 1,023, so that a row is read in whole sectors and many
// classes are no serial chain.  Logits go out as the run of bytes that the rows of the warp's samples are.  (With a
// thread per sample, calls for the logits of a small network with 4,096 classes took 208 us for one sample and 4.2 ms for 3,000,
// 21 ms after a layer that leaves the SM little L1; now 77 us and 3.0 ms, most of it the copy to the host.)
__global__ void k_votes(const int8_t *logits, int cp, int n_classes, conv::FastDiv by_classes, int log_lanes, SampleRun run, int batch,
                        int32_t *__restrict__ counts, int8_t *__restrict__ logits_out)
{
    conv::chain_start();
    const uint32_t thread = blockIdx.x * blockDim.x + threadIdx.x, sub = thread & ((1u << log_lanes) - 1u), lane = threadIdx.x & 31u;
    const uint32_t b = thread >> log_lanes;
    const bool live = b < (uint32_t)batch;
    const unsigned voters = __ballot_sync(0xffffffffu, live && sub == 0);
    conv::chain_wait();
    const int8_t *p = logits + (size_t)b * cp;
    int best = 0, bestv = -1000;
    for (int k0 = (int)sub * 16; live && k0 < n_classes; k0 += 16 << log_lanes) {
        const uint4 v = *reinterpret_cast<const uint4 *>(p + k0);
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const int l = (int)(w[k >> 2] << (24 - 8 * (k & 3))) >> 24;
            if (k0 + k < n_classes && l > bestv) { bestv = l; best = k0 + k; }
        }
    }
    for (int d = 1; d < 1 << log_lanes; d <<= 1) {
        const int v = __shfl_xor_sync(0xffffffffu, bestv, d), o = __shfl_xor_sync(0xffffffffu, best, d);
        if (v > bestv || (v == bestv && o < best)) { bestv = v; best = o; }
    }
    if (live && sub == 0) {
        const size_t at = (size_t)run.at(b).row * n_classes + best;
        const unsigned same = __match_any_sync(voters, (unsigned long long)at);
        if (lane == (uint32_t)__ffs(same) - 1u) atomicAdd(counts + at, __popc(same));
    }
    if (!logits_out) return;
    const uint32_t first = (thread - lane) >> log_lanes;                 // the warp's samples
    if (first >= (uint32_t)batch) return;
    const uint32_t n = min(32u >> log_lanes, (uint32_t)batch - first) * (uint32_t)n_classes;
    int8_t *to = logits_out + (size_t)first * n_classes;
    for (uint32_t i = lane; i < n; i += 128u) {
        int8_t v[4];
#pragma unroll
        for (uint32_t k = 0; k < 4; ++k) {
            uint32_t c;
            const uint32_t row = by_classes.divmod(min(i + 32u * k, n - 1u), c);
            v[k] = logits[(size_t)(first + row) * cp + c];
        }
#pragma unroll
        for (uint32_t k = 0; k < 4; ++k)
            if (i + 32u * k < n) to[i + 32u * k] = v[k];
    }
}

}  // namespace

// ------------------------------------------------------------------ launchers

cudaError_t launch_first_conv(const GLayer &L, const uint8_t *x_chw, int in_c, const NoiseStream &ns, const SampleRun &run,
                              int batch, int8_t *out, cudaStream_t st)
{
    const int wpad = L.win + 2 * L.pad;
    int band = 8;
    while (band > 1 && (size_t)((band - 1) * L.stride + L.kh) * wpad * 4 > 40 * 1024) band >>= 1;
    const size_t smem = (size_t)((band - 1) * L.stride + L.kh) * wpad * 4;
    if (smem > 48 * 1024) return cudaErrorInvalidValue;
    dim3 grid((L.hout + band - 1) / band, batch);
    k_first_conv<<<grid, 128, smem, st>>>(L, x_chw, in_c, ns, run, band, out);
    return cudaGetLastError();
}

cudaError_t launch_noisy_input(const uint8_t *x_chw, int in_c, int in_h, int in_w, const NoiseStream &ns,
                               int batch, int32_t *out_chw, cudaStream_t st)
{
    const int d = in_c * in_h * in_w;
    const int64_t n = (((int64_t)d + 3) >> 2) * batch;
    k_noisy_input<<<(unsigned)((n + 127) / 128), 128, 0, st>>>(x_chw, d, ns, batch, out_chw);
    return cudaGetLastError();
}

cudaError_t launch_conv(const GLayer &L, int batch, const int8_t *in, const int8_t *res, int8_t *out,
                        cudaStream_t st)
{
    const int64_t npx = (int64_t)batch * L.hout * L.wout;
    dim3 grid((unsigned)((npx + 127) / 128), L.coutp >> 4);
    k_conv<<<grid, 128, 0, st>>>(L, batch, in, res, out);
    return cudaGetLastError();
}

cudaError_t launch_gavgpool(const GLayer &L, int batch, const int8_t *in, int8_t *out, cudaStream_t st, bool chained)
{
    const int warps = batch * (((L.cinp >> 2) + 7) >> 3);
    return conv::launch_chained(chained, k_gavgpool, dim3((unsigned)((warps + 3) / 4)), 128, 0, st, L, batch, in, out);
}

cudaError_t launch_maxpool(const GLayer &L, int batch, const int8_t *in, int8_t *out, cudaStream_t st, bool chained)
{
    const uint32_t n = (uint32_t)(L.hout * L.wout * (L.cinp >> 4));
    const conv::FastDiv by_c16 = conv::FastDiv::make((uint32_t)(L.cinp >> 4)), by_w = conv::FastDiv::make((uint32_t)L.wout);
    for (int b = 0; b < batch; b += 65535) {                     // a launch's second grid dimension holds no more
        const dim3 grid((n + 127) / 128, (unsigned)std::min(batch - b, 65535));
        const int8_t *src = in + (size_t)b * L.hin * L.win * L.cinp;
        int8_t *dst = out + (size_t)b * L.hout * L.wout * L.cinp;
        const cudaError_t e = conv::launch_chained(chained, L.kh == 3 && L.kw == 3 ? k_maxpool<3> : k_maxpool<0>, grid, 128, 0, st, L, by_c16, by_w, n, src, dst);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_votes(const int8_t *logits_nhwc, int cp, int n_classes, const SampleRun &run, int batch, int32_t *counts,
                         int8_t *logits_out, cudaStream_t st, bool chained)
{
    int log_lanes = 0;
    while (log_lanes < 5 && 32 << log_lanes <= n_classes) ++log_lanes;
    return conv::launch_chained(chained, k_votes, dim3((unsigned)((((int64_t)batch << log_lanes) + 127) / 128)), 128, 0, st, logits_nhwc, cp, n_classes,
                                conv::FastDiv::make((uint32_t)n_classes), log_lanes, run, batch, counts, logits_out);
}

}  // namespace isc
