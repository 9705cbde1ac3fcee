// What the layer-by-layer tensor-core convolutions share: MMA issue, the 32-bit requantisation, bounded barrier waits
// and asynchronous copies.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "isc_internal.h"
#include "isc_tc.cuh"

namespace isc {
namespace conv {

using namespace tc;

constexpr unsigned long long kWaitLimitNs = 2000000000ull;
constexpr unsigned kHintLoad = 20000, kHintEpi = 20000, kHintMma = 20000;      // suspend-time hint of a barrier wait (ns), by role
__device__ __forceinline__ void mma_i8(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n\t}"
                 ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void commit_to(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ long long mad_wide_u(uint32_t a, uint32_t b, long long c)
{
    long long d;
    asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
}

// Division of numbers below 2^31 by a constant of the launch: one multiplication's high half and a shift.  With
// 2^(s-1) < d <= 2^s and m = floor(2^(31+s) / d) + 1, floor(n / d) = floor(n m / 2^(31+s)) for n < 2^31, because the
// excess n (m - 2^(31+s) / d) / 2^(31+s) <= n / 2^(31+s) < 1 / d.  (d = 1: m = 0.)
struct FastDiv {
    uint32_t d, m, shift;
    __host__ static FastDiv make(uint32_t d)
    {
        if (d == 1) return FastDiv{1, 0, 0};
        uint32_t s = 1;
        while ((1ull << s) < d) ++s;
        return FastDiv{d, (uint32_t)((1ull << (31 + s)) / d + 1), s - 1};
    }
    __device__ __forceinline__ uint32_t div(uint32_t n) const { return m ? __umulhi(n, m) >> shift : n; }
    __device__ __forceinline__ uint32_t divmod(uint32_t n, uint32_t &r) const
    {
        const uint32_t q = div(n);
        r = n - q * d;
        return q;
    }
};

// The layers of a network as a chain of launches: a kernel may start when every block of the one before has started and
// leaves it room, sets itself up (barriers, tensor memory, constants; the stem also draws its noise), and waits for the end
// of the one before (chain_wait: complete, and its results visible) before it touches an activation.  Every kernel of a
// chain waits in every block, so the end of one is the end of all before it.  A kernel that takes tensor memory lets the next
// one start once it holds it: a block that has tensor memory and waits for the one before never keeps a block of that one
// from its own, whatever fits onto an SM together.  ResNet-50 at 100 samples, 57 launches: 1,753 ->
// 1,598 us; 4096 samples of a 20-layer network of 32 to 128 channels twice over: 2,961 -> 2,794 us.
__device__ __forceinline__ void chain_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
template <typename... Params, typename... Args>
cudaError_t launch_chained(bool chained, void (*kernel)(Params...), dim3 grid, unsigned threads, size_t smem, cudaStream_t st, const Args &...args)
{
    if (!chained) {
        kernel<<<grid, threads, smem, st>>>(args...);
        return cudaGetLastError();
    }
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = dim3(threads); cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cfg.attrs = &attr; cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, args...);
    if (e != cudaSuccess) cudaGetLastError();
    return e;
}

// 16 accumulators -> 16 int8 outputs with 32-bit arithmetic.  With s = shift - 1 >= 1,
//   rs((acc + bias) * mult, 31 + shift) + zp_out = (hi32((acc + bias) * mult) + c) >> s,  c = 2^(s-1) + zp_out * 2^s,
// exactly (the rounding half 2^(31+s) is a multiple of 2^32, so the product's low word cannot change the floor), and
//   rs((r - zp_res) * res_mult, n) = hi32(u * m2 + R2),  u = r + 128, m2 = res_mult * 2^(32-n), n = 31 or 32,
// with R2 = (2^(n-1) - (128 + zp_res) * res_mult) * 2^(32-n) (kRes = 1).  kRes = 2 is the same term as a single-precision
// product: round((256 k + u) * m) - c_r for an offset k and a multiplier m that the host has checked on all 256 values of
// u (residual_form; m2 then holds m's bits); 256 k is merged into u by the byte permute that extracts u, and c_r is folded
// into c.  A wide or high multiply takes four issue cycles of a scheduler here, two more than the single-precision one with
// everything around it: cycles per output and scheduler, sixteen warps looping over the sequence alone: add, mul.wide, add,
// shift 6.8, add, mad.hi, shift 6.3; with the residual term by permute, mul.wide, add 12.2, by permute, multiply, add 10.
// `cst` points at this block's constants in shared memory.
template <int kRes>
__device__ __forceinline__ uint4 requant16_fast(const int *acc, uint32_t cst, uint4 rv, uint32_t m2, long long r2, uint32_t k8, int lo)
{
    const uint32_t rw[4] = {rv.x ^ 0x80808080u, rv.y ^ 0x80808080u, rv.z ^ 0x80808080u, rv.w ^ 0x80808080u};
    uint32_t packed[4];
#pragma unroll
    for (int g = 0; g < 4; ++g) {
        int y[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            int4 c;
            asm("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(c.x), "=r"(c.y), "=r"(c.z), "=r"(c.w) : "r"(cst + (4 * g + k) * 16));
            int v = mad_hi(acc[4 * g + k] + c.x, c.y, c.z) >> c.w;
            if (kRes == 1) v += hi32(mad_wide_u(__byte_perm(rw[g], 0u, 0x4440u | (uint32_t)k), m2, r2));
            if (kRes == 2) v += mul_denormal(__byte_perm(rw[g], k8, 0x7650u | (uint32_t)k), m2);
            y[k] = max(v, lo);
        }
        packed[g] = pack4_sat(y[0], y[1], y[2], y[3]);
    }
    return make_uint4(packed[0], packed[1], packed[2], packed[3]);
}

// One output (see requant16_fast); kClamp: the lower clamp is above -128, which the packing saturates at.
template <int kRes, bool kClamp>
__device__ __forceinline__ int requant1(int acc, const int4 &c, uint32_t rword, int k, uint32_t m2, long long r2, uint32_t k8, int lo)
{
    int v = mad_hi(acc + c.x, c.y, c.z) >> c.w;
    if (kRes == 1) v += hi32(mad_wide_u(__byte_perm(rword, 0u, 0x4440u | (uint32_t)k), m2, r2));
    if (kRes == 2) v += mul_denormal(__byte_perm(rword, k8, 0x7650u | (uint32_t)k), m2);
    return kClamp ? max(v, lo) : v;
}

// 16 channels of two rows: a channel's constants are read once for both, because their reads bound the form above (a
// 16-byte broadcast per output: six outputs a clock and SM).  r0, r1: the residual bytes, offset by 128.
template <int kRes, bool kClamp>
__device__ __forceinline__ void requant16x2(const int (&a)[2][16], uint32_t cst, const uint32_t (&r0)[4], const uint32_t (&r1)[4], uint32_t m2, long long r2, uint32_t k8, int lo, uint4 (&o)[2])
{
    uint32_t w0[4], w1[4];
#pragma unroll
    for (int g = 0; g < 4; ++g) {
        int y0[4], y1[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            int4 cs;
            asm("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(cs.x), "=r"(cs.y), "=r"(cs.z), "=r"(cs.w) : "r"(cst + (uint32_t)(4 * g + k) * 16u));
            y0[k] = requant1<kRes, kClamp>(a[0][4 * g + k], cs, r0[g], k, m2, r2, k8, lo);
            y1[k] = requant1<kRes, kClamp>(a[1][4 * g + k], cs, r1[g], k, m2, r2, k8, lo);
        }
        w0[g] = pack4_sat(y0[0], y0[1], y0[2], y0[3]);
        w1[g] = pack4_sat(y1[0], y1[1], y1[2], y1[3]);
    }
    o[0] = make_uint4(w0[0], w0[1], w0[2], w0[3]);
    o[1] = make_uint4(w1[0], w1[1], w1[2], w1[3]);
}

// 32 accumulator columns of this thread's lane, asynchronously; the registers are valid after tmem_ld32_wait(),
// which names them so that no use can move above it
__device__ __forceinline__ void tmem_ld32_issue(uint32_t taddr, int (&v)[2][16])
{
    tmem_ld16_issue(taddr, v[0]);
    tmem_ld16_issue(taddr + 16u, v[1]);
}
__device__ __forceinline__ void tmem_ld32_wait(int (&v)[2][16])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(v[0][0]), "+r"(v[0][1]), "+r"(v[0][2]), "+r"(v[0][3]), "+r"(v[0][4]), "+r"(v[0][5]), "+r"(v[0][6]), "+r"(v[0][7]),
                   "+r"(v[0][8]), "+r"(v[0][9]), "+r"(v[0][10]), "+r"(v[0][11]), "+r"(v[0][12]), "+r"(v[0][13]), "+r"(v[0][14]), "+r"(v[0][15]),
                   "+r"(v[1][0]), "+r"(v[1][1]), "+r"(v[1][2]), "+r"(v[1][3]), "+r"(v[1][4]), "+r"(v[1][5]), "+r"(v[1][6]), "+r"(v[1][7]),
                   "+r"(v[1][8]), "+r"(v[1][9]), "+r"(v[1][10]), "+r"(v[1][11]), "+r"(v[1][12]), "+r"(v[1][13]), "+r"(v[1][14]), "+r"(v[1][15])
                 :: "memory");
}

// Bounded wait of a role for a phase of an mbarrier: false after the limit (the caller raises the error word) or when
// another role has raised the CTA's abort flag.  With `kHintNs` the wait is parked in hardware for up to that long per
// attempt instead of polling (the abort flag and the time limit are looked at every eighth attempt).
template <unsigned kHintNs>
__device__ __forceinline__ bool wait_bar(uint32_t bar, uint32_t parity, const volatile int *abort_flag)
{
    if (mbar_test(bar, parity)) return true;
    const unsigned long long t0 = globaltimer();
    for (int spin = 0;; ++spin) {
        if (kHintNs) {
            // parked in hardware until the phase completes or the hint runs out
            uint32_t done;
            asm volatile("{\n\t.reg .pred p;\n\t"
                         "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
                         "selp.u32 %0, 1, 0, p;\n\t}"
                         : "=r"(done) : "r"(bar), "r"(parity), "r"(kHintNs) : "memory");
            if (done) return true;
        } else if (mbar_try(bar, parity)) {
            return true;
        }
        if ((spin & 7) == 7 && (*abort_flag || globaltimer() - t0 > kWaitLimitNs)) return false;
    }
}

// A wait of a whole warp: every lane polls, all go on together.
__device__ __forceinline__ bool wait_warp(uint32_t bar, uint32_t parity, const volatile int *abort_flag)
{
    return __all_sync(0xffffffffu, wait_bar<kHintMma>(bar, parity, abort_flag)) != 0;
}

// MMA and commit by one lane of a converged warp: predicated, no branch
__device__ __forceinline__ void mma_i8_if(uint32_t lane0, uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 q, %5, 0;\n\t"
                 "@q tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n\t}"
                 ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(lane0) : "memory");
}
__device__ __forceinline__ void commit_if(uint32_t lane0, uint32_t bar)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %1, 0;\n\t"
                 "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}"
                 ::"r"(bar), "r"(lane0) : "memory");
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
// the same through L1: the taps of a 3 x 3 filter read a pixel's row nine times, and every CTA reads the zero-point run
__device__ __forceinline__ void cp_async16_cached(uint32_t dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
// one arrival on `bar` (counted in its initial count) once every cp.async this thread has issued so far is complete
__device__ __forceinline__ void cp_async_arrive(uint32_t bar)
{
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// activations to and from global memory, past the first-level cache
__device__ __forceinline__ void st_global_v4(void *p, const uint32_t (&v)[4])
{
    asm volatile("st.global.L1::no_allocate.v4.u32 [%0], {%1,%2,%3,%4};" ::"l"(p), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]) : "memory");
}
__device__ __forceinline__ void ld_global_v4(const void *p, uint32_t (&v)[4])
{
    asm volatile("ld.global.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "l"(p) : "memory");
}
__device__ __forceinline__ void st_global_v2(void *p, uint32_t a, uint32_t b) { asm volatile("st.global.L1::no_allocate.v2.u32 [%0], {%1,%2};" ::"l"(p), "r"(a), "r"(b) : "memory"); }
__device__ __forceinline__ void st_global_u32(void *p, uint32_t a) { asm volatile("st.global.L1::no_allocate.u32 [%0], %1;" ::"l"(p), "r"(a) : "memory"); }
__device__ __forceinline__ uint32_t ld_global_u32(const void *p)
{
    uint32_t v;
    asm volatile("ld.global.L1::no_allocate.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// A stage ring position: index and how many times the ring has wrapped.
struct Ring {
    int s = 0, use = 0;
    __device__ __forceinline__ void advance(int stages) { if (++s == stages) { s = 0; ++use; } }
};

// Bytes from one row of an epilogue warp's scratch to the next: an odd number of 16-byte columns, so that neither the
// row-wise nor the coalesced access has bank conflicts.
__host__ __device__ __forceinline__ uint32_t epi_row_stride(int n_tile) { return (((uint32_t)n_tile >> 4) | 1u) << 4; }

}  // namespace conv
}  // namespace isc
