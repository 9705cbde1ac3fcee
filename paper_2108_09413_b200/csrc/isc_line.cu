// Line-tiled shared-memory-resident tensor-core engine (sm_100a) for CIFAR-shaped residual networks.
//
// One persistent CTA per SM carries a group of four noisy samples through the whole network.  Activations
// stay in shared memory, every convolution is an implicit GEMM on tcgen05 (kind::i8, int32 accumulators in
// tensor memory) and only vote counts return to global memory (Algorithm 1 steps 1-4, Algorithm 2 steps 1-2).
//
// Layout.  A tensor of C channels and H x W pixels (W = 32, 16 or 8) is stored per plane of 16 channels as
// "lines" of 128 positions of 16 bytes.  Position x * I + b * 4 + s of line l holds pixel (row l + b * L, column x)
// of sample s, where I = 128 / W positions belong to one column, I / 4 row bands b share a line and L = H / (I / 4)
// is the number of lines.  Lines are I positions apart from each other (a gap that always holds the zero-point:
// the left and right padding of every row), there is one more line above and below (the padding rows of the
// first and last band; for the other bands these two lines hold copies of the neighbouring band's edge rows,
// written together with the originals), so
//   * the horizontal neighbours of all 128 positions of a line are the same 128 positions moved by +-I, and
//   * the vertical neighbours of all 128 positions of line l are the same 128 positions of line l +- 1.
// A line is therefore an M = 128 operand tile whose nine filter taps are plain address offsets, with every one
// of its rows a real output pixel.
//
// Stacked convolutions.  For a 3x3, stride-1 convolution the three vertical taps are stacked along N: one MMA
// chain over input line p (K = three horizontal taps x input channels) accumulates into the accumulator
// columns of output lines p-1, p, p+1 at once (N = 3 x cout), because the accumulators of consecutive output
// lines are consecutive column blocks of tensor memory.  The epilogue, once it has read a line's columns, puts there what
// the next convolution on them starts from: its folded biases.  This triples N where an MMA is bound by fetching its
// 128 x 32-byte A operand.  With 16 input channels two lines share their odd K units (three MMAs for two lines).  Strided
// and 1x1 convolutions run unstacked: one chain per output line over all taps.
//
// Roles.  Three issuing warps (lane 0 of each) share the MMA chains of a convolution: the host prepares a table of
// operations (accumulator columns, descriptor offsets, which units of the previous convolution must be stored,
// which units complete) in the order in which their inputs become available; operation i belongs to issuing warp
// i mod 3.  One thread alone cannot feed the tensor pipe: an MMA costs it about a hundred cycles of issue latency and
// a commit as much again, so the loop is kept to the fewest instructions (dependency counters read together, the
// timed wait out of line).  Sixteen epilogue warps requantise: four sets of four warps (one per 32-lane quarter of
// tensor memory) share the items of a convolution, an item being one unit (two or four output lines: one
// "accumulators complete" barrier pair, one "stored" counter) and one 16-channel chunk, in the order in which they
// complete.  An epilogue thread reads accumulators as fragments (tcgen05.ld 16x256b: four positions, four consecutive
// channels of each), so that a channel's constants, held in registers for the pass, serve four outputs and residual and
// result bytes move as words (with a position per thread every output took its constants from shared memory: a ResNet-110
// group 460 -> 397 us; the shared K units of 16 input channels then brought it to 375).  The requantisation is integer arithmetic on a pipe that issues multiplies,
// shifts and packs at half rate: the pass is written for the fewest such instructions (see requant4).  A loader warp copies the next
// convolution's blob once its place is free.  Consecutive convolutions overlap unit by unit.  Input noise (Def. 3.3,
// Eq. 2; Def. 3.4), halo fills and the pool / FC / argmax tail are CTA-wide phases between barriers.
//
// Every device-side wait is bounded by a wall-clock limit; on expiry the CTA raises an abort flag, all
// remaining waits fall through, and the host reports ISC_ERR_TIMEOUT.
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <map>
#include <vector>

#include "isc_line.h"
#include "isc_tc.cuh"

namespace isc {

using namespace tc;

namespace {

constexpr int kG = 4;                       // samples per group
constexpr int kEpiWarps = 16;               // the first warps: epilogue; set = warp / 4, tensor-memory quarter = warp % 4
constexpr int kSets = kEpiWarps / 4;
constexpr int kIssuers = 3;                 // the next warps: lane 0 of each issues every kIssuers-th MMA chain of a convolution
constexpr int kLoaderWarp = kEpiWarps + kIssuers;   // the last warp: weight copies
constexpr int kThreads = 32 * (kEpiWarps + kIssuers + 1);
constexpr int kMaxKsteps = 18;
constexpr int kMaxPhases = 160;
constexpr int kMaxBars = 128;
constexpr int kMaxLines = 32;               // output lines of one convolution
constexpr int kCtrlBytes = 10240;
constexpr int kMaxConv = 128;
// How a network is planned; the first way that succeeds is taken.  `chains`: MMA chains of an operation at most; a record of
// several may name more units than it has room for.  The ways from the third on are for networks that keep three tensors of
// 72 KB and have 6 KB left for blobs: a paired convolution's blob is 1.3 to 1.9 KB larger than an unpaired one's.  Packed:
// tensors from the top, which leaves the room in one piece, and other places; a blob's header ends with its last K-step;
// a strided convolution has the units, and may share the barriers, of a general one.
struct PlanTry { int chains; bool paired, packed; };
constexpr PlanTry kPlanTries[] = {{2, true, false}, {1, true, false}, {4, false, false}, {1, false, false}, {2, true, true}, {1, true, true}, {4, false, true}, {1, false, true}};
constexpr int kPlanUsual = 2, kPackAttempts = 200;
constexpr int kPlanRuleBars = 14, kPlanRuleRoom = 15;          // after another rule's refusal the ways from the third on are no help
constexpr int kSmemLimit = 227 * 1024;
constexpr int kTmemCols = 512;
constexpr int kSideStreams = 8;             // concurrent launches when a launch does not fill the GPU
constexpr unsigned long long kWaitLimitNs = 2000000000ull;   // 2 s per wait

enum { PH_FILL = 0, PH_INPUT = 1, PH_CONV = 2, PH_TAIL = 3 };
enum { ERR_NONE = 0, ERR_WAIT_DONE = 1, ERR_WAIT_WEIGHTS = 2, ERR_WAIT_READY = 3, ERR_WAIT_FULL = 4, ERR_WAIT_DRAIN = 5 };
enum { CF_PAIRED = 1, CF_RES = 2, CF_RES_LONG = 4, CF_SCATTER = 8, CF_GENERAL = 16 };         // CF_PAIRED: chains over two lines; CF_RES_LONG: the residual term is no product; CF_GENERAL: the pass that decides everything at run time
// OPF_WAIT_ALL: every unit of the previous convolution; OPF_WAITS / OPF_WAITS4: the record names counters to test (two /
// four slots in use); bits 4-6: how many of them are distinct; bits 8-9: arrivals; bits 10-12: MMA chains
enum { OPF_WAIT_ALL = 1, OPF_WAITS = 2, OPF_WAITS4 = 8 };

// ---- what the kernel reads -------------------------------------------------------------------

// One entry per phase, copied to shared memory when the kernel starts.
//   CONV: a = shared-memory offset of the blob, b = convolutions that follow each other from here on      FILL: a = offset, b = bytes, c = halo byte
struct alignas(16) PhaseEntry { uint32_t kind, a, b, c; };

// Where the blob of convolution c comes from (global) and goes to (shared).
// and which convolution must be complete before the copy may start: the counters stored[dep_first .. + dep_units)
// must have reached dep_mult * (group * dep_uses + dep_local + 1); dep_units = 0: nothing to wait for.
struct alignas(16) ConvSrc {
    unsigned long long gmem;
    uint32_t bytes_phase, smem_off;                 // bytes | phase << 24; offset | late << 31
    uint32_t dep_first, dep_units, dep_mult, dep_local_uses;     // dep_local | dep_uses << 16
};

// MMA chains over an input line, or over up to two consecutive pairs of lines (paired convolutions), in the form an issuing
// thread consumes: accumulator columns, what to add to the operand descriptors' start addresses, and the barriers (as byte
// offsets, 0xFFFF = none) of its dependencies and completions.
struct alignas(16) LOp {
    uint32_t d_col;         // first accumulator column within the bank
    uint32_t idesc;         // instruction descriptor (N = blocks * cout; paired: blocks = 0)
    uint32_t a_add, b_add;  // 16-byte units: (input line + 1) * pitch, first weight block * block size; paired: kPairInner, or per K-step
                            // k, at bit 7 k: output lines (3 bits), first weight block (2), first output line behind d_col's (2)
    uint16_t wait[4];       // 4 * unit of the previous convolution that must be stored
    uint16_t commit[3];     // 8 * unit of this convolution whose accumulators are complete after the chain
    uint16_t flags;         // OPF_* | distinct waits << 4 | arrivals << 8 | chains << 10
};
// a pair of lines away from the tensor's edges: lines p - 1 .. p + 1, p - 1 .. p + 2, p .. p + 2
constexpr uint32_t kPairInner = (3u | 0u << 3 | 0u << 5) | (4u | 0u << 3 | 0u << 5) << 7 | (3u | 0u << 3 | 1u << 5) << 14;
static_assert(sizeof(LOp) == 32, "one operation is two 16-byte loads");

// Head of every blob: first what an epilogue warp reads, then what only some need.
struct alignas(16) LConvDesc {
    uint32_t flags, n_items, recs_per_item, d_base;         // (unit, chunk) pairs; records of the pass table for each; first accumulator column
    uint32_t bar_full, bar_done, use_local, uses_per_group;  // barrier indices of this class
    uint32_t n_units, c_rel, passes_rel, out_base;          // units (their barriers); constants, pass table; output (line 0, lane 0, plane 0)
    uint32_t res_base, res_m2, res_k8, dup_delta;           // residual operand and its term; bytes from a band's first row to its copy below the band above it, 0: one band
    // geometry of the output and of the scattered input
    uint32_t out_plane, out_pitch16, out_log_lines, out_logI;
    uint32_t in_logI, in_n_lines, out_nb, vec_rel;           // vec_rel: start values for the accumulators' next use, 16 channels each
    // the general pass
    int32_t lo; uint32_t res_r2_lo, res_r2_hi, gen_res_m2;
    // issuing threads
    uint32_t n_ops, n_ksteps, ops_rel, n_chunks;
    uint32_t b_lo0, kstep16, pitch16, cols;                  // b_lo0: low word of the first K-step's weight descriptor (shared-memory base 0)
    uint32_t a_lo[kMaxKsteps + 2];             // low words of the operand descriptors of line -1 (shared-memory base 0)
};
static_assert(sizeof(LConvDesc) % 16 == 0, "blob sections stay 16-byte aligned");

struct FcConst { int32_t mult, n, zp_out, lo, bias, pad0, pad1, pad2; };

struct LineParams {
    const PhaseEntry *ptab;
    const ConvSrc *conv_src;
    const uint8_t *bar_counts;
    int32_t n_bars, n_phases, n_conv, n_groups;
    int32_t in_c, in_H, in_W;
    // What the groups of four samples are: per image, groups_sel groups of the selection phase (n_sel samples from
    // number 0 on), then groups_est of the estimation phase (n_est samples from ns.first_sample on).
    int32_t groups_sel, groups_est, n_sel, n_est, phase_sel;
    unsigned long long image_id0;     // of image 0
    const uint8_t *x;                 // clean images, CHW, one after the other
    NoiseStream ns;                   // ctr3_fixed: the estimation phase's number; ctr2 is not used
    uint32_t input_base, input_pitch16;   // line 0, lane 0 of the first layer's operand region
    // tail
    uint32_t tail_base, tail_plane, tail_pitch16, tail_logI;
    int32_t tail_C, tail_H, tail_W, tail_n_lines;
    int32_t pool_mult, pool_n, pool_zp_in, pool_zp_out, pool_lo;
    const int8_t *fc_w;               // [n_classes][64]
    const FcConst *fc_c;
    int32_t n_classes;
    int32_t *counts;                  // [image][phases in use][n_classes]
    int8_t *logits;                   // [n_est][n_classes] or null (one image, no selection phase)
    int32_t *err;
    unsigned long long *phase_cycles; // [4]: SM cycles per CTA spent in FILL, INPUT, everything else, TAIL, summed over CTAs and launches
    // debug
    const int32_t *acc_init;          // [kTmemCols]: the accumulators' values before the first group
    int32_t stop_phase;
    uint32_t dump_off, dump_bytes;
    uint8_t *dump;
};

struct Ctrl {
    unsigned long long bars[kMaxBars];
    unsigned long long wbar[3], drain;
    uint32_t tmem_base;
    volatile int abort_flag;
    uint32_t stored[kMaxBars];              // per unit: stores of its 16-channel chunks by a warp, counted over the whole run
    int32_t pool_sum[kG][64];               // the tail's sums over the pixels, zero between groups
    alignas(16) int8_t pooled[kG][64];      // its pooled features, one row per sample of the group
    long long cyc[4], cyc_mark;             // thread 0's phase clocks
    PhaseEntry ptab[kMaxPhases];
    ConvSrc csrc[kMaxConv];
};
static_assert(sizeof(Ctrl) <= kCtrlBytes - 16, "control block too large");

// ------------------------------------------------------------------ device helpers
//
// Nothing on a convolution's path may use local memory: with 227 KB of shared memory per SM the first-level cache is too
// small for 640 threads' stacks, and every spilled register or structure on the stack costs a trip to the second level
// (a convolution's fixed cost per warp was 2,900 cycles so).  Hence the kernel makes no calls, and shared memory is addressed
// through the array's constant address.
extern __shared__ __align__(128) uint8_t smem[];
__device__ __forceinline__ Ctrl *the_ctrl() { return reinterpret_cast<Ctrl *>(smem); }
__device__ __forceinline__ uint32_t the_base() { return smem_u32(smem); }
#define CTRL_ADDR(member) (the_base() + (uint32_t)offsetof(Ctrl, member))

// D += A * B: accumulators start from their channels' folded biases (see LPass)
__device__ __forceinline__ void mma_i8(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.eq.b32 p, 0, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n\t}"
                 ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc) : "memory");
}
__device__ __forceinline__ void commit_to(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// 16 columns of all 32 lanes take the values at `vec` (shared memory), one per column.  (In fragment form, four values per
// thread, the store's eight registers had to be copied together each time: 230 instead of 60 cycles of a pass of 1,050.)
__device__ __forceinline__ void tmem_st_columns(uint32_t taddr, uint4 a, uint4 b, uint4 c, uint4 d)
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
                 ::"r"(taddr), "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w),
                   "r"(c.x), "r"(c.y), "r"(c.z), "r"(c.w), "r"(d.x), "r"(d.y), "r"(d.z), "r"(d.w) : "memory");
}
__device__ __forceinline__ void tmem_st_columns(uint32_t taddr, uint32_t vec)
{
    tmem_st_columns(taddr, ld_shared_v4(vec), ld_shared_v4(vec + 16u), ld_shared_v4(vec + 32u), ld_shared_v4(vec + 48u));
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ long long mad_wide_u(uint32_t a, uint32_t b, long long c)
{
    long long d;
    asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
}
// Per-channel requantisation constants of a thread's four channels 4 c .. 4 c + 3 of a chunk, as stored in the blob (48 bytes):
// multipliers, rounding addends, shifts.  The accumulators start from the folded bias.  With s = shift - 1 >= 1,
//   rs(acc * mult, 31 + shift) + zp_out = (hi32(acc * mult) + c) >> s,   c = 2^(s-1) + zp_out * 2^s,
// exactly: the rounding half 2^(31+s) is a multiple of 2^32, so the low word of the product cannot change the floor.
// For s = 0 the half sits in the low word: the result is hi32 + (bit 31 of the low word) + c with c = zp_out.
// A scheduler issues a wide or high multiply in four cycles here, shifts, permutes and packs in two, additions in one: this
// form is the cheapest exact one found (mad.hi, shift; 5.1 cycles per output where add, wide multiply, add, shift take 6.8).
struct ChanConsts { int mult[4], c[4], s[4]; };
__device__ __forceinline__ ChanConsts ld_chan_consts(uint32_t addr)
{
    ChanConsts k;
    asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(k.mult[0]), "=r"(k.mult[1]), "=r"(k.mult[2]), "=r"(k.mult[3]) : "r"(addr));
    asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(k.c[0]), "=r"(k.c[1]), "=r"(k.c[2]), "=r"(k.c[3]) : "r"(addr + 16u));
    asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(k.s[0]), "=r"(k.s[1]), "=r"(k.s[2]), "=r"(k.s[3]) : "r"(addr + 32u));
    return k;
}
constexpr uint32_t kChunkConstBytes = 4 * 48, kVecBytes = 64;
__device__ __forceinline__ long long mul_wide(int a, int b)
{
    long long d;
    asm("mul.wide.s32 %0, %1, %2;" : "=l"(d) : "r"(a), "r"(b));
    return d;
}
__device__ __forceinline__ void red_release_add(uint32_t addr, uint32_t v)
{
    asm volatile("red.release.cta.shared::cta.add.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t ld_volatile_u32(uint32_t addr)
{
    uint32_t v;
    asm volatile("ld.volatile.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t ld_acquire_u32(uint32_t addr)
{
    uint32_t v;
    asm volatile("ld.acquire.cta.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}
// Bounded waits.  On expiry: the abort flag and the error word, wait kind | index of the barrier within the control block << 8 |
// parity waited for << 20 | CTA << 21.
struct Waiter {
    int32_t *err;
    unsigned long long limit_ns = kWaitLimitNs;
    static __device__ __forceinline__ bool aborted() { return ld_volatile_u32(CTRL_ADDR(abort_flag)) != 0u; }
    __device__ __forceinline__ void fail(int code, uint32_t bar, uint32_t parity) const
    {
        the_ctrl()->abort_flag = 1;
        const uint32_t idx = (bar - the_base()) >> 3;
        atomicCAS(err, 0, (int)((uint32_t)code | ((idx & 0xFFFu) << 8) | ((parity & 1u) << 20) | (blockIdx.x << 21)));
    }
    // Wait for a phase of an mbarrier.  Each attempt parks the thread in hardware for a bounded time,
    // so a waiting warp does not compete for issue slots; the clock is read only when the first gives up.
    __device__ __forceinline__ bool barrier(uint32_t bar, uint32_t parity, int code) const
    {
        if (mbar_try(bar, parity)) return true;
        const unsigned long long t0 = globaltimer();
        for (int spin = 0;; ++spin) {
            if (mbar_try(bar, parity)) return true;
            if ((spin & 7) == 7) {
                if (aborted()) return false;
                if (globaltimer() - t0 > limit_ns) { fail(code, bar, parity); return false; }
            }
        }
    }
    // Wait until a counter in shared memory has reached `expected` (counters only grow).
    __device__ __forceinline__ bool counter(uint32_t addr, uint32_t expected, int code) const
    {
        const unsigned long long t0 = globaltimer();
        for (int spin = 0;; ++spin) {
            if ((int32_t)(ld_acquire_u32(addr) - expected) >= 0) return true;
            if ((spin & 15) == 15) {
                if (aborted()) return false;
                if (globaltimer() - t0 > limit_ns) { fail(code, addr, 0); return false; }
            }
        }
    }
};

// ------------------------------------------------------------------ issuing thread

struct PrevConv { uint32_t done_addr, expected, n_lines; };    // counters of its units, their value when stored; n_lines = 0: nothing to wait for

// The barrier of the next blob: three, used in turn.
struct WeightSlot {
    uint32_t slot = 0, parity = 0;
    __device__ __forceinline__ void advance() { if (++slot == 3u) { slot = 0; parity ^= 1u; } }
};

struct IssueCtx {
    uint32_t desc, ops, n_ops, s16, b_lo0, kstep16, d0, full_addr, issuer, pitch16, cols;
};

// How an issuing thread polls a "stored" counter.  A volatile load by default (a weak one could be moved out of the loop): an
// acquiring one costs over a hundred cycles per test on the issue path.  What the counter guards was published by the
// storing warp with a proxy fence and a releasing add; the MMAs that read it are issued after the value was seen (control
// dependency) and after tcgen05.fence::after_thread_sync.  Building with -DISC_ACQUIRE_POLL takes the acquiring form
// instead, so that a divergence could be traced to this choice.
__device__ __forceinline__ uint32_t ld_counter(uint32_t addr)
{
#ifdef ISC_ACQUIRE_POLL
    return ld_acquire_u32(addr);
#else
    return ld_volatile_u32(addr);
#endif
}

// The operations of one convolution that belong to one issuing thread (every kIssuers-th record).  The low words of
// the operand descriptors stay in registers; an operation adds its line and block offsets to their start-address
// fields.  The counters an operation depends on are read together (unused slots repeat the first one) and compared
// once; what the counters guard was made visible to the tensor cores' reads by the storing warp (proxy fence, then a
// releasing add) and is read by MMAs that are issued only after the values have been seen.
__device__ __forceinline__ bool op_wait(const Waiter &w, const PrevConv &prev, uint4 r1)
{
    const uint32_t fl = r1.w >> 16;
    if (fl & OPF_WAIT_ALL) {
        for (uint32_t l = 0; l < prev.n_lines; ++l)
            if (!w.counter(prev.done_addr + 4 * l, prev.expected, ERR_WAIT_DONE)) return false;
    }
    if (fl & OPF_WAITS) {
        const unsigned long long t0 = globaltimer();
        for (int spin = 0;; ++spin) {
            int32_t m = min((int32_t)(ld_counter(prev.done_addr + (r1.x & 0xFFFFu)) - prev.expected),
                            (int32_t)(ld_counter(prev.done_addr + (r1.x >> 16)) - prev.expected));
            if (fl & OPF_WAITS4)
                m = min(m, min((int32_t)(ld_counter(prev.done_addr + (r1.y & 0xFFFFu)) - prev.expected),
                               (int32_t)(ld_counter(prev.done_addr + (r1.y >> 16)) - prev.expected)));
            if (m >= 0) break;
            if ((spin & 63) == 63) {
                if (Waiter::aborted()) return false;
                if (globaltimer() - t0 > w.limit_ns) { w.fail(ERR_WAIT_DONE, prev.done_addr + (r1.x & 0xFFFFu), 0); return false; }
            }
        }
    }
    tc_fence_after();
    return true;
}
__device__ __forceinline__ void op_commit(const IssueCtx &ic, uint4 r1)
{
    const uint32_t nc = (r1.w >> 24) & 3u;
    if (nc) {
        commit_to(ic.full_addr + (r1.z & 0xFFFFu));
        if (nc > 1) {
            commit_to(ic.full_addr + (r1.z >> 16));
            if (nc > 2) commit_to(ic.full_addr + (r1.w & 0xFFFFu));
        }
    }
}

// kChains: an operation is up to four chains over consecutive lines.
template <int KS, bool kChains = false>
__device__ __forceinline__ bool issue_ops(const Waiter &w, const IssueCtx &ic, const PrevConv &prev, uint32_t n_ksteps)
{
    constexpr int NK = KS > 0 ? KS : 1;
    uint32_t alo[NK], blo[NK];
    const uint32_t ahi = (uint32_t)(make_desc(0, 0, 128) >> 32), bhi = (uint32_t)(make_desc(0, 128, 256) >> 32);
    if (KS > 0) {
#pragma unroll
        for (int k4 = 0; k4 < NK; k4 += 4) {
            const uint4 v = ld_shared_v4(ic.desc + offsetof(LConvDesc, a_lo) + 4 * k4);
            const uint32_t vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (k4 + q < NK) alo[k4 + q] = vv[q] + ic.s16;
        }
#pragma unroll
        for (int k = 0; k < NK; ++k) blo[k] = ic.b_lo0 + ic.s16 + (uint32_t)k * ic.kstep16;
    }
    uint32_t at = ic.ops + 32u * ic.issuer;           // the table ends with kIssuers spare records: reads run one ahead
    uint4 n0 = ld_shared_v4(at), n1 = ld_shared_v4(at + 16);
    for (uint32_t i = ic.issuer; i < ic.n_ops; i += kIssuers) {
        const uint4 r0 = n0, r1 = n1;         // d_col, idesc, a_add, b_add | wait 0-1, wait 2-3, commit 0-1, commit 2 and flags
        at += 32u * kIssuers;
        n0 = ld_shared_v4(at); n1 = ld_shared_v4(at + 16);
        if (!op_wait(w, prev, r1)) return false;
        const uint32_t d = ic.d0 + r0.x;
        if (!(r1.w & (7u << 26))) {
            // a record that only carries this thread's arrivals on units it did not add to
        } else if (kChains) {
            const uint32_t n_chains = (r1.w >> 26) & 7u;
            for (uint32_t c = 0; c < n_chains; ++c) {
#pragma unroll
                for (int k = 0; k < NK; ++k)
                    mma_i8(d + c * ic.cols, ((uint64_t)ahi << 32) | (uint64_t)(alo[k] + r0.z + c * ic.pitch16), ((uint64_t)bhi << 32) | (uint64_t)(blo[k] + r0.w), r0.y);
            }
        } else if (KS > 0) {
#pragma unroll
            for (int k = 0; k < NK; ++k)
                mma_i8(d, ((uint64_t)ahi << 32) | (uint64_t)(alo[k] + r0.z), ((uint64_t)bhi << 32) | (uint64_t)(blo[k] + r0.w), r0.y);
        } else {
            for (uint32_t k = 0; k < n_ksteps; ++k) {
                const uint32_t a_lo = lds32(ic.desc + offsetof(LConvDesc, a_lo) + 4 * k) + ic.s16;
                mma_i8(d, ((uint64_t)ahi << 32) | (uint64_t)(a_lo + r0.z), ((uint64_t)bhi << 32) | (uint64_t)(ic.b_lo0 + ic.s16 + k * ic.kstep16 + r0.w), r0.y);
            }
        }
        op_commit(ic, r1);
    }
    return true;
}

// The same for paired convolutions (see build_plan): three MMAs for two lines.
__device__ __forceinline__ bool issue_pairs(const Waiter &w, const IssueCtx &ic, const PrevConv &prev)
{
    const uint32_t ahi = (uint32_t)(make_desc(0, 0, 128) >> 32), bhi = (uint32_t)(make_desc(0, 128, 256) >> 32);
    const uint4 v = ld_shared_v4(ic.desc + offsetof(LConvDesc, a_lo));
    const uint32_t alo[3] = {v.x + ic.s16, v.y + ic.s16, v.z + ic.s16}, c2 = 2u * ic.cols;
    const uint32_t blo[3] = {ic.b_lo0 + ic.s16, ic.b_lo0 + ic.s16 + 3u * c2, ic.b_lo0 + ic.s16 + 7u * c2};
    const uint32_t n1_bits = ic.cols >> 3 << 17;                        // N of one block in the instruction descriptor
    uint32_t at = ic.ops + 32u * ic.issuer;
    uint4 n0 = ld_shared_v4(at), n1 = ld_shared_v4(at + 16);
    for (uint32_t i = ic.issuer; i < ic.n_ops; i += kIssuers) {
        const uint4 r0 = n0, r1 = n1;
        at += 32u * kIssuers;
        n0 = ld_shared_v4(at); n1 = ld_shared_v4(at + 16);
        if (!op_wait(w, prev, r1)) return false;
        uint32_t d = ic.d0 + r0.x, a_add = r0.z;
        const uint32_t n_pairs = (r1.w >> 26) & 7u;
        if (r0.w == kPairInner) {
            for (uint32_t q = 0; q < n_pairs; ++q) {
                mma_i8(d, ((uint64_t)ahi << 32) | (uint64_t)(alo[0] + a_add), ((uint64_t)bhi << 32) | (uint64_t)blo[0], r0.y + 3u * n1_bits);
                mma_i8(d, ((uint64_t)ahi << 32) | (uint64_t)(alo[1] + a_add), ((uint64_t)bhi << 32) | (uint64_t)blo[1], r0.y + 4u * n1_bits);
                mma_i8(d + ic.cols, ((uint64_t)ahi << 32) | (uint64_t)(alo[2] + a_add), ((uint64_t)bhi << 32) | (uint64_t)blo[2], r0.y + 3u * n1_bits);
                d += c2;
                a_add += 2u * ic.pitch16;
            }
        } else if (n_pairs) {
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const uint32_t f = r0.w >> (7 * k);
                mma_i8(d + ((f >> 5) & 3u) * ic.cols, ((uint64_t)ahi << 32) | (uint64_t)(alo[k] + a_add), ((uint64_t)bhi << 32) | (uint64_t)(blo[k] + ((f >> 3) & 3u) * c2),
                       r0.y + (f & 7u) * n1_bits);
            }
        }
        op_commit(ic, r1);
    }
    return true;
}

__device__ __forceinline__ void issue_weights(const ConvSrc *src, uint32_t sbase, uint32_t wbar_addr)
{
    const uint4 v = *reinterpret_cast<const uint4 *>(src);
    const void *gmem = reinterpret_cast<const void *>(((unsigned long long)v.y << 32) | v.x);
    const uint32_t bytes = v.z & 0xFFFFFFu;
    mbar_expect_tx(wbar_addr, bytes);
    bulk_g2s(sbase + (v.w & 0x7FFFFFFFu), gmem, bytes, wbar_addr);
}

// The copy of convolution `target`'s blob, by lane 0 of the loader warp, once the convolution it names is complete:
// the blob takes the place of things that convolution (or an earlier one) was the last to use.
__device__ __forceinline__ bool loader_copy(const LineParams &p, int target, uint32_t wslot, int it)
{
    const Waiter w{p.err};
    const ConvSrc *src = the_ctrl()->csrc + target;
    if ((int)(src->bytes_phase >> 24) > p.stop_phase) return true;
    const uint32_t n = src->dep_units;
    if (n) {
        const uint32_t expected = src->dep_mult * ((uint32_t)it * (src->dep_local_uses >> 16) + (src->dep_local_uses & 0xFFFFu) + 1u);
        const uint32_t first = CTRL_ADDR(stored) + 4u * src->dep_first;
        for (uint32_t l = 0; l < n; ++l)
            if (!w.counter(first + 4 * l, expected, ERR_WAIT_DONE)) return false;
    }
    issue_weights(src, the_base(), CTRL_ADDR(wbar) + 8u * wslot);
    return true;
}

// One convolution's share of an issuing warp, by its lane 0.  Returns false after a wait has expired.
template <bool kRare>
__device__ __forceinline__ bool issuer_conv(const LineParams &p, uint32_t tmem, uint32_t blob_off, WeightSlot ws, uint32_t issuer, int it, PrevConv &prev)
{
    const Waiter w{p.err};
    if (!w.barrier(CTRL_ADDR(wbar) + 8u * ws.slot, ws.parity, ERR_WAIT_WEIGHTS)) return false;
    const uint32_t desc = the_base() + blob_off;
    const uint4 h0 = ld_shared_v4(desc);                                    // flags, n_items, recs_per_item, d_base
    const uint4 h1 = ld_shared_v4(desc + offsetof(LConvDesc, bar_full));    // bar_full, bar_done, use_local, uses_per_group
    const uint4 h2 = ld_shared_v4(desc + offsetof(LConvDesc, n_ops));       // n_ops, n_ksteps, ops_rel, n_chunks
    const uint4 h3 = ld_shared_v4(desc + offsetof(LConvDesc, b_lo0));       // b_lo0, kstep16, pitch16, cols
    const uint32_t n_units = lds32(desc + offsetof(LConvDesc, n_units));
    const uint32_t use = (uint32_t)it * h1.w + h1.z;
    IssueCtx ic;
    ic.desc = desc; ic.ops = desc + h2.z; ic.n_ops = h2.x;
    ic.s16 = the_base() >> 4; ic.b_lo0 = h3.x; ic.kstep16 = h3.y;
    ic.d0 = tmem + h0.w;
    ic.full_addr = CTRL_ADDR(bars) + 8u * (h1.x + (use & 1u) * n_units);      // the class has two sets of barriers, used in turn
    ic.issuer = issuer;
    ic.pitch16 = h3.z;
    ic.cols = h3.w;
    bool ok;
    if (h0.x & CF_PAIRED) ok = issue_pairs(w, ic, prev);
    else if (kRare && h2.y == 2u) ok = issue_ops<2, true>(w, ic, prev, 2);
    else switch (h2.y) {
    case 1: ok = issue_ops<1>(w, ic, prev, 1); break;
    case 3: ok = issue_ops<3>(w, ic, prev, 3); break;
    case 5: ok = issue_ops<5>(w, ic, prev, 5); break;
    case 6: ok = issue_ops<6>(w, ic, prev, 6); break;
    case 9: ok = issue_ops<9>(w, ic, prev, 9); break;
    default: ok = issue_ops<0>(w, ic, prev, h2.y); break;
    }
    if (!ok) return false;
    prev.done_addr = CTRL_ADDR(stored) + 4u * h1.y;
    prev.expected = 4u * h2.w * (use + 1u);
    prev.n_lines = n_units;
    return true;
}

// ------------------------------------------------------------------ epilogue warps

// A thread works on four positions of a line (rows quarter * 32 + lane / 4 + 8 i) and the four channels 4 c .. 4 c + 3 of a chunk
// (c = lane mod 4), one word: constants stay in registers for a whole convolution, and eight positions x 16 bytes make one
// conflict-free store.  (The columns of the weights are ordered so that a thread's accumulator columns are these channels.)
// One record of the pass table: one or two lines of a unit and a chunk.
struct alignas(16) LPass {
    // unit | lines << 8 | chunk << 12 | line 0 first / last row of its band << 16, 17 | line 1 << 18, 19 | start values of line 0, 1 << 20, 26:
    // the accumulators read take the folded biases of the channels that the next convolution on these columns puts there
    uint32_t meta;
    uint32_t lines;         // line 0 | line 1 << 8
    uint32_t tcol[2];       // accumulator columns of the two lines' chunk within the bank
    uint32_t out[2];        // byte offset of the two lines' chunk (line within its plane + plane) in the output
    uint32_t res[2];        // the same in the residual operand
};
static_assert(sizeof(LPass) == 32, "one pass is two 16-byte loads");

// Four outputs of one position.
//   kRes = 1: y += floor((u * m2 + r2) / 2^32), the residual term of the general form.
//   kRes = 2: y += round((256 k + u) * m) - c_r with u = r + 128 the residual byte as an unsigned number, for an offset k
//   and a multiplier m that the planner has checked on all 256 values of u (residual_form): rs((r - zp_res) * res_mult, n).
//   `k8` holds 256 k, which the byte permute that extracts u merges into it; c_r is folded into the rounding addends.
template <int kRes>
__device__ __forceinline__ uint32_t requant4(int a0, int a1, int a2, int a3, const ChanConsts &k, uint32_t rword, uint32_t m2, uint32_t k8, long long r2)
{
    int y0 = mad_hi(a0, k.mult[0], k.c[0]) >> k.s[0], y1 = mad_hi(a1, k.mult[1], k.c[1]) >> k.s[1];
    int y2 = mad_hi(a2, k.mult[2], k.c[2]) >> k.s[2], y3 = mad_hi(a3, k.mult[3], k.c[3]) >> k.s[3];
    if (kRes == 1) {
        y0 += hi32(mad_wide_u(__byte_perm(rword, 0u, 0x4440u), m2, r2));
        y1 += hi32(mad_wide_u(__byte_perm(rword, 0u, 0x4441u), m2, r2));
        y2 += hi32(mad_wide_u(__byte_perm(rword, 0u, 0x4442u), m2, r2));
        y3 += hi32(mad_wide_u(__byte_perm(rword, 0u, 0x4443u), m2, r2));
    }
    if (kRes == 2) {
        y0 += mul_denormal(__byte_perm(rword, k8, 0x7650u), m2);
        y1 += mul_denormal(__byte_perm(rword, k8, 0x7651u), m2);
        y2 += mul_denormal(__byte_perm(rword, k8, 0x7652u), m2);
        y3 += mul_denormal(__byte_perm(rword, k8, 0x7653u), m2);
    }
    return pack4_sat(y0, y1, y2, y3);
}

__device__ __forceinline__ void st_shared_u32(uint32_t addr, uint32_t v) { asm volatile("st.shared.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory"); }
__device__ __forceinline__ void st_shared_u32_if(uint32_t addr, uint32_t v, uint32_t flag)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p st.shared.u32 [%0], %1;\n\t}" ::"r"(addr), "r"(v), "r"(flag) : "memory");
}

// After an item: the stores become visible to the tensor cores' reads, the tensor-memory accesses are ordered
// before the arrival, and the warp counts one stored chunk of the unit.
__device__ __forceinline__ void pass_done(uint32_t counter, int lane)
{
    tmem_st_wait();
    tc_fence_before();
    fence_proxy_async();
    __syncwarp();
    if (lane == 0) red_release_add(counter, 1u);
}

// Stride 2: where position `pos` of even input line number `line` goes (even columns survive, and every row of an even line
// is an even row), relative to the output's line 0, lane 0, plane 0, with its line and band.
struct Scatter { uint32_t log_i, half_lines, log_lines, log_o, pitch; };
__device__ __forceinline__ uint32_t scatter_to(const Scatter &g, uint32_t pos, uint32_t line, uint32_t &oline, uint32_t &oband)
{
    const uint32_t x = pos >> g.log_i, band = (pos & ((1u << g.log_i) - 1u)) >> 2, row = line + band * g.half_lines;
    oline = row & ((1u << g.log_lines) - 1u);
    oband = row >> g.log_lines;
    return (oline * g.pitch + ((x >> 1) << g.log_o) + (oband << 2) + (pos & 3u)) * 16u;
}

// The items (unit, chunk) of a convolution that belong to this warp's set: one wait, one or two records of two lines each,
// one arrival.  kScatter: stride 2, results go to the next geometry (2.1 instead of 4.0 us a convolution of the first
// transition when that was a pass of run-time decisions, line by line).
template <int kRes, bool kScatter>
__device__ __forceinline__ bool epi_conv_fast(Waiter w, uint32_t tmem_lane, uint32_t warp, uint32_t lane, uint32_t desc, uint4 h0, uint4 h1, uint4 h2, uint4 h3, uint32_t use)
{
    const uint32_t tmem0 = tmem_lane + h0.w, full = CTRL_ADDR(bars) + 8u * (h1.x + (use & 1u) * h2.x), done = CTRL_ADDR(stored) + 4u * h1.y;
    const uint32_t parity = (use >> 1) & 1u, word = lane & 3u, row0 = (warp & 3u) * 32u + (lane >> 2);
    const uint32_t out = the_base() + h2.w + (kScatter ? word * 4u : row0 * 16u + word * 4u), res = the_base() + h3.x + row0 * 16u + word * 4u;
    const uint32_t vecs = desc + lds32(desc + offsetof(LConvDesc, vec_rel));
    const uint32_t m2 = h3.y, k8 = h3.z, dup = h3.w;
    const long long r2 = kRes == 1 ? (long long)(((unsigned long long)lds32(desc + offsetof(LConvDesc, res_r2_hi)) << 32) | k8) : 0ll;
    // The bands of a thread's rows: they differ in bits 3 and 4 of the position, of which a band number has bits 2 and 3 at
    // most.  Bit 0, 1: rows of even number have a band above, below; bit 2, 3: those of odd number.
    const uint32_t nb = lds32(desc + offsetof(LConvDesc, out_nb));
    uint32_t bands = 0;
    // Stride 2 (see scatter_to): the rows of a thread are in one band, and steps of 8 positions go on by whole columns, so
    // that the output line is worked out once per input line.
    uint32_t sc_row = 0, sc_at = 0, sc_pitch = 0, sc_log = 0, sc_odd = 0;
    if (kScatter) {
        const uint4 g0 = ld_shared_v4(desc + offsetof(LConvDesc, out_plane)), g1 = ld_shared_v4(desc + offsetof(LConvDesc, in_logI));
        const uint32_t log_i = g1.x, log_o = g0.w;
        sc_pitch = g0.y;
        sc_log = g0.z | log_i << 8 | log_o << 16;
        sc_row = ((row0 & ((1u << log_i) - 1u)) >> 2) * (g1.y >> 1);
        sc_at = (row0 >> (log_i + 1u) << log_o) + (row0 & 3u);
        sc_odd = ((row0 >> log_i) & 1u) | (((row0 + 8u) >> log_i) & 1u) << 1;         // bit j: position row0 + 8 j (+ 16) is in an odd column
    }
    if (!kScatter) {
        const uint32_t a = (row0 >> 2) & (nb - 1u), b = ((row0 >> 2) + 2u) & (nb - 1u);
        bands = (a >= 1u ? 1u : 0u) | (a + 1u < nb ? 2u : 0u) | (b >= 1u ? 4u : 0u) | (b + 1u < nb ? 8u : 0u);
    }
    const uint32_t consts = desc + h2.y + word * 48u, rec_bytes = 32u * h0.z, rec_stop = desc + h2.z + rec_bytes * h0.y;
#pragma unroll 1
    for (uint32_t rec = desc + h2.z + rec_bytes * (warp >> 2); rec < rec_stop; rec += rec_bytes * (kSets - 1)) {
        const uint32_t rec_end = rec + rec_bytes;
        uint4 q0 = ld_shared_v4(rec), q1 = ld_shared_v4(rec + 16u);
        const uint32_t unit = q0.x & 0xFFu;
        const ChanConsts k = ld_chan_consts(consts + ((q0.x >> 12) & 0xFu) * kChunkConstBytes);
        const bool ok = w.barrier(full + 8u * unit, parity, ERR_WAIT_FULL);
        if (!__all_sync(0xffffffffu, ok)) return false;                 // aborted: every other wait falls through too
        tc_fence_after();
#pragma unroll 1
        for (;;) {
            // Four steps: two lines x two halves of 16 positions; the next step's accumulators are requested before this
            // step's arithmetic.  (All 32 accumulators at once left no registers for the addresses.)
            int acc[2][8];
            tmem_ld_frag(tmem0 + q0.z, acc[0]);
#pragma unroll
            for (int st = 0; st < 4; ++st) {
                const int l = st >> 1, h = st & 1;
                int (&v)[8] = acc[st & 1];
                const uint32_t to = out + (l ? q1.y : q1.x);
                const uint32_t from = res + (l ? q1.w : q1.z) + (uint32_t)h * 256u;
                uint32_t r0 = 0, r1 = 0;
                if (kRes) { r0 = lds32(from) ^ 0x80808080u; r1 = lds32(from + 128u) ^ 0x80808080u; }
                tmem_ld_frag_wait(v);
                if (st < 3) tmem_ld_frag(tmem0 + (st == 0 ? q0.z + (16u << 16) : st == 1 ? q0.w : q0.w + (16u << 16)), acc[(st + 1) & 1]);
                if (h == 1) tmem_st_columns(tmem0 + (l ? q0.w : q0.z), vecs + (l ? q0.x >> 26 : (q0.x >> 20) & 63u) * kVecBytes);
                if (kScatter) {
                    // q1 holds the chunk's plane here, not a line's offset
                    const uint32_t lines = 1u << (sc_log & 0xFFu), row = ((q0.y >> (8 * l)) & 0xFFu) + sc_row, oline = row & (lines - 1u), oband = row >> (sc_log & 0xFFu);
                    const uint32_t up = oline == 0u && oband >= 1u, dn = oline + 1u == lines && oband + 1u < nb;
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        if ((sc_odd >> j) & 1u) continue;
                        const uint32_t o = requant4<0>(v[2 * j], v[2 * j + 1], v[2 * j + 4], v[2 * j + 5], k, 0u, 0u, 0u, 0ll);
                        const uint32_t col = (uint32_t)(16 * h + 8 * j) >> (((sc_log >> 8) & 0xFFu) + 1u) << (sc_log >> 16);
                        const uint32_t at = to + (oline * sc_pitch + sc_at + col + (oband << 2)) * 16u;
                        st_shared_u32(at, o);
                        if (dup) {
                            st_shared_u32_if(at + dup, o, up);
                            st_shared_u32_if(at - dup, o, dn);
                        }
                    }
                } else {
                    const uint32_t o0 = requant4<kRes>(v[0], v[1], v[4], v[5], k, r0, m2, k8, r2), at = to + (uint32_t)h * 256u;
                    st_shared_u32(at, o0);
                    const uint32_t o1 = requant4<kRes>(v[2], v[3], v[6], v[7], k, r1, m2, k8, r2);
                    st_shared_u32(at + 128u, o1);
                    const uint32_t edges = (q0.x >> (16 + 2 * l)) & 3u;
                    if (dup && edges) {
                        // first row of a lower band: also the row below the band above it; last row of an upper band: the
                        // row above the next band
                        const uint32_t e = bands & (edges | edges << 2);
                        st_shared_u32_if(at + dup, o0, e & 1u);
                        st_shared_u32_if(at - dup, o0, e & 2u);
                        st_shared_u32_if(at + 128u + dup, o1, e & 4u);
                        st_shared_u32_if(at + 128u - dup, o1, e & 8u);
                    }
                }
            }
            rec += 32u;
            if (rec == rec_end) break;
            q0 = ld_shared_v4(rec);
            q1 = ld_shared_v4(rec + 16u);
        }
        pass_done(done + 4u * unit, (int)lane);
    }
    return true;
}

// The general pass: a lower clamp above -128, a shift of one, a lone line; one line at a time, every property decided at
// run time.
__device__ __forceinline__ bool epi_conv_general(Waiter w, uint32_t tmem_lane, uint32_t warp, uint32_t lane, uint32_t desc, uint4 h0, uint4 h1, uint4 h2, uint4 h3, uint32_t use)
{
    const bool res = h0.x & CF_RES, scatter = h0.x & CF_SCATTER;
    const uint32_t tmem0 = tmem_lane + h0.w, full = CTRL_ADDR(bars) + 8u * (h1.x + (use & 1u) * h2.x), done = CTRL_ADDR(stored) + 4u * h1.y;
    const uint32_t parity = (use >> 1) & 1u, word = lane & 3u, row0 = (warp & 3u) * 32u + (lane >> 2), dup = h3.w;
    const uint4 g0 = ld_shared_v4(desc + offsetof(LConvDesc, out_plane)), g1 = ld_shared_v4(desc + offsetof(LConvDesc, in_logI));
    const uint4 gl = ld_shared_v4(desc + offsetof(LConvDesc, lo));
    const int lo = (int)gl.x;
    const long long r2 = (long long)(((unsigned long long)gl.z << 32) | gl.y);
    const uint32_t nb = g1.z, vecs = desc + g1.w;
    const Scatter g{g1.x, g1.y >> 1, g0.z, g0.w, g0.y};
#pragma unroll 1
    for (uint32_t i = warp >> 2; i < h0.y; i += kSets) {
        const uint32_t rec = desc + h2.z + 32u * i;                   // one record per item
        const uint4 q0 = ld_shared_v4(rec), q1 = ld_shared_v4(rec + 16u);
        const uint32_t unit = q0.x & 0xFFu, n = (q0.x >> 8) & 0xFu;
        const ChanConsts k = ld_chan_consts(desc + h2.y + word * 48u + ((q0.x >> 12) & 0xFu) * kChunkConstBytes);
        const bool ok = w.barrier(full + 8u * unit, parity, ERR_WAIT_FULL);
        if (!__all_sync(0xffffffffu, ok)) return false;
        tc_fence_after();
#pragma unroll 1
        for (uint32_t l = 0; l < n; ++l) {
            const uint32_t tcol = l ? q0.w : q0.z, to = the_base() + h2.w + word * 4u + (l ? q1.y : q1.x), line = (q0.y >> (8u * l)) & 0xFFu;
            const uint32_t from = the_base() + h3.x + word * 4u + (l ? q1.w : q1.z), edges = q0.x >> (16u + 2u * l);
#pragma unroll 1
            for (uint32_t h = 0; h < 2; ++h) {
                int a[8];
                tmem_ld_frag(tmem0 + tcol + (h * 16u << 16), a);
                tmem_ld_frag_wait(a);
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const uint32_t pos = row0 + 16u * h + 8u * (uint32_t)j;
                    const uint32_t rword = res ? lds32(from + pos * 16u) ^ 0x80808080u : 0u;
                    int y[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const long long prod = mul_wide(a[2 * j + (q & 1) + 4 * (q >> 1)], k.mult[q]);
                        int v = k.s[q] ? (hi32(prod) + k.c[q]) >> k.s[q] : hi32(prod) + (int)((uint32_t)lo32(prod) >> 31) + k.c[q];
                        if (res) v += hi32(mad_wide_u((rword >> (8 * q)) & 0xFFu, gl.w, r2));
                        y[q] = max(v, lo);
                    }
                    const uint32_t o = pack4_sat(y[0], y[1], y[2], y[3]);
                    uint32_t at = to + pos * 16u, up, dn;
                    if (scatter) {
                        if ((pos >> g.log_i) & 1u) continue;
                        uint32_t oline, oband;
                        at = to + scatter_to(g, pos, line, oline, oband);
                        up = oline == 0u && oband >= 1u;
                        dn = oline + 1u == (1u << g.log_lines) && oband + 1u < nb;
                    } else {
                        const uint32_t band = (pos >> 2) & (nb - 1u);
                        up = (edges & 1u) && band >= 1u;
                        dn = (edges & 2u) && band + 1u < nb;
                    }
                    st_shared_u32(at, o);
                    if (dup) {
                        st_shared_u32_if(at + dup, o, up);
                        st_shared_u32_if(at - dup, o, dn);
                    }
                }
            }
            tmem_st_columns(tmem0 + tcol, vecs + ((q0.x >> (20u + 6u * l)) & 63u) * kVecBytes);
        }
        pass_done(done + 4u * unit, (int)lane);
    }
    return true;
}

// FILL: the region takes its halo value everywhere
__device__ __forceinline__ void fill_phase(uint32_t off, uint32_t bytes, uint32_t halo)
{
    const uint32_t word = (halo & 0xFFu) * 0x01010101u;
    const uint4 v = make_uint4(word, word, word, word);
    for (uint32_t o = threadIdx.x * 16u; o < bytes; o += kThreads * 16u) st_shared_v4(the_base() + off + o, v);
}

// Which samples a group holds: image, phase, and the range of sample numbers.
struct GroupJob {
    int image, local, n;              // local: index of the group's first sample within the image's phase; n: samples of that phase
    bool sel;
};
__device__ __forceinline__ GroupJob group_job(const LineParams &p, int grp)
{
    GroupJob g;
    const int per_image = p.groups_sel + p.groups_est;
    g.image = grp / per_image;
    const int r = grp - g.image * per_image;
    g.sel = r < p.groups_sel;
    g.local = kG * (g.sel ? r : r - p.groups_sel);
    g.n = g.sel ? p.n_sel : p.n_est;
    return g;
}

// INPUT: one item = four horizontally adjacent pixels of one sample and input channel, one Philox block (Def. 3.3,
// Def. 3.4).  Items of all channels share one index space (3072 items of a 32 x 32 x 3 image for 640 threads; with the
// channels of a pixel in one thread it was 1024, two rounds of which the second is mostly idle).  The levels come from the
// table of bins in global memory: one load that depends on the uniforms instead of the guide's and then one for each step of
// a bisection, which a CTA with nearly no L1 beside its shared memory waits for at L2's latency (a group of the 20-layer
// network 92.5 -> 89.3 us, the call of the tiny CNN 94 -> 84 us).
__device__ __forceinline__ void input_phase(const LineParams &p, int grp)
{
    const int H = p.in_H, W = p.in_W, in_c = p.in_c;
    const int log_wq = 31 - __clz(W >> 2);                  // W is a power of two
    const int quads = kG * H * (W >> 2);
    const uint32_t *__restrict__ cum = p.ns.cum;
    const uint32_t *__restrict__ guide = p.ns.guide;
    const uint2 *__restrict__ bins = p.ns.bins;
    const int T = p.ns.T, steps = p.ns.guide_steps;
    const GroupJob g = group_job(p, grp);
    const unsigned long long image_id = p.image_id0 + (unsigned long long)g.image;
    const uint32_t key0 = p.ns.key0, key1 = p.ns.key1, ctr2 = (uint32_t)image_id;
    const uint32_t ctr3_fixed = (g.sel ? (uint32_t)p.phase_sel : p.ns.ctr3_fixed) | ((uint32_t)(image_id >> 32) & 0xFFFFu) << 16;
    const long long j0 = (g.sel ? 0ll : p.ns.first_sample) + g.local;
    const uint8_t *__restrict__ x = p.x + (size_t)g.image * (size_t)(in_c * H * W);
    int ch = 0;
    for (int i = (int)threadIdx.x, qi = i; i < quads * in_c; i += kThreads, qi += kThreads) {
        while (qi >= quads) { qi -= quads; ++ch; }
        // consecutive threads take consecutive samples: their stores fall into one 64-byte run
        const int s = qi & (kG - 1);
        const int rem = qi >> 2;
        const int y = rem >> log_wq, x4 = rem & ((1 << log_wq) - 1);
        const long long j = j0 + s;
        const uint32_t ctr3 = ctr3_fixed | (uint32_t)(((j >> 32) & 0xFF) << 8);
        const uint32_t e = (uint32_t)((ch * H + y) * W + 4 * x4);
        const uint4 r = philox4x32_10(make_uint4(e >> 2, (uint32_t)(j & 0xFFFFFFFFll), ctr2, ctr3), key0, key1);
        const uint32_t clean = __ldg(reinterpret_cast<const uint32_t *>(x + e));
        int z[4];
        if (bins && noise_levels4_bins(r, 0u, bins, p.ns.bin_bits, z)) {
        } else if (guide) {
            noise_levels4(r, cum, guide, T, steps, z);
        } else {
            const uint32_t u[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) z[k] = noise_level(u[k], cum, T);
        }
        // the input has one row band: line = row, position = column * 4 + sample; the bytes beyond the input channels
        // meet zero weights
        const uint32_t at = the_base() + p.input_base + ((uint32_t)y * p.input_pitch16 + (uint32_t)(4 * x4) * kG + (uint32_t)s) * 16u + (uint32_t)ch;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int v = min(255, max(0, (int)((clean >> (8 * k)) & 0xFFu) + z[k]));
            asm volatile("st.shared.u8 [%0], %1;" ::"r"(at + (uint32_t)k * (kG * 16u)), "r"(v) : "memory");
        }
    }
}

// TAIL: global average pool, FC, argmax and vote (Algorithm 1 steps 1-4), in three steps between barriers.
// First step: a thread adds up four channels (one word) of one sample over a share of the pixels; consecutive threads take
// the words of the four samples of a position (64 contiguous bytes), the shares meet in shared-memory additions.  (One
// thread per channel and sample left most of the CTA idle over 64 to 1024 pixels: with the noise phase before it, a
// network that ends at a 32 x 32 map spent 43 us a group more, the tiny CNN 15 us a call.)
__device__ __forceinline__ void tail_sum(const LineParams &p)
{
    const int units = p.tail_C, parts = kThreads / units, part = (int)threadIdx.x / units, u = (int)threadIdx.x - part * units;       // a unit is (word, sample)
    if (part >= parts) return;
    const int word = u >> 2, s = u & (kG - 1);
    const int log_w = 31 - __clz(p.tail_W), log_n = 31 - __clz(p.tail_n_lines);                                  // powers of two
    const uint32_t base = the_base() + p.tail_base + (uint32_t)(word >> 2) * p.tail_plane + (uint32_t)(word & 3) * 4u + (uint32_t)s * 16u;
    int sum[4] = {0, 0, 0, 0}, n = 0;
    for (int i = part; i < p.tail_H * p.tail_W; i += parts, ++n) {
        const int y = i >> log_w, x = i & (p.tail_W - 1);
        const int line = y & (p.tail_n_lines - 1), band = y >> log_n;
        const uint32_t pos = (uint32_t)line * p.tail_pitch16 + ((uint32_t)x << p.tail_logI) + (uint32_t)(band * 4);
        const int v = (int)lds32(base + pos * 16u);
        sum[0] = __dp4a(v, 1, sum[0]);
        sum[1] = __dp4a(v, 1 << 8, sum[1]);
        sum[2] = __dp4a(v, 1 << 16, sum[2]);
        sum[3] = __dp4a(v, 1 << 24, sum[3]);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) atomicAdd(&the_ctrl()->pool_sum[s][4 * word + k], sum[k] - n * p.pool_zp_in);
}

// Second step: the sums' requantisation.
__device__ __forceinline__ void tail_pool(const LineParams &p)
{
    for (int q = (int)threadIdx.x; q < kG * p.tail_C; q += kThreads) {
        const int s = q & (kG - 1), ch = q >> 2;
        const int sum = the_ctrl()->pool_sum[s][ch];
        the_ctrl()->pool_sum[s][ch] = 0;
        long long v = ((long long)sum * p.pool_mult + (1ll << (p.pool_n - 1))) >> p.pool_n;
        v += p.pool_zp_out;
        v = v < p.pool_lo ? p.pool_lo : v;
        v = v > 127 ? 127 : v;
        the_ctrl()->pooled[s][ch] = (int8_t)v;
    }
}

// Third step: FC, argmax and vote; one warp carries one sample, a lane one class (features beyond the last meet zero weights).
__device__ __forceinline__ void tail_sample(const LineParams &p, int s, int grp)
{
    const int lane = (int)threadIdx.x & 31;
    const int n_classes = p.n_classes;
    const GroupJob g = group_job(p, grp);
    const int sample = g.local + s;                            // index within the image's phase
    const bool counted = sample < g.n;
    int best_v = -1000, best_o = 0x7fffffff;
    uint4 f[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) f[k] = ld_shared_v4(CTRL_ADDR(pooled) + (uint32_t)(64 * s + 16 * k));
    for (int o0 = 0; o0 < n_classes; o0 += 32) {
        const int o = o0 + lane;
        const bool live = o < n_classes;
        const FcConst k = p.fc_c[live ? o : 0];
        const uint4 *wrow = reinterpret_cast<const uint4 *>(p.fc_w + (size_t)(live ? o : 0) * 64);
        int acc = k.bias;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint4 w = __ldg(wrow + q);
            acc = __dp4a((int)f[q].x, (int)w.x, acc);
            acc = __dp4a((int)f[q].y, (int)w.y, acc);
            acc = __dp4a((int)f[q].z, (int)w.z, acc);
            acc = __dp4a((int)f[q].w, (int)w.w, acc);
        }
        long long v = ((long long)acc * k.mult + (1ll << (k.n - 1))) >> k.n;
        v += k.zp_out;
        v = v < k.lo ? k.lo : v;
        v = v > 127 ? 127 : v;
        if (live) {
            if ((int)v > best_v) { best_v = (int)v; best_o = o; }
            if (counted && p.logits) p.logits[(long long)sample * n_classes + o] = (int8_t)v;
        }
    }
    // lowest index among the maxima
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) {
        const int ov = __shfl_xor_sync(0xffffffffu, best_v, d), oo = __shfl_xor_sync(0xffffffffu, best_o, d);
        if (ov > best_v || (ov == best_v && oo < best_o)) { best_v = ov; best_o = oo; }
    }
    if (counted && lane == 0) {
        const int row = p.groups_sel ? 2 * g.image + (g.sel ? 0 : 1) : g.image;
        atomicAdd(p.counts + (size_t)row * n_classes + best_o, 1);
    }
}

// A phase of the whole CTA: everything before it is complete in all warps, and it is before anything after it.  Nothing inside
// can raise the abort flag, so that all warps skip it or none.  Thread 0 keeps the time (phases run between barriers, so one
// thread's clock measures them).
__device__ __forceinline__ void cta_phase(const LineParams &p, uint4 e, int grp)
{
    Ctrl *ctrl = the_ctrl();
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const bool live = !Waiter::aborted();
    if (threadIdx.x == 0) ctrl->cyc_mark = clock64();
    if (live) {
        if (e.x == PH_FILL) fill_phase(e.y, e.z, e.w);
        else if (e.x == PH_INPUT) input_phase(p, grp);
        else tail_sum(p);
    }
    if (e.x == PH_TAIL) {
        __syncthreads();
        if (live) tail_pool(p);
        __syncthreads();
        if (live && threadIdx.x < 32 * kG) tail_sample(p, (int)(threadIdx.x >> 5), grp);
    }
    fence_proxy_async();
    __syncthreads();
    if (threadIdx.x == 0) ctrl->cyc[e.x & 3u] += clock64() - ctrl->cyc_mark;
}

// The roles' shares of the convolutions from phase `ph` on, up to the next phase of the whole CTA.  After the abort flag is
// up a role skips its convolutions and goes on through the phases.
struct RoleState {
    WeightSlot ws;              // of the next convolution (loader: of the next copy)
    bool ok = true;
    PrevConv prev{0u, 0u, 0u};
    int next_copy = 0;
};

template <bool kRare>
__device__ __forceinline__ void epilogue_run(const LineParams &p, uint32_t tmem, uint32_t warp, uint32_t lane, int ph, int stop, int it, RoleState &r)
{
    const Waiter w{p.err};
    const uint32_t tmem_lane = tmem + ((warp & 3u) * 32u << 16);
    for (; ph < stop; ++ph) {
        if (r.ok) r.ok = __all_sync(0xffffffffu, w.barrier(CTRL_ADDR(wbar) + 8u * r.ws.slot, r.ws.parity, ERR_WAIT_WEIGHTS));
        r.ws.advance();
        if (!r.ok) continue;
        const uint32_t desc = the_base() + lds32(CTRL_ADDR(ptab) + 16u * (uint32_t)ph + 4u);
        const uint4 h0 = ld_shared_v4(desc), h1 = ld_shared_v4(desc + 16u), h2 = ld_shared_v4(desc + 32u), h3 = ld_shared_v4(desc + 48u);
        const uint32_t use = (uint32_t)it * h1.w + h1.z;
        if (h0.x & CF_GENERAL) r.ok = epi_conv_general(w, tmem_lane, warp, lane, desc, h0, h1, h2, h3, use);
        else if (h0.x & CF_SCATTER) r.ok = epi_conv_fast<0, true>(w, tmem_lane, warp, lane, desc, h0, h1, h2, h3, use);
        else if (kRare && (h0.x & CF_RES_LONG)) r.ok = epi_conv_fast<1, false>(w, tmem_lane, warp, lane, desc, h0, h1, h2, h3, use);
        else if (h0.x & CF_RES) r.ok = epi_conv_fast<2, false>(w, tmem_lane, warp, lane, desc, h0, h1, h2, h3, use);
        else r.ok = epi_conv_fast<0, false>(w, tmem_lane, warp, lane, desc, h0, h1, h2, h3, use);
    }
}

template <bool kRare>
__device__ __forceinline__ void issuer_run(const LineParams &p, uint32_t tmem, uint32_t issuer, int ph, int stop, int it, RoleState &r)
{
    for (; ph < stop; ++ph, r.ws.advance())
        if (r.ok && !Waiter::aborted()) r.ok = issuer_conv<kRare>(p, tmem, lds32(CTRL_ADDR(ptab) + 16u * (uint32_t)ph + 4u), r.ws, issuer, it, r.prev);
}

__device__ __forceinline__ void loader_run(const LineParams &p, int ph, int stop, int it, RoleState &r)
{
    for (; ph < stop && r.next_copy < p.n_conv; ++ph, ++r.next_copy, r.ws.advance())
        if (r.ok && !Waiter::aborted()) r.ok = loader_copy(p, r.next_copy, r.ws.slot, it);
}

// kRare: the network has convolutions whose residual term is no product, or two K-steps of unpaired lines.  A kernel of its own: the
// first's pass alone, beside the other three, cost every network 0.7 % (ResNet-110 at 100,100 samples 62.0 -> 62.5 ms).
template <bool kRare>
__global__ void __launch_bounds__(kThreads, 1) k_line(const __grid_constant__ LineParams p)
{
    Ctrl *ctrl = the_ctrl();
    const uint32_t warp = warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31u;
    for (int i = threadIdx.x; i < p.n_bars; i += blockDim.x) mbar_init(CTRL_ADDR(bars) + 8u * (uint32_t)i, p.bar_counts[i]);
    if (threadIdx.x == 0) {
        for (uint32_t s = 0; s < 3; ++s) mbar_init(CTRL_ADDR(wbar) + 8u * s, 1);
        mbar_init(CTRL_ADDR(drain), kIssuers);
        ctrl->abort_flag = 0;
    }
    for (int i = threadIdx.x; i < p.n_phases; i += blockDim.x) ctrl->ptab[i] = p.ptab[i];
    for (int i = threadIdx.x; i < p.n_conv; i += blockDim.x) ctrl->csrc[i] = p.conv_src[i];
    for (int i = threadIdx.x; i < kMaxBars; i += blockDim.x) ctrl->stored[i] = 0;
    for (int i = threadIdx.x; i < kG * 64; i += blockDim.x) (&ctrl->pool_sum[0][0])[i] = 0;
    if (warp == 0) tmem_alloc(CTRL_ADDR(tmem_base), kTmemCols);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_proxy_async();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = ctrl->tmem_base;
    // accumulators start from the folded biases of the first convolution that uses them
    if (warp < kEpiWarps) {
        const uint32_t lanes = tmem + ((warp & 3u) * 32u << 16);
        for (uint32_t col = (warp >> 2) * 16u; col < (uint32_t)kTmemCols; col += kSets * 16u) {
            const uint4 *v = reinterpret_cast<const uint4 *>(p.acc_init + col);
            tmem_st_columns(lanes + col, __ldg(v), __ldg(v + 1), __ldg(v + 2), __ldg(v + 3));
        }
        tmem_st_wait();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (threadIdx.x == 0) {
        ctrl->cyc[PH_FILL] = ctrl->cyc[PH_INPUT] = ctrl->cyc[PH_TAIL] = 0;
        ctrl->cyc[PH_CONV] = clock64();         // until the end: the start time; what phases leave of the duration is the convolutions
    }
    const int end = min(p.n_phases, p.stop_phase + 1);
    RoleState r;
    int it = 0;
    for (int grp = blockIdx.x; grp < p.n_groups; grp += gridDim.x, ++it) {
        // the first blob of the group: everything of the previous group is complete
        if (warp == kLoaderWarp && p.n_conv > 0) {
            if (lane == 0 && r.ok && !Waiter::aborted()) r.ok = loader_copy(p, 0, r.ws.slot, it);
            r.ws.advance();
            r.next_copy = 1;
        }
        for (int ph = 0; ph < end;) {
            const uint4 e = ld_shared_v4(CTRL_ADDR(ptab) + 16u * (uint32_t)ph);
            if (e.x != PH_CONV) {
                cta_phase(p, e, grp);
                r.prev.n_lines = 0;
                ++ph;
                continue;
            }
            const int stop = min(end, ph + (int)e.z);
            if (warp < kEpiWarps) {
                epilogue_run<kRare>(p, tmem, warp, lane, ph, stop, it, r);
            } else if (lane == 0) {
                if (warp < kLoaderWarp) issuer_run<kRare>(p, tmem, warp - kEpiWarps, ph, stop, it, r);
                else loader_run(p, ph, stop, it, r);
            }
            ph = stop;
        }
        __syncwarp();
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
    }
    // no tensor-core work may be in flight when tensor memory is released
    if (warp >= kEpiWarps && warp < kLoaderWarp && lane == 0) {
        const Waiter w{p.err};
        commit_to(CTRL_ADDR(drain));
        w.barrier(CTRL_ADDR(drain), 0, ERR_WAIT_DRAIN);
    }
    __syncwarp();
    if (threadIdx.x == 0 && p.phase_cycles) {
        const long long total = clock64() - ctrl->cyc[PH_CONV];
        atomicAdd(p.phase_cycles + PH_FILL, (unsigned long long)ctrl->cyc[PH_FILL]);
        atomicAdd(p.phase_cycles + PH_INPUT, (unsigned long long)ctrl->cyc[PH_INPUT]);
        atomicAdd(p.phase_cycles + PH_TAIL, (unsigned long long)ctrl->cyc[PH_TAIL]);
        atomicAdd(p.phase_cycles + PH_CONV, (unsigned long long)(total - ctrl->cyc[PH_FILL] - ctrl->cyc[PH_INPUT] - ctrl->cyc[PH_TAIL]));
    }
    if (p.dump)
        for (uint32_t o = threadIdx.x * 16u; o < p.dump_bytes; o += blockDim.x * 16u)
            *reinterpret_cast<uint4 *>(p.dump + o) = ld_shared_v4(the_base() + p.dump_off + o);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) tmem_dealloc(tmem, kTmemCols);
}

// The engine's wait code on a barrier and a counter that nothing ever completes: one CTA, one thread, the limit given by
// the caller.  The first wait must run out and raise the abort flag and the error word; the second must then fall
// through at once.  out[0..1] = what the two waits returned, out[2] = the abort flag, out[3] = nanoseconds spent.
__global__ void k_wait_probe(int32_t *err, unsigned long long limit_ns, int32_t *out)
{
    Ctrl *ctrl = the_ctrl();
    if (threadIdx.x == 0) {
        mbar_init(smem_u32(&ctrl->bars[0]), 1);
        ctrl->abort_flag = 0;
        ctrl->stored[0] = 0;
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    __syncthreads();
    if (threadIdx.x == 0) {
        const Waiter w{err, limit_ns};
        const unsigned long long t0 = globaltimer();
        out[0] = w.barrier(smem_u32(&ctrl->bars[0]), 0, ERR_WAIT_FULL) ? 1 : 0;
        out[1] = w.counter(smem_u32(&ctrl->stored[0]), 1u, ERR_WAIT_DONE) ? 1 : 0;
        out[2] = ctrl->abort_flag;
        out[3] = (int32_t)min(globaltimer() - t0, 0x7FFFFFFFull);
    }
}

// =============================================================================== host planner

int ilog2(int v) { int l = 0; while ((1 << l) < v) ++l; return l; }

// Geometry of one tensor in the line layout.
struct LGeo {
    int C = 0, H = 0, W = 0, planes = 0, halo = 0;
    int I = 0, nb = 0, n_lines = 0, pitch = 0;       // positions per column, row bands, lines, line pitch in positions
    uint32_t plane_bytes = 0, bytes = 0, line0 = 0;  // line0: byte offset of line 0, lane 0 within a plane
    int buffer = -1, producer_phase = -1, producer_conv = -1;
    bool scatter_produced = false;
    int last_use_layer = -1;
    bool last_use_as_input = false;
};

bool set_geometry(LGeo &t)
{
    if (t.W != 32 && t.W != 16 && t.W != 8) return false;
    if (t.H != t.W) return false;
    t.planes = (t.C + 15) / 16;
    t.I = 128 / t.W;
    t.nb = t.I / kG;
    t.n_lines = t.H / t.nb;
    t.pitch = 128 + t.I;
    const int positions = t.I + (t.n_lines + 2) * t.pitch + 8;      // leading gap, lines -1 .. n_lines with their gaps, slack
    t.plane_bytes = (uint32_t)positions * 16u;
    t.bytes = t.plane_bytes * (uint32_t)t.planes;
    t.line0 = (uint32_t)(t.I + t.pitch) * 16u;
    return true;
}

struct PlanBuffer { uint32_t bytes = 0, off = 0; int birth = 0, death = 0, halo = 0; };
struct AllocReq { uint32_t bytes; int birth, death, slack; uint32_t *off; int conv; };

// First-fit placement of one request among the allocations that are still busy at its birth, from the bottom or from the top.
bool place(std::vector<AllocReq> &done, AllocReq &r, uint32_t capacity, bool high)
{
    std::vector<std::pair<uint32_t, uint32_t>> busy;
    for (const AllocReq &e : done)
        if (e.death >= r.birth - r.slack) busy.push_back({*e.off, *e.off + e.bytes});
    std::sort(busy.begin(), busy.end());
    uint32_t at = kCtrlBytes;
    if (high) {
        uint32_t end = capacity;
        for (auto b = busy.rbegin(); b != busy.rend() && end >= r.bytes; ++b) {
            if (((end - r.bytes) & ~127u) >= b->second) break;
            end = std::min(end, b->first);
        }
        at = end >= r.bytes ? (end - r.bytes) & ~127u : 0u;
        if (at < kCtrlBytes) return false;
    } else {
        for (const auto &b : busy) {
            if (at + r.bytes <= b.first) break;
            at = std::max(at, (b.second + 127u) & ~127u);
        }
        if (at + r.bytes > capacity) return false;
    }
    *r.off = at;
    done.push_back(r);
    return true;
}

// A plan that does not fit is not an error (another engine runs the model); the rule that refused it is kept for
// line_plan_probe, and ISC_PLAN_DEBUG=1 prints it.
thread_local int g_plan_rule = 0;
#define PLAN_FAIL(id) do { g_plan_rule = (id); if (getenv("ISC_PLAN_DEBUG")) fprintf(stderr, "line engine: plan rule %d failed\n", id); return false; } while (0)

bool no_other_way(const PlanTry &how) { return &how == kPlanTries + kPlanUsual && g_plan_rule != kPlanRuleRoom && g_plan_rule != kPlanRuleBars; }

bool conv_ok(const isc_layer &L, bool first)
{
    if (L.op != ISC_CONV2D) return false;
    if (L.kh != L.kw || (L.kh != 1 && L.kh != 3)) return false;
    if (L.pad != (L.kh - 1) / 2) return false;
    if (L.stride != 1 && L.stride != 2) return false;
    if (first) { if (L.cin > 4 || L.stride != 1) return false; }
    else if (L.cin % 16 != 0 || L.cin > 64) return false;
    if (L.cout % 16 != 0 || L.cout > 64) return false;
    return true;
}

}  // namespace

struct LinePlan {
    int in_c = 0, in_h = 0, in_w = 0, n_classes = 0, n_phases = 0, n_conv = 0, n_bars = 0;
    uint32_t smem_bytes = 0;
    LineParams base;
    std::vector<int> phase_kind;
    std::vector<LGeo> tensors;
    std::vector<uint32_t> tensor_off;
    PhaseEntry *d_ptab = nullptr;
    ConvSrc *d_conv_src = nullptr;
    uint8_t *d_bar_counts = nullptr;
    int32_t *d_acc_init = nullptr;
    uint8_t *d_blob = nullptr;
    int8_t *d_fc_w = nullptr;
    FcConst *d_fc_c = nullptr;
    int32_t *d_err = nullptr;
    unsigned long long *d_phase_cycles = nullptr;
    uint8_t *d_dump = nullptr;
    int sm_count = 0;
    bool rare = false;                   // a convolution needs k_line<true>
    int attr_device = -1;                // the device on which the kernel's shared-memory limit has been raised
    // launches smaller than the GPU (see line_run)
    cudaStream_t side[kSideStreams] = {};
    int side_priority = 0, side_device = 0;
    cudaEvent_t fork_event = nullptr, join_event[kSideStreams] = {};
};

namespace {

// What the planner knows about a convolution phase while it builds the operation and pass tables.
struct ConvPlan {
    int layer = -1, phase = -1;
    int in_tensor = -1, out_tensor = -1;
    bool stacked = false, paired = false, scatter = false, general = false;
    ResidualForm res_form;              // of the residual term, and its constant
    int32_t res_c = 0;
    int recs_per_item = 1;              // records of the pass table per (unit, chunk)
    int m = 0;                          // output lines (ordinals)
    int n_chunks = 0, cols = 0, n_banks = 1;
    int cls = -1, use_local = 0;
    std::vector<LOp> ops;
    std::vector<LPass> passes;
    std::vector<int> done_time;         // per output line: index of the pass that stores its last chunk
    int n_units = 0;
    std::vector<int> unit_of;           // per output line: its unit
    std::vector<int> a_delta;
    std::vector<uint32_t> a_lbo;
    std::vector<std::pair<int, int>> kunits;   // per K-step: indices into `units` (second may be -1)
    struct Unit { int r, s, pl; };             // vertical tap (-1 when stacked), horizontal tap, input plane
    std::vector<Unit> units;
};

bool build_plan(const LayerIn *layers, int n_layers, int in_c, int in_h, int in_w, int n_classes, const PlanTry &how, LinePlan *plan,
                std::vector<uint8_t> *blob_out, std::vector<uint32_t> *blob_offsets, std::vector<PhaseEntry> *ptab_out,
                std::vector<ConvSrc> *csrc_out, std::vector<uint8_t> *bar_counts_out, std::vector<int32_t> *acc_init_out)
{
    const int n_conv_layers = n_layers - 2;
    // ---- tensors of the model (tensor t = output of layer t-1)
    std::vector<LGeo> T((size_t)n_layers + 1);
    T[0].C = in_c; T[0].H = in_h; T[0].W = in_w; T[0].halo = layers[0].d.zp_in;
    for (int i = 0; i < n_conv_layers; ++i) {
        const isc_layer &L = layers[i].d;
        const LGeo &in = T[(size_t)L.in_tensor];
        LGeo &o = T[(size_t)i + 1];
        o.C = L.cout;
        o.H = (in.H + 2 * L.pad - L.kh) / L.stride + 1;
        o.W = (in.W + 2 * L.pad - L.kw) / L.stride + 1;
        o.halo = L.zp_out;
        if (L.stride == 2 && ((in.H & 1) || (in.W & 1))) PLAN_FAIL(1);
    }
    for (int t = 0; t <= n_conv_layers; ++t)
        if (!set_geometry(T[(size_t)t])) PLAN_FAIL(2);
    if (T[0].nb != 1) PLAN_FAIL(3);                 // the input writer knows one row band only
    for (int i = 0; i < n_layers; ++i) {
        const isc_layer &L = layers[i].d;
        T[(size_t)L.in_tensor].last_use_layer = i;
        T[(size_t)L.in_tensor].last_use_as_input = true;
        if (L.res_tensor >= 0) {
            T[(size_t)L.res_tensor].last_use_layer = i;
            T[(size_t)L.res_tensor].last_use_as_input = false;
        }
    }
    // ---- phase skeleton: FILL(input) INPUT, then per convolution [FILL of a fresh output] CONV, then TAIL
    struct Skel { int kind; int layer; int tensor; };
    std::vector<Skel> skel;
    std::vector<PlanBuffer> buffers;
    std::vector<int> layer_phase((size_t)n_layers, -1);
    auto new_buffer = [&](int tensor) {
        PlanBuffer b;
        b.bytes = T[(size_t)tensor].bytes; b.halo = T[(size_t)tensor].halo;
        b.birth = (int)skel.size();
        buffers.push_back(b);
        T[(size_t)tensor].buffer = (int)buffers.size() - 1;
        skel.push_back({PH_FILL, -1, tensor});
    };
    new_buffer(0);
    skel.push_back({PH_INPUT, -1, 0});
    int prev_conv_layer = -1;
    for (int i = 0; i < n_conv_layers; ++i) {
        const isc_layer &L = layers[i].d;
        const int out_t = i + 1;
        LGeo &o = T[(size_t)out_t];
        bool placed = false;
        // (a) in place over the residual operand, when this layer is its last reader
        if (L.res_tensor >= 0 && L.stride == 1 && T[(size_t)L.res_tensor].last_use_layer == i &&
            L.res_tensor != L.in_tensor && T[(size_t)L.res_tensor].halo == o.halo &&
            T[(size_t)L.res_tensor].bytes == o.bytes && T[(size_t)L.res_tensor].W == o.W) {
            o.buffer = T[(size_t)L.res_tensor].buffer;
            placed = true;
        }
        // (b) over a same-shaped tensor whose last reader was the previous convolution, as its input
        if (!placed && L.stride == 1 && prev_conv_layer >= 0)
            for (int t = 1; t <= n_conv_layers && !placed; ++t) {
                const LGeo &x = T[(size_t)t];
                if (x.buffer < 0 || t == out_t || t == L.in_tensor || t == L.res_tensor) continue;
                if (x.last_use_layer != prev_conv_layer || !x.last_use_as_input) continue;
                if (x.C != o.C || x.H != o.H || x.W != o.W || x.halo != o.halo) continue;
                bool newest = true;           // x must be the current tenant of its buffer
                for (int u = t + 1; u <= n_conv_layers; ++u)
                    if (T[(size_t)u].buffer == x.buffer) newest = false;
                if (newest) { o.buffer = x.buffer; placed = true; }
            }
        if (!placed) new_buffer(out_t);
        layer_phase[(size_t)i] = (int)skel.size();
        skel.push_back({PH_CONV, i, -1});
        prev_conv_layer = i;
    }
    const int tail_phase = (int)skel.size();
    skel.push_back({PH_TAIL, -1, n_conv_layers});
    layer_phase[(size_t)n_layers - 2] = tail_phase;
    layer_phase[(size_t)n_layers - 1] = tail_phase;
    const int n_phases = (int)skel.size();
    if (n_phases > kMaxPhases) PLAN_FAIL(4);
    // ---- lifetimes
    for (int t = 0; t <= n_conv_layers; ++t) {
        LGeo &x = T[(size_t)t];
        if (x.buffer < 0) PLAN_FAIL(5);
        int death = x.last_use_layer >= 0 ? layer_phase[(size_t)x.last_use_layer] : -1;
        x.producer_phase = t >= 1 ? layer_phase[(size_t)t - 1] : 1;
        death = std::max(death, x.producer_phase);
        buffers[(size_t)x.buffer].death = std::max(buffers[(size_t)x.buffer].death, death);
    }
    // ---- convolutions: K-steps, operations, passes
    std::vector<ConvPlan> convs;
    std::map<std::pair<int, int>, int> class_of;            // (lines, chunks) -> class
    std::vector<int> class_lines, class_chunks, class_uses;
    for (int ph = 0; ph < n_phases; ++ph) {
        if (skel[(size_t)ph].kind != PH_CONV) continue;
        ConvPlan cp;
        cp.layer = skel[(size_t)ph].layer; cp.phase = ph;
        const isc_layer &L = layers[cp.layer].d;
        cp.in_tensor = L.in_tensor; cp.out_tensor = cp.layer + 1;
        LGeo &in = T[(size_t)cp.in_tensor];
        LGeo &out = T[(size_t)cp.out_tensor];
        out.producer_conv = (int)convs.size();
        cp.scatter = L.stride == 2;
        out.scatter_produced = cp.scatter;
        cp.n_chunks = L.cout / 16; cp.cols = L.cout;
        if (cp.scatter && (in.n_lines & 1)) PLAN_FAIL(6);
        cp.m = cp.scatter ? in.n_lines / 2 : in.n_lines;
        if (cp.m > kMaxLines || cp.m * cp.cols > kTmemCols) PLAN_FAIL(7);
        cp.stacked = L.kh == 3 && L.stride == 1 && in.n_lines >= 2;
        cp.n_banks = kTmemCols / (cp.m * cp.cols) >= 2 ? 2 : 1;
        if (L.res_tensor >= 0) {
            const LGeo &r = T[(size_t)L.res_tensor];
            if (cp.scatter || r.W != out.W || r.H != out.H || r.C != out.C) PLAN_FAIL(8);
            const int res_n = 31 - L.res_shift;
            if (res_n != 31 && res_n != 32) PLAN_FAIL(9);
        }
        // K units and steps
        const int s_lo = L.kw == 3 ? -1 : 0, s_hi = L.kw == 3 ? 1 : 0;
        if (cp.stacked) {
            for (int pl = 0; pl < in.planes; ++pl)
                for (int s = s_lo; s <= s_hi; ++s) cp.units.push_back({-1, s, pl});
        } else {
            const int r_lo = L.kh == 3 ? 0 : 1, r_hi = L.kh == 3 ? 2 : 1;
            for (int pl = 0; pl < in.planes; ++pl)
                for (int r = r_lo; r <= r_hi; ++r)
                    for (int s = s_lo; s <= s_hi; ++s) cp.units.push_back({r, s, pl});
        }
        auto unit_addr = [&](const ConvPlan::Unit &u) {
            const int dr = cp.stacked ? 0 : u.r - 1;
            return (long long)u.pl * in.plane_bytes + ((long long)dr * in.pitch + (long long)u.s * in.I) * 16;
        };
        // Three units (16 input channels): two lines share their odd ones.  The K-steps of lines p and p + 1 are (p: left, centre),
        // (p: right, p + 1: left), (p + 1: centre, right); the middle one adds to four output lines, with zero weights where a line
        // does not reach.  Three MMAs for two lines instead of four with half of every second one empty: stage 1 of a CIFAR
        // ResNet takes 2,450 instead of 2,990 cycles of operand reads a convolution.
        cp.paired = how.paired && cp.stacked && cp.units.size() == 3 && in.n_lines % 2 == 0;
        if (cp.paired) {
            const long long u0 = unit_addr(cp.units[0]), u1 = unit_addr(cp.units[1]), u2 = unit_addr(cp.units[2]), pitch = (long long)in.pitch * 16;
            cp.a_delta = {(int)u0, (int)u2, (int)(pitch + u1)};
            cp.a_lbo = {(uint32_t)(u1 - u0), (uint32_t)(pitch + u0 - u2), (uint32_t)(u2 - u1)};
            cp.kunits = {{0, 1}, {2, 0}, {1, 2}};
        }
        for (size_t a = 0; a < cp.units.size() && !cp.paired; a += 2) {
            if (a + 1 < cp.units.size()) {
                const long long d = unit_addr(cp.units[a + 1]) - unit_addr(cp.units[a]);
                if (d <= 0 || d >= (1 << 18)) PLAN_FAIL(10);
                cp.kunits.push_back({(int)a, (int)a + 1});
                cp.a_delta.push_back((int)unit_addr(cp.units[a]));
                cp.a_lbo.push_back((uint32_t)d);
            } else {
                cp.kunits.push_back({(int)a, -1});
                cp.a_delta.push_back((int)unit_addr(cp.units[a]));
                cp.a_lbo.push_back(16u);
            }
        }
        if ((int)cp.kunits.size() > kMaxKsteps) PLAN_FAIL(11);
        // ---- operations
        const ConvPlan *pv = (!convs.empty() && convs.back().phase == ph - 1) ? &convs.back() : nullptr;
        // same lines and chunks: the same barriers (class) and, with one bank, the same accumulator columns
        const bool same_class = pv && pv->m == cp.m && pv->n_chunks == cp.n_chunks && pv->scatter == cp.scatter;
        // the previous convolution produced this one's input, line for line
        const bool aligned = pv && in.producer_conv == (int)convs.size() - 1 && !pv->scatter;
        // Same class: the same barriers, and with one bank the same accumulator columns.  An operation then waits for
        // the previous convolution's lines of the same numbers as the output lines it adds to, so that no line of
        // this convolution can be stored (and arrive on the line's barrier) before that line of the previous one.
        const bool slots = same_class;
        auto prev_time = [&](int line) { return pv ? pv->done_time[(size_t)line] : 0; };
        auto src_line = [&](int p) -> int {       // which output line of the producer fills input line p (-1: constant)
            if (p >= 0 && p < in.n_lines) return p;
            if (in.nb == 1) return -1;
            return p < 0 ? in.n_lines - 1 : 0;
        };
        struct ProtoOp { int a_line, b_block, n_blocks, d_line, n_chains; std::vector<int> need; std::vector<int> outs; int ready; };
        std::vector<ProtoOp> proto;
        if (cp.paired) {
            for (int p = -1; p <= in.n_lines - 1; p += 2) {
                ProtoOp o;
                o.n_chains = 1;
                o.a_line = p;
                const int y_lo = std::max(p - 1, 0), y_hi = std::min(p + 2, in.n_lines - 1);
                o.d_line = y_lo; o.n_blocks = 3;
                const int y_hi0 = std::min(p + 1, in.n_lines - 1), y_lo2 = std::max(p, 0);
                o.b_block = (y_hi0 - y_lo + 1) | (y_lo - (p - 1)) << 3 | ((y_hi - y_lo + 1) | (y_lo - (p - 1)) << 3) << 7 |
                            ((y_hi - y_lo2 + 1) | (y_lo2 - p) << 3 | (y_lo2 - y_lo) << 5) << 14;
                for (int y = y_lo; y <= y_hi; ++y) o.outs.push_back(y);
                for (int l = p; l <= p + 1 && aligned; ++l)
                    if (src_line(l) >= 0) o.need.push_back(src_line(l));
                if (slots) for (int y = y_lo; y <= y_hi; ++y) o.need.push_back(y);
                proto.push_back(o);
            }
        } else if (cp.stacked) {
            for (int p = -1; p <= in.n_lines; ++p) {
                ProtoOp o;
                o.n_chains = 1;
                o.a_line = p;
                const int y_lo = std::max(p - 1, 0), y_hi = std::min(p + 1, in.n_lines - 1);
                o.b_block = y_lo - (p - 1); o.n_blocks = y_hi - y_lo + 1; o.d_line = y_lo;
                for (int y = y_lo; y <= y_hi; ++y) o.outs.push_back(y);
                if (aligned && src_line(p) >= 0) o.need.push_back(src_line(p));
                if (slots) for (int y = y_lo; y <= y_hi; ++y) o.need.push_back(y);
                proto.push_back(o);
            }
        } else {
            for (int j = 0; j < cp.m; ++j) {
                ProtoOp o;
                o.n_chains = 1;
                const int cline = cp.scatter ? 2 * j : j;
                o.a_line = cline; o.b_block = 0; o.n_blocks = 1; o.d_line = j;
                o.outs.push_back(j);
                if (aligned)
                    for (int r = (L.kh == 3 ? -1 : 0); r <= (L.kh == 3 ? 1 : 0); ++r)
                        if (src_line(cline + r) >= 0) o.need.push_back(src_line(cline + r));
                if (slots) o.need.push_back(j);
                proto.push_back(o);
            }
        }
        for (ProtoOp &o : proto) {
            o.ready = 0;
            for (int l : o.need) o.ready = std::max(o.ready, prev_time(l));
        }
        std::stable_sort(proto.begin(), proto.end(), [](const ProtoOp &a, const ProtoOp &b) { return a.ready < b.ready; });
        // In long paired convolutions two consecutive pairs make one operation, where lines are not paired up to four chains: an issuing
        // thread spends as much on a record as on its MMAs.
        const int step = cp.paired ? 2 : 1;                          // lines of a chain
        if (cp.stacked && (cp.paired || cp.kunits.size() == 2) && cp.m >= 16) {
            std::vector<ProtoOp> merged;
            for (const ProtoOp &o : proto) {
                ProtoOp *l = merged.empty() ? nullptr : &merged.back();
                if (l && l->n_chains < how.chains && l->a_line + step * l->n_chains == o.a_line && l->d_line + step * l->n_chains == o.d_line &&
                    l->n_blocks == o.n_blocks && l->b_block == o.b_block && (!cp.paired || o.b_block == (int)kPairInner)) {
                    l->n_chains += 1;
                    l->ready = std::max(l->ready, o.ready);
                    for (int n : o.need) if (std::find(l->need.begin(), l->need.end(), n) == l->need.end()) l->need.push_back(n);
                    for (int y : o.outs) if (std::find(l->outs.begin(), l->outs.end(), y) == l->outs.end()) l->outs.push_back(y);
                } else {
                    merged.push_back(o);
                }
            }
            proto.swap(merged);
        }
        // completion of each output line = the last operation that contributes to it
        std::vector<int> last_op((size_t)cp.m, -1);
        for (size_t i = 0; i < proto.size(); ++i)
            for (int y : proto[i].outs) last_op[(size_t)y] = (int)i;
        // ---- units: the lines of a pass, in the order of completion; one barrier pair per unit
        std::vector<int> order((size_t)cp.m);
        for (int y = 0; y < cp.m; ++y) order[(size_t)y] = y;
        std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return last_op[(size_t)a] < last_op[(size_t)b]; });
        // A record of the pass table covers `sup` lines; a unit (one "accumulators complete" barrier, one "stored"
        // counter) covers `upl` lines = one or two records.  Long convolutions take four-line units: every barrier
        // arrival costs an issuing thread a tcgen05.commit and every unit costs an epilogue warp a wait and an arrival.
        const int sup = cp.m >= 2 ? 2 : 1;
        // The fast pass covers pairs of lines with the saturating pack as the only clamp.  The residual term is a single-precision
        // product where that exists and its constant fits into every channel's rounding addend, else the general form's.
        bool general = (cp.m & 1) || (L.relu && L.zp_out > -128);
        for (int oc = 0; oc < L.cout; ++oc) general = general || layers[cp.layer].shift[oc] == 1;
        if (!general && L.res_tensor >= 0) {
            cp.res_form = residual_form(L.res_mult, L.res_shift, L.zp_res, &cp.res_c);
            bool fits = cp.res_form.exists();
            for (int oc = 0; oc < L.cout && fits; ++oc) {
                const int sft = layers[cp.layer].shift[oc] - 1;
                fits = sft >= 1 && requant_addend_fits((1ll << (sft - 1)) + ((long long)L.zp_out - cp.res_c) * (1ll << sft));
            }
            if (!fits) { cp.res_form = ResidualForm(); cp.res_c = 0; }
        }
        cp.general = general;
        const int upl = (!general && cp.m >= 16 && cp.m % 4 == 0 && !(how.packed && cp.scatter)) ? 4 : sup;
        cp.recs_per_item = upl / sup;
        cp.n_units = (cp.m + upl - 1) / upl;
        cp.unit_of.assign((size_t)cp.m, 0);
        std::vector<int> unit_last_op((size_t)cp.n_units, -1);
        for (int i = 0; i < cp.m; ++i) {
            const int u = i / upl;
            cp.unit_of[(size_t)order[(size_t)i]] = u;
            unit_last_op[(size_t)u] = std::max(unit_last_op[(size_t)u], last_op[(size_t)order[(size_t)i]]);
        }
        // class: same number of units and chunks = same barriers
        const auto key = std::make_pair(cp.n_units, cp.n_chunks);
        if (!class_of.count(key)) {
            class_of[key] = (int)class_lines.size();
            class_lines.push_back(cp.n_units); class_chunks.push_back(cp.n_chunks); class_uses.push_back(0);
        }
        cp.cls = class_of[key];
        cp.use_local = class_uses[(size_t)cp.cls]++;
        // Maps in several bands: the edge rows of a band are copied into the padding lines of its neighbours, and those copies
        // are ordered line by line through the rows above and below that a stacked filter on the previous convolution's
        // output waits for.  A 1 x 1 convolution, or one of an older tensor, waits for the rows it adds to only: by then the
        // copies that it reads may not be written, and others may still be read that its own will overwrite.
        const bool wait_all = pv && (pv->cls != cp.cls || !same_class || (in.nb > 1 && !(cp.stacked && aligned)));
        // Record i belongs to issuing thread i mod kIssuers; every thread needs a record to carry its arrivals.
        auto null_op = []() { ProtoOp o; o.a_line = 0; o.b_block = 0; o.n_blocks = 0; o.d_line = 0; o.n_chains = 0; o.ready = 0; return o; };
        while (proto.size() < (size_t)kIssuers) proto.push_back(null_op());
        // Each thread arrives on every unit's barrier once: after its last record that adds to the unit, or with any
        // of its records if it has none (at most three arrivals fit a record; empty records are added as needed).
        std::vector<std::vector<int>> commits;
        for (int attempt = 0;; ++attempt) {
            commits.assign(proto.size(), std::vector<int>());
            bool fits = true;
            std::vector<std::vector<char>> has((size_t)cp.n_units, std::vector<char>((size_t)kIssuers, 0));
            for (int u = 0; u < cp.n_units && fits; ++u)
                for (int wi = 0; wi < kIssuers && fits; ++wi) {
                    int last = -1;
                    for (size_t i = (size_t)wi; i < proto.size(); i += kIssuers)
                        for (int y : proto[i].outs)
                            if (cp.unit_of[(size_t)y] == u) last = (int)i;
                    if (last < 0) continue;
                    if (commits[(size_t)last].size() >= 3) fits = false;
                    else { commits[(size_t)last].push_back(u); has[(size_t)u][(size_t)wi] = 1; }
                }
            for (int u = 0; u < cp.n_units && fits; ++u)
                for (int wi = 0; wi < kIssuers && fits; ++wi) {
                    if (has[(size_t)u][(size_t)wi]) continue;
                    // in a long convolution the record just before the unit completes, else any
                    int carrier = -1;
                    for (size_t i = (size_t)wi; i < proto.size(); i += kIssuers)
                        if (commits[i].size() < 3 && (carrier < 0 || (cp.m >= 16 && (int)i <= unit_last_op[(size_t)u]))) carrier = (int)i;
                    if (carrier < 0) fits = false;
                    else commits[(size_t)carrier].push_back(u);
                }
            if (fits) break;
            if (attempt >= 8) PLAN_FAIL(13);
            while (proto.size() % kIssuers) proto.push_back(null_op());
            for (int wi = 0; wi < kIssuers; ++wi) proto.push_back(null_op());
        }
        // No thread may still be reading the table when the convolution is complete (its blob's place may then be
        // reused): every thread's last record must carry an arrival, so empty records at the end are dropped.
        while (!proto.empty() && proto.back().n_blocks == 0 && commits.back().empty()) { proto.pop_back(); commits.pop_back(); }
        for (int wi = 0; wi < kIssuers; ++wi) {
            int last = -1;
            for (size_t i = (size_t)wi; i < proto.size(); i += kIssuers) last = (int)i;
            if (last < 0 || commits[(size_t)last].empty()) PLAN_FAIL(23);
        }
        // each thread waits, once, for what its own records need
        std::vector<std::vector<char>> waited((size_t)kIssuers, std::vector<char>(pv ? (size_t)pv->n_units : 0, 0));
        std::vector<char> all_waited(pv ? (size_t)pv->n_units : 0, 0);
        for (size_t i = 0; i < proto.size(); ++i) {
            const ProtoOp &o = proto[i];
            const size_t wi = i % kIssuers;
            LOp op;
            memset(&op, 0xFF, sizeof(op));
            op.flags = (uint16_t)(o.n_chains << 10);
            op.d_col = (uint32_t)(o.d_line * cp.cols);
            const uint32_t a_fmt_bit = cp.in_tensor == 0 ? 0u : 1u;
            op.idesc = (2u << 4) | (a_fmt_bit << 7) | (1u << 10) | ((128u >> 4) << 24);
            if (!cp.paired) op.idesc |= (uint32_t)((std::max(o.n_blocks, 1) * L.cout) >> 3) << 17;
            op.a_add = (uint32_t)(o.a_line + 1) * (uint32_t)in.pitch;
            op.b_add = cp.paired ? (uint32_t)o.b_block : (uint32_t)o.b_block * (uint32_t)L.cout * 2u;
            if (i < (size_t)kIssuers && wait_all) {
                op.flags |= OPF_WAIT_ALL;
                std::fill(waited[wi].begin(), waited[wi].end(), 1);
            }
            int n_wait = 0, n_commit = 0;
            std::vector<int> need_units;
            for (int l : o.need) need_units.push_back(pv->unit_of[(size_t)l]);
            // A thread may arrive on a unit's barrier only when the barrier's previous use is over.  Between
            // convolutions of one class that use is the previous convolution's unit of the same number; anything
            // older is complete once the previous convolution is (the thread's first record has waited for all of it).
            if (pv && pv->cls == cp.cls)
                for (int u : commits[i]) need_units.push_back(u);
            for (int u : need_units)
                if (!waited[wi][(size_t)u]) {
                    if (n_wait >= 4) PLAN_FAIL(12);
                    op.wait[n_wait++] = (uint16_t)(4 * u);
                    waited[wi][(size_t)u] = 1;
                    all_waited[(size_t)u] = 1;
                }
            for (int u : commits[i]) op.commit[n_commit++] = (uint16_t)(8 * u);
            // unused wait slots repeat the first one, so that the kernel reads two (or four) counters without looking
            if (n_wait) {
                op.flags |= OPF_WAITS | (n_wait > 2 ? OPF_WAITS4 : 0);
                for (int k = n_wait; k < 4; ++k) op.wait[k] = op.wait[0];
            }
            op.flags |= (uint16_t)(n_wait << 4) | (uint16_t)(n_commit << 8);
            cp.ops.push_back(op);
        }
        // "this convolution complete" must imply "the previous one complete": between them the threads wait for all its units
        if (pv && !wait_all)
            for (char wtd : all_waited)
                if (!wtd) PLAN_FAIL(20);
        // ---- passes: unit by unit, chunk by chunk
        cp.done_time.assign((size_t)cp.m, 0);
        int n_items = 0;
        for (int u = 0; u < cp.n_units; ++u)
            for (int ch = 0; ch < cp.n_chunks; ++ch, ++n_items)
              for (int rec = 0; rec < cp.recs_per_item; ++rec) {
                const int first = u * upl + rec * sup;
                const int n = std::min(sup, cp.m - first);
                LPass P;
                memset(&P, 0, sizeof(P));
                P.meta = (uint32_t)u | ((uint32_t)n << 8) | ((uint32_t)ch << 12);
                for (int q = 0; q < n; ++q) {
                    const int line = order[(size_t)first + q];
                    P.lines |= (uint32_t)line << (8 * q);
                    P.tcol[q] = (uint32_t)(line * cp.cols + ch * 16);
                    P.out[q] = (cp.scatter ? 0u : (uint32_t)(line * out.pitch) * 16u) + (uint32_t)ch * out.plane_bytes;
                    P.res[q] = L.res_tensor >= 0 ? (uint32_t)(line * out.pitch) * 16u + (uint32_t)ch * T[(size_t)L.res_tensor].plane_bytes : 0u;
                    if (!cp.scatter) {
                        if (line == 0) P.meta |= 1u << (16 + 2 * q);
                        if (line == out.n_lines - 1) P.meta |= 1u << (17 + 2 * q);
                    }
                    cp.done_time[(size_t)line] = n_items / kSets;
                }
                cp.passes.push_back(P);
              }
        convs.push_back(cp);
    }
    const int n_conv = (int)convs.size();
    if (n_conv > kMaxConv) PLAN_FAIL(22);
    // ---- start values of the accumulators: whoever reads 16 columns leaves in them the folded biases of the channels that
    // the next convolution on these columns (in the cyclic order of the groups) puts there
    std::vector<std::vector<int32_t>> bias((size_t)n_conv);
    for (int c = 0; c < n_conv; ++c) {
        const isc_layer &L = layers[convs[(size_t)c].layer].d;
        const LayerIn &ML = layers[convs[(size_t)c].layer];
        const int per = L.cin * L.kh * L.kw;
        for (int oc = 0; oc < L.cout; ++oc) {
            long long wsum = 0;
            for (int q = 0; q < per; ++q) wsum += ML.w[(size_t)oc * per + q];
            const long long b = (long long)ML.bias[oc] - (long long)L.zp_in * wsum;
            if (b < -(1ll << 31) || b >= (1ll << 31)) PLAN_FAIL(24);
            bias[(size_t)c].push_back((int32_t)b);
        }
    }
    auto bank_base = [&](int c) { const ConvPlan &cp = convs[(size_t)c]; return (cp.n_banks > 1 && (cp.use_local & 1)) ? cp.m * cp.cols : 0; };
    // the convolution after `c` that uses column `col`, and its 16 channels there: *first; -1: none
    auto next_user = [&](int c, int col, int *first) {
        for (int d = 1; d <= n_conv; ++d) {
            const int q = (c + d) % n_conv, at = col - bank_base(q);
            if (at < 0 || at >= convs[(size_t)q].m * convs[(size_t)q].cols) continue;
            *first = at % convs[(size_t)q].cols;
            return q;
        }
        return -1;
    };
    std::vector<std::vector<std::pair<int, int>>> vecs((size_t)n_conv);         // per convolution: (next user, its first channel)
    for (int c = 0; c < n_conv; ++c)
        for (LPass &P : convs[(size_t)c].passes)
            for (uint32_t q = 0; q < ((P.meta >> 8) & 0xFu); ++q) {
                std::pair<int, int> key;
                key.first = next_user(c, bank_base(c) + (int)P.tcol[q], &key.second);
                std::vector<std::pair<int, int>> &v = vecs[(size_t)c];
                const size_t at = (size_t)(std::find(v.begin(), v.end(), key) - v.begin());
                if (at == v.size()) v.push_back(key);
                if (at >= 64) PLAN_FAIL(26);
                P.meta |= (uint32_t)at << (20 + 6 * q);
            }
    // the columns of 16 are in the order of the epilogue's fragments: column 8 h + 2 c + e is channel 4 c + 2 h + e
    auto channel_of = [](int col) { return (col & ~15) | ((col & 6) << 1) | ((col & 8) >> 2) | (col & 1); };
    acc_init_out->assign((size_t)kTmemCols, 0);
    for (int col = 0; col < kTmemCols; col += 16) {
        int first = 0;
        const int q = next_user(n_conv - 1, col, &first);
        for (int b = 0; b < 16 && q >= 0; ++b) (*acc_init_out)[(size_t)col + b] = bias[(size_t)q][(size_t)channel_of(first + b)];
    }
    // ---- barriers: per class, one per output line for "accumulators complete" and one for "line stored"
    std::vector<int> class_full(class_lines.size()), class_done(class_lines.size());
    bar_counts_out->clear();
    for (size_t k = 0; k < class_lines.size(); ++k) {
        class_full[k] = (int)bar_counts_out->size();
        for (int l = 0; l < 2 * class_lines[k]; ++l) bar_counts_out->push_back((uint8_t)kIssuers);    // two sets, one arrival per issuing thread
        class_done[k] = (int)bar_counts_out->size();
        for (int l = 0; l < class_lines[k]; ++l) bar_counts_out->push_back((uint8_t)(4 * class_chunks[k]));
    }
    if ((int)bar_counts_out->size() > kMaxBars) PLAN_FAIL(kPlanRuleBars);
    // ---- blob sizes and shared-memory placement in order of birth
    std::vector<uint32_t> w_bytes((size_t)n_conv), w_off((size_t)n_conv), w_rel((size_t)n_conv), c_rel((size_t)n_conv),
        ops_rel((size_t)n_conv), passes_rel((size_t)n_conv), vec_rel((size_t)n_conv);
    for (int c = 0; c < n_conv; ++c) {
        const ConvPlan &cp = convs[(size_t)c];
        const isc_layer &L = layers[cp.layer].d;
        const uint32_t rows = (uint32_t)(cp.stacked ? 3 : 1) * (uint32_t)L.cout;
        uint32_t at = how.packed ? (uint32_t)(offsetof(LConvDesc, a_lo) + (cp.kunits.size() + 3) / 4 * 16) : (uint32_t)sizeof(LConvDesc);
        ops_rel[(size_t)c] = at; at += ((uint32_t)cp.ops.size() + (uint32_t)kIssuers) * (uint32_t)sizeof(LOp);    // spare records: reads run one ahead
        passes_rel[(size_t)c] = at; at += (uint32_t)cp.passes.size() * (uint32_t)sizeof(LPass);
        at = (at + 127u) & ~127u;
        w_rel[(size_t)c] = at; at += cp.paired ? 10u * (uint32_t)L.cout * 32u : (uint32_t)cp.kunits.size() * rows * 32u;
        c_rel[(size_t)c] = at; at += (uint32_t)(L.cout / 16) * kChunkConstBytes;
        vec_rel[(size_t)c] = at; at += (uint32_t)vecs[(size_t)c].size() * kVecBytes;
        w_bytes[(size_t)c] = (at + 127u) & ~127u;
    }
    std::vector<AllocReq> reqs, placed;
    for (PlanBuffer &b : buffers) reqs.push_back({b.bytes, b.birth, b.death, 0, &b.off, -1});
    for (int c = 0; c < n_conv; ++c)
        reqs.push_back({w_bytes[(size_t)c], c == 0 ? 0 : convs[(size_t)c - 1].phase, convs[(size_t)c].phase, c == 0 ? 0 : 1,
                        &w_off[(size_t)c], c});
    std::stable_sort(reqs.begin(), reqs.end(), [](const AllocReq &a, const AllocReq &b) { return a.birth < b.birth; });
    uint32_t high = kCtrlBytes;
    std::vector<char> late((size_t)n_conv, 0);
    // Packed plans try other places, tensors from the top and blobs from the bottom first and then either at random.
    uint32_t dice = 1;
    auto from_top = [&](const AllocReq &r, int attempt) {
        if (!how.packed) return false;
        if (attempt == 0) return r.conv < 0;
        dice ^= dice << 13; dice ^= dice >> 17; dice ^= dice << 5;
        return (dice & 4u) != 0;
    };
    auto lay_out = [&](int attempt) {
        placed.clear();
        std::fill(late.begin(), late.end(), 0);
        high = kCtrlBytes;
        for (AllocReq &r : reqs) {
            r.slack = r.conv > 0 ? 1 : 0;
            bool ok = place(placed, r, kSmemLimit, from_top(r, attempt));
            if (!ok && r.conv > 0) {
                // A blob is normally copied when the convolution before its own starts, while the one before that may
                // still be in its epilogue (slack 1).  Where that does not fit, it is copied once that one is complete.
                r.slack = 0;
                late[(size_t)r.conv] = 1;
                ok = place(placed, r, kSmemLimit, from_top(r, attempt));
            }
            if (!ok) {
                if (getenv("ISC_PLAN_DEBUG") && attempt == 0) {
                    fprintf(stderr, "line engine: no room for %u bytes born at phase %d (dies %d); busy then:\n", r.bytes, r.birth, r.death);
                    for (const AllocReq &e : placed)
                        if (e.death >= r.birth - r.slack)
                            fprintf(stderr, "  [%u, %u) phases %d..%d\n", *e.off, *e.off + e.bytes, e.birth, e.death);
                }
                return false;
            }
            high = std::max(high, *r.off + r.bytes);
        }
        return true;
    };
    bool laid_out = false;
    for (int attempt = 0; attempt < (how.packed ? kPackAttempts : 1) && !laid_out; ++attempt) laid_out = lay_out(attempt);
    if (!laid_out) PLAN_FAIL(kPlanRuleRoom);
    if (getenv("ISC_PLAN_DEBUG") && atoi(getenv("ISC_PLAN_DEBUG")) > 1)
        for (const AllocReq &r : placed)
            fprintf(stderr, "  %s %d: [%u, %u) phases %d..%d\n", r.conv >= 0 ? "blob" : "tensor", r.conv, *r.off, *r.off + r.bytes, r.birth, r.death);
    plan->tensors = T;
    plan->tensor_off.assign(T.size(), 0);
    for (int t = 0; t <= n_conv_layers; ++t) plan->tensor_off[(size_t)t] = buffers[(size_t)T[(size_t)t].buffer].off;
    // ---- emit phases and blobs
    ptab_out->assign((size_t)n_phases, PhaseEntry{0, 0, 0, 0});
    csrc_out->assign((size_t)n_conv, ConvSrc{0, 0, 0, 0, 0, 0, 0});
    blob_out->clear();
    blob_offsets->assign((size_t)n_conv, 0);
    plan->phase_kind.assign((size_t)n_phases, 0);
    int conv_at = 0;
    for (int ph = 0; ph < n_phases; ++ph) {
        const Skel &S = skel[(size_t)ph];
        PhaseEntry &E = (*ptab_out)[(size_t)ph];
        E.kind = (uint32_t)S.kind;
        plan->phase_kind[(size_t)ph] = S.kind;
        if (S.kind == PH_FILL) {
            E.a = plan->tensor_off[(size_t)S.tensor]; E.b = T[(size_t)S.tensor].bytes; E.c = (uint32_t)(T[(size_t)S.tensor].halo & 0xFF);
            continue;
        }
        if (S.kind != PH_CONV) continue;
        const int c = conv_at++;
        const ConvPlan &cp = convs[(size_t)c];
        const LayerIn &ML = layers[cp.layer];
        const isc_layer &L = ML.d;
        const LGeo &in = T[(size_t)cp.in_tensor], &out = T[(size_t)cp.out_tensor];
        E.a = w_off[(size_t)c];
        for (int q = ph; q < n_phases && skel[(size_t)q].kind == PH_CONV; ++q) E.b += 1;
        std::vector<uint8_t> blob(w_bytes[(size_t)c], 0);
        LConvDesc D;
        memset(&D, 0, sizeof(D));
        plan->rare |= (L.res_tensor >= 0 && !cp.general && !cp.res_form.exists()) || (cp.stacked && cp.kunits.size() == 2);
        D.flags = (L.res_tensor >= 0 ? CF_RES : 0u) | (cp.scatter ? CF_SCATTER : 0u) | (cp.general ? CF_GENERAL : 0u) | (L.res_tensor >= 0 && !cp.res_form.exists() ? CF_RES_LONG : 0u) | (cp.paired ? CF_PAIRED : 0u);
        D.n_items = (uint32_t)(cp.n_units * cp.n_chunks); D.recs_per_item = (uint32_t)cp.recs_per_item; D.d_base = (uint32_t)bank_base(c);
        D.bar_full = (uint32_t)class_full[(size_t)cp.cls]; D.bar_done = (uint32_t)class_done[(size_t)cp.cls];
        D.use_local = (uint32_t)cp.use_local; D.uses_per_group = (uint32_t)class_uses[(size_t)cp.cls];
        D.n_units = (uint32_t)cp.n_units; D.c_rel = c_rel[(size_t)c]; D.passes_rel = passes_rel[(size_t)c];
        D.out_base = plan->tensor_off[(size_t)cp.out_tensor] + out.line0;
        D.dup_delta = out.nb > 1 ? (uint32_t)(out.n_lines * out.pitch - 4) * 16u : 0u;
        D.out_plane = out.plane_bytes; D.out_pitch16 = (uint32_t)out.pitch;
        D.out_log_lines = (uint32_t)ilog2(out.n_lines); D.out_logI = (uint32_t)ilog2(out.I);
        if ((1 << D.out_log_lines) != out.n_lines) PLAN_FAIL(16);
        D.in_logI = (uint32_t)ilog2(in.I); D.in_n_lines = (uint32_t)in.n_lines; D.out_nb = (uint32_t)out.nb; D.vec_rel = vec_rel[(size_t)c];
        D.lo = L.relu ? std::max(-128, L.zp_out) : -128;
        D.n_ops = (uint32_t)cp.ops.size(); D.n_ksteps = (uint32_t)cp.kunits.size(); D.ops_rel = ops_rel[(size_t)c]; D.n_chunks = (uint32_t)cp.n_chunks;
        D.pitch16 = (uint32_t)in.pitch; D.cols = (uint32_t)cp.cols;
        // operand base: line -1, lane 0, plane 0 of the input
        const uint32_t a_base = plan->tensor_off[(size_t)cp.in_tensor] + in.line0 - (uint32_t)in.pitch * 16u;
        if (L.res_tensor >= 0) {
            const LGeo &rt = T[(size_t)L.res_tensor];
            D.res_base = plan->tensor_off[(size_t)L.res_tensor] + rt.line0;
            const int res_n = 31 - L.res_shift;
            const unsigned long long m2 = (unsigned long long)(uint32_t)L.res_mult << (32 - res_n);
            if (L.res_mult <= 0 || m2 >= (1ull << 32)) PLAN_FAIL(17);
            // rs((r - zp) * mult, n) = floor(((u - 128 - zp) * mult + 2^(n-1)) * 2^(32-n) / 2^32), u = r + 128
            const long long r2 = (((1ll << (res_n - 1)) - (128ll + L.zp_res) * (long long)L.res_mult)) * (1ll << (32 - res_n));
            D.gen_res_m2 = (uint32_t)m2;
            D.res_r2_lo = (uint32_t)((unsigned long long)r2 & 0xFFFFFFFFull);
            D.res_r2_hi = (uint32_t)((unsigned long long)r2 >> 32);
            D.res_m2 = cp.res_form.exists() ? cp.res_form.m_bits : (uint32_t)m2;
            D.res_k8 = cp.res_form.exists() ? cp.res_form.k8 : D.res_r2_lo;
        }
        for (size_t k = 0; k < cp.kunits.size(); ++k) {
            const long long a = (long long)a_base + cp.a_delta[k];
            if (a < 0 || (a & 15) || (cp.a_lbo[k] & 15u)) PLAN_FAIL(21);
            D.a_lo[k] = (uint32_t)(a >> 4) | ((cp.a_lbo[k] >> 4) << 16);
        }
        D.b_lo0 = ((w_off[(size_t)c] + w_rel[(size_t)c]) >> 4) | ((128u >> 4) << 16);
        D.kstep16 = (uint32_t)(cp.stacked ? 3 : 1) * (uint32_t)L.cout * 2u;
        // operand reads stay inside the input's region
        for (size_t k = 0; k < cp.kunits.size(); ++k)
            for (const LOp &op : cp.ops) {
                const long long lo_b = (long long)in.line0 - (long long)in.pitch * 16 + (long long)op.a_add * 16 + cp.a_delta[k];
                const long long hi_b = lo_b + cp.a_lbo[k] + 128 * 16 + (long long)std::max(((op.flags >> 10) & 7) - 1, 0) * (cp.paired ? 2 : 1) * in.pitch * 16;
                if (lo_b < 0 || hi_b > (long long)in.bytes) PLAN_FAIL(18);
            }
        memcpy(blob.data(), &D, ops_rel[(size_t)c]);
        memcpy(blob.data() + ops_rel[(size_t)c], cp.ops.data(), cp.ops.size() * sizeof(LOp));
        memcpy(blob.data() + passes_rel[(size_t)c], cp.passes.data(), cp.passes.size() * sizeof(LPass));
        // weights: per K-step, rows = block * cout + column; block b is vertical tap 2 - b when stacked, and 3 - b for the second
        // line's unit of a pair's middle K-step
        const int taps = L.kh * L.kw;
        size_t at_row = 0;
        for (size_t k = 0; k < cp.kunits.size(); ++k) {
            const bool middle = cp.paired && k == 1;
            const uint32_t rows = (uint32_t)(middle ? 4 : cp.stacked ? 3 : 1) * (uint32_t)L.cout;
            const int halves[2] = {cp.kunits[k].first, cp.kunits[k].second};
            for (int hf = 0; hf < 2; ++hf) {
                if (halves[hf] < 0) continue;
                const ConvPlan::Unit &u = cp.units[(size_t)halves[hf]];
                for (uint32_t n = 0; n < rows; ++n) {
                    const int oc = channel_of((int)(n % (uint32_t)L.cout)), blk = (int)(n / (uint32_t)L.cout);
                    const int r = !cp.stacked ? u.r : middle && hf == 1 ? 3 - blk : 2 - blk;
                    if (r < 0 || r > 2) continue;
                    const int tap = L.kh == 3 ? r * 3 + (u.s + 1) : 0;
                    for (int b = 0; b < 16; ++b) {
                        const int ci = u.pl * 16 + b;
                        if (ci >= L.cin) continue;
                        const int8_t wv = ML.w[((size_t)oc * L.cin + ci) * taps + tap];
                        blob[w_rel[(size_t)c] + (at_row + n / 8 * 8) * 32 + (size_t)hf * 128 + (size_t)(n % 8) * 16 + b] = (uint8_t)wv;
                    }
                }
            }
            at_row += rows;
        }
        for (int oc = 0; oc < L.cout; ++oc) {
            const int sh = ML.shift[oc];
            if (sh < 1 || sh > 20) PLAN_FAIL(19);
            const int sft = sh - 1;
            const int32_t cst[3] = {ML.mult[oc], sft ? (int32_t)((1ll << (sft - 1)) + ((long long)L.zp_out - cp.res_c) * (1ll << sft)) : L.zp_out, sft};
            for (int q = 0; q < 3; ++q)
                memcpy(&blob[c_rel[(size_t)c] + (size_t)(oc / 16) * kChunkConstBytes + (size_t)(oc % 16 / 4) * 48 + (size_t)q * 16 + (size_t)(oc % 4) * 4], &cst[q], 4);
            if (sft == 0 && !cp.general) PLAN_FAIL(25);      // a shift of one puts the rounding half in the product's low word
        }
        for (size_t v = 0; v < vecs[(size_t)c].size(); ++v)
            for (int b = 0; b < 16 && vecs[(size_t)c][v].first >= 0; ++b)
                memcpy(&blob[vec_rel[(size_t)c] + v * kVecBytes + (size_t)b * 4], &bias[(size_t)vecs[(size_t)c][v].first][(size_t)channel_of(vecs[(size_t)c][v].second + b)], 4);
        (*blob_offsets)[(size_t)c] = (uint32_t)blob_out->size();
        blob_out->insert(blob_out->end(), blob.begin(), blob.end());
        (*csrc_out)[(size_t)c].bytes_phase = w_bytes[(size_t)c] | ((uint32_t)ph << 24);
        (*csrc_out)[(size_t)c].smem_off = w_off[(size_t)c] | (late[(size_t)c] ? 0x80000000u : 0u);
        {
            // The copy starts while the convolution before this one runs.  The blob's place was last used by the
            // convolution three back or an earlier one (for a late blob: two back), which must be complete by then.
            const int q = late[(size_t)c] ? c - 2 : c - 3;
            ConvSrc &cs = (*csrc_out)[(size_t)c];
            cs.dep_first = cs.dep_units = cs.dep_mult = cs.dep_local_uses = 0;
            if (q >= 0) {
                const ConvPlan &dq = convs[(size_t)q];
                cs.dep_first = (uint32_t)class_done[(size_t)dq.cls];
                cs.dep_units = (uint32_t)dq.n_units;
                cs.dep_mult = 4u * (uint32_t)dq.n_chunks;
                cs.dep_local_uses = (uint32_t)dq.use_local | ((uint32_t)class_uses[(size_t)dq.cls] << 16);
            }
        }
    }
    plan->n_phases = n_phases;
    plan->n_conv = n_conv;
    plan->n_bars = (int)bar_counts_out->size();
    plan->smem_bytes = (high + 127u) & ~127u;
    (void)n_classes;
    return true;
}

}  // namespace

namespace {

// The structure the engine is built for: convolutions, then global average pool, then FC.
bool structure_ok(const LayerIn *layers, int n_layers, int n_classes)
{
    if (n_layers < 3 || n_classes > 128) PLAN_FAIL(101);
    const isc_layer &LP = layers[n_layers - 2].d, &LF = layers[n_layers - 1].d;
    if (LP.op != ISC_GAVGPOOL || LF.op != ISC_FC) PLAN_FAIL(102);
    if (LP.in_tensor != n_layers - 2 || LF.in_tensor != n_layers - 1) PLAN_FAIL(103);
    if (LP.cin > 64 || LP.cin % 16 != 0 || LF.res_tensor >= 0) PLAN_FAIL(104);
    for (int i = 0; i < n_layers - 2; ++i) {
        const isc_layer &L = layers[i].d;
        if (!conv_ok(L, i == 0)) PLAN_FAIL(105);
        if ((i == 0) != (L.in_tensor == 0)) PLAN_FAIL(106);
        if (L.res_tensor == 0) PLAN_FAIL(107);
        // a consumer's zero-point must be the halo value its operand was written with
        if (L.in_tensor > 0 && L.zp_in != layers[L.in_tensor - 1].d.zp_out) PLAN_FAIL(108);
        if (L.in_tensor > i || L.res_tensor > i) PLAN_FAIL(109);
    }
    if (LP.zp_in != layers[n_layers - 3].d.zp_out) PLAN_FAIL(110);
    return true;
}

}  // namespace

int line_plan_probe(const LayerIn *layers, int n_layers, int in_c, int in_h, int in_w, int n_classes, int *rule, uint32_t *smem_bytes)
{
    g_plan_rule = 0;
    *smem_bytes = 0;
    bool ok = structure_ok(layers, n_layers, n_classes);
    if (ok) {
        for (const PlanTry &how : kPlanTries) {
            if (no_other_way(how)) break;
            LinePlan plan;
            std::vector<uint8_t> blob, bar_counts;
            std::vector<uint32_t> blob_off;
            std::vector<PhaseEntry> ptab;
            std::vector<ConvSrc> csrc;
            std::vector<int32_t> acc_init;
            ok = build_plan(layers, n_layers, in_c, in_h, in_w, n_classes, how, &plan, &blob, &blob_off, &ptab, &csrc, &bar_counts, &acc_init);
            if (ok) *smem_bytes = plan.smem_bytes;
            if (ok) break;
        }
    }
    *rule = ok ? 0 : g_plan_rule;
    return ok ? 1 : 0;
}

int line_build(const LayerIn *layers, int n_layers, int in_c, int in_h, int in_w, int n_classes, LinePlan **out)
{
    *out = nullptr;
    if (!structure_ok(layers, n_layers, n_classes)) return ISC_OK;
    const isc_layer &LP = layers[n_layers - 2].d, &LF = layers[n_layers - 1].d;

    LinePlan *plan = nullptr;
    std::vector<uint8_t> blob, bar_counts;
    std::vector<uint32_t> blob_off;
    std::vector<PhaseEntry> ptab;
    std::vector<ConvSrc> csrc;
    std::vector<int32_t> acc_init;
    for (const PlanTry &how : kPlanTries) {
        if (no_other_way(how)) break;
        plan = new LinePlan();
        blob.clear(); bar_counts.clear(); blob_off.clear(); ptab.clear(); csrc.clear();
        if (build_plan(layers, n_layers, in_c, in_h, in_w, n_classes, how, plan, &blob, &blob_off, &ptab, &csrc, &bar_counts, &acc_init)) break;
        delete plan;
        plan = nullptr;
    }
    if (!plan) return ISC_OK;
    plan->in_c = in_c; plan->in_h = in_h; plan->in_w = in_w; plan->n_classes = n_classes;

    int dev = 0;
    cudaDeviceProp prop;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaGetDeviceProperties(&prop, dev) != cudaSuccess) {
        cudaGetLastError(); delete plan; return ISC_ERR_CUDA;
    }
    if (prop.major != 10 || (size_t)prop.sharedMemPerBlockOptin < plan->smem_bytes) { delete plan; return ISC_OK; }
    plan->sm_count = prop.multiProcessorCount;

    // FC parameters (bias folded with the pool output's zero-point)
    const int C = LP.cin;
    std::vector<int8_t> fcw((size_t)n_classes * 64, 0);
    std::vector<FcConst> fcc((size_t)n_classes);
    const LayerIn &MF = layers[n_layers - 1];
    for (int o = 0; o < n_classes; ++o) {
        long long wsum = 0;
        for (int c = 0; c < C; ++c) {
            fcw[(size_t)o * 64 + c] = MF.w[(size_t)o * C + c];
            wsum += MF.w[(size_t)o * C + c];
        }
        FcConst k{};
        k.mult = MF.mult[o]; k.n = 31 + MF.shift[o]; k.zp_out = LF.zp_out;
        k.lo = LF.relu ? std::max(-128, LF.zp_out) : -128;
        k.bias = (int32_t)(MF.bias[o] - (long long)LF.zp_in * wsum);
        fcc[(size_t)o] = k;
    }
    bool cuda_ok = true;
    auto up = [&](void **dst, const void *src, size_t bytes) {
        if (cudaMalloc(dst, std::max<size_t>(bytes, 16)) != cudaSuccess) { cuda_ok = false; *dst = nullptr; return; }
        if (cudaMemcpy(*dst, src, bytes, cudaMemcpyHostToDevice) != cudaSuccess) cuda_ok = false;
    };
    up((void **)&plan->d_blob, blob.data(), blob.size());
    for (size_t c = 0; c < csrc.size(); ++c) csrc[c].gmem = (unsigned long long)(plan->d_blob + blob_off[c]);
    up((void **)&plan->d_ptab, ptab.data(), ptab.size() * sizeof(PhaseEntry));
    up((void **)&plan->d_conv_src, csrc.data(), csrc.size() * sizeof(ConvSrc));
    up((void **)&plan->d_bar_counts, bar_counts.data(), bar_counts.size());
    up((void **)&plan->d_acc_init, acc_init.data(), acc_init.size() * sizeof(int32_t));
    up((void **)&plan->d_fc_w, fcw.data(), fcw.size());
    up((void **)&plan->d_fc_c, fcc.data(), fcc.size() * sizeof(FcConst));
    int32_t zero = 0;
    up((void **)&plan->d_err, &zero, sizeof(zero));
    const unsigned long long zeros4[4] = {0, 0, 0, 0};
    up((void **)&plan->d_phase_cycles, zeros4, sizeof(zeros4));
    if (cuda_ok && cudaMalloc((void **)&plan->d_dump, kSmemLimit) != cudaSuccess) cuda_ok = false;
    if (!cuda_ok) { cudaGetLastError(); line_free(plan); return ISC_ERR_NOMEM; }

    LineParams &b = plan->base;
    memset(&b, 0, sizeof(b));
    b.ptab = plan->d_ptab;
    b.conv_src = plan->d_conv_src;
    b.bar_counts = plan->d_bar_counts;
    b.acc_init = plan->d_acc_init;
    b.n_bars = plan->n_bars;
    b.n_phases = plan->n_phases;
    b.n_conv = plan->n_conv;
    b.in_c = in_c; b.in_H = in_h; b.in_W = in_w;
    b.input_base = plan->tensor_off[0] + plan->tensors[0].line0;
    b.input_pitch16 = (uint32_t)plan->tensors[0].pitch;
    const LGeo &last = plan->tensors[(size_t)n_layers - 2];
    b.tail_base = plan->tensor_off[(size_t)n_layers - 2] + last.line0;
    b.tail_plane = last.plane_bytes; b.tail_pitch16 = (uint32_t)last.pitch; b.tail_logI = (uint32_t)ilog2(last.I);
    b.tail_C = last.C; b.tail_H = last.H; b.tail_W = last.W; b.tail_n_lines = last.n_lines;
    b.pool_mult = layers[n_layers - 2].mult[0];
    b.pool_n = 31 + layers[n_layers - 2].shift[0];
    b.pool_zp_in = LP.zp_in; b.pool_zp_out = LP.zp_out;
    b.pool_lo = LP.relu ? std::max(-128, LP.zp_out) : -128;
    b.fc_w = plan->d_fc_w; b.fc_c = plan->d_fc_c;
    b.n_classes = n_classes;
    b.err = plan->d_err;
    b.phase_cycles = plan->d_phase_cycles;
    b.stop_phase = 1 << 30;
    *out = plan;
    return ISC_OK;
}

static void line_free_streams(LinePlan *p)
{
    for (int i = 0; i < kSideStreams; ++i) {
        if (p->side[i]) cudaStreamDestroy(p->side[i]);
        if (p->join_event[i]) cudaEventDestroy(p->join_event[i]);
        p->side[i] = nullptr;
        p->join_event[i] = nullptr;
    }
    if (p->fork_event) cudaEventDestroy(p->fork_event);
    p->fork_event = nullptr;
}

void line_free(LinePlan *p)
{
    if (!p) return;
    line_free_streams(p);
    cudaFree(p->d_ptab); cudaFree(p->d_conv_src); cudaFree(p->d_bar_counts); cudaFree(p->d_acc_init); cudaFree(p->d_blob); cudaFree(p->d_fc_w);
    cudaFree(p->d_fc_c); cudaFree(p->d_err); cudaFree(p->d_phase_cycles); cudaFree(p->d_dump);
    delete p;
}

// The side streams start after what `st` holds so far.  They have its priority and live on the current device: a call on
// a stream of another priority than the last one's makes them anew (what they held then has been joined and waited for).
static int line_fork(LinePlan *p, cudaStream_t st)
{
    int priority = 0, device = 0;
    if (cudaStreamGetPriority(st, &priority) != cudaSuccess || cudaGetDevice(&device) != cudaSuccess) { cudaGetLastError(); return ISC_ERR_CUDA; }
    if (p->fork_event && (p->side_priority != priority || p->side_device != device)) line_free_streams(p);
    if (!p->fork_event) {
        p->side_priority = priority;
        p->side_device = device;
        bool ok = cudaEventCreateWithFlags(&p->fork_event, cudaEventDisableTiming) == cudaSuccess;
        for (int i = 0; i < kSideStreams && ok; ++i)
            ok = cudaStreamCreateWithPriority(&p->side[i], cudaStreamNonBlocking, priority) == cudaSuccess &&
                 cudaEventCreateWithFlags(&p->join_event[i], cudaEventDisableTiming) == cudaSuccess;
        if (!ok) { cudaGetLastError(); line_free_streams(p); return ISC_ERR_CUDA; }
    }
    bool ok = cudaEventRecord(p->fork_event, st) == cudaSuccess;
    for (int i = 0; i < kSideStreams && ok; ++i) ok = cudaStreamWaitEvent(p->side[i], p->fork_event, 0) == cudaSuccess;
    if (!ok) { cudaGetLastError(); return ISC_ERR_CUDA; }
    return ISC_OK;
}

// ... and `st` goes on after them.
static int line_join(LinePlan *p, cudaStream_t st)
{
    bool ok = true;
    for (int i = 0; i < kSideStreams; ++i)
        ok = cudaEventRecord(p->join_event[i], p->side[i]) == cudaSuccess && cudaStreamWaitEvent(st, p->join_event[i], 0) == cudaSuccess && ok;
    if (!ok) { cudaGetLastError(); return ISC_ERR_CUDA; }
    return ISC_OK;
}

static int line_launch(LinePlan *p, LineParams &q, cudaStream_t st)
{
    const auto kernel = p->rare ? k_line<true> : k_line<false>;
    int device = -1;
    bool ok = cudaGetDevice(&device) == cudaSuccess;
    if (ok && device != p->attr_device) {
        ok = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit) == cudaSuccess;
        if (ok) p->attr_device = device;
    }
    if (!ok) { cudaGetLastError(); return ISC_ERR_CUDA; }
    const int grid = std::max(1, std::min(q.n_groups, p->sm_count));
    kernel<<<grid, kThreads, p->smem_bytes, st>>>(q);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess && getenv("ISC_PLAN_DEBUG")) fprintf(stderr, "line engine: launch failed: %s\n", cudaGetErrorString(e));
    return e == cudaSuccess ? ISC_OK : ISC_ERR_CUDA;
}

int64_t line_wave_samples(const LinePlan *p) { return (int64_t)kG * p->sm_count; }

// Every call's work as launches of at most `batch_hint` samples (0: as few launches as possible).  A launch is a list
// of groups over images and phases: CERTIFY's N0 = 100 samples take 25 of 148 SMs for a whole round when they are launched
// alone.  Launches of less than eight rounds are dealt to side streams, so that the next ones' groups fill the SMs that
// one launch leaves idle (64 groups at 256 samples: 0.49 M samples/s one after the other, 1.19 M so; 1,024 samples on
// ResNet-20 4.3 M, with the fused phases 5.0 M).  From eight rounds on launches run one after the other: 16,384 samples
// each, 27.7 rounds, give 1.28 M samples/s on ResNet-110 where shorter ones that overlap give 1.32 M.
int line_run(LinePlan *p, const LineWork &w, const NoiseStream &ns, int batch_hint, int32_t *err, cudaStream_t st, int64_t *launches)
{
    LineParams q = p->base;
    q.ns = ns;
    q.err = err;
    q.phase_sel = w.phase_sel;
    auto groups = [](int64_t n) { return (int32_t)((n + kG - 1) / kG); };
    if (batch_hint <= 0) {
        q.x = w.x;
        q.image_id0 = w.image_id0;
        q.counts = w.counts;
        q.logits = w.logits;
        q.n_sel = (int32_t)w.n_sel; q.n_est = (int32_t)w.n_est;
        q.groups_sel = groups(w.n_sel); q.groups_est = groups(w.n_est);
        const int64_t n = (int64_t)w.n_images * ((int64_t)q.groups_sel + q.groups_est);
        if (n == 0) return ISC_OK;
        if (n >= (1ll << 31)) return ISC_ERR_ARG;            // callers cut their images into launches far below this
        q.n_groups = (int32_t)n;
        *launches += 1;
        return line_launch(p, q, st);
    }
    const int64_t total = ((w.n_sel + batch_hint - 1) / batch_hint + (w.n_est + batch_hint - 1) / batch_hint) * w.n_images;
    const bool side = total > 1 && batch_hint < 8 * kG * p->sm_count;
    if (side) {
        int rc = line_fork(p, st);
        if (rc) return rc;
    }
    int rc = ISC_OK;
    int64_t at = 0;
    for (int i = 0; i < w.n_images && rc == ISC_OK; ++i)
        for (int ph = w.n_sel ? 0 : 1; ph < 2 && rc == ISC_OK; ++ph) {
            const int64_t n = ph == 0 ? w.n_sel : w.n_est;
            for (int64_t done = 0; done < n && rc == ISC_OK; done += batch_hint, ++at) {
                const int64_t m = std::min<int64_t>(batch_hint, n - done);
                q.x = w.x + (size_t)i * (size_t)(p->in_c * p->in_h * p->in_w);
                q.image_id0 = w.image_id0 + (uint64_t)i;
                q.counts = w.counts + (size_t)(w.n_sel ? 2 * i + ph : i) * p->n_classes;
                q.logits = w.logits ? w.logits + (size_t)done * p->n_classes : nullptr;
                q.n_sel = 0; q.groups_sel = 0;
                q.n_est = (int32_t)m; q.groups_est = groups(m);
                q.ns.ctr3_fixed = ph == 0 ? (uint32_t)w.phase_sel : ns.ctr3_fixed;
                q.ns.first_sample = (ph == 0 ? 0 : ns.first_sample) + done;
                q.n_groups = q.groups_est;
                rc = line_launch(p, q, side ? p->side[at % kSideStreams] : st);
                *launches += 1;
            }
        }
    if (side) {
        const int rj = line_join(p, st);
        if (rc == ISC_OK) rc = rj;
    }
    return rc;
}

// The error word of a launch, read back by the caller after the stream has been synchronised.
int line_status(int32_t e)
{
    if (e == 0) return ISC_OK;
    if (getenv("ISC_PLAN_DEBUG")) fprintf(stderr, "line engine: wait %d on barrier %d parity %d expired in CTA %d\n", e & 0xFF, (e >> 8) & 0xFFF, (e >> 20) & 1, (int)((unsigned)e >> 21));
    return ISC_ERR_TIMEOUT;
}

// The same for the launches that use the plan's own error word, which is cleared.
static int line_check(LinePlan *p)
{
    int32_t e = 0;
    if (cudaMemcpy(&e, p->d_err, sizeof(e), cudaMemcpyDeviceToHost) != cudaSuccess) { cudaGetLastError(); return ISC_ERR_CUDA; }
    if (e != 0) cudaMemset(p->d_err, 0, sizeof(e));
    return line_status(e);
}

int line_wait_probe(LinePlan *p, long long limit_ns, int32_t out[4], cudaStream_t st)
{
    if (limit_ns < 1000 || limit_ns > 100000000ll) return ISC_ERR_ARG;          // 1 us .. 100 ms
    int32_t *d_out = reinterpret_cast<int32_t *>(p->d_dump);                   // the debug read-back buffer
    k_wait_probe<<<1, 32, kCtrlBytes, st>>>(p->d_err, (unsigned long long)limit_ns, d_out);
    if (cudaGetLastError() != cudaSuccess) return ISC_ERR_CUDA;
    if (cudaMemcpyAsync(out, d_out, 4 * sizeof(int32_t), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess) { cudaGetLastError(); return ISC_ERR_CUDA; }
    return line_check(p);
}

int line_phase_cycles(LinePlan *p, unsigned long long out[4])
{
    if (cudaMemcpy(out, p->d_phase_cycles, 4 * sizeof(unsigned long long), cudaMemcpyDeviceToHost) != cudaSuccess) {
        cudaGetLastError();
        return ISC_ERR_CUDA;
    }
    return ISC_OK;
}

// Runs one group (samples ns.first_sample ..) up to the phase that produces `tensor` and returns that
// tensor of the first sample as [C][H][W] int32.
int line_debug_tensor(LinePlan *p, const uint8_t *d_x, const NoiseStream &ns, int tensor, int32_t *out_chw,
                      int32_t *d_counts_scratch, cudaStream_t st, int64_t *launches)
{
    if (tensor < 0 || tensor >= (int)p->tensors.size() || p->tensors[(size_t)tensor].buffer < 0) return ISC_ERR_UNSUPPORTED;
    const LGeo &t = p->tensors[(size_t)tensor];
    LineParams q = p->base;
    q.x = d_x; q.ns = ns; q.counts = d_counts_scratch; q.logits = nullptr;
    q.image_id0 = (unsigned long long)ns.ctr2 | (unsigned long long)(ns.ctr3_fixed >> 16) << 32;
    q.ns.ctr3_fixed &= 0xFFu;
    q.n_sel = 0; q.groups_sel = 0; q.n_est = 1; q.groups_est = 1; q.n_groups = 1;
    q.stop_phase = t.producer_phase;
    q.dump_off = p->tensor_off[(size_t)tensor]; q.dump_bytes = t.bytes; q.dump = p->d_dump;
    int rc = line_launch(p, q, st);
    *launches += 1;
    if (rc) return rc;
    std::vector<uint8_t> h(t.bytes);
    if (cudaMemcpyAsync(h.data(), p->d_dump, t.bytes, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess) { cudaGetLastError(); return ISC_ERR_CUDA; }
    if ((rc = line_check(p))) return rc;
    for (int c = 0; c < t.C; ++c)
        for (int y = 0; y < t.H; ++y)
            for (int x = 0; x < t.W; ++x) {
                const int line = y % t.n_lines, band = y / t.n_lines;
                const size_t at = (size_t)(c / 16) * t.plane_bytes + t.line0 +
                                  ((size_t)line * t.pitch + (size_t)x * t.I + (size_t)band * 4) * 16 + (size_t)(c % 16);
                const uint8_t b = h[at];
                out_chw[((size_t)c * t.H + y) * t.W + x] = tensor == 0 ? (int32_t)b : (int32_t)(int8_t)b;
            }
    return ISC_OK;
}


}  // namespace isc
