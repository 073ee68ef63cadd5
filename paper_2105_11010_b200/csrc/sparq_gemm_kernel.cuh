// Fused SPARQ GEMM / implicit-GEMM convolution for sm_100a.
//
//   acc[m][j] = sum_k T(A)[m][k] * B[j][k]      (Eq. 1 with Eq. 2 applied on the fly)
//
// One persistent CTA per SM walks output tiles of 128 x BN.  Warp roles:
//   warp 0        TMA producer: A tile (tiled 2-D box for the GEMM, im2col box for the
//                 convolution) and B tile into a ring of shared-memory stages; without a transform,
//                 and with ATM, warp 18 fetches B
//   warp 1        allocates tensor memory; one lane issues tcgen05.mma kind::i8
//                 (u8 x s8 -> s32) on each transformed stage
//   warps 2..9    epilogue: tcgen05.ld of a finished accumulator, fp32 scale / bias /
//                 ReLU / requantize, global stores (warp w reads lane quarter w % 4 of its team's
//                 tiles, and its share of their columns)
//   warps 10..17  transform: rewrite the A stage in place with bSPARQ / vSPARQ (or, ATM, into tensor memory)
//
// A stage travels  TMA (async proxy) -> transform warps (generic proxy) -> MMA (async
// proxy); the hand-offs are mbarriers, with fence.proxy.async after the in-place rewrite.
// The 128-byte (64-byte) shared-memory swizzle only permutes 16-byte chunks inside a
// row, and a vSPARQ pair never straddles a 16-byte chunk, so the transform treats the
// stage as a flat array of 16-byte vectors.
//
// Every wait is bounded: when a wait gives up it sets bit 0 of the status word, raises a
// CTA-wide abort flag that makes all later waits return at once, and the kernel still
// runs to its normal end (loops have fixed trip counts), drains its own copies and frees
// its tensor memory.
#pragma once

#include <cuda.h>

#include "sparq_common.cuh"

namespace sparq {

constexpr int kBM = 128;                 // rows of an output tile = MMA M
constexpr int kNumEpiWarps = 8;          // two per tensor-memory lane quarter; without a transform
                                         // (mode NONE) the transform warps are epilogue warps too
constexpr int kNumXfWarps = 8;
// The transform warps work as two teams that take stages (or window pieces) alternately: a
// stage's chain of barrier read, shared-memory loads, arithmetic, stores and fence is mostly
// latency, and one team's chain overlaps the other's.
constexpr int kXfTeams = 2;
constexpr int kXfTeamWarps = kNumXfWarps / kXfTeams;
constexpr int kFirstEpiWarp = 2;
constexpr int kFirstXfWarp = kFirstEpiWarp + kNumEpiWarps;
// Without a transform sparq_gemm_kernel's last warp is a second producer: one thread's chain -- wait,
// announce, two copies -- was the longest of a step where steps are short (batch 64, 7x7x512 -> 512
// 3x3 transformed first 16.5 -> 14.4 us, 56x56x128 -> 128 3x3 stride 2 without a transform 12.8 -> 10.9).
// With a transform a step is longer, and one producer as fast or faster (200704 x 64, K 256, 17.55 us against 17.75).
constexpr int kWeightWarp = kFirstXfWarp + kNumXfWarps;
__host__ __device__ constexpr int gemm_threads(int mode, bool in_tmem) { return 32 * (kWeightWarp + (mode == SPARQ_MODE_NONE || in_tmem ? 1 : 0)); }
// Epilogue warps of a kernel instantiated for `mode`.
__host__ __device__ constexpr int epi_warps(int mode) { return mode == SPARQ_MODE_NONE ? kNumEpiWarps + kNumXfWarps : kNumEpiWarps; }
// Shares that a tile's columns are split into over the groups of one epilogue team.
__host__ __device__ constexpr int epi_parts(int groups, int teams, int bn) { return groups / teams < bn / 32 ? groups / teams : bn / 32; }
constexpr int kMaxStages = 8;
constexpr int kMaxDynSmemGemm = 232448 - 6144;   // 227 KB minus room for the static variables
constexpr int kSmemBudget = 200 * 1024;  // for the stage ring
// Default limit of every device-side wait, in SM clock cycles (about a second).  The limit is a
// kernel argument, so that a diagnostic launch can make a wait run out in microseconds.
constexpr long long kWaitLimitCycles = 2000000000LL;

struct GemmArgs {
    // problem
    int64_t M, N, K;        // GEMM view (K = r*s*c for the convolution)
    int k_blocks;           // number of BK-wide reduction steps
    // convolution geometry (conv = 1) for the im2col producer
    int conv;
    int c_blocks;           // BK-wide channel blocks per filter tap (the last one may reach past C: zero fill)
    int tap_k;              // bytes of a filter row per tap (= C)
    int S;                  // filter width (taps are ordered r-major, s-minor)
    int Ho, Wo;
    int stride_h, stride_w, pad_h, pad_w;
    // transform
    XformDev xf;
    // epilogue
    const float *scale;
    const float *bias;
    int relu;
    float inv_out_scale;
    int32_t *acc_out;
    float *f32_out;
    uint8_t *u8_out;
    unsigned int *status;
    long long wait_limit;   // cycles after which a device-side wait gives up
    // producer-side transform of u8_out (mode NONE = off)
    int next_mode, next_rnd;
    XformDev next_xf;
    // residual input of the epilogue (nullptr = none)
    const uint8_t *residual;
    float residual_scale;
    int stages;             // of the operand ring
    // staged output: bytes per row of the boxes that the epilogue warps store (and fetch the residual)
    // with through shared memory, 0 = straight from registers.  See epi_staged.
    int out_box;
    // small form only: rows of a tile; CTAs of a cluster that share a tile (1 = none)
    int tile_rows, split;
};

// ---- PTX wrappers ---------------------------------------------------------------------

__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(bar), "r"(count));
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(bar) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}

// Non-blocking look at a phase: 1 if it has completed.  Unlike try_wait this never suspends
// the thread, and nothing waits for its result until the value is used.
__device__ __forceinline__ uint32_t mbar_test(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok;
}

// Three looks at once (bit i: barrier i): all reads are in flight together before any answer
// is consumed.
__device__ __forceinline__ uint32_t mbar_test3(uint32_t bar0, uint32_t parity0, uint32_t bar1, uint32_t parity1,
                                               uint32_t bar2, uint32_t parity2)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p, q, r;\n\t.reg .u32 a, b, c;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 q, [%3], %4;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 r, [%5], %6;\n\t"
        "selp.u32 a, 1, 0, p;\n\t"
        "selp.u32 b, 2, 0, q;\n\t"
        "selp.u32 c, 4, 0, r;\n\t"
        "or.b32 a, a, b;\n\t"
        "or.b32 %0, a, c;\n\t}"
        : "=r"(ok) : "r"(bar0), "r"(parity0), "r"(bar1), "r"(parity1), "r"(bar2), "r"(parity2) : "memory");
    return ok;
}

// Bounded wait.  Returns false (after flagging) if the phase did not complete in time or
// if another thread of the CTA already gave up.
//
// EARLY: for a role that touches on-chip memory only and so does not wait for the kernel before, on the barriers of the
// operands that it starts with.  That kernel may release this one early and then take long, which must not count
// against the limit: the first expiry waits for it (at once if it has finished) and starts the clock again.
// (Every role waiting for it in front of its first barrier instead: 32x56x56x64 -> 64 3x3 8.44 -> 8.63 us, the
// ResNet-50 pass at batch 64 744 -> 755; every wait EARLY: 256 x 64 x 576 5.42 -> 5.54.)
template <bool EARLY = false>
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile uint32_t *abort_flag,
                                          unsigned int *status, long long limit_cycles, bool ignore_abort = false)
{
    if (mbar_try_wait(bar, parity)) return true;
    if (!ignore_abort && *abort_flag) return false;
    long long t0 = clock64();
    bool alone = !EARLY;            // the kernel before has finished
    for (uint32_t it = 1;; ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((it & 0x3Fu) == 0) {
            if (!ignore_abort && *abort_flag) return false;
            if (clock64() - t0 > limit_cycles) {
                if (!alone) {
                    dep_wait();
                    alone = true;
                    t0 = clock64();
                    continue;
                }
                *abort_flag = 1u;
                atomicOr(status, 1u);
                return false;
            }
        }
    }
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, uint32_t bar, int x, int y)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
        :: "r"(dst), "l"(map), "r"(bar), "r"(x), "r"(y) : "memory");
}

// Groups of 32 weight rows from row n0 (a multiple of 32), in the order that the map says (natural, or
// that of epi_frag: one instruction for both, the loop that issues it has no time for a decision).
__device__ __forceinline__ void tma_load_row_groups(uint32_t dst, const CUtensorMap *map, uint32_t bar, int k, int n0)
{
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %4, %4, %5}], [%2];"
        :: "r"(dst), "l"(map), "r"(bar), "r"(k), "r"(0), "r"(n0 >> 5) : "memory");
}

// im2col box: `pixels-per-column` output pixels starting at base pixel (w, h, n), channels
// c .. c+box, filter tap offset (woff, hoff); out-of-image taps are filled with zeros.
__device__ __forceinline__ void tma_load_im2col_4d(uint32_t dst, const CUtensorMap *map, uint32_t bar,
                                                   int c, int w, int h, int n, uint16_t woff, uint16_t hoff)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.im2col.mbarrier::complete_tx::bytes "
        "[%0], [%1, {%3, %4, %5, %6}], [%2], {%7, %8};"
        :: "r"(dst), "l"(map), "r"(bar), "r"(c), "r"(w), "r"(h), "r"(n), "h"(woff), "h"(hoff) : "memory");
}

// A box of shared memory into global memory (what lies outside the tensor is clipped); stores of a
// thread form one group per tma_store_commit, and tma_store_wait_read<N> returns once all but
// the last N groups have been read out of shared memory.
__device__ __forceinline__ void tma_store_2d(const CUtensorMap *map, uint32_t src, int x, int y)
{
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%2, %3}], [%1];"
                 :: "l"(map), "r"(src), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void tma_store_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void tma_store_wait_read() { asm volatile("cp.async.bulk.wait_group.read %0;" :: "n"(N) : "memory"); }
__device__ __forceinline__ void tma_store_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

__device__ __forceinline__ void prefetch_tensormap(const CUtensorMap *map)
{
    asm volatile("prefetch.tensormap [%0];" :: "l"(map) : "memory");
}

__device__ __forceinline__ void fence_proxy_async_smem()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// D[tmem] (+)= A[smem] * B[smem], 128 x N x 32, u8 x s8 -> s32, and the commit that signals a barrier once the
// MMAs before it have retired, for a warp that runs its loop converged: every lane executes
// the surrounding code (so that descriptor arithmetic on warp-uniform values can stay in
// the uniform datapath) and only the lane with `elected` != 0 issues.
__device__ __forceinline__ void tc_mma_i8_if(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                             uint32_t accumulate, uint32_t elected)
{
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "setp.ne.b32 q, %5, 0;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n\t}"
        :: "r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(elected) : "memory");
}

// The same with A in tensor memory (row i in lane i, four bytes of K per column).
__device__ __forceinline__ void tc_mma_i8_tmem_if(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc,
                                                  uint32_t accumulate, uint32_t elected)
{
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "setp.ne.b32 q, %5, 0;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::i8 [%0], [%1], %2, %3, p;\n\t}"
        :: "r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(elected) : "memory");
}

__device__ __forceinline__ void tc_commit_if(uint32_t bar, uint32_t elected)
{
    asm volatile(
        "{\n\t.reg .pred q;\n\t"
        "setp.ne.b32 q, %1, 0;\n\t"
        "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}"
        :: "r"(bar), "r"(elected) : "memory");
}

// One lane of a converged warp (the same lane every time it is asked within a launch is not
// guaranteed; callers ask once and keep the answer).
__device__ __forceinline__ uint32_t elect_one()
{
    uint32_t e;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(e));
    return e;
}

// Shared-memory matrix descriptor of a K-major tile whose rows are ROW_BYTES long
// (128 or 64) and swizzled with the matching TMA mode; 8-row groups are contiguous.
template <int ROW_BYTES>
__device__ __forceinline__ uint64_t make_smem_desc(uint32_t saddr)
{
    constexpr uint64_t layout = (ROW_BYTES == 128) ? 2ull : 4ull;   // 128B / 64B swizzle
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);            // start address
    d |= (uint64_t)1 << 16;                              // leading-dimension offset (unused when swizzled)
    d |= (uint64_t)((8 * ROW_BYTES) >> 4) << 32;         // stride between 8-row groups
    d |= (uint64_t)1 << 46;                              // descriptor version of this architecture
    d |= layout << 61;
    return d;
}

// kind::i8 instruction descriptor: s32 accumulator, unsigned A, signed B, both K-major.
__device__ __forceinline__ constexpr uint32_t make_idesc_i8(int n, int m = kBM)
{
    return (2u << 4) | (0u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

// 16 words of each lane's row into 16 columns.
__device__ __forceinline__ void tmem_st_32x16(uint32_t taddr, const uint4 (&v)[4])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
                 :: "r"(taddr), "r"(v[0].x), "r"(v[0].y), "r"(v[0].z), "r"(v[0].w), "r"(v[1].x), "r"(v[1].y), "r"(v[1].z), "r"(v[1].w),
                    "r"(v[2].x), "r"(v[2].y), "r"(v[2].z), "r"(v[2].w), "r"(v[3].x), "r"(v[3].y), "r"(v[3].z), "r"(v[3].w) : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// 32 contiguous bytes with one 256-bit store (dst 32-byte aligned).
__device__ __forceinline__ void st_global_v8(void *dst, const uint32_t (&w)[8])
{
    asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
                 :: "l"(dst), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
                 : "memory");
}

__device__ __forceinline__ void tmem_ld_32x32_issue(uint32_t taddr, uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr) : "memory");
}

// 32 rows x 32 columns of an accumulator as matrix fragments: lane l gets, of each group j of eight
// columns, columns 2 (l % 4) and + 1 of rows l / 4 (r[4j], r[4j + 1]), + 8 (r[4j + 2], r[4j + 3]) and, 16
// places on in r, + 16 and + 24.
__device__ __forceinline__ void tmem_ld_frag_issue(uint32_t taddr, uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x4.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr) : "memory");
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x4.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr + (16u << 16)) : "memory");
}

// Reduction steps of a convolution in order, from step `first`: filter tap (r, s), channel block
// starting at c, and the block's first byte k of a filter.
struct TapWalk {
    int c, r, s, k, tap_k, bk, S;
    __device__ __forceinline__ TapWalk(const GemmArgs &g, int bk_, int first)
    {
        tap_k = g.conv ? g.tap_k : 0x7FFFFFFF;      // a matrix: k only
        bk = bk_; S = g.S;
        c = r = s = k = 0;
        if (g.conv && first) {
            const int tap = first / g.c_blocks;
            c = (first - tap * g.c_blocks) * bk;
            r = tap / S;
            s = tap - r * S;
            k = tap * tap_k + c;
        }
    }
    __device__ __forceinline__ void next()
    {
        c += bk;
        k += bk;
        if (c >= tap_k) {
            k += tap_k - c;
            c = 0;
            if (++s == S) { s = 0; ++r; }
        }
    }
};

// ---- epilogue arithmetic ----------------------------------------------------------------

// Four fp32 values on the output grid -> four bytes clamp(rint(z), 0, 255) in one word, z0 in
// the low byte: a round-to-nearest-even conversion to int32 each (NaN gives 0, the infinities
// the int32 limits), then two instructions that saturate two integers to bytes and pack them
// beside the bytes already there.  Clamping and rounding with fp32 instructions (max, min, add
// of 1.5 * 2^23) and permuting the bytes together took eleven issue slots where this takes six.
__device__ __forceinline__ uint32_t requant_pack4(float z0, float z1, float z2, float z3)
{
    uint32_t hi, w;
    asm("cvt.pack.sat.u8.s32.b32 %0, %1, %2, %3;" : "=r"(hi) : "r"(__float2int_rn(z3)), "r"(__float2int_rn(z2)), "r"(0));
    asm("cvt.pack.sat.u8.s32.b32 %0, %1, %2, %3;" : "=r"(w) : "r"(__float2int_rn(z1)), "r"(__float2int_rn(z0)), "r"(hi));
    return w;
}

// The next layer's transform of one word, inline: one run-time form for every width, set and rounding.
__device__ __forceinline__ uint32_t next_xform_word(uint32_t x, int mode, int rnd, const XformDev &xf)
{
    const uint32_t m = drop_mask<0, true>(x, xf.n, xf.widen_c);
    const uint32_t q = rnd ? apply_mask<true>(x, m, xf.n) : apply_mask<false>(x, m, xf.n);
    if (mode != SPARQ_MODE_VSPARQ) return q;
    uint32_t lone = x;
    if (xf.n < 4) {
        const uint32_t ml = drop_mask<0, false>(x, 2 * xf.n, 0u);
        lone = rnd ? apply_mask<true>(x, ml, 2 * xf.n) : apply_mask<false>(x, ml, 2 * xf.n);
    }
    const uint32_t nz = ((x & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | x;
    const uint32_t partner_nz = prmt(nz, nz, 0xAB89u);
    return (q & partner_nz) | (lone & ~partner_nz);
}

// The next layer's transform on requantized bytes (producer-side SPARQ): four adjacent output
// channels per word, pairs (2j, 2j+1) inside it.  Kept out of line: the epilogue loops are hot
// and every variant inlined at every use made the kernels several times larger than the
// instruction caches, which the warp roles share.
// (Words by value: through a pointer they went to local memory and back, 4-14 % of such a layer.)
struct Words8 {
    uint32_t w[8];
};
static __device__ __noinline__ Words8 next_xform_words(Words8 v, int mode, int rnd, XformDev xf)
{
    auto each = [&](auto f) {
#pragma unroll
        for (int q = 0; q < 8; ++q) v.w[q] = f(v.w[q]);
    };
    if (mode == SPARQ_MODE_VSPARQ) {
        // full sets: the half-precision form
        if (xf.rounds == 0 && xf.n != 4) each([&](uint32_t x) { return xform_word_fullset<SPARQ_MODE_VSPARQ, false, true>(x, xf); });
        else if (xf.rounds == 0 && rnd) each([&](uint32_t x) { return xform_word_fullset<SPARQ_MODE_VSPARQ, true, true>(x, xf); });
        else each([&](uint32_t x) { return next_xform_word(x, mode, rnd, xf); });
    } else {
        each([&](uint32_t x) { return next_xform_word(x, mode, rnd, xf); });
    }
    return v;
}

// Per-thread view of the epilogue's outputs and constants.
struct EpiView {
    int64_t N;
    int32_t *acc_out;
    float *f32_out;
    uint8_t *u8_out;
    float inv_out_scale;
    bool need_f;      // a dequantized output is requested
    bool relu_op;     // the ReLU select has to be executed (see below)
    int gran;         // bytes (columns) that one access to a u8 row may take: 32, 16, 8, 4 or 1, whichever divides N
    int out;          // EpiOut: which instantiation of a kernel the launch takes
    int next_mode;    // SPARQ mode applied to the requantized bytes (producer-side transform)
    int next_rnd;
    XformDev next_xf;
    const uint8_t *residual;   // u8 identity tensor added before the ReLU, or nullptr
    float residual_scale;
};

// The kernels are instantiated per kind of output: requantized bytes only, in whole groups of 32
// columns (epi_lean), the same with a residual, and everything else.  One kernel with all of them
// was slower on every layer: the warp roles share the instruction caches, every kernel starts with
// cold ones, and the code that a launch does not run still spreads the code it does over more
// lines (and takes registers: the largest role decides for all).  128x28x28x128 -> 128 3x3:
// 17.5 -> 16.9 us without the residual's code, 32x56x56x64 -> 64 10.75 -> 10.45.
enum EpiOut { kOutGeneral, kOutBytes, kOutResidual };

// Whether an epilogue of sparq_gemm_kernel works on matrix fragments (epi_frag), with the weight rows in fragment
// order: boxes staged in shared memory, and 256-wide tiles.  Straight to global memory from narrower ones the
// row form, a whole 32 bytes of a row per thread and store, is faster (200704 x 64, K 256, 17.5 us against
// 17.9, without a transform 10.7 against 11.9), and in the window kernel (128x28x28x128 -> 128 3x3
// 15.4 against 15.6, 256-wide tiles 35.6 against 36.4).
__host__ __device__ constexpr bool frag_rows(int out, int bn, int out_box) { return out != kOutGeneral && (bn == 256 || out_box); }

template <class Args>
__host__ __device__ __forceinline__ EpiView make_epi_view(const Args &g)
{
    EpiView e;
    e.N = g.N;
    e.acc_out = g.acc_out;
    e.f32_out = g.f32_out;
    e.u8_out = g.u8_out;
    e.inv_out_scale = g.inv_out_scale;
    e.need_f = (g.f32_out != nullptr) || (g.u8_out != nullptr);
    // relu(y) * inv clamped to [0, 255] equals y * inv clamped when inv > 0, so the ReLU
    // select is only needed when the fp32 value itself is an output
    e.relu_op = g.relu && (g.f32_out != nullptr || !(g.inv_out_scale > 0.0f));
    const bool aligned32 = ((reinterpret_cast<uintptr_t>(g.u8_out) | reinterpret_cast<uintptr_t>(g.f32_out) |
                             reinterpret_cast<uintptr_t>(g.acc_out) | reinterpret_cast<uintptr_t>(g.residual)) & 31u) == 0;
    e.gran = g.N % 32 == 0 && aligned32 ? 32 : g.N % 16 == 0 ? 16 : g.N % 8 == 0 ? 8 : g.N % 4 == 0 ? 4 : 1;
    // (the fragment form keeps offsets over a tile's rows in 32 bits)
    const bool bytes_only = e.u8_out && !g.acc_out && !g.f32_out && g.next_mode == SPARQ_MODE_NONE && !e.relu_op && e.gran == 32 && g.N < 1 << 24;
    e.out = !bytes_only ? kOutGeneral : g.residual ? kOutResidual : kOutBytes;
    e.next_mode = g.next_mode;
    e.next_rnd = g.next_rnd;
    e.next_xf = g.next_xf;
    e.residual = g.residual;
    e.residual_scale = g.residual_scale;
    return e;
}

// Two fp32 values in one 64-bit register and the packed arithmetic of sm_100: each instruction
// performs the IEEE round-to-nearest operation on both halves, so a pair of columns costs one
// issue slot where the scalar form costs two.
__device__ __forceinline__ uint64_t f2_pack(float lo, float hi)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void f2_unpack(uint64_t r, float &lo, float &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(r));
}
__device__ __forceinline__ uint64_t f2_add(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t f2_mul(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t f2_fma(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

// 32 contiguous bytes (src 32-byte aligned) through the read-only path.
__device__ __forceinline__ void ld_global_v8(const void *src, uint32_t (&w)[8])
{
    asm volatile("ld.global.nc.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7])
                 : "l"(src));
}

// Bytes 2H and 2H + 1 of w as two fp32 values: 2^23 + byte as a bit pattern (one permute), minus
// 2^23, both exact.
template <int H>
__device__ __forceinline__ uint64_t bytes_to_f2(uint32_t w)
{
    const uint32_t a = prmt(w, 0x4B000000u, 0x7440u + (2 * H)), b = prmt(w, 0x4B000000u, 0x7440u + (2 * H + 1));
    return f2_add(f2_pack(__uint_as_float(a), __uint_as_float(b)), f2_pack(-8388608.0f, -8388608.0f));
}

// The form every layer of a network uses -- requantized bytes only, whole groups of 32 columns --
// as straight-line code with nothing decided per element and the fp32 steps done two columns at
// a time: per accumulator one int -> float conversion, one fma, (with a residual one more fma,) one
// multiply and the conversion back to an integer, then two saturating packs per four columns.
// Same IEEE sequence per element as epi_general.  (The int -> float conversion beats the add-based
// form for small accumulators: 46.6 against 42.7 outputs per clock and SM, arithmetic alone.)
// res: the 32 columns' residual bytes.
template <bool RES>
__device__ __forceinline__ void epi_lean(const uint32_t (&v)[32], const float *s_scale, const float *s_bias, float inv, float res_scale,
                                         const uint32_t (&res)[8], uint32_t (&w)[8])
{
    const uint64_t inv2 = f2_pack(inv, inv), rs2 = f2_pack(res_scale, res_scale);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const float4 sc = *reinterpret_cast<const float4 *>(&s_scale[4 * q]);
        const float4 bi = *reinterpret_cast<const float4 *>(&s_bias[4 * q]);
        float z[4];
        uint64_t y0 = f2_fma(f2_pack(__int2float_rn((int)v[4 * q]), __int2float_rn((int)v[4 * q + 1])), f2_pack(sc.x, sc.y), f2_pack(bi.x, bi.y));
        uint64_t y1 = f2_fma(f2_pack(__int2float_rn((int)v[4 * q + 2]), __int2float_rn((int)v[4 * q + 3])), f2_pack(sc.z, sc.w), f2_pack(bi.z, bi.w));
        if (RES) {
            y0 = f2_fma(bytes_to_f2<0>(res[q]), rs2, y0);
            y1 = f2_fma(bytes_to_f2<1>(res[q]), rs2, y1);
        }
        f2_unpack(f2_mul(y0, inv2), z[0], z[1]);
        f2_unpack(f2_mul(y1, inv2), z[2], z[3]);
        w[q] = requant_pack4(z[0], z[1], z[2], z[3]);
    }
}

// The same on matrix fragments (tmem_ld_frag_issue): a thread has four rows of eight columns, so that a
// column's scale and bias are read once for four outputs, four 16-byte reads per 32 x 32 outputs where
// a thread per row takes sixteen.  Those reads are broadcasts, but of more than one wavefront each, and shared
// memory is what the epilogue shares with the tensor core's operands: 200704 x 256, K 64, 1600 -> 1370 wavefronts of
// the load / store pipe a tile (425 of them now bank conflicts of the staged boxes).  16384 x 4096, K 512, 42.6 -> 38.7 us,
// 50176 x 256, K 512, without a transform 9.95 -> 9.0, the ResNet-50 pass at batch 64 829 -> 799.
// The eight columns are adjacent outputs because the weight rows lie in shared memory in fragment order:
// row 8j + 2q + b of each group of 32 holds weight row 8q + 2j + b (a five-dimensional tensor map, no
// extra copy), so accumulator columns 2q, 2q + 1 of the groups j = 0..3 are output columns 8q .. 8q + 7.
// scale, bias: of this thread's eight columns.  res, w: bytes of row r in words 2r, 2r + 1.
template <bool RES>
__device__ __forceinline__ void epi_frag(const uint32_t (&v)[32], const float *scale, const float *bias, float inv, float res_scale,
                                         const uint32_t (&res)[8], uint32_t (&w)[8])
{
    const uint64_t inv2 = f2_pack(inv, inv), rs2 = f2_pack(res_scale, res_scale);
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        const float4 sc = *reinterpret_cast<const float4 *>(&scale[4 * p]);
        const float4 bi = *reinterpret_cast<const float4 *>(&bias[4 * p]);
        const uint64_t s0 = f2_pack(sc.x, sc.y), s1 = f2_pack(sc.z, sc.w), b0 = f2_pack(bi.x, bi.y), b1 = f2_pack(bi.z, bi.w);
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int i = 16 * (r >> 1) + 8 * p + 2 * (r & 1);
            uint64_t y0 = f2_fma(f2_pack(__int2float_rn((int)v[i]), __int2float_rn((int)v[i + 1])), s0, b0);
            uint64_t y1 = f2_fma(f2_pack(__int2float_rn((int)v[i + 4]), __int2float_rn((int)v[i + 5])), s1, b1);
            if (RES) {
                y0 = f2_fma(bytes_to_f2<0>(res[2 * r + p]), rs2, y0);
                y1 = f2_fma(bytes_to_f2<1>(res[2 * r + p]), rs2, y1);
            }
            float z[4];
            f2_unpack(f2_mul(y0, inv2), z[0], z[1]);
            f2_unpack(f2_mul(y1, inv2), z[2], z[3]);
            w[2 * r + p] = requant_pack4(z[0], z[1], z[2], z[3]);
        }
    }
}

// The first `cols` of 32 bytes / words at any byte / word address: aligned words / 16-byte pieces put
// together from their neighbours, and single bytes / words at the ends.  (A thread owns a row, so
// every store of a warp falls into 32 lines: their number is what such an epilogue takes.  Row
// lengths that are no multiple of 4 only: 16384 x 1021, K 512, 171 -> 44 us.)
__device__ __forceinline__ void store_bytes_unaligned(uint8_t *dst, const uint32_t (&w)[8], int cols)
{
    const int head = (int)(-reinterpret_cast<uintptr_t>(dst) & 3u), sh = 8 * head;
    const int words = cols > head ? (cols - head) >> 2 : 0, done = head + 4 * words;
#pragma unroll
    for (int i = 0; i < 3; ++i)
        if (i < head && i < cols) dst[i] = (uint8_t)(w[0] >> (8 * i));
#pragma unroll
    for (int q = 0; q < 8; ++q)
        if (q < words) *reinterpret_cast<uint32_t *>(dst + head + 4 * q) = __funnelshift_r(w[q], q < 7 ? w[q + 1] : 0u, sh);
#pragma unroll
    for (int i = 0; i < 32; ++i)
        if ((cols != 32 || i >= 28) && i >= done && i < cols) dst[i] = (uint8_t)(w[i >> 2] >> (8 * (i & 3)));
}
__device__ __forceinline__ void store_words_unaligned(uint32_t *dst, const uint32_t (&v)[32], int cols)
{
    const int head = (int)(-(reinterpret_cast<uintptr_t>(dst) >> 2) & 3u);
    const int quads = cols > head ? (cols - head) >> 2 : 0, done = head + 4 * quads;
    auto at = [&](int i) {      // v[i + head]
        const uint32_t a = head & 1 ? v[i + 1 < 32 ? i + 1 : 31] : v[i], b = head & 1 ? v[i + 3 < 32 ? i + 3 : 31] : v[i + 2 < 32 ? i + 2 : 31];
        return head & 2 ? b : a;
    };
#pragma unroll
    for (int i = 0; i < 3; ++i)
        if (i < head && i < cols) dst[i] = v[i];
#pragma unroll
    for (int q = 0; q < 8; ++q)
        if (q < quads) *reinterpret_cast<uint4 *>(dst + head + 4 * q) = make_uint4(at(4 * q), at(4 * q + 1), at(4 * q + 2), at(4 * q + 3));
#pragma unroll
    for (int i = 0; i < 32; ++i)
        if ((cols != 32 || i >= 28) && i >= done && i < cols) dst[i] = v[i];
}

// The first `cols` of 32 bytes, in accesses of `gran` >= 4 bytes (a divisor of the row length).
__device__ __forceinline__ void store_bytes32(uint8_t *dst, const uint32_t (&w)[8], int cols, int gran)
{
    if (gran == 32) {
        st_global_v8(dst, w);
    } else if (gran == 16) {
#pragma unroll
        for (int i = 0; i < 2; ++i)
            if (16 * i < cols) reinterpret_cast<uint4 *>(dst)[i] = make_uint4(w[4 * i], w[4 * i + 1], w[4 * i + 2], w[4 * i + 3]);
    } else if (gran == 8) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (8 * i < cols) reinterpret_cast<uint2 *>(dst)[i] = make_uint2(w[2 * i], w[2 * i + 1]);
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (4 * i < cols) reinterpret_cast<uint32_t *>(dst)[i] = w[i];
    }
}

__device__ __forceinline__ void load_bytes32(const uint8_t *src, uint32_t (&w)[8], int cols, int gran)
{
#pragma unroll
    for (int i = 0; i < 8; ++i) w[i] = 0u;
    if (gran >= 16) {
#pragma unroll
        for (int i = 0; i < 2; ++i)
            if (16 * i < cols) {
                const uint4 r = __ldg(reinterpret_cast<const uint4 *>(src) + i);
                w[4 * i] = r.x; w[4 * i + 1] = r.y; w[4 * i + 2] = r.z; w[4 * i + 3] = r.w;
            }
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (4 * i < cols) w[i] = __ldg(reinterpret_cast<const uint32_t *>(src) + i);
    }
}

// 32 accumulators of one output row (columns col0 .. col0 + 31) with any combination of outputs and
// any N (ODD: N is no multiple of 4): optional raw store, dequantize, optional fp32 store, requantize
// and store.  v is overwritten.
template <bool ODD>
__device__ __forceinline__ void epi_general(const EpiView &e, uint32_t (&v)[32], int64_t row, int64_t col0,
                                            const float *s_scale, const float *s_bias)
{
    const int64_t off = row * e.N + col0;
    const int cols = (int)(e.N - col0 < 32 ? e.N - col0 : 32);
    auto store32 = [&](void *base) {       // 32 words
        uint32_t *dst = reinterpret_cast<uint32_t *>(base) + off;
        if (ODD) {
            store_words_unaligned(dst, v, cols);
        } else if (e.gran == 32) {
#pragma unroll
            for (int q = 0; q < 4; ++q) st_global_v8(dst + 8 * q, reinterpret_cast<const uint32_t(&)[8]>(v[8 * q]));
        } else {
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (4 * q < cols) reinterpret_cast<uint4 *>(dst)[q] = make_uint4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
        }
    };
    if (e.acc_out) store32(e.acc_out);
    if (!e.need_f) return;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const float4 sc = *reinterpret_cast<const float4 *>(&s_scale[4 * q]);
        const float4 bi = *reinterpret_cast<const float4 *>(&s_bias[4 * q]);
        float y[4];
        f2_unpack(f2_fma(f2_pack(__int2float_rn((int)v[4 * q]), __int2float_rn((int)v[4 * q + 1])), f2_pack(sc.x, sc.y), f2_pack(bi.x, bi.y)), y[0], y[1]);
        f2_unpack(f2_fma(f2_pack(__int2float_rn((int)v[4 * q + 2]), __int2float_rn((int)v[4 * q + 3])), f2_pack(sc.z, sc.w), f2_pack(bi.z, bi.w)), y[2], y[3]);
#pragma unroll
        for (int i = 0; i < 4; ++i) v[4 * q + i] = __float_as_uint(y[i]);
    }
    if (e.residual) {
        uint32_t r[8];
        if (ODD) {
#pragma unroll
            for (int i = 0; i < 8; ++i) r[i] = 0u;
#pragma unroll
            for (int i = 0; i < 32; ++i)
                if (i < cols) r[i >> 2] |= (uint32_t)__ldg(e.residual + off + i) << (8 * (i & 3));
        } else {
            load_bytes32(e.residual + off, r, cols, e.gran);
        }
        const uint64_t rs2 = f2_pack(e.residual_scale, e.residual_scale);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            float y[4];
            f2_unpack(f2_fma(bytes_to_f2<0>(r[q]), rs2, f2_pack(__uint_as_float(v[4 * q]), __uint_as_float(v[4 * q + 1]))), y[0], y[1]);
            f2_unpack(f2_fma(bytes_to_f2<1>(r[q]), rs2, f2_pack(__uint_as_float(v[4 * q + 2]), __uint_as_float(v[4 * q + 3]))), y[2], y[3]);
#pragma unroll
            for (int i = 0; i < 4; ++i) v[4 * q + i] = __float_as_uint(y[i]);
        }
    }
    if (e.relu_op) {
#pragma unroll
        for (int i = 0; i < 32; ++i) v[i] = __float_as_uint(fmaxf(__uint_as_float(v[i]), 0.0f));    // NaN -> 0, like (y > 0 ? y : 0)
    }
    if (e.f32_out) store32(e.f32_out);
    if (e.u8_out) {
        uint32_t w[8];
        const uint64_t inv2 = f2_pack(e.inv_out_scale, e.inv_out_scale);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            float z[4];
            f2_unpack(f2_mul(f2_pack(__uint_as_float(v[4 * q]), __uint_as_float(v[4 * q + 1])), inv2), z[0], z[1]);
            f2_unpack(f2_mul(f2_pack(__uint_as_float(v[4 * q + 2]), __uint_as_float(v[4 * q + 3])), inv2), z[2], z[3]);
            w[q] = requant_pack4(z[0], z[1], z[2], z[3]);
        }
        if (e.next_mode != SPARQ_MODE_NONE) {
            Words8 t;
#pragma unroll
            for (int q = 0; q < 8; ++q) t.w[q] = w[q];
            t = next_xform_words(t, e.next_mode, e.next_rnd, e.next_xf);
#pragma unroll
            for (int q = 0; q < 8; ++q) w[q] = t.w[q];
        }
        if (ODD) store_bytes_unaligned(e.u8_out + off, w, cols);
        else store_bytes32(e.u8_out + off, w, cols, e.gran);
    }
}

// A warp's share of one accumulator: `cols` columns (a multiple of 32) starting at tensor-memory
// address taddr0 (tile-local column cbase), for this thread's output row.  wait_full() blocks
// until the accumulator is complete; when its last columns are in registers the warp hands it
// back by arriving on acc_empty_bar.
//
// 32 columns at a time: the arithmetic alone runs at 46 outputs per clock and SM, so what an
// epilogue takes is latency -- the accumulator's barrier, tensor memory, shared memory behind the
// tensor core's operand fetches -- and long straight-line groups hide most of it.  (Groups of 16 with
// the next one's tensor-memory load in flight measured 20 % slower: every group starts with its
// own exposed scale / bias reads.)  The residual bytes are fetched a group ahead, the first ones
// before the accumulator is waited for.
enum EpiKind { kEpiGeneral, kEpiGeneralOdd, kEpiLean, kEpiLeanResidual };

template <int KIND, class WaitFull>
__device__ __forceinline__ void epi_warp_columns_as(const EpiView &e, uint32_t taddr0, int cbase, int cols, int64_t row, bool row_ok,
                                                    int64_t n0, const float *s_scale, const float *s_bias,
                                                    uint32_t acc_empty_bar, int lane, WaitFull wait_full)
{
    uint32_t rn[8];
    auto fetch_residual = [&](int ct) {       // columns ct .. ct + 31 of the tile
        if (row_ok && n0 + ct < e.N) ld_global_v8(e.residual + row * e.N + n0 + ct, rn);
    };
    if (KIND == kEpiLeanResidual) {
#pragma unroll
        for (int i = 0; i < 8; ++i) rn[i] = 0u;
        fetch_residual(cbase);
    }
    wait_full();
#pragma unroll 1
    for (int c = 0; c < cols; c += 32) {
        uint32_t v[32], r[8];
        tmem_ld_32x32_issue(taddr0 + (uint32_t)c, v);
        if (KIND == kEpiLeanResidual) {
#pragma unroll
            for (int i = 0; i < 8; ++i) r[i] = rn[i];
            if (c + 32 < cols) fetch_residual(cbase + c + 32);
        }
        tmem_ld_wait();
        if (c + 32 == cols) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acc_empty_bar);
        }
        const int ct = cbase + c;                    // column inside the tile
        const int64_t col0 = n0 + ct;
        if (!row_ok || col0 >= e.N) continue;
        if (KIND == kEpiGeneral || KIND == kEpiGeneralOdd) {
            epi_general<KIND == kEpiGeneralOdd>(e, v, row, col0, s_scale + ct, s_bias + ct);
        } else {
            uint32_t w[8];
            epi_lean<KIND == kEpiLeanResidual>(v, s_scale + ct, s_bias + ct, e.inv_out_scale, e.residual_scale, r, w);
            st_global_v8(e.u8_out + row * e.N + col0, w);
        }
    }
}

// A warp's share of one accumulator in fragment form, straight to global memory: each row gets 32 bytes
// of four adjacent threads.  pos: the tile's first output byte of these columns, off[r]: from there to this
// thread's eight bytes in its row r, rows: bit r set where that row exists, left: columns up to N.
// (All that is worked out once per tile, or launch: a 64-bit row position per store cost 4-6 %.)
template <bool RES, class WaitFull>
__device__ __forceinline__ void epi_frag_columns(const EpiView &e, uint32_t taddr0, int cols, int64_t pos, const uint32_t (&off)[4], uint32_t rows,
                                                 int64_t left, const float *s_scale, const float *s_bias, uint32_t acc_empty_bar, int lane, WaitFull wait_full)
{
    s_scale += 8 * (lane & 3);
    s_bias += 8 * (lane & 3);
    const int valid = left < cols ? (int)left : cols;       // a multiple of 32, or none
    uint8_t *out = e.u8_out + pos;
    const uint8_t *residual = e.residual + pos;
    uint32_t rn[8];
    auto fetch_residual = [&](int c) {
        if (c >= valid) return;
#pragma unroll
        for (int r = 0; r < 4; ++r)
            if (rows >> r & 1u) {
                const uint2 b = __ldg(reinterpret_cast<const uint2 *>(residual + c + off[r]));
                rn[2 * r] = b.x;
                rn[2 * r + 1] = b.y;
            }
    };
    if (RES) {
#pragma unroll
        for (int i = 0; i < 8; ++i) rn[i] = 0u;
        fetch_residual(0);
    }
    wait_full();
#pragma unroll 1
    for (int c = 0; c < cols; c += 32) {
        uint32_t v[32], res[8], w[8];
        tmem_ld_frag_issue(taddr0 + (uint32_t)c, v);
        if (RES) {
#pragma unroll
            for (int i = 0; i < 8; ++i) res[i] = rn[i];
            fetch_residual(c + 32);
        }
        tmem_ld_wait();
        if (c + 32 == cols) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acc_empty_bar);
        }
        if (c >= valid) continue;
        epi_frag<RES>(v, s_scale + c, s_bias + c, e.inv_out_scale, e.residual_scale, res, w);
#pragma unroll
        for (int r = 0; r < 4; ++r)
            if (rows >> r & 1u) *reinterpret_cast<uint2 *>(out + c + off[r]) = make_uint2(w[2 * r], w[2 * r + 1]);
    }
}

// OUT: the kind of output that the kernel is instantiated for (EpiOut).
template <int OUT, class WaitFull>
__device__ __forceinline__ void epi_warp_columns(const EpiView &e, uint32_t taddr0, int cbase, int cols, int64_t row, bool row_ok,
                                                 int64_t n0, const float *s_scale, const float *s_bias,
                                                 uint32_t acc_empty_bar, int lane, WaitFull wait_full)
{
    if constexpr (OUT != kOutGeneral) {
        epi_warp_columns_as<OUT == kOutResidual ? kEpiLeanResidual : kEpiLean>(e, taddr0, cbase, cols, row, row_ok, n0, s_scale, s_bias,
                                                                               acc_empty_bar, lane, wait_full);
    } else {
        if (e.gran == 1) epi_warp_columns_as<kEpiGeneralOdd>(e, taddr0, cbase, cols, row, row_ok, n0, s_scale, s_bias, acc_empty_bar, lane, wait_full);
        else epi_warp_columns_as<kEpiGeneral>(e, taddr0, cbase, cols, row, row_ok, n0, s_scale, s_bias, acc_empty_bar, lane, wait_full);
    }
}

// One box of the staged output: 32 rows of `box` (64 or 128) columns, from tensor memory (in fragment form) to
// the warp's shared-memory buffer `buf` (32 rows of `box` bytes, 16-byte pieces swizzled as the
// tensor map says), which a TMA store then takes to global memory as whole 64- or 128-byte
// pieces of a row.  With a residual the buffer holds the identity tensor's box, fetched by TMA,
// and is rewritten in place.
//
// Why: a thread owns an output row, so its own 32-byte stores (and residual loads) of a warp fall
// into 32 different lines; a 51 MB output took 16.6 us that way against 10.5 in whole lines, and
// its residual with it, with little L1 left beside the operand ring, 35 against 20.  (Fetching
// the residual into L2 ahead of the boxes changed nothing: it is not HBM's latency.)  The whole
// layer, M 200704 x K 64 -> N 256: 26.5 -> 23.3 us, with a residual 44.8 -> 33.2; and in fragment form 19.0 ->
// 17.8 and 31.2 -> 28.1 (four buffers of 64 columns a warp, for more residual bytes in flight: 32.0).
// next_residual() is called once the first 32 columns are done.
template <bool RES, class Next>
__device__ __forceinline__ void epi_staged_box(uint32_t taddr, int box, uint32_t buf, const float *s_scale, const float *s_bias,
                                               float inv, float res_scale, uint32_t acc_empty_bar, int lane, Next next_residual)
{
    // this thread's rows lane / 4 + 8r: the swizzle of all four is that of the first
    const uint32_t row = (uint32_t)(lane >> 2), c8 = 8u * (uint32_t)(lane & 3);
    const uint32_t row_buf = buf + row * (uint32_t)box, step = 8u * (uint32_t)box;
    const uint32_t swz = box == 128 ? row & 7u : (row >> 1) & 3u;
    s_scale += c8;
    s_bias += c8;
#pragma unroll 1
    for (int c = 0; c < box; c += 32) {
        uint32_t v[32], res[8], w[8];
        tmem_ld_frag_issue(taddr + (uint32_t)c, v);
        const uint32_t col = (uint32_t)c + c8;
        const uint32_t a = row_buf + (((col >> 4) ^ swz) << 4) + (col & 8u);
        if (RES) {
#pragma unroll
            for (int r = 0; r < 4; ++r)
                asm volatile("ld.shared.v2.u32 {%0,%1}, [%2];" : "=r"(res[2 * r]), "=r"(res[2 * r + 1]) : "r"(a + (uint32_t)r * step));
        }
        tmem_ld_wait();
        if (acc_empty_bar && c + 32 == box) {        // the accumulator's last columns are in registers
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acc_empty_bar);
        }
        epi_frag<RES>(v, s_scale + c, s_bias + c, inv, res_scale, res, w);
#pragma unroll
        for (int r = 0; r < 4; ++r)
            asm volatile("st.shared.v2.u32 [%0], {%1,%2};" :: "r"(a + (uint32_t)r * step), "r"(w[2 * r]), "r"(w[2 * r + 1]) : "memory");
        if (c == 0) next_residual();
    }
}

// Stages the scale and bias of columns n0 .. n0+bn-1 in shared memory for the `threads` threads
// that meet at hardware barrier `bar` (t = this thread's number among them).
template <class Args>
__device__ __forceinline__ void epi_stage_scale_bias(const Args &g, int64_t n0, int bn, int t, int threads, int bar,
                                                     float *s_scale, float *s_bias)
{
    asm volatile("bar.sync %0, %1;" :: "r"(bar), "r"(threads) : "memory");     // previous readers are done
    for (int c = t; c < bn; c += threads) {
        const int64_t col = n0 + c;
        const bool ok = col < g.N;
        s_scale[c] = ok ? __ldg(g.scale + col) : 0.0f;
        s_bias[c] = (ok && g.bias) ? __ldg(g.bias + col) : 0.0f;
    }
    asm volatile("bar.sync %0, %1;" :: "r"(bar), "r"(threads) : "memory");
}

// ---- the kernel ---------------------------------------------------------------------------

template <int BN, int BK>
struct TileCfg {
    static constexpr int kABytes = kBM * BK;
    static constexpr int kBBytes = BN * BK;
    static constexpr int kStageBytes = kABytes + kBBytes;
    // stages of the ring beside `staging` bytes of output boxes
    __host__ __device__ static constexpr int stages(int staging)
    {
        const int n = (staging ? kMaxDynSmemGemm - 1024 - staging : kSmemBudget) / kStageBytes;
        return n > kMaxStages ? kMaxStages : n;
    }
    static constexpr int kAcc = BN == 256 ? 2 : 4;                  // accumulator stages in tensor memory
    static constexpr int kTmemCols = kAcc * BN;
    // With the activations in tensor memory (ATM): stages of weights, and of raw activations in what room is left
    static constexpr int kAtmRoom = kMaxDynSmemGemm - 1024, kAtmStages = 4;
    static constexpr int kAtmRawStages = (kAtmRoom - kAtmStages * kBBytes) / kABytes;
    static constexpr int kAtmSmem = 1024 + kAtmStages * kBBytes + kAtmRawStages * kABytes;
};

template <int BN, int BK, int MODE, int XN, bool RND, int OUT, bool ATM>
__global__ void __launch_bounds__(gemm_threads(MODE, ATM), 1)
sparq_gemm_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
                  const __grid_constant__ CUtensorMap map_out, const __grid_constant__ CUtensorMap map_res, const GemmArgs g)
{
    using Cfg = TileCfg<BN, BK>;
    constexpr bool kTwoProducers = MODE == SPARQ_MODE_NONE || ATM;
    // ATM: the transform warps write their results to tensor memory, which the tensor core reads A from; the
    // raw activations have a ring of their own.
    static_assert(!ATM || (MODE != SPARQ_MODE_NONE && BK == 128 && BN == 256 && OUT == kOutBytes), "A in tensor memory: transformed steps of 128 bytes");
    static_assert(!ATM || (Cfg::kAtmRawStages == 5 && Cfg::kAtmStages * 32 + BN <= 512), "rings with A in tensor memory");
    const int S = ATM ? Cfg::kAtmStages : g.stages;
    extern __shared__ uint8_t smem_raw[];
    // The ring that the transform teams read has two sets of full barriers, for even and odd rounds.  A parity
    // answers for every second phase, so a team may ask a barrier for a phase only once it knows that the one before
    // has completed.  Of a single set, in a ring of an odd number of stages -- three beside the boxes of staged
    // 256-wide tiles, seven of 64-wide ones, five raw ones with ATM -- that phase was the other team's, which
    // nothing orders before the question; a barrier of two sets comes round after twice the stages, with the team
    // that asked it before.  (Reading the stage's empty barrier first is as safe, but one more round trip per
    // step: 200704 x 64, K 256, 16.85 -> 17.05 us, 12544 x 256, K 1024, 8.75 -> 9.05.  Two sets with the counters in
    // every lane: 17.25 and 9.0; in the warp: 16.1 and 8.85.)
    constexpr int kFullSets = MODE != SPARQ_MODE_NONE && !ATM ? 2 : 1, kRawSets = ATM ? 2 : 1;
    __shared__ __align__(8) uint64_t bar_full[kFullSets * kMaxStages], bar_xf[kMaxStages], bar_empty[kMaxStages];
    __shared__ __align__(8) uint64_t bar_raw[ATM ? kRawSets * kMaxStages : 1], bar_raw_empty[ATM ? kMaxStages : 1];
    __shared__ __align__(8) uint64_t bar_res[epi_warps(MODE)][2];       // residual boxes landed
    // tensor memory: accumulators; with ATM one, and four stages of transformed activations
    constexpr int kAcc = ATM ? 1 : Cfg::kAcc;
    constexpr int kTmemCols = ATM ? 512 : Cfg::kTmemCols;
    // The epilogue warps form groups of four (one warp per tensor-memory lane quarter) and the
    // groups teams: team t takes the CTA's tiles of number t modulo the number of teams, so that the
    // epilogues of consecutive tiles -- mostly latency -- overlap.  A CTA with a single tile puts
    // all its groups in one team, each group on its own columns (32 at least; a group too many
    // for the tile's columns stays idle).
    constexpr int kGroups = epi_warps(MODE) / 4;
    constexpr int kMaxTeams = kGroups < kAcc ? kGroups : kAcc;
    __shared__ __align__(8) uint64_t bar_acc_full[kAcc], bar_acc_empty[kAcc], bar_done;
    __shared__ uint32_t tmem_base_slot;
    __shared__ uint32_t abort_word;
    constexpr bool kSharedFull = MODE == SPARQ_MODE_NONE;        // both producers announce on bar_full
    constexpr uint32_t kStillIssuing = 0xFFFFFFFFu;
    __shared__ volatile uint32_t announced[kSharedFull ? 2 : 1];        // stages that each of them announced, once it has stopped
    __shared__ __align__(16) float s_scale[kMaxTeams][BN], s_bias[kMaxTeams][BN];

    // the same in all lanes, and so for the compiler: what a role keeps of its ring costs the lanes' integer pipe nothing
    const int warp = __shfl_sync(0xFFFFFFFFu, (int)(threadIdx.x >> 5), 0);
    const int lane = threadIdx.x & 31;
    volatile uint32_t *abort_flag = &abort_word;

    const int64_t m_tiles = (g.M + kBM - 1) / kBM;
    const int64_t n_tiles = (g.N + BN - 1) / BN;
    // tile indices fit 32 bits (the host refuses larger problems); a 64-bit division per tile
    // and thread costs more instructions than a tile's share of the epilogue arithmetic
    const uint32_t total_tiles = (uint32_t)(m_tiles * n_tiles);
    const uint32_t n_tiles32 = (uint32_t)n_tiles;
    const int teams = total_tiles > gridDim.x ? kMaxTeams : 1;

    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const int SA = ATM ? Cfg::kAtmRawStages : S;
    const uint32_t b_base = smem_base + (uint32_t)(ATM ? SA * Cfg::kABytes : Cfg::kABytes);
    constexpr uint32_t kAStep = ATM ? Cfg::kABytes : Cfg::kStageBytes, kBStep = ATM ? Cfg::kBBytes : Cfg::kStageBytes;
    auto a_stage = [&](int s) { return smem_base + (uint32_t)s * kAStep; };
    auto b_stage = [&](int s) { return b_base + (uint32_t)s * kBStep; };

    if (threadIdx.x == 0) {
        prefetch_tensormap(&map_a);
        prefetch_tensormap(&map_b);
        for (int q = 0; q < kFullSets * S; ++q) mbar_init(smem_u32(&bar_full[q]), kSharedFull ? 2 : 1);
        for (int s = 0; s < S; ++s) {
            mbar_init(smem_u32(&bar_xf[s]), kXfTeamWarps);
            mbar_init(smem_u32(&bar_empty[s]), 1);
        }
        for (int q = 0; ATM && q < kRawSets * SA; ++q) mbar_init(smem_u32(&bar_raw[q]), 1);
        for (int s = 0; ATM && s < SA; ++s) mbar_init(smem_u32(&bar_raw_empty[s]), kXfTeamWarps);
        for (int a = 0; a < kAcc; ++a) {
            mbar_init(smem_u32(&bar_acc_full[a]), 1);
            mbar_init(smem_u32(&bar_acc_empty[a]), 4 * epi_parts(kGroups, teams, BN));
        }
        for (int w = 0; w < epi_warps(MODE); ++w)
            for (int b = 0; b < 2; ++b) mbar_init(smem_u32(&bar_res[w][b]), 1);
        mbar_init(smem_u32(&bar_done), 1);
        abort_word = 0;
        if (kSharedFull) announced[0] = announced[1] = kStillIssuing;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(smem_u32(&tmem_base_slot)), "r"((uint32_t)kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = tmem_base_slot;
    const int kb_count = g.k_blocks;

    if (warp == 0 || (kTwoProducers && warp == kWeightWarp)) {
        // ================= TMA producers =================
        // A thread feeds the whole CTA, a few hundred cycles a step: positions are counters, not divisions,
        // and the abort flag is read only where a wait has given up (every read of shared memory queues
        // behind the tensor core's operand fetches).
        if (lane == 0) {
            constexpr uint32_t kBytes = kTwoProducers ? Cfg::kABytes : Cfg::kStageBytes;     // of the first producer
            // the ring that this thread fills, and its barriers
            const bool raw = ATM && warp == 0;
            const int ring = raw ? SA : S;
            const uint32_t bars_full = smem_u32(raw ? bar_raw : bar_full), bars_empty = smem_u32(raw ? bar_raw_empty : bar_empty);
            const int sets = raw ? kRawSets : kFullSets;
            const uint32_t set = sets == 2 ? 8u * (uint32_t)ring : 0u;       // bytes from one set of full barriers to the other
            uint32_t it = 0;   // running stage counter across tiles
            int s = 0;         // stage it % ring
            uint32_t use = 0;  // it / ring
            bool live = true;
            for (uint32_t tile = blockIdx.x; tile < total_tiles && live; tile += gridDim.x) {
                const uint32_t mt = (n_tiles32 == 1) ? tile : tile / n_tiles32, nt = tile - mt * n_tiles32;
                const int64_t m0 = (int64_t)mt * kBM;
                const int n0 = (int)(nt * BN);
                int base_n = 0, base_h = 0, base_w = 0;
                if (g.conv) {
                    const uint32_t hw = (uint32_t)(g.Ho * g.Wo), m032 = (uint32_t)m0;   // M of a convolution fits 31 bits
                    base_n = (int)(m032 / hw);
                    const int rem = (int)(m032 - (uint32_t)base_n * hw);
                    base_h = (rem / g.Wo) * g.stride_h - g.pad_h;
                    base_w = (rem % g.Wo) * g.stride_w - g.pad_w;
                }
                // The roles that touch the caller's memory wait for the kernel before, each behind what it can work
                // out without it (later waits return at once); the others do not (EARLY waits).  With one wait of all
                // threads behind the set-up, its release was followed by every role's first index arithmetic
                // and the fetch of its code: 0.2 to 0.6 us of each launch, the ResNet-50 pass 798 -> 763 us.
                dep_wait();
                dep_launch();
                // the tile's stages in turn, until the CTA has given up
                auto stages = [&](uint32_t bytes, auto copy) {
                    TapWalk tap(g, BK, 0);
                    for (int kb = 0; kb < kb_count; ++kb, ++it) {
                        if (use > 0 && !mbar_wait(bars_empty + 8u * (uint32_t)s, (use - 1) & 1, abort_flag, g.status, g.wait_limit)) { live = false; break; }
                        const uint32_t full = bars_full + 8u * (uint32_t)s + (use & 1u) * set;
                        mbar_expect_tx(full, bytes);
                        copy(full, tap);
                        tap.next();
                        if (++s == ring) { s = 0; ++use; }
                    }
                };
                auto weights = [&](uint32_t full, const TapWalk &tap) {
                    if (OUT != kOutGeneral) tma_load_row_groups(b_stage(s), &map_b, full, tap.k, n0);
                    else tma_load_2d(b_stage(s), &map_b, full, tap.k, n0);
                };
                if (kTwoProducers && warp == kWeightWarp) {
                    stages(Cfg::kBBytes, weights);
                } else if (g.conv) {
                    // Channels past C arrive as zeros, so whatever the weight block holds
                    // there (the next tap's first bytes) adds nothing.
                    stages(kBytes, [&](uint32_t full, const TapWalk &tap) {
                        tma_load_im2col_4d(a_stage(s), &map_a, full, tap.c, base_w, base_h, base_n, (uint16_t)tap.s, (uint16_t)tap.r);
                        if (!kTwoProducers) weights(full, tap);
                    });
                } else {
                    stages(kBytes, [&](uint32_t full, const TapWalk &tap) {
                        tma_load_2d(a_stage(s), &map_a, full, tap.k, (int)m0);
                        if (!kTwoProducers) weights(full, tap);
                    });
                }
            }
            const int me = warp == 0 ? 0 : 1;
            if (kSharedFull) announced[me] = it;
            // After an abort: wait (bounded) for the copies still in flight, so that none
            // lands after the CTA has exited.
            if (*abort_flag) {
                uint32_t last = it;
                if (kSharedFull) {
                    // The two may have stopped at different stages, at most a ring apart: no stage is released that
                    // both have not announced.  The one behind arrives for the other one's, which complete with
                    // that one's copies then, and waits for them, too.
                    const long long t0 = clock64();
                    uint32_t other;
                    while ((other = announced[me ^ 1]) == kStillIssuing && clock64() - t0 <= g.wait_limit) {}
                    for (uint32_t j = it; other != kStillIssuing && j < other; ++j, ++last) mbar_arrive(bars_full + 8u * (j % (uint32_t)ring));
                }
                const uint32_t first = last > (uint32_t)ring ? last - ring : 0;
                const uint32_t bars = (uint32_t)(sets * ring);
                for (uint32_t j = first; j < last; ++j)
                    mbar_wait(bars_full + 8u * (j % bars), j / bars & 1u, abort_flag, g.status, g.wait_limit, true);
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ================= MMA issuer =================
        // The whole warp runs this loop converged and one elected lane issues, so that the
        // descriptor arithmetic (warp-uniform values only) can stay in the uniform datapath.
        {
            const uint32_t elected = elect_one();
            constexpr uint32_t idesc = make_idesc_i8(BN);
            // descriptors of stage 0; a stage adds its byte offset / 16 to the start-address field
            const uint64_t adesc0 = make_smem_desc<BK>(smem_base);
            const uint64_t bdesc0 = make_smem_desc<BK>(b_base);
            uint32_t local_tile = 0;
            int s = 0;             // stage
            uint32_t ph = 0;       // its phase parity
            bool live = true;
            for (uint32_t tile = blockIdx.x; tile < total_tiles && live; tile += gridDim.x, ++local_tile) {
                const int acc = local_tile % kAcc;
                const uint32_t acc_use = local_tile / kAcc;
                if (acc_use > 0) mbar_wait(smem_u32(&bar_acc_empty[acc]), (acc_use - 1) & 1, abort_flag, g.status, g.wait_limit);
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + (uint32_t)(acc * BN);
                for (int kb = 0; kb < kb_count; ++kb) {
                    if (kSharedFull) {
                        // (a stage that is not there is not released, see the producers)
                        if (!mbar_wait<true>(smem_u32(&bar_full[s]), ph, abort_flag, g.status, g.wait_limit)) { live = false; break; }
                    } else mbar_wait<true>(smem_u32(&bar_xf[s]), ph, abort_flag, g.status, g.wait_limit);
                    if (ATM) mbar_wait(smem_u32(&bar_full[s]), ph, abort_flag, g.status, g.wait_limit);
                    tc_fence_after();
                    const uint64_t adesc = adesc0 + (uint64_t)((uint32_t)s * (kAStep >> 4)), bdesc = bdesc0 + (uint64_t)((uint32_t)s * (kBStep >> 4));
                    const uint32_t a_tmem = tmem_base + 256u + (uint32_t)s * 32u;
#pragma unroll
                    for (int k = 0; k < BK / 32; ++k) {
                        if (ATM) tc_mma_i8_tmem_if(d_tmem, a_tmem + (uint32_t)(k * 8), bdesc + (uint64_t)(k * 2), idesc, (kb > 0 || k > 0) ? 1u : 0u, elected);
                        else tc_mma_i8_if(d_tmem, adesc + (uint64_t)(k * 2), bdesc + (uint64_t)(k * 2), idesc,
                                     (kb > 0 || k > 0) ? 1u : 0u, elected);
                    }
                    tc_commit_if(smem_u32(&bar_empty[s]), elected);       // stage reusable once these MMAs retire
                    if (++s == S) { s = 0; ph ^= 1u; }
                }
                tc_commit_if(smem_u32(&bar_acc_full[acc]), elected);      // accumulator complete
            }
            // all tensor-core work of this CTA has retired before tensor memory is freed
            tc_commit_if(smem_u32(&bar_done), elected);
            mbar_wait(smem_u32(&bar_done), 0, abort_flag, g.status, g.wait_limit, true);
        }
        __syncwarp();
    } else if (warp < kFirstEpiWarp + epi_warps(MODE)) {
        // ================= epilogue =================
        const int quarter = warp & 3;                        // tensor-memory lanes this warp may read
        const int group = (warp - kFirstEpiWarp) >> 2;
        const int team = group % teams;                      // tiles team, team + teams, ...
        const int parts = epi_parts(kGroups, teams, BN), part = group / teams;
        const int cols = BN / parts, cbase = part * cols;    // this warp's share of the tile's columns
        const int team_thread = (part * 4 + quarter) * 32 + lane, team_threads = parts * 128;
        const EpiView ev = make_epi_view(g);
        uint32_t off[4];                                     // epi_frag_columns
#pragma unroll
        for (int r = 0; r < 4; ++r) off[r] = (uint32_t)((lane >> 2) + 8 * r) * (uint32_t)g.N + 8u * (uint32_t)(lane & 3);
        int64_t staged_nt = -1;
        uint32_t local_tile = (uint32_t)team;
        dep_wait();
        if (!ATM && OUT != kOutGeneral && g.out_box) {
            // ---- through shared memory (see epi_staged_box); a reduction long enough for ATM outweighs its output ----
            const int ew = warp - kFirstEpiWarp;
            const uint32_t box_bytes = 32u * (uint32_t)g.out_box;
            const uint32_t stage0 = a_stage(S) + (uint32_t)ew * 2u * box_bytes;
            constexpr bool res = OUT == kOutResidual;
            // boxes of this warp in order: the out_box-wide parts of its columns, tile after tile
            auto fetch = [&](uint32_t n, uint32_t tile, int c) {          // box n's residual, by lane 0
                const uint32_t mt = (n_tiles32 == 1) ? tile : tile / n_tiles32;
                const int x = (int)(tile - mt * n_tiles32) * BN + cbase + c, y = (int)mt * kBM + quarter * 32;
                const uint32_t bar = smem_u32(&bar_res[ew][n & 1u]);
                mbar_expect_tx(bar, box_bytes);
                tma_load_2d(stage0 + (n & 1u) * box_bytes, &map_res, bar, x, y);
            };
            uint32_t n = 0;
            const uint32_t tile_step = (uint32_t)teams * gridDim.x;
            uint32_t tile = blockIdx.x + (uint32_t)team * gridDim.x;
            if (part < parts && tile < total_tiles && res && lane == 0) fetch(0u, tile, 0);
            for (; tile < total_tiles && part < parts; tile += tile_step, local_tile += (uint32_t)teams) {
                const uint32_t mt32 = (n_tiles32 == 1) ? tile : tile / n_tiles32;
                const int64_t nt = tile - mt32 * n_tiles32;
                const int acc = local_tile % kAcc;
                if (nt != staged_nt) {
                    staged_nt = nt;
                    epi_stage_scale_bias(g, nt * BN, BN, team_thread, team_threads, 1 + team, s_scale[team], s_bias[team]);
                }
                mbar_wait(smem_u32(&bar_acc_full[acc]), (local_tile / kAcc) & 1u, abort_flag, g.status, g.wait_limit);
                tc_fence_after();
                const uint32_t taddr0 = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(acc * BN + cbase);
                for (int c = 0; c < cols; c += g.out_box, ++n) {
                    const bool last = c + g.out_box == cols;
                    auto next_residual = [&]() {
                        if (!res || lane != 0) return;
                        const uint32_t nt_tile = last ? tile + tile_step : tile;
                        if (nt_tile >= total_tiles) return;
                        tma_store_wait_read<0>();          // the box before this one has left the buffer
                        fetch(n + 1u, nt_tile, last ? 0 : c + g.out_box);
                    };
                    const uint32_t buf = stage0 + (n & 1u) * box_bytes;
                    if (res) {
                        mbar_wait(smem_u32(&bar_res[ew][n & 1u]), (n >> 1) & 1u, abort_flag, g.status, g.wait_limit);
                    } else {
                        if (lane == 0) tma_store_wait_read<1>();       // box n - 2 has left the buffer
                        __syncwarp();
                    }
                    const float *sc = s_scale[team] + cbase + c, *bi = s_bias[team] + cbase + c;
                    const uint32_t abar = last ? smem_u32(&bar_acc_empty[acc]) : 0u;
                    epi_staged_box<res>(taddr0 + (uint32_t)c, g.out_box, buf, sc, bi, g.inv_out_scale, g.residual_scale, abar, lane, next_residual);
                    fence_proxy_async_smem();
                    __syncwarp();
                    const int x = (int)nt * BN + cbase + c;
                    const int64_t y = (int64_t)mt32 * kBM + quarter * 32;
                    if (lane == 0) {
                        if ((int64_t)x < g.N && y < g.M) tma_store_2d(&map_out, buf, x, (int)y);
                        tma_store_commit();
                    }
                }
            }
            if (lane == 0) {
                // after an abort: wait (bounded) for residual boxes that may still be in flight
                if (*abort_flag && res && n > 0)
                    for (uint32_t q = n > 1 ? n - 2 : 0; q < n; ++q)
                        mbar_wait(smem_u32(&bar_res[ew][q & 1u]), (q >> 1) & 1u, abort_flag, g.status, g.wait_limit, true);
                tma_store_wait_all();
            }
            __syncwarp();
        } else
        for (uint32_t tile = blockIdx.x + (uint32_t)team * gridDim.x; tile < total_tiles && part < parts;
             tile += (uint32_t)teams * gridDim.x, local_tile += (uint32_t)teams) {
            const uint32_t mt32 = (n_tiles32 == 1) ? tile : tile / n_tiles32;
            const int64_t mt = mt32, nt = tile - mt32 * n_tiles32;
            const int acc = local_tile % kAcc;
            const uint32_t acc_use = local_tile / kAcc;
            if (ev.need_f && nt != staged_nt) {              // new column tile: new scale / bias
                staged_nt = nt;
                epi_stage_scale_bias(g, nt * BN, BN, team_thread, team_threads, 1 + team, s_scale[team], s_bias[team]);
            }
            const uint32_t taddr0 = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(acc * BN + cbase);
            auto wait_full = [&]() {
                mbar_wait(smem_u32(&bar_acc_full[acc]), acc_use & 1, abort_flag, g.status, g.wait_limit);
                tc_fence_after();
            };
            const int64_t row0 = mt * kBM + quarter * 32;
            if constexpr (!frag_rows(OUT, BN, 0)) {
                const int64_t row = row0 + lane;
                epi_warp_columns<OUT>(ev, taddr0, cbase, cols, row, row < g.M, nt * BN, s_scale[team], s_bias[team],
                                      smem_u32(&bar_acc_empty[acc]), lane, wait_full);
            } else {
                uint32_t rows = 0;
#pragma unroll
                for (int r = 0; r < 4; ++r) rows |= (row0 + (lane >> 2) + 8 * r < g.M ? 1u : 0u) << r;
                epi_frag_columns<OUT == kOutResidual>(ev, taddr0, cols, row0 * g.N + nt * BN + cbase, off, rows, g.N - nt * BN - cbase, s_scale[team] + cbase,
                                                      s_bias[team] + cbase, smem_u32(&bar_acc_empty[acc]), lane, wait_full);
            }
        }
    } else if (MODE != SPARQ_MODE_NONE) {
        // ================= transform =================
        const int team = (warp - kFirstXfWarp) / kXfTeamWarps;
        const int xt = threadIdx.x - (kFirstXfWarp + team * kXfTeamWarps) * 32;   // 0 .. 127 inside the team
        constexpr int kXfThreads = kXfTeamWarps * 32;
        constexpr int kVecs = Cfg::kABytes / 16;
        constexpr int kPerThread = kVecs / kXfThreads;
        constexpr int kHalf = kPerThread / 2;                       // vectors that a thread works on at a time
        static_assert(kVecs % kXfThreads == 0 && kPerThread % 2 == 0, "A stage must split evenly over a team, and in halves");
        const XformDev xf = g.xf;
        // The team's stages in order: its number, the ring stage and its phase.  A stage's first half is
        // loaded while the second half of the one before is worked on, if it has landed by then: with two
        // warps to a scheduler, the barrier read and the loads' latency at the head of each stage were a
        // tenth of its time: 200704 x 64, K 256, 17.7 -> 16.9 us, 50176 x 128, K 512, 11.4 -> 10.9.
        const uint32_t my_tiles = blockIdx.x < total_tiles ? (total_tiles - blockIdx.x + gridDim.x - 1) / gridDim.x : 0u;
        const uint32_t total = my_tiles * (uint32_t)kb_count;
        auto load = [&](uint4 (&v)[kHalf], int s, int j0) {
#pragma unroll
            for (int j = 0; j < kHalf; ++j)
                asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v[j].x), "=r"(v[j].y), "=r"(v[j].z), "=r"(v[j].w)
                             : "r"(a_stage(s) + (uint32_t)((j0 + j) * kXfThreads + xt) * 16u));
        };
        auto work = [&](uint4 (&v)[kHalf], int s, int j0) {
#pragma unroll
            for (int j = 0; j < kHalf; ++j) {
                v[j].x = xform_fused<MODE, XN, RND>(v[j].x, xf);
                v[j].y = xform_fused<MODE, XN, RND>(v[j].y, xf);
                v[j].z = xform_fused<MODE, XN, RND>(v[j].z, xf);
                v[j].w = xform_fused<MODE, XN, RND>(v[j].w, xf);
                asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};"
                             :: "r"(a_stage(s) + (uint32_t)((j0 + j) * kXfThreads + xt) * 16u),
                                "r"(v[j].x), "r"(v[j].y), "r"(v[j].z), "r"(v[j].w) : "memory");
            }
        };
        if constexpr (ATM) {
            // A thread has one row (of its warp's tensor-memory lanes), half of its 128 bytes at a time; from the
            // raw stage into the transformed one, which has the number of the weight stage beside it.
            const int quarter = warp & 3;
            const uint32_t row = (uint32_t)(quarter * 32 + lane), swz = row & 7u;
            auto load_row = [&](uint4 (&v)[4], int sa, int c0) {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v[j].x), "=r"(v[j].y), "=r"(v[j].z), "=r"(v[j].w)
                                 : "r"(a_stage(sa) + row * 128u + (((uint32_t)(c0 + j) ^ swz) << 4)));
            };
            auto work_row = [&](uint4 (&v)[4]) {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    v[j].x = xform_fused<MODE, XN, RND>(v[j].x, xf);
                    v[j].y = xform_fused<MODE, XN, RND>(v[j].y, xf);
                    v[j].z = xform_fused<MODE, XN, RND>(v[j].z, xf);
                    v[j].w = xform_fused<MODE, XN, RND>(v[j].w, xf);
                }
            };
            uint4 va[4], vb[4];
            int sa = team, s = team;
            int qa = team;                     // full barrier of the raw stage,
            uint32_t pa = 0, use = 0;          // its phase; uses of the transformed one before
            bool loaded = false;
            for (uint32_t it = (uint32_t)team; it < total; it += kXfTeams) {
                if (!loaded) {
                    mbar_wait<true>(smem_u32(&bar_raw[qa]), pa, abort_flag, g.status, g.wait_limit);
                    load_row(va, sa, 0);
                }
                load_row(vb, sa, 4);
                work_row(va);
                if (use > 0) mbar_wait(smem_u32(&bar_empty[s]), (use - 1u) & 1u, abort_flag, g.status, g.wait_limit);
                tc_fence_after();
                const uint32_t dst = tmem_base + ((uint32_t)(quarter * 32) << 16) + 256u + (uint32_t)s * 32u;
                tmem_st_32x16(dst, va);
                int na = sa + kXfTeams;
                if (na >= SA) na -= SA;
                qa += kXfTeams;
                if (qa >= kRawSets * SA) { qa -= kRawSets * SA; pa ^= 1u; }
                loaded = it + kXfTeams < total && __all_sync(0xFFFFFFFFu, mbar_test(smem_u32(&bar_raw[qa]), pa));
                if (loaded) load_row(va, na, 0);
                work_row(vb);
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&bar_raw_empty[sa]));      // the whole stage is in registers
                tmem_st_32x16(dst + 16u, vb);
                tmem_st_wait();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&bar_xf[s]));
                sa = na;
                s += kXfTeams;
                if (s >= S) { s -= S; ++use; }
            }
        } else {
            uint4 va[kHalf], vb[kHalf];
            int s = team;
            int q = team;              // its full barrier,
            uint32_t ph = 0;           // and that barrier's phase
            bool loaded = false;
            for (uint32_t it = (uint32_t)team; it < total; it += kXfTeams) {
                if (!loaded) {
                    mbar_wait<true>(smem_u32(&bar_full[q]), ph, abort_flag, g.status, g.wait_limit);
                    load(va, s, 0);
                }
                load(vb, s, kHalf);
                work(va, s, 0);
                int ns = s + kXfTeams;
                if (ns >= S) ns -= S;
                q += kXfTeams;
                if (q >= kFullSets * S) { q -= kFullSets * S; ph ^= 1u; }
                loaded = it + kXfTeams < total && __all_sync(0xFFFFFFFFu, mbar_test(smem_u32(&bar_full[q]), ph));
                if (loaded) load(va, ns, 0);
                work(vb, s, kHalf);
                fence_proxy_async_smem();       // generic-proxy writes visible to the tensor core
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&bar_xf[s]));
                s = ns;
            }
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;"
                     :: "r"(tmem_base), "r"((uint32_t)kTmemCols) : "memory");
    }
}

struct GemmMaps {
    CUtensorMap a, b, out, res;     // out, res: staged output only
};

// Host launcher for one tile shape; picks the transform variant.  Defined once per
// (BN, BK) in its own translation unit.
template <int BN, int BK>
cudaError_t launch_gemm_shape(const GemmMaps &m, GemmArgs &g, int mode, int n, int rnd, int grid, cudaStream_t st);

template <int BN, int BK, int MODE, int XN, bool RND, int OUT, bool ATM>
cudaError_t launch_gemm_kernel(const GemmMaps &m, GemmArgs &g, int grid, cudaStream_t st)
{
    auto kfn = sparq_gemm_kernel<BN, BK, MODE, XN, RND, OUT, ATM>;
    static bool attr_set[64] = {};   // per device ordinal
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64 || !attr_set[dev]) {
        e = cudaFuncSetAttribute(kfn, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDynSmemGemm);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) attr_set[dev] = true;
    }
    const int staging = g.out_box ? epi_warps(MODE) * 2 * 32 * g.out_box : 0;
    g.stages = TileCfg<BN, BK>::stages(staging);
    const int smem = ATM ? TileCfg<BN, BK>::kAtmSmem : 1024 + g.stages * TileCfg<BN, BK>::kStageBytes + staging;
    return launch_overlapped(kfn, grid, gemm_threads(MODE, ATM), smem, st, m.a, m.b, m.out, m.res, g);
}

// Whether a fused launch of 256-wide tiles puts the transformed activations into tensor memory (ATM).  What a
// step moves through shared memory falls from 1024 to 768 wavefronts (counted, with copies and operand reads), but the accumulator has to
// do with one stage, and a launch starts and ends a little later: from a dozen steps a CTA.  us with / without:
// 16384 x 512, K 4096 (64 steps) 42.1 / 46.7, 12544 x 512, K 1024 (16) 14.3 / 15.0, 28x28x512 -> 1024 stride 2 (12) 13.3 /
// 13.7, 50176 x 256, K 512 (12) 13.04 / 12.97, 12544 x 256, K 1024 (8) 9.14 / 9.08, 6272 x 256, K 1024 (8) 8.4 / 8.05,
// 50176 x 512, K 128 (6) 13.8 / 12.7.  On narrower tiles it gave nothing (50176 x 128, K 512, 11.3 / 10.9).
inline bool a_in_tmem(const GemmArgs &g, int bn, int grid)
{
    const int64_t tiles = (g.M + kBM - 1) / kBM * ((g.N + bn - 1) / bn);
    return g.k_blocks >= 4 && (tiles + grid - 1) / grid * g.k_blocks >= 12;
}

template <int BN, int BK, int MODE, int XN, bool RND>
cudaError_t launch_gemm_variant(const GemmMaps &m, GemmArgs &g, int grid, cudaStream_t st)
{
    const int out = make_epi_view(g).out;
    if constexpr (MODE != SPARQ_MODE_NONE && BK == 128 && BN == 256) {
        if (out == kOutBytes && a_in_tmem(g, BN, grid)) return launch_gemm_kernel<BN, BK, MODE, XN, RND, kOutBytes, true>(m, g, grid, st);
    }
    if (out == kOutBytes) return launch_gemm_kernel<BN, BK, MODE, XN, RND, kOutBytes, false>(m, g, grid, st);
    if (out == kOutResidual) return launch_gemm_kernel<BN, BK, MODE, XN, RND, kOutResidual, false>(m, g, grid, st);
    return launch_gemm_kernel<BN, BK, MODE, XN, RND, kOutGeneral, false>(m, g, grid, st);
}

#define SPARQ_LAUNCH_VARIANT(MODE_, XN_, RND_) return launch_gemm_variant<BN, BK, MODE_, XN_, RND_>(m, g, grid, st)

#define SPARQ_DEFINE_GEMM_SHAPE(BN_, BK_)                                                              \
    template <>                                                                                        \
    cudaError_t launch_gemm_shape<BN_, BK_>(const GemmMaps &m, GemmArgs &g, int mode, int n, int rnd,  \
                                            int grid, cudaStream_t st)                                 \
    {                                                                                                  \
        constexpr int BN = BN_, BK = BK_;                                                              \
        if (mode == SPARQ_MODE_NONE) SPARQ_LAUNCH_VARIANT(SPARQ_MODE_NONE, 4, false);                  \
        if (mode == SPARQ_MODE_BSPARQ) {                                                               \
            if (n == 8) SPARQ_LAUNCH_VARIANT(SPARQ_MODE_BSPARQ, 8, true);                              \
            if (n == 5) { if (rnd) SPARQ_LAUNCH_VARIANT(SPARQ_MODE_BSPARQ, 5, true);                   \
                          else SPARQ_LAUNCH_VARIANT(SPARQ_MODE_BSPARQ, 5, false); }                    \
            if (n == 4) { if (rnd) SPARQ_LAUNCH_VARIANT(SPARQ_MODE_BSPARQ, 4, true);                   \
                          else SPARQ_LAUNCH_VARIANT(SPARQ_MODE_BSPARQ, 4, false); }                    \
            if (rnd) SPARQ_LAUNCH_VARIANT(SPARQ_MODE_BSPARQ, 0, true);                                 \
            else SPARQ_LAUNCH_VARIANT(SPARQ_MODE_BSPARQ, 0, false);                                    \
        }                                                                                              \
        if (n == 8) SPARQ_LAUNCH_VARIANT(SPARQ_MODE_VSPARQ, 8, true);                                  \
        if (n == 5) { if (rnd) SPARQ_LAUNCH_VARIANT(SPARQ_MODE_VSPARQ, 5, true);                       \
                      else SPARQ_LAUNCH_VARIANT(SPARQ_MODE_VSPARQ, 5, false); }                        \
        if (n == 4) { if (rnd) SPARQ_LAUNCH_VARIANT(SPARQ_MODE_VSPARQ, 4, true);                       \
                      else SPARQ_LAUNCH_VARIANT(SPARQ_MODE_VSPARQ, 4, false); }                        \
        if (rnd) SPARQ_LAUNCH_VARIANT(SPARQ_MODE_VSPARQ, 0, true);                                     \
        else SPARQ_LAUNCH_VARIANT(SPARQ_MODE_VSPARQ, 0, false);                                        \
    }

}  // namespace sparq
