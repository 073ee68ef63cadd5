// Fused GEMM / im2col convolution for launches in which no CTA has more than one tile: the layers
// of a network at batch 1, small matrices.  Such a launch is latency from end to end, so this
// form of sparq_gemm_kernel (same operands, stage hand-offs and epilogue arithmetic)
//   - runs ten warps and at most half of an SM's shared memory and registers, so that CTAs of the
//     NEXT launch start beside it (barriers, tensor memory, tensor maps);
//   - has eight worker warps that first transform the stages and then run the epilogue, instead
//     of separate roles of which one always waits;
//   - has tiles of 64 rows as well as of 128 (x 64 columns): a step is bound by the transform of its
//     rows, so half the rows are half the time where the SMs are there;
//   - SHARED: puts a cluster of `split` CTAs on one tile when the tiles leave most SMs idle and the
//     reduction is long.  Each accumulates its part of the reduction steps and sends every row of
//     partial sums to the CTA that owns the row (an equal share of consecutive rows each) through
//     distributed shared memory; the stores signal the owner's barrier with their byte counts,
//     and when all have arrived the owner adds the `split` partial sums -- integers, so in any
//     order -- and writes the outputs.  The partial sums never leave the SMs.  (Through global
//     memory, with a counter per tile, they cost more than the split gave.)  With split = 1 the
//     same path turns the tile around in shared memory, so that int32 and fp32 outputs go out
//     as 256-byte pieces of rows instead of 16 bytes of 32 rows at a time.
// Warps: 0 TMA producer, 1 tensor memory and MMA issue, 2..9 workers.
#pragma once

#include "sparq_gemm_kernel.cuh"

namespace sparq {

constexpr int kSmallBN = 64;
constexpr int kSmallWorkers = 8;
constexpr int kSmallThreads = 32 * (2 + kSmallWorkers);
constexpr int kMaxSplit = 8;
// two CTAs per SM
constexpr int kSmallMaxDynSmem = 232448 / 2 - 3072;

// Rows of a tile that each CTA of its cluster writes.
__host__ __device__ inline int split_rows(int64_t M, int tile_rows, int split)
{
    const int rows = M < tile_rows ? (int)M : tile_rows;
    return (rows + split - 1) / split;
}
// Receive buffer: per sending rank 16 groups of four columns, a group = one 16-byte piece per row of
// the owner, padded by a piece.  A warp's store instruction (one group of consecutive rows) is
// contiguous, and the owner's reads along a row hit different banks.
__host__ __device__ inline int split_group_bytes(int rows) { return (rows + 1) * 16; }
__host__ __device__ inline int split_rank_bytes(int rows) { return kSmallBN / 4 * split_group_bytes(rows); }

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

__device__ __forceinline__ uint32_t map_to_rank(uint32_t saddr, int rank)
{
    uint32_t d;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(saddr), "r"(rank));
    return d;
}

// 16 bytes into another CTA's shared memory; its barrier `bar` counts them when they are there.
__device__ __forceinline__ void store_remote16(uint32_t dst, uint32_t bar, uint32_t a, uint32_t b, uint32_t c, uint32_t d)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%2,%3,%4,%5}, [%1];"
                 :: "r"(dst), "r"(bar), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}

// Four columns (col0 .. col0 + 3) of one output row from their accumulators: every output wanted.
__device__ __forceinline__ void epi_four(const EpiView &e, const int (&a)[4], const float (&sc)[4], const float (&bi)[4], uint32_t res,
                                         int64_t row, int64_t col0, bool full)
{
    const int64_t off = row * e.N + col0;
    const int cols = (int)(e.N - col0 < 4 ? e.N - col0 : 4);
    if (e.acc_out) {
        if (full) {
            *reinterpret_cast<int4 *>(e.acc_out + off) = make_int4(a[0], a[1], a[2], a[3]);
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (i < cols) e.acc_out[off + i] = a[i];
        }
    }
    if (!e.need_f) return;
    float y[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        y[i] = __fmaf_rn(__int2float_rn(a[i]), sc[i], bi[i]);
        if (e.residual) y[i] = __fmaf_rn(__uint2float_rn((res >> (8 * i)) & 0xFFu), e.residual_scale, y[i]);
        if (e.relu_op) y[i] = fmaxf(y[i], 0.0f);            // NaN -> 0, like (y > 0 ? y : 0)
    }
    if (e.f32_out) {
        if (full) {
            *reinterpret_cast<float4 *>(e.f32_out + off) = make_float4(y[0], y[1], y[2], y[3]);
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (i < cols) e.f32_out[off + i] = y[i];
        }
    }
    if (e.u8_out) {
        uint32_t w = requant_pack4(__fmul_rn(y[0], e.inv_out_scale), __fmul_rn(y[1], e.inv_out_scale),
                                   __fmul_rn(y[2], e.inv_out_scale), __fmul_rn(y[3], e.inv_out_scale));
        if (e.next_mode != SPARQ_MODE_NONE) w = next_xform_word(w, e.next_mode, e.next_rnd, e.next_xf);
        if (full) {
            *reinterpret_cast<uint32_t *>(e.u8_out + off) = w;
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (i < cols) e.u8_out[off + i] = (uint8_t)(w >> (8 * i));
        }
    }
}

template <int BK, int MODE, int XN, bool RND, bool SHARED>
__global__ void __launch_bounds__(kSmallThreads, 2)
sparq_gemm_small_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b, const GemmArgs g)
{
    constexpr int BN = kSmallBN;
    const int TM = g.tile_rows;                        // 64 or 128
    const int kABytes = TM * BK, kStageBytes = kABytes + BN * BK;
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bar_full[kMaxStages], bar_xf[kMaxStages], bar_empty[kMaxStages];
    __shared__ __align__(8) uint64_t bar_acc, bar_recv;
    __shared__ uint32_t tmem_base_slot;
    __shared__ uint32_t abort_word;
    __shared__ __align__(16) float s_scale[BN], s_bias[BN];

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    volatile uint32_t *abort_flag = &abort_word;
    const int S = g.stages;
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    auto a_stage = [&](int s) { return smem_base + (uint32_t)s * kStageBytes; };
    auto b_stage = [&](int s) { return smem_base + (uint32_t)s * kStageBytes + kABytes; };
    const uint32_t recv = smem_base + (uint32_t)(S * kStageBytes);         // SHARED: partial sums from the cluster

    // this CTA's tile, and its reduction steps
    const uint32_t split = SHARED ? (uint32_t)g.split : 1u;
    const uint32_t tile = SHARED ? blockIdx.x / split : blockIdx.x;
    const int rank = SHARED ? (int)(blockIdx.x - tile * split) : 0;
    const uint32_t n_tiles = (uint32_t)((g.N + BN - 1) / BN);
    const uint32_t mt = n_tiles == 1 ? tile : tile / n_tiles, nt = tile - mt * n_tiles;
    const int64_t m0 = (int64_t)mt * TM;
    const int n0 = (int)nt * BN;
    const int kb_first = SHARED ? rank * g.k_blocks / (int)split : 0;
    const int kb_last = SHARED ? (rank + 1) * g.k_blocks / (int)split : g.k_blocks;
    const int steps = kb_last - kb_first;
    const int rows_left = g.M - m0 < TM ? (int)(g.M - m0) : TM;          // valid rows of the tile

    if (warp == 0) {
        if (lane == 0) {
            prefetch_tensormap(&map_a);
            prefetch_tensormap(&map_b);
            for (int s = 0; s < S; ++s) {
                mbar_init(smem_u32(&bar_full[s]), 1);
                mbar_init(smem_u32(&bar_xf[s]), kSmallWorkers);
                mbar_init(smem_u32(&bar_empty[s]), 1);
            }
            mbar_init(smem_u32(&bar_acc), 1);
            mbar_init(smem_u32(&bar_recv), 1);
            abort_word = 0;
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        __syncwarp();
    } else if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(smem_u32(&tmem_base_slot)), "r"((uint32_t)BN) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = tmem_base_slot;
    // rows of the tile that this CTA writes
    const int own_rows = SHARED ? split_rows(g.M, TM, (int)split) : TM;
    int own_valid = rows_left - rank * own_rows;
    own_valid = own_valid < 0 ? 0 : own_valid > own_rows ? own_rows : own_valid;
    // (A launch with split = 1 has no clusters, and executes none of their instructions.)
    if (SHARED && split > 1) {
        if (threadIdx.x == 0) mbar_expect_tx(smem_u32(&bar_recv), split * (uint32_t)own_valid * (BN * 4));
        __syncwarp();
        cluster_arrive();       // "barriers ready": waited for before the first remote store
    }
    // Each role waits for the kernel before by itself, behind what it can work out without it (0.1 to 0.3 us of
    // a launch without a transform: 49 x 512, K 2048, 4.1 -> 3.8 us).
    if (warp == 0) {
        // ================= TMA producer =================
        if (lane == 0) {
            int base_w = 0, base_h = 0, base_n = 0;
            if (g.conv) {
                const uint32_t hw = (uint32_t)(g.Ho * g.Wo), m032 = (uint32_t)m0;
                base_n = (int)(m032 / hw);
                const int rem = (int)(m032 - (uint32_t)base_n * hw);
                base_h = (rem / g.Wo) * g.stride_h - g.pad_h;
                base_w = (rem % g.Wo) * g.stride_w - g.pad_w;
            }
            int it = 0, s = 0;
            uint32_t ph = 1;       // phase parity of bar_empty to wait for (1: the ring's first round needs none)
            TapWalk tap(g, BK, kb_first);
            dep_wait();
            dep_launch();
            for (; it < steps; ++it) {
                if (it >= S && !mbar_wait(smem_u32(&bar_empty[s]), ph, abort_flag, g.status, g.wait_limit)) break;
                const uint32_t full = smem_u32(&bar_full[s]);
                const int kx = g.conv ? tap.k : (kb_first + it) * BK;
                mbar_expect_tx(full, kStageBytes);
                if (g.conv) tma_load_im2col_4d(a_stage(s), &map_a, full, tap.c, base_w, base_h, base_n, (uint16_t)tap.s, (uint16_t)tap.r);
                else tma_load_2d(a_stage(s), &map_a, full, kx, (int)m0);
                if (it >= S) tma_load_2d(b_stage(s), &map_b, full, kx, n0);
                tap.next();
                if (++s == S) { s = 0; ph ^= 1u; }
            }
            if (*abort_flag)       // none of this thread's copies may land after the CTA has exited
                for (int j = it > S ? it - S : 0; j < it; ++j)
                    mbar_wait(smem_u32(&bar_full[j % S]), (uint32_t)(j / S) & 1u, abort_flag, g.status, g.wait_limit, true);
        }
        __syncwarp();
    } else if (warp == 1) {
        // ================= MMA issuer =================
        const uint32_t elected = elect_one();
        // The ring's first round of weights, beside the producer's activations: one thread takes about
        // 0.1 us a stage to issue both, in front of the first MMA.
        if (elected) {
            TapWalk tap(g, BK, kb_first);
            dep_wait();
            for (int it = 0; it < S && it < steps; ++it, tap.next())
                tma_load_2d(b_stage(it), &map_b, smem_u32(&bar_full[it]), g.conv ? tap.k : (kb_first + it) * BK, n0);
        }
        __syncwarp();
        const uint32_t idesc = make_idesc_i8(BN, TM);
        const uint64_t adesc0 = make_smem_desc<BK>(smem_base);
        const uint64_t bdesc0 = make_smem_desc<BK>(smem_base + kABytes);
        int s = 0;
        uint32_t ph = 0;
        for (int it = 0; it < steps; ++it) {
            mbar_wait(smem_u32(MODE == SPARQ_MODE_NONE ? &bar_full[s] : &bar_xf[s]), ph, abort_flag, g.status, g.wait_limit);
            tc_fence_after();
            const uint64_t off = (uint64_t)((uint32_t)s * (uint32_t)(kStageBytes >> 4));
#pragma unroll
            for (int k = 0; k < BK / 32; ++k)
                tc_mma_i8_if(tmem_base, adesc0 + off + (uint64_t)(k * 2), bdesc0 + off + (uint64_t)(k * 2), idesc,
                             (it > 0 || k > 0) ? 1u : 0u, elected);
            tc_commit_if(smem_u32(&bar_empty[s]), elected);
            if (++s == S) { s = 0; ph ^= 1u; }
        }
        tc_commit_if(smem_u32(&bar_acc), elected);
        mbar_wait(smem_u32(&bar_acc), 0, abort_flag, g.status, g.wait_limit, true);
        __syncwarp();
    } else {
        // ================= workers =================
        const EpiView ev = make_epi_view(g);
        const int wt = threadIdx.x - 64;                  // 0 .. 255
        // scale and bias on their way while the operands are
        float c_scale[4], c_bias[4];                      // SHARED: of this thread's four columns
        // Column groups of four that exist in this tile, and so rows that the workers write at a time: 512 x 10,
        // K 144, took 6.2 us where only the first three of sixteen threads on a row had columns, 3.2 so.
        const int groups = g.N - n0 < BN ? (int)(g.N - n0 + 3) / 4 : BN / 4;
        const int first_row = wt / groups, row_step = kSmallWorkers * 32 / groups;
        const int cg = wt - first_row * groups, fcol = n0 + cg * 4;
        const bool fvec = (g.N & 3) == 0 && (reinterpret_cast<uintptr_t>(g.residual) & 3u) == 0;
        dep_wait();
        if (ev.need_f) {
            if (SHARED) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const bool ok = fcol + i < g.N;
                    c_scale[i] = ok ? __ldg(g.scale + fcol + i) : 0.0f;
                    c_bias[i] = ok && g.bias ? __ldg(g.bias + fcol + i) : 0.0f;
                }
            } else if (wt < BN) {
                const bool ok = n0 + wt < g.N;
                c_scale[0] = ok ? __ldg(g.scale + n0 + wt) : 0.0f;
                c_bias[0] = ok && g.bias ? __ldg(g.bias + n0 + wt) : 0.0f;
            }
        }
        if (MODE != SPARQ_MODE_NONE) {
            const XformDev xf = g.xf;
            constexpr int kThreads = kSmallWorkers * 32, kPer = kBM * BK / 16 / kThreads;
            // Vectors that a thread works on at a time.  A launch starts with cold instruction caches, and the
            // transforms of 3- and 2-bit windows unrolled four times over are more code than the latency they hide is
            // worth (6opt: 256 x 64 x 576 6.95 -> 6.25 us, 7x7x512 -> 512 3x3, one image, 7.2 -> 6.4, 100 x 1000 x 4096 10.3 ->
            // 9.7); the shorter ones at n = 4 are better unrolled where the reduction is long (100 x 1000 x 4096 7.8 us, in
            // twos 8.3; 3opt 9.9 and 10.2).
            constexpr int kBatch = XN == 4 || XN == 5 ? kPer : 2;
            const int nvec = rows_left * (BK / 16);       // rows past M are padding: nothing to transform
            int s = 0;
            uint32_t ph = 0;
            for (int it = 0; it < steps; ++it) {
                mbar_wait(smem_u32(&bar_full[s]), ph, abort_flag, g.status, g.wait_limit);
                const uint32_t base = a_stage(s) + (uint32_t)wt * 16u;
                auto batch = [&](int j0) {
                    uint4 v[kBatch];
#pragma unroll
                    for (int j = 0; j < kBatch; ++j)
                        if (wt + (j0 + j) * kThreads < nvec)
                            asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v[j].x), "=r"(v[j].y), "=r"(v[j].z), "=r"(v[j].w)
                                         : "r"(base + (uint32_t)((j0 + j) * kThreads * 16)));
#pragma unroll
                    for (int j = 0; j < kBatch; ++j) {
                        if (wt + (j0 + j) * kThreads >= nvec) continue;
                        v[j].x = xform_fused<MODE, XN, RND>(v[j].x, xf);
                        v[j].y = xform_fused<MODE, XN, RND>(v[j].y, xf);
                        v[j].z = xform_fused<MODE, XN, RND>(v[j].z, xf);
                        v[j].w = xform_fused<MODE, XN, RND>(v[j].w, xf);
                        asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};"
                                     :: "r"(base + (uint32_t)((j0 + j) * kThreads * 16)), "r"(v[j].x), "r"(v[j].y), "r"(v[j].z), "r"(v[j].w) : "memory");
                    }
                };
                if constexpr (kBatch == kPer) {
                    batch(0);
                } else {
#pragma unroll 1
                    for (int j0 = 0; wt + j0 * kThreads < nvec; j0 += kBatch) batch(j0);
                }
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&bar_xf[s]));
                if (++s == S) { s = 0; ph ^= 1u; }
            }
        }
        const int quarter = warp & 3, half = (warp - 2) >> 2, cbase = half * 32;
        // tensor-memory lane -> tile row: all 32 lanes of a quarter, or its first 16 for 64-row tiles
        const int trow = TM == 64 ? (lane < 16 ? quarter * 16 + lane : TM) : quarter * 32 + lane;
        const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)cbase;
        auto wait_acc = [&]() {
            mbar_wait(smem_u32(&bar_acc), 0, abort_flag, g.status, g.wait_limit);
            tc_fence_after();
        };
        if constexpr (!SHARED) {
            if (ev.need_f) {
                if (wt < BN) { s_scale[wt] = c_scale[0]; s_bias[wt] = c_bias[0]; }
                asm volatile("bar.sync 1, %0;" :: "n"(kSmallWorkers * 32) : "memory");
            }
            // (handing the accumulator back is not needed here: the barrier named is never waited for)
            if (ev.out == kOutResidual)
                epi_warp_columns<kOutResidual>(ev, taddr, cbase, 32, m0 + trow, trow < rows_left, n0, s_scale, s_bias, smem_u32(&bar_recv), lane, wait_acc);
            else
                epi_warp_columns<kOutBytes>(ev, taddr, cbase, 32, m0 + trow, trow < rows_left, n0, s_scale, s_bias, smem_u32(&bar_recv), lane, wait_acc);
        } else {
            // residual bytes of this thread's four columns of the CTA's row lrow
            auto residual_of = [&](int lrow) {
                uint32_t r = 0u;
                if (!g.residual || lrow >= own_valid || fcol >= g.N) return r;
                const uint8_t *src = g.residual + (m0 + rank * own_rows + lrow) * g.N + fcol;
                if (fvec) return __ldg(reinterpret_cast<const uint32_t *>(src));
                for (int q = 0; q < 4 && fcol + q < g.N; ++q) r |= (uint32_t)__ldg(src + q) << (8 * q);
                return r;
            };
            uint32_t r = residual_of(first_row);
            const uint32_t gbytes = (uint32_t)split_group_bytes(own_rows), rbytes = (uint32_t)split_rank_bytes(own_rows);
            wait_acc();
            uint32_t v[32];
            tmem_ld_32x32_issue(taddr, v);
            if (split == 1) {
                tmem_ld_wait();
                if (trow < rows_left) {
                    const uint32_t dst = recv + (uint32_t)(cbase / 4) * gbytes + (uint32_t)trow * 16u;
#pragma unroll
                    for (int q = 0; q < 8; ++q)
                        asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" :: "r"(dst + (uint32_t)q * gbytes), "r"(v[4 * q]),
                                     "r"(v[4 * q + 1]), "r"(v[4 * q + 2]), "r"(v[4 * q + 3]) : "memory");
                }
                asm volatile("bar.sync 1, %0;" :: "n"(kSmallWorkers * 32) : "memory");
            } else {
                __syncwarp();
                cluster_wait();        // every CTA of the cluster has its barriers ready
                tmem_ld_wait();
                if (trow < rows_left) {
                    const int owner = trow / own_rows, lrow = trow - owner * own_rows;
                    const uint32_t dst = map_to_rank(recv + (uint32_t)rank * rbytes, owner) + (uint32_t)(cbase / 4) * gbytes + (uint32_t)lrow * 16u;
                    const uint32_t bar = map_to_rank(smem_u32(&bar_recv), owner);
#pragma unroll
                    for (int q = 0; q < 8; ++q)
                        store_remote16(dst + (uint32_t)q * gbytes, bar, v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
                }
                mbar_wait(smem_u32(&bar_recv), 0, abort_flag, g.status, g.wait_limit);
            }
            if (first_row < row_step) {        // the last threads have no place in a step
                for (int lrow = first_row; lrow < own_valid; lrow += row_step) {
                    const uint32_t src = recv + (uint32_t)cg * gbytes + (uint32_t)lrow * 16u;
                    int p[kMaxSplit][4];
#pragma unroll
                    for (int q = 0; q < kMaxSplit; ++q) {
                        p[q][0] = p[q][1] = p[q][2] = p[q][3] = 0;
                        if (q < (int)split)
                            asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(p[q][0]), "=r"(p[q][1]), "=r"(p[q][2]), "=r"(p[q][3])
                                         : "r"(src + (uint32_t)q * rbytes));
                    }
                    const uint32_t r_next = residual_of(lrow + row_step);
                    int a[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        a[k] = ((p[0][k] + p[1][k]) + (p[2][k] + p[3][k])) + ((p[4][k] + p[5][k]) + (p[6][k] + p[7][k]));
                    epi_four(ev, a, c_scale, c_bias, r, m0 + rank * own_rows + lrow, fcol, fvec);
                    r = r_next;
                }
            }
        }
        tc_fence_before();
    }
    if (SHARED && split > 1 && warp < 2) {
        __syncwarp();
        cluster_wait();            // matches the arrival above
    }
    __syncthreads();
    // No CTA leaves while a peer may still write to its shared memory.  In a normal run its barrier has
    // counted every byte by now; a CTA that gave up a wait comes here early.  It stays until every
    // other CTA of the cluster has left or is here too (both after its last remote store: every CTA
    // sends all its rows, given up or not, and reaches this point by bounded waits only), and then
    // until the bytes still on their way have landed.  All waits of the CTA lie before the barrier
    // above, so its threads agree on the flag.  (A second cluster barrier in every run cost 0.1 us.)
    if (SHARED && split > 1 && *abort_flag) {
        __syncwarp();
        cluster_arrive();
        cluster_wait();
        mbar_wait(smem_u32(&bar_recv), 0, abort_flag, g.status, g.wait_limit, true);
    }
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem_base), "r"((uint32_t)BN) : "memory");
    }
}

// Host launcher; defined once per BK in its own translation unit.
template <int BK>
cudaError_t launch_gemm_small(const GemmMaps &m, GemmArgs &g, int mode, int n, int rnd, int grid, cudaStream_t st);

template <int BK, int MODE, int XN, bool RND, bool SHARED>
cudaError_t launch_gemm_small_kernel(const GemmMaps &m, GemmArgs &g, int grid, cudaStream_t st)
{
    auto kfn = sparq_gemm_small_kernel<BK, MODE, XN, RND, SHARED>;
    static bool attr_set[64] = {};   // per device ordinal
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64 || !attr_set[dev]) {
        e = cudaFuncSetAttribute(kfn, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmallMaxDynSmem);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) attr_set[dev] = true;
    }
    const int stage = (g.tile_rows + kSmallBN) * BK;
    const int recv = SHARED ? g.split * split_rank_bytes(split_rows(g.M, g.tile_rows, g.split)) : 0;
    const int steps = (g.k_blocks + g.split - 1) / g.split, fit = (kSmallMaxDynSmem - 1024 - recv) / stage;
    g.stages = steps < fit ? steps : fit;        // no more stages than the CTA has reduction steps
    if (g.stages > kMaxStages) g.stages = kMaxStages;
    return launch_overlapped_cluster(kfn, grid, g.split, kSmallThreads, 1024 + g.stages * stage + recv, st, m.a, m.b, g);
}

#define SPARQ_LAUNCH_SMALL(MODE_, XN_, RND_)                                                           \
    return g.split > 1 || make_epi_view(g).out == kOutGeneral ? launch_gemm_small_kernel<BK, MODE_, XN_, RND_, true>(m, g, grid, st)          \
                       : launch_gemm_small_kernel<BK, MODE_, XN_, RND_, false>(m, g, grid, st)

#define SPARQ_DEFINE_GEMM_SMALL(BK_)                                                                   \
    template <>                                                                                        \
    cudaError_t launch_gemm_small<BK_>(const GemmMaps &m, GemmArgs &g, int mode, int n, int rnd,       \
                                       int grid, cudaStream_t st)                                      \
    {                                                                                                  \
        constexpr int BK = BK_;                                                                        \
        if (mode == SPARQ_MODE_NONE) SPARQ_LAUNCH_SMALL(SPARQ_MODE_NONE, 4, false);                    \
        if (mode == SPARQ_MODE_BSPARQ) {                                                               \
            if (n == 8) SPARQ_LAUNCH_SMALL(SPARQ_MODE_BSPARQ, 8, true);                                \
            if (n == 5 && rnd) SPARQ_LAUNCH_SMALL(SPARQ_MODE_BSPARQ, 5, true);                         \
            if (n == 5) SPARQ_LAUNCH_SMALL(SPARQ_MODE_BSPARQ, 5, false);                               \
            if (n == 4 && rnd) SPARQ_LAUNCH_SMALL(SPARQ_MODE_BSPARQ, 4, true);                         \
            if (n == 4) SPARQ_LAUNCH_SMALL(SPARQ_MODE_BSPARQ, 4, false);                               \
            if (rnd) SPARQ_LAUNCH_SMALL(SPARQ_MODE_BSPARQ, 0, true);                                   \
            SPARQ_LAUNCH_SMALL(SPARQ_MODE_BSPARQ, 0, false);                                           \
        }                                                                                              \
        if (n == 8) SPARQ_LAUNCH_SMALL(SPARQ_MODE_VSPARQ, 8, true);                                    \
        if (n == 5 && rnd) SPARQ_LAUNCH_SMALL(SPARQ_MODE_VSPARQ, 5, true);                             \
        if (n == 5) SPARQ_LAUNCH_SMALL(SPARQ_MODE_VSPARQ, 5, false);                                   \
        if (n == 4 && rnd) SPARQ_LAUNCH_SMALL(SPARQ_MODE_VSPARQ, 4, true);                             \
        if (n == 4) SPARQ_LAUNCH_SMALL(SPARQ_MODE_VSPARQ, 4, false);                                   \
        if (rnd) SPARQ_LAUNCH_SMALL(SPARQ_MODE_VSPARQ, 0, true);                                       \
        SPARQ_LAUNCH_SMALL(SPARQ_MODE_VSPARQ, 0, false);                                               \
    }

}  // namespace sparq
