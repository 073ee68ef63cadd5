// Product with 2:4 sparse weights and vSPARQ on the selected pairs, in one kernel: the expansion of
// the activations (six candidate pairs per group of four, 12 bytes per 4; sparq_sparse24.cu) happens
// between shared memory and shared memory instead of through HBM.
//
// A CTA takes tiles of 256 rows x BN columns (two 128-row accumulators that share every weight
// block).  Warps:
//   0        TMA producer: raw activations (256 rows x 128 bytes) into a ring of two, expanded
//            weights (BN rows x 128 bytes of K' = 3K) into the expanded stages
//   1        tensor memory, MMA issue: 8 MMAs per expanded stage
//   2..5     epilogue
//   6..21    expansion: a thread owns one row and four of its eight 16-byte pieces; each piece (four
//            groups) becomes 48 bytes, so a raw stage becomes exactly three expanded ones (threads of
//            the first half fill stage 0 and the first half of stage 1, the others the rest)
// The expansion is what bounds it: per four activations one bSPARQ transform (11
// instructions at n = 4) and, for each of three output words, a permuted copy of the transformed and
// of the raw bytes, a permuted mask of "partner is non-zero" and a select -- 26 instructions
// where transforming each of the six pairs took 57 -- and 256-row tiles halve the weight traffic
// out of L2, which would bound it otherwise.  The two-kernel form moved 3 bytes per activation
// to HBM and back.  M 100352, K 1152: N 128 164 -> 62 us, N 64 161 -> 60, N 256 176 -> 114;
// N 128 with 3opt 219 -> 71, 6opt 253 -> 69.  (Expanded into tensor memory instead of shared memory: N 128 62, N 256
// 117, K 512 N 512 107 in place of 99.)
#pragma once

#include "sparq_gemm_kernel.cuh"
#include "sparq_expand24.cuh"

namespace sparq {

constexpr int kX24Rows = 256;
constexpr int kX24EpiWarps = 4, kX24XfWarps = 16;
constexpr int kX24FirstXf = 2 + kX24EpiWarps;
constexpr int kX24Threads = 32 * (kX24FirstXf + kX24XfWarps);
constexpr int kX24RawBytes = kX24Rows * 128;
constexpr int kX24RawStages = 2, kX24Stages = 3;

template <int BN>
struct X24Cfg {
    static constexpr int kStageBytes = kX24RawBytes + BN * 128;      // expanded activations, weights
    static constexpr int kSmemBytes = 1024 + kX24RawStages * kX24RawBytes + kX24Stages * kStageBytes;
    static constexpr int kTmemCols = 4 * BN;                          // two tiles of two accumulators
};

// OUT: kOutBytes, or kOutGeneral for every other kind of output.
template <int BN, int XN, bool RND, int OUT>
__global__ void __launch_bounds__(kX24Threads, 1)
sparq_gemm_sparse24_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b, const GemmArgs g)
{
    using Cfg = X24Cfg<BN>;
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bar_raw_full[kX24RawStages], bar_raw_empty[kX24RawStages];
    __shared__ __align__(8) uint64_t bar_w_full[kX24Stages], bar_x_full[kX24Stages], bar_empty[kX24Stages];
    __shared__ __align__(8) uint64_t bar_acc_full[2], bar_acc_empty[2], bar_done;
    __shared__ uint32_t tmem_base_slot;
    __shared__ uint32_t abort_word;
    __shared__ __align__(16) float s_scale[BN], s_bias[BN];

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    volatile uint32_t *abort_flag = &abort_word;
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    auto raw_stage = [&](int s) { return smem_base + (uint32_t)(s * kX24RawBytes); };
    const uint32_t exp_base = smem_base + (uint32_t)(kX24RawStages * kX24RawBytes);
    auto x_stage = [&](int s) { return exp_base + (uint32_t)(s * Cfg::kStageBytes); };
    auto w_stage = [&](int s) { return x_stage(s) + (uint32_t)kX24RawBytes; };

    const uint32_t n_tiles = (uint32_t)((g.N + BN - 1) / BN);
    const uint32_t total_tiles = (uint32_t)((g.M + kX24Rows - 1) / kX24Rows) * n_tiles;
    const int steps = g.k_blocks;          // raw steps of 128 activations = three expanded ones each

    if (threadIdx.x == 0) {
        prefetch_tensormap(&map_a);
        prefetch_tensormap(&map_b);
        for (int s = 0; s < kX24RawStages; ++s) {
            mbar_init(smem_u32(&bar_raw_full[s]), 1);
            mbar_init(smem_u32(&bar_raw_empty[s]), kX24XfWarps);
        }
        for (int s = 0; s < kX24Stages; ++s) {
            mbar_init(smem_u32(&bar_w_full[s]), 1);
            mbar_init(smem_u32(&bar_x_full[s]), s == 1 ? kX24XfWarps : kX24XfWarps / 2);
            mbar_init(smem_u32(&bar_empty[s]), 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(smem_u32(&bar_acc_full[a]), 1);
            mbar_init(smem_u32(&bar_acc_empty[a]), 2 * kX24EpiWarps);      // once per accumulator and warp
        }
        mbar_init(smem_u32(&bar_done), 1);
        abort_word = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(smem_u32(&tmem_base_slot)), "r"((uint32_t)Cfg::kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = tmem_base_slot;
    if (warp == 0) {
        // ================= TMA producer =================
        if (lane == 0) {
            uint32_t ri = 0, wi = 0;          // raw and weight stages issued
            uint32_t use = 0;                 // raw steps issued before this one
            bool live = true;
            for (uint32_t tile = blockIdx.x; tile < total_tiles && live; tile += gridDim.x) {
                const uint32_t mt = n_tiles == 1 ? tile : tile / n_tiles;
                const int n0 = (int)(tile - mt * n_tiles) * BN, m0 = (int)mt * kX24Rows;
                // every role waits for the kernel before, in front of its first access or bounded wait (later waits return at
                // once); EARLY waits in the roles that need not cost 1.5 % here
                dep_wait();
                dep_launch();
                for (int kb = 0; kb < steps && live; ++kb, ++use) {
                    const int s = (int)(use & 1u);
                    if (use >= 2 && !mbar_wait(smem_u32(&bar_raw_empty[s]), ((use >> 1) - 1u) & 1u, abort_flag, g.status, g.wait_limit)) { live = false; break; }
                    const uint32_t full = smem_u32(&bar_raw_full[s]);
                    mbar_expect_tx(full, kX24RawBytes);
                    tma_load_2d(raw_stage(s), &map_a, full, kb * 128, m0);
                    ++ri;
                    for (int j = 0; j < 3; ++j) {
                        if (use > 0 && !mbar_wait(smem_u32(&bar_empty[j]), (use - 1u) & 1u, abort_flag, g.status, g.wait_limit)) { live = false; break; }
                        mbar_expect_tx(smem_u32(&bar_w_full[j]), BN * 128);
                        tma_load_2d(w_stage(j), &map_b, smem_u32(&bar_w_full[j]), kb * 384 + j * 128, n0);
                        ++wi;
                    }
                }
            }
            if (*abort_flag) {       // none of this thread's copies may land after the CTA has exited
                for (uint32_t q = ri > 2 ? ri - 2 : 0; q < ri; ++q)
                    mbar_wait(smem_u32(&bar_raw_full[q & 1u]), (q >> 1) & 1u, abort_flag, g.status, g.wait_limit, true);
                for (uint32_t q = wi > 3 ? wi - 3 : 0; q < wi; ++q)
                    mbar_wait(smem_u32(&bar_w_full[q % 3u]), (q / 3u) & 1u, abort_flag, g.status, g.wait_limit, true);
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ================= MMA issuer =================
        const uint32_t elected = elect_one();
        constexpr uint32_t idesc = make_idesc_i8(BN);
        uint32_t local_tile = 0, ph = 0;
        dep_wait();
        for (uint32_t tile = blockIdx.x; tile < total_tiles; tile += gridDim.x, ++local_tile) {
            const uint32_t acc = local_tile & 1u, acc_use = local_tile >> 1;
            if (acc_use > 0) mbar_wait(smem_u32(&bar_acc_empty[acc]), (acc_use - 1u) & 1u, abort_flag, g.status, g.wait_limit);
            tc_fence_after();
            const uint32_t d_tmem = tmem_base + acc * (uint32_t)(2 * BN);
            for (int kb = 0; kb < steps; ++kb, ph ^= 1u) {
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    mbar_wait(smem_u32(&bar_w_full[j]), ph, abort_flag, g.status, g.wait_limit);
                    mbar_wait(smem_u32(&bar_x_full[j]), ph, abort_flag, g.status, g.wait_limit);
                    tc_fence_after();
                    const uint64_t adesc = make_smem_desc<128>(x_stage(j)), bdesc = make_smem_desc<128>(w_stage(j));
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            tc_mma_i8_if(d_tmem + (uint32_t)(h * BN), adesc + (uint64_t)(h * (kBM * 128 >> 4) + k * 2),
                                         bdesc + (uint64_t)(k * 2), idesc, (kb > 0 || j > 0 || k > 0) ? 1u : 0u, elected);
                    tc_commit_if(smem_u32(&bar_empty[j]), elected);
                }
            }
            tc_commit_if(smem_u32(&bar_acc_full[acc]), elected);
        }
        tc_commit_if(smem_u32(&bar_done), elected);
        mbar_wait(smem_u32(&bar_done), 0, abort_flag, g.status, g.wait_limit, true);
        __syncwarp();
    } else if (warp < kX24FirstXf) {
        // ================= epilogue =================
        const int quarter = warp & 3;
        const int et = threadIdx.x - 64;
        const EpiView ev = make_epi_view(g);
        int64_t staged_nt = -1;
        uint32_t local_tile = 0;
        dep_wait();
        for (uint32_t tile = blockIdx.x; tile < total_tiles; tile += gridDim.x, ++local_tile) {
            const uint32_t mt = n_tiles == 1 ? tile : tile / n_tiles;
            const int64_t nt = tile - mt * n_tiles;
            const uint32_t acc = local_tile & 1u, ph = (local_tile >> 1) & 1u;
            if (ev.need_f && nt != staged_nt) {
                staged_nt = nt;
                epi_stage_scale_bias(g, nt * BN, BN, et, kX24EpiWarps * 32, 1, s_scale, s_bias);
            }
            for (int h = 0; h < 2; ++h) {
                const int64_t row = (int64_t)mt * kX24Rows + h * kBM + quarter * 32 + lane;
                const uint32_t taddr0 = tmem_base + ((uint32_t)(quarter * 32) << 16) + acc * (uint32_t)(2 * BN) + (uint32_t)(h * BN);
                auto wait_full = [&]() {
                    mbar_wait(smem_u32(&bar_acc_full[acc]), ph, abort_flag, g.status, g.wait_limit);
                    tc_fence_after();
                };
                const uint32_t empty = smem_u32(&bar_acc_empty[acc]);
                epi_warp_columns<OUT>(ev, taddr0, 0, BN, row, row < g.M, nt * BN, s_scale, s_bias, empty, lane, wait_full);
            }
        }
    } else {
        // ================= expansion =================
        const int xw = warp - kX24FirstXf, half = xw >> 3;                // half 0: pieces 0..3 of a row, 1: pieces 4..7
        const uint32_t row = (uint32_t)((xw & 7) * 32 + lane), swz = row & 7u;
        const XformDev xf = g.xf;
        uint32_t use = 0;
        // stages this half fills, first and second
        const int s0 = half ? 1 : 0, s1 = half ? 2 : 1;
        dep_wait();
        for (uint32_t tile = blockIdx.x; tile < total_tiles; tile += gridDim.x) {
            const uint32_t mt = n_tiles == 1 ? tile : tile / n_tiles;
            const bool live_row = (int64_t)mt * kX24Rows + (xw & 7) * 32 < g.M;      // any row of this warp
            for (int kb = 0; kb < steps; ++kb, ++use) {
                const int rs = (int)(use & 1u);
                mbar_wait(smem_u32(&bar_raw_full[rs]), (use >> 1) & 1u, abort_flag, g.status, g.wait_limit);
                uint4 v[4];
                if (live_row) {
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v[j].x), "=r"(v[j].y), "=r"(v[j].z), "=r"(v[j].w)
                                     : "r"(raw_stage(rs) + row * 128u + ((((uint32_t)(half * 4 + j)) ^ swz) << 4)));
                }
                auto wait_stage = [&](int s) {
                    if (use > 0) mbar_wait(smem_u32(&bar_empty[s]), (use - 1u) & 1u, abort_flag, g.status, g.wait_limit);
                };
                auto signal_stage = [&](int s) {
                    fence_proxy_async_smem();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&bar_x_full[s]));
                };
                wait_stage(s0);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    // output pieces 3j .. 3j + 2 of this half's twelve; half 0: 0..7 in stage 0, 8..11 in
                    // stage 1 (chunks 0..3); half 1: 0..3 in stage 1 (chunks 4..7), 4..11 in stage 2
                    uint32_t o[12];
                    if (live_row) {
                        expand_group<XN, RND>(v[j].x, xf, o[0], o[1], o[2]);
                        expand_group<XN, RND>(v[j].y, xf, o[3], o[4], o[5]);
                        expand_group<XN, RND>(v[j].z, xf, o[6], o[7], o[8]);
                        expand_group<XN, RND>(v[j].w, xf, o[9], o[10], o[11]);
                    }
#pragma unroll
                    for (int i = 0; i < 3; ++i) {
                        const int p = 3 * j + i;
                        // the first piece of the second stage: the first one is complete
                        if (p == (half ? 4 : 8)) { signal_stage(s0); wait_stage(s1); }
                        const bool second = p >= (half ? 4 : 8);
                        const uint32_t chunk = (uint32_t)((half * 12 + p) & 7);
                        const uint32_t dst = x_stage(second ? s1 : s0) + row * 128u + ((chunk ^ swz) << 4);
                        if (live_row)
                            asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};"
                                         :: "r"(dst), "r"(o[4 * i]), "r"(o[4 * i + 1]), "r"(o[4 * i + 2]), "r"(o[4 * i + 3]) : "memory");
                    }
                }
                signal_stage(s1);
                if (lane == 0) mbar_arrive(smem_u32(&bar_raw_empty[rs]));
            }
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem_base), "r"((uint32_t)Cfg::kTmemCols) : "memory");
    }
}

}  // namespace sparq
