// Stride-1 R x S convolution with the activation transform applied once per staged input
// row ("window" kernel).
//
// The im2col form of the fused kernel stages a shifted copy of the input for every filter
// tap, so every input byte is copied into shared memory and transformed R*S times.  Here a
// CTA's output tile is TR whole output rows of one image, laid out with the PADDED width
// Wp = W + 2*pad_w (slot i = tr * Wp + ow; the S-1 slots at the end of each row are junk and
// are never stored).  With that layout tap (r, s) of slot i reads padded-input pixel
// i + r*Wp + s: every tap is the SAME shared-memory matrix shifted by r*Wp + s rows.
//
// Up to G consecutive tiles of one image form a GROUP that shares one window buffer of
// G*TR + R-1 input rows, so the R-1 halo rows between neighbouring tiles are staged and
// transformed once instead of once per tile.  The window arrives in pieces -- the first is
// TR+R-1 rows, every later one TR rows -- each with its own pair of barriers, and tile j of
// the group needs pieces 0..j only: the tensor core starts on the first tile while later
// pieces are still in flight or being transformed.
//   * tiled TMA boxes (CB channels x Wp x piece rows, zero fill outside the image) bring the
//     pieces in, once per channel block; the swizzle of a box is a function of the
//     shared-memory address, so pieces written at consecutive row offsets form one
//     consistently swizzled matrix,
//   * the transform warps rewrite each piece in place once (bSPARQ / vSPARQ, Sections 3.1-3.2),
//   * the MMA warp issues tcgen05.mma kind::i8 for every (channel block, tap) with an A
//     descriptor whose start address is advanced by (j*TR*Wp + r*Wp + s) rows.
// Each CTA owns a contiguous range of the tile sequence (balanced to within one tile) and
// cuts it into groups at image boundaries.
// Weights either stay resident in shared memory for the whole kernel (B_RESIDENT: all
// R*S*C/CB blocks of BN x CB, loaded once per CTA) or stream through a ring of stages.
// Warp roles, bounded waits and the epilogue are those of sparq_gemm_kernel.
#pragma once

#include "sparq_gemm_kernel.cuh"

namespace sparq {

struct WindowArgs {
    // GEMM view for the epilogue
    int64_t N;              // cout
    int64_t K;              // r * s * c
    // geometry
    int n_img, H, W, C, R, S, pad_h, pad_w, Ho, Wo;
    int Wp;                 // W + 2 * pad_w, rounded up to even where that costs no row (host)
    int TR;                 // output rows per tile
    int tiles_per_img;      // ceil(Ho / TR)
    int c_blocks;           // ceil(C / CB); channels past C arrive as zeros, activations and weights alike
    int G;                  // most tiles that share one window (1 when there are several column tiles)
    int piece0_bytes;       // CB * Wp * (TR + R - 1): first piece of a group, one channel block
    int piece_bytes;        // CB * Wp * TR: every later piece
    int plane_bytes;        // shared-memory bytes reserved per channel block (>= rows the MMA may touch)
    int win_bufs;           // window buffers in the ring
    int b_stages;           // weight stages (stream mode) or resident blocks (resident mode)
    int team_copy;          // 256-wide tiles: room behind the weight stages for the second epilogue team's scale and bias
    uint32_t n_tiles;       // column tiles
    uint32_t units;         // n_img * tiles_per_img * n_tiles, column tile fastest
    uint32_t groups;        // streamed weights on 128-wide tiles: n_img * n_tiles * ceil(tiles_per_img / G) whole
                            // groups of up to G row tiles of one (image, column tile), which share one pass over
                            // the weights; CTAs own whole groups there, contiguous shares of the unit sequence else
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
    const uint8_t *residual;
    float residual_scale;
};

// dynamic shared memory the kernel may ask for: 227 KB minus room for its static variables
constexpr int kWindowMaxDynSmem = 232448 - 4096;
// With streamed weights the epilogue teams keep scale and bias of their own column tiles.  On 256-wide
// tiles the second team's lie in dynamic memory, where there is room (else one team): as static
// variables they took a stage of the ring, or the whole kernel, from shapes that just fit
// (64x35x35x384 -> 192 3x3 102 us, by the im2col kernel 150).
constexpr int kTeamCopyBytes = 2 * 256 * 4;
constexpr int kMaxWinBufs = 4;
constexpr int kMaxG = 8;
constexpr int kMaxBStages = 12;
// Two warps issue MMAs, taking the tiles of a CTA alternately (each owns one of the two
// accumulators): whatever one of them does between two tiles -- commits, barrier reads that
// queue behind the tensor core's own shared-memory traffic, descriptor set-up -- happens
// while the other one's MMAs keep the tensor core busy.
constexpr int kMmaBWarp = kFirstXfWarp + kNumXfWarps;      // the second issuer is the last warp
constexpr int kWindowThreads = 32 * (kMmaBWarp + 1);

__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap *map, uint32_t bar, int c, int w, int h, int n)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
        :: "r"(dst), "l"(map), "r"(bar), "r"(c), "r"(w), "r"(h), "r"(n) : "memory");
}

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap *map, uint32_t bar, int x, int y, int z)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
        :: "r"(dst), "l"(map), "r"(bar), "r"(x), "r"(y), "r"(z) : "memory");
}

// Walks the groups of one CTA's share of the tile sequence.  Every warp role runs the same
// walk, so that window buffers, accumulators and barrier phases line up without any
// communication.
template <bool BY_GROUP>
struct GroupWalk {
    uint32_t u, u_end;          // units (BY_GROUP: whole groups) still to do: [u, u_end)
    uint32_t n_tiles, tpi, G;
    uint32_t img, tin, nt, cnt; // current group: image, first tile inside it, column tile, tiles

    __device__ __forceinline__ GroupWalk(const WindowArgs &g)
    {
        // the sequence is split into gridDim.x contiguous shares that differ by at most one
        const uint32_t total = BY_GROUP ? g.groups : g.units;
        const uint32_t q = total / gridDim.x, rem = total - q * gridDim.x;
        u = blockIdx.x * q + (blockIdx.x < rem ? blockIdx.x : rem);
        u_end = u + q + (blockIdx.x < rem ? 1u : 0u);
        n_tiles = g.n_tiles; tpi = (uint32_t)g.tiles_per_img; G = (uint32_t)g.G;
        img = tin = nt = cnt = 0;
    }
    __device__ __forceinline__ bool next()
    {
        if (u >= u_end) return false;
        if (BY_GROUP) {
            // group number u = (image * n_tiles + column tile) * gpt + k: tiles k*G .. of that image
            const uint32_t gpt = (tpi + G - 1) / G;
            const uint32_t key = u / gpt, k = u - key * gpt;
            img = key / n_tiles;
            nt = key - img * n_tiles;
            tin = k * G;
            cnt = tpi - tin < G ? tpi - tin : G;
            u += 1;
            return true;
        }
        uint32_t mt = u;
        nt = 0;
        if (n_tiles != 1) { mt = u / n_tiles; nt = u - mt * n_tiles; }
        img = mt / tpi;
        tin = mt - img * tpi;
        uint32_t c = 1;
        if (n_tiles == 1) {
            c = tpi - tin;
            if (c > G) c = G;
            if (c > u_end - u) c = u_end - u;
        }
        cnt = c;
        u += c;
        return true;
    }
};

template <int BN, int CB, int MODE, int XN, bool RND, bool B_RESIDENT, int OUT>
__global__ void __launch_bounds__(kWindowThreads, 1)
sparq_conv_window_kernel(const __grid_constant__ CUtensorMap map_x0, const __grid_constant__ CUtensorMap map_x1,
                         const __grid_constant__ CUtensorMap map_w, const WindowArgs g)
{
    extern __shared__ uint8_t smem_raw[];
    // one pair per (window buffer, piece): bytes landed / piece transformed
    __shared__ __align__(8) uint64_t bar_win_full[kMaxWinBufs * kMaxG], bar_win_xf[kMaxWinBufs * kMaxG];
    __shared__ __align__(8) uint64_t bar_win_empty[kMaxWinBufs];
    __shared__ __align__(8) uint64_t bar_b_full[kMaxBStages], bar_b_empty[kMaxBStages];
    // Accumulator stages in tensor memory; tile number t uses stage t % kAcc.  Streamed weights on
    // 128-wide tiles: the tiles of a group are accumulated TOGETHER during one pass over the
    // weights (kBatched), so a group holds up to two stages and four let the next group start
    // while the previous one is in its epilogue.
    constexpr bool kBatched = !B_RESIDENT && BN == 128;
    // Streamed weights pass through a ring that is shorter than one tile's blocks, in tile order:
    // two issuers on different tiles would wait on the same stage barriers several phases apart,
    // which a parity wait cannot tell apart.  One issuer then; two take the tiles alternately with
    // resident weights.
    constexpr uint32_t kIssuers = B_RESIDENT ? 2 : 1;
    // 128-wide tiles without a transform keep one team of sixteen warps and, with resident weights, two
    // stages: nothing slows the issuers down there, so with four stages they finish tiles in pairs
    // and the epilogues run after them in a burst (128x28x28x128 -> 128 3x3: 16.5 -> 15.2 us).
    constexpr bool kOneTeam = BN == 128 && MODE == SPARQ_MODE_NONE;
    constexpr int kAcc = BN == 256 || (kOneTeam && B_RESIDENT) ? 2 : 4;
    // epilogue teams: as in sparq_gemm_kernel
    constexpr int kGroups = epi_warps(MODE) / 4;
    constexpr int kMaxTeams = kOneTeam ? 1 : kGroups < kAcc ? kGroups : kAcc;
    const int teams = kMaxTeams > 1 && g.units > gridDim.x && (BN != 256 || g.team_copy) ? kMaxTeams : 1;
    __shared__ __align__(8) uint64_t bar_acc_full[kAcc], bar_acc_empty[kAcc], bar_done;
    __shared__ uint32_t tmem_base_slot;
    __shared__ uint32_t abort_word;
    // one column tile (resident weights): the teams share one copy, all writing the same values
    constexpr int kCopies = B_RESIDENT || BN == 256 ? 1 : kMaxTeams;
    __shared__ __align__(16) float s_scale_all[kCopies][BN], s_bias_all[kCopies][BN];

    constexpr int kBBlock = BN * CB;                   // one (tap, channel block) of weights
    constexpr int kTmemCols = kAcc * BN;
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    volatile uint32_t *abort_flag = &abort_word;

    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t win_bytes = (uint32_t)g.plane_bytes * (uint32_t)g.c_blocks;
    auto win_buf = [&](int b) { return smem_base + (uint32_t)b * win_bytes; };
    const uint32_t b_base = smem_base + (uint32_t)g.win_bufs * win_bytes;
    auto b_slot = [&](int s) { return b_base + (uint32_t)s * kBBlock; };
    // byte offset of piece j inside a channel block's plane, and its size
    auto piece_off = [&](int j) { return j ? (uint32_t)((j * g.TR + g.R - 1) * g.Wp * CB) : 0u; };
    auto piece_len = [&](int j) { return (uint32_t)(j ? g.piece_bytes : g.piece0_bytes); };

    const int taps = g.R * g.S;
    const int kb_count = taps * g.c_blocks;            // weight blocks per tile
    if (threadIdx.x == 0) {
        prefetch_tensormap(&map_x0);
        prefetch_tensormap(&map_x1);
        prefetch_tensormap(&map_w);
    }
    if (warp == 0) {
        // barrier set-up spread over the lanes of one warp
        for (int b = lane; b < kMaxWinBufs * kMaxG; b += 32) {
            mbar_init(smem_u32(&bar_win_full[b]), 1);
            mbar_init(smem_u32(&bar_win_xf[b]), kNumXfWarps);
        }
        if (lane < kMaxWinBufs) mbar_init(smem_u32(&bar_win_empty[lane]), 2);     // one arrival per issuing warp
        if (lane < kMaxBStages) {
            mbar_init(smem_u32(&bar_b_full[lane]), 1);
            mbar_init(smem_u32(&bar_b_empty[lane]), 1);
        }
        if (lane < kAcc) {
            mbar_init(smem_u32(&bar_acc_full[lane]), 1);
            mbar_init(smem_u32(&bar_acc_empty[lane]), 4 * epi_parts(kGroups, teams, BN));
        }
        if (lane == 0) {
            mbar_init(smem_u32(&bar_done), 2);
            abort_word = 0;
        }
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
    // this CTA's share of the tile sequence: kernel arguments only, so it is worked out (two
    // integer divisions) while the previous kernel may still be running
    GroupWalk<kBatched> walk(g);
    bool have = walk.next();       // the first group, too
    // All weight blocks, once per CTA: every CTA reads the same bytes, so they come out of L2 one
    // reader after the other.  They follow the first piece of activations, which the transform waits
    // for.  map_w is the (channels, filters, taps) view; tap t of channel block cb goes into slot
    // cb * taps + t.  3x3 filters arrive with one copy a channel block on stage barrier 0; other sizes with
    // one a filter row, each on a barrier of its own, so that the first tile starts on the first row
    // (17x35x35x48 -> 64 5x5: 12.9 -> 11.9 us; in the unrolled 3x3 loop the waits cost more than they gave,
    // 128x28x28x128 -> 128 16.0 -> 16.5).
    const bool by_row = B_RESIDENT && !(g.R == 3 && g.S == 3);
    auto issue_resident_weights = [&]() {
        const int copies = by_row ? g.R : 1, copy_taps = by_row ? g.S : taps;
        if (!by_row) mbar_expect_tx(smem_u32(&bar_b_full[0]), (uint32_t)kb_count * kBBlock);
        for (int cb = 0, q = 0; cb < g.c_blocks; ++cb)
            for (int r = 0; r < copies; ++r, ++q) {
                const uint32_t full = smem_u32(&bar_b_full[by_row ? q : 0]);
                if (by_row) mbar_expect_tx(full, (uint32_t)copy_taps * kBBlock);
                tma_load_3d(b_slot(cb * taps + r * copy_taps), &map_w, full, cb * CB, 0, r * copy_taps);
            }
    };
    bool b_issued = false;

    if (warp == 0) {
        // ================= TMA producer =================
        if (lane == 0) {
            uint32_t gi = 0;                   // group counter
            int rb = 0; uint32_t ruse = 0;     // its window buffer (gi % win_bufs) and that buffer's use count (gi / win_bufs)
            uint32_t it = 0;      // streamed weight-block counter,
            int bs = 0; uint32_t buse = 0;     // its stage (it % b_stages) and that stage's use count
            for (; have; have = walk.next()) {
                const int b = rb;                 // window buffer of this group and how often it was used before
                const uint32_t use = ruse;
                if (use > 0 && !mbar_wait(smem_u32(&bar_win_empty[b]), (use - 1) & 1, abort_flag, g.status, g.wait_limit)) break;
                const int oh0 = (int)walk.tin * g.TR;
                // the roles that touch the caller's memory wait for the kernel before (later waits return at once), the
                // others do not (EARLY waits)
                dep_wait();
                dep_launch();
                for (int j = 0; j < g.G; ++j) {
                    const uint32_t wfull = smem_u32(&bar_win_full[b * kMaxG + j]);
                    if (j < (int)walk.cnt) {
                        mbar_expect_tx(wfull, piece_len(j) * (uint32_t)g.c_blocks);
                        const int h0 = oh0 - g.pad_h + (j ? j * g.TR + g.R - 1 : 0);
                        uint32_t dst = win_buf(b) + piece_off(j);
                        for (int cb = 0; cb < g.c_blocks; ++cb, dst += (uint32_t)g.plane_bytes)
                            tma_load_4d(dst, j ? &map_x1 : &map_x0, wfull, cb * CB, -g.pad_w, h0, (int)walk.img);
                    } else {
                        // a piece this group does not have: complete its phase so that the
                        // parity of every barrier of the buffer advances once per use
                        mbar_arrive(wfull);
                    }
                    if (B_RESIDENT && !b_issued) {       // behind the first piece, which the transform waits for
                        issue_resident_weights();
                        b_issued = true;
                    }
                }
                ++gi;
            if (++rb == g.win_bufs) { rb = 0; ++ruse; }
                if (!B_RESIDENT) {
                    bool stop = false;
                    const int passes = kBatched ? 1 : (int)walk.cnt;     // batched: one pass serves the whole group
                    for (int j = 0; j < passes && !stop; ++j) {
                        for (int cb = 0; cb < g.c_blocks && !stop; ++cb) {
                            for (int tap = 0; tap < taps; ++tap, ++it) {
                                const int sb = bs;
                                if (buse > 0 && !mbar_wait(smem_u32(&bar_b_empty[sb]), (buse - 1) & 1, abort_flag, g.status, g.wait_limit)) { stop = true; break; }
                                const uint32_t full = smem_u32(&bar_b_full[sb]);
                                mbar_expect_tx(full, kBBlock);
                                tma_load_3d(b_slot(sb), &map_w, full, cb * CB, (int)(walk.nt * BN), tap);
                                if (++bs == g.b_stages) { bs = 0; ++buse; }
                            }
                        }
                    }
                    if (stop) break;
                }
            }
            if (*abort_flag) {
                // wait (bounded) for copies still in flight so that none lands after exit
                const uint32_t gfirst = gi > (uint32_t)g.win_bufs ? gi - g.win_bufs : 0;
                for (uint32_t q = gfirst; q < gi; ++q)
                    for (int j = 0; j < g.G; ++j)
                        mbar_wait(smem_u32(&bar_win_full[(q % g.win_bufs) * kMaxG + j]), (q / g.win_bufs) & 1,
                                  abort_flag, g.status, g.wait_limit, true);
                if (B_RESIDENT) {
                    for (int q = 0; b_issued && q < (by_row ? g.c_blocks * g.R : 1); ++q)
                        mbar_wait(smem_u32(&bar_b_full[q]), 0, abort_flag, g.status, g.wait_limit, true);
                } else {
                    const uint32_t first = it > (uint32_t)g.b_stages ? it - g.b_stages : 0;
                    for (uint32_t q = first; q < it; ++q)
                        mbar_wait(smem_u32(&bar_b_full[q % g.b_stages]), (q / g.b_stages) & 1, abort_flag, g.status, g.wait_limit, true);
                }
            }
        }
        __syncwarp();
    } else if (warp == 1 || warp == kMmaBWarp) {
        // ================= MMA issuers =================
        // Issuer `me` (0: warp 1, 1: the last warp) takes the tiles whose running number has
        // parity `me`; tile number t goes into accumulator stage t % kAcc.  Each warp runs its loop converged and one elected
        // lane issues: the descriptor arithmetic below is on warp-uniform values only (kernel
        // arguments, loop counters), which lets it stay in the uniform datapath that feeds
        // tcgen05.mma.
        {
            const uint32_t me = (warp == 1) ? 0u : 1u;
            const uint32_t elected = elect_one();
            constexpr uint32_t idesc = make_idesc_i8(BN);
            // descriptors of window buffer 0 and of weight slot 0; offsets are added in units of
            // 16 bytes to the start-address field (the low word never carries into the next field)
            const uint64_t win_desc0 = make_smem_desc<CB>(smem_base);
            const uint64_t b_desc0 = make_smem_desc<CB>(b_base);
            uint32_t wt = 0;                   // tile counter (both issuers count every tile)
            uint32_t gi = 0;                   // group counter
            int rb = 0; uint32_t ruse = 0;     // its window buffer (gi % win_bufs) and that buffer's use count (gi / win_bufs)
            int s = 0;  uint32_t bph = 0;      // streamed weight stage and its phase parity
            // descriptor steps, in 16-byte units: one padded input row, one channel-block plane,
            // the rows of one tile
            const uint32_t row16 = (uint32_t)(g.Wp * CB) >> 4;
            const uint32_t plane16 = (uint32_t)g.plane_bytes >> 4;
            const uint32_t tile16 = (uint32_t)(g.TR * g.Wp * CB) >> 4;
            if (B_RESIDENT) mbar_wait<true>(smem_u32(&bar_b_full[0]), 0, abort_flag, g.status, g.wait_limit);
            bool weights_there = !by_row;      // else waited for row by row, during this issuer's first tile
            for (; have; have = walk.next()) {
                const int b = rb;
                const uint32_t wph = ruse & 1u;
                const uint64_t a_grp = win_desc0 + (uint64_t)((uint32_t)b * (win_bytes >> 4));
                bool issued = false;
                // Barrier reads go through the shared-memory pipe, which the tensor core's operand
                // fetches keep saturated, so a read takes hundreds of cycles.  The two barriers of
                // this issuer's NEXT tile of the group are therefore looked at (non-blocking, both
                // reads in flight together) after the first few MMAs of the current tile have been
                // queued; when both say "ready" -- the usual case -- that tile starts without
                // touching shared memory.
                uint32_t pre_acc = 0, pre_ops = 0;
                if constexpr (kBatched) {
                    // One pass over the streamed weights for all tiles of the group: every weight
                    // block is fetched from L2 once per group instead of once per tile.  Warp 1
                    // issues; the other issuer only keeps its counters in step.
                    const int cnt = (int)walk.cnt;
                    if (me == 0) {
                        issued = true;
                        for (int j = 0; j < cnt; ++j) {
                            const uint32_t t = wt + (uint32_t)j, use = t / (uint32_t)kAcc;
                            if (use > 0) mbar_wait(smem_u32(&bar_acc_empty[t & (uint32_t)(kAcc - 1)]), (use - 1) & 1, abort_flag, g.status, g.wait_limit);
                        }
                        // all pieces of the group: the transform warps finish them in order; without a
                        // transform the copies land in any order
                        if (MODE == SPARQ_MODE_NONE) {
                            for (int j = 0; j < cnt; ++j)
                                mbar_wait<true>(smem_u32(&bar_win_full[b * kMaxG + j]), wph, abort_flag, g.status, g.wait_limit);
                        } else {
                            mbar_wait<true>(smem_u32(&bar_win_xf[b * kMaxG + cnt - 1]), wph, abort_flag, g.status, g.wait_limit);
                        }
                        tc_fence_after();
                        uint64_t a_cb = a_grp;
                        for (uint32_t cb = 0; cb < (uint32_t)g.c_blocks; ++cb, a_cb += plane16) {
                            uint64_t a_r = a_cb;
                            for (int r = 0; r < g.R; ++r, a_r += row16) {
                                for (int sx = 0; sx < g.S; ++sx) {
                                    mbar_wait(smem_u32(&bar_b_full[s]), bph, abort_flag, g.status, g.wait_limit);
                                    tc_fence_after();
                                    const uint64_t bdesc = b_desc0 + (uint64_t)((uint32_t)s * (uint32_t)(kBBlock >> 4));
                                    const uint64_t a_tap = a_r + (uint64_t)(uint32_t)(sx * (CB >> 4));
                                    const uint32_t first = (cb == 0 && r == 0 && sx == 0) ? 0u : 1u;
                                    for (int j = 0; j < cnt; ++j) {
                                        const uint32_t d_tmem = tmem_base + ((wt + (uint32_t)j) & (uint32_t)(kAcc - 1)) * (uint32_t)BN;
                                        const uint64_t adesc = a_tap + (uint64_t)((uint32_t)j * tile16);
#pragma unroll
                                        for (int k = 0; k < CB / 32; ++k)
                                            tc_mma_i8_if(d_tmem, adesc + (uint64_t)(k * 2), bdesc + (uint64_t)(k * 2), idesc,
                                                         (first || k > 0) ? 1u : 0u, elected);
                                    }
                                    tc_commit_if(smem_u32(&bar_b_empty[s]), elected);
                                    if (++s == g.b_stages) { s = 0; bph ^= 1u; }
                                }
                            }
                        }
                        for (int j = 0; j < cnt; ++j)
                            tc_commit_if(smem_u32(&bar_acc_full[(wt + (uint32_t)j) & (uint32_t)(kAcc - 1)]), elected);
                    }
                    wt += (uint32_t)cnt;
                } else
                for (int j = 0; j < (int)walk.cnt; ++j, ++wt) {
                    if (kIssuers == 2 ? (wt & 1u) != me : me != 0u) {
                        if (!B_RESIDENT) {
                            // the other issuer consumes this tile's weight stages
                            s += kb_count;
                            while (s >= g.b_stages) { s -= g.b_stages; bph ^= 1u; }
                        }
                        continue;
                    }
                    issued = true;
                    const uint32_t acc = wt & (uint32_t)(kAcc - 1);
                    const uint32_t acc_use = wt / (uint32_t)kAcc;
                    const uint32_t d_tmem = tmem_base + acc * (uint32_t)BN;
                    if (acc_use > 0 && !pre_acc) mbar_wait(smem_u32(&bar_acc_empty[acc]), (acc_use - 1) & 1, abort_flag, g.status, g.wait_limit);
                    // Tile j reads pieces 0..j.  The transform warps finish pieces in order, so with
                    // a transform piece j's barrier covers the earlier ones.  Without one the copies
                    // land in any order: this issuer waits for pieces j-1 and j (its previous tile
                    // of the group, j-2, waited for the two before).
                    const uint32_t ops_bar = smem_u32(MODE == SPARQ_MODE_NONE ? &bar_win_full[b * kMaxG + j] : &bar_win_xf[b * kMaxG + j]);
                    if (!pre_ops) {
                        if (MODE == SPARQ_MODE_NONE && j > 0) mbar_wait<!B_RESIDENT>(ops_bar - 8u, wph, abort_flag, g.status, g.wait_limit);
                        mbar_wait<!B_RESIDENT>(ops_bar, wph, abort_flag, g.status, g.wait_limit);
                    }
                    tc_fence_after();
                    pre_acc = pre_ops = 0;
                    constexpr uint32_t step = kIssuers;                 // this issuer's next tile is number wt + step
                    const bool look_ahead = j + (int)step < (int)walk.cnt;
                    auto look = [&]() {
                        if (!look_ahead) return;
                        // a stage's first use needs no wait (the piece barrier stands in for it in the look)
                        const uint32_t nacc = (wt + step) & (uint32_t)(kAcc - 1), nuse = (wt + step) / (uint32_t)kAcc;
                        const uint32_t m = mbar_test3(nuse ? smem_u32(&bar_acc_empty[nacc]) : ops_bar, nuse ? (nuse - 1u) & 1u : wph,
                                                      ops_bar + 8u, wph, ops_bar + 8u * step, wph);
                        pre_acc = nuse ? (m & 1u) : 1u;
                        pre_ops = (MODE == SPARQ_MODE_NONE) ? (uint32_t)((m & 6u) == 6u) : (m >> 2);
                    };
                    const uint64_t a_desc0 = a_grp + (uint64_t)((uint32_t)j * tile16);
                    // One (tap, channel block) of the tile: wait for its weights when they are
                    // streamed, then CB / 32 MMAs.  The descriptors are sums of warp-uniform
                    // loop-carried values (no table, no division), so the address arithmetic of
                    // consecutive MMAs is a couple of adds.
                    auto issue_block = [&](const bool first, const uint32_t slot, const uint64_t adesc) {
                        uint64_t bdesc;
                        if (B_RESIDENT) {
                            bdesc = b_desc0 + (uint64_t)(slot * (uint32_t)(kBBlock >> 4));
                        } else {
                            mbar_wait(smem_u32(&bar_b_full[s]), bph, abort_flag, g.status, g.wait_limit);
                            tc_fence_after();
                            bdesc = b_desc0 + (uint64_t)((uint32_t)s * (uint32_t)(kBBlock >> 4));
                        }
#pragma unroll
                        for (int k = 0; k < CB / 32; ++k)
                            tc_mma_i8_if(d_tmem, adesc + (uint64_t)(k * 2), bdesc + (uint64_t)(k * 2), idesc,
                                         (!first || k > 0) ? 1u : 0u, elected);
                        if (!B_RESIDENT) {
                            tc_commit_if(smem_u32(&bar_b_empty[s]), elected);
                            if (++s == g.b_stages) { s = 0; bph ^= 1u; }
                        }
                    };
                    // channel block outer, tap inner: the order of the resident slots
                    uint64_t a_cb = a_desc0;
                    const uint32_t cbs = (uint32_t)g.c_blocks;
                    uint32_t slot = 0;
                    if (g.R == 3 && g.S == 3) {
                        for (uint32_t cb = 0; cb < cbs; ++cb, a_cb += plane16, slot += 9u) {
#pragma unroll
                            for (int r = 0; r < 3; ++r) {
#pragma unroll
                                for (int sx = 0; sx < 3; ++sx)
                                    issue_block(cb == 0 && r == 0 && sx == 0, slot + (uint32_t)(r * 3 + sx),
                                                a_cb + (uint64_t)((uint32_t)r * row16 + (uint32_t)(sx * (CB >> 4))));
                                if (r == 0 && cb == 0) look();
                            }
                        }
                    } else {
                        for (uint32_t cb = 0; cb < cbs; ++cb, a_cb += plane16) {
                            uint64_t a_r = a_cb;
                            for (int r = 0; r < g.R; ++r, a_r += row16) {
                                if (B_RESIDENT && !weights_there) {
                                    mbar_wait(smem_u32(&bar_b_full[cb * (uint32_t)g.R + (uint32_t)r]), 0, abort_flag, g.status, g.wait_limit);
                                    tc_fence_after();
                                }
                                for (int sx = 0; sx < g.S; ++sx, ++slot)
                                    issue_block(cb == 0 && r == 0 && sx == 0, slot, a_r + (uint64_t)(uint32_t)(sx * (CB >> 4)));
                                if (r == 0 && cb == 0) look();
                            }
                        }
                    }
                    weights_there = true;
                    tc_commit_if(smem_u32(&bar_acc_full[acc]), elected);      // accumulator complete
                }
                // The buffer goes back to the producer once both issuers have arrived and their
                // MMAs have retired.  With a transform, first make sure that every transform warp
                // is past all of this use's barriers (they arrive on the last piece's barrier
                // last), so that none of them can still be waiting on a phase when the producer
                // starts the next.
                if (MODE != SPARQ_MODE_NONE && (int)walk.cnt < g.G)
                    mbar_wait<!B_RESIDENT>(smem_u32(&bar_win_xf[b * kMaxG + g.G - 1]), wph, abort_flag, g.status, g.wait_limit);
                if (issued) {
                    tc_commit_if(smem_u32(&bar_win_empty[b]), elected);
                } else {
                    // No tile of this group was this issuer's.  It arrives only once the producer has
                    // started this use of the buffer (its first piece has landed), i.e. after the
                    // previous use's phase of the barrier has completed.
                    mbar_wait<!B_RESIDENT>(smem_u32(&bar_win_full[b * kMaxG]), wph, abort_flag, g.status, g.wait_limit);
                    if (elected) mbar_arrive(smem_u32(&bar_win_empty[b]));
                }
                ++gi;
            if (++rb == g.win_bufs) { rb = 0; ++ruse; }
            }
            // all tensor-core work of this CTA has retired before tensor memory is freed
            tc_commit_if(smem_u32(&bar_done), elected);
            mbar_wait(smem_u32(&bar_done), 0, abort_flag, g.status, g.wait_limit, true);
        }
        __syncwarp();
    } else if (warp < kFirstEpiWarp + epi_warps(MODE)) {
        // ================= epilogue =================
        const int quarter = warp & 3;
        const int group = (warp - kFirstEpiWarp) >> 2;
        const uint32_t team = (uint32_t)(group % teams);     // tiles whose number is team modulo teams
        const int parts = epi_parts(kGroups, teams, BN), part = group / teams;
        const int cols = BN / parts, cbase = part * cols;
        const int team_thread = (part * 4 + quarter) * 32 + lane, team_threads = parts * 128;
        float *s_scale = s_scale_all[kCopies == 1 ? 0 : team], *s_bias = s_bias_all[kCopies == 1 ? 0 : team];
        if (BN == 256 && team) {
            s_scale = reinterpret_cast<float *>(smem_raw + (b_slot(g.b_stages) - smem_u32(smem_raw)));
            s_bias = s_scale + BN;
        }
        const EpiView ev = make_epi_view(g);
        uint32_t wt = 0;
        int64_t staged_nt = -1;
        // this thread's slot inside a tile: row tr of the tile, padded column ow
        const int slot = quarter * 32 + lane;
        const int tr = slot / g.Wp;
        const int ow = slot - tr * g.Wp;
        const bool slot_ok = (tr < g.TR) && (ow < g.Wo);
        dep_wait();
        for (; have && part < parts; have = walk.next()) {
            for (int j = 0; j < (int)walk.cnt; ++j, ++wt) {
                if (wt % (uint32_t)teams != team) continue;
                const int64_t nt = (int64_t)walk.nt;
                const uint32_t acc = wt % (uint32_t)kAcc, acc_use = wt / (uint32_t)kAcc;
                if (ev.need_f && nt != staged_nt) {
                    staged_nt = nt;
                    epi_stage_scale_bias(g, nt * BN, BN, team_thread, team_threads, 1 + (int)team, s_scale, s_bias);
                }
                const int oh = ((int)walk.tin + j) * g.TR + tr;
                const bool row_ok = slot_ok && (oh < g.Ho);
                const int64_t row = ((int64_t)walk.img * g.Ho + oh) * g.Wo + ow;
                const uint32_t taddr0 = tmem_base + ((uint32_t)(quarter * 32) << 16) + acc * BN + (uint32_t)cbase;
                epi_warp_columns<OUT>(ev, taddr0, cbase, cols, row, row_ok, nt * BN, s_scale, s_bias,
                                 smem_u32(&bar_acc_empty[acc]), lane, [&]() {
                                     mbar_wait(smem_u32(&bar_acc_full[acc]), acc_use & 1u, abort_flag, g.status, g.wait_limit);
                                     tc_fence_after();
                                 });
            }
        }
    } else if (MODE != SPARQ_MODE_NONE) {
        // ================= transform: once per piece =================
        const uint32_t xt = threadIdx.x - kFirstXfWarp * 32;
        constexpr uint32_t kXfThreads = kNumXfWarps * 32;
        // Vectors in flight per thread.  Two keep the loop shorter (instruction cache), four hide more of
        // the shared-memory latency behind the tensor core's operand fetches, which are denser on
        // 128-wide tiles: 32x56x56x64 -> 64 3x3 9.25 us with two, 9.4 with one, 9.6 with four;
        // 128x28x28x128 -> 128 3x3 18.2, (three) 16.25, 15.95.  (With the half-precision transform 8.6, 8.6, 8.75 and
        // 15.1, 15.05, 15.05.)
        constexpr int kBatch = BN == 64 ? 2 : 4;
        const XformDev xf = g.xf;
        // Trimming pairs at n = 4 takes 12 packed-integer instructions and 14 in half precision; here, where the
        // transform is not the longest stage, the shorter one wins (128x28x28x128 -> 128 15.55 us against 15.85).
        auto word = [&](uint32_t x) {
            if constexpr (XN == 4 && !RND && MODE == SPARQ_MODE_VSPARQ) return xform_word<MODE, 4, false, false>(x, xf);
            else return xform_fused<MODE, XN, RND>(x, xf);
        };
        uint32_t gi = 0;
        int rb = 0; uint32_t ruse = 0;         // window buffer of the group (gi % win_bufs) and its use count (gi / win_bufs)
        for (; have; have = walk.next()) {
            const int b = rb;
            const uint32_t wph = ruse & 1u;
            for (int j = 0; j < g.G; ++j) {
                mbar_wait<true>(smem_u32(&bar_win_full[b * kMaxG + j]), wph, abort_flag, g.status, g.wait_limit);
                if (j < (int)walk.cnt) {
                    const uint32_t nvec = piece_len(j) >> 4;
                    uint32_t pbase = win_buf(b) + piece_off(j);
                    for (int cb = 0; cb < g.c_blocks; ++cb, pbase += (uint32_t)g.plane_bytes) {
                        // independent 16-byte vectors per thread and step; the last step of a piece may be short
                        for (uint32_t v0 = xt; v0 < nvec; v0 += kBatch * kXfThreads) {
                            uint4 v[kBatch];
                            bool ok[kBatch];
#pragma unroll
                            for (int q = 0; q < kBatch; ++q) {
                                ok[q] = v0 + (uint32_t)q * kXfThreads < nvec;
                                if (ok[q])
                                    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];"
                                                 : "=r"(v[q].x), "=r"(v[q].y), "=r"(v[q].z), "=r"(v[q].w)
                                                 : "r"(pbase + (v0 + (uint32_t)q * kXfThreads) * 16u));
                            }
#pragma unroll
                            for (int q = 0; q < kBatch; ++q) {
                                if (!ok[q]) continue;
                                v[q].x = word(v[q].x);
                                v[q].y = word(v[q].y);
                                v[q].z = word(v[q].z);
                                v[q].w = word(v[q].w);
                                asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};"
                                             :: "r"(pbase + (v0 + (uint32_t)q * kXfThreads) * 16u),
                                                "r"(v[q].x), "r"(v[q].y), "r"(v[q].z), "r"(v[q].w) : "memory");
                            }
                        }
                    }
                    fence_proxy_async_smem();
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&bar_win_xf[b * kMaxG + j]));
            }
            ++gi;
            if (++rb == g.win_bufs) { rb = 0; ++ruse; }
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

template <int BN, int CB, bool B_RESIDENT>
cudaError_t launch_window_shape(const CUtensorMap &mx0, const CUtensorMap &mx1, const CUtensorMap &mw, const WindowArgs &g,
                                int mode, int n, int rnd, int grid, int smem_bytes, cudaStream_t st);

template <int BN, int CB, int MODE, int XN, bool RND, bool RES, int OUT>
cudaError_t launch_window_kernel(const CUtensorMap &mx0, const CUtensorMap &mx1, const CUtensorMap &mw, const WindowArgs &g,
                                 int grid, int smem_bytes, cudaStream_t st)
{
    auto kfn = sparq_conv_window_kernel<BN, CB, MODE, XN, RND, RES, OUT>;
    static bool attr_set[64] = {};   // per device ordinal
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64 || !attr_set[dev]) {
        e = cudaFuncSetAttribute(kfn, cudaFuncAttributeMaxDynamicSharedMemorySize, kWindowMaxDynSmem);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) attr_set[dev] = true;
    }
    return launch_overlapped(kfn, grid, kWindowThreads, smem_bytes, st, mx0, mx1, mw, g);
}

template <int BN, int CB, int MODE, int XN, bool RND, bool RES>
cudaError_t launch_window_variant(const CUtensorMap &mx0, const CUtensorMap &mx1, const CUtensorMap &mw, const WindowArgs &g,
                                  int grid, int smem_bytes, cudaStream_t st)
{
    const int out = make_epi_view(g).out;
    if (out == kOutBytes) return launch_window_kernel<BN, CB, MODE, XN, RND, RES, kOutBytes>(mx0, mx1, mw, g, grid, smem_bytes, st);
    if (out == kOutResidual) return launch_window_kernel<BN, CB, MODE, XN, RND, RES, kOutResidual>(mx0, mx1, mw, g, grid, smem_bytes, st);
    return launch_window_kernel<BN, CB, MODE, XN, RND, RES, kOutGeneral>(mx0, mx1, mw, g, grid, smem_bytes, st);
}

#define SPARQ_LAUNCH_WINDOW_VARIANT(MODE_, XN_, RND_)                                                  \
    return launch_window_variant<BN, CB, MODE_, XN_, RND_, RES>(mx0, mx1, mw, g, grid, smem_bytes, st)

#define SPARQ_DEFINE_WINDOW_SHAPE(BN_, CB_, RES_)                                                      \
    template <>                                                                                        \
    cudaError_t launch_window_shape<BN_, CB_, RES_>(const CUtensorMap &mx0, const CUtensorMap &mx1,    \
                                                    const CUtensorMap &mw,                             \
                                                    const WindowArgs &g, int mode, int n, int rnd,     \
                                                    int grid, int smem_bytes, cudaStream_t st)         \
    {                                                                                                  \
        constexpr int BN = BN_, CB = CB_;                                                              \
        constexpr bool RES = RES_;                                                                     \
        if (mode == SPARQ_MODE_NONE) SPARQ_LAUNCH_WINDOW_VARIANT(SPARQ_MODE_NONE, 4, false);           \
        if (mode == SPARQ_MODE_BSPARQ) {                                                               \
            if (n == 8) SPARQ_LAUNCH_WINDOW_VARIANT(SPARQ_MODE_BSPARQ, 8, true);                       \
            if (n == 5) { if (rnd) SPARQ_LAUNCH_WINDOW_VARIANT(SPARQ_MODE_BSPARQ, 5, true);            \
                          else SPARQ_LAUNCH_WINDOW_VARIANT(SPARQ_MODE_BSPARQ, 5, false); }             \
            if (n == 4) { if (rnd) SPARQ_LAUNCH_WINDOW_VARIANT(SPARQ_MODE_BSPARQ, 4, true);            \
                          else SPARQ_LAUNCH_WINDOW_VARIANT(SPARQ_MODE_BSPARQ, 4, false); }             \
            if (rnd) SPARQ_LAUNCH_WINDOW_VARIANT(SPARQ_MODE_BSPARQ, 0, true);                          \
            else SPARQ_LAUNCH_WINDOW_VARIANT(SPARQ_MODE_BSPARQ, 0, false);                             \
        }                                                                                              \
        if (n == 8) SPARQ_LAUNCH_WINDOW_VARIANT(SPARQ_MODE_VSPARQ, 8, true);                           \
        if (n == 5) { if (rnd) SPARQ_LAUNCH_WINDOW_VARIANT(SPARQ_MODE_VSPARQ, 5, true);                \
                      else SPARQ_LAUNCH_WINDOW_VARIANT(SPARQ_MODE_VSPARQ, 5, false); }                 \
        if (n == 4) { if (rnd) SPARQ_LAUNCH_WINDOW_VARIANT(SPARQ_MODE_VSPARQ, 4, true);                \
                      else SPARQ_LAUNCH_WINDOW_VARIANT(SPARQ_MODE_VSPARQ, 4, false); }                 \
        if (rnd) SPARQ_LAUNCH_WINDOW_VARIANT(SPARQ_MODE_VSPARQ, 0, true);                              \
        else SPARQ_LAUNCH_WINDOW_VARIANT(SPARQ_MODE_VSPARQ, 0, false);                                 \
    }

}  // namespace sparq
