// Host side of the fused entry points: validation, tile-shape choice, TMA tensor maps
// (tiled for the GEMM view, im2col for the convolution), launch.
#include <cuda.h>

#include <cstdlib>
#include <cstring>
#include <mutex>

#include "sparq_conv_window_kernel.cuh"
#include "sparq_gemm_small_kernel.cuh"

namespace sparq {


// Limit of the device-side waits of every fused launch, in SM cycles.
static long long g_wait_limit = kWaitLimitCycles;

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *,
                                  CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);
typedef CUresult (*EncodeIm2colFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                   const cuuint64_t *, const int *, const int *, cuuint32_t, cuuint32_t,
                                   const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                   CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static int driver_fn(const char *name, void **fn)
{
    cudaDriverEntryPointQueryResult q;
    cudaError_t e = cudaGetDriverEntryPointByVersion(name, fn, 12000, cudaEnableDefault, &q);
    if (e != cudaSuccess) return cuda_error(e, name);
    if (q != cudaDriverEntryPointSuccess || !*fn)
        return set_error(SPARQ_ERR_CUDA, "driver entry point %s is unavailable", name);
    return SPARQ_OK;
}

static CUtensorMapSwizzle swizzle_for(int bk) { return bk == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B; }

// A tensor map is a pure function of the arguments it is encoded from (address, extents,
// strides, box, swizzle), and encoding one costs the host several microseconds -- as much as
// a small layer takes on the device.  Networks call the same layers with the same buffers
// over and over, so encoded maps are kept in a small direct-mapped table keyed by those
// arguments.  Host memory only; nothing to release.
struct MapKey {
    uint64_t v[14];
    bool operator==(const MapKey &o) const { return memcmp(v, o.v, sizeof(v)) == 0; }
};
struct MapSlot { bool used; MapKey key; CUtensorMap map; };
constexpr int kMapSlots = 256;
static MapSlot g_map_cache[kMapSlots];
static std::mutex g_map_mutex;

// Forgets the cached tensor maps (host memory only; they are re-encoded on demand).
void release_gemm_state()
{
    std::lock_guard<std::mutex> lock(g_map_mutex);
    for (MapSlot &s : g_map_cache) s.used = false;
}

static unsigned map_hash(const MapKey &k)
{
    uint64_t h = 1469598103934665603ull;
    for (uint64_t x : k.v) { h ^= x; h *= 1099511628211ull; h ^= h >> 29; }
    return (unsigned)(h % kMapSlots);
}
static bool map_lookup(const MapKey &k, CUtensorMap *out)
{
    std::lock_guard<std::mutex> lock(g_map_mutex);
    const MapSlot &s = g_map_cache[map_hash(k)];
    if (!s.used || !(s.key == k)) return false;
    *out = s.map;
    return true;
}
static void map_store(const MapKey &k, const CUtensorMap &m)
{
    std::lock_guard<std::mutex> lock(g_map_mutex);
    MapSlot &s = g_map_cache[map_hash(k)];
    s.used = true; s.key = k; s.map = m;
}

// 2-D K-contiguous matrix [rows][K] with row pitch ld bytes; box = bk x box_rows.
static int encode_2d(CUtensorMap *map, const void *ptr, int64_t K, int64_t rows, int64_t ld, int bk, int box_rows)
{
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        int rc = driver_fn("cuTensorMapEncodeTiled", (void **)&fn);
        if (rc != SPARQ_OK) return rc;
    }
    const MapKey key = {{1, (uint64_t)(uintptr_t)ptr, (uint64_t)K, (uint64_t)rows, (uint64_t)ld, (uint64_t)bk, (uint64_t)box_rows}};
    if (map_lookup(key, map)) return SPARQ_OK;
    cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)ld};
    cuuint32_t box[2] = {(cuuint32_t)bk, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void *>(ptr), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_for(bk), CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return set_error(SPARQ_ERR_CUDA, "cuTensorMapEncodeTiled failed with CUresult %d", (int)r);
    map_store(key, *map);
    return SPARQ_OK;
}

// The weight matrix [rows][K] in groups of 32 rows (rows a multiple of 32).  Row 8j + 2q + b of a group in
// shared memory is matrix row 8q + 2j + b as epi_frag wants it (frag), else the same.  Dimensions (K, b, q, j, group).
static int encode_row_groups(CUtensorMap *map, const void *ptr, int64_t K, int64_t rows, int64_t ld, int bk, int box_rows, bool frag)
{
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        int rc = driver_fn("cuTensorMapEncodeTiled", (void **)&fn);
        if (rc != SPARQ_OK) return rc;
    }
    const MapKey key = {{5, (uint64_t)(uintptr_t)ptr, (uint64_t)K, (uint64_t)rows, (uint64_t)ld, (uint64_t)bk, (uint64_t)box_rows, (uint64_t)frag}};
    if (map_lookup(key, map)) return SPARQ_OK;
    const cuuint64_t pitch = (cuuint64_t)ld;
    cuuint64_t dims[5] = {(cuuint64_t)K, 2, 4, 4, (cuuint64_t)rows / 32};
    cuuint64_t strides[4] = {pitch, (frag ? 8 : 2) * pitch, (frag ? 2 : 8) * pitch, 32 * pitch};
    cuuint32_t box[5] = {(cuuint32_t)bk, 2, 4, 4, (cuuint32_t)box_rows / 32};
    cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 5, const_cast<void *>(ptr), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_for(bk), CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return set_error(SPARQ_ERR_CUDA, "cuTensorMapEncodeTiled (weights) failed with CUresult %d", (int)r);
    map_store(key, *map);
    return SPARQ_OK;
}

// Weights as the GEMM kernels read them.
static int encode_b(CUtensorMap *map, const void *ptr, int64_t K, int64_t rows, int64_t ld, int bk, int bn, const GemmArgs &g, bool small)
{
    const int out = make_epi_view(g).out;
    if (small || out == kOutGeneral) return encode_2d(map, ptr, K, rows, ld, bk, bn);
    return encode_row_groups(map, ptr, K, rows, ld, bk, bn, frag_rows(out, bn, g.out_box));
}

// NHWC activation tensor read as im2col columns of `rows` output pixels x bk channels.
static int encode_im2col(CUtensorMap *map, const void *ptr, int n, int h, int w, int c, int r, int s,
                         int stride_h, int stride_w, int pad_h, int pad_w, int bk, int rows)
{
    static EncodeIm2colFn fn = nullptr;
    if (!fn) {
        int rc = driver_fn("cuTensorMapEncodeIm2col", (void **)&fn);
        if (rc != SPARQ_OK) return rc;
    }
    const MapKey key = {{2, (uint64_t)(uintptr_t)ptr, (uint64_t)n, (uint64_t)h, (uint64_t)w, (uint64_t)c, (uint64_t)r, (uint64_t)s,
                         (uint64_t)stride_h, (uint64_t)stride_w, (uint64_t)(int64_t)pad_h, (uint64_t)(int64_t)pad_w, (uint64_t)bk, (uint64_t)rows}};
    if (map_lookup(key, map)) return SPARQ_OK;
    cuuint64_t dims[4] = {(cuuint64_t)c, (cuuint64_t)w, (cuuint64_t)h, (cuuint64_t)n};
    cuuint64_t strides[3] = {(cuuint64_t)c, (cuuint64_t)c * w, (cuuint64_t)c * w * h};
    // Base pixels (the filter's top-left tap) run from -pad to dim - 1 + upper.
    int lower[2] = {-pad_w, -pad_h};
    int upper[2] = {pad_w - (s - 1), pad_h - (r - 1)};
    cuuint32_t estr[4] = {1, (cuuint32_t)stride_w, (cuuint32_t)stride_h, 1};
    CUresult res = fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, const_cast<void *>(ptr), dims, strides, lower, upper,
                      (cuuint32_t)bk, (cuuint32_t)rows, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_for(bk),
                      CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (res != CUDA_SUCCESS) return set_error(SPARQ_ERR_CUDA, "cuTensorMapEncodeIm2col failed with CUresult %d", (int)res);
    map_store(key, *map);
    return SPARQ_OK;
}

static int device_info(int *sms)
{
    int dev = 0, major = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
    if (e != cudaSuccess) return cuda_error(e, "device query");
    if (major != 10) return set_error(SPARQ_ERR_UNSUPPORTED, "the fused kernels need an sm_100 device (found sm_%d0)", major);
    return SPARQ_OK;
}

// Validates e->next_transform and turns it into kernel arguments (mode NONE when absent).
static int next_transform_args(const sparq_epilogue *e, int64_t N, int *mode, int *rnd, XformDev *xf)
{
    *mode = SPARQ_MODE_NONE;
    *rnd = 0;
    *xf = XformDev{0u, 0, 4};
    fill_fullset(xf, 4, 0);
    if (!e->next_transform || e->next_transform->mode == SPARQ_MODE_NONE) return SPARQ_OK;
    XformArgs nx;
    int rc = validate_params(e->next_transform, &nx);
    if (rc != SPARQ_OK) return rc;
    if (!e->u8_out) return set_error(SPARQ_ERR_INVALID_ARG, "next_transform needs u8_out");
    if (N % 4) return set_error(SPARQ_ERR_UNSUPPORTED, "next_transform needs N (%lld) to be a multiple of 4", (long long)N);
    *mode = nx.mode;
    *rnd = nx.rnd;
    *xf = XformDev{nx.widen_c, nx.widen_rounds, nx.n};
    fill_fullset(xf, nx.n, nx.rnd);
    return SPARQ_OK;
}

static int check_epilogue(const sparq_epilogue *e)
{
    if (!e) return set_error(SPARQ_ERR_INVALID_ARG, "sparq_epilogue is NULL");
    if (!e->acc_out && !e->f32_out && !e->u8_out)
        return set_error(SPARQ_ERR_INVALID_ARG, "no output requested (acc_out, f32_out and u8_out are all NULL)");
    if ((e->f32_out || e->u8_out) && !e->scale)
        return set_error(SPARQ_ERR_INVALID_ARG, "scale is NULL but a dequantized output is requested");
    if ((e->acc_out && ((uintptr_t)e->acc_out & 15u)) || (e->f32_out && ((uintptr_t)e->f32_out & 15u)) ||
        (e->u8_out && ((uintptr_t)e->u8_out & 15u)))
        return set_error(SPARQ_ERR_UNSUPPORTED, "output pointers must be 16-byte aligned");
    if (e->residual) {
        if (!e->f32_out && !e->u8_out)
            return set_error(SPARQ_ERR_INVALID_ARG, "residual needs a dequantized output (f32_out or u8_out)");
        if ((uintptr_t)e->residual & 15u)
            return set_error(SPARQ_ERR_UNSUPPORTED, "residual must be 16-byte aligned");
    }
    return SPARQ_OK;
}

// Bytes per output element that the epilogue writes.
static double out_bytes(const sparq_epilogue *e) { return (e->acc_out ? 4 : 0) + (e->f32_out ? 4 : 0) + (e->u8_out ? 1 : 0); }

// A contraction as its tiles are estimated: `blocks` reduction steps of wide * 128 bytes, `fetch` cycles per row of A
// and B in each, `ow` bytes of output per element (without a residual's, which the staged form hides: counted, 50176 x
// 512, K 128, with one took 128-wide tiles, 16.6 us against 15.8).
struct Steps {
    int64_t blocks;
    double wide, fetch, ow;
};
static Steps gemm_steps(int64_t K, double ow) { return {(K + 127) / 128, 1.0, 2.2, ow}; }
static int conv_bk(int c) { return c % 128 == 0 ? 128 : 64; }
static Steps conv_steps(int64_t taps, int c, double ow)
{
    if (conv_bk(c) == 128) return {taps * (c / 128), 1.0, 1.3, ow};
    // 64-byte rows cost nearly as much as 128-byte ones, and the last block's that reach past C two to three
    // times that (128-wide tiles, 3x3: 500 cycles a step with 64 channels, 925 with 32, 1700 with 16)
    const int full = c / 64, rest = c % 64, per_tap = full + (rest ? 1 : 0);
    const double last = rest == 0 ? 0.0 : rest == 32 ? 2.1 : rest == 48 ? 3.05 : 3.5;
    return {taps * per_tap, 0.5, (1.15 * full + last) / per_tap, ow};
}

// Cycles that the transform takes of a 128-byte step.  (Measured, 128-wide tiles, pairs: n = 4 with all
// placements 1090, with fewer 1450, 3 and 2 bits 1945, restricted 2720; without the pair rule the 3- and 2-bit
// sets are as quick as n = 4.)
static double xform_cycles(const XformArgs &x)
{
    if (x.mode == SPARQ_MODE_NONE) return 0.0;
    if (x.n == 4) return x.widen_rounds ? 1450.0 : 1150.0;
    return x.widen_rounds || x.mode == SPARQ_MODE_VSPARQ ? 2000.0 : 1150.0;
}

// Cycles that one CTA spends with 128 x bn tiles, the estimate that tile width and form are chosen by.  A step
// takes the longest of
//   transform of the A stage   xform_cycles per 128 bytes (xf; 0 without one),
//   MMA                        2 * bn cycles per 128 bytes,
//   operand fetch from L2      Steps::fetch per row of A and B
// plus a hand-over; a tile its steps or its epilogue, in ceil(tiles / SMs) passes.  Narrow tiles add CTAs but re-fetch
// and re-transform A once per column tile.  A fit of the choices (not the times) to 1700 layers measured in every
// form.  Over 2400 others that are too large for the small form it costs 2.3 % against the fastest form, 2.5 % of them
// lose more than 20 %.  The estimate before (one cost for all transforms, 64-byte rows at half price): 4.7 % and 6.8 %,
// and 5.5 % of the layers lost against the one before that, up to 1.9 times: 5151 x 1680, K 2608, at 2 bits 50.7 us fused,
// 36.6 transformed first; 8x44x44x48 -> 488 5x5 49.6 transformed first, 39.4 fused.
static double tile_cycles(int64_t M, int64_t N, const Steps &k, int bn, int sms, double xf)
{
    const int64_t tiles = ((M + kBM - 1) / kBM) * ((N + bn - 1) / bn);
    const int64_t rounds = (tiles + sms - 1) / sms;
    double step = 2.0 * bn * k.wide;
    const double fetch = k.fetch * (kBM + bn);
    if (fetch > step) step = fetch;
    if (xf * k.wide > step) step = xf * k.wide;
    const double epi = bn * (2.6 + 2.1 * k.ow), walk = (double)k.blocks * (step + 105.0);
    return (double)rounds * (walk > 1.35 * epi ? walk : 1.35 * epi) + epi;     // + the last tile's epilogue
}

// The tile width with the lowest estimate.
static int pick_bn(int64_t M, int64_t N, const Steps &k, int sms, double xf, double *cycles = nullptr)
{
    const int cand[3] = {256, 128, 64};
    int best = 64;
    double best_cost = 0.0;
    for (int i = 0; i < 3; ++i) {
        const int bn = cand[i];
        if (bn > 64 && N <= bn / 2) continue;          // would be mostly padding
        const double cost = tile_cycles(M, N, k, bn, sms, xf);
        if (best_cost == 0.0 || cost < best_cost) {
            best_cost = cost;
            best = bn;
        }
    }
    if (cycles) *cycles = best_cost;
    return best;
}

// The small form (sparq_gemm_small_kernel): launches whose 64-wide tiles all run at once.  tile_rows = 0
// where they do not.  Tiles of 64 or 128 rows, and 1 to 8 CTAs of a cluster on a tile, by the time
// of the serial walk along K: a step takes such a launch about 0.25 us, and 0.35 us more for the
// transform of 128 rows (packed integers; the half-precision one at n = 4 takes less); sharing a tile costs about 1.6 us, and writing 128 rows out 0.4 (173 x 128 x 256,
// fp32, without a transform: 4.3 us with 128 rows, 3.8 with 64).  Measured (us, one image, 128-row
// tiles, 1 / 2 / 4 / 8 CTAs on each): 7x7x2048 -> 512 9.4 / 9.1 / 6.1 / 4.8, 14x14x1024 -> 256 6.9 /
// 8.7 / 6.3 / 5.0, 28x28x512 -> 128 5.6 / 7.1 / 5.6, 7x7x512 -> 2048 4.7 / 6.3 / 5.1; chosen by this
// rule, against the full kernel before: 7x7x512 -> 512 3x3 30.1 -> 6.7, 14x14x256 -> 256 3x3 14.9 ->
// 5.5, 14x14x1024 -> 256 8.9 -> 4.2, 28x28x128 -> 512 with a residual 4.6 -> 3.1, 256 x 64 x 576
// with int32 and fp32 outputs 8.7 -> 6.5.
struct SmallForm {
    int tile_rows, split;
};
static SmallForm pick_small(int64_t M, int64_t N, int64_t k_blocks, int sms, bool transform)
{
    SmallForm best = {0, 1};
    double best_cost = 0.0;
    const int64_t n_tiles = (N + kSmallBN - 1) / kSmallBN;
    for (int rows = kBM; rows >= 64; rows /= 2) {
        const int64_t tiles = (M + rows - 1) / rows * n_tiles;
        const double step = 0.25 + (transform ? 0.35 * (double)(M < rows ? M : rows) / kBM : 0.0);
        for (int split = 1; split <= kMaxSplit && tiles * split <= sms && k_blocks >= split; split *= 2) {
            const double cost = 0.4 * rows / kBM + (double)((k_blocks + split - 1) / split) * step + (split > 1 ? 1.6 : 0.0) + (split == 2 ? 0.4 : 0.0);
            if (!best.tile_rows || cost < best_cost - 0.05) { best = {rows, split}; best_cost = cost; }
        }
    }
    return best;
}

// Whether to write T(A) to scratch memory once and contract that, instead of transforming every
// staged tile: worth it when A is staged several times -- several column tiles, several filter
// taps -- because the in-kernel transform is what such a step takes.  The extra pass costs about
// 3.7 us and 2 bytes of traffic per activation (2.8 TB/s of activations), and the contraction reads them again
// (89x56x56x352 -> 24 at 2 bits: 53.2 us fused, 65.5 transformed first).
static bool transform_first(int64_t M, int64_t N, const Steps &k, const XformArgs &x, size_t act_bytes, int sms)
{
    if (pick_small(M, N, k.blocks, sms, true).tile_rows) return false;
    if ((M + kBM - 1) / kBM * ((N + 63) / 64) >= (int64_t)1 << 31) return false;      // near the refused sizes: refused, if at all, with nothing enqueued
    double fused, plain;
    pick_bn(M, N, k, sms, xform_cycles(x), &fused);
    pick_bn(M, N, k, sms, 0.0, &plain);
    const double clk = 1900.0;      // cycles per us
    const double read = clk * (double)act_bytes / 6.0e6;
    return (plain > read ? plain : read) + clk * (3.7 + (double)act_bytes / 2.8e6) < 0.99 * fused;
}

// Variant argument of the launchers (XN of xform_fused): 4 = n = 4 with all five placements, 5 = n = 4
// with fewer, 8 = another full placement set (6opt, 7opt), 0 = restricted sets of n < 4.
static int variant_n(const XformArgs &x) { return x.n == 4 ? (x.widen_rounds ? 5 : 4) : (x.widen_rounds ? 0 : 8); }

// Kernel-side transform constants.
static XformDev xform_dev(const XformArgs &x)
{
    XformDev d{x.widen_c, x.widen_rounds, x.n};
    fill_fullset(&d, x.n, x.rnd);
    return d;
}

static cudaError_t launch(int bn, int bk, bool small, const GemmMaps &m, GemmArgs &g, const XformArgs &x, int grid, cudaStream_t st)
{
    if (small && bk == 64) return launch_gemm_small<64>(m, g, x.mode, variant_n(x), x.rnd, grid, st);
    if (small) return launch_gemm_small<128>(m, g, x.mode, variant_n(x), x.rnd, grid, st);
    if (bn == 64 && bk == 64) return launch_gemm_shape<64, 64>(m, g, x.mode, variant_n(x), x.rnd, grid, st);
    if (bn == 64) return launch_gemm_shape<64, 128>(m, g, x.mode, variant_n(x), x.rnd, grid, st);
    if (bn == 128 && bk == 64) return launch_gemm_shape<128, 64>(m, g, x.mode, variant_n(x), x.rnd, grid, st);
    if (bn == 128) return launch_gemm_shape<128, 128>(m, g, x.mode, variant_n(x), x.rnd, grid, st);
    if (bk == 64) return launch_gemm_shape<256, 64>(m, g, x.mode, variant_n(x), x.rnd, grid, st);
    return launch_gemm_shape<256, 128>(m, g, x.mode, variant_n(x), x.rnd, grid, st);
}

static int fill_common(GemmArgs *g, const XformArgs &x, const sparq_epilogue *e, unsigned int *status)
{
    g->xf = xform_dev(x);
    g->scale = e->scale;
    g->bias = e->bias;
    g->relu = e->relu ? 1 : 0;
    g->inv_out_scale = e->inv_out_scale;
    g->acc_out = e->acc_out;
    g->f32_out = e->f32_out;
    g->u8_out = e->u8_out;
    g->status = status;
    g->wait_limit = g_wait_limit;
    g->residual = e->residual;
    g->residual_scale = e->residual_scale;
    return next_transform_args(e, g->N, &g->next_mode, &g->next_rnd, &g->next_xf);
}

// Chooses the staged output (epi_staged_box) and encodes its tensor maps: for requantized bytes in
// whole groups of 32 columns, when a warp's share of a tile is at least 64 columns wide.  The
// staging buffers cost ring stages, and a hand-over per box where a CTA has a single tile, so the
// output (and residual) bytes of a tile have to weigh at least 5/8 of its operands': 56x56x64 ->
// 256 with a residual 44 -> 33 us, 14x14x256 -> 1024 with one 16 -> 15; 28x28x256 -> 512 without
// one would lose (19 -> 20.5), 7x7x512 -> 2048 with one too (13.0 -> 13.6).
static int output_maps(GemmMaps *m, GemmArgs *g, int mode, int bn, int64_t tiles, int grid)
{
    g->out_box = 0;
    if (make_epi_view(*g).out == kOutGeneral || tiles <= grid) return SPARQ_OK;
    const int64_t out_bytes = (int64_t)kBM * bn * (g->residual ? 2 : 1), operand_bytes = (int64_t)(kBM + bn) * g->K;
    if (8 * out_bytes < 5 * operand_bytes) return SPARQ_OK;
    const int groups = epi_warps(mode) / 4, acc = bn == 256 ? 2 : 4;
    const int teams = groups < acc ? groups : acc;
    const int cols = bn / epi_parts(groups, teams, bn), widest = mode == SPARQ_MODE_NONE ? 64 : 128;
    const int box = cols < widest ? cols : widest;
    if (box < 64) return SPARQ_OK;
    g->out_box = box;
    int rc = encode_2d(&m->out, g->u8_out, g->N, g->M, g->N, box, 32);
    if (rc == SPARQ_OK && g->residual) rc = encode_2d(&m->res, g->residual, g->N, g->M, g->N, box, 32);
    return rc;
}

int gemm_with_status(const uint8_t *A, int64_t lda, const int8_t *B, int64_t ldb, int64_t M, int64_t N, int64_t K,
                     const XformArgs &x, const sparq_epilogue *e, unsigned int *status, cudaStream_t st);

// Parameters of a contraction whose activations are already transformed.
static XformArgs plain_a8w8()
{
    XformArgs x = {};
    x.mode = SPARQ_MODE_NONE;
    x.n = 4;
    return x;
}

// The fused GEMM with the library's own status word (allocated on first use).
static int gemm_impl(const uint8_t *A, int64_t lda, const int8_t *B, int64_t ldb, int64_t M, int64_t N, int64_t K,
                     const XformArgs &x, const sparq_epilogue *e, cudaStream_t st)
{
    unsigned int *status = nullptr;
    int rc = get_status_word(&status);
    if (rc != SPARQ_OK) return rc;
    int sms = 0;
    if (x.mode != SPARQ_MODE_NONE && lda == K && (rc = device_info(&sms)) == SPARQ_OK &&
        transform_first(M, N, gemm_steps(K, out_bytes(e)), x, (size_t)M * (size_t)K, sms)) {
        if (uint8_t *ta = (uint8_t *)workspace_alloc((size_t)M * (size_t)K, st)) {
            rc = quantize_rows(A, ta, (size_t)M, (size_t)K, x, true, st);
            if (rc == SPARQ_OK) rc = gemm_with_status(ta, K, B, ldb, M, N, K, plain_a8w8(), e, status, st);
            workspace_free(ta, st);
            return rc;
        }
    }
    return gemm_with_status(A, lda, B, ldb, M, N, K, x, e, status, st);
}

// NHWC activation tensor read as a box of cb channels x wp columns x rows input rows of one
// image (zero fill outside the image).
static int encode_window(CUtensorMap *map, const void *ptr, int n, int h, int w, int c, int cb, int wp, int rows)
{
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        int rc = driver_fn("cuTensorMapEncodeTiled", (void **)&fn);
        if (rc != SPARQ_OK) return rc;
    }
    const MapKey key = {{3, (uint64_t)(uintptr_t)ptr, (uint64_t)n, (uint64_t)h, (uint64_t)w, (uint64_t)c, (uint64_t)cb, (uint64_t)wp, (uint64_t)rows}};
    if (map_lookup(key, map)) return SPARQ_OK;
    cuuint64_t dims[4] = {(cuuint64_t)c, (cuuint64_t)w, (cuuint64_t)h, (cuuint64_t)n};
    cuuint64_t strides[3] = {(cuuint64_t)c, (cuuint64_t)c * w, (cuuint64_t)c * w * h};
    cuuint32_t box[4] = {(cuuint32_t)cb, (cuuint32_t)wp, (cuuint32_t)rows, 1};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, const_cast<void *>(ptr), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_for(cb), CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return set_error(SPARQ_ERR_CUDA, "cuTensorMapEncodeTiled (window) failed with CUresult %d", (int)r);
    map_store(key, *map);
    return SPARQ_OK;
}

// Weights [cout][taps][c] as (channels, filters, taps): a box brings cb channels of bn filters and
// box_taps taps into consecutive bn x cb shared-memory blocks (a whole filter, a filter row, a tap);
// channels past c arrive as zeros.
static int encode_weights(CUtensorMap *map, const void *ptr, int c, int cout, int taps, int cb, int bn, int box_taps)
{
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        int rc = driver_fn("cuTensorMapEncodeTiled", (void **)&fn);
        if (rc != SPARQ_OK) return rc;
    }
    const MapKey key = {{4, (uint64_t)(uintptr_t)ptr, (uint64_t)c, (uint64_t)cout, (uint64_t)taps, (uint64_t)cb, (uint64_t)bn, (uint64_t)box_taps}};
    if (map_lookup(key, map)) return SPARQ_OK;
    cuuint64_t dims[3] = {(cuuint64_t)c, (cuuint64_t)cout, (cuuint64_t)taps};
    cuuint64_t strides[2] = {(cuuint64_t)c * taps, (cuuint64_t)c};
    cuuint32_t box[3] = {(cuuint32_t)cb, (cuuint32_t)bn, (cuuint32_t)box_taps};
    cuuint32_t estr[3] = {1, 1, 1};
    const CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, const_cast<void *>(ptr), dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_for(cb), CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return set_error(SPARQ_ERR_CUDA, "cuTensorMapEncodeTiled (weights) failed with CUresult %d", (int)r);
    map_store(key, *map);
    return SPARQ_OK;
}

constexpr int kMaxDynSmem = kWindowMaxDynSmem;

// ---- which form a stride-1 convolution takes ---------------------------------------------------------
// Estimates in us, least-squares fits to 840 measured layers (1-128 images of 7..56 pixels, 16-512
// channels and filters, 3x3 / 5x5 / 7x7, five transforms and none), with the packed-integer transform at n = 4 and one wait
// of all roles for the kernel before.  Root mean square error then: window with streamed weights on
// 128-wide tiles 7 %, on 256-wide ones 22 %, small form 10 %, im2col form 11 %.  Both forms have become faster since;
// only the start of the small one was measured again (2.5 -> 1.9 us).  They are compared where either
// form can win by a factor: few tiles (over 493 layers the choice cost 0.2 % against the faster form, at
// worst 20 %; always the window 48 %), half-empty channel blocks (1.4 %; always the window 13 %) and
// rings of two stages.
// The transform's work relative to the 4-bit form with all placements.
static double xform_weight(const XformArgs &x)
{
    return x.mode == SPARQ_MODE_NONE ? 0.0 : x.n == 4 ? (x.widen_rounds ? 1.2 : 1.0) : (x.widen_rounds ? 2.0 : 1.35);
}
// Bytes per output element that the epilogue moves.
static double out_weight(const sparq_epilogue *e) { return out_bytes(e) + (e->residual ? 1 : 0); }
static double small_us(const SmallForm &f, int64_t M, int64_t k_blocks, int bk, double xw)
{
    const double rows = (double)(M < f.tile_rows ? M : f.tile_rows) / kBM * bk / 128.0;
    return 1.9 + (double)((k_blocks + f.split - 1) / f.split) * (0.21 + (0.09 + 0.60 * xw) * rows) + (f.split > 1 ? 1.3 : 0.0);
}
static double im2col_us(int64_t M, int64_t N, int taps, int c, const XformArgs &x, double ow, int sms)
{
    const int bk = conv_bk(c);
    const double xw = xform_weight(x);
    const Steps k = conv_steps(taps, c, ow);
    const int bn = pick_bn(M, N, k, sms, xform_cycles(x));
    const double rounds = (double)(((M + kBM - 1) / kBM * ((N + bn - 1) / bn) + sms - 1) / sms), blocks = rounds * k.blocks;
    return 2.6 + blocks * bk / 128.0 * ((bn == 64 ? 0.05 : bn == 128 ? 0.10 : 0.13) + (bn == 256 ? 0.46 : 0.48) * xw) + 0.22 * blocks +
           0.47 * rounds * bn / 128.0 * ow;
}
// The same layer by the im2col path, in the form that would be launched there.
static double im2col_path_us(int64_t M, int64_t N, int taps, int c, const XformArgs &x, double ow, int sms)
{
    const int64_t k_blocks = conv_steps(taps, c, ow).blocks;
    const SmallForm f = pick_small(M, N, k_blocks, sms, x.mode != SPARQ_MODE_NONE);
    return f.tile_rows ? small_us(f, M, k_blocks, conv_bk(c), xform_weight(x)) : im2col_us(M, N, taps, c, x, ow, sms);
}

// How the window kernel tiles a convolution.
struct WindowPlan {
    int wp, cb, tr, c_blocks, tiles_per_img, bn, n_tiles;
    int64_t units;
    bool resident;
    int grp, win_bufs, b_stages, plane_bytes;
    bool team_copy;
    int smem_bytes;
};

// Stride-1 filters larger than 1x1: false where the window kernel's tiling does not fit, or another form
// is expected to be faster.  ow: out_weight of the epilogue; scratch(bytes): whether T(x) may be
// written to scratch memory.
template <class Scratch>
static bool plan_window(WindowPlan *q, int n, int h, int w, int c, int cout, int r, int s, int pad_w, int ho, int wo,
                        const XformArgs &x, double ow, int sms, Scratch scratch)
{
    int wp = w + 2 * pad_w;
    if (wp > 128 || wo < 1) return false;
    // channel blocks; the last one's tail is zero fill.  Few channels and many filters: 128-wide blocks
    // that are half empty, because 64-channel blocks exist on 64-wide tiles only.
    const int cb = (c <= 64 && cout <= 64) ? 64 : 128;
    int tr = 128 / wp;
    if (tr > ho) tr = ho;
    if (tr < 1 || tr * wo < 64) return false;               // less than half of the MMA rows would be useful
    // Pieces land at multiples of tr * wp rows, which must be a multiple of 128 bytes: an even row
    // width makes it so for 64-byte rows.
    if (cb == 64 && (wp & 1) && wp + 1 <= 128 && (128 / (wp + 1) >= tr)) ++wp;
    const int c_blocks = (c + cb - 1) / cb;
    const int taps = r * s;
    const int kb_count = taps * c_blocks;
    const bool half_empty = cb == 128 && c <= 64;
    const int64_t M = (int64_t)n * ho * wo;
    const double xw = xform_weight(x);
    const int tiles_per_img = (ho + tr - 1) / tr;
    const int64_t m_tiles = (int64_t)n * tiles_per_img;

    int bn;
    if (cb == 64) {
        bn = 64;
    } else {
        bn = (cout > 128 && m_tiles * ((cout + 255) / 256) >= sms) ? 256 : 128;
    }
    const int b_block = bn * cb;
    const int n_tiles = (cout + bn - 1) / bn;
    const int64_t units = m_tiles * n_tiles;
    if (units >= (int64_t)1 << 31) return false;
    const int grid = (int)(units < sms ? units : sms);

    // Shared memory of one window buffer when up to `grp` tiles share it: a plane (one channel
    // block) holds every row the MMA of the group's last tile may touch.
    auto plane_for = [&](int grp) {
        const int rows_alloc = (grp - 1) * tr * wp + (r - 1) * wp + (s - 1) + 128;
        return (rows_alloc * cb + 1023) / 1024 * 1024;
    };
    // Tiles per group: with one column tile, as many as a CTA's share of the tile sequence
    // has (more would never be used) while two window buffers still fit beside the weights.
    // A later piece must land on a 128-byte boundary (TMA destination alignment).
    int gmax = 1;
    if (n_tiles == 1) {
        gmax = (int)((units + grid - 1) / grid);
        if (gmax > tiles_per_img) gmax = tiles_per_img;
        if (gmax > kMaxG) gmax = kMaxG;
        if (cb == 64 && (((tr * wp) & 1) || (((r - 1) * wp) & 1))) gmax = 1;
    }
    bool resident = false, batched = false;
    int win_bufs = 2, b_stages = 0, grp = 1;
    if (bn != 256 && n_tiles == 1 && c_blocks * r <= kMaxBStages && 1024 + 2 * plane_for(1) * c_blocks + kb_count * b_block <= kMaxDynSmem) {
        resident = true;
        b_stages = kb_count;
        grp = gmax;
        while (grp > 1 && 1024 + 2 * plane_for(grp) * c_blocks + kb_count * b_block > kMaxDynSmem) --grp;
        // more buffers only help while a CTA has more groups than buffers
        const int groups_per_cta = (int)((units + grid - 1) / grid + grp - 1) / grp + 1;
        while (win_bufs < kMaxWinBufs && win_bufs < groups_per_cta &&
               1024 + (win_bufs + 1) * plane_for(grp) * c_blocks + kb_count * b_block <= kMaxDynSmem) ++win_bufs;
        // A tile per CTA at most: mostly the time of its weights, 3.35 us + 13 per MB (56x56x64 -> 64 3x3 3.8 us,
        // 28x28x128 -> 128 5.3); the small form may share them out (one image of the latter 5.2 -> 4.6, of
        // 20x20x96 -> 112 6.3 -> 4.3; 56x56x64 stays).
        if (units <= sms && pick_small(M, cout, (int64_t)taps * ((c + 127) / 128), sms, xw > 0.0).tile_rows &&
            im2col_path_us(M, cout, taps, c, x, ow, sms) < 0.97 * (3.35 + 13.2e-6 * kb_count * b_block)) return false;
    } else {
        if (bn == 64) return false;                          // only the resident form is built for 64-wide tiles
        // 128-wide tiles: up to two row tiles of one (image, column tile) are accumulated together
        // during ONE pass over the streamed weights (four accumulator stages: two groups in
        // flight), which halves the weight traffic out of L2 -- the bound of these layers.
        batched = bn == 128;
        double window_us = 0.0;
        auto consider = [&](int g) {
            const int bytes = plane_for(g) * c_blocks;
            // a CTA that owns a single group needs no second window buffer: the room goes to the
            // weight ring, whose depth (bytes in flight) bounds how fast one SM can pull the weights
            const int64_t groups = (int64_t)n * n_tiles * ((tiles_per_img + g - 1) / g);
            int bufs = batched && groups <= sms ? 1 : 2;
            int stages = (kMaxDynSmem - 1024 - bufs * bytes) / b_block;
            if (stages > kMaxBStages) stages = kMaxBStages;
            if (stages < 2) return;
            // spare room beyond four weight stages goes to a third window buffer
            if (bufs == 2 && stages > 4 && 1024 + 3 * bytes + 4 * b_block <= kMaxDynSmem) {
                bufs = 3;
                stages = (kMaxDynSmem - 1024 - 3 * bytes) / b_block;
                if (stages > kMaxBStages) stages = kMaxBStages;
            }
            const double rows = (double)((batched ? tr * g : tr) + r - 1) * wp / 128.0, ring = stages == 2 ? 0.09 : 0.0;
            const double us =
                batched ? 3.9 + (double)((groups + sms - 1) / sms) * (kb_count * (0.066 + 0.159 * g + ring) + c_blocks * rows * (0.73 * xw + 0.23))
                        : 6.0 + (double)((units + sms - 1) / sms) * (kb_count * (0.373 + ring) + c_blocks * rows * (0.65 * xw + 0.46));
            if (b_stages == 0 || us < window_us) { window_us = us; grp = g; win_bufs = bufs; b_stages = stages; }
        };
        if (batched) {
            // one tile a group or two: two halve the weight traffic, one has more CTAs where they are few
            // (8x28x28x256 -> 192: 10.9 us with one, 15.2 with two)
            consider(1);
            if (tiles_per_img > 1 && kMaxDynSmem - 1024 - 2 * plane_for(2) * c_blocks >= 4 * b_block) consider(2);
        } else {
            int g = gmax;
            while (g > 1 && kMaxDynSmem - 1024 - 2 * plane_for(g) * c_blocks < 4 * b_block) --g;
            consider(g);
        }
        if (b_stages == 0) return false;
        // Few tiles: the small form, whose long reduction a cluster can share, may be faster (one image
        // of 14x14x256 -> 256 3x3: 6.9 us against 14.6) or not (8x14x14x512 -> 512 5x5: 82 against 33).
        // Half-empty channel blocks: the im2col form reads 64-channel ones, half the multiplications
        // and operand bytes for one transform per tap (64x17x17x64 -> 256 3x3: 8.3 us against 12.7;
        // 17x35x35x32 -> 160 7x7 at 2 bits 45 against 25).
        if (half_empty || (batched && pick_small(M, cout, (int64_t)taps * ((c + 127) / 128), sms, xw > 0.0).tile_rows)) {
            if (im2col_path_us(M, cout, taps, c, x, ow, sms) < window_us) return false;
        } else if (batched && b_stages == 2) {
            // a ring this short leaves the tensor core waiting; transformed once, the im2col form may win
            // (16x56x56x256 -> 64 5x5 at 3 bits, restricted: 56 us against 100)
            const size_t act_bytes = (size_t)n * h * w * (size_t)c;
            const double first = xw > 0.0 && scratch(act_bytes) ? 2.5 + (double)act_bytes / 2.9e6 + im2col_us(M, cout, taps, c, plain_a8w8(), ow, sms) : 1e30;
            if (first < window_us || im2col_path_us(M, cout, taps, c, x, ow, sms) < window_us) return false;
        }
    }
    *q = {wp, cb, tr, c_blocks, tiles_per_img, bn, n_tiles, units, resident, grp, win_bufs, b_stages, plane_for(grp), false, 0};
    q->smem_bytes = 1024 + win_bufs * q->plane_bytes * c_blocks + b_stages * b_block;
    q->team_copy = bn == 256 && q->smem_bytes + kTeamCopyBytes <= kMaxDynSmem;
    if (q->team_copy) q->smem_bytes += kTeamCopyBytes;
    return true;
}

// Returns 1 if the window kernel was launched, 0 if the convolution should take another form, < 0 on error.
static int try_window_conv(const uint8_t *x_in, int n, int h, int w, int c, const int8_t *wgt, int cout, int r, int s,
                           int pad_h, int pad_w, int ho, int wo, const XformArgs &x, const sparq_epilogue *e,
                           int sms, unsigned int *status, cudaStream_t st)
{
    WindowPlan q;
    if (!plan_window(&q, n, h, w, c, cout, r, s, pad_w, ho, wo, x, out_weight(e), sms, [&](size_t bytes) { return workspace_possible(bytes, st); }))
        return 0;
    const int cb = q.cb, wp = q.wp, tr = q.tr, bn = q.bn;
    CUtensorMap mx, mx1, mw;
    int rc = encode_window(&mx, x_in, n, h, w, c, cb, wp, tr + r - 1);
    if (rc != SPARQ_OK) return rc;
    rc = encode_window(&mx1, x_in, n, h, w, c, cb, wp, tr);
    if (rc != SPARQ_OK) return rc;
    const int64_t K = (int64_t)r * s * c;
    rc = encode_weights(&mw, wgt, c, cout, r * s, cb, bn, !q.resident ? 1 : r == 3 && s == 3 ? r * s : s);   // as the kernel copies them
    if (rc != SPARQ_OK) return rc;

    WindowArgs g;
    memset(&g, 0, sizeof(g));
    g.N = cout; g.K = K;
    g.n_img = n; g.H = h; g.W = w; g.C = c; g.R = r; g.S = s; g.pad_h = pad_h; g.pad_w = pad_w; g.Ho = ho; g.Wo = wo;
    g.Wp = wp; g.TR = tr; g.tiles_per_img = q.tiles_per_img; g.c_blocks = q.c_blocks;
    g.G = q.grp;
    g.piece0_bytes = cb * wp * (tr + r - 1);
    g.piece_bytes = cb * wp * tr;
    g.n_tiles = (uint32_t)q.n_tiles;
    g.units = (uint32_t)q.units;
    int grid = (int)(q.units < sms ? q.units : sms);
    if (!q.resident && bn == 128) {
        // CTAs own whole groups, so that a group is never cut at a share boundary
        const int64_t groups = (int64_t)n * q.n_tiles * ((q.tiles_per_img + q.grp - 1) / q.grp);
        g.groups = (uint32_t)groups;
        grid = (int)(groups < sms ? groups : sms);
    }
    g.plane_bytes = q.plane_bytes;
    g.win_bufs = q.win_bufs;
    g.b_stages = q.b_stages;
    g.team_copy = q.team_copy ? 1 : 0;
    g.xf = xform_dev(x);
    g.scale = e->scale; g.bias = e->bias; g.relu = e->relu ? 1 : 0; g.inv_out_scale = e->inv_out_scale;
    g.acc_out = e->acc_out; g.f32_out = e->f32_out; g.u8_out = e->u8_out;
    g.status = status;
    g.wait_limit = g_wait_limit;
    g.residual = e->residual;
    g.residual_scale = e->residual_scale;
    rc = next_transform_args(e, g.N, &g.next_mode, &g.next_rnd, &g.next_xf);
    if (rc != SPARQ_OK) return rc;
    cudaError_t ce;
    if (bn == 64) ce = launch_window_shape<64, 64, true>(mx, mx1, mw, g, x.mode, variant_n(x), x.rnd, grid, q.smem_bytes, st);
    else if (bn == 128 && q.resident) ce = launch_window_shape<128, 128, true>(mx, mx1, mw, g, x.mode, variant_n(x), x.rnd, grid, q.smem_bytes, st);
    else if (bn == 128) ce = launch_window_shape<128, 128, false>(mx, mx1, mw, g, x.mode, variant_n(x), x.rnd, grid, q.smem_bytes, st);
    else ce = launch_window_shape<256, 128, false>(mx, mx1, mw, g, x.mode, variant_n(x), x.rnd, grid, q.smem_bytes, st);
    if (ce != cudaSuccess) return cuda_error(ce, "sparq_conv_window_kernel launch");
    return 1;
}

// Tile choice, tensor maps and launch of the fused GEMM.  The caller brings the status word (a
// device pointer); nothing here allocates device memory.
int gemm_with_status(const uint8_t *A, int64_t lda, const int8_t *B, int64_t ldb, int64_t M, int64_t N, int64_t K,
                     const XformArgs &x, const sparq_epilogue *e, unsigned int *status, cudaStream_t st)
{
    int sms = 0;
    int rc = device_info(&sms);
    if (rc != SPARQ_OK) return rc;
    const int64_t pad128 = (K + 127) / 128 * 128, pad64 = (K + 63) / 64 * 64;
    // the step that pads K the least; ties go to the wider one -- and so does a long reduction whose
    // padding stays below an eighth (K = 576: five 128-byte steps instead of nine 64-byte ones: each
    // step is a hand-off between three warp roles, which is what a small launch is made of)
    const int bk = (pad64 < pad128 && !(pad64 >= 320 && pad128 * 8 <= pad64 * 9)) ? 64 : 128;
    const SmallForm small = pick_small(M, N, (K + bk - 1) / bk, sms, x.mode != SPARQ_MODE_NONE);
    const int bn = small.tile_rows ? kSmallBN : pick_bn(M, N, gemm_steps(K, out_bytes(e)), sms, xform_cycles(x));
    const int tile_rows = small.tile_rows ? small.tile_rows : kBM;
    GemmMaps m = {};
    rc = encode_2d(&m.a, A, K, M, lda, bk, tile_rows);
    if (rc != SPARQ_OK) return rc;
    GemmArgs g;
    memset(&g, 0, sizeof(g));
    g.M = M; g.N = N; g.K = K;
    g.k_blocks = (int)((K + bk - 1) / bk);
    rc = fill_common(&g, x, e, status);
    if (rc != SPARQ_OK) return rc;
    const int64_t tiles = ((M + tile_rows - 1) / tile_rows) * ((N + bn - 1) / bn);
    if (tiles >= ((int64_t)1 << 31)) return set_error(SPARQ_ERR_UNSUPPORTED, "more than 2^31 output tiles");
    g.tile_rows = tile_rows;
    g.split = small.split;
    const int grid = small.tile_rows ? (int)tiles * small.split : (int)(tiles < sms ? tiles : sms);
    if ((rc = output_maps(&m, &g, x.mode, bn, tiles, grid)) != SPARQ_OK) return rc;
    if ((rc = encode_b(&m.b, B, K, N, ldb, bk, bn, g, small.tile_rows != 0)) != SPARQ_OK) return rc;
    cudaError_t ce = launch(bn, bk, small.tile_rows != 0, m, g, x, grid, st);
    if (ce != cudaSuccess) return cuda_error(ce, "sparq_gemm_kernel launch");
    return SPARQ_OK;
}

// The convolution through an im2col tensor map (strides, and whatever the window kernel does not tile).
static int im2col_conv(const uint8_t *x_in, int n, int h, int w, int c, const int8_t *wgt, int cout, int r, int s,
                       int stride_h, int stride_w, int pad_h, int pad_w, int ho, int wo, const XformArgs &x, const sparq_epilogue *e,
                       int sms, unsigned int *status, cudaStream_t st)
{
    const int64_t M = (int64_t)n * ho * wo, K = (int64_t)r * s * c;
    const int bk = conv_bk(c);
    const Steps k = conv_steps((int64_t)r * s, c, out_bytes(e));
    const SmallForm small = pick_small(M, cout, k.blocks, sms, x.mode != SPARQ_MODE_NONE);
    const int bn = small.tile_rows ? kSmallBN : pick_bn(M, cout, k, sms, xform_cycles(x));
    int rc;
    const int tile_rows = small.tile_rows ? small.tile_rows : kBM;
    GemmMaps m = {};
    rc = encode_im2col(&m.a, x_in, n, h, w, c, r, s, stride_h, stride_w, pad_h, pad_w, bk, tile_rows);
    if (rc != SPARQ_OK) return rc;
    GemmArgs g;
    memset(&g, 0, sizeof(g));
    g.M = M; g.N = cout; g.K = K;
    // A channel count that is not a multiple of 64 takes a last block that reaches past C: the
    // im2col copy fills those channels with zeros.
    g.c_blocks = (c + bk - 1) / bk;
    g.k_blocks = r * s * g.c_blocks;
    g.conv = 1;
    g.tap_k = c;
    g.S = s;
    g.Ho = ho; g.Wo = wo;
    g.stride_h = stride_h; g.stride_w = stride_w; g.pad_h = pad_h; g.pad_w = pad_w;
    rc = fill_common(&g, x, e, status);
    if (rc != SPARQ_OK) return rc;
    const int64_t tiles = ((M + tile_rows - 1) / tile_rows) * ((cout + bn - 1) / bn);
    if (tiles >= ((int64_t)1 << 31)) return set_error(SPARQ_ERR_UNSUPPORTED, "more than 2^31 output tiles");
    g.tile_rows = tile_rows;
    g.split = small.split;
    const int grid = small.tile_rows ? (int)tiles * small.split : (int)(tiles < sms ? tiles : sms);
    if ((rc = output_maps(&m, &g, x.mode, bn, tiles, grid)) != SPARQ_OK) return rc;
    if ((rc = encode_b(&m.b, wgt, K, cout, K, bk, bn, g, small.tile_rows != 0)) != SPARQ_OK) return rc;
    cudaError_t ce = launch(bn, bk, small.tile_rows != 0, m, g, x, grid, st);
    if (ce != cudaSuccess) return cuda_error(ce, "sparq_gemm_kernel (convolution) launch");
    return SPARQ_OK;
}

cudaError_t launch_x24(int bn, const CUtensorMap &ma, const CUtensorMap &mb, const GemmArgs &g, int n, int rnd, int grid, cudaStream_t st);

// The 2:4 product with the expansion inside the kernel (sparq_gemm_sparse24_kernel), arguments checked by
// the caller.  Returns 1 if it launched, 0 if expanding into the workspace first is expected to be faster, < 0 on error.
int gemm_sparse24_fused(const uint8_t *A, const int8_t *w_exp, int64_t M, int64_t N, int64_t K, const XformArgs &x,
                        const sparq_epilogue *e, cudaStream_t st)
{
    int sms = 0, rc = device_info(&sms);
    if (rc != SPARQ_OK) return rc;
    // A tile of 256 rows is expanded once per column tile, about 4200 cycles per 128 activations of its
    // rows; the other form moves 4 bytes per activation through HBM and multiplies at K' = 3K.  Few
    // tiles: that product can be shared by clusters.
    const int64_t steps = (K + 127) / 128, steps3 = (3 * K + 127) / 128;
    if (pick_small(M, N, steps3, sms, false).tile_rows) return 0;
    const int bn = N <= 64 ? 64 : 128;
    const int64_t tiles = (M + 255) / 256 * ((N + bn - 1) / bn);
    double plain;
    pick_bn(M, N, gemm_steps(3 * K, out_bytes(e)), sms, 0.0, &plain);
    const double fused = (double)((tiles + sms - 1) / sms) * (double)steps * 4200.0;
    if (tiles >= (int64_t)1 << 31 || fused > plain + 1900.0 * (2.5 + (double)M * (double)K * 4.0 / 6.0e6)) return 0;
    CUtensorMap ma, mb;
    if ((rc = encode_2d(&ma, A, K, M, K, 128, 256)) != SPARQ_OK) return rc;
    if ((rc = encode_2d(&mb, w_exp, 3 * K, N, 3 * K, 128, bn)) != SPARQ_OK) return rc;
    unsigned int *status = nullptr;
    if ((rc = get_status_word(&status)) != SPARQ_OK) return rc;
    GemmArgs g;
    memset(&g, 0, sizeof(g));
    g.M = M; g.N = N; g.K = 3 * K;
    g.k_blocks = (int)steps;
    if ((rc = fill_common(&g, x, e, status)) != SPARQ_OK) return rc;
    const cudaError_t ce = launch_x24(bn, ma, mb, g, variant_n(x), x.rnd, (int)(tiles < sms ? tiles : sms), st);
    return ce == cudaSuccess ? 1 : cuda_error(ce, "sparq_gemm_sparse24_kernel launch");
}

int check_epilogue_args(const sparq_epilogue *e) { return check_epilogue(e); }

// e->next_transform for N output columns: before anything is enqueued, for entry points of several kernels.
int check_next_transform(const sparq_epilogue *e, int64_t N)
{
    int mode, rnd;
    XformDev xf;
    return next_transform_args(e, N, &mode, &rnd, &xf);
}

}  // namespace sparq

using namespace sparq;

extern "C" int sparq_gemm_s8(const uint8_t *A, int64_t lda, const int8_t *B, int64_t ldb,
                             int64_t M, int64_t N, int64_t K,
                             const sparq_params *p, const sparq_epilogue *e, void *stream)
{
    XformArgs x;
    int rc = validate_params(p, &x);
    if (rc != SPARQ_OK) return rc;
    rc = check_epilogue(e);
    if (rc != SPARQ_OK) return rc;
    if (M < 0 || N < 0 || K < 0) return set_error(SPARQ_ERR_INVALID_ARG, "negative dimension");
    if (M == 0 || N == 0) return SPARQ_OK;
    if (!A || !B) return set_error(SPARQ_ERR_INVALID_ARG, "A or B is NULL");
    if (K == 0 || K % 16 || K > 65536) return set_error(SPARQ_ERR_UNSUPPORTED, "K = %lld must be a multiple of 16 in [16, 65536]", (long long)K);
    if (lda < K || ldb < K || lda % 16 || ldb % 16)
        return set_error(SPARQ_ERR_UNSUPPORTED, "lda/ldb must be multiples of 16 and at least K");
    if (((uintptr_t)A | (uintptr_t)B) & 15u) return set_error(SPARQ_ERR_UNSUPPORTED, "A and B must be 16-byte aligned");
    if (M > (int64_t)1 << 31 || N > (int64_t)1 << 31) return set_error(SPARQ_ERR_UNSUPPORTED, "M or N too large");
    if ((rc = check_next_transform(e, N)) != SPARQ_OK) return rc;
    return gemm_impl(A, lda, B, ldb, M, N, K, x, e, (cudaStream_t)stream);
}

extern "C" int sparq_conv2d_nhwc_s8(const uint8_t *x_in, int n, int h, int w, int c,
                                    const int8_t *wgt, int cout, int r, int s,
                                    int stride_h, int stride_w, int pad_h, int pad_w,
                                    const sparq_params *p, const sparq_epilogue *e, void *stream)
{
    XformArgs x;
    int rc = validate_params(p, &x);
    if (rc != SPARQ_OK) return rc;
    rc = check_epilogue(e);
    if (rc != SPARQ_OK) return rc;
    if (n < 0 || h < 0 || w < 0 || c < 0 || cout < 0) return set_error(SPARQ_ERR_INVALID_ARG, "negative dimension");
    if (r < 1 || s < 1 || stride_h < 1 || stride_w < 1 || pad_h < 0 || pad_w < 0)
        return set_error(SPARQ_ERR_INVALID_ARG, "filter size and strides must be >= 1, pads >= 0");
    if (r > 7 || s > 7 || stride_h > 8 || stride_w > 8 || pad_h >= r || pad_w >= s)
        return set_error(SPARQ_ERR_UNSUPPORTED, "filter up to 7x7, strides up to 8, pads below the filter size");
    if (n == 0 || cout == 0) return SPARQ_OK;
    if (h + 2 * pad_h < r || w + 2 * pad_w < s) return set_error(SPARQ_ERR_INVALID_ARG, "filter larger than the padded image");
    if (!x_in || !wgt) return set_error(SPARQ_ERR_INVALID_ARG, "x or wgt is NULL");
    if (c == 0 || c % 16) return set_error(SPARQ_ERR_UNSUPPORTED, "c = %d must be a positive multiple of 16", c);
    if (((uintptr_t)x_in | (uintptr_t)wgt) & 15u) return set_error(SPARQ_ERR_UNSUPPORTED, "x and wgt must be 16-byte aligned");
    const int ho = (h + 2 * pad_h - r) / stride_h + 1;
    const int wo = (w + 2 * pad_w - s) / stride_w + 1;
    const int64_t M = (int64_t)n * ho * wo;
    const int64_t K = (int64_t)r * s * c;
    if (K > 65536) return set_error(SPARQ_ERR_UNSUPPORTED, "r*s*c = %lld exceeds 65536", (long long)K);
    // Beyond, the kernels' 32-bit coordinates (of a matrix row, of an output pixel) would wrap.
    const bool matrix = r == 1 && s == 1 && stride_h == 1 && stride_w == 1 && pad_h == 0 && pad_w == 0;
    if (M > (matrix ? (int64_t)1 << 31 : (int64_t)0xFFFFFFFF)) return set_error(SPARQ_ERR_UNSUPPORTED, "%lld output pixels are too many for one call", (long long)M);
    if ((rc = check_next_transform(e, cout)) != SPARQ_OK) return rc;
    cudaStream_t st = (cudaStream_t)stream;

    // A 1x1 filter with unit stride reads the NHWC tensor as the M x c matrix it already is.
    if (matrix) return gemm_impl(x_in, c, wgt, c, M, cout, c, x, e, st);

    int sms = 0;
    rc = device_info(&sms);
    if (rc != SPARQ_OK) return rc;
    unsigned int *status = nullptr;
    rc = get_status_word(&status);
    if (rc != SPARQ_OK) return rc;
    if (stride_h == 1 && stride_w == 1) {
        rc = try_window_conv(x_in, n, h, w, c, wgt, cout, r, s, pad_h, pad_w, ho, wo, x, e, sms, status, st);
        if (rc != 0) return rc < 0 ? rc : SPARQ_OK;
    }
    const size_t act_bytes = (size_t)n * h * w * (size_t)c;
    if (x.mode != SPARQ_MODE_NONE && transform_first(M, cout, conv_steps((int64_t)r * s, c, out_bytes(e)), x, act_bytes, sms)) {
        if (uint8_t *tx = (uint8_t *)workspace_alloc(act_bytes, st)) {
            rc = quantize_rows(x_in, tx, (size_t)n * h * w, (size_t)c, x, true, st);
            if (rc == SPARQ_OK) rc = im2col_conv(tx, n, h, w, c, wgt, cout, r, s, stride_h, stride_w, pad_h, pad_w, ho, wo, plain_a8w8(), e, sms, status, st);
            workspace_free(tx, st);
            return rc;
        }
    }
    return im2col_conv(x_in, n, h, w, c, wgt, cout, r, s, stride_h, stride_w, pad_h, pad_w, ho, wo, x, e, sms, status, st);
}

extern "C" int sparq_selftest_form(int n, int h, int w, int c, int cout, int r, int s, int stride_h, int stride_w, int pad_h, int pad_w,
                                   const sparq_params *p, int sms)
{
    XformArgs x;
    const int rc = validate_params(p, &x);
    if (rc != SPARQ_OK) return rc;
    if (n < 1 || h < 1 || w < 1 || c < 16 || c % 16 || cout < 1 || r < 1 || s < 1 || r > 7 || s > 7 || stride_h < 1 || stride_w < 1 ||
        pad_h < 0 || pad_w < 0 || pad_h >= r || pad_w >= s || h + 2 * pad_h < r || w + 2 * pad_w < s || sms < 1)
        return set_error(SPARQ_ERR_INVALID_ARG, "bad convolution geometry");
    const int ho = (h + 2 * pad_h - r) / stride_h + 1, wo = (w + 2 * pad_w - s) / stride_w + 1;
    const int64_t M = (int64_t)n * ho * wo;
    const bool matrix = r == 1 && s == 1 && stride_h == 1 && stride_w == 1;
    WindowPlan q;
    auto scratch = [](size_t bytes) { return bytes <= kWorkspaceMaxBytes; };
    if (!matrix && stride_h == 1 && stride_w == 1 && plan_window(&q, n, h, w, c, cout, r, s, pad_w, ho, wo, x, 1.0, sms, scratch))
        return q.resident ? SPARQ_FORM_WINDOW_RESIDENT : SPARQ_FORM_WINDOW_STREAMED;
    const Steps k = matrix ? gemm_steps(c, 1.0) : conv_steps((int64_t)r * s, c, 1.0);
    const size_t act_bytes = (size_t)n * h * w * (size_t)c;
    if (x.mode != SPARQ_MODE_NONE && transform_first(M, cout, k, x, act_bytes, sms) && scratch(act_bytes)) return SPARQ_FORM_TRANSFORM_FIRST;
    return pick_small(M, cout, k.blocks, sms, x.mode != SPARQ_MODE_NONE).tile_rows ? SPARQ_FORM_SMALL : SPARQ_FORM_FULL;
}
