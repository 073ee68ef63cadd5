// Standalone bSPARQ / vSPARQ transform (Sections 3.1-3.2): uint8 in, uint8 out.
//
// Fast path: the tensor is a flat array of 16-byte vectors.  With an even row length
// every pair (2j, 2j+1) of a row is also an aligned byte pair of the flat array, so rows
// need no special care.  Each thread streams kVec independent 16-byte loads, transforms
// the sixteen 32-bit words in registers and streams them back; the kernel is bound by
// HBM traffic (one byte read, one written per activation).
//
// Odd row lengths with the pair rule: pairs of an odd row are shifted by one byte against the flat
// array's, and the last value of a row has no partner.  Same vectors, with the partner of every
// byte taken from a mask of non-zero bytes shifted to either side.
//
// Generic path: one thread per pair with the scalar form of the same definitions; used
// for unaligned buffers, odd rows shorter than a vector, and the last bytes of other tensors.
#include <type_traits>

#include "sparq_common.cuh"

namespace sparq {

constexpr int kThreads = 256;
constexpr int kVec = 4;  // 16-byte vectors per thread per iteration

__device__ __forceinline__ uint4 ld_stream(const uint4 *p)
{
    uint4 v;
    asm volatile("ld.global.cs.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}

__device__ __forceinline__ void st_stream(uint4 *p, uint4 v)
{
    asm volatile("st.global.cs.v4.u32 [%0], {%1,%2,%3,%4};"
                 :: "l"(p), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}

// release_first: the next launch starts while this one works, for a contraction that reads the result (one
// CTA per SM, set up meanwhile).  Else it starts at the end: blocks of a streaming successor that take
// the free places of the SMs early are spread over them unevenly (10 MB: 4.5 -> 5.4 us).
// XN: the form of the transform, as in xform_fused.  The 3- and 2-bit full sets take the half-precision
// one: with the packed-integer form at their compile-time width the kernel was bound by the integer
// pipe (2^28 activations, vSPARQ: 6opt 105 -> 82 us, 7opt 119 -> 82 us, the measured copy rate).
template <int MODE, int XN, bool RND>
__global__ void __launch_bounds__(kThreads)
quantize_vec_kernel(const uint4 *in, uint4 *out, size_t nvec, XformDev d, int release_first)
{
    dep_wait();
    if (release_first) dep_launch();
    const size_t tile = (size_t)kThreads * kVec;
    for (size_t base = (size_t)blockIdx.x * tile; base < nvec; base += (size_t)gridDim.x * tile) {
        uint4 v[kVec];
        size_t idx[kVec];
#pragma unroll
        for (int j = 0; j < kVec; ++j) {
            idx[j] = base + (size_t)j * kThreads + threadIdx.x;
            if (idx[j] < nvec) v[j] = ld_stream(in + idx[j]);
        }
#pragma unroll
        for (int j = 0; j < kVec; ++j) {
            if (idx[j] < nvec) {
                uint4 o;
                o.x = xform_fused<MODE, XN, RND>(v[j].x, d);
                o.y = xform_fused<MODE, XN, RND>(v[j].y, d);
                o.z = xform_fused<MODE, XN, RND>(v[j].z, d);
                o.w = xform_fused<MODE, XN, RND>(v[j].w, d);
                st_stream(out + idx[j], o);
            }
        }
    }
    if (!release_first) dep_launch();
}

// vSPARQ on rows of odd length (>= 16, so that a vector meets at most one row boundary).  Column parity is
// the parity of (flat index + row): in even rows byte pairs are those of the flat array, in odd rows
// they are shifted by one.  200000 x 1025: 437 us a pair per thread, 142 us here (bound by the integer
// pipe: both masks, the blend at a row's end and two windows).  magic = floor(2^64 / row_len).  `bytes`: of the whole tensor, whose bytes
// beside a vector are read for its outer partners (in place too: the transform keeps zero zero and
// everything else non-zero).
constexpr int kOddVec = 2;
// Below, a pair per thread spreads over more SMs (16 KB: 1.85 us against 2.45; 100 KB 2.0 against 2.1).
constexpr size_t kOddVecMin = 128 << 10;
template <int XN, bool RND>
__global__ void __launch_bounds__(kThreads)
quantize_odd_rows_kernel(const uint8_t *in, uint8_t *out, size_t bytes, size_t row_len, unsigned long long magic, XformDev d)
{
    dep_wait();
    const size_t nvec = (bytes + 15) / 16, tile = (size_t)kThreads * kOddVec;
    for (size_t base = (size_t)blockIdx.x * tile; base < nvec; base += (size_t)gridDim.x * tile) {
        uint4 v[kOddVec];
        uint32_t before[kOddVec], after[kOddVec];
        size_t idx[kOddVec];
#pragma unroll
        for (int j = 0; j < kOddVec; ++j) {
            idx[j] = base + (size_t)j * kThreads + threadIdx.x;
            if (idx[j] >= nvec) continue;
            if (16 * idx[j] + 16 <= bytes) {
                v[j] = *reinterpret_cast<const uint4 *>(in + 16 * idx[j]);
            } else {                                                       // the tensor's last bytes
                uint32_t t[4] = {0u, 0u, 0u, 0u};
#pragma unroll
                for (int i = 0; i < 15; ++i)
                    if (16 * idx[j] + i < bytes) t[i >> 2] |= (uint32_t)in[16 * idx[j] + i] << (8 * (i & 3));
                v[j] = make_uint4(t[0], t[1], t[2], t[3]);
            }
            before[j] = idx[j] ? in[16 * idx[j] - 1] : 0u;
            after[j] = 16 * idx[j] + 16 < bytes ? in[16 * idx[j] + 16] : 0u;
        }
#pragma unroll
        for (int j = 0; j < kOddVec; ++j) {
            if (idx[j] >= nvec) continue;
            const size_t i0 = 16 * idx[j];
            size_t row = (size_t)__umul64hi(i0, magic);
            if ((row + 1) * row_len <= i0) ++row;                          // the estimate is at most one short
            const size_t end = (row + 1) * row_len - i0;                   // bytes of this row from here on
            const int cut = end < 17 ? (int)end : 17;                      // 17: the row goes on past the vector
            const uint32_t x[4] = {v[j].x, v[j].y, v[j].z, v[j].w};
            uint32_t nz[6], o[4];
            nz[0] = before[j] ? 0x80000000u : 0u;
            nz[5] = after[j] ? 0x80u : 0u;
#pragma unroll
            for (int w = 0; w < 4; ++w) nz[w + 1] = (((x[w] & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | x[w]);
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                const uint32_t left = prmt(nz[w], nz[w + 1], 0x6543u), right = prmt(nz[w + 1], nz[w + 2], 0x4321u);   // byte i: of i - 1, i + 1
                const uint32_t flat = prmt(nz[w + 1], nz[w + 1], 0xAB89u);          // partner non-zero, flat pairs
                const uint32_t shifted = prmt(left, right, 0xFAD8u);                // bytes l0 r1 l2 r3
                // bytes of this word that belong to the next row
                const int first = cut - 4 * w;                                       // first byte of the next row
                const uint32_t nxt = first <= 0 ? 0xFFFFFFFFu : first >= 4 ? 0u : 0xFFFFFFFFu << (8 * first);
                const uint32_t a = row & 1 ? shifted : flat, b = row & 1 ? flat : shifted;
                uint32_t partner = (a & ~nxt) | (b & nxt);
                if (first >= 1 && first <= 4) partner &= ~(0xFFu << (8 * (first - 1)));   // the row's last value has no partner
                uint32_t q, l;
                window_and_lone<XN, RND>(x[w], d, q, l);
                o[w] = (q & partner) | (l & ~partner);
            }
            if (i0 + 16 <= bytes) {
                st_stream(reinterpret_cast<uint4 *>(out + i0), make_uint4(o[0], o[1], o[2], o[3]));
            } else {
#pragma unroll
                for (int i = 0; i < 15; ++i)
                    if (i0 + i < bytes) out[i0 + i] = (uint8_t)(o[i >> 2] >> (8 * (i & 3)));
            }
        }
    }
    dep_launch();
}

// ---- scalar definitions (generic path) -----------------------------------------------

// One activation: leading one -> lowest allowed placement that covers it -> trim / round.
__device__ unsigned scalar_window(unsigned x, int w, unsigned mask, int rnd)
{
    if (x == 0) return 0;
    int p = 31 - __clz((int)x);
    int s = p - w + 1;
    if (s < 0) s = 0;
    while (!((mask >> s) & 1u)) ++s;          // the top placement is always allowed
    unsigned q = (x >> s) << s;
    if (rnd && s > 0 && ((x >> (s - 1)) & 1u)) {
        unsigned up = q + (1u << s);
        if (up <= 255u) q = up;               // otherwise stay at the all-ones top window
    }
    return q;
}

__global__ void quantize_pair_kernel(const uint8_t *in, uint8_t *out,
                                     size_t rows, size_t row_len, XformArgs a)
{
    dep_wait();
    const size_t pairs_per_row = (row_len + 1) / 2;
    const size_t total = rows * pairs_per_row;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += (size_t)gridDim.x * blockDim.x) {
        size_t r = i / pairs_per_row, j = i % pairs_per_row;
        size_t k0 = r * row_len + 2 * j;
        bool has_b = (2 * j + 1) < row_len;
        unsigned x0 = in[k0], x1 = has_b ? in[k0 + 1] : 0u;
        unsigned q0, q1;
        if (a.mode == SPARQ_MODE_NONE) {
            q0 = x0; q1 = x1;
        } else if (a.mode == SPARQ_MODE_VSPARQ && (x0 == 0 || x1 == 0)) {
            // the lone non-zero owns 2n bits, at any shift 0 .. 8-2n
            int w2 = 2 * a.n;
            unsigned full = (1u << (8 - w2 + 1)) - 1u;
            q0 = (w2 >= 8) ? x0 : scalar_window(x0, w2, full, a.rnd);
            q1 = (w2 >= 8) ? x1 : scalar_window(x1, w2, full, a.rnd);
        } else {
            q0 = scalar_window(x0, a.n, a.mask, a.rnd);
            q1 = scalar_window(x1, a.n, a.mask, a.rnd);
        }
        out[k0] = (uint8_t)q0;
        if (has_b) out[k0 + 1] = (uint8_t)q1;
    }
    dep_launch();
}

// Launches `kernel<XN, RND>` (given as a generic lambda over integral constants) for the parameters.
template <class F>
static cudaError_t by_variant(const XformArgs &a, F go)
{
    using std::integral_constant;
    if (a.widen_rounds > 0 && a.n == 4) return a.rnd ? go(integral_constant<int, 5>(), std::true_type()) : go(integral_constant<int, 5>(), std::false_type());
    if (a.widen_rounds > 0 && a.n == 3) return a.rnd ? go(integral_constant<int, 3>(), std::true_type()) : go(integral_constant<int, 3>(), std::false_type());
    if (a.widen_rounds > 0) return a.rnd ? go(integral_constant<int, 2>(), std::true_type()) : go(integral_constant<int, 2>(), std::false_type());
    if (a.n != 4) return go(integral_constant<int, 8>(), std::true_type());
    return a.rnd ? go(integral_constant<int, 4>(), std::true_type()) : go(integral_constant<int, 4>(), std::false_type());
}

template <int MODE>
static cudaError_t launch_vec(const uint4 *in, uint4 *out, size_t nvec, const XformArgs &a, int blocks, bool feeds, cudaStream_t st)
{
    XformDev d{a.widen_c, a.widen_rounds, a.n};
    fill_fullset(&d, a.n, a.rnd);
    return by_variant(a, [&](auto xn, auto rnd) {
        return launch_overlapped(quantize_vec_kernel<MODE, decltype(xn)::value, decltype(rnd)::value>, blocks, kThreads, 0, st, in, out, nvec, d, (int)feeds);
    });
}

static cudaError_t launch_odd_rows(const uint8_t *in, uint8_t *out, size_t bytes, size_t row_len, const XformArgs &a, int blocks, cudaStream_t st)
{
    XformDev d{a.widen_c, a.widen_rounds, a.n};
    fill_fullset(&d, a.n, a.rnd);
    const unsigned long long magic = ~0ull / row_len;       // floor(2^64 / row_len): row_len is odd and above 1
    return by_variant(a, [&](auto xn, auto rnd) {
        return launch_overlapped(quantize_odd_rows_kernel<decltype(xn)::value, decltype(rnd)::value>, blocks, kThreads, 0, st, in, out, bytes, row_len, magic, d);
    });
}

int quantize_rows(const uint8_t *in, uint8_t *out, size_t rows, size_t row_len, const XformArgs &a, bool feeds, cudaStream_t st)
{
    if (rows == 0 || row_len == 0) return SPARQ_OK;
    if (!in || !out) return set_error(SPARQ_ERR_INVALID_ARG, "in/out pointer is NULL");
    if (rows > ((size_t)1 << 62) / row_len) return set_error(SPARQ_ERR_INVALID_ARG, "rows * row_len overflows");
    const size_t total = rows * row_len;
    if (in != out) {
        const uint8_t *lo = in < (const uint8_t *)out ? in : out;
        const uint8_t *hi = in < (const uint8_t *)out ? out : in;
        if (lo + total > hi) return set_error(SPARQ_ERR_INVALID_ARG, "in and out overlap partially");
    }
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return cuda_error(e, "device query");

    const bool pairs_flat = (a.mode != SPARQ_MODE_VSPARQ) || (row_len % 2 == 0);
    const bool aligned = (((uintptr_t)in | (uintptr_t)out) & 15u) == 0;
    size_t done = 0;
    if (pairs_flat && aligned && total >= 16) {
        const size_t nvec = total / 16;
        const size_t tile = (size_t)kThreads * kVec;
        size_t want = (nvec + tile - 1) / tile;
        size_t cap = (size_t)sms * 64;   // grid-stride beyond this many blocks
        int blocks = (int)(want < cap ? want : cap);
        const uint4 *vi = (const uint4 *)in;
        uint4 *vo = (uint4 *)out;
        if (a.mode == SPARQ_MODE_NONE) e = launch_vec<SPARQ_MODE_NONE>(vi, vo, nvec, a, blocks, feeds, st);
        else if (a.mode == SPARQ_MODE_BSPARQ) e = launch_vec<SPARQ_MODE_BSPARQ>(vi, vo, nvec, a, blocks, feeds, st);
        else e = launch_vec<SPARQ_MODE_VSPARQ>(vi, vo, nvec, a, blocks, feeds, st);
        if (e != cudaSuccess) return cuda_error(e, "quantize_vec_kernel launch");
        done = nvec * 16;
        if (done == total) return SPARQ_OK;
    }
    if (!pairs_flat && aligned && row_len >= 16 && total > kOddVecMin) {
        const size_t tile = (size_t)kThreads * kOddVec, want = ((total + 15) / 16 + tile - 1) / tile, cap = (size_t)sms * 64;
        e = launch_odd_rows(in, out, total, row_len, a, (int)(want < cap ? want : cap), st);
        if (e != cudaSuccess) return cuda_error(e, "quantize_odd_rows_kernel launch");
        return SPARQ_OK;
    }
    // Remainder (or everything, when the fast path does not apply).  With pairs_flat the
    // remaining bytes start at an even offset and form one pseudo-row.
    size_t g_rows = pairs_flat ? 1 : rows;
    size_t g_len = pairs_flat ? total - done : row_len;
    size_t npairs = g_rows * ((g_len + 1) / 2);
    size_t want = (npairs + 255) / 256;
    size_t cap = (size_t)sms * 32;
    int blocks = (int)(want < cap ? want : cap);
    if (blocks < 1) blocks = 1;
    e = launch_overlapped(quantize_pair_kernel, blocks, 256, 0, st, in + done, out + done, g_rows, g_len, a);
    if (e != cudaSuccess) return cuda_error(e, "quantize_pair_kernel launch");
    return SPARQ_OK;
}

}  // namespace sparq

using namespace sparq;

extern "C" int sparq_quantize(const uint8_t *in, uint8_t *out, size_t rows, size_t row_len,
                              const sparq_params *p, void *stream)
{
    XformArgs a;
    const int rc = validate_params(p, &a);
    return rc != SPARQ_OK ? rc : quantize_rows(in, out, rows, row_len, a, false, (cudaStream_t)stream);
}
