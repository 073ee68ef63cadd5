// Shared host/device pieces of the SPARQ library: error reporting, parameter
// validation, and the packed (4 activations per 32-bit word) form of the
// bSPARQ / vSPARQ transform used by both the standalone kernel and the fused GEMM.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "sparq.h"

namespace sparq {

// ---- host side ---------------------------------------------------------------------

int set_error(int code, const char *fmt, ...);
int cuda_error(cudaError_t e, const char *what);

// Host-validated, kernel-ready description of the transform.
struct XformArgs {
    int mode;           // SPARQ_MODE_*
    int n;              // window bits: 2, 3, 4
    int rnd;            // 0 trim, 1 nearest
    int widen_rounds;   // longest run of consecutive disallowed shifts
    uint32_t widen_c;   // per byte: bit d set for every disallowed shift d (0 < d < 8-n)
    uint32_t mask;      // placement mask as given
};

// Checks `p` (Section 3.1 placement sets, Section 5.1 widths) and fills `x`.
int validate_params(const sparq_params *p, XformArgs *x);

// Device status word shared by all kernels of this library on the current device.
// Bit 0: a bounded wait expired.  Allocated on first use, freed by sparq_shutdown().
int get_status_word(unsigned int **dptr);

// The standalone transform (sparq_quantize) with validated parameters.  feeds: the next launch is the
// contraction that reads `out`.
int quantize_rows(const uint8_t *in, uint8_t *out, size_t rows, size_t row_len, const XformArgs &a, bool feeds, cudaStream_t st);

// Stream-ordered scratch memory (sparq_workspace.cu): valid for work enqueued on `st` after the call
// and before the matching workspace_free.  Any thread, any stream.  nullptr when there is none to be
// had, and while the stream is being captured (the caller then takes a path without it).
// A larger scratch tensor is not worth taking from the user's device: its caller has a path without.
constexpr size_t kWorkspaceMaxBytes = (size_t)1 << 30;
bool workspace_possible(size_t bytes, cudaStream_t st);     // whether it is worth asking
void *workspace_alloc(size_t bytes, cudaStream_t st);
void workspace_free(void *p, cudaStream_t st);

// ---- overlapped launches ----------------------------------------------------------------
// The library's kernels are launched with programmatic stream serialization: a kernel may start,
// and set itself up, while its predecessor on the stream is finishing.  dep_wait() blocks until
// every earlier kernel has completed and its writes are visible; no thread touches the caller's
// memory before it.  dep_launch() lets the next kernel start.
#ifdef __CUDACC__
__device__ __forceinline__ void dep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <class Kernel, class... Args>
cudaError_t launch_overlapped_cluster(Kernel kernel, int grid, int cluster, int threads, int smem_bytes, cudaStream_t st, const Args &...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = (size_t)smem_bytes;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)cluster;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

template <class Kernel, class... Args>
cudaError_t launch_overlapped(Kernel kernel, int grid, int threads, int smem_bytes, cudaStream_t st, const Args &...args)
{
    return launch_overlapped_cluster(kernel, grid, 1, threads, smem_bytes, st, args...);
}
#endif

// ---- device side -------------------------------------------------------------------

#define SPARQ_HD __host__ __device__ __forceinline__

// prmt.b32: byte i of the result is byte (sel nibble i & 7) of {b:a}; nibble bit 3 asks
// for that byte's top bit replicated over all eight bits instead.
SPARQ_HD uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel)
{
#ifdef __CUDA_ARCH__
    uint32_t d;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
    return d;
#else
    uint64_t src = ((uint64_t)b << 32) | a;
    uint32_t d = 0;
    for (int i = 0; i < 4; ++i) {
        uint32_t nib = (sel >> (4 * i)) & 0xFu;
        uint32_t byte = (uint32_t)(src >> (8 * (nib & 7u))) & 0xFFu;
        if (nib & 8u) byte = (byte & 0x80u) ? 0xFFu : 0u;
        d |= byte << (8 * i);
    }
    return d;
#endif
}

// Kernel-side copy of the placement-set constants of XformArgs.
struct XformDev {
    uint32_t widen_c;
    int rounds;
    int n;
    // Full placement sets only (every shift 0..8-n allowed; see xform_word_fullset): per 16-bit
    // half, twice in a word -- the rounding increment, the mask of the kept bits and the
    // largest sum that still trims to the top window, of the n-bit window (f_*) and of the 2n-bit
    // window of a lone non-zero (l_*).
    uint32_t f_add, f_mask, f_top;
    uint32_t l_add, l_mask, l_top;
};

// binary16 bit pattern of an integer 0 < v < 2048 (exact)
inline uint32_t half_bits_of_int(uint32_t v)
{
    int p = 0;
    while ((v >> (p + 1)) != 0) ++p;
    return ((uint32_t)(p + 15) << 10) | ((v << (10 - p)) & 0x3FFu);
}

// Constants of xform_word_fullset for window width n and the rounding flag (at n = 4 it has its own, and a lone
// non-zero keeps all bits).
inline void fill_fullset(XformDev *d, int n, int rnd)
{
    auto set = [&](int w, uint32_t *add, uint32_t *mask, uint32_t *top) {
        const uint32_t m16 = (0xFFFFu << (11 - w)) & 0xFFFFu;      // sign, exponent and the top w-1 fraction bits
        const uint32_t a16 = rnd ? (1u << (10 - w)) : 0u;          // half of the lowest kept bit
        *mask = m16 * 0x00010001u;
        *add = a16 * 0x00010001u;
        *top = (half_bits_of_int(((1u << w) - 1u) << (8 - w)) | (~m16 & 0xFFFFu)) * 0x00010001u;
    };
    set(n, &d->f_add, &d->f_mask, &d->f_top);
    if (n < 4) set(2 * n, &d->l_add, &d->l_mask, &d->l_top);
}

// Mask of the bits BELOW the window for each of the four bytes of x (Section 3.1: the
// window's top bit is the leading one, or the window sits at the bottom).  The window
// width is WT when WT != 0, else the run-time value w_rt.  With WIDEN, a window that landed
// on a disallowed placement moves up to the next allowed one: one step `m |= (m << 1) & c`
// moves every byte that sits on a disallowed shift up by one and leaves the others alone,
// so three unconditional steps cover the longest possible run (n - 1 <= 3) and need no
// branch.
template <int WT, bool WIDEN>
SPARQ_HD uint32_t drop_mask(uint32_t x, int w_rt, uint32_t widen_c)
{
    const int w = WT ? WT : w_rt;
    const uint32_t low = 0x01010101u * (0xFFu >> w);
    uint32_t m = (x >> w) & low;                 // bits of x above the lowest window
    m |= (m >> 1) & 0x7F7F7F7Fu;                 // smear the leading one downwards
    if (!WT || 8 - WT > 2) m |= (m >> 2) & 0x3F3F3F3Fu;
    if (!WT || 8 - WT > 4) m |= (m >> 4) & 0x0F0F0F0Fu;
    if (WIDEN) {
        m |= (m << 1) & widen_c;
        m |= (m << 1) & widen_c;
        m |= (m << 1) & widen_c;
    }
    return m;
}

// Trim or round four bytes given their drop masks (w = window width).  Rounding adds
// half a window LSB; a byte that would overflow 8 bits (only possible at the highest
// placement, where the half is 0x80 >> w) keeps its trimmed value, i.e. saturates to
// the all-ones window.
template <bool RND>
SPARQ_HD uint32_t apply_mask(uint32_t x, uint32_t m, int w)
{
    if (!RND) return x & ~m;
    uint32_t half = m ^ ((m >> 1) & 0x7F7F7F7Fu);   // (m + 1) >> 1 per byte
    uint32_t x7 = x & 0x7F7F7F7Fu, x8 = x & 0x80808080u;
    uint32_t lo = x7 + half;                        // no carry leaves a byte
    uint32_t ovf = lo & x8;                         // bit 7: x + half >= 256
    lo -= ovf >> w;
    return (lo ^ x8) & ~m;
}

// T on four packed activations (bytes 0,1 and bytes 2,3 are the pairs of Eq. 2).
// N = 2, 3, 4 fixes the window width at compile time; N = 0 takes it from d.n.
// WIDEN = false is only valid for full placement sets (d.rounds == 0).
template <int MODE, int N, bool RND, bool WIDEN>
SPARQ_HD uint32_t xform_word(uint32_t x, const XformDev &d)
{
    if (MODE == SPARQ_MODE_NONE) return x;
    const int n = N ? N : d.n;
    uint32_t q = apply_mask<RND>(x, drop_mask<N, WIDEN>(x, n, d.widen_c), n);
    if (MODE == SPARQ_MODE_BSPARQ) return q;
    // vSPARQ: a byte whose partner is zero keeps the 2n-bit budget (all 8 bits for n = 4;
    // a 2n-bit window at any shift 0..8-2n otherwise, Section 5.1).
    uint32_t lone = x;
    if (N == 2 || N == 3) {
        lone = apply_mask<RND>(x, drop_mask<(N == 4 ? 0 : 2 * N), false>(x, 2 * n, 0u), 2 * n);
    } else if (N == 0) {
        // run-time width: n = 4 gives a window of 8 bits, whose drop mask is empty
        const int w2 = 2 * n;
        lone = apply_mask<RND>(x, w2 < 8 ? drop_mask<0, false>(x, w2, 0u) : 0u, w2 < 8 ? w2 : 7);
    }
    uint32_t nz = ((x & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | x;   // bit 7 of each byte: byte != 0
    uint32_t partner_nz = prmt(nz, nz, 0xAB89u);           // swap within pairs, replicate bit 7
    return (q & partner_nz) | (lone & ~partner_nz);
}

#ifdef __CUDACC__
// ---- full placement sets: the window through the floating-point unit --------------------------
// With every shift allowed, bSPARQ keeps the n most significant bits starting at the leading
// one (Section 3.1) -- which is what a binary floating-point number with n - 1 fraction bits
// holds.  A byte b is exact in binary16 (11 significant bits); as bit patterns, two bytes per
// 32-bit register:
//     0x6400 | b               = 1024 + b       (one byte permute per pair)
//     (1024 + b) - 1024        = b, normalized: the subtraction finds the leading one
//     min(bits + half, top)    the rounding increment, ties up, a carry moving into the exponent
//                              (31 -> 32); top is the last pattern below 256, so that 248.. stay in
//                              the top window (one fused add-and-minimum on 16-bit halves)
//     . & mask                 = b rounded to n significant bits; without the increment: trimmed
//     . + 1024                 = the integer back in the low byte of each half
// 11 instructions per four activations for any width, 16 with the pair rule at n = 4 (25 at n < 4,
// with its second, 2n-bit window).
//
// What the transform costs is the integer pipe: a logical operation, shift, permute or minimum takes it
// two cycles a warp, an integer add one and a half, half-precision arithmetic two of another pipe.
// The packed-integer form of n = 4 is 19 instructions, 17 of them logical or shifts: 32.2 cycles per
// word and scheduler with two warps on it; this form 22.9.  56x56x256 -> 64 at batch 64 20.9 -> 17.6
// us, 14x14x1024 -> 256 10.4 -> 9.5, the ResNet-50 pass 894 -> 841 us, one image 240 -> 229.
// (Tried: choosing by the partner with multiplications in the half-precision pipe, 26.4 cycles with two
// warps and 22.5 with four; zero masks per half, 25.0; halves of both kinds, 23.2 and 19.8.)
__device__ __forceinline__ uint32_t h2_sub(uint32_t a, uint32_t b)
{
    uint32_t d;
    asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}
__device__ __forceinline__ uint32_t h2_add(uint32_t a, uint32_t b)
{
    uint32_t d;
    asm("add.rn.f16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}

constexpr uint32_t kHalf1024 = 0x64006400u;

// Four bytes as normalized halves: bytes 0, 1 in lo, bytes 2, 3 in hi.
__device__ __forceinline__ void bytes_to_halves(uint32_t x, uint32_t &lo, uint32_t &hi)
{
    lo = h2_sub(prmt(x, 0x64646464u, 0x4140u), kHalf1024);
    hi = h2_sub(prmt(x, 0x64646464u, 0x4342u), kHalf1024);
}

// The window of four activations given as halves, back in bytes.
template <bool ADD>
__device__ __forceinline__ uint32_t window_of_halves(uint32_t lo, uint32_t hi, uint32_t add, uint32_t mask, uint32_t top)
{
    if (ADD) {
        lo = __viaddmin_u16x2(lo, add, top);
        hi = __viaddmin_u16x2(hi, add, top);
    }
    return prmt(h2_add(lo & mask, kHalf1024), h2_add(hi & mask, kHalf1024), 0x6420u);
}

// FIXED4: n = 4 with rounding RND, constants at compile time; otherwise n < 4, width and rounding as in d.
template <int MODE, bool FIXED4, bool RND>
__device__ __forceinline__ uint32_t xform_word_fullset(uint32_t x, const XformDev &d)
{
    if (MODE == SPARQ_MODE_NONE) return x;
    uint32_t lo, hi;
    bytes_to_halves(x, lo, hi);
    const uint32_t q = FIXED4 ? window_of_halves<RND>(lo, hi, 0x00400040u, 0xFF80FF80u, 0x5BFF5BFFu)
                              : window_of_halves<true>(lo, hi, d.f_add, d.f_mask, d.f_top);
    if (MODE == SPARQ_MODE_BSPARQ) return q;
    // vSPARQ: a byte whose partner is zero keeps the 2n-bit window (the whole byte for n = 4)
    uint32_t lone = x;
    if (!FIXED4) lone = window_of_halves<true>(lo, hi, d.l_add, d.l_mask, d.l_top);
    const uint32_t nz = ((x & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | x;   // bit 7 of each byte: byte != 0
    const uint32_t partner_nz = prmt(nz, nz, 0xAB89u);           // swap within pairs, replicate bit 7
    return (q & partner_nz) | (lone & ~partner_nz);
}

// The transform of a fused kernel instantiated for (MODE, XN, RND): XN = 4 is n = 4 with all
// five placements (half precision, constants at compile time), XN = 5 n = 4 with fewer (3opt, 2opt: the
// packed-integer form with the width fixed and the placement widening), XN = 8 any other full placement set
// (6opt, 7opt; either rounding, through the constants; RND unused), XN = 0 the general
// packed-integer form with run-time width and the placement widening (restricted sets of n < 4); XN = 3
// and 2 are that with the width fixed, in the standalone kernels only, which the integer pipe bounds
// there (the fused kernels would need two more instantiations of everything for rare sets).
template <int MODE, int XN, bool RND>
__device__ __forceinline__ uint32_t xform_fused(uint32_t x, const XformDev &d)
{
    if (XN == 8 || XN == 4) return xform_word_fullset<MODE, XN == 4, RND>(x, d);
    if (XN == 5) return xform_word<MODE, 4, RND, true>(x, d);
    if (XN == 3) return xform_word<MODE, 3, RND, true>(x, d);
    if (XN == 2) return xform_word<MODE, 2, RND, true>(x, d);
    return xform_word<MODE, 0, RND, true>(x, d);
}

// The two values that vSPARQ chooses between for each of four activations, whatever pairs they form: q,
// its own window, and l, what it keeps beside a zero (the whole byte for n = 4).  XN as above.
template <int XN, bool RND>
__device__ __forceinline__ void window_and_lone(uint32_t x, const XformDev &d, uint32_t &q, uint32_t &l)
{
    q = xform_fused<SPARQ_MODE_BSPARQ, XN, RND>(x, d);
    l = x;
    if (XN != 4 && XN != 5) {
        if (XN == 8) {
            uint32_t lo, hi;
            bytes_to_halves(x, lo, hi);
            l = window_of_halves<true>(lo, hi, d.l_add, d.l_mask, d.l_top);
        } else {
            l = apply_mask<RND>(x, drop_mask<0, false>(x, 2 * d.n, 0u), 2 * d.n);
        }
    }
}
#endif

}  // namespace sparq
