// Packed SPARQ stream: what the multiplier of Eq. 4 consumes instead of the 8-bit activation --
// two n-bit inputs per pair (a 2n-bit data field) and the pair's control state (both
// placements, or where a lone value sits; Sections 3.1 and 5.1).
//
//   data plane   per unit of 16 activations the 8 pairs' fields (in1 << n) | in2, pair j at bits
//                [j*2n, (j+1)*2n) of a little-endian integer of 2n bytes (n = 4: a byte a pair)
//   ctrl plane   per unit the 8 pair states, CB bits each, pair j at bits [j*CB, (j+1)*CB) of a
//                little-endian integer of CB bytes
//   state        both non-zero: id(shift1) * ns + id(shift2) with ns placements in the set and
//                id = rank of the shift in the set; a lone value (vSPARQ) owns the pair's
//                2n-bit window at shift s_l in 0 .. 8-2n and travels as that window's two n-bit
//                halves: ns*ns + s_l in the first slot, ns*ns + (9 - 2n) + s_l in the second
//
// Both kernels stream: a thread owns whole units (one 16-byte vector of activations <-> 2n data
// bytes + CB control bytes); planes whose share of a unit is not a power of two go through a
// warp-private staging area, so that global accesses are whole words.  What a value or a state
// means is looked up in tables replicated once per lane in shared memory (word (index, lane) at
// word address index * 32 + lane), so that a warp's 32 look-ups hit 32 different banks
// whatever the data.
//
// Bound: HBM by bytes (1 + n/8 + CB/16 an activation), instruction issue and look-ups close
// behind.  Decoding is one table word and one two-term dot product (dp2a) per pair, where a look-up
// per input took twice the table reads; the next chunk's loads are in flight while a chunk is
// worked on, which 64 registers and two blocks per SM (one table each) leave room for: three
// blocks at 40 registers without the prefetch measured 29 + 19 us.  51.4 M activations, encode +
// decode, back to back: n = 4 5opt 43.4 -> 33.7 us (5.5 TB/s, 0.84 of measured copy), n = 3 6opt
// 127.6 -> 37.7 us, n = 2 7opt 124 -> 33.3 us.
#include "sparq_common.cuh"

namespace sparq {

namespace {

constexpr int kThreads = 512;
constexpr int kUnits = 4;                        // units per thread per tile
constexpr int kEncWords = 512, kDecWords = 64;

// Encoder table.  The data field and the state of a pair are the SUM of one half-word per
// slot, half-word = data contribution | state contribution << 8.  Word index = x * 2 + z
// with x the slot's activation and z = 1 when the partner slot is zero (vSPARQ only):
//   low half, first slot    z = 0: window(x) << n | (id(x) * ns) << 8
//                           z = 1: lone(x) | (ns*ns + s_l) << 8
//   high half, second slot  z = 0: window(x) | id(x) << 8
//                           z = 1: lone(x) | (ns*ns + 9 - 2n + s_l) << 8, 0 for x = 0
// Decoder table.  The two activations of a pair as (first | second << 8) are a linear function
// of its two n-bit inputs, in1 * P + in2 * Q, with word[state] = Q | P << 16 (Eq. 4 with unit
// weights: each input shifted and routed to the slot the state names).
template <int WORDS>
struct Table {
    uint32_t w[WORDS];
};
using EncTable = Table<kEncWords>;
using DecTable = Table<kDecWords>;

__device__ __forceinline__ uint4 ld_stream16(const void *p)
{
    uint4 v;
    asm volatile("ld.global.cs.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}

__device__ __forceinline__ void st_stream16(void *p, uint4 v)
{
    asm volatile("st.global.cs.v4.u32 [%0], {%1,%2,%3,%4};"
                 :: "l"(p), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}

// One copy of the table per lane (all threads of the block call this).
template <int WORDS>
__device__ __forceinline__ void fill_table(uint32_t *s_tab, const Table<WORDS> &tab)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = warp; i < WORDS; i += kThreads / 32) s_tab[i * 32 + lane] = tab.w[i];
}

// BITS-bit field `st` into bits [POS, POS + BITS) of the 64-bit word (lo, hi)
template <int POS, int BITS>
__device__ __forceinline__ void put_field(uint32_t &lo, uint32_t &hi, uint32_t st)
{
    if constexpr (POS >= 32) {
        hi |= st << (POS - 32);
    } else {
        lo |= st << POS;
        if constexpr (POS + BITS > 32) hi |= st >> (32 - POS);
    }
}

// Bits [POS, ...) of (lo, hi) moved to bit 0; what lies above is the caller's to mask.
template <int POS>
__device__ __forceinline__ uint32_t from_bit(uint32_t lo, uint32_t hi)
{
    if constexpr (POS >= 32) return hi >> (POS - 32);
    else if constexpr (POS == 0) return lo;
    else return __funnelshift_r(lo, hi, POS);
}

// Two pairs (one 32-bit word of activations): their sums data | state << 8.
// lanes = (lane * 4) in every byte: the lane's offset inside a table word row.
template <int MODE>
__device__ __forceinline__ void pack_word(uint32_t x, uint32_t lanes, const uint8_t *s_tab, uint32_t &s0, uint32_t &s1)
{
    uint32_t low = lanes;                                                // byte: z << 7 | lane << 2
    if (MODE == SPARQ_MODE_VSPARQ) {
        const uint32_t nz = ((x & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | x;      // bit 7 of each byte: byte != 0
        low = (~prmt(nz, nz, 0xAB89u) & 0x80808080u) | lanes;            // bit 7: the partner is zero
    }
    // byte offsets of the four look-ups: activation << 8 | z << 7 | lane << 2
    const uint32_t o01 = prmt(x, low, 0x1504u), o23 = prmt(x, low, 0x3726u);
    auto half = [&](uint32_t off) { return (uint32_t)*reinterpret_cast<const uint16_t *>(s_tab + off); };
    s0 = half(o01 & 0xFFFFu) + half((o01 >> 16) + 2u);
    s1 = half(o23 & 0xFFFFu) + half((o23 >> 16) + 2u);
}

// low bytes of four words -> one word
__device__ __forceinline__ uint32_t bytes4(uint32_t a, uint32_t b, uint32_t c, uint32_t d)
{
    return prmt(prmt(a, b, 0x0040u), prmt(c, d, 0x0040u), 0x5410u);
}

// A warp owns chunks of kUnits * 32 consecutive units (unit (i, lane) of a chunk is
// chunk0 + i * 32 + lane, so its loads and stores are contiguous); the chunk's bytes in each
// plane are contiguous too, and go through a warp-private staging area, so the only block-wide
// barrier is the one after the table fill.
constexpr int kChunkUnits = kUnits * 32;

// A chunk's `bytes` bytes of a plane between its staging area and global memory, as words plus a
// byte tail (the plane's side is 16-byte aligned: a chunk starts at a multiple of 128 units).
// PER = bytes per unit.
template <int PER>
__device__ __forceinline__ void plane_out(uint8_t *dst, const uint8_t *s, uint32_t bytes, int lane)
{
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const uint32_t o = (uint32_t)(k * 32 + lane) * 4u;
        if (o + 4u <= bytes) __stcs(reinterpret_cast<uint32_t *>(dst + o), *reinterpret_cast<const uint32_t *>(s + o));
    }
    if ((uint32_t)lane < (bytes & 3u)) dst[(bytes & ~3u) + lane] = s[(bytes & ~3u) + lane];
}
template <int PER>
__device__ __forceinline__ void plane_load(uint32_t (&r)[PER], const uint8_t *src, uint32_t bytes, int lane)
{
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const uint32_t o = (uint32_t)(k * 32 + lane) * 4u;
        r[k] = o + 4u <= bytes ? __ldcs(reinterpret_cast<const uint32_t *>(src + o)) : 0u;
    }
}
template <int PER>
__device__ __forceinline__ void plane_stage(uint8_t *s, const uint32_t (&r)[PER], const uint8_t *src, uint32_t bytes, int lane)
{
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const uint32_t o = (uint32_t)(k * 32 + lane) * 4u;
        if (o + 4u <= bytes) *reinterpret_cast<uint32_t *>(s + o) = r[k];
    }
    if ((uint32_t)lane < (bytes & 3u)) s[(bytes & ~3u) + lane] = src[(bytes & ~3u) + lane];
}

// The PER (<= 6) bytes of unit `idx` of a staged chunk, as a 64-bit integer: they span at most two
// words, because idx * PER mod 4 plus PER never exceeds 8 for PER = 2 .. 6.
template <int PER>
__device__ __forceinline__ void staged_unit(const uint8_t *s, int idx, uint32_t &lo, uint32_t &hi)
{
    const uint32_t off = (uint32_t)(idx * PER), sh = (off & 3u) * 8u;
    const uint32_t *w = reinterpret_cast<const uint32_t *>(s + (off & ~3u));
    const uint32_t w0 = w[0], w1 = w[1];
    lo = __funnelshift_r(w0, w1, sh);
    hi = w1 >> sh;
}

// Bytes per warp of a staged plane (a word beyond the last unit may be read).
template <int PER>
__host__ __device__ constexpr int stage_bytes() { return (kChunkUnits * PER + 4 + 15) / 16 * 16; }
// The data plane is staged only for n = 3; 8 and 4 bytes a unit are whole words as they are.
template <int N>
__host__ __device__ constexpr int data_stage_bytes() { return N == 3 ? stage_bytes<6>() : 0; }

// Resident blocks per SM of both kernels: what 64 registers a thread allow.
constexpr int kCodecBlocks = 2;

template <int MODE, int N, int CB>
__global__ void __launch_bounds__(kThreads, kCodecBlocks)
pack_kernel(const uint8_t *__restrict__ in, uint8_t *__restrict__ data, uint8_t *__restrict__ ctrl,
            size_t units, const __grid_constant__ EncTable tab)
{
    extern __shared__ __align__(128) uint8_t smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint8_t *s_ctrl = smem + kEncWords * 128 + warp * (stage_bytes<CB>() + data_stage_bytes<N>());
    uint8_t *s_data = s_ctrl + stage_bytes<CB>();
    fill_table(reinterpret_cast<uint32_t *>(smem), tab);
    __syncthreads();
    dep_wait();
    dep_launch();
    const uint32_t lanes = (uint32_t)lane * 0x04040404u;
    const size_t n_chunks = (units + kChunkUnits - 1) / kChunkUnits;
    const size_t stride = (size_t)gridDim.x * (kThreads / 32);
    // the next chunk's loads are in flight while this one is encoded
    uint4 nxt[kUnits];
    auto fetch = [&](size_t ch) {
#pragma unroll
        for (int i = 0; i < kUnits; ++i) {
            const size_t u = ch * kChunkUnits + (size_t)(i * 32 + lane);
            nxt[i] = u < units ? ld_stream16(in + 16 * u) : make_uint4(0u, 0u, 0u, 0u);
        }
    };
    size_t ch = (size_t)blockIdx.x * (kThreads / 32) + warp;
    if (ch < n_chunks) fetch(ch);
    for (; ch < n_chunks; ch += stride) {
        const size_t chunk0 = ch * kChunkUnits;
        const size_t left = units - chunk0;
        const uint32_t cnt = (uint32_t)(left < (size_t)kChunkUnits ? left : (size_t)kChunkUnits);
        uint4 v[kUnits];
#pragma unroll
        for (int i = 0; i < kUnits; ++i) v[i] = nxt[i];
        if (ch + stride < n_chunks) fetch(ch + stride);
#pragma unroll
        for (int i = 0; i < kUnits; ++i) {
            if ((uint32_t)(i * 32 + lane) >= cnt) continue;
            const size_t u = chunk0 + (size_t)(i * 32 + lane);
            uint32_t s[8];
            pack_word<MODE>(v[i].x, lanes, smem, s[0], s[1]);
            pack_word<MODE>(v[i].y, lanes, smem, s[2], s[3]);
            pack_word<MODE>(v[i].z, lanes, smem, s[4], s[5]);
            pack_word<MODE>(v[i].w, lanes, smem, s[6], s[7]);
            if constexpr (N == 4) {
                __stcs(reinterpret_cast<uint2 *>(data) + u, make_uint2(bytes4(s[0], s[1], s[2], s[3]), bytes4(s[4], s[5], s[6], s[7])));
            } else {
                uint32_t lo = 0u, hi = 0u;
                put_field<0 * 2 * N, 2 * N>(lo, hi, s[0] & 0xFFu);
                put_field<1 * 2 * N, 2 * N>(lo, hi, s[1] & 0xFFu);
                put_field<2 * 2 * N, 2 * N>(lo, hi, s[2] & 0xFFu);
                put_field<3 * 2 * N, 2 * N>(lo, hi, s[3] & 0xFFu);
                put_field<4 * 2 * N, 2 * N>(lo, hi, s[4] & 0xFFu);
                put_field<5 * 2 * N, 2 * N>(lo, hi, s[5] & 0xFFu);
                put_field<6 * 2 * N, 2 * N>(lo, hi, s[6] & 0xFFu);
                put_field<7 * 2 * N, 2 * N>(lo, hi, s[7] & 0xFFu);
                if constexpr (N == 2) {
                    __stcs(reinterpret_cast<uint32_t *>(data) + u, lo);
                } else {
                    uint16_t *sd = reinterpret_cast<uint16_t *>(s_data + (i * 32 + lane) * 6);
                    sd[0] = (uint16_t)lo; sd[1] = (uint16_t)(lo >> 16); sd[2] = (uint16_t)hi;
                }
            }
            uint32_t lo = 0u, hi = 0u;
            put_field<0 * CB, CB>(lo, hi, s[0] >> 8);
            put_field<1 * CB, CB>(lo, hi, s[1] >> 8);
            put_field<2 * CB, CB>(lo, hi, s[2] >> 8);
            put_field<3 * CB, CB>(lo, hi, s[3] >> 8);
            put_field<4 * CB, CB>(lo, hi, s[4] >> 8);
            put_field<5 * CB, CB>(lo, hi, s[5] >> 8);
            put_field<6 * CB, CB>(lo, hi, s[6] >> 8);
            put_field<7 * CB, CB>(lo, hi, s[7] >> 8);
            uint8_t *sc = s_ctrl + (i * 32 + lane) * CB;
            if constexpr (CB % 2 == 0) {
#pragma unroll
                for (int k = 0; k < CB; k += 2) *reinterpret_cast<uint16_t *>(sc + k) = (uint16_t)((k < 4 ? lo : hi) >> (8 * (k & 3)));
            } else {
#pragma unroll
                for (int k = 0; k < CB; ++k) sc[k] = (uint8_t)((k < 4 ? lo : hi) >> (8 * (k & 3)));
            }
        }
        __syncwarp();
        plane_out<CB>(ctrl + chunk0 * CB, s_ctrl, cnt * CB, lane);
        if constexpr (N == 3) plane_out<6>(data + chunk0 * 6, s_data, cnt * 6u, lane);
        __syncwarp();
    }
}

// Pair J's two activations (first | second << 8) from its inputs' bytes: digits holds in2, in1 of
// two pairs (J even: bytes 0, 1; J odd: bytes 2, 3).
template <int J, int CB>
__device__ __forceinline__ uint32_t unpack_pair(uint32_t clo, uint32_t chi, uint32_t digits, uint32_t base, const uint8_t *s_tab)
{
    constexpr int p = J * CB;
    constexpr uint32_t mask = ((1u << CB) - 1u) << 7;
    uint32_t st;
    if constexpr (p < 7) st = clo << (7 - p);
    else st = from_bit<p - 7>(clo, chi);
    const uint32_t w = *reinterpret_cast<const uint32_t *>(s_tab + ((st & mask) | base));    // state << 7 | lane << 2
    return (J & 1) ? __dp2a_hi(w, digits, 0u) : __dp2a_lo(w, digits, 0u);
}

// The n-bit inputs of pairs 2K and 2K + 1 as bytes (in2, in1, in2, in1).
template <int N, int K>
__device__ __forceinline__ uint32_t digits_of(uint32_t dlo, uint32_t dhi)
{
    if constexpr (N == 4) {
        const uint32_t w = K < 2 ? dlo : dhi;
        return prmt(w & 0x0F0F0F0Fu, (w >> 4) & 0x0F0F0F0Fu, (K & 1) ? 0x7362u : 0x5140u);
    } else {
        constexpr uint32_t fm = (1u << (2 * N)) - 1u, nm = ((1u << N) - 1u) * 0x01010101u;
        const uint32_t t = from_bit<K * 4 * N>(dlo, dhi);
        const uint32_t u = (t & fm) | ((t << (16 - 2 * N)) & (fm << 16));    // one field per half
        return (u | (u << (8 - N))) & nm;                                     // one input per byte
    }
}

template <int N, int CB>
__global__ void __launch_bounds__(kThreads, kCodecBlocks)
unpack_kernel(const uint8_t *__restrict__ data, const uint8_t *__restrict__ ctrl, uint8_t *__restrict__ out,
              size_t units, const __grid_constant__ DecTable tab)
{
    extern __shared__ __align__(128) uint8_t smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint8_t *s_ctrl = smem + kDecWords * 128 + warp * (stage_bytes<CB>() + data_stage_bytes<N>());
    uint8_t *s_data = s_ctrl + stage_bytes<CB>();
    fill_table(reinterpret_cast<uint32_t *>(smem), tab);
    __syncthreads();
    dep_wait();
    dep_launch();
    const uint32_t base = (uint32_t)lane * 4u;
    const size_t n_chunks = (units + kChunkUnits - 1) / kChunkUnits;
    const size_t stride = (size_t)gridDim.x * (kThreads / 32);
    // the next chunk's loads are in flight while this one is decoded
    constexpr int kDataRegs = N == 3 ? 6 : N == 4 ? 2 * kUnits : kUnits;
    uint32_t cn[CB], dn[kDataRegs];
    auto count = [&](size_t ch) {
        const size_t left = units - ch * kChunkUnits;
        return (uint32_t)(left < (size_t)kChunkUnits ? left : (size_t)kChunkUnits);
    };
    auto fetch = [&](size_t ch) {
        const uint32_t cnt = count(ch);
        plane_load<CB>(cn, ctrl + ch * kChunkUnits * CB, cnt * CB, lane);
        if constexpr (N == 3) {
            plane_load<6>(dn, data + ch * kChunkUnits * 6, cnt * 6u, lane);
        } else {
#pragma unroll
            for (int i = 0; i < kUnits; ++i) {
                const size_t u = ch * kChunkUnits + (size_t)(i * 32 + lane);
                const bool ok = (uint32_t)(i * 32 + lane) < cnt;
                if constexpr (N == 4) {
                    const uint2 d = ok ? __ldcs(reinterpret_cast<const uint2 *>(data) + u) : make_uint2(0u, 0u);
                    dn[2 * i] = d.x; dn[2 * i + 1] = d.y;
                } else {
                    dn[i] = ok ? __ldcs(reinterpret_cast<const uint32_t *>(data) + u) : 0u;
                }
            }
        }
    };
    size_t ch = (size_t)blockIdx.x * (kThreads / 32) + warp;
    if (ch < n_chunks) fetch(ch);
    for (; ch < n_chunks; ch += stride) {
        const size_t chunk0 = ch * kChunkUnits;
        const uint32_t cnt = count(ch);
        uint32_t dlo[kUnits], dhi[kUnits];
        if constexpr (N == 3) {
            plane_stage<6>(s_data, dn, data + chunk0 * 6, cnt * 6u, lane);
        } else {
#pragma unroll
            for (int i = 0; i < kUnits; ++i) {
                dlo[i] = N == 4 ? dn[2 * i] : dn[i];
                dhi[i] = N == 4 ? dn[2 * i + 1] : 0u;
            }
        }
        plane_stage<CB>(s_ctrl, cn, ctrl + chunk0 * CB, cnt * CB, lane);
        if (ch + stride < n_chunks) fetch(ch + stride);
        __syncwarp();
#pragma unroll
        for (int i = 0; i < kUnits; ++i) {
            if ((uint32_t)(i * 32 + lane) >= cnt) continue;
            uint32_t clo, chi;
            staged_unit<CB>(s_ctrl, i * 32 + lane, clo, chi);
            if constexpr (N == 3) staged_unit<6>(s_data, i * 32 + lane, dlo[i], dhi[i]);
            const uint32_t g0 = digits_of<N, 0>(dlo[i], dhi[i]), g1 = digits_of<N, 1>(dlo[i], dhi[i]);
            const uint32_t g2 = digits_of<N, 2>(dlo[i], dhi[i]), g3 = digits_of<N, 3>(dlo[i], dhi[i]);
            const uint32_t p0 = unpack_pair<0, CB>(clo, chi, g0, base, smem), p1 = unpack_pair<1, CB>(clo, chi, g0, base, smem);
            const uint32_t p2 = unpack_pair<2, CB>(clo, chi, g1, base, smem), p3 = unpack_pair<3, CB>(clo, chi, g1, base, smem);
            const uint32_t p4 = unpack_pair<4, CB>(clo, chi, g2, base, smem), p5 = unpack_pair<5, CB>(clo, chi, g2, base, smem);
            const uint32_t p6 = unpack_pair<6, CB>(clo, chi, g3, base, smem), p7 = unpack_pair<7, CB>(clo, chi, g3, base, smem);
            st_stream16(out + 16 * (chunk0 + (size_t)(i * 32 + lane)),
                        make_uint4(prmt(p0, p1, 0x5410u), prmt(p2, p3, 0x5410u), prmt(p4, p5, 0x5410u), prmt(p6, p7, 0x5410u)));
        }
        __syncwarp();
    }
}

int set_size(uint32_t mask) { return __builtin_popcount(mask); }

// Placements of a lone value's 2n-bit window.
int lone_shifts(int n) { return 9 - 2 * n; }

int state_bits(const XformArgs &x)
{
    const int ns = set_size(x.mask);
    const int states = ns * ns + (x.mode == SPARQ_MODE_VSPARQ ? 2 * lone_shifts(x.n) : 0);
    int bits = 0;
    while ((1 << bits) < states) ++bits;
    return bits;
}

// Validates the parameters of the packed form: a SPARQ mode.
int check_pack_params(const sparq_params *p, XformArgs *x)
{
    int rc = validate_params(p, x);
    if (rc != SPARQ_OK) return rc;
    if (x->mode == SPARQ_MODE_NONE) return set_error(SPARQ_ERR_INVALID_ARG, "the packed form needs mode BSPARQ or VSPARQ");
    return SPARQ_OK;
}

int check_stream(const void *a, const void *b, const void *c, size_t rows, size_t row_len, size_t *units)
{
    if (!a || !b || !c) return set_error(SPARQ_ERR_INVALID_ARG, "a stream pointer is NULL");
    if (row_len % 16) return set_error(SPARQ_ERR_UNSUPPORTED, "row_len (%zu) must be a multiple of 16", row_len);
    if (rows > ((size_t)1 << 62) / row_len) return set_error(SPARQ_ERR_INVALID_ARG, "rows * row_len overflows");
    if ((((uintptr_t)a | (uintptr_t)b | (uintptr_t)c) & 15u) != 0)
        return set_error(SPARQ_ERR_UNSUPPORTED, "stream pointers must be 16-byte aligned");
    *units = rows * row_len / 16;
    return SPARQ_OK;
}

// Lowest shift allowed by `mask` at which a w-bit window holds q.
int placement_of(uint32_t q, int w, uint32_t mask)
{
    for (int s = 0;; ++s)
        if (((mask >> s) & 1u) && (q >> s) < (1u << w)) return s;
}

int rank_of(int s, uint32_t mask) { return __builtin_popcount(mask & ((1u << s) - 1u)); }

// The table of the calling thread's last parameters is kept: a network packs every layer with the
// same ones, and computing it takes the host longer than a launch.
const EncTable &encoder_table(const XformArgs &x)
{
    static thread_local EncTable tab;
    static thread_local XformArgs key = {-1, 0, 0, 0, 0u, 0u};
    if (x.mode == key.mode && x.n == key.n && x.rnd == key.rnd && x.mask == key.mask) return tab;
    key = x;
    const XformDev d{x.widen_c, x.widen_rounds, x.n};
    const int ns = set_size(x.mask), n = x.n, w2 = 2 * n, nl = lone_shifts(n);
    const uint32_t lone_mask = (1u << nl) - 1u;
    const bool pairs = x.mode == SPARQ_MODE_VSPARQ;
    for (uint32_t v = 0; v < 256; ++v) {
        // window of bSPARQ(v), and what is kept of v beside a zero, from the packed transform
        const uint32_t q = (x.rnd ? xform_word<SPARQ_MODE_BSPARQ, 0, true, true>(v, d)
                                  : xform_word<SPARQ_MODE_BSPARQ, 0, false, true>(v, d)) & 0xFFu;
        const uint32_t l = (x.rnd ? xform_word<SPARQ_MODE_VSPARQ, 0, true, true>(v, d)
                                  : xform_word<SPARQ_MODE_VSPARQ, 0, false, true>(v, d)) & 0xFFu;
        const int s = placement_of(q, n, x.mask), sl = placement_of(l, w2, lone_mask);
        const uint32_t id = (uint32_t)rank_of(s, x.mask), win = q >> s;
        const uint32_t first = (win << n) | ((id * ns) << 8), second = win | (id << 8);
        tab.w[2 * v] = first | (second << 16);
        const uint32_t field = l >> sl;
        const uint32_t first_z = field | ((uint32_t)(ns * ns + sl) << 8), second_z = v ? (field | ((uint32_t)(ns * ns + nl + sl) << 8)) : 0u;
        tab.w[2 * v + 1] = pairs ? (first_z | (second_z << 16)) : tab.w[2 * v];
    }
    return tab;
}

DecTable decoder_table(const XformArgs &x)
{
    DecTable tab;
    const int ns = set_size(x.mask), n = x.n, nl = lone_shifts(n);
    int shift_of[8], r = 0;
    for (int s = 0; s <= 8 - n; ++s)
        if ((x.mask >> s) & 1u) shift_of[r++] = s;
    for (int st = 0; st < kDecWords; ++st) {
        uint32_t p = 0, q = 0;                                    // states a valid stream never holds: 0
        if (st < ns * ns) {                                       // two windows
            p = 1u << shift_of[st / ns];
            q = 256u << shift_of[st % ns];
        } else if (x.mode == SPARQ_MODE_VSPARQ && st < ns * ns + 2 * nl) {
            const int t = st - ns * ns, sl = t % nl;              // lone value: its halves at s_l + n and s_l
            q = (t < nl ? 1u : 256u) << sl;
            p = q << n;
        }
        tab.w[st] = q | (p << 16);
    }
    return tab;
}

// Launch with the table's and the staging's shared memory (above the default limit for the
// encoder); as many blocks as stay resident, each of which fills its table once.
template <int WORDS, class Kernel, class... Args>
int launch_codec(Kernel kernel, const char *what, int stage_per_warp, int blocks_per_sm, size_t units, cudaStream_t st, Args... args)
{
    const int smem = WORDS * 128 + stage_per_warp * (kThreads / 32);
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return cuda_error(e, what);
    const size_t want = (units + kThreads * kUnits - 1) / (kThreads * kUnits), cap = (size_t)sms * blocks_per_sm;
    e = launch_overlapped(kernel, (int)(want < cap ? want : cap), kThreads, smem, st, args...);
    return e == cudaSuccess ? SPARQ_OK : cuda_error(e, what);
}

template <int MODE, int N, int CB>
int launch_pack(const uint8_t *in, uint8_t *data, uint8_t *ctrl, size_t units, const XformArgs &x, cudaStream_t st)
{
    return launch_codec<kEncWords>(pack_kernel<MODE, N, CB>, "pack_kernel launch", stage_bytes<CB>() + data_stage_bytes<N>(), kCodecBlocks, units, st,
                                   in, data, ctrl, units, encoder_table(x));
}

template <int N, int CB>
int launch_unpack(const uint8_t *data, const uint8_t *ctrl, uint8_t *out, size_t units, const XformArgs &x, cudaStream_t st)
{
    return launch_codec<kDecWords>(unpack_kernel<N, CB>, "unpack_kernel launch", stage_bytes<CB>() + data_stage_bytes<N>(), kCodecBlocks, units, st,
                                   data, ctrl, out, units, decoder_table(x));
}

// F<N, CB>::run(args...) for the stream's field and state widths (n = 4: 2 .. 5 state bits, n = 3
// and 2: 4 .. 6, narrower sets of theirs included).
#define SPARQ_CODEC_CASE(FN, N_, CB_, ...) case CB_: return FN<N_, CB_>(__VA_ARGS__)
#define SPARQ_CODEC_SWITCH(FN, n, cb, ...)                                              \
    do {                                                                                \
        if ((n) == 4) switch (cb) {                                                     \
            SPARQ_CODEC_CASE(FN, 4, 2, __VA_ARGS__); SPARQ_CODEC_CASE(FN, 4, 3, __VA_ARGS__); \
            SPARQ_CODEC_CASE(FN, 4, 4, __VA_ARGS__); SPARQ_CODEC_CASE(FN, 4, 5, __VA_ARGS__); \
        }                                                                               \
        if ((n) == 3) switch (cb) {                                                     \
            SPARQ_CODEC_CASE(FN, 3, 4, __VA_ARGS__); SPARQ_CODEC_CASE(FN, 3, 5, __VA_ARGS__); \
            SPARQ_CODEC_CASE(FN, 3, 6, __VA_ARGS__);                                    \
        }                                                                               \
        if ((n) == 2) switch (cb) {                                                     \
            SPARQ_CODEC_CASE(FN, 2, 4, __VA_ARGS__); SPARQ_CODEC_CASE(FN, 2, 5, __VA_ARGS__); \
            SPARQ_CODEC_CASE(FN, 2, 6, __VA_ARGS__);                                    \
        }                                                                               \
        return set_error(SPARQ_ERR_UNSUPPORTED, "no codec kernel for %d-bit windows with %d control bits", n, cb); \
    } while (0)

template <int N, int CB>
int launch_pack_v(const uint8_t *i, uint8_t *d, uint8_t *c, size_t u, const XformArgs &x, cudaStream_t s) { return launch_pack<SPARQ_MODE_VSPARQ, N, CB>(i, d, c, u, x, s); }
template <int N, int CB>
int launch_pack_b(const uint8_t *i, uint8_t *d, uint8_t *c, size_t u, const XformArgs &x, cudaStream_t s) { return launch_pack<SPARQ_MODE_BSPARQ, N, CB>(i, d, c, u, x, s); }

int pack_switch(const uint8_t *in, uint8_t *data, uint8_t *ctrl, size_t units, const XformArgs &x, cudaStream_t st)
{
    const int cb = state_bits(x);
    if (x.mode == SPARQ_MODE_VSPARQ) SPARQ_CODEC_SWITCH(launch_pack_v, x.n, cb, in, data, ctrl, units, x, st);
    SPARQ_CODEC_SWITCH(launch_pack_b, x.n, cb, in, data, ctrl, units, x, st);
}

int unpack_switch(const uint8_t *data, const uint8_t *ctrl, uint8_t *out, size_t units, const XformArgs &x, cudaStream_t st)
{
    SPARQ_CODEC_SWITCH(launch_unpack, x.n, state_bits(x), data, ctrl, out, units, x, st);
}

}  // namespace

}  // namespace sparq

using namespace sparq;

extern "C" int sparq_packed_ctrl_bits(const sparq_params *p)
{
    XformArgs x;
    const int rc = check_pack_params(p, &x);
    return rc != SPARQ_OK ? rc : state_bits(x);
}

extern "C" int sparq_pack(const uint8_t *in, size_t rows, size_t row_len, const sparq_params *p,
                          uint8_t *data, uint8_t *ctrl, void *stream)
{
    XformArgs x;
    int rc = check_pack_params(p, &x);
    if (rc != SPARQ_OK) return rc;
    if (rows == 0 || row_len == 0) return SPARQ_OK;
    size_t units = 0;
    if ((rc = check_stream(in, data, ctrl, rows, row_len, &units)) != SPARQ_OK) return rc;
    return pack_switch(in, data, ctrl, units, x, (cudaStream_t)stream);
}

extern "C" int sparq_unpack(const uint8_t *data, const uint8_t *ctrl, size_t rows, size_t row_len,
                            const sparq_params *p, uint8_t *out, void *stream)
{
    XformArgs x;
    int rc = check_pack_params(p, &x);
    if (rc != SPARQ_OK) return rc;
    if (rows == 0 || row_len == 0) return SPARQ_OK;
    size_t units = 0;
    if ((rc = check_stream(data, ctrl, out, rows, row_len, &units)) != SPARQ_OK) return rc;
    return unpack_switch(data, ctrl, out, units, x, (cudaStream_t)stream);
}
