// The streaming kernels of libmxq.  Common shape: every lane owns a "unit" of 32 bytes of the
// widest stream it touches (one 256-bit global access), a warp sweeps tiles of 32*U consecutive
// units, and every tile gets a warp of its own: many small CTAs that the hardware schedules as
// earlier ones retire, which keeps the loads of new CTAs overlapped with the arithmetic and stores
// of older ones (a persistent wave with a stride loop measured 10-20 % slower on these streams).
//
//   quantize / fake_quant : unit = 32 B of FP32/BF16 input (8 / 16 elements); a block of 32
//                           elements spans 4 / 2 adjacent lanes, whose maxima meet by xor-shuffles.
//   slice_scale           : unit = 32 element codes = one block per lane, no cross-lane traffic.
//   dequantize            : to 16-bit outputs a unit is 32 element codes (64 B out); to FP32 it is 32 B
//                           of output (8 elements), see dequantize_wide_kernel.
//
// Every kernel lets its successor start launching at once, asks L2 for its own input lines, and only
// then waits for its predecessor (see pdl_release / prefetch_tile / pdl_acquire in mxq_access.cuh).
//
// All of them are bound by HBM traffic, with the integer/logic pipe (64 lanes per clock per SM) as
// the second bound; the arithmetic below is shaped to stay under it: packed 16-bit maxima, MXINT rounding as
// packed FP16 multiply-adds (round-down FP32 adds for FP32 sources), codes packed by multiply-adds, signs
// by byte permutes, the sm_100a narrowing conversion instructions for MXFP.
#pragma once
#include <cstdint>
#include <tuple>
#include <type_traits>
#include <utility>
#include <cuda_runtime.h>

#include "mxq_access.cuh"
#include "mxq_codec.cuh"

namespace mxq {


template <int N, class Fn>
__device__ __forceinline__ void static_for(Fn&& fn)
{
    [&]<int... I>(std::integer_sequence<int, I...>) { (fn(std::integral_constant<int, I>{}), ...); }
    (std::make_integer_sequence<int, N>{});
}

// ------------------------------------------------------------------------------------------
// Where a block's scale byte goes
// ------------------------------------------------------------------------------------------
// The kernels that produce scale bytes write them through put_scale(), overloaded on the type of
// the destination: a plain pointer (byte of block i at scales[i], the library's stored form), or a
// TiledScales record, which places them in the 128-row x 4-column tiles a block-scaled tensor-core
// matrix multiply reads (the step that consumes W_t, Sec. 3.5): tile (r / 128, c / 4) is 512
// consecutive bytes and holds the byte of row r, block-column c at
// (r mod 32) * 16 + (r div 32 mod 4) * 4 + c mod 4.

__device__ __forceinline__ void put_scale(uint8_t* scales, size_t blk, uint32_t byte)
{
    st_u8(scales + blk, byte);
}

// Division of a 32-bit block index by the row length in blocks, by multiply and shift (the
// round-up method for an invariant divisor: with s = ceil(log2 d) and m = floor(2^32 (2^s - d) / d) + 1,
// n / d = (t + ((n - t) >> min(s, 1))) >> max(s - 1, 0) where t is the high word of m * n).  The host
// fills in m and the two shifts (see make_tiled_scales in mxq_launch.h).
struct TiledScales {
    uint8_t* base;
    uint32_t kblocks;      // block-columns per row (the divisor)
    uint32_t magic, shift1, shift2;
    uint32_t col_tiles;    // ceil(kblocks / 4)
    uint32_t rows;         // of the matrix (for the padding)
};

inline TiledScales make_tiled_scales(uint8_t* base, uint32_t kblocks, uint32_t rows = 0)      // 1 <= kblocks <= 2^31
{
    uint32_t s = 0;
    while ((1ull << s) < kblocks) ++s;
    const uint64_t m = ((1ull << 32) * ((1ull << s) - kblocks)) / kblocks + 1;
    return TiledScales{base, kblocks, (uint32_t)m, s < 1 ? s : 1u, s > 1 ? s - 1 : 0u, (kblocks + 3) / 4, rows};
}

// Byte offset of block `blk` (row-major index, below 2^32) inside the tiled buffer.
__host__ __device__ __forceinline__ size_t tiled_scale_offset(const TiledScales& t, size_t blk)
{
    const uint32_t n = (uint32_t)blk;
#ifdef __CUDA_ARCH__
    const uint32_t hi = __umulhi(t.magic, n);
#else
    const uint32_t hi = (uint32_t)(((uint64_t)t.magic * n) >> 32);
#endif
    const uint32_t r = (hi + ((n - hi) >> t.shift1)) >> t.shift2;
    const uint32_t c = n - r * t.kblocks;
    const size_t tile = (size_t)(r >> 7) * t.col_tiles + (c >> 2);
    return tile * 512 + (r & 31u) * 16u + ((r >> 5) & 3u) * 4u + (c & 3u);
}

__device__ __forceinline__ void put_scale(const TiledScales& t, size_t blk, uint32_t byte)
{
    st_u8(t.base + tiled_scale_offset(t, blk), byte);
}

// Tiles that the matrix covers only in part hold byte 0 where no block lands.  Those bytes are written by CTAs of
// their own behind the grid's last data CTA, kPadPerThread pieces per thread: the 4-byte pieces of the rows below
// the matrix, then the rest of the last piece of every row whose block-columns do not fill it.  (A memset of the
// whole buffer in front of the kernel cost a launch and, having no programmatic launch, the overlap with the
// kernel before it: a call on a 1000 x 4096 BF16 matrix, to E4M3, 13.0 us with it and 10.4 without, through the same binding.)
constexpr int kPadPerThread = 4;

__host__ __device__ __forceinline__ size_t tiled_pad_pieces(const TiledScales& t)
{
    const uint32_t below = (0u - t.rows) & 127u;
    return (size_t)below * t.col_tiles + ((t.kblocks & 3u) ? t.rows : 0u);
}

// CTAs of `threads` threads that the padding takes.
inline size_t tiled_pad_ctas(const TiledScales& t, int threads)
{
    const size_t per = (size_t)threads * kPadPerThread;
    return (tiled_pad_pieces(t) + per - 1) / per;
}

template <int THREADS>
__device__ __forceinline__ void fill_scale_padding(const TiledScales& t, size_t pad_cta)
{
    const uint32_t below = (0u - t.rows) & 127u;
    const size_t nbelow = (size_t)below * t.col_tiles, npieces = tiled_pad_pieces(t);
#pragma unroll
    for (int j = 0; j < kPadPerThread; ++j) {
        const size_t i = pad_cta * (THREADS * kPadPerThread) + j * THREADS + threadIdx.x;
        if (i >= npieces) return;
        const bool row_below = i < nbelow;
        const size_t r = row_below ? t.rows + i % below : i - nbelow;
        const size_t ct = row_below ? i / below : t.col_tiles - 1;
        uint8_t* piece = t.base + ((r >> 7) * t.col_tiles + ct) * 512 + (r & 31) * 16 + ((r >> 5) & 3) * 4;
        if (row_below) {
            st_u32(piece, 0);
        } else {
            for (uint32_t c = t.kblocks & 3u; c < 4; ++c) st_u8(piece + c, 0);
        }
    }
}

// For a kernel whose grid may end in such CTAs: true (and the padding written) if this is one of them.  `cta`
// counts from the matrix's first CTA, each of which covers `per_cta` lane units.
template <int THREADS, class SCALES>
__device__ __forceinline__ bool is_padding_cta(const SCALES& scales, size_t cta, size_t nunits, uint32_t per_cta)
{
    if constexpr (std::is_same_v<SCALES, TiledScales>) {
        if (cta * per_cta >= nunits) {
            pdl_acquire();
            fill_scale_padding<THREADS>(scales, cta - (nunits + per_cta - 1) / per_cta);
            return true;
        }
    }
    return false;
}

// ------------------------------------------------------------------------------------------
// Source element types
// ------------------------------------------------------------------------------------------

struct F32 {
    static constexpr int id = MXQ_F32;
    static constexpr int size = 4;
    static constexpr int epl = 8;     // elements per 32-byte lane unit
};
struct BF16 {
    static constexpr int id = MXQ_BF16;
    static constexpr int size = 2;
    static constexpr int epl = 16;
};

// Element i of a lane unit as FP32 (exact widening for BF16).
template <class T, int I>
__device__ __forceinline__ float unit_elem(const uint32_t (&w)[8])
{
    if constexpr (T::size == 4) return __uint_as_float(w[I]);
    else return __uint_as_float((I & 1) ? (w[I >> 1] & 0xFFFF0000u) : (w[I >> 1] << 16));
}

__device__ __forceinline__ float max3_abs_nan(float a, float b, float c)
{
    float d;
    asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(fabsf(a)), "f"(fabsf(b)), "f"(fabsf(c)));
    return d;
}

// FP32 bit pattern of max |element| over the lane unit, for BF16 its upper half; any NaN yields a NaN pattern, an
// infinity the infinity pattern (both >= 0x7F800000, both larger than every finite pattern).
template <class T>
__device__ __forceinline__ uint32_t unit_amax_bits(const uint32_t (&w)[8])
{
    if constexpr (T::size == 4) {
        float m0 = max3_abs_nan(__uint_as_float(w[0]), __uint_as_float(w[1]), __uint_as_float(w[2]));
        float m1 = max3_abs_nan(__uint_as_float(w[3]), __uint_as_float(w[4]), __uint_as_float(w[5]));
        float m2 = max3_abs_nan(__uint_as_float(w[6]), __uint_as_float(w[7]), m0);
        float m;
        asm("max.NaN.f32 %0, %1, %2;" : "=f"(m) : "f"(m1), "f"(m2));
        return __float_as_uint(m) & 0x7FFFFFFFu;
    } else {
        // BF16 magnitudes are ordered like their 15-bit patterns: packed 16-bit integer maxima.
        constexpr uint32_t kAbs = 0x7FFF7FFFu;
        uint32_t a = __vimax3_s16x2(w[0] & kAbs, w[1] & kAbs, w[2] & kAbs);
        uint32_t b = __vimax3_s16x2(w[3] & kAbs, w[4] & kAbs, w[5] & kAbs);
        uint32_t c = __vimax3_s16x2(w[6] & kAbs, w[7] & kAbs, a);
        const uint32_t m = __vmaxu2(b, c);
        return max(m, m << 16);                               // (the low half is not part of the result)
    }
}

template <int LPB>
__device__ __forceinline__ uint32_t group_max(uint32_t v)
{
#pragma unroll
    for (int o = 1; o < LPB; o <<= 1) v = max(v, __shfl_xor_sync(0xFFFFFFFFu, v, o));
    return v;
}

// ------------------------------------------------------------------------------------------
// MXINT rounding on the FP16 pipe
// ------------------------------------------------------------------------------------------
// FP16 subnormals are the integers 0 ... 1023 times 2^-24, their bit patterns those integers.  A fused multiply-add whose
// result lies there therefore rounds to an integer, two elements per instruction, on the FMA pipe; the
// integer/logic pipe, which bounds these kernels, is left for packing.

__device__ __forceinline__ uint32_t hfma2(uint32_t a, uint32_t b, uint32_t c)
{
    uint32_t d;
    asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}

__device__ __forceinline__ uint32_t hfma2_relu(uint32_t a, uint32_t b, uint32_t c)      // negative results become +0
{
    uint32_t d;
    asm("fma.rn.relu.f16x2 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}

__device__ __forceinline__ uint32_t mul_bf16x2(uint32_t a, uint32_t b)
{
    uint32_t d;
    asm("mul.rn.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}

__host__ __device__ constexpr uint32_t both_halves(uint32_t h) { return h | h << 16; }

// m * 2^e as an FP16 bit pattern; exact for integers m of up to 11 significant bits in FP16's range.
__host__ __device__ constexpr uint32_t half_bits(int m, int e)
{
    const uint32_t sign = m < 0 ? 0x8000u : 0u;
    uint32_t f = (uint32_t)(m < 0 ? -m : m);
    for (; f >= 2048u; f >>= 1) ++e;
    for (; f < 1024u && e > -24; f <<= 1) --e;
    for (; e < -24; f >>= 1) ++e;
    return sign | (f < 1024u ? f : (f - 1024u) | (uint32_t)(e + 25) << 10);
}

// The MXINT codes (Eq. 3, Eq. 4) of two values r, given as the FP16 pair p = r 2^-E with |r| <= 128, each XORed with
// M = 2^(B-1) - 1.  The first multiply-add rounds M + r (1 + 2^-10) to an integer; the factor turns ties away from zero and
// is too small to carry any other value of eight significant bits (|r| 2^-10 is below their spacing) over a halfway point.
// Negative sums (r below -M) become 0 = the symmetric clip; the second one is the same clip of the other side:
// 2M - (M + q) = M - q, and (M - q) ^ M is the two's complement of q in B bits.
//   MIN : the second clip as a packed integer minimum on the logic pipe instead (the first sum then takes -r, so that it is
//         M - q already).
template <int B, int E, bool MIN = false>
__device__ __forceinline__ uint32_t round_halves(uint32_t p)
{
    constexpr uint32_t M = (1u << (B - 1)) - 1u;
    constexpr uint32_t c = half_bits(1025, E - 34);                // 2^(E - 24) (1 + 2^-10)
    if constexpr (MIN) {
        const uint32_t r = hfma2_relu(p, both_halves(c | 0x8000u), both_halves(M));
        return __vminu2(r, both_halves(2 * M));
    } else {
        const uint32_t r = hfma2_relu(p, both_halves(c), both_halves(M));
        return hfma2_relu(r, both_halves(half_bits(-1, 0)), both_halves(2 * M));
    }
}

// Word number `word` of the bitstream that repeats one B-bit code.
template <int B>
__host__ __device__ constexpr uint32_t code_pattern(uint32_t code, int word)
{
    uint32_t v = 0;
    for (int i = 0; i < 32; ++i) v |= (code >> ((32 * word + i) % B) & 1u) << i;
    return v;
}

// XORs every B-bit code of the bitstream with M = 2^(B-1) - 1 (see round_halves).
template <int B, int NW>
__device__ __forceinline__ void unbias_codes(uint32_t (&out)[NW])
{
    static_for<NW>([&](auto j) {
        constexpr uint32_t pattern = code_pattern<B>((1u << (B - 1)) - 1u, decltype(j)::value);
        out[decltype(j)::value] ^= pattern;
    });
}

// Two 2B-bit fields in the low bits of the halves of y -> their 4B-bit stream in the top bits (the rest clear).
template <int B>
__device__ __forceinline__ uint32_t join_halves_top(uint32_t y)
{
    constexpr uint32_t k = 1u << (16 - 2 * B);
    return (y & 0xFFFFu) * (k * (k - 1u)) + y * k;
}

// Two W-bit fields in the low bits of the halves of y -> their 2W-bit stream in the low bits (the rest clear): one operation less
// than join_halves_top, on the logic pipe.
template <int W>
__device__ __forceinline__ uint32_t join_halves_low(uint32_t y)
{
    return (y >> 16) * ((1u << W) - (1u << 16)) + y;
}

// NZ streams of W bits, each in the low bits of its word (the rest clear) -> the little-endian bitstream: a multiply-add
// per stream and a shift where one crosses a word; three byte permutes join four streams of 24 bits.
template <int W, int NZ, int NW>
__device__ __forceinline__ void pack_low_streams(const uint32_t (&z)[NZ], uint32_t (&out)[NW])
{
    static_assert(NW * 32 >= NZ * W, "output too small");
    if constexpr (W == 24 && NZ % 4 == 0) {
#pragma unroll
        for (int g = 0; g < NZ / 4; ++g) {
            out[3 * g + 0] = __byte_perm(z[4 * g + 0], z[4 * g + 1], 0x4210);
            out[3 * g + 1] = __byte_perm(z[4 * g + 1], z[4 * g + 2], 0x5421);
            out[3 * g + 2] = __byte_perm(z[4 * g + 2], z[4 * g + 3], 0x6542);
        }
    } else {
        static_for<NZ>([&](auto j) {
            constexpr int J = decltype(j)::value;
            constexpr int off = J * W, wi = off >> 5, sh = off & 31;
            if constexpr (sh == 0) out[wi] = z[J];
            else out[wi] += z[J] * (1u << sh);
            if constexpr (sh + W > 32) out[wi + 1] = z[J] >> (32 - sh);
        });
    }
}

// ------------------------------------------------------------------------------------------
// Q_f: quantize (Eq. 1-3)
// ------------------------------------------------------------------------------------------

// Four B-bit codes, one per byte, -> their 4B-bit stream c0 | c1 << B | c2 << 2B | c3 << 3B in the TOP bits of
// the result (the bits below clear).  Every field only ever moves LEFT relative to c3, so the moves are
// multiply-adds (the multiply pipe) instead of shifts and selects on the logic pipe: with the codes in the
// top bits of their bytes, w + (2^(8-B) - 1) (w & 0x00FF00FF) moves bytes 0 and 2 up by 8 - B, which joins each
// byte pair into a 2B-bit field at the top of its half; y + (2^(16-2B) - 1) (y & 0xFFFF) joins the two fields.
template <int B>
__device__ __forceinline__ uint32_t squeeze_top(uint32_t w)            // codes in the top B bits, the rest clear
{
    constexpr int D = 8 - B;
    const uint32_t y = (w & 0x00FF00FFu) * ((1u << D) - 1u) + w;
    return (y & 0x0000FFFFu) * ((1u << (2 * D)) - 1u) + y;
}

template <int B>
__device__ __forceinline__ uint32_t squeeze_low(uint32_t w)            // codes in the low B bits, the rest clear
{
    constexpr int D = 8 - B;
    const uint32_t y = (w & 0x00FF00FFu) * (((1u << D) - 1u) << D) + w * (1u << D);
    return (y & 0x0000FFFFu) * ((1u << (2 * D)) - 1u) + y;
}

// NZ streams of four B-bit codes, each in the top 4B bits of its word (the rest clear) -> the little-endian
// bitstream.  Pieces that move left are multiply-adds, pieces that move right shift-adds; for 6 bits the
// pieces are whole bytes and three byte permutes join four streams.
template <int B, int NZ, int NW>
__device__ __forceinline__ void pack_streams(const uint32_t (&z)[NZ], uint32_t (&out)[NW])
{
    constexpr int W = 4 * B;                                             // bits per stream
    static_assert(NW * 32 >= NZ * W, "output too small");
    if constexpr (B == 6 && NZ % 4 == 0) {
#pragma unroll
        for (int g = 0; g < NZ / 4; ++g) {
            out[3 * g + 0] = __byte_perm(z[4 * g + 0], z[4 * g + 1], 0x5321);
            out[3 * g + 1] = __byte_perm(z[4 * g + 1], z[4 * g + 2], 0x6532);
            out[3 * g + 2] = __byte_perm(z[4 * g + 2], z[4 * g + 3], 0x7653);
        }
    } else {
        static_for<NZ>([&](auto j) {
            constexpr int J = decltype(j)::value;
            constexpr int off = J * W, wi = off >> 5, sh = off & 31;
            // the field has to go from bit 32 - W to bit sh
            uint32_t v;
            if constexpr (sh <= 32 - W) v = z[J] >> (32 - W - sh);
            else v = z[J] * (1u << (sh - (32 - W)));
            if constexpr (sh == 0) out[wi] = v;
            else out[wi] += v;
            if constexpr (sh + W > 32) out[wi + 1] = z[J] >> (64 - W - sh);
        });
    }
}

// Codes of a BF16 lane unit in an MXINT format, inv = 2^-shared_exp, two elements per instruction: r = v inv, exact in BF16
// wherever it does not round to 0 anyway; r 2^-122, whose BF16 exponent field fits FP16's five bits, so that the
// pattern moved up by three bits under its sign is the FP16 number r 2^-10 (what is lost below BF16's smallest normal is below
// r = 2^-4).
template <class F, int NW>
__device__ __forceinline__ void quantize_unit_bf16_int(const uint32_t (&w)[8], float inv, uint32_t (&out)[NW])
{
    constexpr int B = F::bits;
    const uint32_t inv2 = __byte_perm(__float_as_uint(inv), 0, 0x3232);
    constexpr uint32_t k122 = both_halves((127u - 122u) << 7);
    uint32_t z[4];
    static_for<4>([&](auto qi) {
        constexpr int Q = decltype(qi)::value;
        uint32_t r[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const uint32_t x = mul_bf16x2(mul_bf16x2(w[2 * Q + i], inv2), k122);
            r[i] = round_halves<B, 10>(((x & 0x7FFF7FFFu) * 8u) | (x & 0x80008000u));
        }
        if constexpr (B == 8) {
            z[Q] = __byte_perm(r[0], r[1], 0x6420);
        } else {
            // c0 | c1 << B of each pair lands in the upper half
            constexpr uint32_t j = 0x10000u + (1u << B);
            const uint32_t y = __byte_perm(r[0] * j, r[1] * j, 0x7632);
            if constexpr (B == 4) z[Q] = y;
            else z[Q] = join_halves_top<B>(y);
        }
    });
    if constexpr (B == 8) {
#pragma unroll
        for (int i = 0; i < 4; ++i) out[i] = z[i];
    } else if constexpr (B == 4) {
        out[0] = __byte_perm(z[0], z[1], 0x6420);
        out[1] = __byte_perm(z[2], z[3], 0x6420);
    } else {
        pack_streams<B>(z, out);
    }
    unbias_codes<B>(out);
}

// MXINT codes of four consecutive elements (Eq. 3), one per byte in the low F::bits bits.
//   v0..v3 : the raw elements, inv = 2^-shared_exp (|v| inv < 2^(bits-1), exact)
//   full   : 0xFF in the bytes whose element is negative, 0x00 elsewhere
// One round-down FFMA per element adds 2^15 + 0.5, where the FP32 spacing is 2^-8: byte 1 of the
// sum is floor(|r| + 0.5), the magnitude rounded to nearest with ties away from zero.  Three byte
// permutes gather the four magnitudes; clip and sign are then applied to all four at once.
template <class F>
__device__ __forceinline__ uint32_t quantize_int_quad(float v0, float v1, float v2, float v3, float inv, uint32_t full)
{
    constexpr float kMagic = 32768.5f;
    constexpr uint32_t k01 = 0x01010101u;
    constexpr uint32_t kInv255 = 0xFEFEFEFFu;                  // 255^-1 mod 2^32: mask -> 0/1 per byte
    constexpr uint32_t kMask = k01 * F::mask;
    const uint32_t y0 = __float_as_uint(__fmaf_rd(fabsf(v0), inv, kMagic));
    const uint32_t y1 = __float_as_uint(__fmaf_rd(fabsf(v1), inv, kMagic));
    const uint32_t y2 = __float_as_uint(__fmaf_rd(fabsf(v2), inv, kMagic));
    const uint32_t y3 = __float_as_uint(__fmaf_rd(fabsf(v3), inv, kMagic));
    uint32_t q = __byte_perm(__byte_perm(y0, y1, 0x0051), __byte_perm(y2, y3, 0x0051), 0x5410);
    q -= (q >> (F::bits - 1)) & k01;                           // 2^(b-1) -> 2^(b-1) - 1 (symmetric clip)
    if constexpr (F::bits == 8) {
        // negate in 7 bits, then set the sign bit: no carry leaves a byte even for a negative zero
        const uint32_t z = (q ^ (full & 0x7F7F7F7Fu)) + full * kInv255;
        return z ^ (full & 0x80808080u);
    } else {
        return ((q ^ (full & kMask)) + full * kInv255) & kMask;
    }
}

// 0xFF / 0x00 per byte: the signs of elements 4Q .. 4Q+3 of an FP32 lane unit, straight from the raw words.
template <int Q>
__device__ __forceinline__ uint32_t unit_sign_bytes(const uint32_t (&w)[8])
{
    uint32_t a, b;
    asm("prmt.b32 %0, %1, %2, 0x00FB;" : "=r"(a) : "r"(w[4 * Q]), "r"(w[4 * Q + 1]));
    asm("prmt.b32 %0, %1, %2, 0x00FB;" : "=r"(b) : "r"(w[4 * Q + 2]), "r"(w[4 * Q + 3]));
    return __byte_perm(a, b, 0x5410);
}

// Codes of one lane unit, packed as a little-endian bitstream.
template <class T, class F, int NW>
__device__ __forceinline__ void quantize_unit(const uint32_t (&w)[8], float inv, uint32_t (&out)[NW])
{
    if constexpr (F::kind == KIND_INT) {
        static_assert(T::size == 4, "BF16 -> MXINT: quantize_unit_bf16_int");
        constexpr int NQ = T::epl / 4;
        uint32_t z[NQ];
        static_for<NQ>([&](auto qi) {
            constexpr int Q = decltype(qi)::value;
            z[Q] = quantize_int_quad<F>(unit_elem<T, 4 * Q>(w), unit_elem<T, 4 * Q + 1>(w), unit_elem<T, 4 * Q + 2>(w),
                                        unit_elem<T, 4 * Q + 3>(w), inv, unit_sign_bytes<Q>(w));
        });
        if constexpr (F::bits == 8) {
#pragma unroll
            for (int j = 0; j < NQ; ++j) out[j] = z[j];
        } else if constexpr (F::bits == 4) {
            // c0 | c1 << 4 lands in byte 0 and c2 | c3 << 4 in byte 2 of z | z >> 4
#pragma unroll
            for (int j = 0; j < NQ / 2; ++j)
                out[j] = __byte_perm(z[2 * j] | (z[2 * j] >> 4), z[2 * j + 1] | (z[2 * j + 1] >> 4), 0x6420);
        } else {
#pragma unroll
            for (int j = 0; j < NQ; ++j) z[j] = squeeze_low<F::bits>(z[j]);
            pack_streams<F::bits>(z, out);
        }
    } else if constexpr (F::bits == 4) {
        // two codes to the byte
        static_for<T::epl / 2>([&](auto i) {
            constexpr int I = decltype(i)::value;
            put_code<8, I>(out, quantize_fp_hw_pair<F>(unit_elem<T, 2 * I>(w) * inv, unit_elem<T, 2 * I + 1>(w) * inv));
        });
    } else {
        // four elements at a time, squeezed as one word; E3M3 / E2M2 through the hardware neighbour format.  (BF16, 2^25 elements,
        // against a shift and an OR per code: E2M3 16.1 -> 14.4 us, E3M2 15.7 -> 14.3; E3M3 17.7 -> 17.2, E2M2 17.2 -> 16.8.  E2M1,
        // two codes to a byte already, took 13.9 -> 14.5 with eight elements to a word and stays with pairs.)
        constexpr int NQ = T::epl / 4;
        uint32_t z[NQ];
        float k = inv;
        if constexpr (!F::hw_cvt) k *= SoftFp<F>::pre_scale;     // exact: both are powers of two
        static_for<NQ>([&](auto qi) {
            constexpr int Q = decltype(qi)::value;
            const float r0 = unit_elem<T, 4 * Q>(w) * k, r1 = unit_elem<T, 4 * Q + 1>(w) * k;
            const float r2 = unit_elem<T, 4 * Q + 2>(w) * k, r3 = unit_elem<T, 4 * Q + 3>(w) * k;
            if constexpr (!F::hw_cvt) z[Q] = squeeze_top<F::bits>(quantize_fp_soft_quad_top<F>(r0, r1, r2, r3));
            else if constexpr (F::bits == 8) z[Q] = quantize_fp_hw_quad<F>(r0, r1, r2, r3);
            else z[Q] = squeeze_low<F::bits>(quantize_fp_hw_quad<F>(r0, r1, r2, r3));
        });
        if constexpr (F::bits == 8) {
#pragma unroll
            for (int j = 0; j < NQ; ++j) out[j] = z[j];
        } else {
            pack_streams<F::bits>(z, out);
        }
    }
}

// One warp tile (32 U lane units) of one tensor; shared by the single-tensor and the batched kernels.
// Every lane of the warp must call it (the block maxima meet by shuffles).
template <class T, class F, int BLOCK, int U, class SCALES>
__device__ __forceinline__ void quantize_tile(const uint8_t* __restrict__ src, size_t nunits, uint8_t* __restrict__ codes,
                                              const SCALES& scales, size_t tile, uint8_t* stage)
{
    constexpr int LPB = BLOCK / T::epl;                 // lanes per block
    static_assert(LPB >= 1 && LPB <= 32, "block must cover at least one lane unit");
    constexpr int OB = T::epl * F::bits / 8;            // code bytes per lane unit
    constexpr int NW = code_words(T::epl, F::bits);
    const int lane = threadIdx.x & 31;
    const size_t u0 = tile * (32 * U) + lane;
    uint32_t w[U][8];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const size_t unit = u0 + u * 32;
        if (unit < nunits) ld256(w[u], src + unit * 32);
        else {
#pragma unroll
            for (int j = 0; j < 8; ++j) w[u][j] = 0;
        }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const size_t unit = u0 + u * 32;
        const uint32_t amax = group_max<LPB>(unit_amax_bits<T>(w[u]));
        const BlockScale s = block_scale<F>(amax);
        uint32_t out[NW];
        if constexpr (T::size == 2 && F::kind == KIND_INT) quantize_unit_bf16_int<F>(w[u], s.inv, out);
        else quantize_unit<T, F>(w[u], s.inv, out);
        if (s.byte == 0xFFu) {
#pragma unroll
            for (int j = 0; j < NW; ++j) out[j] = 0;
        }
        if constexpr (StagedTile<OB>::use) store_bytes<OB>(stage + (u * 32 + lane) * OB, out);
        if (unit < nunits) {
            if constexpr (!StagedTile<OB>::use) store_bytes<OB>(codes + unit * OB, out);
            if (lane % LPB == 0) put_scale(scales, unit / LPB, s.byte);
        }
    }
    if constexpr (StagedTile<OB>::use) {
        const size_t first = tile * (32 * U), left = nunits - first;
        flush_stage<32 * U * OB>(stage, codes + first * OB, (uint32_t)(left < 32 * U ? left : 32 * U) * OB);
    }
}

// The staging area of the calling warp for a quantize tile (null when a lane's code piece is stored
// directly).  Must be called by every thread of the CTA, outside divergent code.
template <class T, class F, int U, int THREADS>
__device__ __forceinline__ uint8_t* quantize_stage()
{
    constexpr int OB = T::epl * F::bits / 8;
    if constexpr (StagedTile<OB>::use) {
        __shared__ __align__(128) uint8_t stage_area[(THREADS / 32) * 32 * U * OB];
        return stage_area + (threadIdx.x >> 5) * (32 * U * OB);
    } else {
        return nullptr;
    }
}

// Resident CTAs (of 128 threads) per SM the quantizer is compiled for: 16, i.e. 32 registers (against the compiler's own choice, 2^25 elements
// and more, BF16 -> MXINT7 and MXINT3 and FP32 -> MXINT7 3 - 4 % faster, MXINT5, 4 and 2 1 %, E3M3 4 %, E2M2 6 %, MXINT8 and MXINT6 1 %
// slower, E4M3 4 %, E2M1 3 %), but 12 from FP32 to tiled E4M3, which in 32 registers loads one lane unit after the other (2^23.5
// elements 10.7 us against 9.2, 2^25 25.6 and 24.6; the other tiled formats lose up to 5 % with 12 in the largest launches).
template <class T, class F, class SCALES>
__host__ __device__ constexpr int quantize_min_ctas()
{
    return !std::is_same_v<SCALES, uint8_t*> && T::size == 4 && F::bits == 8 ? 12 : 16;
}

template <class T, class F, int BLOCK, int U, int THREADS, class SCALES = uint8_t*>
__global__ void __launch_bounds__(THREADS, quantize_min_ctas<T, F, SCALES>() * 128 / THREADS)
quantize_kernel(const uint8_t* __restrict__ src, size_t nunits, uint8_t* __restrict__ codes, SCALES scales)
{
    pdl_release();
    const size_t tile = (size_t)blockIdx.x * (THREADS / 32) + (threadIdx.x >> 5);
    uint8_t* stage = quantize_stage<T, F, U, THREADS>();
    if (is_padding_cta<THREADS>(scales, blockIdx.x, nunits, THREADS * U)) return;
    prefetch_tile<U, 32>(src, tile, nunits);
    pdl_acquire();
    if (tile * (32 * U) < nunits) quantize_tile<T, F, BLOCK, U>(src, nunits, codes, scales, tile, stage);
}

// ------------------------------------------------------------------------------------------
// Fused fake-quant forward (Eq. 6 in reconstructed form)
// ------------------------------------------------------------------------------------------

__device__ __forceinline__ float fma_keep_plus_zero(float a, float b)
{
    // a * b + (+0): turns a -0 product into +0 and changes nothing else
    float d;
    asm("fma.rn.f32 %0, %1, %2, 0f00000000;" : "=f"(d) : "f"(a), "f"(b));
    return d;
}

// two FP32 values out of a packed narrow-float pair produced by quantize_fp_hw_pair
template <class F>
__device__ __forceinline__ float2 widen_hw_pair(uint32_t d)
{
    uint32_t h2;
    if constexpr (F::id == MXQ_FP8_E4M3) asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(h2) : "h"((uint16_t)d));
    else if constexpr (F::id == MXQ_FP6_E3M2) asm("cvt.rn.f16x2.e3m2x2 %0, %1;" : "=r"(h2) : "h"((uint16_t)d));
    else if constexpr (F::id == MXQ_FP6_E2M3) asm("cvt.rn.f16x2.e2m3x2 %0, %1;" : "=r"(h2) : "h"((uint16_t)d));
    else asm("{ .reg .b8 t; cvt.u8.u32 t, %1; cvt.rn.f16x2.e2m1x2 %0, t; }" : "=r"(h2) : "r"(d));
    float2 f;
    asm("{ .reg .b16 l, h; mov.b32 {l, h}, %2; cvt.f32.f16 %0, l; cvt.f32.f16 %1, h; }"
        : "=f"(f.x), "=f"(f.y) : "r"(h2));
    return f;
}

// Two inputs of an MXFP fake-quant divided by the target's X, in FP32 (exact).  E3M3 / E2M2: divided by a further 2^k,
// which makes them values of their hardware neighbour format (see SoftFp).
template <class F, int MODE>
__device__ __forceinline__ void fake_quant_scaled(float v0, float v1, float inv, float& r0, float& r1)
{
    using A = Fmt<MXQ_FP8_E4M3>;
    constexpr bool via = MODE == MXQ_FQ_VIA_ANCHOR && F::id != A::id;
    constexpr int de = A::emax - F::emax;
    constexpr int k = [] { if constexpr (F::hw_cvt) return 0; else return SoftFp<F>::k; }();
    if constexpr (via) {
        // anchor codes -> exact FP16 values -> divide by 2^(de + k) (exact) -> FP32
        uint32_t a = quantize_fp_hw_pair<A>(v0 * inv, v1 * inv);
        uint32_t h2;
        asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(h2) : "h"((uint16_t)a));
        constexpr uint32_t kHalf = (uint32_t)(15 - de - k) << 10;          // 2^-(de + k) as FP16
        asm("mul.rn.f16x2 %0, %0, %1;" : "+r"(h2) : "r"(kHalf | (kHalf << 16)));
        asm("{ .reg .b16 l, h; mov.b32 {l, h}, %2; cvt.f32.f16 %0, l; cvt.f32.f16 %1, h; }"
            : "=f"(r0), "=f"(r1) : "r"(h2));
    } else {
        const float inv_k = inv * __uint_as_float((uint32_t)(127 - k) << 23);  // exact: powers of two
        r0 = v0 * inv_k;
        r1 = v1 * inv_k;
    }
}

// Element-format value (the real number P) of two inputs after quantization, as FP32.
//   DIRECT     : P = quantize_F(v inv)                       (inv = 2^-shared_exp of F)
//   VIA_ANCHOR : P = Q_{A->F}(quantize_A(v inv))             (inv = 2^-shared_exp of the anchor A)
template <class F, int MODE>
__device__ __forceinline__ float2 fake_quant_pair(float v0, float v1, float inv)
{
    using A = Fmt<F::kind == KIND_INT ? MXQ_INT8 : MXQ_FP8_E4M3>;
    constexpr bool via = MODE == MXQ_FQ_VIA_ANCHOR && F::id != A::id;
    constexpr int de = A::emax - F::emax;
    float2 p;
    if constexpr (F::kind == KIND_INT) {
        // floor(x + 0.5) for 0 <= x < 2^22 on the FP32 pipes alone: a round-down add of 2^22 + 0.5 lands
        // on the 0.5 grid of [2^22, 2^23), a round-down add of another 2^22 on the integer grid of
        // [2^23, 2^24).  The value stays biased by 2^23 until the clip.
        auto one = [&](float v) {
            float y = __fmaf_rd(fabsf(v), inv, 4194304.5f);                            // 2^22 + h, h = |r| + 0.5 on the 0.5 grid
            if constexpr (via) {
                // Eq. 4 on the anchor magnitude q8 = floor(h): floor(q8 / 2^de + 0.5) = floor(h / 2^de + 0.5),
                // since flooring before a division by an integer changes nothing.  So the anchor's integer
                // step is skipped: one more round-down multiply-add onto the 0.5 grid.
                // (Clipping q8 to 127 first would change nothing either: 127 and 128 both end in the clipped bin.)
                constexpr float kScale = 1.0f / (float)(1 << de);
                constexpr float kBias = 4194304.5f - 4194304.0f / (float)(1 << de);    // exact in FP32
                y = __fmaf_rd(y, kScale, kBias);
            }
            float z = __fadd_rd(y, 4194304.0f);                                        // 2^23 + floor(.)
            z = fminf(z, 8388608.0f + (float)F::max_mag);                              // symmetric clip
            const float qf = z - 8388608.0f;                                           // exact small integer
            return __uint_as_float(__float_as_uint(qf) | (__float_as_uint(v) & 0x80000000u));
        };
        p.x = one(v0);
        p.y = one(v1);
    } else {
        float r0, r1;
        fake_quant_scaled<F, MODE>(v0, v1, inv, r0, r1);
        p = widen_hw_pair<F>(quantize_fp_hw_pair<F>(r0, r1));
    }
    return p;
}

// The same of four inputs, for the two formats without a narrowing instruction: the clip works on four codes at a time
// (BF16, 2^25 elements, against two at a time: E3M3 direct 21.0 -> 19.9 us, through the anchor 22.9 -> 21.2; E2M2 21.3 -> 20.0, 22.8 -> 21.1).
template <class F, int MODE>
__device__ __forceinline__ void fake_quant_soft_quad(float v0, float v1, float v2, float v3, float inv, float (&p)[4])
{
    using H = Fmt<SoftFp<F>::hw>;
    float r0, r1, r2, r3;
    fake_quant_scaled<F, MODE>(v0, v1, inv, r0, r1);
    fake_quant_scaled<F, MODE>(v2, v3, inv, r2, r3);
    const uint32_t c = quantize_fp_soft_quad<F>(r0, r1, r2, r3);
    const float2 a = widen_hw_pair<H>(c & 0xFFFFu), b = widen_hw_pair<H>(c >> 16);
    p[0] = a.x * SoftFp<F>::post_scale;
    p[1] = a.y * SoftFp<F>::post_scale;
    p[2] = b.x * SoftFp<F>::post_scale;
    p[3] = b.y * SoftFp<F>::post_scale;
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi)
{
    uint32_t d;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
    return d;
}

// One warp tile (32 U lane units) of one tensor; shared by the single-tensor and the batched kernels.
// Every lane of the warp must call it (the block maxima meet by shuffles).
template <class T, class F, int BLOCK, int MODE, int U>
__device__ __forceinline__ void fake_quant_tile(const uint8_t* src, size_t nunits, uint8_t* dst, size_t tile)
{
    using A = Fmt<F::kind == KIND_INT ? MXQ_INT8 : MXQ_FP8_E4M3>;
    constexpr bool via = MODE == MXQ_FQ_VIA_ANCHOR && F::id != A::id;
    using S = std::conditional_t<via, A, F>;            // the format whose scale Eq. 1 computes
    constexpr int de = A::emax - F::emax;
    constexpr int LPB = BLOCK / T::epl;
    static_assert(LPB >= 1 && LPB <= 32, "block must cover at least one lane unit");
    const size_t u0 = tile * (32 * U) + (threadIdx.x & 31);
    uint32_t w[U][8];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const size_t unit = u0 + u * 32;
        if (unit < nunits) ld256(w[u], src + unit * 32);
        else {
#pragma unroll
            for (int j = 0; j < 8; ++j) w[u][j] = 0;
        }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const size_t unit = u0 + u * 32;
        const uint32_t amax = group_max<LPB>(unit_amax_bits<T>(w[u]));
        const BlockScale s = block_scale<S>(amax);
        // X of the target format: the anchor's byte moved up by de, saturating (Eq. 4-5)
        const uint32_t byte = via ? min(s.byte + (uint32_t)de, 254u) : s.byte;
        const float X = scale_value(byte);
        uint32_t out[8];
        if constexpr (F::kind == KIND_FP && !F::hw_cvt) {
            static_for<T::epl / 4>([&](auto i) {
                constexpr int I = 4 * decltype(i)::value;
                float p[4];
                fake_quant_soft_quad<F, MODE>(unit_elem<T, I>(w[u]), unit_elem<T, I + 1>(w[u]), unit_elem<T, I + 2>(w[u]),
                                              unit_elem<T, I + 3>(w[u]), s.inv, p);
                if constexpr (T::size == 4) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) out[I + j] = __float_as_uint(p[j] * X);
                } else {
                    out[I / 2] = pack_bf16x2(p[0] * X, p[1] * X);
                    out[I / 2 + 1] = pack_bf16x2(p[2] * X, p[3] * X);
                }
            });
        } else {
            static_for<T::epl / 2>([&](auto i) {
                constexpr int I = decltype(i)::value;
                const float v0 = unit_elem<T, 2 * I>(w[u]), v1 = unit_elem<T, 2 * I + 1>(w[u]);
                float2 p = fake_quant_pair<F, MODE>(v0, v1, s.inv);
                float y0, y1;
                if constexpr (F::kind == KIND_INT) {          // MXINT zero reconstructs to +0
                    y0 = fma_keep_plus_zero(p.x, X);
                    y1 = fma_keep_plus_zero(p.y, X);
                } else {
                    y0 = p.x * X;
                    y1 = p.y * X;
                }
                if constexpr (T::size == 4) {
                    out[2 * I] = __float_as_uint(y0);
                    out[2 * I + 1] = __float_as_uint(y1);
                } else {
                    out[I] = pack_bf16x2(y0, y1);
                }
            });
        }
        if (unit < nunits) {
            if (s.byte == 0xFFu) st256_splat(dst + unit * 32, T::size == 4 ? 0x7FC00000u : 0x7FC07FC0u);   // poisoned block
            else st256(dst + unit * 32, out);
        }
    }
}

template <class T, class F, int BLOCK, int MODE, int U, int THREADS>
__global__ void __launch_bounds__(THREADS, 2048 / THREADS)
fake_quant_kernel(const uint8_t* src, size_t nunits, uint8_t* dst)   // dst may equal src
{
    pdl_release();
    const size_t tile = (size_t)blockIdx.x * (THREADS / 32) + (threadIdx.x >> 5);
    prefetch_tile<U, 32>(src, tile, nunits);
    pdl_acquire();
    if (tile * (32 * U) < nunits) fake_quant_tile<T, F, BLOCK, MODE, U>(src, nunits, dst, tile);
}

// Which tensor of a batch owns a tile.  The batched kernels lay the tiles of all tensors end to end;
// the items (sorted by tile_begin) ride in the kernel parameters.  A plain binary search over a few
// hundred items costs eight dependent constant-memory reads.  The host therefore adds a coarse index: the
// tile space is cut into at most 256 segments of 2^shift tiles, coarse[k] is the item that owns the first
// tile of segment k (coarse[last + 1] the last item), and a tile's owner lies between the entries of its
// segment's two ends -- usually the same item or neighbours, so the search that remains takes zero
// to two steps.
struct TileIndex {
    uint32_t shift;
    uint16_t coarse[258];
};

template <class ITEM>
inline void build_tile_index(TileIndex& ix, const ITEM* items, int count, size_t total_tiles)
{
    ix.shift = 0;
    while ((total_tiles >> ix.shift) > 255) ++ix.shift;
    const size_t nseg = total_tiles ? ((total_tiles - 1) >> ix.shift) + 1 : 1;
    int it = 0;
    for (size_t k = 0; k < nseg; ++k) {
        const size_t first = k << ix.shift;
        while (it + 1 < count && items[it + 1].tile_begin <= first) ++it;
        ix.coarse[k] = (uint16_t)it;
    }
    for (size_t k = nseg; k < 258; ++k) ix.coarse[k] = (uint16_t)(count - 1);
}

// `items` is an array inside a __grid_constant__ kernel parameter; tile < total_tiles.
template <class ITEM>
__host__ __device__ __forceinline__ int find_item(const ITEM* items, const TileIndex& ix, size_t tile)
{
    const uint32_t k = (uint32_t)(tile >> ix.shift);
    int lo = ix.coarse[k], hi = ix.coarse[k + 1];
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (items[mid].tile_begin <= tile) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// A tile of the batched kernels is what one CTA converts, THREADS / 32 consecutive warp tiles of ONE tensor: the owner
// is found once per CTA from the block index, by uniform instructions, and the tensor's pointers live in uniform
// registers.  (With a lookup per warp tile they took two registers each in every lane: MXINT8 -> MXINT4 over four
// decoder layers 219 -> 208 us, BF16 -> MXINT8 over eight 840 -> 804 us with one lookup per CTA.)  The calling warp's
// tile in the tensor that starts at CTA tile `tile_begin`:
template <int THREADS>
__device__ __forceinline__ size_t item_warp_tile(size_t tile_begin)
{
    return (blockIdx.x - tile_begin) * (THREADS / 32) + (threadIdx.x >> 5);
}

// The fake-quant of a whole set of tensors (every quantized weight of a model in one QAT step, Eq. 6)
// in one launch: the tiles of all tensors laid end to end, the item table in the kernel's parameters.
struct FqDeviceItem {
    const uint8_t* src;
    uint8_t* dst;
    size_t nunits;
    size_t tile_begin;     // first global tile index of this tensor
};

template <int K>
struct FqItemBlock {
    FqDeviceItem items[K];
    TileIndex index;
};

template <class T, class F, int BLOCK, int MODE, int U, int R, int THREADS, int K>
__global__ void __launch_bounds__(THREADS, 14)
fake_quant_batched_kernel(const __grid_constant__ FqItemBlock<K> blk)
{
    pdl_release();
    // the item table is a kernel parameter, so the lookup may run before the dependency wait
    const FqDeviceItem& t = blk.items[find_item(blk.items, blk.index, blockIdx.x)];
    // a warp converts R consecutive warp tiles of the tensor, one after the other
    const size_t first = item_warp_tile<THREADS>(t.tile_begin) * R;
#pragma unroll
    for (int r = 0; r < R; ++r) prefetch_tile<U, 32>(t.src, first + r, t.nunits);
    pdl_acquire();
#pragma unroll 1
    for (int r = 0; r < R; ++r)
        if ((first + r) * (32 * U) < t.nunits) fake_quant_tile<T, F, BLOCK, MODE, U>(t.src, t.nunits, t.dst, first + r);
}

// Q_f (Eq. 1-3) over a whole set of tensors in one launch (the anchor checkpoint of a model, Sec. 3.5:
// every linear weight quantized once and stored): tiles of all tensors end to end, items in the parameters.
struct QDeviceItem {
    const uint8_t* src;
    uint8_t* codes;
    uint8_t* scales;
    size_t nunits;
    size_t tile_begin;
};

template <int K>
struct QItemBlock {
    QDeviceItem items[K];
    TileIndex index;
};

// Resident CTAs (of 128 threads) per SM: 14 (against the compiler's own choice BF16 -> MXINT7 and MXINT5 of 2^25 elements and more take
// 3 % less, the other formats the same to 1 %), but 12 from BF16 to E3M3 and E2M2, whose four-code clip wants more registers in small
// sets (2^16 elements 2.09 us with 14, 2.0 with 12; 2^22.5 5.06 and 4.5, 2^25 17.2 and 16.7, 2^28 131 either way).
template <class T, class F>
__host__ __device__ constexpr int quantize_batched_min_ctas()
{
    return T::size == 2 && F::kind == KIND_FP && !F::hw_cvt ? 12 : 14;
}

template <class T, class F, int BLOCK, int U, int THREADS, int K>
__global__ void __launch_bounds__(THREADS, quantize_batched_min_ctas<T, F>())
quantize_batched_kernel(const __grid_constant__ QItemBlock<K> blk)
{
    pdl_release();
    uint8_t* stage = quantize_stage<T, F, U, THREADS>();
    // the item table is a kernel parameter, so the lookup may run before the dependency wait
    const QDeviceItem& t = blk.items[find_item(blk.items, blk.index, blockIdx.x)];
    const size_t tile = item_warp_tile<THREADS>(t.tile_begin);
    prefetch_tile<U, 32>(t.src, tile, t.nunits);
    pdl_acquire();
    if (tile * (32 * U) < t.nunits)                       // whole warps
        quantize_tile<T, F, BLOCK, U>(t.src, t.nunits, t.codes, t.scales, tile, stage);
}

// ------------------------------------------------------------------------------------------
// Q_{h->l}: Slice-and-Scale (Eq. 4-5).  One lane = 32 codes.
// ------------------------------------------------------------------------------------------

// Four consecutive codes, number J, of a little-endian bitstream of B-bit codes (B < 8), in 16-bit lanes: c0 | c1 << B in the
// lower half, c2 | c3 << B in the upper one; the bits above 2B of the upper half are undefined.
template <int B, int J, int NW>
__device__ __forceinline__ uint32_t code_quad_lanes(const uint32_t (&in)[NW])
{
    constexpr int off = 4 * B * J, wi = off >> 5, sh = off & 31;
    if constexpr (B == 4) {
        return __byte_perm(in[wi], 0, sh == 0 ? 0x4140 : 0x4342);
    } else {
        uint32_t f;
        if constexpr (sh == 0) f = in[wi];
        else if constexpr (sh + 4 * B <= 32) f = in[wi] >> sh;
        else f = __funnelshift_r(in[wi], in[wi + 1], sh);
        constexpr uint32_t k = 1u << (16 - 2 * B);
        return f * k - (f & ((1u << (2 * B)) - 1u)) * (k - 1u);
    }
}

// Four MXINT codes, number J of the lane's 32, as FP16 pairs, the codes 0 and 2 in .a, 1 and 3 in .b: the value of code p
// is p 2^(8-b_h) 2^-17, the same for every source width, so that de = b_h - b_l becomes 8 - b_l below.  The
// biased code u = p + 2^(b_h - 1) under the exponent of 1024 is the FP16 number 1024 + u; one multiply-add takes the bias off.
struct IntHalves {
    uint32_t a, b;
};

template <class FH, int J, int NW>
__device__ __forceinline__ IntHalves int_halves(const uint32_t (&in)[NW])
{
    constexpr int B = FH::bits;
    constexpr uint32_t one = both_halves(half_bits(1, -9 - B));
    constexpr uint32_t bias = both_halves(half_bits(-(1024 + (1 << (B - 1))), -9 - B));
    IntHalves h;
    if constexpr (B == 8) {
        const uint32_t u = in[J] ^ 0x80808080u;
        h.a = hfma2(__byte_perm(u, 0x64646464u, 0x4240), one, bias);
        h.b = hfma2(__byte_perm(u, 0x64646464u, 0x4341), one, bias);
    } else {
        constexpr uint32_t m = both_halves(FH::mask), k = both_halves(0x6400u + (1u << (B - 1)));
        const uint32_t y = code_quad_lanes<B, J>(in);
        h.a = hfma2((y & m) ^ k, one, bias);
        h.b = hfma2(((y >> B) & m) ^ k, one, bias);
    }
    return h;
}

__device__ __forceinline__ bool has_e4m3_nan(uint32_t x)
{
    return (((x & 0x7F7F7F7Fu) + 0x01010101u) & 0x80808080u) != 0;
}

// Eq. 5 on E4M3 codes through the conversion instructions: exact widening to FP16, exact division
// by 2^de, FP32, narrowing cvt (nearest even, saturating).  Register halves and bytes are split and
// joined with mov so that no shift or mask is spent on them.

// four E4M3 codes of one word as two FP16 pairs (exact).  Kept apart from the scaling so that two
// targets converted from the same word share it.
__device__ __forceinline__ void e4m3_word_to_f16(uint32_t w, uint32_t& a, uint32_t& b)
{
    asm("{ .reg .b16 l, h; mov.b32 {l, h}, %2; cvt.rn.f16x2.e4m3x2 %0, l; cvt.rn.f16x2.e4m3x2 %1, h; }"
        : "=r"(a), "=r"(b) : "r"(w));
}

// Four codes, number J of the lane's 32, of an MXFP format below eight bits as two FP16 pairs: one code per byte,
// then the widening conversion.  E3M3 and E2M2 have none; with the sign bit one position up their codes are codes of E4M3 and E3M2
// (same mantissa, see SoftFp) that stand for 2^-fp_source_shift() times the value.
template <class FH>
__host__ __device__ constexpr int fp_source_shift()
{
    return FH::id == MXQ_FP7_E3M3 ? 4 : FH::id == MXQ_FP5_E2M2 ? 2 : 0;
}

template <class FH, int J, int NW>
__device__ __forceinline__ void fp_quad_to_f16(const uint32_t (&in)[NW], uint32_t& a, uint32_t& b)
{
    constexpr int B = FH::bits;
    static_assert(FH::kind == KIND_FP && B < 8 && B > 4);
    const uint32_t y = code_quad_lanes<B, J>(in);
    uint32_t w = (y & both_halves(FH::mask << B)) * (1u << (8 - B)) + (y & both_halves(FH::mask));
    if constexpr (!FH::hw_cvt) w += w & (0x01010101u << (B - 1));
    if constexpr (FH::id == MXQ_FP7_E3M3)
        e4m3_word_to_f16(w, a, b);
    else if constexpr (FH::id == MXQ_FP6_E2M3)
        asm("{ .reg .b16 l, h; mov.b32 {l, h}, %2; cvt.rn.f16x2.e2m3x2 %0, l; cvt.rn.f16x2.e2m3x2 %1, h; }"
            : "=r"(a), "=r"(b) : "r"(w));
    else
        asm("{ .reg .b16 l, h; mov.b32 {l, h}, %2; cvt.rn.f16x2.e3m2x2 %0, l; cvt.rn.f16x2.e3m2x2 %1, h; }"
            : "=r"(a), "=r"(b) : "r"(w));
}

// two FP16 pairs (four MXFP codes), divided by 2^DE, as four FP32 values
template <int DE>
__device__ __forceinline__ void fp_pairs_scaled(uint32_t a, uint32_t b, float (&f)[4])
{
    constexpr uint32_t kHalf = (uint32_t)(15 - DE) << 10;      // 2^-de as FP16
    asm("{ .reg .b16 l, h; .reg .b32 a, b;\n"
        "  mul.rn.f16x2 a, %4, %6;  mul.rn.f16x2 b, %5, %6;\n"
        "  mov.b32 {l, h}, a;  cvt.f32.f16 %0, l;  cvt.f32.f16 %1, h;\n"
        "  mov.b32 {l, h}, b;  cvt.f32.f16 %2, l;  cvt.f32.f16 %3, h; }"
        : "=f"(f[0]), "=f"(f[1]), "=f"(f[2]), "=f"(f[3]) : "r"(a), "r"(b), "r"(kHalf | (kHalf << 16)));
}

// Four MXFP codes, given as two FP16 pairs, in a 5-, 6- or 7-bit MXFP format, the codes in the top bits of their
// bytes.  `nans` has 0x7F in the bytes whose anchor code was a NaN code (see e4m3_word_clean).
//   E2M3, E3M2: divided by 2^de (exact in FP16), widened to FP32, narrowing conversion.
//   E3M3      : no narrowing instruction, but it is E4M3 with fewer binades (see SoftFp): the same through the
//               conversion to E4M3 of the value divided by a further 2^4.
//   E2M2      : the same through E5M2 (bias 15, a further 2^14), whose conversion takes the FP16 pair itself, without
//               the trip through FP32 (the E4M3 conversion of FP16 pairs is slower than that trip).  The FP16 product
//               is exact where it matters: it loses bits only below the smallest halfway point 2^-17, where every
//               value rounds to zero either way (anchor codes have four significant bits).
// From E4M3 nothing is clipped: its largest value 448 / 2^de (7, 28, 28, 7) does not exceed the target's largest (7.5, 28, 30, 7;
// E2M3, E3M2, E3M3, E2M2).  From the narrower sources E3M3 -> E3M2 (30 against 28) relies on the conversion's saturation, and E2M2 as a
// target on a clip of its own (7.5 against 7).
template <class FH, class FL>
__device__ __forceinline__ uint32_t ss_fp_pairs_top(uint32_t a, uint32_t b, uint32_t nans)
{
    constexpr int de = FH::emax - FL::emax - fp_source_shift<FH>(), D = 8 - FL::bits;
    constexpr uint32_t k01 = 0x01010101u;
    constexpr uint32_t kMag = k01 * FL::max_mag;
    uint32_t c;
    if constexpr (FL::id == MXQ_FP5_E2M2 && FH::id != MXQ_FP8_E4M3) {
        // E3M3 and E2M3 go up to 7.5 2^de, which rounds beyond the target's largest: the quantizer's conversion clips it
        float f[4];
        fp_pairs_scaled<de + SoftFp<FL>::k>(a, b, f);
        return quantize_fp_soft_quad_top<FL>(f[0], f[1], f[2], f[3]);
    } else if constexpr (FL::id == MXQ_FP5_E2M2) {
        constexpr uint32_t kHalf = 1u << (24 - (de + 14));           // 2^-20 as an FP16 subnormal
        asm("{ .reg .b16 l, h; .reg .b32 a, b; mul.rn.f16x2 a, %1, %3; mul.rn.f16x2 b, %2, %3;\n"
            "  cvt.rn.satfinite.e5m2x2.f16x2 l, a; cvt.rn.satfinite.e5m2x2.f16x2 h, b; mov.b32 %0, {l, h}; }"
            : "=r"(c) : "r"(a), "r"(b), "r"(kHalf | (kHalf << 16)));
        return ((c & kMag) << D) | (c & 0x80808080u);
    } else {
        constexpr int k = FL::id == MXQ_FP7_E3M3 ? 4 : 0;
        float f[4];
        fp_pairs_scaled<de + k>(a, b, f);
        if constexpr (FL::id == MXQ_FP7_E3M3)
            asm("{ .reg .b16 l, h; cvt.rn.satfinite.e4m3x2.f32 l, %2, %1; cvt.rn.satfinite.e4m3x2.f32 h, %4, %3; mov.b32 %0, {l, h}; }"
                : "=r"(c) : "f"(f[0]), "f"(f[1]), "f"(f[2]), "f"(f[3]));
        else if constexpr (FL::id == MXQ_FP6_E2M3)
            asm("{ .reg .b16 l, h; cvt.rn.satfinite.e2m3x2.f32 l, %2, %1; cvt.rn.satfinite.e2m3x2.f32 h, %4, %3; mov.b32 %0, {l, h}; }"
                : "=r"(c) : "f"(f[0]), "f"(f[1]), "f"(f[2]), "f"(f[3]));
        else
            asm("{ .reg .b16 l, h; cvt.rn.satfinite.e3m2x2.f32 l, %2, %1; cvt.rn.satfinite.e3m2x2.f32 h, %4, %3; mov.b32 %0, {l, h}; }"
                : "=r"(c) : "f"(f[0]), "f"(f[1]), "f"(f[2]), "f"(f[3]));
        if constexpr (FL::mu == 3) c |= nans & kMag;
        if constexpr (FL::id == MXQ_FP7_E3M3) return ((c & kMag) << D) | (c & 0x80808080u);
        else return c << D;
    }
}

// eight MXFP codes (given as their four FP16 pairs) -> eight E2M1 codes in one word; values up to 7 or 7.5 saturate at 6
template <class FH>
__device__ __forceinline__ uint32_t ss_fp_pairs_to_e2m1(uint32_t a0, uint32_t b0, uint32_t a1, uint32_t b1)
{
    constexpr int de = FH::emax - 2 - fp_source_shift<FH>();
    float f[4], g[4];
    fp_pairs_scaled<de>(a0, b0, f);
    fp_pairs_scaled<de>(a1, b1, g);
    uint32_t d;
    asm("{ .reg .b8 a, b, c, e;\n"
        "  cvt.rn.satfinite.e2m1x2.f32 a, %2, %1;  cvt.rn.satfinite.e2m1x2.f32 b, %4, %3;\n"
        "  cvt.rn.satfinite.e2m1x2.f32 c, %6, %5;  cvt.rn.satfinite.e2m1x2.f32 e, %8, %7;\n"
        "  mov.b32 %0, {a, b, c, e}; }"
        : "=r"(d) : "f"(f[0]), "f"(f[1]), "f"(f[2]), "f"(f[3]), "f"(g[0]), "f"(g[1]), "f"(g[2]), "f"(g[3]));
    return d;
}

// From E4M3 to every target, one element at a time (exact, slow): for units with NaN codes.
template <class FH, class FL, int NWI, int NWO>
__device__ __forceinline__ void ss_unit_by_element(const uint32_t (&in)[NWI], uint32_t (&out)[NWO])
{
#pragma unroll
    for (int j = 0; j < NWO; ++j) out[j] = 0;
    static_for<32>([&](auto i) {
        constexpr int I = decltype(i)::value;
        const uint32_t c = get_code<FH::bits, I>(in);
        put_code<FL::bits, I>(out, ss_fp_elem<FH, FL>(c));
    });
}

__device__ __forceinline__ bool unit_has_e4m3_nan(const uint32_t (&in)[8])
{
    bool nan = false;
#pragma unroll
    for (int j = 0; j < 8; ++j) nan |= has_e4m3_nan(in[j]);
    return nan;
}

// A word of four E4M3 codes with every NaN code (0x7F) replaced by the largest finite one (0x7E, the sign
// kept); `nans` gets 0x7F in the bytes that held one.
__device__ __forceinline__ uint32_t e4m3_word_clean(uint32_t x, uint32_t& nans)
{
    const uint32_t m = ((x & 0x7F7F7F7Fu) + 0x01010101u) & 0x80808080u;
    nans = m - (m >> 7);
    return x - (m >> 7);
}

// Eight codes (the quads 2J and 2J + 1 of a lane's 32) in a lower format: two streams for pack_streams, or,
// for the 4-bit formats, one finished output word.  MXINT codes stay XORed with M until ss_finish.
template <class FL, int J, bool MIN, bool LOW>
__device__ __forceinline__ void ss_int_quad_pair(const IntHalves& w0, const IntHalves& w1, uint32_t (&z)[8])
{
    constexpr int B = FL::bits, E = 9 + B;                     // r = p 2^(8-b_h) / 2^(8-B)
    const uint32_t y0 = round_halves<B, E, MIN>(w0.b) * (1u << B) + round_halves<B, E, MIN>(w0.a);
    const uint32_t y1 = round_halves<B, E, MIN>(w1.b) * (1u << B) + round_halves<B, E, MIN>(w1.a);
    if constexpr (B == 4) {
        z[J] = __byte_perm(y0, y1, 0x6420);
    } else {
        z[2 * J] = LOW ? join_halves_low<2 * B>(y0) : join_halves_top<B>(y0);
        z[2 * J + 1] = LOW ? join_halves_low<2 * B>(y1) : join_halves_top<B>(y1);
    }
}

template <class FH, class FL, int J>
__device__ __forceinline__ void ss_fp_quad_pair(const uint32_t (&h)[4], const uint32_t (&nans)[2], uint32_t (&z)[8])
{
    if constexpr (FL::bits == 4) {
        z[J] = ss_fp_pairs_to_e2m1<FH>(h[0], h[1], h[2], h[3]);
    } else {
        z[2 * J] = squeeze_top<FL::bits>(ss_fp_pairs_top<FH, FL>(h[0], h[1], nans[0]));
        z[2 * J + 1] = squeeze_top<FL::bits>(ss_fp_pairs_top<FH, FL>(h[2], h[3], nans[1]));
    }
}

template <class FL, bool LOW = false, int NWO>
__device__ __forceinline__ void ss_finish(const uint32_t (&z)[8], uint32_t (&out)[NWO])
{
    if constexpr (FL::bits == 4) {
#pragma unroll
        for (int j = 0; j < 4; ++j) out[j] = z[j];
    } else if constexpr (LOW) {
        pack_low_streams<4 * FL::bits>(z, out);
    } else {
        pack_streams<FL::bits>(z, out);
    }
    if constexpr (FL::kind == KIND_INT) unbias_codes<FL::bits>(out);
}

template <int I, class... FL>
using ss_target_t = typename std::tuple_element<I, std::tuple<FL...>>::type;

// Which clip of round_halves: the packed minimum from MXINT8, where the FMA pipe has become the fuller one (2^26 codes, multiply-add
// against minimum: -> 6 + 4 bits 27.6 and 25.3 us, 7 + 5 31.3 and 29.7, 6 + 4 + 2 32.7 and 30.9, -> 2 15.8 and 15.0, -> 7 20.5 and
// 20.1); the multiply-add from narrower sources, whose unpacking is logic (MXINT6 -> MXINT4 14.3 and 16.2, MXINT4 -> MXINT2 12.4 and
// 13.7), and to 5 bits, where the minimum costs registers (-> 5 19.3 and 21.5; 5 + 4 over four layers 299 and, spilling, 385).
template <class FH, class FL>
__host__ __device__ constexpr bool ss_min_clip()
{
    return FH::bits == 8 && FL::bits != 5;
}

// Streams joined in the low bits instead of the top ones: in a set whose targets all have more than five bits, which is 7 + 6 (2^24 codes 8.6 us
// against 9.9, 2^22 4.0 and 4.7, 2^25.8 24.8 and 25.4).  With a narrower target the top form is the faster one or the
// difference is small: 7 + 4 bits 9.2 and 7.8, 6 + 4 8.6 and 7.4, 7 + 5 8.9 and 8.8.
template <class FH, class... FL>
__host__ __device__ constexpr bool ss_low_join()
{
    return FH::id == MXQ_INT8 && sizeof...(FL) > 1 && ((FL::bits > 5) && ...);
}

// The 32 codes of one lane to one or more lower formats, eight codes at a time so that what
// the targets share (the FP16 values, and which codes are NaN) lives only that long.  E4M3 anchors:
// NAN_CODES = false promises that none of the codes is a NaN code.  A NaN code maps to the largest magnitude with
// its sign: so does the largest finite code, 448, wherever the target's largest mantissa is 1.75 or less
// (448 / 2^de = 1.75 * 2^emax); for the three-bit mantissas (largest 1.875) the magnitude bits of the target
// code are set as well.
template <bool NAN_CODES, class FH, class... FL, int NW>
__device__ __forceinline__ void ss_unit(const uint32_t (&in)[NW], uint32_t (&z)[sizeof...(FL)][8])
{
    static_for<4>([&](auto jj) {
        constexpr int J = decltype(jj)::value;
        if constexpr (FH::kind == KIND_INT) {
            const IntHalves w0 = int_halves<FH, 2 * J>(in), w1 = int_halves<FH, 2 * J + 1>(in);
            static_for<(int)sizeof...(FL)>([&](auto i) {
                constexpr int I = decltype(i)::value;
                using F = ss_target_t<I, FL...>;
                ss_int_quad_pair<F, J, ss_min_clip<FH, F>(), ss_low_join<FH, FL...>()>(w0, w1, z[I]);
            });
        } else {
            uint32_t h[4], nans[2] = {0, 0};
            if constexpr (FH::bits == 8) {
                e4m3_word_to_f16(NAN_CODES ? e4m3_word_clean(in[2 * J], nans[0]) : in[2 * J], h[0], h[1]);
                e4m3_word_to_f16(NAN_CODES ? e4m3_word_clean(in[2 * J + 1], nans[1]) : in[2 * J + 1], h[2], h[3]);
            } else {
                fp_quad_to_f16<FH, 2 * J>(in, h[0], h[1]);
                fp_quad_to_f16<FH, 2 * J + 1>(in, h[2], h[3]);
            }
            static_for<(int)sizeof...(FL)>([&](auto i) {
                constexpr int I = decltype(i)::value;
                ss_fp_quad_pair<FH, ss_target_t<I, FL...>, J>(h, nans, z[I]);
            });
        }
    });
}

// The 32 MXINT8 codes of one lane to ONE lower format, with fewer instructions than the general form above takes for a
// single target: the codes come as sign-extended 16-bit pairs (one byte permute per pair, no exclusive OR), one packed
// add-with-maximum brings them under the exponent of 1024 and clips the negative side at -M, and the rounding's relu clips the other
// one.  For 3 and 2 bits the pairs hold codes four apart, so that eight codes join inside the halves.  Instructions per
// lane unit against the general form: -> 7 bits 186 and 197, 6 175 and 185, 4 127 and 131, 3 141 and 166, 2 130 and 155.  Where it is
// used and where not: see the kernels.
template <class FL, int NWO>
__device__ __forceinline__ void ss_int8_unit(const uint32_t (&in)[8], uint32_t (&out)[NWO])
{
    constexpr int B = FL::bits;
    constexpr uint32_t M = FL::max_mag;
    constexpr uint32_t one = both_halves(half_bits(1, -17)), bias = both_halves(half_bits(-(1024 + 128), -17));
    constexpr uint32_t factor = both_halves(half_bits(1025, B - 25) | 0x8000u);        // -(1 + 2^-10), see round_halves
    const auto round_pair = [&](uint32_t p) {                                          // -> M - q
        const uint32_t h = __viaddmax_s16x2(p, both_halves(0x6480u), both_halves(0x6480u - (M << (8 - B))));
        return hfma2_relu(hfma2(h, one, bias), factor, both_halves(M));
    };
    // selector bit 3 replicates the sign of the byte
    if constexpr (B <= 3) {
        uint32_t z[4];
        static_for<4>([&](auto jj) {
            constexpr int J = decltype(jj)::value;
            const uint32_t w0 = in[2 * J], w1 = in[2 * J + 1];
            uint32_t p0, p1, p2, p3;
            asm("prmt.b32 %0, %1, %2, 0xC480;" : "=r"(p0) : "r"(w0), "r"(w1));
            asm("prmt.b32 %0, %1, %2, 0xD591;" : "=r"(p1) : "r"(w0), "r"(w1));
            asm("prmt.b32 %0, %1, %2, 0xE6A2;" : "=r"(p2) : "r"(w0), "r"(w1));
            asm("prmt.b32 %0, %1, %2, 0xF7B3;" : "=r"(p3) : "r"(w0), "r"(w1));
            constexpr uint32_t k = 1u << B;
            const uint32_t y = (round_pair(p3) * k + round_pair(p2)) * (k * k) + (round_pair(p1) * k + round_pair(p0));
            if constexpr (B == 3) z[J] = join_halves_low<12>(y);
            else z[J] = y;
        });
        if constexpr (B == 3) {
            pack_low_streams<24>(z, out);
        } else {
            out[0] = __byte_perm(z[0], z[1], 0x6420);
            out[1] = __byte_perm(z[2], z[3], 0x6420);
        }
    } else {
        uint32_t y[8];
        static_for<8>([&](auto jj) {
            constexpr int J = decltype(jj)::value;
            uint32_t a, b;
            asm("prmt.b32 %0, %1, %1, 0xA280;" : "=r"(a) : "r"(in[J]));
            asm("prmt.b32 %0, %1, %1, 0xB391;" : "=r"(b) : "r"(in[J]));
            y[J] = round_pair(b) * (1u << B) + round_pair(a);
            if constexpr (B > 4) y[J] = join_halves_low<2 * B>(y[J]);
        });
        if constexpr (B == 4) {
#pragma unroll
            for (int j = 0; j < 4; ++j) out[j] = __byte_perm(y[2 * j], y[2 * j + 1], 0x6420);
        } else {
            pack_low_streams<4 * B>(y, out);
        }
    }
    unbias_codes<B>(out);
}

// Convert the 32 codes of one lane.  in: 8*FH::bits/8... words of the high format's bitstream.  SHORT: by ss_int8_unit (MXINT8 only).
template <class FH, class FL, bool SHORT, int NWI, int NWO>
__device__ __forceinline__ void slice_scale_unit(const uint32_t (&in)[NWI], uint32_t (&out)[NWO])
{
    if constexpr (FH::id == FL::id) {
#pragma unroll
        for (int j = 0; j < NWO; ++j) out[j] = in[j];
    } else if constexpr (SHORT) {
        static_assert(FH::id == MXQ_INT8, "MXINT8 only");
        ss_int8_unit<FL>(in, out);
    } else {
        uint32_t z[1][8];
        if constexpr (!FH::has_nan) {
            ss_unit<false, FH, FL>(in, z);
            ss_finish<FL>(z[0], out);
        } else if (!unit_has_e4m3_nan(in)) {
            ss_unit<false, FH, FL>(in, z);
            ss_finish<FL>(z[0], out);
        } else {
            // an E4M3 NaN code (never produced by the quantizer): the slow path, which costs this kernel nothing
            // where ss_unit<true> slows the 6-bit targets by 1.5 %
            ss_unit_by_element<FH, FL>(in, out);
        }
    }
}

// Scale bytes are an element-wise stream of their own: byte -> min(byte + de, 254), 0xFF kept.
__device__ __forceinline__ uint8_t ss_scale_byte(uint32_t b, int de)
{
    return (uint8_t)(b == 0xFFu ? 0xFFu : min(b + (uint32_t)de, 254u));
}

// One warp tile (32 U lane units) of one tensor; shared by the single-tensor and the batched
// kernels.  The scale bytes are an element-wise stream of their own: lane unit i also converts
// scale i, or, with HALVES (block 16, two scales per lane unit), its own two as one 16-bit access: MXINT8 -> MXINT4 of
// 2^25 codes 9.1 us, E4M3 -> E2M3 11.3, where a second pass over the upper half of the scales took 10.8 and 12.7.  (A
// run-time choice between the two forms cost the larger blocks 2 - 9 %.)
template <class FH, class FL, int U, bool HALVES, bool SHORT = false, class SCALES>
__device__ __forceinline__ void slice_scale_tile(const uint8_t* __restrict__ codes, const uint8_t* __restrict__ scales,
                                                 size_t nunits, size_t nscales, uint8_t* __restrict__ out_codes,
                                                 const SCALES& out_scales, size_t tile, uint8_t* stage)
{
    constexpr int IB = 4 * FH::bits, OB = 4 * FL::bits;      // bytes per lane unit
    constexpr int NWI = IB / 4, NWO = OB / 4;
    constexpr int de = FH::emax - FL::emax;
    const size_t u0 = tile * (32 * U) + (threadIdx.x & 31);
    uint32_t w[U][NWI];
    uint32_t sb[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const size_t unit = u0 + u * 32;
        if (unit < nunits) load_words<NWI>(w[u], codes + unit * IB);
        else {
#pragma unroll
            for (int j = 0; j < NWI; ++j) w[u][j] = 0;
        }
        if constexpr (HALVES) sb[u] = unit < nunits ? ld_u16(scales + unit * 2) : 0;
        else sb[u] = unit < nscales ? ld_u8(scales + unit) : 0;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const size_t unit = u0 + u * 32;
        if constexpr (HALVES) {
            if (unit < nunits) st_u16(out_scales + unit * 2, ss_scale_byte(sb[u] & 0xFFu, de) | ss_scale_byte(sb[u] >> 8, de) << 8);
        } else {
            if (unit < nscales) put_scale(out_scales, unit, ss_scale_byte(sb[u], de));
        }
        uint32_t out[NWO];
        slice_scale_unit<FH, FL, SHORT>(w[u], out);
        if constexpr (StagedTile<OB>::use) store_bytes<OB>(stage + (u * 32 + (threadIdx.x & 31)) * OB, out);
        else if (unit < nunits) store_bytes<OB>(out_codes + unit * OB, out);
    }
    if constexpr (StagedTile<OB>::use) {
        const size_t first = tile * (32 * U), left = nunits - first;
        flush_stage<32 * U * OB>(stage, out_codes + first * OB, (uint32_t)(left < 32 * U ? left : 32 * U) * OB);
    }
}

// The staging area of the calling warp for a Slice-and-Scale tile (null when the target's pieces are
// single vectors).  Must be called by every thread of the CTA, outside divergent code.
template <class FL, int U, int THREADS>
__device__ __forceinline__ uint8_t* slice_scale_stage()
{
    constexpr int OB = 4 * FL::bits;
    if constexpr (StagedTile<OB>::use) {
        __shared__ __align__(128) uint8_t stage_area[(THREADS / 32) * 32 * U * OB];
        return stage_area + (threadIdx.x >> 5) * (32 * U * OB);
    } else {
        return nullptr;
    }
}

// Resident CTAs (of 128 threads) per SM the single-tensor kernel is compiled for, i.e. its register budget; 10 against 14, mean over
// 2^24 to 2^26.5 codes.  MXINT to five bits and more and to two gets room for 48 registers (with 14 MXINT8 -> 7 / 6 / 5 / 2 bits are 7 / 8 / 6 / 5 %
// slower), MXINT8 -> 4 and 3 fit 32 (with 10 1 and 5 % slower; from MXINT7, 6 and 5 to 3 bits 10 would be 3 - 6 % faster, the other narrow
// sources take the same), and so do the MXFP ones (block 32: the same to 2 %).  With tiled scale outputs 14 CTAs would spill, so
// those keep 12.
//   SMALL : see slice_scale_is_small.
template <class FH, class FL, class SCALES, bool SMALL>
__host__ __device__ constexpr int slice_scale_min_ctas()
{
    if constexpr (!std::is_same_v<SCALES, uint8_t*>) return 12;
    else return SMALL || (FH::kind == KIND_INT && FL::bits != 4 && FL::bits != 3) ? 10 : 14;
}

// MXINT8 in a launch of about one wave.  The next launch's CTAs are resident early (see mxq_access.cuh): as many as fit beside
// this one's at once, the others wherever one of this one's has ended, so the more fit the more unevenly they spread, which a grid of
// one wave does not make up for.  Kernels with ss_int8_unit and at most 10 CTAs to an SM (12 to 4 bits, whose code leaves room for no
// fewer), against the larger launches' kernels: 2^23.25 codes -> 7 bits 3.9 and 4.4 us, 6 3.8 and 4.3, 4 3.3 and 4.0, 3 3.6 and 4.3; 2^22 -> 7 3.2
// and 3.5, 3 3.0 and 3.2.  They stop at one wave (2^24 codes -> 6 bits 5.4 and 5.2), and to 4 bits also below five CTAs per SM, where the
// other one is the faster (2^22 codes 2.65 and 2.4).  5 and 2 bits have one kernel (5 bits with 10 CTAs: 2^22.75 codes 4.2 us
// against 3.2; 2 bits: at most 12 either way).
template <class FH, class FL>
__host__ __device__ constexpr bool slice_scale_has_small()
{
    return FH::id == MXQ_INT8 && (FL::bits == 7 || FL::bits == 6 || FL::bits == 4 || FL::bits == 3);
}

template <class FL>
inline bool slice_scale_is_small(size_t ctas)
{
    return ctas > (size_t)148 * (FL::bits == 4 ? 5 : 0) && ctas <= (size_t)148 * (FL::bits > 4 ? 10 : 12);
}

template <class FH, class FL, int U, int THREADS, class SCALES = uint8_t*, bool HALVES = false, bool SMALL = false>
__global__ void __launch_bounds__(THREADS, slice_scale_min_ctas<FH, FL, SCALES, SMALL>())
slice_scale_kernel(const uint8_t* __restrict__ codes, const uint8_t* __restrict__ scales, size_t nunits,
                   size_t nscales, uint8_t* __restrict__ out_codes, SCALES out_scales)
{
    // (to 7 bits the general form is as fast in larger launches, to 6, 5 and 4 faster: 2^25 codes -> 6 9.8 us against 10.1, 2^24.5 -> 5
    // 7.5 and 7.7; to 3 bits it takes 8.9 against 8.0, to 2 the same but 4.25 against 3.4 at 2^23.5)
    constexpr bool kShort = FH::id == MXQ_INT8 && (SMALL || FL::bits <= 3);
    pdl_release();
    const size_t tile = (size_t)blockIdx.x * (THREADS / 32) + (threadIdx.x >> 5);
    uint8_t* stage = slice_scale_stage<FL, U, THREADS>();
    if (is_padding_cta<THREADS>(out_scales, blockIdx.x, nunits, THREADS * U)) return;
    prefetch_tile<U, 4 * FH::bits>(codes, tile, nunits);
    pdl_acquire();
    if (tile * (32 * U) < nunits)
        slice_scale_tile<FH, FL, U, HALVES, kShort>(codes, scales, nunits, nscales, out_codes, out_scales, tile, stage);
}

// Several targets from one read of the anchor (the elastic-serving case: one stored checkpoint, several lower
// precisions wanted at once).  Per element 1.03 bytes are read once instead of once per target, and what the
// conversions share (the FP16 values of the codes) is computed once.  The set of targets is a compile-time list: a kernel that
// walks a run-time list of formats keeps the shared words in registers across a switch and took 38 - 46 us for MXINT8 -> {7, 5, 3}
// bits of 2^25.8 codes (block 64) where these take 30 (a pass per target: 50; the bytes alone: 26.7).  Compiled for 12
// resident CTAs (40 registers): with 10, 2^25.8 codes to {7, 5, 3} take 29.0 us against 28.9, {6, 4} 21.7 and 21.5, {7, 5} 25.1 and 24.7,
// and launches of one or two waves gain or lose up to 20 % with their size ({6, 4} of 2^23.5 codes 4.9 against 5.4, 2^24 7.6 and 7.25); with
// 14 most sets spill.  Sets of four spill at 12 and get 10.  A few still spill: {5, 3, 2} 48 bytes, {4, 3}, {4, 2}, {5, 4, 3}, {5, 4, 2} and
// {7, 6, 4, 3} 4, {7, 6, 4, 2}, {7, 4, 3, 2} and {6, 4, 3, 2} 8, {E3M3, E3M2, E2M3} 12, {E3M3, E3M2, E2M2} 4.  Of the MXINT8 ones none is
// slower for it than with the integer rounding, which spilled in one of them (2^26 codes: {5, 3, 2} 31.3 -> 30.8 us, {4, 2} 22.6 -> 20.3,
// {5, 4, 2} 30.6 -> 27.5, {7, 6, 4, 2} 40.8 -> 38.2; 2^24: 10.7 -> 9.8, 6.7 -> 6.2, 10.6 -> 9.2, 12.5 -> 11.8).
struct SsOut {
    uint8_t* codes;
    uint8_t* scales;
};

template <int N>
struct SsOuts {
    SsOut t[N];
};

// Bytes of staging area per lane unit that the targets before number I need (I = the count: all of them).
template <int I, class... FL>
__host__ __device__ constexpr int ss_stage_offset()
{
    constexpr int ob[] = {(StagedTile<4 * FL::bits>::use ? 4 * FL::bits : 0)...};
    int sum = 0;
    for (int i = 0; i < I; ++i) sum += ob[i];
    return sum;
}

// One CTA tile (THREADS * U lane units, 32 U consecutive ones per warp) of an 8-bit anchor into all targets; shared
// by the single-tensor and the batched kernels.  `first` is the tile's first unit: it depends on the block
// alone, so the 64-bit bases of all streams live in uniform registers and a lane adds 32-bit offsets.
template <class FH, int U, int THREADS, class... FL>
__device__ __forceinline__ void slice_scale_set_tile(const uint8_t* __restrict__ codes, const uint8_t* __restrict__ scales,
                                                     size_t nunits, size_t nscales, const SsOut* outs, size_t first,
                                                     uint8_t* stage)
{
    static_assert(FH::bits == 8, "an 8-bit anchor");
    constexpr int N = sizeof...(FL);
    constexpr uint32_t kTile = THREADS * U;
    const uint32_t lane = threadIdx.x & 31, warp0 = (threadIdx.x >> 5) * (32 * U), l0 = warp0 + lane;
    // units and scales of the tensor inside this tile (a block of 64 or 128 has fewer scales than units: the
    // first tiles carry them)
    const uint32_t valid = nunits - first < kTile ? (uint32_t)(nunits - first) : kTile;
    const uint32_t valid_scales = first >= nscales ? 0u : nscales - first < kTile ? (uint32_t)(nscales - first) : kTile;
    codes += first * 32;
    uint32_t w[U][8];
    uint32_t sb[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        if (l0 + u * 32 < valid) ld256(w[u], codes + (l0 + u * 32) * 32);
        else {
#pragma unroll
            for (int j = 0; j < 8; ++j) w[u][j] = 0;
        }
        sb[u] = l0 + u * 32 < valid_scales ? ld_u8(scales + first + (l0 + u * 32)) : 0;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
        if (l0 + u * 32 < valid_scales) {
            static_for<N>([&](auto i) {
                constexpr int I = decltype(i)::value;
                st_u8(outs[I].scales + first + (l0 + u * 32), ss_scale_byte(sb[u], FH::emax - ss_target_t<I, FL...>::emax));
            });
        }
        uint32_t z[N][8];
        // one NaN-code check, all conversions in one straight line
        if (FH::kind == KIND_INT || !unit_has_e4m3_nan(w[u])) ss_unit<false, FH, FL...>(w[u], z);
        else if constexpr (FH::kind == KIND_FP) ss_unit<true, FH, FL...>(w[u], z);
        static_for<N>([&](auto i) {
            constexpr int I = decltype(i)::value;
            using F = ss_target_t<I, FL...>;
            constexpr int OB = 4 * F::bits;
            uint32_t out[OB / 4];
            ss_finish<F, ss_low_join<FH, FL...>()>(z[I], out);
            if constexpr (StagedTile<OB>::use)
                store_bytes<OB>(stage + 32 * U * ss_stage_offset<I, FL...>() + (u * 32 + lane) * OB, out);
            else if (l0 + u * 32 < valid) store_bytes<OB>(outs[I].codes + first * OB + (l0 + u * 32) * OB, out);
        });
    }
    if constexpr (ss_stage_offset<N, FL...>() > 0) {
        if (warp0 < valid) {                                    // whole warps
            const uint32_t mine = valid - warp0 < 32 * U ? valid - warp0 : 32 * U;
            static_for<N>([&](auto i) {
                constexpr int I = decltype(i)::value;
                constexpr int OB = 4 * ss_target_t<I, FL...>::bits;
                if constexpr (StagedTile<OB>::use)
                    flush_stage_async<32 * U * OB>(stage + 32 * U * ss_stage_offset<I, FL...>(),
                                                   outs[I].codes + first * OB + warp0 * OB, mine * OB);
            });
            stage_wait<0>();
        }
    }
    if (nscales > nunits) {                                     // block 16: two scales per lane unit
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const size_t i = nunits + first + (l0 + u * 32);
            if (i < nscales) {
                const uint32_t b = ld_u8(scales + i);
                static_for<N>([&](auto k) {
                    constexpr int I = decltype(k)::value;
                    st_u8(outs[I].scales + i, ss_scale_byte(b, FH::emax - ss_target_t<I, FL...>::emax));
                });
            }
        }
    }
}

// Asks L2 for the tile's input lines (see prefetch_tile): lane l of the CTA for the line of each of its U units.
template <int U, int THREADS, int UNIT_BYTES>
__device__ __forceinline__ void prefetch_cta_tile(const uint8_t* base, size_t first, size_t nunits)
{
    const uint32_t l0 = (threadIdx.x >> 5) * (32 * U) + (threadIdx.x & 31);
    base += first * UNIT_BYTES;
    const uint32_t valid = nunits - first < THREADS * U ? (uint32_t)(nunits - first) : THREADS * U;
#pragma unroll
    for (int u = 0; u < U; ++u)
        if (l0 + u * 32 < valid) asm volatile("prefetch.global.L2 [%0];" :: "l"(base + (l0 + u * 32) * UNIT_BYTES));
}

// The staging areas of the calling warp (null where every target's pieces are stored directly).
// Must be called by every thread of the CTA, outside divergent code.
template <int U, int THREADS, class... FL>
__device__ __forceinline__ uint8_t* slice_scale_set_stage()
{
    constexpr int kWarp = 32 * U * ss_stage_offset<(int)sizeof...(FL), FL...>();
    if constexpr (kWarp > 0) {
        __shared__ __align__(128) uint8_t area[(THREADS / 32) * kWarp];
        return area + (threadIdx.x >> 5) * kWarp;
    } else {
        return nullptr;
    }
}

template <class FH, int U, int THREADS, class... FL>
__global__ void __launch_bounds__(THREADS, sizeof...(FL) >= 4 ? 10 : 12)
slice_scale_set_kernel(const uint8_t* __restrict__ codes, const uint8_t* __restrict__ scales, size_t nunits, size_t nscales,
                       const __grid_constant__ SsOuts<(int)sizeof...(FL)> outs)
{
    pdl_release();
    const size_t first = (size_t)blockIdx.x * (THREADS * U);
    uint8_t* stage = slice_scale_set_stage<U, THREADS, FL...>();
    prefetch_cta_tile<U, THREADS, 32>(codes, first, nunits);
    pdl_acquire();
    slice_scale_set_tile<FH, U, THREADS, FL...>(codes, scales, nunits, nscales, outs.t, first, stage);
}

// Device-side item of the batched conversion (one tensor), with its place in the flattened
// tile space of the whole batch.
struct SsDeviceItem {
    const uint8_t* codes;
    const uint8_t* scales;
    uint8_t* out_codes;
    uint8_t* out_scales;
    size_t nunits;
    size_t nscales;
    size_t tile_begin;     // first global tile index of this tensor
};

// All tensors in one launch: the tiles of every tensor are laid end to end and every CTA finds the
// tensor its tile belongs to by a search of the item table, so small tensors do not leave SMs idle.
template <class FH, class FL, int U, int THREADS>
__global__ void __launch_bounds__(THREADS)
slice_scale_batched_kernel(const SsDeviceItem* __restrict__ items, const TileIndex* __restrict__ index)
{
    pdl_release();
    uint8_t* stage = slice_scale_stage<FL, U, THREADS>();
    pdl_acquire();
    // items are sorted by tile_begin: the last one that starts at or before this CTA's tile owns it
    // (table and index are device memory written by the copy in front of this launch: read after the wait)
    const SsDeviceItem& t = items[find_item(items, *index, blockIdx.x)];
    const size_t tile = item_warp_tile<THREADS>(t.tile_begin);
    if (tile * (32 * U) < t.nunits)                       // whole warps
        slice_scale_tile<FH, FL, U, false>(t.codes, t.scales, t.nunits, t.nscales, t.out_codes, t.out_scales, tile, stage);
}

// The same launch with the item table carried in the kernel's parameter space (K items, 56 bytes
// each, plus the coarse index: K = 64 stays near the classic 4 KB of parameters, K = 512 uses the
// 32 KB that sm_70 and later allow).  No device buffer, no host-to-device copy in front of the kernel.
template <int K>
struct SsItemBlock {
    SsDeviceItem items[K];
    TileIndex index;
};

// (Compiled for 12 resident CTAs: against the compiler's own choice, seven tensors of 2^25 to 2^28 codes in all, E4M3 -> E2M3 and E3M2 7 % faster,
// MXINT8 -> 3 bits 5 %, -> 7, 5 and E3M3, E2M2 2 %, the others the same but MXINT8 -> 6 bits, 3 % slower.  SMALL: see
// slice_scale_is_small; seven tensors of 2^23 codes -> 7 bits 4.0 us against 4.4, 6 3.8 and 4.3, 3 3.4 and 3.8.)
template <class FH, class FL, int U, int THREADS, int K, bool SMALL = false>
__global__ void __launch_bounds__(THREADS, SMALL ? 10 : 12)
slice_scale_batched_param_kernel(const __grid_constant__ SsItemBlock<K> blk)
{
    // (2^25 codes, short against general form: -> 7 bits 10.7 us and 11.5, 3 8.4 and 8.9, 2^24 -> 2 4.05 and 4.3, 4 4.2 and 4.3)
    constexpr bool kShort = FH::id == MXQ_INT8 && FL::bits < 8 && (SMALL || (FL::bits != 6 && FL::bits != 5));
    pdl_release();
    uint8_t* stage = slice_scale_stage<FL, U, THREADS>();
    // parameters: readable before the wait
    const SsDeviceItem& t = blk.items[find_item(blk.items, blk.index, blockIdx.x)];
    const size_t tile = item_warp_tile<THREADS>(t.tile_begin);
    prefetch_tile<U, 4 * FH::bits>(t.codes, tile, t.nunits);
    pdl_acquire();
    if (tile * (32 * U) < t.nunits)                       // whole warps
        slice_scale_tile<FH, FL, U, false, kShort>(t.codes, t.scales, t.nunits, t.nscales, t.out_codes, t.out_scales, tile, stage);
}

// Two targets from one read of every anchor of a set of tensors (the whole-model conversion of Sec. 3.5
// for a deployment that serves two lower precisions at once): items of 72 bytes, 256 per launch.
struct SsPairDeviceItem {
    const uint8_t* codes;
    const uint8_t* scales;
    SsOut out[2];
    size_t nunits;
    size_t nscales;
    size_t tile_begin;
};

template <int K>
struct SsPairItemBlock {
    SsPairDeviceItem items[K];
    TileIndex index;
};

// (Resident CTAs: for MXINT8 ten, because twelve spill for some pairs -- four layers to 5 + 4 bits 363 us against 292, 6 + 4 305 and
// 302, 7 + 5 361 and 358; for E4M3 twelve.)
template <class FH, class FL1, class FL2, int U, int THREADS, int K>
__global__ void __launch_bounds__(THREADS, FH::kind == KIND_INT ? 10 : 12)
slice_scale_pair_batched_kernel(const __grid_constant__ SsPairItemBlock<K> blk)
{
    pdl_release();
    uint8_t* stage = slice_scale_set_stage<U, THREADS, FL1, FL2>();
    const SsPairDeviceItem& t = blk.items[find_item(blk.items, blk.index, blockIdx.x)];
    const size_t first = (blockIdx.x - t.tile_begin) * (THREADS * U);
    prefetch_cta_tile<U, THREADS, 32>(t.codes, first, t.nunits);
    pdl_acquire();
    slice_scale_set_tile<FH, U, THREADS, FL1, FL2>(t.codes, t.scales, t.nunits, t.nscales, t.out, first, stage);
}

// The batched conversion with every tensor's scale bytes written in the tiled order (block 32): the
// item carries the matrix's TiledScales record in place of a plain pointer.  K = 256 items of 72 bytes
// ride in the kernel parameters.
struct SsTiledDeviceItem {
    const uint8_t* codes;
    const uint8_t* scales;
    uint8_t* out_codes;
    TiledScales out_scales;
    size_t nunits;
    size_t tile_begin;
};

template <int K>
struct SsTiledItemBlock {
    SsTiledDeviceItem items[K];
    TileIndex index;
};

template <class FH, class FL, int U, int THREADS, int K>
__global__ void __launch_bounds__(THREADS)
slice_scale_tiled_batched_kernel(const __grid_constant__ SsTiledItemBlock<K> blk)
{
    pdl_release();
    uint8_t* stage = slice_scale_stage<FL, U, THREADS>();
    // parameters: readable before the wait
    const SsTiledDeviceItem& t = blk.items[find_item(blk.items, blk.index, blockIdx.x)];
    if (is_padding_cta<THREADS>(t.out_scales, blockIdx.x - t.tile_begin, t.nunits, THREADS * U)) return;
    const size_t tile = item_warp_tile<THREADS>(t.tile_begin);
    prefetch_tile<U, 4 * FH::bits>(t.codes, tile, t.nunits);
    pdl_acquire();
    if (tile * (32 * U) < t.nunits)                       // whole warps
        slice_scale_tile<FH, FL, U, false>(t.codes, t.scales, t.nunits, t.nunits, t.out_codes, t.out_scales, tile, stage);
}

// ------------------------------------------------------------------------------------------
// Reconstruction V^ = X P.  One lane = 32 codes.
// ------------------------------------------------------------------------------------------

// Two kernels.  For 16-bit outputs a lane takes 32 codes (one block: 16 - 32 bytes of codes in one
// vector load) and writes 64 bytes; for FP32 outputs that shape would spread every store instruction
// of a warp over 32 different 128-byte lines (measured 84 % of the copy rate), so there a lane unit
// is 32 bytes of OUTPUT instead and every store instruction covers 1 KB of consecutive addresses
// (98 %).  The second shape was 1 - 2 % slower than the first for BF16 outputs.

template <class F, class T, int U>
__device__ __forceinline__ void dequantize_tile(const uint8_t* __restrict__ codes, const uint8_t* __restrict__ scales,
                                                size_t nunits, int units_per_scale_shift, int scales_per_unit,
                                                uint8_t* __restrict__ dst, size_t tile)
{
    constexpr int IB = 4 * F::bits, NWI = IB / 4;
    constexpr int OBYTES = 32 * T::size;                      // 64 or 128 bytes out per lane
    const int lane = threadIdx.x & 31;
    const size_t u0 = tile * (32 * U) + lane;
    uint32_t w[U][NWI];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const size_t unit = u0 + u * 32;
        if (unit < nunits) load_words<NWI>(w[u], codes + unit * IB);
        else {
#pragma unroll
            for (int j = 0; j < NWI; ++j) w[u][j] = 0;
        }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const size_t unit = u0 + u * 32;
        if (unit >= nunits) continue;
        // scales_per_unit is 1 (block >= 32: one scale shared by 2^shift units) or 2 (block 16)
        uint32_t sbyte[2];
        if (scales_per_unit == 1) {
            sbyte[0] = sbyte[1] = ld_u8(scales + (unit >> units_per_scale_shift));
        } else {
            sbyte[0] = ld_u8(scales + unit * 2);
            sbyte[1] = ld_u8(scales + unit * 2 + 1);
        }
        uint8_t* o = dst + unit * OBYTES;
        // four 32-byte stores for FP32 (8 elements each), two for BF16 (16 elements each)
        constexpr int EPS = 32 / T::size;
        static_for<32 / EPS>([&](auto k) {
            constexpr int K = decltype(k)::value;
            const uint32_t sbk = sbyte[(K * EPS) / 16];
            uint32_t out[8];
            if (sbk == 0xFFu) {
#pragma unroll
                for (int j = 0; j < 8; ++j) out[j] = T::size == 4 ? 0x7FC00000u : 0x7FC07FC0u;
            } else if (F::id == MXQ_FP8_E4M3 && T::size == 2 &&
                       !(has_e4m3_nan(w[u][(4 * K) % NWI]) | has_e4m3_nan(w[u][(4 * K + 1) % NWI]) |
                         has_e4m3_nan(w[u][(4 * K + 2) % NWI]) | has_e4m3_nan(w[u][(4 * K + 3) % NWI]))) {
                // MXFP8 anchor codes (no NaN code among these 16): the widening conversion gives the
                // exact values, one FP32 multiply applies the scale as in the generic path below
                const float X = scale_value(sbk);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    uint32_t a, b;
                    e4m3_word_to_f16(w[u][(4 * K + j) % NWI], a, b);
                    float f0, f1, f2, f3;
                    asm("{ .reg .b16 l, h; mov.b32 {l, h}, %4; cvt.f32.f16 %0, l; cvt.f32.f16 %1, h;\n"
                        "  mov.b32 {l, h}, %5; cvt.f32.f16 %2, l; cvt.f32.f16 %3, h; }"
                        : "=f"(f0), "=f"(f1), "=f"(f2), "=f"(f3) : "r"(a), "r"(b));
                    out[2 * j] = pack_bf16x2(f0 * X, f1 * X);
                    out[2 * j + 1] = pack_bf16x2(f2 * X, f3 * X);
                }
            } else {
                const float X = scale_value(sbk);
                static_for<EPS / 2>([&](auto i) {
                    constexpr int I = K * EPS + 2 * decltype(i)::value;
                    const uint32_t c0 = get_code<F::bits, I>(w[u]), c1 = get_code<F::bits, I + 1>(w[u]);
                    float y0 = decode<F>(c0) * X;
                    float y1 = decode<F>(c1) * X;
                    // an E4M3 NaN code reconstructs to the canonical quiet NaN
                    bool n0 = false, n1 = false;
                    if constexpr (F::has_nan) {
                        n0 = (c0 & 0x7Fu) == 0x7Fu;
                        n1 = (c1 & 0x7Fu) == 0x7Fu;
                    }
                    if constexpr (T::size == 4) {
                        out[I - K * EPS] = n0 ? 0x7FC00000u : __float_as_uint(y0);
                        out[I - K * EPS + 1] = n1 ? 0x7FC00000u : __float_as_uint(y1);
                    } else {
                        uint32_t p = pack_bf16x2(y0, y1);
                        if (n0) p = (p & 0xFFFF0000u) | 0x7FC0u;
                        if (n1) p = (p & 0x0000FFFFu) | 0x7FC00000u;
                        out[(I - K * EPS) / 2] = p;
                    }
                });
            }
            st256(o + K * 32, out);
        });
    }
}

template <class F, class T, int U, int THREADS>
__global__ void __launch_bounds__(THREADS)
dequantize_kernel(const uint8_t* __restrict__ codes, const uint8_t* __restrict__ scales, size_t nunits,
                  int units_per_scale_shift, int scales_per_unit, uint8_t* __restrict__ dst)
{
    pdl_release();
    const size_t tile = (size_t)blockIdx.x * (THREADS / 32) + (threadIdx.x >> 5);
    pdl_acquire();
    if (tile * (32 * U) < nunits)
        dequantize_tile<F, T, U>(codes, scales, nunits, units_per_scale_shift, scales_per_unit, dst, tile);
}


// A lane unit is 32 bytes of OUTPUT (16 BF16 or 8 FP32 elements), so that every store instruction
// of a warp covers 1 KB of consecutive addresses; the codes of a unit are 2 x bits or bits bytes,
// read with the widest access their alignment allows.  A unit never straddles a block (blocks are
// at least 16 elements), so it needs one scale: scales[unit >> scale_shift].
template <class F, class T, int U>
__device__ __forceinline__ void dequantize_wide_tile(const uint8_t* __restrict__ codes, const uint8_t* __restrict__ scales,
                                                     size_t nunits, int scale_shift, uint8_t* __restrict__ dst, size_t tile)
{
    constexpr int EPL = T::epl;                               // elements per lane unit
    constexpr int IB = EPL * F::bits / 8;                     // code bytes per lane unit
    constexpr int NWI = (IB + 3) / 4;
    const size_t u0 = tile * (32 * U) + (threadIdx.x & 31);
    uint32_t w[U][NWI];
    uint32_t sb[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const size_t unit = u0 + u * 32;
        if constexpr (IB == 3 || (IB > 4 && IB < 8)) {
            // lanes beyond the end take the last unit: inside a branch the shifts would wait for one unit's words before the
            // next unit's are asked for (2^14 codes of 6 bits 1.7 us instead of 1.4)
            const size_t mine = unit < nunits ? unit : nunits - 1;
            load_piece<IB>(w[u], codes, mine);
            sb[u] = ld_u8(scales + (mine >> scale_shift));
        } else if (unit < nunits) {
            load_bytes<IB>(w[u], codes + unit * IB);
            sb[u] = ld_u8(scales + (unit >> scale_shift));
        } else {
#pragma unroll
            for (int j = 0; j < NWI; ++j) w[u][j] = 0;
            sb[u] = 0;
        }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const size_t unit = u0 + u * 32;
        uint32_t out[8];
        const float X = scale_value(min(sb[u], 254u));
        static_for<EPL / 2>([&](auto i) {
            constexpr int I = 2 * decltype(i)::value;
            const uint32_t c0 = get_code<F::bits, I>(w[u]), c1 = get_code<F::bits, I + 1>(w[u]);
            float y0 = decode<F>(c0) * X;
            float y1 = decode<F>(c1) * X;
            // an E4M3 NaN code reconstructs to the canonical quiet NaN
            bool n0 = false, n1 = false;
            if constexpr (F::has_nan) {
                n0 = (c0 & 0x7Fu) == 0x7Fu;
                n1 = (c1 & 0x7Fu) == 0x7Fu;
            }
            if constexpr (T::size == 4) {
                out[I] = n0 ? 0x7FC00000u : __float_as_uint(y0);
                out[I + 1] = n1 ? 0x7FC00000u : __float_as_uint(y1);
            } else {
                uint32_t p = pack_bf16x2(y0, y1);
                if (n0) p = (p & 0xFFFF0000u) | 0x7FC0u;
                if (n1) p = (p & 0x0000FFFFu) | 0x7FC00000u;
                out[I / 2] = p;
            }
        });
        if (sb[u] == 0xFFu) {                                 // poisoned block
#pragma unroll
            for (int j = 0; j < 8; ++j) out[j] = T::size == 4 ? 0x7FC00000u : 0x7FC07FC0u;
        }
        if (unit < nunits) st256(dst + unit * 32, out);
    }
}

template <class F, class T, int U, int THREADS>
__global__ void __launch_bounds__(THREADS)
dequantize_wide_kernel(const uint8_t* __restrict__ codes, const uint8_t* __restrict__ scales, size_t nunits, int scale_shift,
                       uint8_t* __restrict__ dst)
{
    pdl_release();
    const size_t tile = (size_t)blockIdx.x * (THREADS / 32) + (threadIdx.x >> 5);
    pdl_acquire();
    if (tile * (32 * U) < nunits) dequantize_wide_tile<F, T, U>(codes, scales, nunits, scale_shift, dst, tile);
}

// Reconstruction of a whole set of tensors in one launch (tiles end to end, items in the parameters).
// `shift` and `scales_per_unit` are those of the single-tensor kernel of the same output type.
struct DqDeviceItem {
    const uint8_t* codes;
    const uint8_t* scales;
    uint8_t* dst;
    size_t nunits;
    size_t tile_begin;
};

template <int K>
struct DqItemBlock {
    DqDeviceItem items[K];
    TileIndex index;
};

template <class F, class T, int U, int THREADS, int K>
__global__ void __launch_bounds__(THREADS)
dequantize_batched_kernel(const __grid_constant__ DqItemBlock<K> blk, int shift, int scales_per_unit)
{
    pdl_release();
    const DqDeviceItem& t = blk.items[find_item(blk.items, blk.index, blockIdx.x)];
    const size_t tile = item_warp_tile<THREADS>(t.tile_begin);
    pdl_acquire();
    if (tile * (32 * U) >= t.nunits) return;              // whole warps
    if constexpr (T::size == 4) dequantize_wide_tile<F, T, U>(t.codes, t.scales, t.nunits, shift, t.dst, tile);
    else dequantize_tile<F, T, U>(t.codes, t.scales, t.nunits, shift, scales_per_unit, t.dst, tile);
}

// ------------------------------------------------------------------------------------------
// Straight-through backward: a plain copy
// ------------------------------------------------------------------------------------------

template <int U, int THREADS>
__global__ void __launch_bounds__(THREADS)
copy_kernel(const uint8_t* __restrict__ src, size_t nbytes, uint8_t* __restrict__ dst)
{
    pdl_release();
    const size_t nunits = nbytes / 32;
    const int lane = threadIdx.x & 31;
    const size_t warp = (size_t)blockIdx.x * (THREADS / 32) + (threadIdx.x >> 5);
    const size_t ntiles = (nunits + 32 * U - 1) / (32 * U);
    prefetch_tile<U, 32>(src, warp, nunits);
    pdl_acquire();
    if (const size_t tile = warp; tile < ntiles) {
        const size_t u0 = tile * (32 * U) + lane;
        uint32_t w[U][8];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (u0 + u * 32 < nunits) ld256(w[u], src + (u0 + u * 32) * 32);
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (u0 + u * 32 < nunits) st256(dst + (u0 + u * 32) * 32, w[u]);
    }
    // ragged tail (n * size need not be a multiple of 32 bytes)
    const size_t tid = (size_t)blockIdx.x * THREADS + threadIdx.x;
    for (size_t i = nunits * 32 + tid; i < nbytes; i += (size_t)gridDim.x * THREADS) st_u8(dst + i, ld_u8(src + i));
}

}  // namespace mxq
