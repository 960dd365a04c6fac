// fx.cuh -- FP64 products on the 5th-generation tensor cores from exact integer pieces
// (the error-free splitting of Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 2012):
// an operand row or column is put on a fixed-point grid of 56 bits below its largest
// entry and cut into seven signed 8-bit digits, exact in FP16; the products of digits i and
// j with i + j = l accumulate exactly in one FP32 accumulator per level l <= 6 (integers
// below 2^24 for up to 128 products); the level sums are joined in 64-bit integers and
// rounded once.  The error of a product is bounded relative to the product of the two
// operands' largest entries (28 x 2^-56 at most, about 2^-56 to 2^-54 rms), not to the result.  Shared by the variance kernel (diag_fx.cu) and the Schur complements
// (factor.cu).
#pragma once
#include <cuda_fp16.h>

#include <cstdint>

#include "tcgen05.cuh"

namespace spi {
namespace {

constexpr int kDig = 7;                            // digits of an operand, levels of a product
constexpr unsigned long long kDigBias = 0x0080808080808080ULL;

// Shared-memory matrix descriptor: K-major, no swizzle, 128 bytes between the core
// matrices (8 rows x 16 bytes) of a K step, `sbo` bytes between 8-row groups.
__device__ __forceinline__ uint64_t fx_desc(uint32_t saddr, uint32_t sbo) {
    return (uint64_t)((saddr & 0x3FFFF) >> 4) | ((uint64_t)(128 >> 4) << 16) | ((uint64_t)(sbo >> 4) << 32) |
           ((uint64_t)1 << 46);
}
__device__ __forceinline__ void fx_mma(uint32_t tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}"
                 :: "r"(tmem), "l"(a), "l"(b), "r"(idesc), "r"(acc));
}
__device__ __forceinline__ void fx_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                 :: "r"(tc_smem_u32(bar)));
}
// 8 accumulator columns of 16 lanes (no wait): lane l of the warp receives columns
// 2 (l % 4), 2 (l % 4) + 1 of rows l / 4 (r[0], r[1]) and l / 4 + 8 (r[2], r[3]), so that a
// warp's accesses to the rows of Z take whole 64-byte segments.
__device__ __forceinline__ void fx_ld16x8(uint32_t taddr, uint32_t (&r)[4]) {
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x1.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(taddr));
}

__device__ __forceinline__ int fx_exp(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }

// The biased exponent of v, far below any other for zero (subnormal values count as zero).
__device__ __forceinline__ int fx_scaled_exp(double v) {
    const int e = fx_exp(v);
    return e ? e : -1000000;
}
// The same, kFxNonFinite for an infinity or NaN: an exponent sum above kFxNonFinite / 2 marks
// a product with such a factor.
constexpr int kFxNonFinite = 1 << 20;
__device__ __forceinline__ int fx_scaled_exp_nf(double v) {
    const int e = fx_exp(v);
    return e == 0x7ff ? kFxNonFinite : e ? e : -1000000;
}
// v on the grid 2^(E - 1022 - 55) (v's own exponent e <= E): rounded to an integer below
// 2^55 in magnitude, plus kDigBias.  The mantissa, three bits up, is shifted right by E - e;
// the last bit is rounded off after the bias (and the sign) have been added.
__device__ __forceinline__ unsigned long long fx_fix(double v, int e, int E) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const unsigned long long mant = ((b & 0x000FFFFFFFFFFFFFULL) | 0x0010000000000000ULL) << 3;
    const unsigned long long x = mant >> min(E - e, 63);
    const unsigned long long sg = (unsigned long long)((long long)b >> 63);
    return ((x ^ sg) - sg + (2ULL * kDigBias + 1ULL)) >> 1;
}

// Digit plane q (0 = most significant) of two fixed-point values (with kDigBias added:
// each byte is a digit + 128, the seventh byte 0 .. 256) as a pair of FP16 integers.
template <int kQ>
__device__ __forceinline__ uint32_t fx_digit2(unsigned long long a, unsigned long long b) {
    const uint32_t al = (uint32_t)a, ah = (uint32_t)(a >> 32);
    const uint32_t bl = (uint32_t)b, bh = (uint32_t)(b >> 32);
    uint32_t t;
    if constexpr (kQ == 0) t = (__byte_perm(ah, bh, 0x7632) & 0x01FF01FFu) | 0x64006400u;
    else if constexpr (kQ == 1) t = (__byte_perm(ah, bh, 0x5511) & 0x00FF00FFu) | 0x64006400u;
    else if constexpr (kQ == 2) t = (__byte_perm(ah, bh, 0x4400) & 0x00FF00FFu) | 0x64006400u;
    else if constexpr (kQ == 3) t = (__byte_perm(al, bl, 0x7733) & 0x00FF00FFu) | 0x64006400u;
    else if constexpr (kQ == 4) t = (__byte_perm(al, bl, 0x6622) & 0x00FF00FFu) | 0x64006400u;
    else if constexpr (kQ == 5) t = (__byte_perm(al, bl, 0x5511) & 0x00FF00FFu) | 0x64006400u;
    else t = (__byte_perm(al, bl, 0x4400) & 0x00FF00FFu) | 0x64006400u;
    // 0x6400 + u is 1024 + u in FP16; minus 1152 leaves the digit
    const __half2 r = __hsub2(*reinterpret_cast<const __half2*>(&t), __half2half2(__ushort_as_half(0x6480)));
    return *reinterpret_cast<const uint32_t*>(&r);
}
// The digits of eight fixed-point values (consecutive in K) into the seven planes, 16 bytes each.
template <int kQ>
__device__ __forceinline__ void fx_store_planes(unsigned char* dst, size_t plane, const unsigned long long (&x)[8]) {
    if constexpr (kQ < kDig) {
        uint4 u;
        u.x = fx_digit2<kQ>(x[0], x[1]);
        u.y = fx_digit2<kQ>(x[2], x[3]);
        u.z = fx_digit2<kQ>(x[4], x[5]);
        u.w = fx_digit2<kQ>(x[6], x[7]);
        *reinterpret_cast<uint4*>(dst + kQ * plane) = u;
        fx_store_planes<kQ + 1>(dst, plane, x);
    }
}

// The digits of four values into the planes, 8 bytes each.
template <int kQ>
__device__ __forceinline__ void fx_store_planes4(unsigned char* dst, size_t plane, const unsigned long long (&x)[4]) {
    if constexpr (kQ < kDig) {
        uint2 u;
        u.x = fx_digit2<kQ>(x[0], x[1]);
        u.y = fx_digit2<kQ>(x[2], x[3]);
        *reinterpret_cast<uint2*>(dst + kQ * plane) = u;
        fx_store_planes4<kQ + 1>(dst, plane, x);
    }
}

// The seven level sums of one output (integers, exact in FP32; level l weighs
// 2^-(14 + 8 l)) as one integer in units of 2^-55: levels 0-3 fit two 32-bit words, levels
// 4-6 are shifted down by 7 bits, the last with rounding.
// An FP32 integer of at most 2^22 in magnitude becomes a two's-complement one by adding
// 1.5 2^23 (the sum's low bits; FP32 additions run at eight times the rate of the
// conversion instruction): levels 0 and 1, and level 6 after its shift.
__device__ __forceinline__ long long fx_join(const uint32_t (&t)[kDig]) {
    constexpr float kMagic = 12582912.0f;
    constexpr int kBits = 0x4B400000;
    const int i0 = __float_as_int(__uint_as_float(t[0]) + kMagic) - kBits;
    const int i1 = __float_as_int(__uint_as_float(t[1]) + kMagic) - kBits;
    const int i6 = __float_as_int(fmaf(__uint_as_float(t[6]), 0.0078125f, kMagic)) - kBits;
    const int i2 = __float2int_rn(__uint_as_float(t[2])), i3 = __float2int_rn(__uint_as_float(t[3]));
    const int i4 = __float2int_rn(__uint_as_float(t[4])), i5 = __float2int_rn(__uint_as_float(t[5]));
    const int p01 = i0 * 256 + i1, p23 = i2 * 256 + i3, p56 = i5 * 2 + i6;
    return (long long)i4 * 512 + p56 + (long long)p23 * (1 << 17) + ((long long)p01 << 33);
}
// The same when every level sum is at most 2^22 (up to 32 products): all levels by the
// addition, the sums of levels 4-6 in 32 bits, the constants folded (modulo 2^32).
__device__ __forceinline__ long long fx_join_small(const uint32_t (&t)[kDig]) {
    constexpr float kMagic = 12582912.0f;
    constexpr uint32_t kBits = 0x4B400000u;
    uint32_t i[kDig];
#pragma unroll
    for (int l = 0; l < kDig - 1; ++l) i[l] = __float_as_uint(__uint_as_float(t[l]) + kMagic);
    i[6] = __float_as_uint(fmaf(__uint_as_float(t[6]), 0.0078125f, kMagic));
    const int p01 = (int)(i[0] * 256u + i[1] - kBits * 257u), p23 = (int)(i[2] * 256u + i[3] - kBits * 257u);
    const int p456 = (int)(i[4] * 512u + i[5] * 2u + i[6] - kBits * 515u);
    return (long long)p456 + (long long)p23 * (1 << 17) + ((long long)p01 << 33);
}
// v 2^(e - 55) rounded to FP64 (e the sum of the row's and the column's exponents).
__device__ __forceinline__ double fx_value(long long v, int e) {
    const unsigned long long sg = (unsigned long long)(v >> 63);
    const unsigned long long u = ((unsigned long long)v ^ sg) - sg;
    const int lz = __clzll((long long)u);
    const unsigned long long r = ((u << (lz - 1)) + 0x200ULL) >> 10;  // leading bit at 52 (a carry raises the exponent)
    const int ex = 1023 + 63 - 55 + e - lz;  // biased exponent of the leading bit
    if (u == 0 || ex <= 0) return 0.0;
    if (ex > 2046) return __longlong_as_double((long long)((sg & 0x8000000000000000ULL) | 0x7ff0000000000000ULL));
    const unsigned long long bits = r + ((unsigned long long)(uint32_t)(ex - 1) << 52);
    return __longlong_as_double((long long)(bits | (sg & 0x8000000000000000ULL)));
}

// The exponent of s, the power of two next to sqrt(d), and 2^e.
__device__ __forceinline__ int fx_scale_exp(double d) { return (fx_exp(d) - 1023) >> 1; }
__device__ __forceinline__ double fx_pow2(int e) { return __hiloint2double((1023 + e) << 20, 0); }

}  // namespace
}  // namespace spi
