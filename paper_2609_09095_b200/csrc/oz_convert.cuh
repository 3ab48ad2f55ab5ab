// Conversion of FP64 elements into plane bytes (Algorithm 2): the quantised integer in four balanced FP32 limbs,
// residues of every modulus from packed multiply-adds on them, digits by one more rounded division (odd squares) or
// from a small table (powers of two and non-squares).  Shared by the deconstruction kernels and by the product
// kernel that converts its A operand on the fly.
// Internal to liboz_b200.so; every function is device-inline and lives in the including file's
// anonymous namespace.
#pragma once

#include <utility>

#include "oz_internal.h"

namespace oz {
namespace {

// Eq. 1 for one element, integer form (any sigma): a' = quant(x 2^sigma) as a 64-bit integer.  While 2^sigma is a normal
// double, split_limbs() multiplies by it instead: exact in FP64 (a product that underflows is far below 1/2 and rounds to
// zero either way), and the hardware conversion rounds to nearest-even or toward zero.
__device__ __noinline__ long long quantise(double x, int sigma, bool tz)
{
    unsigned long long bits = static_cast<unsigned long long>(__double_as_longlong(x));
    int be = static_cast<int>((bits >> 52) & 0x7FF);
    unsigned long long frac = bits & 0xFFFFFFFFFFFFFull;
    unsigned long long sig = be ? (frac | (1ull << 52)) : frac;
    int ex = be ? be - 1023 : -1022;
    int sh = 52 - ex - sigma;                       // |x| 2^sigma = sig / 2^sh
    unsigned long long q;
    if (sh <= 0) {
        q = sig << (sh < -63 ? 63 : -sh);
    } else {
        if (sh > 63) sh = 63;                       // sig < 2^53: anything past 54 rounds to zero
        if (tz) q = sig >> sh;
        else q = (sig + ((1ull << (sh - 1)) - 1ull) + ((sig >> sh) & 1ull)) >> sh;  // ties to even
    }
    return (bits >> 63) ? -static_cast<long long>(q) : static_cast<long long>(q);
}

// ---- residues in FP32 ---------------------------------------------------------------------------
// The quantised integer is cut into four BALANCED limbs at bits 0, 16, 31 and 45 (16, 15, 14 bits and
// the signed rest), each held exactly in FP32, and
//     v = l0 + c1 l1 + c2 l2 + c3 l3,   c_q = 2^(bit q) mod m, balanced,
// is an integer below 2^24 in magnitude: three fused multiply-adds, exact.  rint(v / m) comes from a
// multiplication by the rounded reciprocal and the 1.5 * 2^23 constant, one more multiply-add leaves the
// balanced residue r.  The quotient is the nearest integer as long as |v| |m inv - 1| < 1/2 (v / m is never
// closer than 1 / (2m) to a half-integer for odd m), which residue_exact() checks for every modulus.
// Every instruction works on a packed pair of elements: six for two residues, where 16-bit integer limbs
// take seven for one.  What bounds the conversion is instruction issue (and the look-ups' shared-memory
// wavefronts), so both the packed arithmetic and the digits of the odd squares, which need no table,
// come straight off its time: 204 -> 146 thread-instructions per element of A on set S, 190 -> 137 of B.
constexpr int kLimbBit1 = 16, kLimbBit2 = 31, kLimbBit3 = 45;
// Largest |a'|, as 2^q, of an element whose product does not vanish: CS and MAXEXP stay below sqrt(M/2); the
// accurate rule reaches sqrt(32) 2^(L/2) with L = floor(log2 of its budget) = 110, 112, 116.  (Elements
// that only meet zeros may be larger under the accurate rule; their residues then are arbitrary but
// bounded, see kLutGuard.)
__host__ __device__ constexpr double max_operand(int set)
{
    constexpr double sqrt_half = 0.7071067811865476;
    return sqrt_half * (set == 0 ? 0x1p58 : (set == 1 ? 0x1p59 : 0x1p61));
}
__host__ __device__ constexpr float inv_of(uint32_t m) { return 1.0f / static_cast<float>(m); }
__host__ __device__ constexpr int balanced_pow2(int e, uint32_t m)
{
    const int v = static_cast<int>(pow2_mod(e, m));
    return 2 * v > static_cast<int>(m) ? v - static_cast<int>(m) : v;
}
__host__ __device__ constexpr double abs_d(double x) { return x < 0 ? -x : x; }
__host__ __device__ constexpr bool residue_exact(int set, uint32_t m)
{
    const double v = 32768.0 + 16384.0 * abs_d(balanced_pow2(kLimbBit1, m)) + 8192.0 * abs_d(balanced_pow2(kLimbBit2, m)) +
                     (max_operand(set) * 0x1p-45 + 1.0) * abs_d(balanced_pow2(kLimbBit3, m));
    const double delta = abs_d(static_cast<double>(inv_of(m)) * m - 1.0);
    return v < 16777216.0 && v * delta < 0.5;
}

constexpr float kRintF = 12582912.0f;        // 1.5 * 2^23: the low mantissa bits of x + kRintF hold rint(x)

// NP pairs of consecutive elements: pair q holds elements 2q and 2q + 1
template <int NP>
struct Limbs {
    float2 l0[NP], l1[NP], l2[NP], l3[NP];
    uint32_t low[2 * NP];                    // bits 0..14 are those of a' (the power-of-two moduli)
};

// limbs of one quantised value
__device__ __forceinline__ void limb_fields(long long a, float &f0, float &f1, float &f2, float &f3, uint32_t &low)
{
    constexpr unsigned long long kBias = (1ull << 15) + (1ull << 30) + (1ull << 44) + (1ull << 63);
    const unsigned long long p = static_cast<unsigned long long>(a) + kBias;
    const uint32_t lo = static_cast<uint32_t>(p), hi = static_cast<uint32_t>(p >> 32);
    // a field OR 2^23's exponent is the float 2^23 + field
    low = __byte_perm(lo, 0x4B000000u, 0x7610);
    f0 = __uint_as_float(low);
    f1 = __uint_as_float(((lo >> 16) & 0x7FFFu) | 0x4B000000u);
    f2 = __uint_as_float((__funnelshift_r(lo, hi, 31) & 0x3FFFu) | 0x4B000000u);
    f3 = __uint_as_float((hi >> 13) | 0x4B000000u);
}

template <int NP>
__device__ __forceinline__ void limb_pair(long long a0, long long a1, int q, Limbs<NP> &L)
{
    constexpr float k23 = 8388608.0f;
    float f0[2], f1[2], f2[2], f3[2];
    limb_fields(a0, f0[0], f1[0], f2[0], f3[0], L.low[2 * q]);
    limb_fields(a1, f0[1], f1[1], f2[1], f3[1], L.low[2 * q + 1]);
    L.l0[q] = __fadd2_rn(make_float2(f0[0], f0[1]), make_float2(-(k23 + 32768.0f), -(k23 + 32768.0f)));
    L.l1[q] = __fadd2_rn(make_float2(f1[0], f1[1]), make_float2(-(k23 + 16384.0f), -(k23 + 16384.0f)));
    L.l2[q] = __fadd2_rn(make_float2(f2[0], f2[1]), make_float2(-(k23 + 8192.0f), -(k23 + 8192.0f)));
    L.l3[q] = __fadd2_rn(make_float2(f3[0], f3[1]), make_float2(-(k23 + 262144.0f), -(k23 + 262144.0f)));
}

// limbs of the quantised values of 2 NP elements
template <int NP>
__device__ __forceinline__ void split_limbs(const double (&x)[2 * NP], int sigma, bool tz, Limbs<NP> &L)
{
    if (sigma >= -1000 && sigma <= 1000) {       // 2^sigma is a normal number: always, except for lines of (nearly) subnormals; no sigma is below -979
        const double scale = __hiloint2double((1023 + sigma) << 20, 0);
        if (!tz) {
#pragma unroll
            for (int q = 0; q < NP; ++q) limb_pair(__double2ll_rn(x[2 * q] * scale), __double2ll_rn(x[2 * q + 1] * scale), q, L);
        } else {
#pragma unroll
            for (int q = 0; q < NP; ++q) limb_pair(__double2ll_rz(x[2 * q] * scale), __double2ll_rz(x[2 * q + 1] * scale), q, L);
        }
    } else if constexpr (NP == 2) {
        // Four elements a thread (the product kernel, whose tiles wait for their slowest row): sigma > 1000, the line holds numbers
        // below 2^-880 only, which 2^1000 lifts into the normal range without rounding.  (3000 x 100 x 1500 in storage mode F with three
        // such rows, set E: 385 us a call with the integer form, 354 with two multiplications; with eight or sixteen elements a thread
        // they cost the other lines registers that spill.)
        const double scale = __hiloint2double((1023 + sigma - 1000) << 20, 0);
        auto lifted = [&](double v) {
            const double y = v * 0x1p1000 * scale;
            return tz ? __double2ll_rz(y) : __double2ll_rn(y);
        };
#pragma unroll
        for (int q = 0; q < NP; ++q) limb_pair(lifted(x[2 * q]), lifted(x[2 * q + 1]), q, L);
    } else {
#pragma unroll
        for (int q = 0; q < NP; ++q) limb_pair(quantise(x[2 * q], sigma, tz), quantise(x[2 * q + 1], sigma, tz), q, L);
    }
}

__device__ __forceinline__ float2 dup(float x) { return make_float2(x, x); }

// balanced residues of a pair
template <int SET, int I, int NP>
__device__ __forceinline__ float2 residue_pair(const Limbs<NP> &L, int q)
{
    constexpr uint32_t m = modulus(SET, I);
    static_assert(residue_exact(SET, m), "exact limb sum and quotient");
    constexpr float c1 = balanced_pow2(kLimbBit1, m), c2 = balanced_pow2(kLimbBit2, m), c3 = balanced_pow2(kLimbBit3, m);
    float2 v = __ffma2_rn(L.l1[q], dup(c1), L.l0[q]);
    v = __ffma2_rn(L.l2[q], dup(c2), v);
    v = __ffma2_rn(L.l3[q], dup(c3), v);
    const float2 quot = __fadd2_rn(__ffma2_rn(v, dup(inv_of(m)), dup(kRintF)), dup(-kRintF));
    return __ffma2_rn(quot, dup(-static_cast<float>(m)), v);
}

// One word of the table, which is written once, before a block barrier.  Free to move otherwise: the caller's address has
// to depend on something that is read behind that barrier (elements from shared memory, or the table's own address).
__device__ __forceinline__ uint32_t lds_u32(uint32_t addr)
{
    uint32_t v;
    asm("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}

// The table in shared memory.  A look-up's byte offset comes out of FP32 arithmetic as the bit pattern of a denormal, exact while
// those bits stay below 2^24.  Near: the table's address is part of that sum.  Far: in a cluster a block's shared addresses carry its
// rank above bit 24, so the address is added to the offset as an integer.
struct NearTable {
    uint32_t addr;
    __device__ __forceinline__ float base(uint32_t words) const { return __uint_as_float(addr + 4 * words); }
    __device__ __forceinline__ uint32_t at(uint32_t bits) const { return lds_u32(bits); }
    __device__ __forceinline__ uint32_t word(uint32_t i) const { return lds_u32(addr + 4 * i); }
};
struct FarTable {
    uint32_t addr;
    __device__ __forceinline__ float base(uint32_t words) const { return __uint_as_float(4 * words); }
    __device__ __forceinline__ uint32_t at(uint32_t bits) const { return lds_u32(addr + bits); }
    __device__ __forceinline__ uint32_t word(uint32_t i) const { return lds_u32(addr + 4 * i); }
};

// two E4M3 bytes (x in the low one); every digit is representable, so nothing is rounded
__device__ __forceinline__ uint32_t e4m3_pair(float2 d)
{
    uint16_t h;
    asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(h) : "f"(d.y), "f"(d.x));
    return h;
}

// four values whose low bytes are wanted -> one word
__device__ __forceinline__ uint32_t pack_low_bytes(uint32_t a, uint32_t b, uint32_t c, uint32_t d)
{
    return __byte_perm(__byte_perm(a, b, 0x0040), __byte_perm(c, d, 0x0040), 0x5410);
}

template <int N>
__device__ __forceinline__ void store_words(uint8_t *out, const uint32_t (&w)[N])
{
    if constexpr (N == 4) *reinterpret_cast<uint4 *>(out) = make_uint4(w[0], w[1], w[2], w[3]);
    else if constexpr (N == 2) *reinterpret_cast<uint2 *>(out) = make_uint2(w[0], w[1]);
    else *reinterpret_cast<uint32_t *>(out) = w[0];
}

// Digits of four integer-valued numbers to base BASE, both rounded: d1 = rint(r / BASE), d0 = r - BASE d1
template <int BASE, bool E4M3>
__device__ __forceinline__ void digit_words(const float2 (&r)[2], uint32_t &w0, uint32_t &w1)
{
    float2 d0[2], d1[2], t1[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        t1[h] = __ffma2_rn(r[h], dup(inv_of(BASE)), dup(kRintF));
        d1[h] = __fadd2_rn(t1[h], dup(-kRintF));
        d0[h] = __ffma2_rn(d1[h], dup(-static_cast<float>(BASE)), r[h]);
    }
    if constexpr (E4M3) {
        w0 = e4m3_pair(d0[0]) | (e4m3_pair(d0[1]) << 16);
        w1 = e4m3_pair(d1[0]) | (e4m3_pair(d1[1]) << 16);
    } else {
        const float2 u0 = __fadd2_rn(d0[0], dup(kRintF)), u1 = __fadd2_rn(d0[1], dup(kRintF));
        w0 = pack_low_bytes(__float_as_uint(u0.x), __float_as_uint(u0.y), __float_as_uint(u1.x), __float_as_uint(u1.y));
        w1 = pack_low_bytes(__float_as_uint(t1[0].x), __float_as_uint(t1[0].y), __float_as_uint(t1[1].x), __float_as_uint(t1[1].y));
    }
}

// One modulus (compile-time index I of set SET) for 2 NP consecutive inner-dimension elements: residues,
// digits, and 1, 2 or 3 plane stores of 2 NP bytes.  Digits come from the table for the power-of-two and the
// non-square moduli (Lemma 1's carry makes the latter irregular) and from one more rounded division for the
// odd squares.  lut: the set's table.
template <int SET, int LAYOUT, int I, int NP, class Table>
__device__ __forceinline__ void convert_modulus(const Limbs<NP> &L, const Table &lut, uint8_t *out, int64_t plane_stride)
{
    static_assert(NP % 2 == 0, "whole words");
    constexpr uint32_t m = modulus(SET, I);
    constexpr int plane = first_plane(SET, I, LAYOUT);
    constexpr bool pow2 = (m & (m - 1)) == 0;
    constexpr int s = square_root(m);
    constexpr int NW = NP / 2;                       // plane words
    constexpr bool e4m3 = LAYOUT == kLayoutDigits || LAYOUT == kLayoutMerged || LAYOUT == kLayoutTwo || LAYOUT == kLayoutFour;   // else INT8
    if constexpr (LAYOUT == kLayoutNative) {         // one plane: the centred residue itself
        uint32_t w[NW];
#pragma unroll
        for (int g = 0; g < NW; ++g) {
            if constexpr (pow2) {
                static_assert(!pow2 || m == 256, "the low byte of a' is its centred residue modulo 256");
                w[g] = pack_low_bytes(L.low[4 * g], L.low[4 * g + 1], L.low[4 * g + 2], L.low[4 * g + 3]);
            } else {
                const float2 r0 = __fadd2_rn(residue_pair<SET, I>(L, 2 * g), dup(kRintF));
                const float2 r1 = __fadd2_rn(residue_pair<SET, I>(L, 2 * g + 1), dup(kRintF));
                w[g] = pack_low_bytes(__float_as_uint(r0.x), __float_as_uint(r0.y), __float_as_uint(r1.x), __float_as_uint(r1.y));
            }
        }
        store_words(out + plane * plane_stride, w);
    } else if constexpr (two_plane_layout(LAYOUT)) {
        // no table: 121 thread-instructions per element of A on set S where three planes take 127 and conflicting look-ups
        constexpr bool four = s == 0 && (LAYOUT == kLayoutFour || LAYOUT == kLayoutFourI8);
        constexpr int base = s ? s : 16;
        uint32_t w[4][NW];
#pragma unroll
        for (int g = 0; g < NW; ++g) {
            float2 r[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if constexpr (pow2) {        // the lowest limb carries the residue
                    const float2 l = L.l0[2 * g + h];
                    const float2 quot = __fadd2_rn(__ffma2_rn(l, dup(inv_of(m)), dup(kRintF)), dup(-kRintF));
                    r[h] = __ffma2_rn(quot, dup(-static_cast<float>(m)), l);
                } else {
                    r[h] = residue_pair<SET, I>(L, 2 * g + h);
                }
            }
            digit_words<base, e4m3>(r, w[0][g], w[1][g]);
            if constexpr (four) {            // f = 16 e mod m, balanced
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float2 quot = __fadd2_rn(__ffma2_rn(r[h], dup(16.0f * inv_of(m)), dup(kRintF)), dup(-kRintF));
                    r[h] = __ffma2_rn(quot, dup(-static_cast<float>(m)), __fmul2_rn(r[h], dup(16.0f)));
                }
                digit_words<base, e4m3>(r, w[2][g], w[3][g]);
            }
        }
#pragma unroll
        for (int d = 0; d < (four ? 4 : 2); ++d) store_words(out + (plane + d) * plane_stride, w[d]);
    } else if constexpr (s != 0 && !pow2) {
        // odd square: both digits balanced and free of ties
        uint32_t w0[NW], w1[NW];
#pragma unroll
        for (int g = 0; g < NW; ++g) {
            const float2 r[2] = {residue_pair<SET, I>(L, 2 * g), residue_pair<SET, I>(L, 2 * g + 1)};
            digit_words<s, e4m3>(r, w0[g], w1[g]);
        }
        store_words(out + plane * plane_stride, w0);
        store_words(out + (plane + 1) * plane_stride, w1);
    } else {
        // table word: byte 0 = d0, 1 = d1, 2 = d0+d1, 3 = the byte the merged layouts swap in (FP8: the pre-scaled
        // -16*d1 for d1; INT8: -d0 for d0, with 4*d1 made by a byte-wise shift)
        uint32_t w0[NW], w1[NW], w2[NW];
#pragma unroll
        for (int g = 0; g < NW; ++g) {
            uint32_t t[4];
            if constexpr (pow2) {
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    t[e] = lut.word(lut_offset(SET, I) + (L.low[4 * g + e] & (m - 1)));
            } else {
                // byte offset 4 (r + bias) as the bits of a denormal: one multiply-add, no conversion
                constexpr int bias = static_cast<int>(m / 2) + kLutGuard;
                const float2 base = dup(lut.base(lut_offset(SET, I) + bias));
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float2 a = __ffma2_rn(residue_pair<SET, I>(L, 2 * g + h), dup(0x1p-147f), base);
                    t[2 * h] = lut.at(__float_as_uint(a.x));
                    t[2 * h + 1] = lut.at(__float_as_uint(a.y));
                }
            }
            const uint32_t t01 = __byte_perm(t[0], t[1], 0x5140), t23 = __byte_perm(t[2], t[3], 0x5140);
            const uint32_t first = __byte_perm(t01, t23, 0x5410), second = __byte_perm(t01, t23, 0x7632);
            const uint32_t u01 = __byte_perm(t[0], t[1], 0x7362), u23 = __byte_perm(t[2], t[3], 0x7362);
            const uint32_t extra = __byte_perm(u01, u23, 0x7632);
            constexpr bool kI8 = s == 0 && (LAYOUT == kLayoutMergedI8A || LAYOUT == kLayoutMergedI8B);
            w0[g] = s == 0 && LAYOUT == kLayoutMergedI8A ? extra : first;
            w1[g] = s == 0 && LAYOUT == kLayoutMerged ? extra : (kI8 ? ((second << 2) & 0xFCFCFCFCu) : second);
            w2[g] = __byte_perm(u01, u23, 0x5410);
        }
        store_words(out + plane * plane_stride, w0);
        store_words(out + (plane + 1) * plane_stride, w1);
        if constexpr (s == 0) store_words(out + (plane + 2) * plane_stride, w2);
    }
}

template <int SET, int LAYOUT, int NP, class Table, int... I>
__device__ __forceinline__ void convert_all_moduli(std::integer_sequence<int, I...>, const Limbs<NP> &L, const Table &lut,
                                                   uint8_t *out, int64_t plane_stride)
{
    (convert_modulus<SET, LAYOUT, I>(L, lut, out, plane_stride), ...);
}

}  // namespace
}  // namespace oz
