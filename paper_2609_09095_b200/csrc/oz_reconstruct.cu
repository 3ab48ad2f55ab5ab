// Reconstruction (Algorithm 3; Eq. 4-5 and the last step of Sec. 2 (iv)): residues -> the integer
// c' in [-M/2, M/2), unscaled by 2^-(sigma_i + tau_j) and rounded once to FP64.
//
// The paper's SIMT branch walks Garner's mixed-radix digits (r(r-1)/2 multiply-reduce steps).
// CRT fixes c' uniquely, so any exact evaluation gives the same integer; this kernel uses the
// weighted form over groups of moduli.  With P_g the product of the two or three moduli of group g,
//     c' = sum_g u_g N_g  -  kappa M,     N_g = M / P_g,     u_g = sum_{i in g} c_i a_i,
// where a_i is 0 modulo the other moduli of its group and (N_g)^-1 modulo m_i, balanced: u_g is a 32-bit integer that two or
// three integer multiply-adds form from the stored residues, and one conversion serves the whole group.  Every N_g and M is cut
// into a high and a middle part of at most 21 signed bits and the rest: the sums of the first two are integers below 2^53
// (group_bounds()) and formed EXACTLY by FP64 fused multiply-adds, that of the third is off by less than kRestError.
// kappa = round(S/M) comes from a floating estimate; error-free additions then give the correctly rounded FP64 value unless
// c' lies within kRestError of a rounding boundary, is so small that this error counts, or lies near +-M/2.  The first two kinds are settled
// from c' modulo 2^64 (settle_rows()); for the last, an exact path: the 128-bit integer, an exact range test for the lift to [-M/2, M/2), and one
// round-to-nearest-even done in integer arithmetic.  A term for every modulus, three parts of 38 or 40 bits each, took 36 (S) to 45 (A)
// FP64 multiply-adds and 12 to 15 conversions an output where this takes 18 and 6 (A: 15 and 5).
// A thread handles four rows of a column, two where the outputs are few.
#include <utility>

#include "oz_internal.h"

namespace oz {
namespace {

// ---- groups of moduli -----------------------------------------------------------------------------
constexpr int kMaxGroups = 6;
__host__ __device__ constexpr int set_groups(int set) { return set == 2 ? 5 : 6; }
// Moduli of a group (indices, -1: none): those that keep the sum of the bounds of |u_g| small, so that the rest's error is small.
__host__ __device__ constexpr int group_member(int set, int g, int e)
{
    constexpr int S[6][3] = {{5, 9, -1}, {3, 4, -1}, {7, 10, -1}, {1, 2, -1}, {0, 6, -1}, {8, 11, -1}};
    constexpr int E[6][3] = {{7, 11, 12}, {5, 8, -1}, {4, 9, -1}, {0, 6, -1}, {1, 3, -1}, {2, 10, -1}};
    constexpr int A[6][3] = {{1, 9, 11}, {6, 7, 12}, {0, 3, 4}, {2, 5, 8}, {10, 13, 14}, {-1, -1, -1}};
    return set == 0 ? S[g][e] : set == 1 ? E[g][e] : A[g][e];
}
// places of the middle and of the high part
__host__ __device__ constexpr int mid_bit(int set) { return set == 0 ? 52 : set == 1 ? 55 : 54; }
__host__ __device__ constexpr int high_bit(int set) { return mid_bit(set) + 21; }

struct Wide { uint64_t lo, hi; };                 // 128-bit constants at compile time
__host__ __device__ constexpr Wide wide_mul(Wide w, uint64_t m)      // m below 2^31, no overflow
{
    const uint64_t p0 = (w.lo & 0xFFFFFFFFull) * m, p1 = (w.lo >> 32) * m + (p0 >> 32);
    return {(p0 & 0xFFFFFFFFull) | (p1 << 32), w.hi * m + (p1 >> 32)};
}
__host__ __device__ constexpr uint64_t group_product(int set, int g)
{
    uint64_t p = 1;
    for (int e = 0; e < 3; ++e)
        if (group_member(set, g, e) >= 0) p *= static_cast<uint64_t>(modulus(set, group_member(set, g, e)));
    return p;
}
__host__ __device__ constexpr bool in_group(int set, int g, int i)
{
    return group_member(set, g, 0) == i || group_member(set, g, 1) == i || group_member(set, g, 2) == i;
}
// N_g; g = -1: M
__host__ __device__ constexpr Wide group_weight(int set, int g)
{
    Wide w{1, 0};
    for (int i = 0; i < set_r(set); ++i)
        if (g < 0 || !in_group(set, g, i)) w = wide_mul(w, static_cast<uint64_t>(modulus(set, i)));
    return w;
}
// N = high 2^high_bit + mid 2^mid_bit + rest, the last two balanced
struct Parts { int64_t high, mid, rest; };
__host__ __device__ constexpr Parts split_parts(int set, Wide w)
{
    const int b = mid_bit(set), c = high_bit(set) - b;
    Parts p{};
    p.rest = static_cast<int64_t>(w.lo & ((1ull << b) - 1));
    uint64_t up = (w.lo >> b) | (w.hi << (64 - b));
    if (p.rest >> (b - 1)) { p.rest -= 1ll << b; ++up; }
    p.mid = static_cast<int64_t>(up & ((1ull << c) - 1));
    up >>= c;
    if (p.mid >> (c - 1)) { p.mid -= 1ll << c; ++up; }
    p.high = static_cast<int64_t>(up);
    return p;
}
// a_i of member e of group g
__host__ __device__ constexpr int64_t member_weight(int set, int g, int e)
{
    const int i = group_member(set, g, e);
    if (i < 0) return 0;
    const uint64_t m = static_cast<uint64_t>(modulus(set, i)), P = group_product(set, g);
    uint64_t other = 1;                              // M / m_i modulo m_i
    for (int j = 0; j < set_r(set); ++j)
        if (j != i) other = other * static_cast<uint64_t>(modulus(set, j)) % m;
    uint64_t inv = 1;
    while (other * inv % m != 1) ++inv;
    const uint64_t a = P / m * inv % P;
    return 2 * a > P ? static_cast<int64_t>(a) - static_cast<int64_t>(P) : static_cast<int64_t>(a);
}
// Largest number that stands for a residue: all that a form can hold; two bytes, as everything in the public layout of sets S and E: below 2 m,
// but for the groups of three, whose sums would leave 32 bits: there the public layout's numbers are reduced first.
__host__ __device__ constexpr bool reduced_first(int set, int i)
{
    bool three = false;
    for (int g = 0; g < set_groups(set); ++g) three = three || (in_group(set, g, i) && group_member(set, g, 2) >= 0);
    return set != 2 && three;
}
__host__ __device__ constexpr int64_t largest_number(int set, int i)
{
    const int64_t form = stored_form(set, i) == kStoredByte ? 255 : stored_form(set, i) == kStoredTen ? 1023 : 0, twice = 2 * modulus(set, i) - 1;
    return set == 2 || reduced_first(set, i) || form > twice ? form : twice;
}
__host__ __device__ constexpr int64_t abs64(int64_t x) { return x < 0 ? -x : x; }
// bound of |u_g|: the terms of one sign
__host__ __device__ constexpr int64_t group_reach(int set, int g)
{
    int64_t pos = 0, neg = 0;
    for (int e = 0; e < 3; ++e) {
        if (group_member(set, g, e) < 0) continue;
        const int64_t t = largest_number(set, group_member(set, g, e)) * member_weight(set, g, e);
        if (t > 0) pos += t;
        else neg -= t;
    }
    return pos > neg ? pos : neg;
}
__host__ __device__ constexpr double pow2d(int e) { double v = 1.0; for (int i = 0; i < e; ++i) v *= 2.0; return v; }
struct Bounds { double high, mid, rest, kappa; bool words; };
// of the three sums in units of their places, with kappa M taken off (which makes the high one small); every u_g in 32 bits
__host__ __device__ constexpr Bounds group_bounds(int set)
{
    Bounds b{0.0, 0.0, 0.0, 1.0, true};
    for (int g = 0; g < set_groups(set); ++g) {
        const Parts p = split_parts(set, group_weight(set, g));
        const double u = static_cast<double>(group_reach(set, g));
        b.high += u * static_cast<double>(abs64(p.high));
        b.mid += u * static_cast<double>(abs64(p.mid));
        b.rest += u * static_cast<double>(abs64(p.rest));
        b.kappa += u / static_cast<double>(group_product(set, g));
        if (u >= 2147483648.0 || abs64(p.high) >= (1ll << 21)) b.words = false;
    }
    const Parts m = split_parts(set, group_weight(set, -1));
    b.mid += b.kappa * static_cast<double>(abs64(m.mid));
    b.rest += b.kappa * static_cast<double>(abs64(m.rest));
    return b;
}
// Bound, as a power of two, of what the rest's multiply-adds (one a group and one of kappa M) and the last addition to it lose
__host__ __device__ constexpr int rest_error_log2(int set)
{
    const double e = group_bounds(set).rest * (set_groups(set) + 3) / pow2d(53);
    int l = 0;
    while (pow2d(l) < e) ++l;
    return l;
}
template <int SET> constexpr int kRestErrorLog2 = rest_error_log2(SET);
template <int SET> constexpr bool kExact = group_bounds(SET).words && group_bounds(SET).high < 9007199254740992.0 &&
                                           group_bounds(SET).mid < 9007199254740992.0 && mid_bit(SET) > kRestErrorLog2<SET> + 4;
static_assert(kExact<0> && kExact<1> && kExact<2>, "the high and middle sums are exact, every group's integer fits 32 bits");

// High words of doubles: below the first, the rest's error may reach a quarter of an ulp; from the second on (M / 2 but for its last bits),
// the lift is decided exactly.
__host__ __device__ constexpr uint32_t small_word(int set) { return static_cast<uint32_t>(1023 + rest_error_log2(set) + 56) << 20; }
__host__ __device__ constexpr uint32_t half_M_word(int set)
{
    Wide w = group_weight(set, -1);
    int bits = 128;
    while (!(w.hi >> 63)) { w.hi = (w.hi << 1) | (w.lo >> 63); w.lo <<= 1; --bits; }
    return (static_cast<uint32_t>(1023 + bits - 2) << 20 | static_cast<uint32_t>((w.hi >> 43) & 0xFFFFFu)) - 1u;
}
__host__ __device__ constexpr double inverse_M(int set)
{
    const Wide w = group_weight(set, -1);
    return 1.0 / (static_cast<double>(w.hi) * pow2d(64) + static_cast<double>(w.lo));
}

// ---- kernels ----------------------------------------------------------------------------------------
// Constants that do not fit an instruction's immediate operand (the high and middle parts do: 21 significant bits)
struct ReconConst { double rest[kMaxGroups], M_rest, inv_M; };
template <int SET>
constexpr ReconConst recon_constants()
{
    ReconConst c{};
    for (int g = 0; g < set_groups(SET); ++g) c.rest[g] = static_cast<double>(split_parts(SET, group_weight(SET, g)).rest);
    c.M_rest = static_cast<double>(split_parts(SET, group_weight(SET, -1)).rest);
    c.inv_M = inverse_M(SET);
    return c;
}
__constant__ ReconConst c_recon[kNumSets] = {recon_constants<0>(), recon_constants<1>(), recon_constants<2>()};

// Up to this many outputs two rows a thread (from 1200 x 1200 on four are faster): 512 x 512 on set S 23.7 us a call, with four rows 25.7; 700 x 700 x 300 29.3 and 30.6.
constexpr int64_t kFewOutputs = 700000;
// Public layout: blocks of 128 threads, nine an SM with two rows a thread (56 registers).  6000 x 6000 update, set E, with 8 / 9 / 10: 288 / 274 / 281 us
constexpr int kPublicThreads = 128;
constexpr double kRint = 6755399441055744.0;          // 1.5 * 2^52: (x + kRint) - kRint = rint(x)

// x * 2^scale for a finite double x (exact unless the result leaves the normal range)
__device__ __forceinline__ double scale_pow2(double x, int scale)
{
    int hi = __double2hiint(x);
    int be = (hi >> 20) & 0x7FF;
    int nb = be + scale;
    if (be != 0 && nb >= 1 && nb <= 2046) return __hiloint2double(hi + (scale << 20), __double2loint(x));
    return scalbn(x, scale);        // zero, or a result outside the normal range
}

// The numbers of a thread's rows: lo the low bytes, hi the bits above them in the same bytes (ten-bit form); two-byte form: lo the first
// two rows, hi the others
struct Numbers { uint32_t lo[kMaxR], hi[kMaxR]; };

template <uint32_t SELECT>
__device__ __forceinline__ uint32_t permute(uint32_t a, uint32_t b)
{
    uint32_t v;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(v) : "r"(a), "r"(b), "n"(SELECT));
    return v;
}

// number of modulus I in row H of the thread
template <int SET, bool PRIVATE, int H, int I>
__device__ __forceinline__ uint32_t number(const Numbers &w)
{
    constexpr int form = PRIVATE || residue_bytes(SET) == 1 ? stored_form(SET, I) : static_cast<int>(kStoredPair);
    if constexpr (form == kStoredByte) {
        return permute<0x4440u + H>(w.lo[I], 0u);
    } else if constexpr (form == kStoredTen) {
        return permute<0xCC40u + 0x1111u * H>(w.lo[I], w.hi[I]);              // above the two bytes: the sign of one below 4
    } else {
        const uint32_t c = permute<(H & 1) ? 0x4432u : 0x4410u>(H < 2 ? w.lo[I] : w.hi[I], 0u);
        return !PRIVATE && reduced_first(SET, I) ? min(c, c - static_cast<uint32_t>(modulus(SET, I))) : c;
    }
}

template <int SET, bool PRIVATE, int H, int G>
__device__ __forceinline__ int group_value(const Numbers &w)
{
    constexpr int i0 = group_member(SET, G, 0), i1 = group_member(SET, G, 1), i2 = group_member(SET, G, 2);
    constexpr uint32_t a0 = static_cast<uint32_t>(member_weight(SET, G, 0)), a1 = static_cast<uint32_t>(member_weight(SET, G, 1)),
                       a2 = static_cast<uint32_t>(member_weight(SET, G, 2));
    uint32_t u = number<SET, PRIVATE, H, i0>(w) * a0;
    u = number<SET, PRIVATE, H, i1>(w) * a1 + u;
    if constexpr (i2 >= 0) u = number<SET, PRIVATE, H, i2>(w) * a2 + u;
    return static_cast<int>(u);
}

template <int SET, bool PRIVATE, int H, int G>
__device__ __forceinline__ void crt_term(const Numbers &w, double &X0, double &X1, double &X2)
{
    constexpr Parts p = split_parts(SET, group_weight(SET, G));
    constexpr double high = static_cast<double>(p.high) * pow2d(high_bit(SET)), mid = static_cast<double>(p.mid) * pow2d(mid_bit(SET));
    const double d = __int2double_rn(group_value<SET, PRIVATE, H, G>(w)), rest = c_recon[SET].rest[G];
    X0 = G == 0 ? d * rest : fma(d, rest, X0);
    X1 = G == 0 ? d * mid : fma(d, mid, X1);
    X2 = G == 0 ? d * high : fma(d, high, X2);
}

template <int SET, bool PRIVATE, int H, int... G>
__device__ __forceinline__ void crt_sum(std::integer_sequence<int, G...>, const Numbers &w, double &X0, double &X1, double &X2)
{
    (crt_term<SET, PRIVATE, H, G>(w, X0, X1, X2), ...);
}

template <int SET, bool PRIVATE, int H, int... G>
__device__ __forceinline__ void group_values(std::integer_sequence<int, G...>, const Numbers &w, int (&u)[kMaxGroups])
{
    ((u[G] = group_value<SET, PRIVATE, H, G>(w)), ...);
}

template <int SET, int... G>
__device__ __forceinline__ unsigned __int128 exact_sum(std::integer_sequence<int, G...>, const int (&u)[kMaxGroups])
{
    unsigned __int128 v = 0;
    auto term = [&](int ug, Wide N) {
        v += static_cast<unsigned __int128>(static_cast<__int128>(ug)) * ((static_cast<unsigned __int128>(N.hi) << 64) | N.lo);
    };
    (term(u[G], group_weight(SET, G)), ...);
    return v;
}

// The numbers of a thread from the public layout: ROWS consecutive rows of a column.  WORDS: one 32-bit load covers them; else an element
// each, the last row again for those behind it, so that no load waits for a branch (3001 x 2999 update, an odd
// leading dimension: with a branch a modulus 227 us on S, 181 on A; now 94 and 107).
template <int SET, bool WORDS>
struct PublicLoader {
    static constexpr bool kPrivate = false;
    const unsigned char *base;
    int64_t stride;                  // bytes from modulus to modulus
    int nrows;
    template <int I>
    __device__ __forceinline__ void load_one(Numbers &w) const
    {
        constexpr int RB = residue_bytes(SET);
        w.hi[I] = 0u;
        const unsigned char *src = base + I * stride;
        if constexpr (WORDS) {
            w.lo[I] = *reinterpret_cast<const uint32_t *>(src);        // ldr is a multiple of ROWS: in bounds
        } else if constexpr (RB == 2) {
            const uint16_t *e = reinterpret_cast<const uint16_t *>(src);
            w.lo[I] = e[0] | static_cast<uint32_t>(e[nrows > 1 ? 1 : 0]) << 16;
        } else {
            w.lo[I] = src[0] | static_cast<uint32_t>(src[nrows > 1 ? 1 : 0]) << 8 | static_cast<uint32_t>(src[nrows > 2 ? 2 : 0]) << 16 |
                      static_cast<uint32_t>(src[nrows > 3 ? 3 : 0]) << 24;
        }
    }
    template <int I> __device__ __forceinline__ void finish_one(Numbers &) const {}
};

// Threads of a block of the private layout's kernel: one warp for each chunk of sixteen rows and, of two rows a thread, each half of it; eight columns.  1024
// threads on an SM: numbers, sums and old values of C take 64 registers.  16384 x 16384 update, set S, in blocks of 256 threads 1709 us, of 128
// 1611 us, the same with 896 threads on an SM (72 registers), 1893 with 1152 (56, spills).
__host__ __device__ constexpr int tiled_threads(int rows) { return rows == 4 ? 128 : 256; }
constexpr int kPieces = 4;             // thread blocks to a patch

// From a patch of the private array: chunk, column, word of the chunk; of two rows a thread, the half of the word.  Where a thread stands follows from its number.
template <int SET, int ROWS, bool SPREAD>
struct PatchLoader {
    static constexpr bool kPrivate = true;
    const unsigned char *patch;
    static __device__ __forceinline__ uint32_t chunk() { return SPREAD ? (threadIdx.x >> 5) & 3u : (threadIdx.x >> 2) & 3u; }
    static __device__ __forceinline__ uint32_t half_word() { return ROWS == 4 ? 0u : SPREAD ? threadIdx.x >> 7 : (threadIdx.x >> 4) & 1u; }
    static __device__ __forceinline__ uint32_t column_of() { return blockIdx.x % kPieces * 8 + (SPREAD ? (threadIdx.x >> 2) & 7u : threadIdx.x / (64 / ROWS)); }
    static __device__ __forceinline__ uint32_t word_of() { return threadIdx.x & 3u; }
    template <int I>
    __device__ __forceinline__ void load_one(Numbers &w) const
    {
        constexpr int form = stored_form(SET, I);
        const uint32_t c = chunk(), half = half_word(), column = column_of(), word = word_of();
        const unsigned char *src = patch + stored_start(SET, I);           // a compile-time offset from one address
        w.hi[I] = 0u;
        if constexpr (form == kStoredPair) {
            w.lo[I] = *reinterpret_cast<const uint32_t *>(src + ((2 * c + (ROWS == 2 ? half : 0u)) * 32 + column) * 16 + word * 4);
            if constexpr (ROWS == 4) w.hi[I] = *reinterpret_cast<const uint32_t *>(src + ((2 * c + 1) * 32 + column) * 16 + word * 4);
        } else {
            w.lo[I] = *reinterpret_cast<const uint32_t *>(src + (c * 32 + column) * 16 + word * 4);
            if constexpr (form == kStoredTen) w.hi[I] = *reinterpret_cast<const uint32_t *>(src + 2048 + column * 16 + c * 4);
        }
    }
    template <int I>
    __device__ __forceinline__ void finish_one(Numbers &w) const       // the thread's rows of what was loaded
    {
        const uint32_t skip = 16 * half_word(), word = word_of();
        if constexpr (stored_form(SET, I) == kStoredTen) w.hi[I] = (w.hi[I] >> (2 * word + skip)) & 0x03030303u;        // the thread's bits
        if constexpr (stored_form(SET, I) != kStoredPair && ROWS == 2) w.lo[I] >>= skip;
    }
};

template <class Loader, int... I>
__device__ __forceinline__ void load_numbers(std::integer_sequence<int, I...>, const Loader &from, Numbers &w)
{
    (from.template load_one<I>(w), ...);
    (from.template finish_one<I>(w), ...);
}

// row h, no compile-time constant here, in the place of the first one
template <int SET, bool PRIVATE>
__device__ __forceinline__ void first_row(Numbers &w, int h)
{
#pragma unroll
    for (int i = 0; i < set_r(SET); ++i) {
        if (PRIVATE ? stored_form(SET, i) == kStoredPair : residue_bytes(SET) == 2) {
            w.lo[i] = (h < 2 ? w.lo[i] : w.hi[i]) >> (16 * (h & 1));
        } else {
            w.lo[i] >>= 8 * h;
            w.hi[i] >>= 8 * h;
        }
    }
}

// ---- results that a floating sum with an inexact rest leaves undecided: near a rounding boundary, or small ----
// r is an integer near c', and c' modulo 2^64 takes two integer multiply-adds a group: c' - r is the difference modulo 2^64 with its sign,
// exact as a double, and r + (c' - r) is c' correctly rounded by that one addition.  For |r| below 2^kSettledLog2: the difference, the rest's error and half an
// ulp of r, stays below 2^53, and kappa is far from a tie.  Products with structural zeros, decaying or graded operands have such results by the
// million: 4000 x 4000 x 500 updates of graded operands (N(0,1) exp(-|i - j| / 5), results 2^-30 to 2^-80 of the bound) by the 128-bit sum below, row after
// row, 604 us a call on S, 601 on E, 434 on A, by this form 416, 410 and 299, where every result settled by the floating sum takes 380, 400 and 270.
constexpr int kSettledLog2 = 104;
template <int SET> constexpr bool kSettles = kRestErrorLog2<SET> < 50 && static_cast<double>(half_M_word(SET) >> 20) > 1023.0 + kSettledLog2 + 4.0;
static_assert(kSettles<0> && kSettles<1> && kSettles<2>, "a difference that a double holds, kappa within a tenth of an integer");
__device__ __forceinline__ bool settles(double r) { return 2u * static_cast<uint32_t>(__double2hiint(r)) < 2u * (static_cast<uint32_t>(1023 + kSettledLog2) << 20); }

// kappa = round(sum of u_g / P_g) by integers: 2^share_bits() / P_g fits 31 bits
__host__ __device__ constexpr int share_bits(int set)
{
    uint64_t least = group_product(set, 0);
    for (int g = 1; g < set_groups(set); ++g) least = group_product(set, g) < least ? group_product(set, g) : least;
    int b = 31;
    while (b < 50 && ((2ull << b) / least) >> 31 == 0) ++b;
    return b;
}
__host__ __device__ constexpr int32_t share_factor(int set, int g) { return static_cast<int32_t>((1ull << share_bits(set)) / group_product(set, g)); }
template <int SET> constexpr bool kShares = group_bounds(SET).kappa * pow2d(share_bits(SET)) < pow2d(62) &&
                                            set_groups(SET) * pow2d(31) < pow2d(share_bits(SET) - 3);
static_assert(kShares<0> && kShares<1> && kShares<2>, "the sum of the shares fits 63 bits and is within an eighth");

// + u w modulo 2^64, the low word of w balanced
__device__ __forceinline__ void add_low(int u, uint64_t w, uint64_t &low, uint32_t &high)
{
    const int32_t l = static_cast<int32_t>(static_cast<uint32_t>(w));
    low += static_cast<uint64_t>(static_cast<int64_t>(u) * l);
    high += static_cast<uint32_t>(u) * static_cast<uint32_t>((w - static_cast<uint64_t>(static_cast<int64_t>(l))) >> 32);
}

// an integer r, |r| < 2^116, modulo 2^64
__device__ __forceinline__ uint64_t low_bits(double r)
{
    const uint64_t bits = static_cast<uint64_t>(__double_as_longlong(r)), sig = (bits & 0xFFFFFFFFFFFFFull) | (1ull << 52);
    const int e = (__double2hiint(r) >> 20 & 0x7FF) - 1075;
    const uint64_t v = e >= 0 ? sig << (e & 63) : e >= -52 ? sig >> (-e & 63) : 0ull;
    return __double2hiint(r) < 0 ? 0ull - v : v;
}

template <int SET, int... G>
__device__ __forceinline__ double settled(std::integer_sequence<int, G...>, const int (&u)[kMaxGroups], double r)
{
    int64_t share = 1ll << (share_bits(SET) - 1);
    ((share += static_cast<int64_t>(u[G]) * share_factor(SET, G)), ...);
    uint64_t low = 0ull;
    uint32_t high = 0u;
    (add_low(u[G], group_weight(SET, G).lo, low, high), ...);
    add_low(-static_cast<int>(share >> share_bits(SET)), group_weight(SET, -1).lo, low, high);
    return r + static_cast<double>(static_cast<int64_t>(low + (static_cast<uint64_t>(high) << 32) - low_bits(r)));
}

// The thread's rows (bit h) whose c' is zero if it is below 2^(kRestErrorLog2 + 3) in magnitude.  It is zero where the products of two
// groups, together larger than that, divide it: a third of the work of settle_rows(), for products with structural zeros.
template <int SET, int ROWS, class Loader, int... H>
__device__ __forceinline__ uint32_t zero_rows(std::integer_sequence<int, H...>, const Loader &from)
{
    constexpr int64_t P0 = static_cast<int64_t>(group_product(SET, 0)), P1 = static_cast<int64_t>(group_product(SET, 1));
    static_assert(static_cast<double>(P0) * static_cast<double>(P1) > pow2d(kRestErrorLog2<SET> + 4), "two groups tell");
    constexpr int a2 = group_member(SET, 0, 2), b2 = group_member(SET, 1, 2);
    Numbers w = {};
    load_numbers(std::integer_sequence<int, group_member(SET, 0, 0), group_member(SET, 0, 1), group_member(SET, 1, 0), group_member(SET, 1, 1)>{}, from, w);
    if constexpr (a2 >= 0) load_numbers(std::integer_sequence<int, a2>{}, from, w);
    if constexpr (b2 >= 0) load_numbers(std::integer_sequence<int, b2>{}, from, w);
    return ((group_value<SET, Loader::kPrivate, H, 0>(w) % static_cast<int>(P0) == 0 && group_value<SET, Loader::kPrivate, H, 1>(w) % static_cast<int>(P1) == 0 ? 1u << H : 0u) | ...);
}

template <int SET, int ROWS, class Loader, int... H>
__device__ __forceinline__ void settle_rows(std::integer_sequence<int, H...>, const Loader &from, double (&r)[ROWS])
{
    Numbers w;
    load_numbers(std::make_integer_sequence<int, set_r(SET)>{}, from, w);
    auto one = [&](auto index) {
        constexpr int h = decltype(index)::value;
        constexpr auto groups = std::make_integer_sequence<int, set_groups(SET)>{};
        int u[kMaxGroups] = {};
        group_values<SET, Loader::kPrivate, h>(groups, w, u);
        r[h] = settles(r[h]) ? settled<SET>(groups, u, r[h]) : r[h];
    };
    (one(std::integral_constant<int, H>{}), ...);
}

// alpha 2^-(sa + sb) c' (alpha = 1 or -1, as a sign bit) where only the scale is out of reach: r is c' correctly rounded.  NaN for a line with
// Inf/NaN.  The sum of the shifts is taken in 64 bits; beyond 2^20 the result is zero or infinite whatever c' is.
__device__ __forceinline__ bool marked(int sa, int sb) { return sb == OZ_NONFINITE_SHIFT || sa == OZ_NONFINITE_SHIFT; }
__device__ __forceinline__ int far_sum(int sa, int sb)
{
    return static_cast<int>(min(max(static_cast<long long>(sa) + sb, -(1ll << 20)), 1ll << 20));
}
__device__ __noinline__ double row_value_far(double r, int sa, int sb, int alpha_sign)
{
    const double alpha = __hiloint2double(0x3FF00000 ^ alpha_sign, 0);
    if (marked(sa, sb)) return __longlong_as_double(0x7FF8000000000000ll) * alpha;
    return scale_pow2(r, -far_sum(sa, sb)) * alpha;
}

// The same where c' itself has to be formed: the sum modulo 2^128 (|c'| is below 2^118), exact lift to [-M/2, M/2),
// round-to-nearest-even conversion in integer arithmetic, power-of-two scale.
// `from` reads the numbers once more: held until here they would cost the common case a third of its registers.
template <int SET, class Loader>
__device__ __noinline__ double row_value_exact(Loader from, int h, int sa, int sb, int alpha_sign)
{
    const double alpha = __hiloint2double(0x3FF00000 ^ alpha_sign, 0);
    if (marked(sa, sb)) return __longlong_as_double(0x7FF8000000000000ll) * alpha;
    Numbers w;
    load_numbers(std::make_integer_sequence<int, set_r(SET)>{}, from, w);
    first_row<SET, Loader::kPrivate>(w, h);
    int u[kMaxGroups] = {};
    group_values<SET, Loader::kPrivate, 0>(std::make_integer_sequence<int, set_groups(SET)>{}, w, u);
    constexpr Wide Mw = group_weight(SET, -1);
    const __int128 M = static_cast<__int128>((static_cast<unsigned __int128>(Mw.hi) << 64) | Mw.lo);
    const __int128 Mh = M >> 1;     // M is even for every set (each holds a power of two)
    double share = 0.0;             // S / M
#pragma unroll
    for (int g = 0; g < set_groups(SET); ++g) share += static_cast<double>(u[g]) / static_cast<double>(group_product(SET, g));
    const __int128 kappa = static_cast<__int128>(__double2int_rn(share));
    __int128 v = static_cast<__int128>(exact_sum<SET>(std::make_integer_sequence<int, set_groups(SET)>{}, u) -
                                       static_cast<unsigned __int128>(M) * static_cast<unsigned __int128>(kappa));
    if (v >= Mh) v -= M;
    else if (v < -Mh) v += M;
    unsigned long long lo = static_cast<unsigned long long>(v);
    long long hi = static_cast<long long>(v >> 64);
    const bool neg = hi < 0;
    if (neg) {
        lo = 0ull - lo;
        hi = ~hi + (lo == 0ull ? 1 : 0);
    }
    // nearest double, ties to even: top 64 bits with a sticky bit far below the rounding position
    const unsigned long long uhi = static_cast<unsigned long long>(hi);
    const int lz = __clzll(static_cast<long long>(uhi | 1ull));          // uhi < 2^54: lz in [10, 63]
    const unsigned long long top = (uhi << lz) | (lo >> (64 - lz));
    const unsigned long long rest = lo << lz;
    const unsigned long long mant = uhi ? (top | (rest ? 1ull : 0ull)) : lo;
    const double d = scale_pow2(__ull2double_rn(mant), (uhi ? 64 - lz : 0) - far_sum(sa, sb));
    return (neg ? -d : d) * alpha;
}

// One row: r, and whether it is c' correctly rounded.
// X2 + X1 = s + err by a fast two-sum, which is error-free because X2 is a multiple of 2^high_bit and so of ulp(X1)
// (|X1| < 2^(53 + mid_bit)); t = err + X0, where X0 is off by its multiply-adds' roundings; s + t = r + rem exactly (s is a multiple of
// 2^mid_bit and so of ulp(t)).  All that is lost is below 2^kRestErrorLog2, so r is c' correctly rounded where rem enlarged by that much
// does not move it and |r| is in the range of range_word(): from 2^56 times that error on, so that the other side is no nearer, a power of two
// included, and below M / 2.
template <int SET, bool PRIVATE, int H>
__device__ __forceinline__ bool row_value(const Numbers &w, double &r)
{
    constexpr Parts M = split_parts(SET, group_weight(SET, -1));
    constexpr double M1 = static_cast<double>(M.mid) * pow2d(mid_bit(SET)), M2 = static_cast<double>(M.high) * pow2d(high_bit(SET));
    double X0 = 0.0, X1 = 0.0, X2 = 0.0;
    crt_sum<SET, PRIVATE, H>(std::make_integer_sequence<int, set_groups(SET)>{}, w, X0, X1, X2);
    const double minus_kappa = kRint - fma(X2 + X1, c_recon[SET].inv_M, kRint);
    X0 = fma(minus_kappa, c_recon[SET].M_rest, X0);
    X1 = fma(minus_kappa, M1, X1);              // exact: integers below 2^53 in units of their places
    X2 = fma(minus_kappa, M2, X2);
    const double s = X2 + X1, err = X1 - (s - X2);
    const double t = err + X0;
    r = s + t;
    const double rem = t - (r - s);
    constexpr int kErrorWord = (1023 + kRestErrorLog2<SET>) << 20;
    const double more = rem + __hiloint2double((__double2hiint(rem) & INT32_MIN) | kErrorWord, 0);
    return r + more == r;
}
// below kRangeSpan for |r| in that range (the sign shifted out)
template <int SET> constexpr uint32_t kRangeSpan = 2u * (half_M_word(SET) - small_word(SET));
template <int SET>
__device__ __forceinline__ uint32_t range_word(double r) { return 2u * static_cast<uint32_t>(__double2hiint(r)) - 2u * small_word(SET); }

template <bool PRIVATE> __device__ __forceinline__ constexpr int row_of(int h) { return (h & 1) + (PRIVATE ? 8 : 2) * (h >> 1); }
// alpha 2^-(sa + sb) c' for all rows of a thread, one of which at least is not as row_value() leaves it.  sure: the rows that
// row_value() calls rounded (bit h).
template <int ROWS> struct Results { double r[ROWS]; };
template <int ROWS> struct Shifts { int s[ROWS]; };
template <int SET, int ROWS, class Loader, int... H>
__device__ __forceinline__ Results<ROWS> finish_rows(std::integer_sequence<int, H...> rows, const Loader &from, Results<ROWS> v, const Shifts<ROWS> &sa, int sb,
                                                     int alpha_sign, int nrows, uint32_t sure)
{
    // rows of C whose result is not known to be rounded; those among them near zero
    uint32_t open = 0u, least = 0u;
    constexpr uint32_t small = 2u * (static_cast<uint32_t>(1023 + kRestErrorLog2<SET> + 2) << 20);       // |c'| is below twice the bound of |r|
#pragma unroll
    for (int h = 0; h < ROWS; ++h) {
        if (((sure >> h & 1u) && range_word<SET>(v.r[h]) < kRangeSpan<SET>) || marked(sa.s[h], sb) || row_of<Loader::kPrivate>(h) >= nrows) continue;
        open |= 1u << h;
        if (2u * static_cast<uint32_t>(__double2hiint(v.r[h])) < small) least |= 1u << h;
    }
    if (open != 0u && open == least) {
        const uint32_t zeros = zero_rows<SET, ROWS>(rows, from) & open;
#pragma unroll
        for (int h = 0; h < ROWS; ++h) v.r[h] = zeros >> h & 1u ? 0.0 : v.r[h];
        open &= ~zeros;
    }
    if (open != 0u) {
        settle_rows<SET, ROWS>(rows, from, v.r);
#pragma unroll
        for (int h = 0; h < ROWS; ++h)
            if (settles(v.r[h])) open &= ~(1u << h);
    }
#pragma unroll
    for (int h = 0; h < ROWS; ++h) {
        const uint32_t sum = static_cast<uint32_t>(sa.s[h]) + static_cast<uint32_t>(sb);
        if (open >> h & 1u) v.r[h] = row_value_exact<SET>(from, h, sa.s[h], sb, alpha_sign);
        else if (sum + 904u <= 1924u && static_cast<uint32_t>(sa.s[h]) + (1u << 30) < 1u << 31)
            v.r[h] *= __hiloint2double(static_cast<int>((1023u - sum) << 20) ^ alpha_sign, 0);
        else v.r[h] = row_value_far(v.r[h], sa.s[h], sb, alpha_sign);
    }
    return v;
}

// Out of line for four rows a thread of the private layout, whose registers are full: what it needs then costs the common case none of them (all but
// two variants without spills; inline, which keeps the numbers from the first load, 20 to 50 bytes: plain 4000 x 4000 x 500 updates 2 percent slower).
template <int SET, int ROWS, class Loader, int... H>
__device__ __noinline__ Results<ROWS> finish_rows_call(std::integer_sequence<int, H...> rows, Loader from, Results<ROWS> v, Shifts<ROWS> sa, int sb,
                                                       int alpha_sign, int nrows, uint32_t sure)
{
    return finish_rows<SET, ROWS>(rows, from, v, sa, sb, alpha_sign, nrows, sure);
}

// scalar stores of up to two consecutive rows; `first` / `second`: which of them are written.  A zero without an old value is +0, as in the stores of pairs.
__device__ __forceinline__ void store_pair(double *out, double p0, double p1, bool first, bool second, double beta)
{
    if (first) out[0] = (beta != 0.0 ? out[0] : 0.0) + p0;
    if (second) out[1] = (beta != 0.0 ? out[1] : 0.0) + p1;
}

// ROWS rows of a column, row_of(0) .. from `row` on: reconstruct, update C with fast alpha 2^-(sa + sb) c'.
// For beta = 1 the old values of C are requested before the arithmetic starts, so that their latency
// hides behind it.  nrows: rows of C from `row` on.  `keep`: bit h set = the thread's row h is written (rows that go to the native FP64 path are not).
// The tests of a thread's rows are taken together: one branch a thread, which almost none takes.
template <int SET, int ROWS, class Loader, int... H>
__device__ __forceinline__ void reconstruct_rows(std::integer_sequence<int, H...>, const Loader &from, int64_t row, int nrows, int sb,
                                                 const int32_t *__restrict__ shiftA, double alpha, double beta,
                                                 double *out, bool vecC, uint32_t keep)
{
    constexpr bool PRIVATE = Loader::kPrivate;
    // all residue loads are issued before any arithmetic: independent requests in flight per
    // thread, kept packed so that they fit the register budget
    Numbers w;
    load_numbers(std::make_integer_sequence<int, set_r(SET)>{}, from, w);
    int sa[ROWS];
#pragma unroll
    for (int h = 0; h < ROWS; ++h) sa[h] = row_of<PRIVATE>(h) < nrows ? shiftA[row + row_of<PRIVATE>(h)] : 0;
    const bool whole = vecC && nrows > row_of<PRIVATE>(ROWS - 1) && (keep & ((1u << ROWS) - 1u)) == ((1u << ROWS) - 1u);
    double2 old[ROWS / 2];
#pragma unroll
    for (int h = 0; h < ROWS / 2; ++h) old[h] = make_double2(0.0, 0.0);
    if (whole && beta != 0.0) {
#pragma unroll
        for (int h = 0; h < ROWS / 2; ++h) old[h] = *reinterpret_cast<const double2 *>(out + row_of<PRIVATE>(2 * h));
    }
    const int alpha_sign = alpha < 0.0 ? INT32_MIN : 0;
    double r[ROWS];
    bool rounded[ROWS];
    ((rounded[H] = row_value<SET, PRIVATE, H>(w, r[H])), ...);
    // 2^-(sa + sb) and r 2^-(sa + sb) are normal for sums in [-904, 1020] (1 <= |r| < 2^118); the sum is taken in 32 bits, which a shift of
    // at most 2^30, unlike the mark of a row with Inf/NaN, cannot wrap into that range whatever the column's is, its mark among them
    uint32_t scale[ROWS], far = 0u, wide = 0u, range = 0u;
    bool all = true;
    const uint32_t scale0 = (1023u + 904u) << 20 ^ static_cast<uint32_t>(alpha_sign);
#pragma unroll
    for (int h = 0; h < ROWS; ++h) {
        const uint32_t sum = static_cast<uint32_t>(sa[h]) + static_cast<uint32_t>(sb) + 904u;
        far = max(far, sum);
        wide |= static_cast<uint32_t>(sa[h]) + (1u << 30);
        range = max(range, range_word<SET>(r[h]));
        scale[h] = scale0 - (sum << 20);                 // high word of alpha 2^-(sa + sb)
        all = all && rounded[h];
    }
    if (!(all && far <= 1924u && wide < 1u << 31 && range < kRangeSpan<SET>)) {
        uint32_t sure = 0u;
#pragma unroll
        for (int h = 0; h < ROWS; ++h) sure |= rounded[h] ? 1u << h : 0u;
        Results<ROWS> v;
        if constexpr (PRIVATE && ROWS == 4) v = finish_rows_call<SET, ROWS>(std::integer_sequence<int, H...>{}, from, {{r[H]...}}, {{sa[H]...}}, sb, alpha_sign, nrows, sure);
        else v = finish_rows<SET, ROWS>(std::integer_sequence<int, H...>{}, from, {{r[H]...}}, {{sa[H]...}}, sb, alpha_sign, nrows, sure);
#pragma unroll
        for (int h = 0; h < ROWS; ++h) {
            r[h] = v.r[h];
            scale[h] = 0x3FF00000u;
        }
    }
#pragma unroll
    for (int p = 0; p < ROWS / 2; ++p) {
        const int first = row_of<PRIVATE>(2 * p);
        const double f0 = __hiloint2double(static_cast<int>(scale[2 * p]), 0), f1 = __hiloint2double(static_cast<int>(scale[2 * p + 1]), 0);
        if (whole) *reinterpret_cast<double2 *>(out + first) = make_double2(fma(r[2 * p], f0, old[p].x), fma(r[2 * p + 1], f1, old[p].y));
        else store_pair(out + first, r[2 * p] * f0, r[2 * p + 1] * f1, nrows > first && (keep >> (2 * p) & 1u), nrows > first + 1 && (keep >> (2 * p + 1) & 1u), beta);
    }
}

// Each thread reconstructs ROWS consecutive rows of one column: the residues of those rows are one
// 32-bit word per modulus (two uint16 for S and E, four uint8 for the all-byte set A).
template <int SET, bool WORDS>
__global__ void __launch_bounds__(kPublicThreads, residue_bytes(SET) == 2 ? 9 : 8)
reconstruct_kernel(const void *__restrict__ Rv, int64_t ldr, int64_t mod_stride, int64_t m,
                   int64_t n, const int32_t *__restrict__ shiftA, const int32_t *__restrict__ shiftB,
                   double alpha, double beta, double *__restrict__ C, int64_t ldc, int vecC)
{
    dependency_release();
    dependency_wait();
    constexpr int RB = residue_bytes(SET), ROWS = 4 / RB;
    // grid.x covers the row groups of a column, grid.y (and .z beyond 65535) the columns: no division
    const int64_t row = (blockIdx.x * static_cast<int64_t>(kPublicThreads) + threadIdx.x) * ROWS;
    if (row >= m) return;
    const int64_t j = blockIdx.y + 65535ll * blockIdx.z;
    if (j >= n) return;
    const int nrows = m - row < ROWS ? static_cast<int>(m - row) : ROWS;

    const PublicLoader<SET, WORDS> from{static_cast<const unsigned char *>(Rv) + (j * ldr + row) * RB, mod_stride * RB, nrows};
    reconstruct_rows<SET, ROWS>(std::make_integer_sequence<int, ROWS>{}, from, row, nrows, shiftB[j], shiftA, alpha, beta, C + row + j * ldc, vecC != 0, 0xFu);
}

// Same reconstruction from the tile-ordered private array that the whole-method GEMM writes (see
// ResidueTiling).  A thread takes four rows of one column: one 32-bit word of low bytes per modulus, and a word of high bits that the
// four threads of a 16-byte chunk share.  A warp takes one chunk of eight neighbouring columns: its loads of low bytes are whole
// 128-byte lines and its accesses to C eight pieces of 64 contiguous bytes; its next ones and the warps of a thread block, which
// take the other chunks of the same columns, complete those to whole lines of C.
// ACCESS: how C is taken, in pairs of elements (even ldc, C on a multiple of 16 bytes), or singly, stored or updated.  Updates of single
// elements, whose loads and stores in eight pieces each cost more the more there are, give a warp consecutive words of one column: 512
// contiguous bytes of C for residue loads that touch eight lines.  1009 x 983 x 256, set S: 39 us a call against 52; 4501 x 4400 x 128: 400
// against 732; plain stores are faster in pieces (34 us against 36, 334 against 352).
// The loads wait for DRAM as long as the arithmetic takes, so the first block of a patch asks for the patch that is `ahead` of it, in the order of the
// blocks, to be brought into L2: 16384 x 16384 update, set S, 1803 -> 1725 us (old values of C too: 1760; only those: 1922), 8192 x 8192 on set A
// 401 -> 363 us.  (Patches in a ring of shared memory, two ahead, two blocks of 512 threads an SM: 2920 us.)
// grid: x = (piece of the patch, patch within the tile, CTA rank of the pair), y = tile column, z = tile row
// SKIP: rows flagged in `skip` are left untouched (they are re-issued on the native FP64 path).
enum { kPairs, kSingleStores, kSingleUpdates };
// ROWS: four, or two where the outputs are few and a thread's chain of arithmetic counts (launch_reconstruct_tiled())
template <int SET, bool SKIP, int ACCESS, int ROWS>
__global__ void __launch_bounds__(tiled_threads(ROWS), 1024 / tiled_threads(ROWS))
reconstruct_tiled_kernel(const void *__restrict__ Rv, int cg, int tiles_n, int tn0,
                         int64_t m, int64_t n, int64_t col0, int64_t col1,
                         const int32_t *__restrict__ shiftA, const int32_t *__restrict__ shiftB,
                         double alpha, double beta, double *__restrict__ C, int64_t ldc,
                         const unsigned char *__restrict__ skip, uint32_t ahead)
{
    dependency_release();
    dependency_wait();
    constexpr bool spread = ACCESS != kSingleUpdates;
    using Loader = PatchLoader<SET, ROWS, spread>;
    const uint32_t wi = (blockIdx.x / kPieces) & 15u;
    const uint32_t rank = blockIdx.x / (kPieces * 16);     // 0, or 0..1 with CTA pairs
    const uint32_t tn = static_cast<uint32_t>(tn0) + blockIdx.y, tm = blockIdx.z;
    const uint32_t patch = ((tm * static_cast<uint32_t>(tiles_n) + tn) * static_cast<uint32_t>(cg) + rank) * 16 + wi;
    if (ahead != 0 && threadIdx.x == 0 && blockIdx.x % kPieces == 0) {
        const uint32_t next = patch + ahead;
        if (next < static_cast<uint32_t>(tiles_n) * gridDim.z * static_cast<uint32_t>(cg) * 16)
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;"
                         ::"l"(static_cast<const unsigned char *>(Rv) + next * static_cast<int64_t>(patch_bytes(SET))), "r"(patch_bytes(SET)) : "memory");
    }
    const int64_t row = static_cast<int64_t>(tm) * 256 + (wi >> 2) * 64 + Loader::chunk() * 16 + Loader::half_word() * 8 + Loader::word_of() * 2;
    const int64_t j = (static_cast<int64_t>(tn) * cg + rank) * 128 + (wi & 3u) * 32 + Loader::column_of();
    if (row >= m || j >= n || j < col0 || j >= col1) return;
    const int nrows = m - row < 16 ? static_cast<int>(m - row) : 16;
    uint32_t keep = 0xFu;
    if constexpr (SKIP) {
        keep = 0u;
#pragma unroll
        for (int h = 0; h < ROWS; ++h)
            if (row_of<true>(h) < nrows && !skip[row + row_of<true>(h)]) keep |= 1u << h;
        if (!keep) return;
    }
    const Loader from{static_cast<const unsigned char *>(Rv) + patch * static_cast<int64_t>(patch_bytes(SET))};
    reconstruct_rows<SET, ROWS>(std::make_integer_sequence<int, ROWS>{}, from, row, nrows, shiftB[j], shiftA, alpha, beta, C + row + j * ldc, ACCESS == kPairs, keep);
}

}  // namespace

oz_status_t launch_reconstruct(int64_t m, int64_t n, const void *R, int64_t ldr,
                               int64_t mod_stride, const int32_t *shiftA, const int32_t *shiftB,
                               int set, double alpha, double beta, double *C, int64_t ldc,
                               cudaStream_t stream)
{
    // one 32-bit load per modulus covers a thread's rows when every row group starts on a 4-byte boundary
    const int rows = 4 / residue_bytes(set);
    const bool words = ldr % rows == 0 && mod_stride % rows == 0 && (reinterpret_cast<uintptr_t>(R) & 3u) == 0;
    int vecC = ((ldc & 1) == 0 && (reinterpret_cast<uintptr_t>(C) & 15u) == 0) ? 1 : 0;
    int64_t bx = ((m + rows - 1) / rows + kPublicThreads - 1) / kPublicThreads;
    if (bx > 0x7FFFFFFFll) return OZ_ERR_UNSUPPORTED;
    if (n > 65535ll * 65535ll) return OZ_ERR_UNSUPPORTED;
    dim3 grid(static_cast<unsigned>(bx), static_cast<unsigned>(n < 65535 ? n : 65535),
              static_cast<unsigned>((n + 65534) / 65535));
    auto kernel = words ? (set == 2 ? reconstruct_kernel<2, true> : set == 0 ? reconstruct_kernel<0, true> : reconstruct_kernel<1, true>)
                        : (set == 2 ? reconstruct_kernel<2, false> : set == 0 ? reconstruct_kernel<0, false> : reconstruct_kernel<1, false>);
    OZ_CUDA_CHECK(launch(kernel, grid, kPublicThreads, 0, stream, R, ldr, mod_stride, m, n, shiftA, shiftB, alpha, beta, C, ldc, vecC));
    count_launch();
    OZ_CUDA_CHECK(cudaGetLastError());
    return OZ_OK;
}

oz_status_t launch_reconstruct_tiled(int64_t m, int64_t n, const void *R, const int32_t *shiftA,
                                     const int32_t *shiftB, int set, double alpha, double beta,
                                     double *C, int64_t ldc, int64_t col0, int64_t col1,
                                     cudaStream_t stream, const unsigned char *skip)
{
    if (col1 <= col0) return OZ_OK;
    const ResidueTiling t = residue_tiling(m, n, set);
    const int tn0 = static_cast<int>(col0 / t.tile_cols);
    const int ntn = static_cast<int>((col1 + t.tile_cols - 1) / t.tile_cols) - tn0;
    // there the threads of four rows do not fill the chip
    const bool few = m * n <= kFewOutputs;
    if (t.tiles_m > 65535 || ntn > 65535) return OZ_ERR_UNSUPPORTED;
    const int vecC = ((ldc & 1) == 0 && (reinterpret_cast<uintptr_t>(C) & 15u) == 0) ? 1 : 0;
    const dim3 grid(static_cast<unsigned>(kPieces * 16 * t.cg), static_cast<unsigned>(ntn),
                    static_cast<unsigned>(t.tiles_m));
    // Blocks that become resident beside the GEMM's keep the multiprocessor's memory split at the GEMM's (28 KiB of L1) for
    // the whole kernel: worth the overlapped launch up to a million outputs only (16384 x 16384: 11.4 -> 11.9 ms a call)
    const bool early = m * n <= (1ll << 20);
    // one round of resident blocks ahead; not for a panel, whose blocks do not walk the array from end to end
    const int64_t patches = static_cast<int64_t>(t.tiles_m) * t.tiles_n * t.cg * 16;
    if (patches > 0x7FFFFFFFll) return OZ_ERR_UNSUPPORTED;       // as the residue GEMM
    const uint32_t ahead = ntn == t.tiles_n ? static_cast<uint32_t>(1024 / tiled_threads(few ? 2 : 4) * sm_count() / kPieces) : 0u;
#define OZ_RECON_KERNEL(SET_, SKIP_, ROWS_)                                             \
    (vecC          ? reconstruct_tiled_kernel<SET_, SKIP_, kPairs, ROWS_>               \
     : beta == 0.0 ? reconstruct_tiled_kernel<SET_, SKIP_, kSingleStores, ROWS_>        \
                   : reconstruct_tiled_kernel<SET_, SKIP_, kSingleUpdates, ROWS_>)
#define OZ_RECON_TILED(SET_)                                                                                         \
    OZ_CUDA_CHECK(launch_if(early, few ? (skip ? OZ_RECON_KERNEL(SET_, true, 2) : OZ_RECON_KERNEL(SET_, false, 2))   \
                                       : (skip ? OZ_RECON_KERNEL(SET_, true, 4) : OZ_RECON_KERNEL(SET_, false, 4)), grid, tiled_threads(few ? 2 : 4), 0, stream, R, t.cg, \
                         t.tiles_n, tn0, m, n, col0, col1, shiftA, shiftB, alpha, beta, C, ldc, skip, ahead))
    if (set == 2) OZ_RECON_TILED(2);
    else if (set == 0) OZ_RECON_TILED(0);
    else OZ_RECON_TILED(1);
#undef OZ_RECON_TILED
#undef OZ_RECON_KERNEL
    count_launch();
    OZ_CUDA_CHECK(cudaGetLastError());
    return OZ_OK;
}

}  // namespace oz
