// Deconstruction (Algorithm 2; scaling of Eq. 1): FP64 operand -> per-line shifts and K-major
// 8-bit residue planes.
//
// Kernels of the three-pass form, in launch order (the scans serve both operands of a product at once where both take it):
//   scan_sample    clears the per-line scratch (largest exponent, non-finite flag, sums) and guesses every line's largest exponent from 32 samples
//   scan pass 2    largest floor(log2|x|) of every line, Inf/NaN detection, and for the guess and the next two exponents the exact integer sum of
//                  ceil(|x| 2^(9-E))^2
//   scan pass 1    the sums of the lines whose exponent was not among those
// (scan_init, pass 0 without sums and pass 1 of all lines where there is no room for the guesses' sums, too few elements for them to pay, or no need of
// sums: rule MAXEXP and the accurate one, which end with pass 0)
//   scan_finalize  shift[line] (sigma_i or tau_j of Eq. 1)
//   convert        quantise, reduce modulo every modulus, split into digits, store the planes
// Small operands take one kernel instead of the five, both operands of a product together where they fit; lines that fit a
// cluster's shared memory are read once by deconstruct_cluster_kernel.
//
// The scan is split over the inner dimension with integer atomics (max / or / add), so its
// result does not depend on the order of the partial results: the shifts are bit-reproducible.
//
// The residues modulo every m_i and their digits come from FP32 arithmetic on balanced limbs and a small
// per-modulus table in shared memory (oz_convert.cuh; the paper's byte-plane identity of paragraph "O2" on
// limbs of 14 to 16 bits).
#include <utility>

#include "oz_internal.h"
#include "oz_convert.cuh"

namespace oz {
namespace {

constexpr int kConvThreads = 256;
constexpr int kChunk = 128;            // inner-dimension elements of a conversion tile
constexpr int kTileLines = 16;         // lines of a conversion tile: two per warp
constexpr int kTileRow = (kChunk + 2) * 8;            // side 1: bytes of a tile row, an odd number of 16-byte chunks
constexpr int kTileBytes = kTileLines * kTileRow;    // side 0 needs kTileLines * kChunk * 8 of them
static_assert(kTileBytes % 128 == 0, "tile alignment");

// resident blocks per SM: four where no table takes shared memory and 64 registers are enough (three against four: 131072 x 128 x 4096 on
// INT8 digits 7645 and 7326 us a call, native planes of 32768 x 1024 337 and 324 us on side 0, 281 and 273 on side 1)
__host__ __device__ constexpr int conv_blocks(int layout) { return layout == kLayoutNative || two_plane_layout(layout) ? 4 : 3; }

struct ScanScratch {
    unsigned long long *sumsq;  // [lines]  sum of squared magnitudes (accurate rule: maximum of the bound product)
    int *emax;                  // [lines]  largest exponent, INT32_MIN for a line of zeros
    int *nonfinite;             // [lines]  bit 31: the line holds Inf/NaN; bits 0..30: sum of the magnitudes
};
constexpr int kNonfiniteBit = INT32_MIN;

__host__ __device__ inline ScanScratch carve_scratch(void *scratch, int64_t lines)
{
    ScanScratch s;
    char *base = static_cast<char *>(scratch);
    s.sumsq = reinterpret_cast<unsigned long long *>(base);
    s.emax = reinterpret_cast<int *>(base + 8 * lines);
    s.nonfinite = reinterpret_cast<int *>(base + 12 * lines);
    return s;
}

__device__ __forceinline__ const double *element(const double *X, int64_t ldx, int side,
                                                 int64_t line, int64_t kk)
{
    return side == 0 ? X + line + kk * ldx : X + kk + line * ldx;
}

// classification of a double: returns 0 zero, 1 finite non-zero (e = floor(log2|x|)), 2 Inf/NaN
__device__ __forceinline__ int classify(double x, int *e)
{
    unsigned long long bits = static_cast<unsigned long long>(__double_as_longlong(x));
    int be = static_cast<int>((bits >> 52) & 0x7FF);
    unsigned long long frac = bits & 0xFFFFFFFFFFFFFull;
    if (be == 0x7FF) return 2;
    if (be == 0) {
        if (frac == 0) return 0;
        *e = -1011 - __clzll(static_cast<long long>(frac));   // subnormal: normalise the fraction
        return 1;
    }
    *e = be - 1023;
    return 1;
}

// ceil(|x| scale), scale a power of two and a normal number.  The product is exact unless it leaves the normal range; rounded up there, a non-zero x
// counts as 1 however small.
__device__ __forceinline__ unsigned int magnitude(double x, double scale) { return __double2uint_ru(__dmul_ru(fabs(x), scale)); }

// ceil(|x| 2^(9-E)) in integer arithmetic (lines of subnormals, where 2^(9-E) is no normal double)
__device__ __forceinline__ unsigned int scaled_magnitude(double x, int E)
{
    const unsigned long long bits = static_cast<unsigned long long>(__double_as_longlong(x));
    const int be = static_cast<int>((bits >> 52) & 0x7FF);
    const unsigned long long frac = bits & 0xFFFFFFFFFFFFFull;
    if (be == 0x7FF || (be == 0 && frac == 0)) return 0u;
    const unsigned long long sig = be ? (frac | (1ull << 52)) : frac;
    const int ex = be ? be - 1023 : -1022;
    const int sh = 43 + E - ex;                           // |x| 2^(9-E) = sig / 2^sh
    if (sh >= 64) return 1u;
    if (sh <= 0) return static_cast<unsigned int>(sig << (-sh));
    return static_cast<unsigned int>((sig >> sh) + ((sig & ((1ull << sh) - 1ull)) ? 1ull : 0ull));
}

// The norm sums of a line need its largest exponent, which is known only when the whole line has been read.  So the exponent is guessed low, from a sample
// of kSamples elements, and the sums are taken for it and the next ones while the line is read for the first time: ceil(|x| 2^(9 - E - 1)) is
// ceil(ceil(|x| 2^(9 - E)) / 2).  Lines whose exponent lies elsewhere are read again.  These arrays lie in the operand's planes, which the conversion
// fills later; exponent null: two passes.
constexpr int kGuesses = 3, kSamples = 32;
struct ScanGuess {
    unsigned long long *sumsq;  // [kGuesses][lines]
    unsigned int *l1;           // [kGuesses][lines]
    int *exponent;              // [lines]  INT32_MIN: none
};
constexpr int kGuessBytes = kGuesses * 12 + 4;       // a line
__host__ __device__ inline ScanGuess carve_guess(void *spare, int64_t lines)
{
    char *base = static_cast<char *>(spare);
    if (!spare) return {nullptr, nullptr, nullptr};
    return {reinterpret_cast<unsigned long long *>(base), reinterpret_cast<unsigned int *>(base + 8 * kGuesses * lines),
            reinterpret_cast<int *>(base + 12 * kGuesses * lines)};
}
__device__ __forceinline__ bool guessed(int exponent, int guess)
{
    return guess != INT32_MIN && exponent != INT32_MIN && static_cast<unsigned int>(exponent) - static_cast<unsigned int>(guess) < static_cast<unsigned int>(kGuesses);
}

// One operand of a scan.  lines = 0: none.
struct ScanSide {
    const double *X;
    int64_t ldx, lines;
    int64_t kspan;              // inner indices of a block
    uint32_t line_blocks;       // blocks across the lines
    uint32_t blocks;            // in all
    ScanScratch s;
    ScanGuess g;
};

// The scans take one operand or both operands of a product in one launch: blocks [0, a.blocks) serve side 0, the others
// side 1 (2048^3 under the accurate rule: thirteen dependent launches before, nine now, 383 -> 345 us a call).
__global__ void scan_init_kernel(ScanScratch sa, int64_t linesA, ScanScratch sb, int64_t linesB)
{
    dependency_release();
    dependency_wait();
    int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
    const bool side = i >= linesA;
    if (side) i -= linesA;
    const ScanScratch s = side ? sb : sa;
    if (i >= (side ? linesB : linesA)) return;
    s.sumsq[i] = 0ull;
    s.emax[i] = INT32_MIN;
    s.nonfinite[i] = 0;
}

// The same and a guess of every line's exponent.  Blocks of 32 lines (side 0) or eight, one a warp.
// No guess where the samples' exponents lie kWide eighths or more below the largest in the mean (side 0: of the block's lines): other elements of most
// such lines lie above the guesses, and the sums would be in vain.  Mean distances and hits with 4096 elements: U(-1,1) 1.0, all; N(0,1) 2.3, all;
// (U(0,1) - 1/2) exp(s N(0,1)), s = 1/2: 2.3, 99 percent; 0.7: 2.9, 84; 1: 3.6, 54; 2: 6.3, 10.  On side 0 a missed line is read again with all that lie beside it, on side 1 alone.
// oz_prepare_operand with guesses for all lines of all operands -> like this (two passes), us.  (U(0,1) - 1/2) exp(2 N(0,1)): rows of A 37647 x 1700 595 -> 580
// (574), 1000 x 16000 147 -> 144 (142), 281 x 16000 57.7 -> 54.7 (52.8); columns of B 9411 x 1700 152 -> 150 (145), 2647 x 1700 48.7 -> 43.1 (43.5).  U(-1,1):
// 503 -> 505 (574), 122 -> 121 (142), 47.3 -> 47.8 (52.8); 135 -> 132 (146), 44.9 -> 43.1 (43.5).
constexpr unsigned int kWide0 = 25, kWide1 = 42;
constexpr int64_t kGuessed1 = 6000000;       // elements of side 1
__global__ void __launch_bounds__(256)
scan_sample_kernel(const __grid_constant__ ScanSide a, const __grid_constant__ ScanSide b, int64_t k)
{
    __shared__ unsigned int tops[8][32], belows[8][32];
    dependency_release();
    dependency_wait();
    const uint32_t blocksA = static_cast<uint32_t>((a.lines + 31) / 32);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool side = blockIdx.x >= blocksA;
    const ScanSide &p = side ? b : a;
    unsigned int top = 0u, below = 0u;       // below: distances, and from bit 16 on the samples that they belong to
    int64_t line;
    auto distance = [](unsigned int high, unsigned int from) {        // of a high word, zeros and subnormals left out
        const unsigned int e = high >> 20 & 0x7FFu;
        return e ? 0x10000u + min((from >> 20) - e, 15u) : 0u;
    };
    if (!side) {
        line = static_cast<int64_t>(blockIdx.x) * 32 + lane;
        constexpr int PER = kSamples / 8;
        unsigned int high[PER];
#pragma unroll
        for (int u = 0; u < PER; ++u)
            high[u] = line < p.lines && p.g.exponent ? static_cast<unsigned int>(__double2hiint(p.X[line + (warp * PER + u) * k / kSamples * p.ldx])) & 0x7FFFFFFFu : 0u;
#pragma unroll
        for (int u = 0; u < PER; ++u) top = max(top, high[u]);
#pragma unroll
        for (int u = 0; u < PER; ++u) below += distance(high[u], top);
        tops[warp][lane] = top;
        belows[warp][lane] = below;
        __syncthreads();
        if (warp != 0) return;
#pragma unroll
        for (int w = 1; w < 8; ++w) top = max(top, tops[w][lane]);
        below = 0u;
#pragma unroll
        for (int w = 0; w < 8; ++w) below += belows[w][lane] + (belows[w][lane] >> 16) * min((top >> 20) - (tops[w][lane] >> 20), 15u);
        below = (below >> 16 << 20) + (below & 0xFFFFu);           // of a line at most 32 samples, 960
        below = __reduce_add_sync(0xFFFFFFFFu, below);
        below = (below >> 20) * kWide0 <= (below & 0xFFFFFu) * 8u ? 1u : 0u;
    } else {
        line = static_cast<int64_t>(blockIdx.x - blocksA) * 8 + warp;
        static_assert(kSamples == 32, "one sample a lane, four in a sector");
        const unsigned int high = line < p.lines && p.g.exponent ? static_cast<unsigned int>(__double2hiint(p.X[(lane >> 2) * k / 8 + (lane & 3) + line * p.ldx])) & 0x7FFFFFFFu : 0u;
        top = __reduce_max_sync(0xFFFFFFFFu, high);
        below = __reduce_add_sync(0xFFFFFFFFu, distance(high, top));
        if (lane != 0) return;
        below = (below >> 16) * kWide1 <= (below & 0xFFFFu) * 8u ? 1u : 0u;
    }
    if (line >= p.lines) return;
    p.s.sumsq[line] = 0ull;
    p.s.emax[line] = INT32_MIN;
    p.s.nonfinite[line] = 0;
    if (!p.g.exponent) return;
    const int E = static_cast<int>(top >> 20) - 1023;
    // 2^(9 - E) a normal number, as the sums' fast form needs it; no guess from zeros and subnormals, Inf or NaN
    p.g.exponent[line] = below == 0u && top >= 0x00100000u && top < 0x7FF00000u && 9 - E >= -1000 && 9 - E <= 1000 - kGuesses ? E : INT32_MIN;
#pragma unroll
    for (int c = 0; c < kGuesses; ++c) {
        p.g.sumsq[c * p.lines + line] = 0ull;
        p.g.l1[c * p.lines + line] = 0u;
    }
}

// of squares up to 2^20, at most n of them: below 4096 in one word
__device__ __forceinline__ unsigned long long warp_sum(unsigned long long v, int64_t n)
{
    if (n < 4096) return __reduce_add_sync(0xFFFFFFFFu, static_cast<unsigned int>(v));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}

// One pass over the operand.  PASS 0: largest exponent + non-finite flag.  PASS 1: sum of squares, of the lines whose exponent was not guessed.
// PASS 2: pass 0 and the sums for every guess.
// side 0: thread = line, loop over a k-range (loads coalesced across lines).
// side 1: warp = line, lanes stride over a k-range (loads coalesced along k), shuffle reduction.
template <int SIDE, int PASS>
__device__ __forceinline__ void scan_block(const ScanSide &p, int64_t k, uint32_t block)
{
    const double *__restrict__ X = p.X;
    const ScanScratch &s = p.s;
    const int64_t ldx = p.ldx, lines = p.lines;
    const uint32_t kb0 = block / p.line_blocks, lb = block - kb0 * p.line_blocks;
    int64_t k0 = static_cast<int64_t>(kb0) * p.kspan;
    int64_t k1 = k0 + p.kspan < k ? k0 + p.kspan : k;
    int lane = threadIdx.x & 31;
    int64_t line;
    int64_t kstart, kstep;
    if (SIDE == 0) {
        line = lb * 256ll + threadIdx.x;
        kstart = k0;
        kstep = 1;
    } else {
        line = lb * 8ll + (threadIdx.x >> 5);
        kstart = k0 + lane;
        kstep = 32;
    }
    bool live = line < lines;
    int emax = INT32_MIN;
    unsigned int top = 0u;        // PASS 0, 2: largest high word of |x|
    unsigned long long acc = 0;
    unsigned int l1 = 0;          // sum of the magnitudes abar <= 2^10 (exponent-span check): below 2^30 for k <= 2^20
    int E = 0;
    if (PASS == 1 && live) {
        E = s.nonfinite[line] < 0 ? INT32_MIN : s.emax[line];      // INT32_MIN: nothing to add
        if (p.g.exponent && guessed(E, p.g.exponent[line])) live = false;
    }
    if (PASS == 2) E = live && p.g.exponent ? p.g.exponent[line] : INT32_MIN;
    const unsigned int beyond = E == INT32_MIN ? 0u : static_cast<unsigned int>(E + 1023 + kGuesses) << 20;       // PASS 2: above the guesses
    unsigned long long sums[kGuesses] = {};
    unsigned int l1s[kGuesses] = {};
    // 2^(9-E) as a double, when it is a normal number (not for lines of subnormals only)
    const bool fast_scale = PASS >= 1 && E != INT32_MIN && 9 - E >= -1000 && 9 - E <= 1000;
    const double scale9 = __hiloint2double((1023 + (fast_scale ? 9 - E : 0)) << 20, 0);
    if (live && !(PASS == 1 && E == INT32_MIN)) {
        // batches of 8 independent loads keep enough bytes in flight to run at memory speed
        for (int64_t kb = kstart; kb < k1; kb += 8 * kstep) {
            double xs[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                int64_t kk = kb + u * kstep;
                xs[u] = kk < k1 ? *element(X, ldx, SIDE, line, kk) : 0.0;
            }
            if (PASS != 1) {
#pragma unroll
                for (int u = 0; u < 8; ++u) top = max(top, static_cast<unsigned int>(__double2hiint(xs[u])) & 0x7FFFFFFFu);
            }
            if (PASS == 2) {
                if (top < beyond) {
                    // what is added for a guess below the line's exponent may wrap and is never read
                    unsigned int part[kGuesses] = {};
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const unsigned int abar = magnitude(xs[u], scale9);
#pragma unroll
                        for (int c = 0; c < kGuesses; ++c) {
                            const unsigned int half = (abar + ((1u << c) - 1u)) >> c;
                            part[c] += half * half;
                            l1s[c] += half;
                        }
                    }
#pragma unroll
                    for (int c = 0; c < kGuesses; ++c) sums[c] += part[c];
                }
            } else if (PASS == 1) {
                unsigned int part = 0u;           // eight terms of at most 2^20
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const double x = xs[u];
                    unsigned int abar;
                    if (fast_scale) {
                        abar = magnitude(x, scale9);
                    } else {
                        abar = scaled_magnitude(x, E);
                    }
                    part += abar * abar;
                    l1 += abar;
                }
                acc += part;
            }
        }
    }
    if (PASS != 1) {
        // The high words order like the exponents; where only zeros and subnormals were seen, the exponents come
        // from the whole words.
        if (SIDE == 1) top = __reduce_max_sync(0xFFFFFFFFu, top);
        if (top >= 0x00100000u) {
            emax = static_cast<int>(top >> 20) - 1023;
        } else if (live) {
            // (zeros in every tenth row of A, 131072 x 4096: one load at a time 6579 us a deconstruction, by eight 5355)
            for (int64_t kb = kstart; kb < k1; kb += 8 * kstep) {
                double xs[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) xs[u] = kb + u * kstep < k1 ? *element(X, ldx, SIDE, line, kb + u * kstep) : 0.0;
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    int e;
                    if (classify(xs[u], &e) == 1 && e > emax) emax = e;
                }
            }
            if (SIDE == 1) emax = __reduce_max_sync(0xFFFFFFFFu, emax);
        }
    } else if (SIDE == 1) {
        acc = warp_sum(acc, p.kspan);
        l1 = __reduce_add_sync(0xFFFFFFFFu, l1);
    }
    const bool reached = PASS == 2 && top < beyond;       // (side 1: by the whole warp) a guess may hold
    if (SIDE == 1 && reached) {
#pragma unroll
        for (int c = 0; c < kGuesses; ++c) {
            sums[c] = warp_sum(sums[c], p.kspan);
            l1s[c] = __reduce_add_sync(0xFFFFFFFFu, l1s[c]);
        }
    }
    if (!live || (SIDE == 1 && lane != 0)) return;
    if (reached) {
#pragma unroll
        for (int c = 0; c < kGuesses; ++c)
            if (sums[c]) {
                atomicAdd(&p.g.sumsq[c * lines + line], sums[c]);
                atomicAdd(&p.g.l1[c * lines + line], l1s[c]);
            }
    }
    if (PASS != 1) {
        if (top >= 0x7FF00000u) atomicOr(&s.nonfinite[line], kNonfiniteBit);
        else if (emax != INT32_MIN) atomicMax(&s.emax[line], emax);
    } else if (acc) {
        atomicAdd(&s.sumsq[line], acc);
        atomicAdd(&s.nonfinite[line], static_cast<int>(l1));     // never reaches bit 31
    }
}

template <int PASS>
__global__ void __launch_bounds__(256)
scan_kernel(const __grid_constant__ ScanSide a, const __grid_constant__ ScanSide b, int64_t k)
{
    dependency_release();
    dependency_wait();
    if (blockIdx.x < a.blocks) scan_block<0, PASS>(a, k, blockIdx.x);
    else scan_block<1, PASS>(b, k, blockIdx.x - a.blocks);
}

// Largest p with 4^p S <= G^2 (S = sum of squares > 0, G^2 as two words): from the bit lengths, and one comparison.
__device__ __forceinline__ int norm_exponent(unsigned long long S, unsigned long long g2lo, unsigned long long g2hi)
{
    const int bits_g = g2hi ? 128 - __clzll(static_cast<long long>(g2hi)) : 64 - __clzll(static_cast<long long>(g2lo));
    const int p = (bits_g - (64 - __clzll(static_cast<long long>(S)))) >> 1;      // G^2 has at least as many bits as S
    const unsigned __int128 scaled = static_cast<unsigned __int128>(S) << (2 * p);
    const unsigned __int128 G2 = (static_cast<unsigned __int128>(g2hi) << 64) | g2lo;
    return scaled <= G2 ? p : p - 1;
}

// Flatness of a line, floor(2^16 l1^2 / (k S)), at most 2^16 since l1^2 <= k S (l1 < 2^30, S <= 2^40): the quotient of
// the rounded FP64 values is off by less than 2^-30 of one, so the exact floor is its integer part or a neighbour.
__device__ __forceinline__ unsigned int line_flatness(unsigned int l1, unsigned long long S, int64_t k)
{
    const unsigned __int128 num = static_cast<unsigned __int128>(static_cast<unsigned long long>(l1) * l1) << 16;
    const unsigned long long den = static_cast<unsigned long long>(k) * S;
    const double approx = static_cast<double>(static_cast<unsigned long long>(l1) * l1) * 65536.0 / static_cast<double>(den);
    unsigned long long q = static_cast<unsigned long long>(approx);
    if (static_cast<unsigned __int128>(q) * den > num) --q;
    else if (static_cast<unsigned __int128>(q + 1) * den <= num) ++q;
    return static_cast<unsigned int>(q);
}

// shift[line]: MAXEXP  t - 1 - E;  CS  p + 9 - E with p the largest integer such that
// 4^p * S <= G^2  (G^2 passed as two 64-bit words).
struct FinalizeSide {
    ScanScratch s;
    int64_t lines;
    int tbits;
    int32_t *shift;
    ScanGuess g;
};
__global__ void scan_finalize_kernel(const __grid_constant__ FinalizeSide a, const __grid_constant__ FinalizeSide b, int64_t k, int rule,
                                     unsigned long long g2lo, unsigned long long g2hi,
                                     unsigned int esc_threshold, unsigned int *status)
{
    dependency_release();
    dependency_wait();
    int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
    const int side = i < a.lines ? 0 : 1;
    if (side) i -= a.lines;
    const ScanScratch s = side ? b.s : a.s;
    int32_t *shift = side ? b.shift : a.shift;
    unsigned int flatness = 0xFFFFFFFFu;
    bool bad = false;
    if (i < (side ? b.lines : a.lines)) {
        const int E = s.emax[i];
        bad = s.nonfinite[i] < 0;
        if (bad) {
            shift[i] = OZ_NONFINITE_SHIFT;
        } else if (E == INT32_MIN) {
            shift[i] = 0;
        } else if (rule == 0) {
            shift[i] = (side ? b.tbits : a.tbits) - 1 - E;
        } else {
            const ScanGuess g = side ? b.g : a.g;
            if (g.exponent && guessed(E, g.exponent[i])) {       // the sums of the guess go where those of a second pass would be
                const int64_t at = (E - g.exponent[i]) * (side ? b.lines : a.lines) + i;
                s.sumsq[i] = g.sumsq[at];
                s.nonfinite[i] = static_cast<int>(g.l1[at]);
            }
            shift[i] = norm_exponent(s.sumsq[i], g2lo, g2hi) + 9 - E;
            flatness = line_flatness(static_cast<unsigned int>(s.nonfinite[i]), s.sumsq[i], k);
        }
    }
    // Exponent-span check (Algorithm 1, "ESC check"): the smallest flatness of each operand's lines is kept in
    // the device status block and judged against the set's threshold when the status is queried.  One update a warp and side: a
    // warp may hold lines of both, and its lanes would queue up at the two words (8000 lines: 8.6 us, 4.4 with one update).
    const unsigned int qa = __reduce_min_sync(0xFFFFFFFFu, side ? 0xFFFFFFFFu : flatness);
    const unsigned int qb = __reduce_min_sync(0xFFFFFFFFu, side ? flatness : 0xFFFFFFFFu);
    bad = __any_sync(0xFFFFFFFFu, bad);
    if ((threadIdx.x & 31) == 0) {
        if (bad) atomicOr(status, 1u << OZ_ERR_NONFINITE_INPUT);
        if (qa != 0xFFFFFFFFu) atomicMin(status + 1, qa);
        if (qb != 0xFFFFFFFFu) atomicMin(status + 2, qb);
        if (min(qa, qb) != 0xFFFFFFFFu) status[3] = esc_threshold;
    }
}

// ---- out-of-range rows (Algorithm 1, last line; Algorithm 3, "ESC range check; re-issue out-of-range
// rows on the native-FP64 path") ------------------------------------------------------------------
// flatness of one scanned line from its norm sums, capped at 2^16; 0xFFFFFFFF for a line that does
// not count (zeros only, or Inf/NaN)
__device__ __forceinline__ unsigned int scanned_flatness(const ScanScratch &s, int64_t i, int64_t k)
{
    const int nf = s.nonfinite[i];
    if (nf < 0 || s.emax[i] == INT32_MIN) return 0xFFFFFFFFu;
    const unsigned int q = line_flatness(static_cast<unsigned int>(nf), s.sumsq[i], k);
    return q > 65536u ? 65536u : q;
}

// One block.  Row i of the product is re-issued when q(a_i) * min_j q(b_j) < threshold.  Writes the
// flag of every row, the re-issued rows in ascending order, their number, and adds that number to the
// device status block (word 4).
__global__ void __launch_bounds__(1024)
esc_rows_kernel(ScanScratch sA, int64_t m, ScanScratch sB, int64_t n, int64_t k, unsigned int threshold,
                unsigned char *flag, int *list, unsigned int *count, unsigned int *status)
{
    __shared__ unsigned int red[32];
    __shared__ unsigned int base;
    dependency_release();
    dependency_wait();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    unsigned int qb = 0xFFFFFFFFu;
    for (int64_t j = tid; j < n; j += blockDim.x) qb = min(qb, scanned_flatness(sB, j, k));
    qb = __reduce_min_sync(0xFFFFFFFFu, qb);
    if (lane == 0) red[warp] = qb;
    if (tid == 0) base = 0u;
    __syncthreads();
    qb = red[lane];
    qb = __reduce_min_sync(0xFFFFFFFFu, qb);
    if (qb > 65536u) qb = 65536u;
    __syncthreads();
    for (int64_t i0 = 0; i0 < m; i0 += blockDim.x) {
        const int64_t i = i0 + tid;
        bool out = false;
        if (i < m) {
            const unsigned int qa = scanned_flatness(sA, i, k);
            out = qa != 0xFFFFFFFFu && static_cast<unsigned long long>(qa) * qb < threshold;
            flag[i] = out ? 1 : 0;
        }
        // ordered compaction: position = rows re-issued so far + those of lower threads
        const unsigned int ballot = __ballot_sync(0xFFFFFFFFu, out);
        if (lane == 0) red[warp] = __popc(ballot);
        __syncthreads();
        unsigned int before = base;
        for (int w = 0; w < warp; ++w) before += red[w];
        if (out) list[before + __popc(ballot & ((1u << lane) - 1u))] = static_cast<int>(i);
        __syncthreads();
        if (tid == 0) {
            unsigned int total = 0;
            for (int w = 0; w < 32; ++w) total += red[w];
            base += total;
        }
        __syncthreads();
    }
    if (tid == 0) {
        *count = base;
        if (base) atomicAdd(status + 4, base);
    }
}

// ---- accurate mode (Sec. 2 "The FP8 variant": the additional FP8 product that estimates a
// magnitude bound, the "+1" of the 3r + 1 schedule) ------------------------------------------
// Magnitude digit of one element: the smallest integer of the E4M3 grid {0..16, 18, 20, .., 32} that
// is >= |x| 2^(4-E), E the largest exponent of the line; integer arithmetic on the bit pattern.
__device__ __noinline__ uint32_t bound_digit_exact(double x, int E)
{
    unsigned long long bits = static_cast<unsigned long long>(__double_as_longlong(x));
    int be = static_cast<int>((bits >> 52) & 0x7FF);
    unsigned long long frac = bits & 0xFFFFFFFFFFFFFull;
    if (be == 0x7FF || (be == 0 && frac == 0)) return 0u;
    unsigned long long sig = be ? (frac | (1ull << 52)) : frac;
    int ex = be ? be - 1023 : -1022;
    int sh = 48 + E - ex;                                 // |x| 2^(4-E) = sig / 2^sh
    unsigned long long g;
    if (sh >= 64) g = 1ull;
    else if (sh <= 0) g = sig << (-sh);
    else g = (sig >> sh) + ((sig & ((1ull << sh) - 1ull)) ? 1ull : 0ull);
    uint32_t d = static_cast<uint32_t>(g);
    if (d > 16u && (d & 1u)) ++d;                         // above 16 the grid holds the even integers
    return d;
}

// What a line's digits are made with: dead (a line of zeros, or with Inf/NaN) gives zeros
struct BoundLine {
    int E;
    bool dead, fast;
    double scale;
};
__device__ __forceinline__ BoundLine bound_line(const ScanScratch &s, int64_t line, bool live)
{
    BoundLine b;
    b.E = live ? s.emax[line] : INT32_MIN;
    b.dead = !live || b.E == INT32_MIN || s.nonfinite[line] < 0;
    const int up = b.dead ? 0 : 4 - b.E;                  // (no sum with the mark of a line of zeros)
    b.fast = up >= -1000 && up <= 1000;                   // 2^(4-E) as a double
    b.scale = __hiloint2double((1023 + (b.fast ? up : 0)) << 20, 0);
    return b;
}
__device__ __forceinline__ uint32_t bound_digit(double x, const BoundLine &b)
{
    if (!b.fast) return bound_digit_exact(x, b.E);
    const uint32_t d = magnitude(x, b.scale);
    return d > 16u ? (d + 1u) & ~1u : d;
}

// One byte per element: the E4M3 code of its magnitude digit, K-major like the residue planes
// (out[line * pitch + kk]; bytes kk in [k, pitch) are zero), both operands in one launch.  A block takes 32 lines x 64 inner
// indices of side 0, loaded along the lines, or 8 lines x 256 of side 1, one line a warp; the bytes go through shared memory
// so that pieces of 64 and 256 bytes are stored.  (18 + 16 us for two 2048 x 2048 operands when the digits were 64-bit shifts, their
// codes came from constant memory at divergent addresses and a thread had four elements between two barriers.)
struct BoundSide {
    const double *X;
    int64_t ldx, lines;
    ScanScratch s;
    uint8_t *out;
    uint32_t blocks;
};
__global__ void __launch_bounds__(256)
bound_plane_kernel(const __grid_constant__ BoundSide a, const __grid_constant__ BoundSide b, int64_t k, int64_t pitch)
{
    __shared__ __align__(16) unsigned char tile[32 * 80];        // 64 bytes a row, padded; side 1: 256 bytes a warp
    dependency_release();
    dependency_wait();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto code2 = [](uint32_t d0, uint32_t d1) { return e4m3_pair(make_float2(static_cast<float>(d0), static_cast<float>(d1))); };
    if (blockIdx.x < a.blocks) {
        const uint32_t ltiles = static_cast<uint32_t>((a.lines + 31) / 32), kc = blockIdx.x / ltiles;
        const int64_t line0 = static_cast<int64_t>(blockIdx.x - kc * ltiles) * 32, line = line0 + lane, k0 = static_cast<int64_t>(kc) * 64;
        const BoundLine bl = bound_line(a.s, line, line < a.lines);
        double x[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int64_t kk = k0 + 8 * warp + u;
            x[u] = !bl.dead && kk < k ? a.X[line + kk * a.ldx] : 0.0;
        }
        uint32_t w[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) w[u] = code2(bound_digit(x[2 * u], bl), bound_digit(x[2 * u + 1], bl));
        *reinterpret_cast<uint2 *>(tile + lane * 80 + 8 * warp) = make_uint2(w[0] | (w[1] << 16), w[2] | (w[3] << 16));
        __syncthreads();
        const int lr = threadIdx.x >> 3, kq = (threadIdx.x & 7) * 8;
        const int64_t oline = line0 + lr, okk = k0 + kq;
        if (oline < a.lines && okk < pitch)      // a pitch is a multiple of 16
            *reinterpret_cast<uint2 *>(a.out + oline * pitch + okk) = *reinterpret_cast<const uint2 *>(tile + lr * 80 + kq);
    } else {
        const uint32_t block = blockIdx.x - a.blocks, kchunks = static_cast<uint32_t>((pitch + 255) / 256), lt = block / kchunks;
        const int64_t line = static_cast<int64_t>(lt) * 8 + warp, k0 = static_cast<int64_t>(block - lt * kchunks) * 256;
        if (line >= b.lines) return;
        const BoundLine bl = bound_line(b.s, line, true);
        const double *src = b.X + line * b.ldx;
        double x[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int64_t kk = k0 + lane + 32 * u;
            x[u] = !bl.dead && kk < k ? src[kk] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < 8; u += 2) {
            const uint32_t w = code2(bound_digit(x[u], bl), bound_digit(x[u + 1], bl));
            tile[warp * 256 + lane + 32 * u] = static_cast<unsigned char>(w);
            tile[warp * 256 + lane + 32 * u + 32] = static_cast<unsigned char>(w >> 8);
        }
        __syncwarp();
        if (k0 + 8 * lane < pitch)
            *reinterpret_cast<uint2 *>(b.out + line * pitch + k0 + 8 * lane) = *reinterpret_cast<const uint2 *>(tile + warp * 256 + 8 * lane);
    }
}

// shift[line] of the accurate rule from the line's maximum of the bound product (the bit pattern of
// a non-negative integer-valued float, accumulated with atomicMax in the low word of sumsq[line]):
//   ((L - ceil(log2 max)) >> 1) + 4 - E
__global__ void accurate_finalize_kernel(const __grid_constant__ FinalizeSide a, const __grid_constant__ FinalizeSide b, int L,
                                         unsigned int *status)
{
    dependency_release();
    dependency_wait();
    int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
    const bool side = i >= a.lines;
    if (side) i -= a.lines;
    const ScanScratch s = side ? b.s : a.s;
    int32_t *shift = side ? b.shift : a.shift;
    if (i >= (side ? b.lines : a.lines)) return;
    if (s.nonfinite[i] < 0) {
        shift[i] = OZ_NONFINITE_SHIFT;
        atomicOr(status, 1u << OZ_ERR_NONFINITE_INPUT);
        return;
    }
    const int E = s.emax[i];
    if (E == INT32_MIN) { shift[i] = 0; return; }
    const uint32_t v = static_cast<uint32_t>(__uint_as_float(static_cast<uint32_t>(s.sumsq[i])));
    const int clog = v <= 1u ? 0 : 32 - __clz(static_cast<int>(v - 1u));
    shift[i] = ((L - clog) >> 1) + 4 - E;
}

// 2 NP consecutive inner-dimension elements of one line -> 2 NP bytes of every stored plane.
template <int SET, int LAYOUT, int NP, class Table>
__device__ __forceinline__ void convert(const double (&x)[2 * NP], int sigma, bool tz, const Table &lut, uint8_t *out,
                                        int64_t plane_stride)
{
    Limbs<NP> L;
    split_limbs<NP>(x, sigma, tz, L);
    convert_all_moduli<SET, LAYOUT>(std::make_integer_sequence<int, set_r(SET)>{}, L, lut, out, plane_stride);
}

// copies the digit table to shared memory (16-byte pieces)
template <int SET, int LAYOUT>
__device__ __forceinline__ void load_table(uint32_t *lut, const uint32_t *__restrict__ lut_global, int tid, int nthreads)
{
    for (int i = tid; i < lut_words_of(SET, LAYOUT) / 4; i += nthreads)
        reinterpret_cast<uint4 *>(lut)[i] = reinterpret_cast<const uint4 *>(lut_global)[i];
}

// Side 1: 16-byte chunk of a tile row that holds the element pair c: the eight lanes of a quarter warp, which read
// chunks 4 l + e or 8 l + e (l = 0..7), then hit eight different bank groups
__device__ __forceinline__ int tile_chunk(int c) { return c ^ ((c >> 3) & 7); }

// Whether an operand's elements may travel two at a time: 16-byte aligned columns
__host__ __device__ inline bool element_pairs(const double *X, int64_t ldx)
{
    return (ldx & 1) == 0 && (reinterpret_cast<uintptr_t>(X) & 15u) == 0;
}

// asynchronous copies of one (8 bytes) or two (16 bytes) elements; nothing is read and zeros are written for bytes = 0
__device__ __forceinline__ void copy8(uint32_t dst, const double *src, bool live)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(live ? 8 : 0) : "memory");
}
__device__ __forceinline__ void copy16(uint32_t dst, const double *src, int bytes)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void copy16(uint32_t dst, const double *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

// The block's copies of a tile of 16 lines x 128 inner indices; what lies beyond the lines or beyond k becomes zeros.
// Side 0 keeps a tile as [index in an octet][octet][line], 128 bytes a row, the 16-byte pieces of a row XORed with half the
// octet's number: two lines travel in one copy, and neither the copies nor the reads, of one or two octets at compile-time
// offsets from one address, conflict.
__device__ __forceinline__ void request_side0(const double *__restrict__ X, int64_t ldx, int64_t lines, int64_t k, bool pairs,
                                              int64_t line0, int64_t k0, uint32_t base)
{
    if (pairs) {
        // a thread copies lines 2c, 2c + 1 of inner indices kq + 32 u, octets kq / 8 + 4 u
        const int c = threadIdx.x & 7, kq = threadIdx.x >> 3;
        const uint32_t dst = base + ((kq & 7) * 16 + (kq >> 3)) * 128 + ((c ^ (kq >> 4)) << 4);
        const double *src = X + line0 + 2 * c + (k0 + kq) * ldx;
        if (line0 + kTileLines <= lines && k0 + kChunk <= k) {
#pragma unroll
            for (int u = 0; u < 4; ++u) copy16((dst ^ (u << 5)) + u * 512, src + 32 * u * ldx);
        } else {
            const int64_t left = lines - (line0 + 2 * c);
            const int bytes = left >= 2 ? 16 : (left == 1 ? 8 : 0);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const bool in = bytes && k0 + kq + 32 * u < k;
                copy16((dst ^ (u << 5)) + u * 512, in ? src + 32 * u * ldx : X, in ? bytes : 0);
            }
        }
    } else {
        // line l of inner indices kq + 16 u, octets kq / 8 + 2 u
        const int l = threadIdx.x & 15, kq = threadIdx.x >> 4;
        const uint32_t dst = base + ((kq & 7) * 16 + (kq >> 3)) * 128 + ((l >> 1) << 4) + (l & 1) * 8;
        const double *src = X + line0 + l + (k0 + kq) * ldx;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const bool in = line0 + l < lines && k0 + kq + 16 * u < k;
            copy8((dst ^ (u << 4)) + u * 256, in ? src + 16 * u * ldx : X, in);
        }
    }
}
// side 1: a warp copies one row, 128 elements of a line
__device__ __forceinline__ void request_row(const double *__restrict__ X, int64_t ldx, int64_t lines, int64_t k, bool pairs,
                                            int64_t line, int64_t k0, uint32_t row)
{
    const int lane = threadIdx.x & 31;
    const bool live = line < lines;
    const int kleft = static_cast<int>(k - k0 < kChunk ? k - k0 : kChunk);        // <= 0: padding only
    const double *src = X + (live ? line : 0) * ldx + k0;
    if (pairs) {
#pragma unroll
        for (int u = 0; u < kChunk / 64; ++u) {
            const int c = lane + 32 * u;
            if (live && kleft == kChunk) {
                copy16(row + tile_chunk(c) * 16, src + 2 * c);
            } else {
                const int left = live ? (kleft - 2 * c) * 8 : 0;
                const int bytes = left >= 16 ? 16 : (left > 0 ? left : 0);
                copy16(row + tile_chunk(c) * 16, bytes ? src + 2 * c : X, bytes);
            }
        }
    } else {
#pragma unroll
        for (int u = 0; u < kChunk / 32; ++u) {
            const int kk = lane + 32 * u;
            const bool in = live && kk < kleft;
            copy8(row + tile_chunk(kk >> 1) * 16 + (kk & 1) * 8, in ? src + kk : X, in);
        }
    }
}
// this thread's eight elements of a tile: line 2 warp + lane / 16, octet lane % 16
template <int SIDE>
__device__ __forceinline__ void tile_octet(const unsigned char *tile, double (&x)[8])
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, oct = lane & 15;
    if constexpr (SIDE == 0) {
        const double *src = reinterpret_cast<const double *>(tile + oct * 128 + ((warp ^ (oct >> 1)) << 4)) + (lane >> 4);
#pragma unroll
        for (int e = 0; e < 8; ++e) x[e] = src[e * 256];
    } else {
        const double2 *row = reinterpret_cast<const double2 *>(tile + (warp * 2 + (lane >> 4)) * kTileRow);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const double2 v = row[tile_chunk(oct * 4 + e)];
            x[2 * e] = v.x;
            x[2 * e + 1] = v.y;
        }
    }
}

// two consecutive octets of a tile: the same line, octets 2 j and 2 j + 1
template <int SIDE>
__device__ __forceinline__ void tile_octets(const unsigned char *tile, int j, double (&x)[16])
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if constexpr (SIDE == 0) {
        const double *src = reinterpret_cast<const double *>(tile + j * 256 + ((warp ^ j) << 4)) + (lane >> 4);
#pragma unroll
        for (int e = 0; e < 16; ++e) x[e] = src[(e & 7) * 256 + (e >> 3) * 16];
    } else {
        const double2 *row = reinterpret_cast<const double2 *>(tile + (warp * 2 + (lane >> 4)) * kTileRow);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const double2 v = row[tile_chunk(j * 8 + e)];
            x[2 * e] = v.x;
            x[2 * e + 1] = v.y;
        }
    }
}

// A block takes tiles of 16 lines x 128 inner indices through shared memory (on side 0 that is the
// transposition: loads run along the lines, plane stores along k) and a thread converts eight consecutive
// elements of one line, so that half a warp stores 128 contiguous bytes of every plane.  The next tile's
// elements are copied asynchronously while this one is converted.  BY_LINE (side 1, planes kept line by line): the 16 rows
// of a tile are consecutive 128-element pieces of a line, and of the next lines behind it, so that a tile stores 2 KiB at
// a time in that layout too.
// Bound: with digit planes DRAM (32768 x 1024, set S on FP8, side 0: 251 us, 243 with the arithmetic left out: 38 bytes an element at
// 5.1 TB/s), on native residues instruction issue and the FP32 pipe (60 % busy each; 184 us against 131), and, line by line
// on side 0, the planes' scattered 128-byte writes.  What surrounds the arithmetic was a third of the instructions: tiles are
// numbered without divisions, shifts are loaded with the elements, whole tiles are copied without a test.  147 -> 127
// thread-instructions per element of A on set S, 125 -> 105 on native residues (205 -> 184 us).
template <int SET, int SIDE, int LAYOUT, bool BY_LINE>
__global__ void __launch_bounds__(kConvThreads, conv_blocks(LAYOUT))
convert_kernel(const double *__restrict__ X, int64_t ldx, int64_t lines, int64_t k,
               const int32_t *__restrict__ shift, const uint32_t *__restrict__ lut_global,
               uint8_t *__restrict__ planes, const __grid_constant__ PlaneGeom geom, int tz)
{
    const int64_t row_pitch = geom.row_pitch;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    uint32_t *lut = reinterpret_cast<uint32_t *>(smem_raw + 2 * kTileBytes);
    const uint32_t lut_addr = static_cast<uint32_t>(__cvta_generic_to_shared(lut));
    const uint32_t tile_addr = static_cast<uint32_t>(__cvta_generic_to_shared(smem_raw));
    dependency_release();
    load_table<SET, LAYOUT>(lut, lut_global, threadIdx.x, kConvThreads);      // written once, before any call
    dependency_wait();

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // work items are numbered in 32 bits (checked on the host)
    const uint32_t nchunks = static_cast<uint32_t>((row_pitch + kChunk - 1) / kChunk);
    const uint32_t ltiles = static_cast<uint32_t>((lines + kTileLines - 1) / kTileLines);
    const uint32_t items = BY_LINE ? (static_cast<uint32_t>(lines) * nchunks + kTileLines - 1) / kTileLines : ltiles * nchunks;
    const bool pairs = element_pairs(X, ldx);
    const int li = warp * 2 + (lane >> 4), oct = lane & 15;        // this thread's line and octet of a tile (see tile_octet)

    // Position of a tile: slow index q (side 0: chunk, side 1: line tile) and fast index `rest`, so that neighbouring blocks
    // take neighbouring lines (side 0) or neighbouring inner indices; BY_LINE: line and chunk of this warp's first row.  A step
    // over the grid adds one constant to each, and one carry.
    const uint32_t fast_count = SIDE == 0 ? ltiles : nchunks;
    const uint32_t start = BY_LINE ? blockIdx.x * kTileLines + 2 * warp : blockIdx.x, step = BY_LINE ? gridDim.x * kTileLines : gridDim.x;
    uint32_t q = start / fast_count, rest = start - q * fast_count;
    const uint32_t dq = step / fast_count, dr = step - dq * fast_count;
    auto advance = [&] {
        q += dq;
        rest += dr;
        if (rest >= fast_count) {
            rest -= fast_count;
            ++q;
        }
    };
    // this thread's line and the first inner index of the tile (BY_LINE: of the row)
    auto place = [&](int64_t &line, int64_t &k0) {
        if constexpr (BY_LINE) {
            line = q;
            uint32_t chunk = rest;
            if ((lane >> 4) && ++chunk == nchunks) {      // the row behind: next piece of the line, or the next line
                chunk = 0;
                ++line;
            }
            k0 = static_cast<int64_t>(chunk) * kChunk;
        } else {
            line = static_cast<int64_t>(SIDE == 0 ? rest : q) * kTileLines + li;
            k0 = static_cast<int64_t>(SIDE == 0 ? q : rest) * kChunk;
        }
    };
    // elements of a tile; rows beyond the lines and inner indices beyond k become zeros
    auto request = [&](int buf) {
        const uint32_t base = tile_addr + buf * kTileBytes;
        if constexpr (SIDE == 0) {
            request_side0(X, ldx, lines, k, pairs, static_cast<int64_t>(rest) * kTileLines, static_cast<int64_t>(q) * kChunk, base);
        } else {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                int64_t line, k0;
                if constexpr (BY_LINE) {
                    line = q;
                    uint32_t chunk = rest;
                    if (h && ++chunk == nchunks) {
                        chunk = 0;
                        ++line;
                    }
                    k0 = static_cast<int64_t>(chunk) * kChunk;
                } else {
                    line = static_cast<int64_t>(q) * kTileLines + warp * 2 + h;
                    k0 = static_cast<int64_t>(rest) * kChunk;
                }
                request_row(X, ldx, lines, k, pairs, line, k0, base + (warp * 2 + h) * kTileRow);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };

    int buf = 0;
    int64_t line = 0, k0 = 0, next_line = 0, next_k0 = 0;
    int sigma = 0, next_sigma = 0;
    if (blockIdx.x < items) {
        place(line, k0);
        request(0);
        sigma = line < lines ? shift[line] : 0;
    }
    for (uint32_t item = blockIdx.x; item < items; item += gridDim.x, buf ^= 1) {
        const bool more = items - item > gridDim.x;
        if (more) {
            advance();
            place(next_line, next_k0);
            request(buf ^ 1);
            next_sigma = next_line < lines ? shift[next_line] : 0;
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();                 // this tile (and, the first time, the table) is there
        if (line < lines && k0 + oct * 8 < row_pitch) {
            double x[8];
            tile_octet<SIDE>(smem_raw + buf * kTileBytes, x);
            if (sigma == OZ_NONFINITE_SHIFT) {       // its planes are zeros
                sigma = 0;
#pragma unroll
                for (int e = 0; e < 8; ++e) x[e] = 0.0;
            }
            convert<SET, LAYOUT, 4>(x, sigma, tz != 0, NearTable{lut_addr},
                                 planes + (k0 >> 7) * geom.chunk_stride + line * geom.line_stride + oct * 8, geom.plane_stride);
        }
        __syncthreads();                 // the tile may be overwritten
        line = next_line;
        k0 = next_k0;
        sigma = next_sigma;
    }
}

// ---- whole deconstruction of a group of lines in one kernel ------------------------------------
// When a few whole lines fit in shared memory next to the look-up table, a thread block loads them
// once and takes everything from there: largest exponent, the norm sums, the shift, and the
// conversion into planes.  The operand is then read from HBM once (8 bytes per element instead of
// 24 with the three-pass kernels above) and one launch replaces five.  The arithmetic is the same,
// function by function, so the outputs are identical; the sums are integers, hence independent of
// the order in which the warps add them.  Not for the accurate rule, whose shifts need the other
// operand.
struct FusedParams {
    const double *X;
    int64_t ldx, lines, k;
    int group;                 // lines per thread block pass
    int pitch;                 // doubles per line in shared memory: odd (conflict-free across lines)
    int side, rule, tbits, tz;
    unsigned long long g2lo, g2hi;
    unsigned int esc_threshold;
    const uint32_t *lut_global;
    uint8_t *planes;
    PlaneGeom geom;
    int32_t *shift;
    unsigned int *status;
    ScanScratch scan;          // where the lines' scan results go as well, for the row check; null: nowhere
};

// a line's scan results, as the scan kernels leave them
__device__ __forceinline__ void keep_scan(const ScanScratch &s, int64_t line, unsigned long long sumsq, int emax, bool bad, unsigned int l1)
{
    if (!s.emax) return;
    s.sumsq[line] = sumsq;
    s.emax[line] = emax;
    s.nonfinite[line] = bad ? kNonfiniteBit : static_cast<int>(l1);
}

// position of inner index kk in a line's buffer: one spare double behind every eight, so that threads that read
// eight consecutive elements each (stride 9) touch all banks
__host__ __device__ constexpr int padded(int kk) { return kk + (kk >> 3); }
__host__ __device__ constexpr int fused_pitch(int k) { return padded(k) | 1; }

struct FusedLine {             // per-line results in shared memory
    unsigned long long sumsq;
    unsigned int top;          // largest high word of |x|
    int emax, shift;           // emax: of lines of zeros and subnormals only
    unsigned int l1;
    __device__ bool bad() const { return top >= 0x7FF00000u; }
    // largest exponent: the high words order like the exponents
    __device__ int exponent() const { return top >= 0x00100000u ? static_cast<int>(top >> 20) - 1023 : emax; }
    __device__ void clear()
    {
        sumsq = 0ull;
        top = 0u;
        emax = INT32_MIN;
        l1 = 0u;
    }
};

// The shift of a line from its scan results, with its contribution to the device status block
__device__ __forceinline__ int line_shift(const FusedParams &p, const FusedLine &r)
{
    if (r.bad()) {
        atomicOr(p.status, 1u << OZ_ERR_NONFINITE_INPUT);
        return OZ_NONFINITE_SHIFT;
    }
    const int emax = r.exponent();
    if (emax == INT32_MIN) return 0;
    if (p.rule == 0) return p.tbits - 1 - emax;
    atomicMin(p.status + 1 + p.side, line_flatness(r.l1, r.sumsq, p.k));
    p.status[3] = p.esc_threshold;
    return norm_exponent(r.sumsq, p.g2lo, p.g2hi) + 9 - emax;
}

// line groups block, block + nblocks, .. of one operand
template <int SET, int SIDE, int LAYOUT>
__device__ __forceinline__ void deconstruct_lines(const FusedParams &p, int block, int nblocks, unsigned char *smem_raw)
{
    uint32_t *lut = reinterpret_cast<uint32_t *>(smem_raw);
    const uint32_t lut_addr = static_cast<uint32_t>(__cvta_generic_to_shared(lut));
    double *buf = reinterpret_cast<double *>(smem_raw + lut_words_of(SET, LAYOUT) * 4);
    FusedLine *both = reinterpret_cast<FusedLine *>(buf + static_cast<size_t>(p.group) * p.pitch);      // 2 x 32, used in turn
    const int nthreads = blockDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = nthreads >> 5;
    dependency_release();
    load_table<SET, LAYOUT>(lut, p.lut_global, tid, nthreads);      // written once, before any call
    dependency_wait();
    const int64_t ngroups = (p.lines + p.group - 1) / p.group;
    const int k = static_cast<int>(p.k);
    if (tid < p.group) both[tid].clear();
    FusedLine *res = both;
    for (int64_t g = block; g < ngroups; g += nblocks) {
        const int64_t line0 = g * p.group;
        const int nl = static_cast<int>(p.lines - line0 < p.group ? p.lines - line0 : p.group);
        __syncthreads();                 // the previous group's conversion has finished with buf / res, this one's res is clear
        // ---- load: nl lines x k doubles, coalesced along the operand's leading dimension; the largest high word of |x| of
        // every line on the way
        if (SIDE == 0) {
            // element (line, kk) at X[line + kk ldx]: consecutive threads take consecutive lines
            // (the group size is a power of two on this side: a thread stays on one line)
            const int gshift = 31 - __clz(p.group), l = tid & (p.group - 1), kstep = nthreads >> gshift;
            unsigned int top = 0u;
            if (l < nl) {
                const double *src = p.X + line0 + l;
                double *dst = buf + l * p.pitch;
                for (int kk = tid >> gshift; kk < k; kk += 4 * kstep) {
                    double v[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) v[u] = kk + u * kstep < k ? src[static_cast<int64_t>(kk + u * kstep) * p.ldx] : 0.0;
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        if (kk + u * kstep < k) dst[padded(kk + u * kstep)] = v[u];
                        top = max(top, static_cast<unsigned int>(__double2hiint(v[u])) & 0x7FFFFFFFu);
                    }
                }
            }
            for (int o = p.group; o < 32; o <<= 1) top = max(top, __shfl_xor_sync(0xFFFFFFFFu, top, o));
            if (lane < p.group && top) atomicMax(&res[l].top, top);
        } else {
            // batches of independent loads: enough bytes in flight to run at memory speed
            for (int l0 = 0; l0 < nl; l0 += 4) {
                unsigned int top[4] = {0u, 0u, 0u, 0u};
                for (int kk = tid; kk < k; kk += nthreads) {
                    double v[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) v[u] = l0 + u < nl ? p.X[kk + (line0 + l0 + u) * p.ldx] : 0.0;
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        if (l0 + u < nl) buf[(l0 + u) * p.pitch + padded(kk)] = v[u];
                        top[u] = max(top[u], static_cast<unsigned int>(__double2hiint(v[u])) & 0x7FFFFFFFu);
                    }
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const unsigned int t = __reduce_max_sync(0xFFFFFFFFu, top[u]);
                    if (lane == 0 && l0 + u < nl && t) atomicMax(&res[l0 + u].top, t);
                }
            }
        }
        __syncthreads();
        FusedLine *next = res == both ? both + 32 : both;
        if (tid < p.group) next[tid].clear();
        // ---- the scans: a line is cut into `segs` pieces, one warp per piece
        const int segs = nwarps >= nl ? nwarps / nl : 1;
        const int span = (k + segs - 1) / segs;
        // lines of zeros and subnormals: exponents from the whole words
        if (__any_sync(0xFFFFFFFFu, lane < nl && res[lane].top < 0x00100000u)) {
            for (int item = warp; item < nl * segs; item += nwarps) {
                const int l = item / segs, seg = item - l * segs;
                const int k0 = seg * span, k1 = min(k, k0 + span);
                if (res[l].top >= 0x00100000u) continue;                 // warp-uniform
                int emax = INT32_MIN;
                for (int kk = k0 + lane; kk < k1; kk += 32) {
                    int e;
                    if (classify(buf[l * p.pitch + padded(kk)], &e) == 1 && e > emax) emax = e;
                }
                emax = __reduce_max_sync(0xFFFFFFFFu, emax);
                if (lane == 0 && emax != INT32_MIN) atomicMax(&res[l].emax, emax);
            }
            __syncthreads();
        }
        if (p.rule == 1) {
            for (int item = warp; item < nl * segs; item += nwarps) {
                const int l = item / segs, seg = item - l * segs;
                const int k0 = seg * span, k1 = min(k, k0 + span);
                const int E = res[l].exponent();
                if (E == INT32_MIN || res[l].bad()) continue;            // warp-uniform
                const bool fast_scale = 9 - E >= -1000 && 9 - E <= 1000;
                const double scale9 = __hiloint2double((1023 + (fast_scale ? 9 - E : 0)) << 20, 0);
                unsigned long long acc = 0ull;
                unsigned int l1 = 0u;
                const double *src = buf + l * p.pitch;
                if (fast_scale) {
                    // (left to itself the compiler unrolls the short body so far that small calls pay for its size: 64^3 from cold caches 11.0 us
                    // a deconstruction on set S, 12.2 on E, like this 9.4 and 10.6; 1000 x 1000 12.4 and 12.1)
#pragma unroll 2
                    for (int kk = k0 + lane; kk < k1; kk += 32) {
                        const unsigned int abar = magnitude(src[padded(kk)], scale9);
                        acc += abar * abar;                              // at most 2^20
                        l1 += abar;
                    }
                } else {
                    for (int kk = k0 + lane; kk < k1; kk += 32) {
                        const unsigned int abar = scaled_magnitude(src[padded(kk)], E);
                        acc += abar * abar;
                        l1 += abar;
                    }
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, o);
                l1 = __reduce_add_sync(0xFFFFFFFFu, l1);
                if (lane == 0 && acc) {
                    atomicAdd(&res[l].sumsq, acc);
                    atomicAdd(&res[l].l1, l1);
                }
            }
            __syncthreads();
        }
        // ---- the shift of every line (same arithmetic as scan_finalize_kernel)
        if (tid < nl) {
            const int sh = line_shift(p, res[tid]);
            res[tid].shift = sh;
            p.shift[line0 + tid] = sh;
            keep_scan(p.scan, line0 + tid, res[tid].sumsq, res[tid].exponent(), res[tid].bad(), res[tid].l1);
        }
        __syncthreads();
        // ---- conversion: a thread takes eight consecutive inner indices of one line; a step over the block adds a constant to
        // its line and octet, and one carry
        const int octs = static_cast<int>(p.geom.row_pitch >> 3);       // row_pitch is a multiple of 16
        const int line_step = nthreads / octs, oct_step = nthreads - line_step * octs;
        for (int l = tid / octs, o = tid - tid / octs * octs; l < nl;) {
            const int kb = 8 * o;
            int sigma = res[l].shift;
            const double *src = buf + l * p.pitch + 9 * o;               // padded(8 o)
            double x[8];
            if (sigma != OZ_NONFINITE_SHIFT && kb + 8 <= k) {
#pragma unroll
                for (int e = 0; e < 8; ++e) x[e] = src[e];
            } else {
                const bool dead = sigma == OZ_NONFINITE_SHIFT;
#pragma unroll
                for (int e = 0; e < 8; ++e) x[e] = (!dead && kb + e < k) ? src[e] : 0.0;
                if (dead) sigma = 0;
            }
            convert<SET, LAYOUT, 4>(x, sigma, p.tz != 0, NearTable{lut_addr},
                                  p.planes + (kb >> 7) * p.geom.chunk_stride + (line0 + l) * p.geom.line_stride + (kb & 127),
                                  p.geom.plane_stride);
            l += line_step;
            o += oct_step;
            if (o >= octs) {
                o -= octs;
                ++l;
            }
        }
        res = next;
    }
}

template <int SET, int SIDE, int LAYOUT>
__global__ void __launch_bounds__(1024, 1)
deconstruct_fused_kernel(const __grid_constant__ FusedParams p)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    deconstruct_lines<SET, SIDE, LAYOUT>(p, blockIdx.x, gridDim.x, smem_raw);
}

// Both operands of a product: the first `blocksA` blocks take A, the others B.  One launch in place of two on two
// streams with their fork and join.
struct PairParams {
    FusedParams a, b;
    int blocksA;
};

template <int SET, int LAYOUTA, int LAYOUTB>
__global__ void __launch_bounds__(1024, 1)
deconstruct_pair_kernel(const __grid_constant__ PairParams p)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int block = blockIdx.x;
    if (block < p.blocksA) deconstruct_lines<SET, 0, LAYOUTA>(p.a, block, p.blocksA, smem_raw);
    else deconstruct_lines<SET, 1, LAYOUTB>(p.b, block - p.blocksA, gridDim.x - p.blocksA, smem_raw);
}

// Lines per thread-block pass of the fused kernel and its launch shape; group = 0: not applicable
// (the lines are too long for shared memory).
// Largest operand of the one-kernel form; above, clusters or three passes.  A call with the limit at 2 M, 4 M and 8 M elements: 3000 x 300 x
// 1200, set S, 125, 116 and 126 us; 4000 x 1000 x 1000 230, 225 and 225; 2500 x 2500 x 1024 308, 308 and 298; 2300 x 2300 x 2000 467, 467 and
// 478 (native 255, 255 and 270); only a tall operand of few rounds would go on winning (5000 x 200 x 1000 137, 138 and 119).
constexpr int64_t kFusedMaxElems = 1ll << 22;
struct FusedShape { int group, threads, grid; size_t smem; };

// `big`: one block of 1024 threads per SM instead of two of 512 (lines too long for two); `slots`: resident blocks
// that this operand may count on
FusedShape fused_shape(int set, int layout, int side, int64_t lines, int64_t k, bool big, int64_t slots)
{
    FusedShape f{0, 0, 0, 0};
    if (k < 1 || k > 32768 || lines < 1) return f;
    // The one-kernel form wins where the call is bound by launch latency; larger operands keep the
    // three-pass kernels, whose many small blocks hide the memory latency better.
    if (lines * k > kFusedMaxElems) return f;
    const int64_t line_bytes = static_cast<int64_t>(fused_pitch(static_cast<int>(k))) * 8;
    const int64_t fixed = lut_words_of(set, layout) * 4 + 64 * static_cast<int64_t>(sizeof(FusedLine)) + 64;
    int64_t group = ((big ? 224 : 110) * 1024 - fixed) / line_bytes;
    // side 0 loads `group` consecutive doubles per inner index
    if (group < (side == 0 ? (big ? 4 : 8) : (big ? 1 : 2))) return f;
    if (group > 32) group = 32;
    // small operands: fewer lines per block, so that the blocks cover the machine (a 256 x 256 operand
    // with 32 lines per block would run on 8 SMs)
    if (slots < 1) slots = 1;
    int64_t spread = (lines + slots - 1) / slots;
    // side 0: at least four consecutive lines (whole 32-byte sectors), eight where few blocks are enough
    // (500^3: 24.7 us a call with four, 28.0 with eight; 256^3: 20.2 and 19.0)
    const int floor_group = side == 0 ? (lines * k >= (1ll << 17) ? 4 : 8) : 1;
    if (spread < floor_group) spread = floor_group;
    if (spread < group) group = spread;
    if (side == 0) {
        int pow2 = 1;
        while (pow2 * 2 <= group) pow2 *= 2;
        // up rather than down: a second round costs more than fuller blocks (1300 x 300 x 1400: 70.9 and 78.0 us)
        if (group > pow2 && (pow2 * 2) * line_bytes + fixed <= (big ? 224 : 110) * 1024 && pow2 < 32) pow2 *= 2;
        group = pow2;
    } else if (group > lines) {
        group = lines;
    }
    f.group = static_cast<int>(group);
    f.threads = big ? 1024 : 512;
    f.smem = static_cast<size_t>(fixed + group * line_bytes);
    const int64_t ngroups = (lines + group - 1) / group;
    f.grid = static_cast<int>(ngroups < slots ? ngroups : slots);
    return f;
}

template <int SET, int SIDE, int LAYOUT>
oz_status_t launch_fused(const FusedParams &p, const FusedShape &f, bool alone, cudaStream_t stream)
{
    static std::atomic<unsigned long long> ready{0};
    OZ_CUDA_CHECK(allow_shared(deconstruct_fused_kernel<SET, SIDE, LAYOUT>, kMaxShared, ready));
    OZ_CUDA_CHECK(launch_if(alone, deconstruct_fused_kernel<SET, SIDE, LAYOUT>, dim3(f.grid), f.threads, f.smem, stream, p));
    count_launch();
    return OZ_OK;
}

template <int SET, int LAYOUTA, int LAYOUTB>
oz_status_t launch_pair(const PairParams &p, const FusedShape &fa, const FusedShape &fb, cudaStream_t stream)
{
    static std::atomic<unsigned long long> ready{0};
    OZ_CUDA_CHECK(allow_shared(deconstruct_pair_kernel<SET, LAYOUTA, LAYOUTB>, kMaxShared, ready));
    OZ_CUDA_CHECK(launch(deconstruct_pair_kernel<SET, LAYOUTA, LAYOUTB>, dim3(fa.grid + fb.grid), fa.threads,
                         fa.smem > fb.smem ? fa.smem : fb.smem, stream, p));
    count_launch();
    return OZ_OK;
}

// parameters of the one-kernel form for one operand
FusedParams fused_params(int side, int64_t lines, int64_t k, const double *X, int64_t ldx, int set, const Route &rt,
                         uint8_t *planes, const PlaneGeom &geom, int32_t *shift, void *scratch, int group)
{
    FusedParams p{};
    if (rt.fallback) p.scan = carve_scratch(scratch, lines);      // the row check reads the scan results
    p.X = X; p.ldx = ldx; p.lines = lines; p.k = k;
    p.group = group;
    p.pitch = fused_pitch(static_cast<int>(k));
    p.side = side; p.rule = rt.rule; p.tz = rt.quant;
    int tA = 0, tB = 0;
    budget_maxexp(set, k, &tA, &tB);
    p.tbits = side == 0 ? tA : tB;
    uint64_t g2lo = 0, g2hi = 0;
    cs_bound_squared(set, k, &g2lo, &g2hi);
    p.g2lo = g2lo; p.g2hi = g2hi;
    p.esc_threshold = esc_threshold(set);
    p.lut_global = device_lut(set, rt.substrate);
    p.planes = planes; p.geom = geom;
    p.shift = shift;
    p.status = device_status_word();
    return p;
}

// ---- whole deconstruction by clusters ---------------------------------------------------------
// Operands above the one-kernel form: a cluster of up to five blocks holds 16 whole lines in its shared memory, `tiles` tiles of
// 128 inner indices a block, so that the operand is read once where scans and conversion read it three times (24 -> 8 bytes an
// element).  A half-warp owns a line in every block; its partial results (largest high word, then the norm sums)
// travel to the other blocks of the cluster through distributed shared memory, one cluster barrier each.  Blocks stay
// resident and walk the strips of 16 lines; a tile's place is refilled with the next strip as soon as it has been converted, so
// that loads run beside the arithmetic.  Same functions and integer sums as the other forms: the same bits.
// Bound: the phases of a strip, one behind the other, with 16 warps an SM to cover them.  8192 x 1024, set S on FP8: 89 us a side, 3.6 TB/s of
// the bytes it cannot do without where their traffic alone runs at 5.2 to 5.5; issue slots 41 % busy, no pipe above 31 %, the waits
// spread over dependent arithmetic, table look-ups, global loads and barriers.  6144 x 3072 native, clusters of four: 157 us, 2.8 TB/s, issue 46 %, FP32
// pipe 44 %.
struct ClusterParams {
    FusedParams f;               // group, pitch: not used
    int tiles;
};
constexpr int kClusterMax = 8;
struct ClusterExchange {         // per line and block of the cluster
    unsigned long long sumsq[kTileLines][kClusterMax];
    unsigned int l1[kTileLines][kClusterMax];
    unsigned int key[2][kTileLines][kClusterMax];      // strips in turn: without norm sums, one barrier a strip is all there is
};
// Largest exponents as keys that order like them: the high word of |x|, or 1100 + e of a subnormal, 0 for zeros only
constexpr unsigned int kFirstNormal = 0x00100000u, kFirstNonfinite = 0x7FF00000u;
__device__ __forceinline__ int key_exponent(unsigned int key)
{
    return key >= kFirstNormal ? static_cast<int>(key >> 20) - 1023 : (key ? static_cast<int>(key) - 1100 : INT32_MIN);
}
__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t cluster_blocks()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t remote(const void *p, uint32_t rank)
{
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(static_cast<uint32_t>(__cvta_generic_to_shared(p))), "r"(rank));
    return a;
}
__device__ __forceinline__ void store_remote(uint32_t addr, unsigned int v) { asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory"); }
__device__ __forceinline__ void store_remote(uint32_t addr, unsigned long long v) { asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(addr), "l"(v) : "memory"); }
__device__ __forceinline__ void cluster_barrier()
{
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <int SET, int SIDE, int LAYOUT>
__global__ void __launch_bounds__(kConvThreads, 2)
deconstruct_cluster_kernel(const __grid_constant__ ClusterParams cp)
{
    const FusedParams &p = cp.f;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int T = cp.tiles;
    ClusterExchange &ex = *reinterpret_cast<ClusterExchange *>(smem_raw + T * kTileBytes);
    uint32_t *lut = reinterpret_cast<uint32_t *>(smem_raw + T * kTileBytes + sizeof(ClusterExchange));
    const uint32_t lut_addr = static_cast<uint32_t>(__cvta_generic_to_shared(lut));
    const uint32_t tile_addr = static_cast<uint32_t>(__cvta_generic_to_shared(smem_raw));
    dependency_release();
    load_table<SET, LAYOUT>(lut, p.lut_global, threadIdx.x, kConvThreads);      // written once, before any call
    dependency_wait();

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int li = warp * 2 + (lane >> 4), oct = lane & 15;
    const unsigned int half = lane < 16 ? 0xFFFFu : 0xFFFF0000u;
    const uint32_t rank = cluster_rank(), C = cluster_blocks();
    const bool pairs = element_pairs(p.X, p.ldx);
    const int64_t nchunks = (p.geom.row_pitch + kChunk - 1) / kChunk, strips = (p.lines + kTileLines - 1) / kTileLines;
    const int64_t chunk0 = static_cast<int64_t>(rank) * T;
    const int nt = static_cast<int>(nchunks - chunk0 < T ? (nchunks - chunk0 > 0 ? nchunks - chunk0 : 0) : T);
    auto request = [&](int64_t strip, int t) {
        const uint32_t base = tile_addr + t * kTileBytes;
        const int64_t line0 = strip * kTileLines, k0 = (chunk0 + t) * kChunk;
        if constexpr (SIDE == 0) {
            request_side0(p.X, p.ldx, p.lines, p.k, pairs, line0, k0, base);
        } else {
            request_row(p.X, p.ldx, p.lines, p.k, pairs, line0 + warp * 2, k0, base + warp * 2 * kTileRow);
            request_row(p.X, p.ldx, p.lines, p.k, pairs, line0 + warp * 2 + 1, k0, base + (warp * 2 + 1) * kTileRow);
        }
    };
    const int64_t first = blockIdx.x / C, step = gridDim.x / C;
    cluster_barrier();                   // every block of the cluster has started: its shared memory may be written
    int turn = 0;
    if (first < strips)
        for (int t = 0; t < nt; ++t) request(first, t);
    for (int64_t strip = first; strip < strips; strip += step, turn ^= 1) {
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();                 // the strip (and, the first time, the table) is there
        const int64_t line = strip * kTileLines + li;
        // ---- largest exponent
        unsigned int key = 0u;
        for (int t = 0; t < nt; ++t) {
            double x[8];
            tile_octet<SIDE>(smem_raw + t * kTileBytes, x);
#pragma unroll
            for (int e = 0; e < 8; ++e) key = max(key, static_cast<unsigned int>(__double2hiint(x[e])) & 0x7FFFFFFFu);
        }
        key = __reduce_max_sync(half, key);
        if (__any_sync(0xFFFFFFFFu, key < kFirstNormal)) {        // zeros and subnormals only: exponents from the whole words
            unsigned int small = 0u;
            for (int t = 0; t < nt; ++t) {
                double x[8];
                tile_octet<SIDE>(smem_raw + t * kTileBytes, x);
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    int ex1;
                    if (classify(x[e], &ex1) == 1 && ex1 < -1022) small = max(small, static_cast<unsigned int>(ex1 + 1100));
                }
            }
            small = __reduce_max_sync(half, small);
            if (key < kFirstNormal) key = small;
        }
        if (static_cast<uint32_t>(oct) < C) store_remote(remote(&ex.key[turn][li][rank], oct), key);
        cluster_barrier();
        key = __reduce_max_sync(half, static_cast<uint32_t>(oct) < C ? ex.key[turn][li][oct] : 0u);
        const int E = key_exponent(key);
        const bool bad = key >= kFirstNonfinite;
        // ---- norm sums
        unsigned long long S = 0ull;
        unsigned int l1 = 0u;
        if (p.rule == 1) {
            if (!bad && E != INT32_MIN) {        // uniform over the half-warp
                const bool fast_scale = 9 - E >= -1000 && 9 - E <= 1000;
                const double scale9 = __hiloint2double((1023 + (fast_scale ? 9 - E : 0)) << 20, 0);
                for (int t = 0; t < nt; ++t) {
                    double x[8];
                    tile_octet<SIDE>(smem_raw + t * kTileBytes, x);
                    unsigned int part = 0u;           // eight terms of at most 2^20
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        unsigned int abar;
                        if (fast_scale) {
                            abar = magnitude(x[e], scale9);
                        } else {
                            abar = scaled_magnitude(x[e], E);
                        }
                        part += abar * abar;
                        l1 += abar;
                    }
                    S += part;
                }
            }
            __syncwarp();
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) S += __shfl_xor_sync(0xFFFFFFFFu, S, o);
            l1 = __reduce_add_sync(half, l1);
            if (static_cast<uint32_t>(oct) < C) {
                store_remote(remote(&ex.sumsq[li][rank], oct), S);
                store_remote(remote(&ex.l1[li][rank], oct), l1);
            }
            cluster_barrier();
            S = static_cast<uint32_t>(oct) < C ? ex.sumsq[li][oct] : 0ull;
            l1 = __reduce_add_sync(half, static_cast<uint32_t>(oct) < C ? ex.l1[li][oct] : 0u);
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) S += __shfl_xor_sync(0xFFFFFFFFu, S, o);
        }
        // ---- the shift (same arithmetic as scan_finalize_kernel)
        int sigma = 0;
        if (oct == 0 && line < p.lines) {
            if (bad) sigma = OZ_NONFINITE_SHIFT;
            else if (E != INT32_MIN) sigma = p.rule == 0 ? p.tbits - 1 - E : norm_exponent(S, p.g2lo, p.g2hi) + 9 - E;
            if (rank == 0) {
                p.shift[line] = sigma;
                keep_scan(p.scan, line, S, E, bad, l1);
                if (bad) {
                    atomicOr(p.status, 1u << OZ_ERR_NONFINITE_INPUT);
                } else if (E != INT32_MIN && p.rule == 1) {
                    atomicMin(p.status + 1 + p.side, line_flatness(l1, S, p.k));
                    p.status[3] = p.esc_threshold;
                }
            }
        }
        sigma = __shfl_sync(0xFFFFFFFFu, sigma, lane & 16);
        // ---- conversion, tile by tile, each followed by the copy of the next strip's
        const bool more = strip + step < strips;
        for (int t = 0; t < nt; t += 2) {        // a thread takes 16 elements: the half-warps' halves take two tiles at once
            const int tt = t + (oct >> 3);
            const int64_t chunk = chunk0 + tt;
            const int k_in = (oct & 7) * 16;                 // first of this thread's indices in the tile
            if (tt < nt && line < p.lines && chunk * kChunk + k_in < p.geom.row_pitch) {
                double x[16];
                tile_octets<SIDE>(smem_raw + tt * kTileBytes, oct & 7, x);
                int sig = sigma;
                if (sig == OZ_NONFINITE_SHIFT) {       // its planes are zeros
                    sig = 0;
#pragma unroll
                    for (int e = 0; e < 16; ++e) x[e] = 0.0;
                }
                convert<SET, LAYOUT, 8>(x, sig, p.tz != 0, FarTable{lut_addr},
                                        p.planes + chunk * p.geom.chunk_stride + line * p.geom.line_stride + k_in, p.geom.plane_stride);
            }
            if (more) {
                __syncthreads();             // these tiles have been read
                request(strip + step, t);
                if (t + 1 < nt) request(strip + step, t + 1);
            }
        }
    }
    cluster_barrier();                   // no block leaves while another may still write to it
}

// Clusters of this many blocks that are resident at once on the current device, asked once per device.  One kernel stands for all:
// each has 127 or 128 registers, 256 threads and no more than half of a multiprocessor's shared memory, so two blocks a
// multiprocessor.  (A cluster stays inside a group of multiprocessors, which three and more do not fill: 148, 93, 71 and 56 clusters of
// two to five blocks on 148 multiprocessors.)
cudaError_t resident_clusters(int blocks, int *clusters)
{
    static std::atomic<int> known[64][kClusterMax + 1];
    int dev = 0;
    cudaError_t rc = cudaGetDevice(&dev);
    if (rc != cudaSuccess) return rc;
    std::atomic<int> &here = known[dev & 63][blocks];
    *clusters = here.load(std::memory_order_relaxed);
    if (*clusters) return cudaSuccess;
    const auto kernel = deconstruct_cluster_kernel<2, 0, kLayoutNative>;
    constexpr size_t half = kMaxShared / 2 - 1024;
    static std::atomic<unsigned long long> ready{0};
    if ((rc = allow_shared(kernel, kMaxShared, ready)) != cudaSuccess) return rc;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(kConvThreads);
    cfg.gridDim = dim3(static_cast<unsigned>(blocks));
    cfg.dynamicSmemBytes = half;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = static_cast<unsigned>(blocks);
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    rc = cudaOccupancyMaxActiveClusters(clusters, kernel, &cfg);
    if (rc != cudaSuccess) return rc;
    if (*clusters < 1) *clusters = 1;
    here.store(*clusters, std::memory_order_relaxed);
    return cudaSuccess;
}

// Blocks of a cluster and tiles of a block for lines of `chunks` tiles, two blocks on an SM; blocks = 0: three passes.
// Clusters of one block win at every size measured up to 800 MB, and of two in the two-plane layouts, which need no table (90316 x 26 x 803 on A
// 1181 us a call against 1254 in three passes, 41247 x 22 x 901 517 against 540).  Larger ones are weighed against the three passes, which
// read operands of this size from L2 and fill their last wave better: in units of what the passes take for a million elements, a strip
// costs a cluster 0.44 a tile and 0.2 (rounds of resident clusters), and either form its start.  That is the time of every
// layout measured, 384 to 3700 inner indices and 4.5 to 40 million elements, within 6 percent (rms).  Clusters of three and more
// have to win by 8 percent: what they leave of the machine to the other operand's kernels is not in the sum.  3000 x 2500 x 1700, set S, 580 us with
// clusters of three on both sides, 541 without; 2100^3 474 and 443; 6144 x 6144 x 3072 native 1836 with clusters of four, 1860
// without.  Above 256 MiB a cluster of three or more spreads its reads over too much memory (side 0: 128 bytes from each of k
// columns; 60000 x 200 x 2500 native 2000 us a call against 2300), and so does any cluster above 1 GiB; beyond five blocks one table
// and one block less per SM hide too little (4096^3, set S: 331 us against 402).  Operands that are copied element by element (an odd
// leading dimension, or off the 16-byte boundary) cost the passes nothing more and a cluster of two a tenth on side 0, larger ones a fifth, and a
// twentieth on side 1 (medians over the same sizes; 40113 x 135 x 1071 by clusters 1024 us a call, by passes 913).
struct ClusterShape { int blocks, tiles; size_t smem; };
ClusterShape cluster_shape(int set, int layout, int side, int64_t lines, int64_t k, int64_t chunks, bool pairs)
{
    const size_t fixed = lut_words_of(set, layout) * 4 + sizeof(ClusterExchange);
    const int most = static_cast<int>((226 * 1024 / 2 - 1024 - fixed) / kTileBytes);
    const int64_t blocks = (chunks + most - 1) / most, bytes = 8 * lines * k;
    if (blocks > 5 || bytes > (blocks <= 2 ? 1ll << 30 : 1ll << 28)) return {0, 0, 0};
    const int tiles = static_cast<int>((chunks + blocks - 1) / blocks);
    if (blocks > (two_plane_layout(layout) ? 2 : 1)) {
        int clusters = 1;
        if (resident_clusters(static_cast<int>(blocks), &clusters) != cudaSuccess) return {0, 0, 0};
        const int64_t strips = (lines + kTileLines - 1) / kTileLines, rounds = (strips + clusters - 1) / clusters;
        const double by_clusters = (static_cast<double>(rounds) * (0.44 * tiles + 0.2) + 0.6) * (pairs ? 1.0 : side == 1 ? 1.05 : blocks == 2 ? 1.1 : 1.2);
        const double by_passes = 1e-6 * static_cast<double>(lines * k) + (side == 0 ? 1.4 : 0.6);
        if (by_clusters >= (blocks == 2 ? 1.0 : 0.92) * by_passes) return {0, 0, 0};
    }
    return {static_cast<int>(blocks), tiles, fixed + static_cast<size_t>(tiles) * kTileBytes};
}

template <int SET, int SIDE, int LAYOUT>
oz_status_t launch_cluster(const ClusterParams &p, const ClusterShape &shape, bool alone, cudaStream_t stream)
{
    const auto kernel = deconstruct_cluster_kernel<SET, SIDE, LAYOUT>;
    static std::atomic<unsigned long long> ready{0};
    OZ_CUDA_CHECK(allow_shared(kernel, kMaxShared, ready));
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(kConvThreads);
    cfg.dynamicSmemBytes = shape.smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = static_cast<unsigned>(shape.blocks);
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    int clusters = 1;
    OZ_CUDA_CHECK(resident_clusters(shape.blocks, &clusters));
    const int64_t strips = (p.f.lines + kTileLines - 1) / kTileLines;
    // as many as share the strips evenly
    const int64_t rounds = (strips + clusters - 1) / clusters, used = (strips + rounds - 1) / rounds;
    cfg.gridDim = dim3(static_cast<unsigned>(used * shape.blocks));
    cfg.numAttrs = alone ? 2 : 1;
    OZ_CUDA_CHECK(cudaLaunchKernelEx(&cfg, kernel, p));
    count_launch();
    OZ_CUDA_CHECK(cudaGetLastError());
    return OZ_OK;
}

template <int SET, int SIDE, int LAYOUT>
oz_status_t launch_convert(const double *X, int64_t ldx, int64_t lines, int64_t k,
                           const int32_t *shift, const uint32_t *lut, uint8_t *planes,
                           const PlaneGeom &geom, int tz, bool alone, cudaStream_t stream)
{
    constexpr size_t smem = lut_words_of(SET, LAYOUT) * 4 + 2 * kTileBytes;
    constexpr bool kByLine = SIDE == 1 && LAYOUT != kLayoutNative && !two_plane_layout(LAYOUT);
    static std::atomic<unsigned long long> ready[2] = {{0}, {0}};
    const bool by_line = kByLine && geom.line_stride != kChunk;
    const auto kernel = by_line ? convert_kernel<SET, SIDE, LAYOUT, kByLine> : convert_kernel<SET, SIDE, LAYOUT, false>;
    OZ_CUDA_CHECK(allow_shared(kernel, smem, ready[by_line]));
    const int64_t nchunks = (geom.row_pitch + kChunk - 1) / kChunk;
    if (lines * nchunks >= 0x7FFFFFFFll) return OZ_ERR_UNSUPPORTED;   // item numbers are 32-bit
    const int64_t need = ((lines + kTileLines - 1) / kTileLines) * nchunks;
    // persistent blocks: as many as are resident at once (each copies the table once)
    const int64_t cap = static_cast<int64_t>(conv_blocks(LAYOUT)) * sm_count();
    int grid = static_cast<int>(need < cap ? need : cap);
    OZ_CUDA_CHECK(launch_if(alone, kernel, dim3(grid), kConvThreads, smem, stream,
                         X, ldx, lines, k, shift, lut, planes, geom, tz));
    count_launch();
    OZ_CUDA_CHECK(cudaGetLastError());
    return OZ_OK;
}

}  // namespace

// scan_init + the scan passes of the route's scale rule [+ the shifts, except for the accurate rule, whose shifts come
// later from the bound product], of one operand or (both pointers) of both
oz_status_t launch_scan(const ScanJob *a, const ScanJob *b, int64_t k, int set, const Route &rt, bool alone, cudaStream_t stream)
{
    // (a side of fewer elements than kGuessed1 has no guesses: its second pass from L2 costs no more than they do)
    auto guessing = [&](const ScanJob *j, int side) { return j && rt.rule == 1 && k >= kSamples && j->spare && (side == 0 || j->lines * k >= kGuessed1); };
    const bool guesses = guessing(a, 0) || guessing(b, 1);
    auto scan_side = [&](const ScanJob *j, int side) {
        ScanSide p{};
        if (!j) return p;
        p.X = j->X; p.ldx = j->ldx; p.lines = j->lines;
        p.s = carve_scratch(j->scratch, j->lines);
        p.g = carve_guess(guessing(j, side) ? j->spare : nullptr, j->lines);
        // split the inner dimension so that the scan fills the machine even for few lines
        const int64_t line_blocks = side == 0 ? (j->lines + 255) / 256 : (j->lines + 7) / 8;
        const int64_t want_split = (148 * 8 + line_blocks - 1) / line_blocks, max_split = (k + 63) / 64;
        int64_t split = want_split < max_split ? want_split : max_split;
        if (split < 1) split = 1;
        if (split > 65535) split = 65535;
        p.kspan = (k + split - 1) / split;
        split = k > 0 ? (k + p.kspan - 1) / p.kspan : 0;
        p.line_blocks = static_cast<uint32_t>(line_blocks);
        p.blocks = static_cast<uint32_t>(line_blocks * split);
        return p;
    };
    const ScanSide sa = scan_side(a, 0), sb = scan_side(b, 1);
    const unsigned blocks1d = static_cast<unsigned>((sa.lines + sb.lines + 255) / 256);
    const dim3 grid(sa.blocks + sb.blocks);
    if (guesses) {
        OZ_CUDA_CHECK(launch_if(alone, scan_sample_kernel, dim3(static_cast<unsigned>((sa.lines + 31) / 32 + (sb.lines + 7) / 8)), 256, 0, stream, sa, sb, k));
        OZ_CUDA_CHECK(launch_if(alone, scan_kernel<2>, grid, 256, 0, stream, sa, sb, k));
        OZ_CUDA_CHECK(launch_if(alone, scan_kernel<1>, grid, 256, 0, stream, sa, sb, k));
        count_launch(3);
    } else {
        OZ_CUDA_CHECK(launch_if(alone, scan_init_kernel, dim3(blocks1d), 256, 0, stream, sa.s, sa.lines, sb.s, sb.lines));
        count_launch();
        if (k > 0) {
            OZ_CUDA_CHECK(launch_if(alone, scan_kernel<0>, grid, 256, 0, stream, sa, sb, k));
            count_launch();
            if (rt.rule == 1) {
                OZ_CUDA_CHECK(launch_if(alone, scan_kernel<1>, grid, 256, 0, stream, sa, sb, k));
                count_launch();
            }
        }
    }
    if (rt.rule != 2) {
        int tA = 0, tB = 0;
        budget_maxexp(set, k, &tA, &tB);
        uint64_t g2lo = 0, g2hi = 0;
        cs_bound_squared(set, k, &g2lo, &g2hi);
        const FinalizeSide fa{sa.s, sa.lines, tA, a ? a->shift : nullptr, sa.g}, fb{sb.s, sb.lines, tB, b ? b->shift : nullptr, sb.g};
        OZ_CUDA_CHECK(launch_if(alone, scan_finalize_kernel, dim3(blocks1d), 256, 0, stream, fa, fb, k, rt.rule, g2lo, g2hi,
                             esc_threshold(set), device_status_word()));
        count_launch();
    }
    OZ_CUDA_CHECK(cudaGetLastError());
    return OZ_OK;
}

// accurate rule: the lines' magnitude digits as one K-major E4M3 plane per operand (after launch_scan)
oz_status_t launch_bound_planes(const ScanJob &a, uint8_t *planeA, const ScanJob &b, uint8_t *planeB, int64_t k, int64_t pitch,
                                cudaStream_t stream)
{
    const int64_t blocksA = ((a.lines + 31) / 32) * ((pitch + 63) / 64), blocksB = ((b.lines + 7) / 8) * ((pitch + 255) / 256);
    if (blocksA + blocksB >= 0x7FFFFFFFll) return OZ_ERR_UNSUPPORTED;
    const BoundSide pa{a.X, a.ldx, a.lines, carve_scratch(a.scratch, a.lines), planeA, static_cast<uint32_t>(blocksA)};
    const BoundSide pb{b.X, b.ldx, b.lines, carve_scratch(b.scratch, b.lines), planeB, static_cast<uint32_t>(blocksB)};
    OZ_CUDA_CHECK(launch(bound_plane_kernel, dim3(static_cast<unsigned>(blocksA + blocksB)), 256, 0, stream, pa, pb, k, pitch));
    count_launch();
    OZ_CUDA_CHECK(cudaGetLastError());
    return OZ_OK;
}

// accurate rule: where the bound product accumulates the maximum of line `l` (a 32-bit word, zero
// after launch_scan): word stride 2 from this address
unsigned int *bound_maxima(void *scratch, int64_t lines)
{
    return reinterpret_cast<unsigned int *>(carve_scratch(scratch, lines).sumsq);
}

// accurate rule: shifts from the maxima of the bound product
oz_status_t launch_accurate_finalize(const ScanJob &a, const ScanJob &b, int budget_log2, cudaStream_t stream)
{
    const FinalizeSide fa{carve_scratch(a.scratch, a.lines), a.lines, 0, a.shift, {}}, fb{carve_scratch(b.scratch, b.lines), b.lines, 0, b.shift, {}};
    OZ_CUDA_CHECK(launch(accurate_finalize_kernel, dim3(static_cast<unsigned>((a.lines + b.lines + 255) / 256)), 256, 0, stream,
                         fa, fb, budget_log2, device_status_word()));
    count_launch();
    OZ_CUDA_CHECK(cudaGetLastError());
    return OZ_OK;
}

// quantise, reduce, look up, store: the planes of one operand from its shifts
oz_status_t launch_convert_planes(int side, int64_t lines, int64_t k, const double *X, int64_t ldx,
                                  int set, const Route &rt, uint8_t *planes, const PlaneGeom &geom,
                                  const int32_t *shift, bool alone, cudaStream_t stream)
{
    const uint32_t *lut = device_lut(set, rt.substrate);
#define OZ_CONVERT(SET_, SIDE_, LAYOUT_)                                                                 \
    launch_convert<SET_, SIDE_, LAYOUT_>(X, ldx, lines, k, shift, lut, planes, geom, rt.quant, alone, stream)
#define OZ_CONVERT_SET(SET_)                                                                                          \
    (layout == kLayoutDigits      ? (side == 0 ? OZ_CONVERT(SET_, 0, kLayoutDigits) : OZ_CONVERT(SET_, 1, kLayoutDigits))      \
     : layout == kLayoutDigitsI8  ? (side == 0 ? OZ_CONVERT(SET_, 0, kLayoutDigitsI8) : OZ_CONVERT(SET_, 1, kLayoutDigitsI8))  \
     : layout == kLayoutMerged    ? OZ_CONVERT(SET_, 0, kLayoutMerged)                                                   \
     : layout == kLayoutMergedI8A ? OZ_CONVERT(SET_, 0, kLayoutMergedI8A)                                                \
     : layout == kLayoutMergedI8B ? OZ_CONVERT(SET_, 1, kLayoutMergedI8B)                                                \
     : layout == kLayoutTwo       ? OZ_CONVERT(SET_, 0, kLayoutTwo)                                                      \
     : layout == kLayoutTwoI8     ? OZ_CONVERT(SET_, 0, kLayoutTwoI8)                                                    \
     : layout == kLayoutFour      ? OZ_CONVERT(SET_, 1, kLayoutFour)                                                     \
                                  : OZ_CONVERT(SET_, 1, kLayoutFourI8))
    const int layout = rt.layout(side);
    if (layout == kLayoutNative) return side == 0 ? OZ_CONVERT(2, 0, kLayoutNative) : OZ_CONVERT(2, 1, kLayoutNative);
    if (set == 0) return OZ_CONVERT_SET(0);
    if (set == 1) return OZ_CONVERT_SET(1);
    return OZ_CONVERT_SET(2);
#undef OZ_CONVERT_SET
#undef OZ_CONVERT
}

// the one-kernel form's shape for an operand by itself, group = 0: three passes
static FusedShape lone_shape(int side, int64_t lines, int64_t k, int set, const Route &rt)
{
    const int sms = sm_count();
    FusedShape f = fused_shape(set, rt.layout(side), side, lines, k, false, 2ll * sms);
    if (f.group <= 0) f = fused_shape(set, rt.layout(side), side, lines, k, true, sms);
    return f;
}

// The cluster form: planes in the private layout, lines that fit a cluster, and the layouts of the schedules that calls take by
// default (merged, native, A of the two-plane schedule; B's digits on FP8 are those of either schedule).  INT8 calls with
// OZ_ACC_SEPARATE therefore take three passes on both operands and FP8 calls with it on A; so does B of the two-plane schedule, whose 128
// lines at most exceed 4 M elements from k = 32768 on, beyond any cluster.
static ClusterShape by_clusters(int side, int64_t lines, int64_t k, int set, const Route &rt, const PlaneGeom &geom, const double *X, int64_t ldx)
{
    const int layout = rt.layout(side);
    const bool built = layout == kLayoutNative || (side == 0 ? layout != kLayoutDigits && layout != kLayoutDigitsI8
                                                             : layout == kLayoutDigits || layout == kLayoutMergedI8B);
    if (!built || geom.line_stride != kChunk || k < 1) return {0, 0, 0};
    return cluster_shape(set, layout, side, lines, k, (geom.row_pitch + kChunk - 1) / kChunk, element_pairs(X, ldx));
}

bool three_passes(int side, const ScanJob &j, int64_t k, int set, const Route &rt)
{
    return lone_shape(side, j.lines, k, set, rt).group <= 0 &&
           by_clusters(side, j.lines, k, set, rt, private_planes(j.lines, round_up(k, kChunk)), j.X, j.ldx).blocks == 0;
}

oz_status_t launch_deconstruct(int side, int64_t lines, int64_t k, const double *X, int64_t ldx,
                               int set, const Route &rt, uint8_t *planes, const PlaneGeom &geom,
                               int32_t *shift, void *scratch, bool alone, cudaStream_t stream)
{
    if (rt.rule == 2) return OZ_ERR_UNSUPPORTED;      // the accurate rule needs both operands
    const FusedShape f = lone_shape(side, lines, k, set, rt);
    if (f.group > 0) {
        const FusedParams p = fused_params(side, lines, k, X, ldx, set, rt, planes, geom, shift, scratch, f.group);
        const int layout = rt.layout(side);
#define OZ_FUSED(SET_, SIDE_, LAYOUT_) launch_fused<SET_, SIDE_, LAYOUT_>(p, f, alone, stream)
#define OZ_FUSED_SET(SET_)                                                                                          \
    (layout == kLayoutDigits      ? (side == 0 ? OZ_FUSED(SET_, 0, kLayoutDigits) : OZ_FUSED(SET_, 1, kLayoutDigits))      \
     : layout == kLayoutDigitsI8  ? (side == 0 ? OZ_FUSED(SET_, 0, kLayoutDigitsI8) : OZ_FUSED(SET_, 1, kLayoutDigitsI8))  \
     : layout == kLayoutMerged    ? OZ_FUSED(SET_, 0, kLayoutMerged)                                                   \
     : layout == kLayoutMergedI8A ? OZ_FUSED(SET_, 0, kLayoutMergedI8A)                                                \
     : layout == kLayoutMergedI8B ? OZ_FUSED(SET_, 1, kLayoutMergedI8B)                                                \
     : layout == kLayoutTwo       ? OZ_FUSED(SET_, 0, kLayoutTwo)                                                      \
     : layout == kLayoutTwoI8     ? OZ_FUSED(SET_, 0, kLayoutTwoI8)                                                    \
     : layout == kLayoutFour      ? OZ_FUSED(SET_, 1, kLayoutFour)                                                     \
                                  : OZ_FUSED(SET_, 1, kLayoutFourI8))
        if (layout == kLayoutNative) return side == 0 ? OZ_FUSED(2, 0, kLayoutNative) : OZ_FUSED(2, 1, kLayoutNative);
        if (set == 0) return OZ_FUSED_SET(0);
        if (set == 1) return OZ_FUSED_SET(1);
        return OZ_FUSED_SET(2);
#undef OZ_FUSED_SET
#undef OZ_FUSED
    }
    const ClusterShape c = by_clusters(side, lines, k, set, rt, geom, X, ldx);
    if (c.blocks) {
        ClusterParams p;
        p.f = fused_params(side, lines, k, X, ldx, set, rt, planes, geom, shift, scratch, 0);
        p.tiles = c.tiles;
        const int layout = rt.layout(side);
#define OZ_CLUSTER(SET_, SIDE_, LAYOUT_) launch_cluster<SET_, SIDE_, LAYOUT_>(p, c, alone, stream)
#define OZ_CLUSTER_SET(SET_)                                                                                    \
    (layout == kLayoutMerged      ? OZ_CLUSTER(SET_, 0, kLayoutMerged)                                         \
     : layout == kLayoutMergedI8A ? OZ_CLUSTER(SET_, 0, kLayoutMergedI8A)                                      \
     : layout == kLayoutMergedI8B ? OZ_CLUSTER(SET_, 1, kLayoutMergedI8B)                                      \
     : layout == kLayoutTwo       ? OZ_CLUSTER(SET_, 0, kLayoutTwo)                                            \
     : layout == kLayoutTwoI8     ? OZ_CLUSTER(SET_, 0, kLayoutTwoI8)                                          \
                                  : OZ_CLUSTER(SET_, 1, kLayoutDigits))
        if (layout == kLayoutNative) return side == 0 ? OZ_CLUSTER(2, 0, kLayoutNative) : OZ_CLUSTER(2, 1, kLayoutNative);
        if (set == 0) return OZ_CLUSTER_SET(0);
        if (set == 1) return OZ_CLUSTER_SET(1);
        return OZ_CLUSTER_SET(2);
#undef OZ_CLUSTER_SET
#undef OZ_CLUSTER
    }
    const ScanJob job{lines, X, ldx, shift, scratch, geom.row_pitch >= kGuessBytes ? planes : nullptr};
    oz_status_t st = launch_scan(side == 0 ? &job : nullptr, side == 1 ? &job : nullptr, k, set, rt, alone, stream);
    if (st != OZ_OK) return st;
    return launch_convert_planes(side, lines, k, X, ldx, set, rt, planes, geom, shift, alone, stream);
}

oz_status_t launch_deconstruct_pair(const OperandJob &a, const OperandJob &b, int64_t k, int set, const Route &rt,
                                    bool *taken, cudaStream_t stream)
{
    *taken = false;
    if (rt.rule == 2) return OZ_OK;      // shifts from both operands
    const int sms = sm_count();
    // The resident blocks are shared out by the operands' sizes.  Taken when both operands then finish in one round
    // (1009 x 983 x 1021: 77.0 -> 68.8 us a call; 1300 x 300 x 1400, one large block per SM: 81.5 -> 70.8); with more rounds the
    // two streams do as well or better (1800^3: 286 against 309).
    FusedShape fa, fb;
    bool one_round = false;
    for (const bool big : {false, true}) {
        const int64_t slots = (big ? 1 : 2) * static_cast<int64_t>(sms);
        fa = fused_shape(set, rt.layout(0), 0, a.lines, k, big, slots * a.lines / (a.lines + b.lines));
        fb = fused_shape(set, rt.layout(1), 1, b.lines, k, big, slots - fa.grid);
        one_round = fa.group > 0 && fb.group > 0 && static_cast<int64_t>(fa.grid) * fa.group >= a.lines &&
                    static_cast<int64_t>(fb.grid) * fb.group >= b.lines;
        if (one_round) break;
    }
    if (!one_round) return OZ_OK;
    PairParams p;
    p.a = fused_params(0, a.lines, k, a.X, a.ldx, set, rt, a.planes, a.geom, a.shift, a.scratch, fa.group);
    p.b = fused_params(1, b.lines, k, b.X, b.ldx, set, rt, b.planes, b.geom, b.shift, b.scratch, fb.group);
    p.blocksA = fa.grid;
    *taken = true;
    const int layout = rt.layout(0);
#define OZ_PAIR(SET_)                                                                                       \
    (layout == kLayoutMerged      ? launch_pair<SET_, kLayoutMerged, kLayoutDigits>(p, fa, fb, stream)      \
     : layout == kLayoutMergedI8A ? launch_pair<SET_, kLayoutMergedI8A, kLayoutMergedI8B>(p, fa, fb, stream) \
     : layout == kLayoutDigitsI8  ? launch_pair<SET_, kLayoutDigitsI8, kLayoutDigitsI8>(p, fa, fb, stream)  \
     : layout == kLayoutTwo       ? launch_pair<SET_, kLayoutTwo, kLayoutFour>(p, fa, fb, stream)           \
     : layout == kLayoutTwoI8     ? launch_pair<SET_, kLayoutTwoI8, kLayoutFourI8>(p, fa, fb, stream)       \
                                  : launch_pair<SET_, kLayoutDigits, kLayoutDigits>(p, fa, fb, stream))
    if (layout == kLayoutNative) return launch_pair<2, kLayoutNative, kLayoutNative>(p, fa, fb, stream);
    return set == 0 ? OZ_PAIR(0) : set == 1 ? OZ_PAIR(1) : OZ_PAIR(2);
#undef OZ_PAIR
}

// flags, ordered list and number of the rows that go to the native FP64 path, from the scan results
// that the deconstruction of both operands left in their scratch blocks
oz_status_t launch_esc_rows(void *scratchA, int64_t m, void *scratchB, int64_t n, int64_t k, int set,
                            unsigned char *flag, int *list, unsigned int *count, cudaStream_t stream)
{
    OZ_CUDA_CHECK(launch(esc_rows_kernel, dim3(1), 1024, 0, stream, carve_scratch(scratchA, m), m,
                         carve_scratch(scratchB, n), n, k, esc_threshold(set), flag, list, count, device_status_word()));
    count_launch();
    OZ_CUDA_CHECK(cudaGetLastError());
    return OZ_OK;
}

}  // namespace oz
