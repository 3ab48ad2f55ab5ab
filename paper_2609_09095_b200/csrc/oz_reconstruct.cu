// Reconstruction (Algorithm 3; Eq. 4-5 and the last step of Sec. 2 (iv)): residues -> the integer
// c' in [-M/2, M/2), unscaled by 2^-(sigma_i + tau_j) and rounded once to FP64.
//
// The paper's SIMT branch walks Garner's mixed-radix digits (r(r-1)/2 multiply-reduce steps).
// CRT fixes c' uniquely, so any exact evaluation gives the same integer; this kernel uses the
// weighted form
//     c' = sum_i c_i V_i  -  kappa M,     V_i = ((M/m_i)^-1 mod m_i) (M/m_i) mod M,
// with every V_i and M cut into three 38-bit chunks (40-bit for the all-byte set).  A stored
// residue is below 2 m_i < 2^11.1 (the whole-method calls keep a representative in (0, 2 m_i); 2^8
// for the byte set), so each of the three chunk sums is an integer below 2^53 -- at most 2^52.8 --
// and is formed EXACTLY by FP64 fused multiply-adds (r MACs per chunk).  kappa = round(S/M) comes from a floating estimate; the
// carry-normalised chunks are then summed with error-free additions, which give the correctly
// rounded FP64 value directly unless c' lies within a hair of a rounding boundary, of a power of
// two or of +-M/2 -- those rare outputs take an exact path: the 128-bit integer, an exact range
// test for the lift to [-M/2, M/2), and one round-to-nearest-even done in integer arithmetic.
// A thread handles the consecutive rows whose residues share one 32-bit word per modulus (two
// uint16, or four uint8 for the all-byte set).
#include <cstring>
#include <utility>

#include "oz_internal.h"

namespace oz {
namespace {

struct ReconConst {
    double V[kMaxR][3];        // V_i = V0 + V1 + V2, the chunks in place: V1 and V2 are multiples of 2^cw and 2^(2cw)
    double Mc[3];              // M   = M0 + M1 + M2 likewise
    double inv_M;              // 1/M (rounded)
    int half_M_guard;          // high word of (M/2) (1 - 2^-30): from it on the lift is decided exactly
    unsigned long long M_lo, M_hi;
};

__constant__ ReconConst c_recon[kNumSets];

// Chunk width: 38 bits for S and E (stored residues < 2^11.1, 13 terms: sums < 2^52.8); 40 bits for
// the 117.8-bit set A (residues < 2^8, 15 terms: sums < 2^52), so that three chunks cover M.
__host__ __device__ constexpr int chunk_bits(int set) { return set == 2 ? 40 : 38; }
__host__ __device__ constexpr double pow2d(int e) { double v = 1.0; for (int i = 0; i < e; ++i) v *= 2.0; return v; }
// Resident blocks per SM.  The loads of a thread are independent, so this many keep memory busy; the registers they leave
// (48, 64) hold everything.  16384 x 16384 update, set S, with 4 / 5 / 6 blocks: 2.18 / 2.17 / 2.17 ms; 6144 x 6144, set A, with
// 3 / 4 / 5 blocks: 288 / 289 / 298 us.  Before the mapping and the arithmetic below: 2.35 ms and 327 us.  One more where single elements
// of C are updated, since their old values are waited for in turn; not for plain stores, whose blocks of 40 registers would fit beside a
// GEMM's and become resident with it (499 x 366 x 2755 under the accurate rule 94 -> 102 us a call).
template <int SET, bool SINGLE_UPDATES = false> constexpr int kReconBlocks = (residue_bytes(SET) == 2 ? 5 : 4) + (SINGLE_UPDATES ? 1 : 0);
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

// w packs the residues of consecutive rows (two uint16 or four uint8); HALF selects the row
template <int SET, int HALF, int I>
__device__ __forceinline__ void crt_term(uint32_t w, double &S0, double &S1, double &S2)
{
    const ReconConst &K = c_recon[SET];
    constexpr int BITS = 8 * residue_bytes(SET);
    const uint32_t c = (w >> (BITS * HALF)) & ((1u << BITS) - 1u);
    // exact; the hardware conversion keeps this off the FP64 pipe, which bounds the kernel
    double cd = __uint2double_rn(c);
    S0 = fma(cd, K.V[I][0], S0);
    S1 = fma(cd, K.V[I][1], S1);
    S2 = fma(cd, K.V[I][2], S2);
}

template <int SET, int HALF, int... I>
__device__ __forceinline__ void crt_sum(std::integer_sequence<int, I...>, const uint32_t (&c)[kMaxR],
                                        double &S0, double &S1, double &S2)
{
    (crt_term<SET, HALF, I>(c[I], S0, S1, S2), ...);
}

// Exact tail (rare path): the three chunks as a 128-bit integer, exact lift to [-M/2, M/2),
// round-to-nearest-even conversion in integer arithmetic, power-of-two scale.
__device__ __forceinline__ double finish_exact(double X0, double X1, double X2, int shift_sum, int set)
{
    const ReconConst &K = c_recon[set];
    const int cw = chunk_bits(set);
    const long long t0 = __double2ll_rn(X0), t1 = __double2ll_rn(X1 * (1.0 / pow2d(cw))), t2 = __double2ll_rn(X2 * (1.0 / pow2d(2 * cw)));
    // v = t0 + t1 2^cw + t2 2^(2cw) as a two's-complement (hi:lo) pair
    unsigned long long lo = static_cast<unsigned long long>(t0) + (static_cast<unsigned long long>(t1) << cw);
    long long hi = (t0 >> 63) + (t1 >> (64 - cw)) + (lo < static_cast<unsigned long long>(t0) ? 1 : 0) +
                   static_cast<long long>(static_cast<unsigned long long>(t2) << (2 * cw - 64));
    const __int128 M = static_cast<__int128>((static_cast<unsigned __int128>(K.M_hi) << 64) | K.M_lo);
    const __int128 Mh = M >> 1;     // M is even for every set (each holds a power of two)
    __int128 v = static_cast<__int128>((static_cast<unsigned __int128>(static_cast<unsigned long long>(hi)) << 64) | lo);
    if (v >= Mh) v -= M;
    else if (v < -Mh) v += M;
    lo = static_cast<unsigned long long>(v);
    hi = static_cast<long long>(v >> 64);
    const bool neg = hi < 0;
    if (neg) {
        lo = 0ull - lo;
        hi = ~hi + (lo == 0ull ? 1 : 0);
    }
    // nearest double, ties to even: top 64 bits with a sticky bit far below the rounding position
    const unsigned long long uhi = static_cast<unsigned long long>(hi);
    const int lz = __clzll(static_cast<long long>(uhi | 1ull));          // uhi < 2^49: lz in [15, 63]
    const unsigned long long top = (uhi << lz) | (lo >> (64 - lz));
    const unsigned long long rest = lo << lz;
    unsigned long long mant = uhi ? (top | (rest ? 1ull : 0ull)) : lo;
    int scale = (uhi ? 64 - lz : 0) - shift_sum;
    double d = scale_pow2(__ull2double_rn(mant), scale);
    return neg ? -d : d;
}

// The three chunks summed: r is c' correctly rounded if the result is true (see row_value())
template <int SET>
__device__ __forceinline__ bool round_chunks(double X0, double X1, double X2, double &r)
{
    const double s = X2 + X1, err = X1 - (s - X2);
    const double t = err + X0;
    r = s + t;
    const double rem = t - (r - s);
    return fma(rem, 1.0 + 0x1p-29, r) == r && (__double2hiint(r) & 0x7FFFFFFF) < c_recon[SET].half_M_guard;
}

// alpha 2^-(sa + sb) c' (alpha = 1 or -1, as a sign bit: in a register pair of its own it spilled) where the fast path does not apply: NaN for a line with Inf/NaN; else from r, where that is c' correctly
// rounded and only the scale is out of reach, or by integers.  The sum of the shifts is taken in 64 bits; beyond 2^20 the result is
// zero or infinite whatever c' is.
template <int SET>
__device__ __noinline__ double row_value_exact(double X0, double X1, double X2, int sa, int sb, int alpha_sign)
{
    const double alpha = __hiloint2double(0x3FF00000 ^ alpha_sign, 0);
    if (sb == OZ_NONFINITE_SHIFT || sa == OZ_NONFINITE_SHIFT) return __longlong_as_double(0x7FF8000000000000ll) * alpha;
    const int sum = static_cast<int>(min(max(static_cast<long long>(sa) + sb, -(1ll << 20)), 1ll << 20));
    double r;
    return (round_chunks<SET>(X0, X1, X2, r) ? scale_pow2(r, -sum) : finish_exact(X0, X1, X2, sum, SET)) * alpha;
}

// Whether a row's shift may enter the 32-bit sums of the fast path: |sa| <= 2^30, which the mark of a row with Inf/NaN exceeds.  No sum
// with a column's shift, whatever that is and the mark of a column among them, then wraps into the range of row_value().
__device__ __forceinline__ bool ordinary_row(int sa)
{
    return static_cast<uint32_t>(sa) + (1u << 30) <= 1u << 31;
}

// One row of the thread's group: value = fast alpha 2^-(sa + sb) c', returned as the rounded integer r and the power of
// two to multiply it by (exact, and left to the caller so that an update of C is one fused multiply-add).
// The chunks are not carry-normalised.  X2 + X1 = s + err by a fast two-sum, which is error-free because X2 is a multiple of
// 2^(2cw) and so of ulp(X1) (|X1| < 2^(53+cw)); t = err + X0 loses at most 2^-52 of |err| + |X0|, and nothing below 2^53,
// which |X0| < 2^52.1 alone does not reach: what it loses is below 2^-40 of half an ulp of s; s + t = r + rem exactly (s is a
// multiple of 2^cw and so of ulp(t)).  Hence r is c' correctly rounded unless c' lies within 2^-29 of half an ulp from a
// rounding boundary -- adding rem, enlarged by 2^-29, then moves r -- or so near to +-M/2 that the lift may apply.
// 50 FP64 operations per output on set S where the carries and a test by exponents took 63.
template <int SET, int HALF>
__device__ __forceinline__ void row_value(const uint32_t (&c)[kMaxR], int sa, int sb, int alpha_sign,
                                          double &r, double &scale)
{
    const ReconConst &K = c_recon[SET];
    double X0 = 0.0, X1 = 0.0, X2 = 0.0;
    crt_sum<SET, HALF>(std::make_integer_sequence<int, set_r(SET)>{}, c, X0, X1, X2);
    const double kappa = fma(X2 + X1, K.inv_M, kRint) - kRint;
    X0 = fma(-kappa, K.Mc[0], X0);              // exact: integers below 2^53 (times 2^cw, 2^(2cw))
    X1 = fma(-kappa, K.Mc[1], X1);
    X2 = fma(-kappa, K.Mc[2], X2);
    const bool rounded = round_chunks<SET>(X0, X1, X2, r);
    const uint32_t shift_sum = static_cast<uint32_t>(sa) + static_cast<uint32_t>(sb);
    scale = __hiloint2double(static_cast<int>((1023u - shift_sum) << 20) ^ alpha_sign, 0);
    // in range: 2^-shift_sum and r 2^-shift_sum are normal; r is zero or 1 <= |r| < 2^118
    if (!(ordinary_row(sa) && shift_sum + 904u <= 1924u && rounded)) {
        r = row_value_exact<SET>(X0, X1, X2, sa, sb, alpha_sign);
        scale = 1.0;
    }
}

// scalar stores of up to two consecutive rows; `first` / `second`: which of them are written
__device__ __forceinline__ void store_pair(double *out, double p0, double p1, bool first, bool second, double beta)
{
    if (first) out[0] = beta != 0.0 ? out[0] + p0 : p0;
    if (second) out[1] = beta != 0.0 ? out[1] + p1 : p1;
}

// the ROWS consecutive rows of column j whose residues are packed in w[]: reconstruct, update C.
// For beta = 1 the old values of C are requested before the arithmetic starts, so that their latency
// hides behind it.  `keep`: bit h set = row h is written (rows that go to the native FP64 path are not).
template <int SET>
__device__ __forceinline__ void reconstruct_rows(const uint32_t (&w)[kMaxR], int64_t row, int nrows, int sb,
                                                 const int32_t *__restrict__ shiftA, double alpha, double beta,
                                                 double *out, bool vecC, uint32_t keep = 0xFu)
{
    constexpr int ROWS = 4 / residue_bytes(SET);
    int sa[ROWS];
#pragma unroll
    for (int h = 0; h < ROWS; ++h) sa[h] = h < nrows ? shiftA[row + h] : 0;
    const bool whole = vecC && nrows == ROWS && (keep & ((1u << ROWS) - 1u)) == ((1u << ROWS) - 1u);
    double2 old[ROWS / 2];
#pragma unroll
    for (int h = 0; h < ROWS / 2; ++h) old[h] = make_double2(0.0, 0.0);
    if (whole && beta != 0.0) {
#pragma unroll
        for (int h = 0; h < ROWS / 2; ++h) old[h] = *reinterpret_cast<const double2 *>(out + 2 * h);
    }
    const int alpha_sign = alpha < 0.0 ? INT32_MIN : 0;
    {
        double r0, r1 = 0.0, f0, f1 = 1.0;
        row_value<SET, 0>(w, sa[0], sb, alpha_sign, r0, f0);
        if (nrows > 1) row_value<SET, 1>(w, sa[1], sb, alpha_sign, r1, f1);
        if (whole) *reinterpret_cast<double2 *>(out) = make_double2(fma(r0, f0, old[0].x), fma(r1, f1, old[0].y));
        else store_pair(out, r0 * f0, r1 * f1, (keep & 1u) != 0, nrows > 1 && (keep & 2u) != 0, beta);
    }
    if constexpr (ROWS == 4) {
        if (nrows > 2) {
            double r2, r3 = 0.0, f2, f3 = 1.0;
            row_value<SET, 2>(w, sa[2], sb, alpha_sign, r2, f2);
            if (nrows > 3) row_value<SET, 3>(w, sa[3], sb, alpha_sign, r3, f3);
            if (whole) *reinterpret_cast<double2 *>(out + 2) = make_double2(fma(r2, f2, old[1].x), fma(r3, f3, old[1].y));
            else store_pair(out + 2, r2 * f2, r3 * f3, (keep & 4u) != 0, nrows > 3 && (keep & 8u) != 0, beta);
        }
    }
}

// Each thread reconstructs ROWS consecutive rows of one column: the residues of those rows are one
// 32-bit word per modulus (two uint16 for S and E, four uint8 for the all-byte set A).
template <int SET>
__global__ void __launch_bounds__(256, kReconBlocks<SET>)
reconstruct_kernel(const void *__restrict__ Rv, int64_t ldr, int64_t mod_stride, int64_t m,
                   int64_t n, const int32_t *__restrict__ shiftA, const int32_t *__restrict__ shiftB,
                   double alpha, double beta, double *__restrict__ C, int64_t ldc, int vecR, int vecC)
{
    dependency_release();
    dependency_wait();
    constexpr int RB = residue_bytes(SET), ROWS = 4 / RB, r = set_r(SET);
    // grid.x covers the row groups of a column, grid.y (and .z beyond 65535) the columns: no division
    const int64_t row = (blockIdx.x * 256ll + threadIdx.x) * ROWS;
    if (row >= m) return;
    const int64_t j = blockIdx.y + 65535ll * blockIdx.z;
    if (j >= n) return;
    const int nrows = m - row < ROWS ? static_cast<int>(m - row) : ROWS;

    // all residue loads are issued before any arithmetic: r independent requests in flight per
    // thread, kept packed so that they fit the register budget
    uint32_t w[kMaxR];
    const unsigned char *base = static_cast<const unsigned char *>(Rv) + (j * ldr + row) * RB;
#pragma unroll
    for (int i = 0; i < r; ++i) {
        const unsigned char *src = base + i * mod_stride * RB;
        if (vecR) {
            w[i] = *reinterpret_cast<const uint32_t *>(src);       // ldr is a multiple of ROWS: in bounds
        } else {
            uint32_t v = 0;
#pragma unroll
            for (int h = 0; h < ROWS; ++h) {
                if (h < nrows) {
                    uint32_t e = RB == 2 ? reinterpret_cast<const uint16_t *>(src)[h] : src[h];
                    v |= e << (8 * RB * h);
                }
            }
            w[i] = v;
        }
    }
    reconstruct_rows<SET>(w, row, nrows, shiftB[j], shiftA, alpha, beta, C + row + j * ldc, vecC != 0);
}

// Same reconstruction from the tile-ordered private array that the whole-method GEMM writes (see
// ResidueTiling).  A thread takes one 32-bit word of a 32-column x 64-row block, i.e. ROWS consecutive
// rows of one column.  A warp takes one 16-byte chunk of eight neighbouring columns: its residue loads are whole
// 128-byte lines and its accesses to C eight pieces of 64 (128) contiguous bytes; the warps of a thread block, which
// take the other chunks of the same columns, complete those to whole lines of C.
// ACCESS: how C is taken, in pairs of elements (even ldc, C on a multiple of 16 bytes), or singly, stored or updated.  Updates of single
// elements, whose loads and stores in eight pieces each cost more the more there are, give a warp consecutive words of one column: 512
// contiguous bytes of C for residue loads that touch eight lines.  1009 x 983 x 256, set S: 39 us a call against 52; 4501 x 4400 x 128: 400
// against 732; plain stores are faster in pieces (34 us against 36, 334 against 352).
// grid: x = (piece of the block, block within the tile, CTA rank of the pair), y = tile column, z = tile row
// SKIP: rows flagged in `skip` are left untouched (they are re-issued on the native FP64 path).
enum { kPairs, kSingleStores, kSingleUpdates };
template <int SET, bool SKIP, int ACCESS>
__global__ void __launch_bounds__(256, kReconBlocks<SET, ACCESS == kSingleUpdates>)
reconstruct_tiled_kernel(const void *__restrict__ Rv, int cg, int tiles_n, int tn0,
                         int64_t m, int64_t n, int64_t col0, int64_t col1,
                         const int32_t *__restrict__ shiftA, const int32_t *__restrict__ shiftB,
                         double alpha, double beta, double *__restrict__ C, int64_t ldc,
                         const unsigned char *__restrict__ skip)
{
    dependency_release();
    dependency_wait();
    constexpr int RB = residue_bytes(SET), ROWS = 4 / RB, r = set_r(SET);
    constexpr int kBlockWords = 64 * 32 * RB / 4;          // words of one 32 x 64 block: 1024 or 512
    constexpr int kColWords = 64 / ROWS;                   // words of one column of the block: 32 or 16
    constexpr int kCtaCols = 256 / kColWords;              // columns per thread block: 8 or 16
    constexpr int kPieces = 32 / kCtaCols;                 // thread blocks per residue block: 4 or 2
    const uint32_t piece = blockIdx.x % kPieces;
    const uint32_t wi = (blockIdx.x / kPieces) & 15u;
    const uint32_t rank = blockIdx.x / (kPieces * 16);     // 0, or 0..1 with CTA pairs
    const uint32_t tn = static_cast<uint32_t>(tn0) + blockIdx.y, tm = blockIdx.z;
    constexpr int kChunks = kColWords / 4;                 // 16-byte chunks of one column: 8 or 4
    const uint32_t warp = threadIdx.x >> 5, sub = threadIdx.x & 3u;
    constexpr bool spread = ACCESS != kSingleUpdates;
    const uint32_t c = spread ? warp % kChunks : (threadIdx.x >> 2) % kChunks;
    const uint32_t lane = piece * kCtaCols + (spread ? warp / kChunks * 8 + ((threadIdx.x >> 2) & 7u) : threadIdx.x / kColWords);   // column of the block
    const int64_t row = static_cast<int64_t>(tm) * 256 + (wi >> 2) * 64 + c * (16 / RB) + sub * ROWS;
    const int64_t j = (static_cast<int64_t>(tn) * cg + rank) * 128 + (wi & 3u) * 32 + lane;
    if (row >= m || j >= n || j < col0 || j >= col1) return;
    const int nrows = m - row < ROWS ? static_cast<int>(m - row) : ROWS;
    uint32_t keep = 0xFu;
    if constexpr (SKIP) {
        keep = 0u;
#pragma unroll
        for (int h = 0; h < ROWS; ++h)
            if (h < nrows && !skip[row + h]) keep |= 1u << h;
        if (!keep) return;
    }
    const int64_t wb = ((static_cast<int64_t>(tm) * tiles_n + tn) * cg + rank) * 16 + wi;
    // the r blocks of this patch are consecutive: modulus i at a compile-time offset
    const unsigned char *base = static_cast<const unsigned char *>(Rv) +
                                ((wb * r) * kBlockWords + c * 128 + lane * 4 + sub) * 4;
    uint32_t w[kMaxR];
#pragma unroll
    for (int i = 0; i < r; ++i) w[i] = *reinterpret_cast<const uint32_t *>(base + i * (kBlockWords * 4));
    reconstruct_rows<SET>(w, row, nrows, shiftB[j], shiftA, alpha, beta, C + row + j * ldc, ACCESS == kPairs, keep);
}

}  // namespace

oz_status_t upload_reconstruct_constants()
{
    static ReconConst host[kNumSets];
    for (int set = 0; set < kNumSets; ++set) {
        unsigned __int128 M = 1;
        for (int i = 0; i < set_r(set); ++i) M *= static_cast<unsigned>(modulus(set, i));
        const int cw = chunk_bits(set);
        const unsigned __int128 mask = (static_cast<unsigned __int128>(1) << cw) - 1;
        auto chunks = [&](unsigned __int128 v, double (&out)[3]) {
            out[0] = static_cast<double>(static_cast<unsigned long long>(v & mask));
            out[1] = static_cast<double>(static_cast<unsigned long long>((v >> cw) & mask)) * pow2d(cw);
            out[2] = static_cast<double>(static_cast<unsigned long long>(v >> (2 * cw))) * pow2d(2 * cw);
        };
        ReconConst &K = host[set];
        for (int i = 0; i < kMaxR; ++i) K.V[i][0] = K.V[i][1] = K.V[i][2] = 0.0;
        for (int i = 0; i < set_r(set); ++i) {
            unsigned mi = static_cast<unsigned>(modulus(set, i));
            unsigned __int128 W = M / mi;
            unsigned wm = static_cast<unsigned>(W % mi), inv = 0;
            for (unsigned c = 1; c < mi; ++c)
                if ((static_cast<unsigned long long>(wm) * c) % mi == 1) { inv = c; break; }
            unsigned __int128 V = W * inv;          // < M, and V = 1 mod m_i, 0 mod the other moduli
            chunks(V, K.V[i]);
        }
        chunks(M, K.Mc);
        K.inv_M = 1.0 / static_cast<double>(M);
        const double guard = 0.5 * static_cast<double>(M) * (1.0 - 0x1p-30);
        uint64_t guard_bits;
        memcpy(&guard_bits, &guard, sizeof(guard));
        K.half_M_guard = static_cast<int>(guard_bits >> 32);
        K.M_lo = static_cast<unsigned long long>(M);
        K.M_hi = static_cast<unsigned long long>(M >> 64);
    }
    OZ_CUDA_CHECK(cudaMemcpyToSymbol(c_recon, host, sizeof(host)));
    return OZ_OK;
}

oz_status_t launch_reconstruct(int64_t m, int64_t n, const void *R, int64_t ldr,
                               int64_t mod_stride, const int32_t *shiftA, const int32_t *shiftB,
                               int set, double alpha, double beta, double *C, int64_t ldc,
                               cudaStream_t stream)
{
    // one 32-bit load per modulus covers a thread's rows when every row group starts on a 4-byte boundary
    const int rows = 4 / residue_bytes(set);
    int vecR = (ldr % rows == 0 && mod_stride % rows == 0 && (reinterpret_cast<uintptr_t>(R) & 3u) == 0) ? 1 : 0;
    int vecC = ((ldc & 1) == 0 && (reinterpret_cast<uintptr_t>(C) & 15u) == 0) ? 1 : 0;
    int64_t bx = ((m + rows - 1) / rows + 255) / 256;
    if (bx > 0x7FFFFFFFll) return OZ_ERR_UNSUPPORTED;
    if (n > 65535ll * 65535ll) return OZ_ERR_UNSUPPORTED;
    dim3 grid(static_cast<unsigned>(bx), static_cast<unsigned>(n < 65535 ? n : 65535),
              static_cast<unsigned>((n + 65534) / 65535));
    auto kernel = set == 2 ? reconstruct_kernel<2> : set == 0 ? reconstruct_kernel<0> : reconstruct_kernel<1>;
    OZ_CUDA_CHECK(launch(kernel, grid, 256, 0, stream, R, ldr, mod_stride, m, n, shiftA, shiftB, alpha, beta, C, ldc, vecR, vecC));
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
    const int pieces = 64 * 32 * residue_bytes(set) / 4 / 256;
    if (t.tiles_m > 65535 || ntn > 65535) return OZ_ERR_UNSUPPORTED;
    const int vecC = ((ldc & 1) == 0 && (reinterpret_cast<uintptr_t>(C) & 15u) == 0) ? 1 : 0;
    const dim3 grid(static_cast<unsigned>(pieces * 16 * t.cg), static_cast<unsigned>(ntn),
                    static_cast<unsigned>(t.tiles_m));
    // Blocks that become resident beside the GEMM's keep the multiprocessor's memory split at the GEMM's (28 KiB of L1) for
    // the whole kernel: worth the overlapped launch up to a million outputs only (16384 x 16384: 11.4 -> 11.9 ms a call)
    const bool early = m * n <= (1ll << 20);
#define OZ_RECON_KERNEL(SET_, SKIP_)                                                    \
    (vecC          ? reconstruct_tiled_kernel<SET_, SKIP_, kPairs>                      \
     : beta == 0.0 ? reconstruct_tiled_kernel<SET_, SKIP_, kSingleStores>               \
                   : reconstruct_tiled_kernel<SET_, SKIP_, kSingleUpdates>)
#define OZ_RECON_TILED(SET_)                                                                                         \
    OZ_CUDA_CHECK(launch_if(early, skip ? OZ_RECON_KERNEL(SET_, true) : OZ_RECON_KERNEL(SET_, false), grid, 256, 0, stream, R, t.cg, \
                         t.tiles_n, tn0, m, n, col0, col1, shiftA, shiftB, alpha, beta, C, ldc, skip))
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
