// Internal declarations shared by the translation units of liboz_b200.so.
// Nothing here is part of the public ABI (see include/oz.h).
#pragma once

#include <atomic>
#include <cuda_runtime.h>
#include <stdint.h>

#include "oz.h"

namespace oz {

constexpr int kMaxR = 15;          // moduli in the largest supported set (A)
constexpr int kMaxPlanes = 44;     // stored planes of set A with two-limb digits
// The plane look-up table of a set: the packed plane bytes of the residues of the moduli whose digits are not
// computed (lut_span() words each).  kLutGuard: entries in front of and behind those of the balanced residues, so that an
// operand element beyond the exact range of the conversion (see max_operand()) still indexes the table.
constexpr int kLutGuard = 8;
constexpr int kLutWords = 4160;    // >= lut_words() of any set (S: 4132, E: 2808, A: 3704)

// ---- modulus sets (Sec. 2 step (ii) for S; "Candidate E" and "Candidate A" paragraphs) ---
constexpr int kNumSets = 3;
__host__ __device__ constexpr int set_r(int set) { return set == 0 ? 12 : (set == 1 ? 13 : 15); }

__host__ __device__ constexpr int modulus(int set, int i)
{
    constexpr int S[15] = {1089, 1024, 961, 841, 625, 529, 511, 509, 503, 499, 491, 487, 1, 1, 1};
    constexpr int E[15] = {1089, 1024, 961, 841, 625, 529, 251, 247, 241, 239, 233, 229, 227, 1, 1};
    constexpr int A[15] = {256, 255, 253, 251, 247, 241, 239, 233, 229, 227, 223, 217, 211, 199, 197};
    return set == 0 ? S[i] : (set == 1 ? E[i] : A[i]);
}

// bytes of one stored residue in [0, m): the moduli of set A fit a byte
__host__ __device__ constexpr int residue_bytes(int set) { return set == 2 ? 1 : 2; }

// How the private residue array of the whole-method calls stores a residue of modulus i: some representative in [0, m + 1], modulo 2^10
// or 2^8 where m is that, in one byte, in ten bits (moduli up to 1024) or in two bytes.  (Set A: canonical.)
enum { kStoredByte, kStoredTen, kStoredPair };
__host__ __device__ constexpr int form_of(int m) { return m <= 256 ? kStoredByte : m <= 1024 ? kStoredTen : kStoredPair; }
__host__ __device__ constexpr int form_bytes(int form) { return form == kStoredByte ? 2048 : form == kStoredTen ? 2560 : 4096; }
__host__ __device__ constexpr int stored_form(int set, int i) { return form_of(modulus(set, i)); }
// where a modulus' residues of a 32 x 64 patch of the output (see ResidueTiling) begin, form_bytes() each, and bytes of a whole patch.  (Sums over the moduli
// before it, for constants: the host takes them along, fill_mod_info().)
__host__ __device__ constexpr int stored_start(int set, int i)
{
    int o = 0;
    for (int j = 0; j < i; ++j) o += form_bytes(stored_form(set, j));
    return o;
}
__host__ __device__ constexpr int patch_bytes(int set) { return stored_start(set, set_r(set)); }

// square root of a square modulus, 0 otherwise
__host__ __device__ constexpr int square_root(int m)
{
    for (int s = 2; s * s <= m; ++s)
        if (s * s == m) return s;
    return 0;
}

// Plane layouts of one operand:
//   kLayoutDigits  2 (square) or 3 digit planes per modulus: d0, d1[, d0+d1]   (Sec. 2 "FP8 variant")
//   kLayoutNative  1 plane: the centred residue itself as an INT8 operand (byte moduli only;
//                  Sec. 2 "The substrate transition")
//   kLayoutMerged  the A operand of the merged-accumulator schedule (discussion of Table "tuples",
//                  N_acc = 2): the d1 plane of every non-square modulus holds the pre-scaled -16*d1
//                  (d1 enters only through d1*e1); same plane count as kLayoutDigits
//   kLayoutMergedI8A / kLayoutMergedI8B  the same schedule on INT8 digit planes, where -16*d1 does
//                  not fit a byte: both operands carry 4*d1 in place of d1 and the A operand -d0
//                  in place of d0, so that (-d0) e0 + (4 d1)(4 e1) = -(d0 e0 - 16 d1 e1)
//   kLayoutDigitsI8  kLayoutDigits with INT8 instead of E4M3 bytes
//   kLayoutTwo / kLayoutFour (and their INT8 forms)  the two-plane schedule of the whole-method calls with few columns:
//                  A holds d0 and d1 of every modulus, B the digits e0, e1 of e and, for a non-square, f0, f1 of
//                  f = 16 e mod m.  Digits to the base s (squares) or 16, each rounded to nearest: the schedule needs no
//                  digit sums, so no carry of Lemma 1 and no table
constexpr int kLayoutDigits = 0, kLayoutNative = 1, kLayoutMerged = 2, kLayoutMergedI8A = 3,
              kLayoutMergedI8B = 4, kLayoutDigitsI8 = 5, kLayoutTwo = 6, kLayoutTwoI8 = 7, kLayoutFour = 8, kLayoutFourI8 = 9;
constexpr int kNumLayouts = 10;
__host__ __device__ constexpr bool two_plane_layout(int layout) { return layout >= kLayoutTwo; }

__host__ __device__ constexpr int planes_of(int m, int layout = kLayoutDigits)
{
    return layout == kLayoutNative ? 1 : (square_root(m) || layout == kLayoutTwo || layout == kLayoutTwoI8) ? 2 : two_plane_layout(layout) ? 4 : 3;
}

__host__ __device__ constexpr int first_plane(int set, int i, int layout = kLayoutDigits)
{
    int p = 0;
    for (int j = 0; j < i; ++j) p += planes_of(modulus(set, j), layout);
    return p;
}

__host__ __device__ constexpr int p_store(int set, int layout = kLayoutDigits)
{
    return first_plane(set, set_r(set), layout);
}

// The same, tabulated at compile time for the host code that runs on every call (the functions above walk the
// set and search square roots).
struct SetTables {
    int root[3][kMaxR];                         // square root of a square modulus, 0 otherwise
    int first[3][kNumLayouts][kMaxR + 1];               // first plane of modulus i per layout; [r]: the number of planes
};
constexpr SetTables make_set_tables()
{
    SetTables t{};
    for (int set = 0; set < 3; ++set)
        for (int i = 0; i < set_r(set); ++i) {
            t.root[set][i] = square_root(modulus(set, i));
            for (int layout = 0; layout < kNumLayouts; ++layout)
                t.first[set][layout][i + 1] = t.first[set][layout][i] + planes_of(modulus(set, i), layout);
        }
    return t;
}
constexpr SetTables kSetTables = make_set_tables();

// largest k for which the merged accumulator d0 e0 - 16 d1 e1 stays exact in FP32: the merged term
// reaches 4095 on the 9-bit tail of S and 1088 on byte moduli
__host__ __device__ constexpr int64_t merged_k_limit(int set) { return set == 0 ? 4097 : 15420; }

// table words of one modulus: canonical residues of a power of two, balanced residues between two guards of a
// non-square, none for an odd square (its digits are computed)
__host__ __device__ constexpr int lut_span(int m)
{
    return (m & (m - 1)) == 0 ? m : (square_root(m) ? 0 : m + 2 * kLutGuard);
}

__host__ __device__ constexpr int lut_offset(int set, int i)
{
    int o = 0;
    for (int j = 0; j < i; ++j) o += lut_span(modulus(set, j));
    return o;
}

// words of a set's table, rounded up to whole 16-byte groups
__host__ __device__ constexpr int lut_words(int set) { return (lut_offset(set, set_r(set)) + 3) / 4 * 4; }
static_assert(lut_words(0) <= kLutWords && lut_words(1) <= kLutWords && lut_words(2) <= kLutWords, "table size");

// table words that a conversion into `layout` needs: native residues and the two-plane schedule need none
__host__ __device__ constexpr int lut_words_of(int set, int layout)
{
    return layout == kLayoutNative || two_plane_layout(layout) ? 0 : lut_words(set);
}

// 2^e mod m
__host__ __device__ constexpr uint32_t pow2_mod(int e, uint32_t m)
{
    uint32_t v = 1 % m;
    for (int j = 0; j < e; ++j) v = (v * 2u) % m;
    return v;
}

// floor(2^32 / m)
__host__ __device__ constexpr uint32_t barrett_magic(uint32_t m)
{
    return static_cast<uint32_t>(0x100000000ull / m);
}

inline int64_t round_up(int64_t v, int64_t a) { return (v + a - 1) / a * a; }

// ---- route decoding ----------------------------------------------------------------------
struct Route {
    int substrate;  // 0 fp8, 1 int8 (two-limb digits), 2 int8 native (one residue plane, set A only)
    int acc;        // 0 unspecified, 1 merged accumulators, 2 separate accumulators, 3 two-plane schedule (internal)
    bool automatic; // the schedule was left to the library
    bool native() const { return substrate == 2; }
    bool merged() const { return acc == 1; }
    bool two_plane() const { return acc == 3; }
    // plane layout of the operand on `side` (0: rows of A, 1: columns of B)
    int layout(int side) const
    {
        if (native()) return kLayoutNative;
        if (two_plane()) return (side == 0 ? kLayoutTwo : kLayoutFour) + (substrate == 1 ? 1 : 0);
        if (!merged()) return substrate == 1 ? kLayoutDigitsI8 : kLayoutDigits;
        if (substrate == 1) return side == 0 ? kLayoutMergedI8A : kLayoutMergedI8B;
        return side == 0 ? kLayoutMerged : kLayoutDigits;
    }
    bool hosted;    // whole-method calls: CRT recombination on the INT8 tensor pipe (OZ_RECON_TENSOR)
    bool fallback;  // oz_dgemm / oz_dgemm_ex: out-of-range rows re-issued on the native FP64 path
    bool fused;     // oz_dgemm / oz_dgemm_ex: A converted inside the product kernel (storage mode F)
    int quant;      // 0 rn, 1 tz
    int rule;       // 0 maxexp, 1 cs, 2 accurate (shifts from the extra bound product)
};
bool decode_route(uint32_t route, Route *out);
bool decode_route_for_set(int set, uint32_t route, Route *out);
oz_status_t resolve_schedule(int set, int64_t k, int64_t n, bool automatic, Route *rt);   // merged or separate accumulators   // also rejects native INT8 off set A

// ---- per-device state --------------------------------------------------------------------
// Builds the lookup tables and constant blocks on the current device the first time it is used.
oz_status_t ensure_device_ready();

// device addresses of the per-device objects (valid after ensure_device_ready())
const uint32_t *device_lut(int set, int substrate);  // substrate 0, 1: kLutWords packed plane bytes
unsigned int *device_status_word();

void count_launch(int n = 1);

// quantisation budgets (host)
void budget_maxexp(int set, int64_t k, int *tA, int *tB);
void cs_bound_squared(int set, int64_t k, uint64_t *lo, uint64_t *hi);  // G^2 as 128 bits

// Where a plane keeps byte (line, kk): (kk / 128) chunk_stride + line line_stride + kk % 128.
//   public:   lines of row_pitch bytes (line_stride = row_pitch, chunk_stride = 128)
//   private:  K chunk by K chunk, the 128-byte pieces of all lines one behind the other (line_stride = 128,
//             chunk_stride = 128 lines; row_pitch = k rounded up to 128, so the size is that of the public layout).
//             A 128-line TMA box is then 16 KiB of consecutive bytes, and a conversion tile stores 2 KiB at a time instead
//             of 128-byte pieces a row pitch apart (32768 x 4096, side 0, set S: 1.39 against 1.61 ms).
struct PlaneGeom {
    int64_t plane_stride, row_pitch, line_stride, chunk_stride;
};
inline PlaneGeom public_planes(int64_t plane_stride, int64_t row_pitch) { return {plane_stride, row_pitch, row_pitch, 128}; }
inline PlaneGeom private_planes(int64_t lines, int64_t pitch) { return {lines * pitch, pitch, 128, 128 * lines}; }

// ---- stage launchers (host side of each .cu) ---------------------------------------------
// `alone`: no other chain of kernels runs beside this one (see launch_if())
oz_status_t launch_deconstruct(int side, int64_t lines, int64_t k, const double *X, int64_t ldx,
                               int set, const Route &rt, uint8_t *planes, const PlaneGeom &geom,
                               int32_t *shift, void *scratch, bool alone, cudaStream_t stream);

// Tile-ordered private residue array of the whole-method calls.  The output is cut into tiles of
// 256 rows x tile_cols columns (128, or 256 when CTA pairs are used); a tile is 16 patches (32 with
// pairs: rank-major) of 32 columns x 64 rows, one per epilogue warp, patch w = quarter + 4 * part
// covering columns 32 * quarter .. +31 (of the rank's 128) and rows 64 * part .. +63.
// Order in memory: tile row, tile column, CTA rank, patch, modulus -- the residues of one patch are consecutive, modulus
// after modulus (stored_start()).  Those of a modulus are stored as [16-byte chunk c][column], chunk c holding 16
// consecutive rows (two-byte form: 8), word s of it rows 2 s, 2 s + 1, 2 s + 8 and 2 s + 9 -- the rows of one thread of the
// reconstruction, four of which then access 64 contiguous bytes of C (row_of()).  Ten-bit form: the low bytes like that, then 16 bytes
// a column with the high bits, word c for the rows of chunk c: bits 2 s and 2 s + 1 of its byte e belong to byte e of word s.
// Set S takes 15.75 bytes an output, where two bytes a residue take 24; E 15.25 instead of 26; A 15.
struct ResidueTiling {
    int cg;              // 1: tiles of 128 columns, 2: CTA pairs, tiles of 256 columns
    int tile_cols;
    int tiles_m, tiles_n;
    int64_t mod_stride;  // elements per modulus in total (tiles are stored whole, padding included)
};
ResidueTiling residue_tiling(int64_t m, int64_t n, int set);

// Both operands of a product in one launch, when the one-kernel form takes both (*taken says whether it did);
// otherwise nothing is launched
struct OperandJob {
    int64_t lines;
    const double *X;
    int64_t ldx;
    uint8_t *planes;
    PlaneGeom geom;
    int32_t *shift;
    void *scratch;
};
oz_status_t launch_deconstruct_pair(const OperandJob &a, const OperandJob &b, int64_t k, int set, const Route &rt,
                                    bool *taken, cudaStream_t stream);

// pieces of launch_deconstruct, and the steps of the accurate rule between them.  The scans take side 0 (a), side 1 (b) or both.
struct ScanJob {
    int64_t lines;
    const double *X;
    int64_t ldx;
    int32_t *shift;
    void *scratch;
    void *spare;                // the operand's first plane, which the conversion fills after the scan, for sums in between; null: none
};
// whether launch_deconstruct() takes the scans and the conversion into private planes (else the one-kernel or the cluster form)
bool three_passes(int side, const ScanJob &job, int64_t k, int set, const Route &rt);
oz_status_t launch_scan(const ScanJob *a, const ScanJob *b, int64_t k, int set, const Route &rt, bool alone, cudaStream_t stream);
oz_status_t launch_convert_planes(int side, int64_t lines, int64_t k, const double *X, int64_t ldx,
                                  int set, const Route &rt, uint8_t *planes, const PlaneGeom &geom,
                                  const int32_t *shift, bool alone, cudaStream_t stream);
oz_status_t launch_bound_planes(const ScanJob &a, uint8_t *planeA, const ScanJob &b, uint8_t *planeB, int64_t k, int64_t pitch,
                                cudaStream_t stream);
unsigned int *bound_maxima(void *scratch, int64_t lines);      // one word per line, word stride 2
oz_status_t launch_accurate_finalize(const ScanJob &a, const ScanJob &b, int budget_log2, cudaStream_t stream);
// the bound product on the tensor cores: rowmax[2 i] / colmax[2 j] receive (atomicMax) the bit pattern
// of max_j / max_i of sum_k GA[i][k] GB[j][k], an integer-valued FP32 number; k <= kBoundKMax
constexpr int64_t kBoundKMax = 16384;
oz_status_t launch_bound_gemm(int64_t m, int64_t n, int64_t k, const uint8_t *GA, int64_t pitchA,
                              const uint8_t *GB, int64_t pitchB, unsigned int *rowmax,
                              unsigned int *colmax, cudaStream_t stream);
int accurate_budget_log2(int set);
// exponent-span check: threshold of the set against the product of the two operands' flatness codes
unsigned int esc_threshold(int set);

// tiled: R is the tile-ordered private array (ldr and mod_stride are then ignored), and the planes are in the private layout
oz_status_t launch_residue_gemm(int64_t m, int64_t n, int64_t k, const uint8_t *PA,
                                int64_t strideA, int64_t pitchA, const uint8_t *PB,
                                int64_t strideB, int64_t pitchB, int set, const Route &rt,
                                void *R, int64_t ldr, int64_t mod_stride, bool tiled,
                                cudaStream_t stream);

// Whether a whole-method call takes the two-plane schedule (planes private to the call, schedule left to the library)
bool two_plane_applies(int64_t m, int64_t n, const Route &rt);

// Storage mode F: residue products with A converted on the fly inside the kernel (n <= 128, merged
// schedule on digit planes, k within the exact depth of one accumulator); public residue layout
bool fused_gemm_applies(int64_t m, int64_t n, int64_t k, int set, const Route &rt);
oz_status_t launch_fused_gemm(int64_t m, int64_t n, int64_t k, const double *A, int64_t lda, const int32_t *shiftA,
                              const uint8_t *PB, int64_t pitchB, int set, const Route &rt,
                              void *R, int64_t ldr, int64_t mod_stride, cudaStream_t stream);

// reconstruction from the tile-ordered array, columns [col0, col1) of the m x n output
oz_status_t launch_reconstruct_tiled(int64_t m, int64_t n, const void *R, const int32_t *shiftA,
                                     const int32_t *shiftB, int set, double alpha, double beta,
                                     double *C, int64_t ldc, int64_t col0, int64_t col1,
                                     cudaStream_t stream, const unsigned char *skip_rows = nullptr);

oz_status_t launch_reconstruct(int64_t m, int64_t n, const void *R, int64_t ldr,
                               int64_t mod_stride, const int32_t *shiftA, const int32_t *shiftB,
                               int set, double alpha, double beta, double *C, int64_t ldc,
                               cudaStream_t stream);

// uploads the constants of the reconstruction on the tensor pipe, of every set, to the current device
oz_status_t upload_hosted_constants();

// reconstruction from the tile-ordered array with the CRT recombination on the INT8 tensor pipe
oz_status_t launch_reconstruct_hosted(int64_t m, int64_t n, const void *R, const int32_t *shiftA,
                                      const int32_t *shiftB, int set, double alpha, double beta,
                                      double *C, int64_t ldc, int64_t col0, int64_t col1,
                                      cudaStream_t stream);

// Out-of-range rows (Algorithm 1, last line; Algorithm 3, "ESC range check"): flags, ascending list and
// number of the rows that go to the native FP64 path, from the scan results that the
// deconstruction left in the two scratch blocks; and the native path itself
oz_status_t launch_esc_rows(void *scratchA, int64_t m, void *scratchB, int64_t n, int64_t k, int set,
                            unsigned char *flag, int *list, unsigned int *count, cudaStream_t stream);
oz_status_t launch_native_rows(int64_t m, int64_t n, int64_t k, const double *A, int64_t lda,
                               const double *B, int64_t ldb, const int *list, const unsigned int *count,
                               const int32_t *shiftB, double alpha, double beta, double *C, int64_t ldc,
                               cudaStream_t stream);

// ---- launching ---------------------------------------------------------------------------
// The kernels of a call are launched as programmatic dependents of their predecessors on the stream: their blocks may
// become resident, and set up what needs no global memory, while the predecessor's last blocks run.  In return every
// kernel executes dependency_wait() on every path (so that its own completion implies its predecessor's) and before its
// first access to global memory, but for the tables that ensure_device_ready() has put there before any launch, and
// lets its successor in with dependency_release() at once.  256^3: 22.9 -> 19.0 us of GPU time a call together with the joint deconstruction of both operands.
#ifdef __CUDACC__
__device__ __forceinline__ void dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void dependency_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// dependent = false: an ordinary launch, for the chains of kernels that run beside another stream's: there the blocks that
// wait early would hold the registers and shared memory that the other chain needs (2003 x 1999 x 1501 with the row
// check: 505 -> 621 us, 6912 x 6912 x 1024: 2.25 -> 2.34 ms).
template <class... Params, class... Args>
cudaError_t launch_if(bool dependent, void (*kernel)(Params...), dim3 grid, int threads, size_t smem, cudaStream_t stream, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(static_cast<unsigned>(threads));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = dependent ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}

template <class... Params, class... Args>
cudaError_t launch(void (*kernel)(Params...), dim3 grid, int threads, size_t smem, cudaStream_t stream, Args... args)
{
    return launch_if(true, kernel, grid, threads, smem, stream, args...);
}

// Opts a kernel in to dynamic shared memory beyond 48 KiB, once per device (one flag per call site's kernel).
template <class Kernel>
cudaError_t allow_shared(Kernel kernel, size_t bytes, std::atomic<unsigned long long> &done)
{
    int dev = 0;
    cudaError_t rc = cudaGetDevice(&dev);
    if (rc != cudaSuccess) return rc;
    const unsigned long long bit = 1ull << (dev & 63);
    if (done.load(std::memory_order_relaxed) & bit) return cudaSuccess;
    rc = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(bytes));
    if (rc == cudaSuccess) done.fetch_or(bit, std::memory_order_relaxed);
    return rc;
}
#endif
constexpr size_t kMaxShared = 227 * 1024;      // dynamic shared memory a block may have

// multiprocessors of the current device (read once per device)
int sm_count();

#define OZ_CUDA_CHECK(expr)                                  \
    do {                                                     \
        cudaError_t e__ = (expr);                            \
        if (e__ != cudaSuccess) return OZ_ERR_CUDA;          \
    } while (0)

}  // namespace oz
