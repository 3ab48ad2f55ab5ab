// The native FP64 path for out-of-range rows (Algorithm 1, last line: "native-FP64 fallback for
// out-of-range rows"; Algorithm 3: "ESC range check; re-issue out-of-range rows on the native-FP64
// path").  The paper names the step and leaves its arithmetic open; the reading taken here:
// every entry of a re-issued row is the compensated inner product of its row of A and column of B,
//     for kk = 0 .. k-1:   p = a b,  pe = fma(a, b, -p)            (a b = p + pe exactly)
//                          s = acc + p,  se = its exact rounding error (error-free sum)
//                          comp += pe + se,  acc = s
//     P = acc + comp,
// FP64 operations only, in this order, so that the value is a function of the data alone (no
// dependence on tiling or on the number of threads) and meets the same 2u (|A||B|) contract as the
// emulated rows.  C(i,j) = alpha P (beta = 0) or C(i,j) + alpha P (beta = 1) from the caller's old
// C: the reconstruction leaves the re-issued rows untouched.
//
// Work distribution: the re-issued rows come as an ascending list whose length only the device knows.  Two resident
// blocks an SM walk tiles of 32 x 32 outputs (2 x 2 a thread), or each half of a block by itself tiles of 8 x 16 (one a thread), chosen
// from the length by small_tiles().  The next inner indices are on their way while a stage is worked on, of small tiles two stages of 64 (the gathered
// rows come from as many DRAM pages: with 32 indices a stage 10 of 2500 rows x 900 x 2500 took 614 us a call instead of 399).  Bound: the FP64 pipe, ten
// instructions of two cycles per multiply-add and warp.  Against tiles of 16 x 16 that a whole block took, in whole rounds: 3 of 300 rows x 300 x 3000
// 247 -> 139 us a call, 700 rows x 40 x 2000 160 -> 112, 60 of 2003 x 1999 x 1501 495 -> 463.
#include "oz_internal.h"

namespace oz {
namespace {

constexpr int kFbThreads = 256, kFbBlocksPerSm = 2;
constexpr int kLargeStage = 32, kSmallStage = 64;       // inner indices per stage
constexpr int kLarge = 32;                       // rows and columns of a large tile
constexpr int kSmallRows = 8, kSmallCols = 16;   // of a small one
constexpr int kLargeRow = kLarge + 2;            // doubles per staged index of a large tile: rows stay 16-byte aligned
constexpr int kSmallLine = kSmallStage + 2;         // doubles per staged line of a small tile: two indices in one load, no bank conflicts
constexpr int kSmallDoubles = 3 * (kSmallRows + kSmallCols) * kSmallLine;       // three stages of a half block
constexpr int kFbSharedDoubles = 2 * kLargeStage * kLargeRow > 2 * kSmallDoubles ? 2 * kLargeStage * kLargeRow : 2 * kSmallDoubles;

struct NativeParams {
    int64_t m, n, k, lda, ldb, ldc;
    const double *A, *B;
    const int *list;
    const unsigned int *count;
    const int32_t *shiftB;
    double alpha, beta;
    double *C;
};

// one multiply-add of an entry: acc + a b with the rounding errors of both operations collected in comp
__device__ __forceinline__ void native_step(double a, double b, double &acc, double &comp)
{
    const double q = __dmul_rn(a, b);
    const double qe = __fma_rn(a, b, -q);
    const double s = __dadd_rn(acc, q);
    const double bb = __dsub_rn(s, acc);
    const double se = __dadd_rn(__dsub_rn(acc, __dsub_rn(s, bb)), __dsub_rn(q, bb));
    comp = __dadd_rn(comp, __dadd_rn(qe, se));
    acc = s;
}

__device__ __forceinline__ void native_store(const NativeParams &p, int64_t row, int64_t j, double acc, double comp)
{
    const double v = p.shiftB[j] == OZ_NONFINITE_SHIFT ? __longlong_as_double(0x7FF8000000000000ll) : __dadd_rn(acc, comp);
    double *out = p.C + row + j * p.ldc;
    const double x = __dmul_rn(p.alpha, v);
    *out = p.beta != 0.0 ? __dadd_rn(*out, x) : x;
}

__device__ __forceinline__ void native_large(const NativeParams &p, int64_t rows, double *shared, int64_t *row_of)
{
    constexpr int S = kLarge, T = 2, K = kLargeStage, P = kLargeRow;
    double *As = shared, *Bs = shared + K * P;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int64_t tcols = (p.n + S - 1) / S, tiles = tcols * ((rows + S - 1) / S);
    for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
        const int64_t r0 = t / tcols * S, c0 = (t - t / tcols * tcols) * S;
        __syncthreads();                         // the previous tile's rows have been used
        if (tid < S) row_of[tid] = r0 + tid < rows ? p.list[r0 + tid] : -1;
        __syncthreads();

        double acc[T][T], comp[T][T];
#pragma unroll
        for (int r = 0; r < T; ++r)
#pragma unroll
            for (int c = 0; c < T; ++c) acc[r][c] = comp[r][c] = 0.0;

        // A: consecutive threads take consecutive re-issued rows of one inner index;
        // B: consecutive threads take consecutive inner indices of one column
        const int ar = tid & (S - 1), ak = tid / S, bk = tid & (K - 1), bc = tid / K;
        const int64_t arow = row_of[ar];
        double av[4], bv[4];
        auto request = [&](int64_t k0) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int64_t kk = k0 + ak + u * (kFbThreads / S);
                av[u] = (arow >= 0 && kk < p.k) ? p.A[arow + kk * p.lda] : 0.0;
                const int64_t c = c0 + bc + u * (kFbThreads / K);
                bv[u] = (c < p.n && k0 + bk < p.k) ? p.B[(k0 + bk) + c * p.ldb] : 0.0;
            }
        };
        request(0);
        for (int64_t k0 = 0; k0 < p.k; k0 += K) {
            const int kn = p.k - k0 < K ? static_cast<int>(p.k - k0) : K;
            if (k0) __syncthreads();             // the previous stage has been read
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                As[(ak + u * (kFbThreads / S)) * P + ar] = av[u];
                Bs[bk * P + bc + u * (kFbThreads / K)] = bv[u];
            }
            __syncthreads();
            if (k0 + K < p.k) request(k0 + K);
#pragma unroll 8
            for (int kk = 0; kk < kn; ++kk) {
                const double2 a = *reinterpret_cast<const double2 *>(As + kk * P + ty * T);
                const double2 b = *reinterpret_cast<const double2 *>(Bs + kk * P + tx * T);
                native_step(a.x, b.x, acc[0][0], comp[0][0]);
                native_step(a.x, b.y, acc[0][1], comp[0][1]);
                native_step(a.y, b.x, acc[1][0], comp[1][0]);
                native_step(a.y, b.y, acc[1][1], comp[1][1]);
            }
        }
#pragma unroll
        for (int c = 0; c < T; ++c) {
            const int64_t j = c0 + tx * T + c;
            if (j >= p.n) continue;
#pragma unroll
            for (int r = 0; r < T; ++r)
                if (row_of[ty * T + r] >= 0) native_store(p, row_of[ty * T + r], j, acc[r][c], comp[r][c]);
        }
    }
}

extern __shared__ __align__(16) double fb_shared[];

// half: this half of the block's number; it keeps its own barrier and shared memory.  (Out of line: inlined it costs the large tiles 2 percent.)
__device__ __noinline__ void native_small(const NativeParams &p, int64_t rows, int half)
{
    double *shared = fb_shared + half * kSmallDoubles;
    constexpr int K = kSmallStage, L = kSmallLine, kStage = (kSmallRows + kSmallCols) * L;
    const int tid = threadIdx.x & 127, tx = tid & 15, ty = tid >> 4;
    const uint32_t base = static_cast<uint32_t>(__cvta_generic_to_shared(shared));
    const int64_t tcols = (p.n + kSmallCols - 1) / kSmallCols, tiles = tcols * ((rows + kSmallRows - 1) / kSmallRows);
    auto sync = [&] { asm volatile("bar.sync %0, 128;" ::"r"(half + 1) : "memory"); };
    const int nk = static_cast<int>((p.k + K - 1) / K);
    for (int64_t t = blockIdx.x + static_cast<int64_t>(half) * gridDim.x; t < tiles; t += 2 * gridDim.x) {      // few tiles: one to an SM
        const int64_t r0 = t / tcols * kSmallRows, c0 = (t - t / tcols * tcols) * kSmallCols;
        // Copies: a thread takes four indices of one row of A (consecutive threads consecutive rows) and one index of eight columns of B.  Rows and columns
        // behind the last one repeat it and are not stored; indices behind k are not read.
        const int ar = tid & 7, ak = tid >> 3, bk = tid & 63, bc = tid >> 6;
        const double *a_next = p.A + p.list[r0 + ar < rows ? r0 + ar : rows - 1] + ak * p.lda;
        const double *b_next = p.B + bk;
        int64_t b_off[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) b_off[u] = (c0 + bc + 2 * u < p.n ? c0 + bc + 2 * u : p.n - 1) * p.ldb;
        const uint32_t a_dst = base + static_cast<uint32_t>(ar * L + ak) * 8, b_dst = base + static_cast<uint32_t>((kSmallRows + bc) * L + bk) * 8;
        auto copy = [](uint32_t dst, const double *src, bool in) {
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(in ? 8 : 0) : "memory");
        };
        auto request = [&](int stage, int left) {       // left: indices from this stage's first one to k
            const uint32_t off = static_cast<uint32_t>(stage * kStage) * 8;
            if (left >= K) {
#pragma unroll
                for (int u = 0; u < 4; ++u) copy(a_dst + off + 128 * u, a_next + 16 * u * p.lda, true);
#pragma unroll
                for (int u = 0; u < 8; ++u) copy(b_dst + off + 2 * L * 8 * u, b_next + b_off[u], true);
            } else {
#pragma unroll
                for (int u = 0; u < 4; ++u) copy(a_dst + off + 128 * u, ak + 16 * u < left ? a_next + 16 * u * p.lda : p.A, ak + 16 * u < left);
#pragma unroll
                for (int u = 0; u < 8; ++u) copy(b_dst + off + 2 * L * 8 * u, bk < left ? b_next + b_off[u] : p.B, bk < left);
            }
            a_next += K * p.lda;
            b_next += K;
        };
        double acc = 0.0, comp = 0.0;
        const int k = static_cast<int>(p.k);
        request(0, k);
        asm volatile("cp.async.commit_group;" ::: "memory");
        if (nk > 1) request(1, k - K);
        asm volatile("cp.async.commit_group;" ::: "memory");
        int stage = 0;
        for (int i = 0; i < nk; ++i) {
            asm volatile("cp.async.wait_group 1;" ::: "memory");
            sync();                              // this stage is there, and the one before it has been read
            if (i + 2 < nk) request(stage == 0 ? 2 : stage - 1, k - (i + 2) * K);
            asm volatile("cp.async.commit_group;" ::: "memory");
            const double *As = shared + stage * kStage + ty * L, *Bs = shared + stage * kStage + (kSmallRows + tx) * L;
            const int kn = k - i * K < K ? k - i * K : K;
            if (kn == K) {
#pragma unroll 8
                for (int kk = 0; kk < K; kk += 2) {
                    const double2 a = *reinterpret_cast<const double2 *>(As + kk), b = *reinterpret_cast<const double2 *>(Bs + kk);
                    native_step(a.x, b.x, acc, comp);
                    native_step(a.y, b.y, acc, comp);
                }
            } else {
                for (int kk = 0; kk < kn; ++kk) native_step(As[kk], Bs[kk], acc, comp);
            }
            if (++stage == 3) stage = 0;
        }
        if (r0 + ty < rows && c0 + tx < p.n) native_store(p, p.list[r0 + ty], c0 + tx, acc, comp);
        sync();                                  // the stages may be filled again
    }
}

// Small tiles while they cost less: a tile of 8 x 16 takes an SM 27.5 cycles an inner index next to others, a round of 32 x 32 tiles over the resident
// blocks 365, whether one or both blocks of an SM have a tile (a last round of a few tiles somewhat less).  Calls with the small and the large ones, us, by
// rounds: 600 rows x 3000 x 300, 96 and 7: 473, 435; 150 x 5000 x 400, 41 and 3: 354, 339; 400 x 3000 x 600, 64 and 5: 595, 578; 450 x 3200 x 500, 78 and 6: 651, 676;
// 225 x 2000 x 1000, 25 and 2: 423, 448; 300 x 3000 x 1500, 49 and 4: 1182, 1315; 1200 x 1600 x 400, 102 and 7: 647, 607.
__device__ __forceinline__ bool small_tiles(int64_t rows, int64_t n, int64_t sms)
{
    const int64_t large = ((rows + kLarge - 1) / kLarge) * ((n + kLarge - 1) / kLarge), slots = kFbBlocksPerSm * sms;
    const int64_t small = ((rows + kSmallRows - 1) / kSmallRows) * ((n + kSmallCols - 1) / kSmallCols);
    return 3 * ((small + sms - 1) / sms) < 40 * ((large + slots - 1) / slots);
}

__global__ void __launch_bounds__(kFbThreads, kFbBlocksPerSm)
native_rows_kernel(const __grid_constant__ NativeParams p, int sms)
{
    dependency_release();
    dependency_wait();
    const int64_t rows = *p.count;
    if (rows == 0) return;
    __shared__ int64_t row_of[kLarge];
    if (small_tiles(rows, p.n, sms)) native_small(p, rows, static_cast<int>(threadIdx.x >> 7));
    else native_large(p, rows, fb_shared, row_of);
}

}  // namespace

oz_status_t launch_native_rows(int64_t m, int64_t n, int64_t k, const double *A, int64_t lda,
                               const double *B, int64_t ldb, const int *list, const unsigned int *count,
                               const int32_t *shiftB, double alpha, double beta, double *C, int64_t ldc,
                               cudaStream_t stream)
{
    // refused as ever: more than 65535 groups of 64 rows, or 2^31 groups of 64 columns
    if ((m + 63) / 64 > 65535 || (n + 63) / 64 > 2147483647ll) return OZ_ERR_UNSUPPORTED;
    const int sms = sm_count();
    NativeParams p{m, n, k, lda, ldb, ldc, A, B, list, count, shiftB, alpha, beta, C};
    // as many blocks as are resident at once, or fewer where even the smallest tiles are fewer
    const int64_t most = ((m + kSmallRows - 1) / kSmallRows) * ((n + kSmallCols - 1) / kSmallCols), cap = static_cast<int64_t>(kFbBlocksPerSm) * sms;
    constexpr size_t shared = kFbSharedDoubles * sizeof(double);
    static std::atomic<unsigned long long> ready{0};
    OZ_CUDA_CHECK(allow_shared(native_rows_kernel, shared, ready));
    OZ_CUDA_CHECK(launch(native_rows_kernel, dim3(static_cast<unsigned>(most < cap ? most : cap)), kFbThreads, shared, stream, p, sms));
    count_launch();
    OZ_CUDA_CHECK(cudaGetLastError());
    return OZ_OK;
}

}  // namespace oz
