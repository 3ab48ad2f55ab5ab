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
// Work distribution: the re-issued rows come as an ascending list whose length only the device knows.  Resident
// blocks (two per SM) walk tiles of S x S outputs, S = 32 (2 x 2 a thread) or 16 (one a thread), chosen from the
// length by small_tiles().  1024 / S inner indices are staged in shared memory at a time and the next ones
// are requested before the arithmetic.  Bound: the FP64 pipe, ten instructions per multiply-add, 0.88 of it
// when every row is re-issued (3000 x 3000 x 1500: 8.56 ms; 8.53 with 64 x 64 tiles in one pass over the grid).  With few
// rows those tiles left most SMs idle; now 60 of 2003 rows x 1999 x 1501 take 0.20 instead of 0.71 ms, 85 of
// 3000 rows x 3000 x 3000 0.60 instead of 1.39, 3 of 300 rows x 300 x 3000 0.13 instead of 1.35.
#include "oz_internal.h"

namespace oz {
namespace {

constexpr int kFbThreads = 256, kFbBlocksPerSm = 2;
constexpr int kFbStage = 1024;                   // elements of each operand per stage
constexpr int kFbStageDoubles = 64 * (16 + 2);   // one staged operand: the larger of (1024 / S) (S + 2)
static_assert(32 * (32 + 2) <= kFbStageDoubles, "stage size");

struct NativeParams {
    int64_t m, n, k, lda, ldb, ldc;
    const double *A, *B;
    const int *list;
    const unsigned int *count;
    const int32_t *shiftB;
    double alpha, beta;
    double *C;
};

// A round of 32 x 32 tiles over the resident blocks takes 0.20 us per inner index whether one or both blocks of an
// SM have a tile (the chains of dependent additions bound it), a round of 16 x 16 tiles 0.066 us: the smaller tiles
// win while their rounds are fewer than three times those of the larger.
__device__ __forceinline__ bool small_tiles(int64_t rows, int64_t n, int64_t slots)
{
    const int64_t tiles32 = ((rows + 31) / 32) * ((n + 31) / 32), tiles16 = ((rows + 15) / 16) * ((n + 15) / 16);
    return (tiles16 + slots - 1) / slots < 3 * ((tiles32 + slots - 1) / slots);
}

template <int S>
__device__ __forceinline__ void native_tiles(const NativeParams &p, int64_t rows, double *As, double *Bs, int64_t *row_of)
{
    constexpr int T = S / 16;                    // outputs of a thread per direction
    constexpr int K = kFbStage / S;              // inner indices per stage
    constexpr int kUnroll = T == 1 ? 16 : 8;      // keeps several inner indices' chains in flight
    constexpr int P = S + 2;                     // doubles per staged index: rows stay 16-byte aligned
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
#pragma unroll kUnroll
            for (int kk = 0; kk < kn; ++kk) {
                double a[T], b[T];
                if constexpr (T == 1) {
                    a[0] = As[kk * P + ty];
                    b[0] = Bs[kk * P + tx];
                } else {
#pragma unroll
                    for (int h = 0; h < T; h += 2) {
                        const double2 a2 = *reinterpret_cast<const double2 *>(As + kk * P + ty * T + h);
                        const double2 b2 = *reinterpret_cast<const double2 *>(Bs + kk * P + tx * T + h);
                        a[h] = a2.x; a[h + 1] = a2.y;
                        b[h] = b2.x; b[h + 1] = b2.y;
                    }
                }
#pragma unroll
                for (int r = 0; r < T; ++r)
#pragma unroll
                    for (int c = 0; c < T; ++c) {
                        const double q = __dmul_rn(a[r], b[c]);
                        const double qe = __fma_rn(a[r], b[c], -q);
                        const double s = __dadd_rn(acc[r][c], q);
                        const double bb = __dsub_rn(s, acc[r][c]);
                        const double se = __dadd_rn(__dsub_rn(acc[r][c], __dsub_rn(s, bb)), __dsub_rn(q, bb));
                        comp[r][c] = __dadd_rn(comp[r][c], __dadd_rn(qe, se));
                        acc[r][c] = s;
                    }
            }
        }

        const double nan = __longlong_as_double(0x7FF8000000000000ll);
#pragma unroll
        for (int c = 0; c < T; ++c) {
            const int64_t j = c0 + tx * T + c;
            if (j >= p.n) continue;
            const bool bad = p.shiftB[j] == OZ_NONFINITE_SHIFT;
#pragma unroll
            for (int r = 0; r < T; ++r) {
                const int64_t row = row_of[ty * T + r];
                if (row < 0) continue;
                const double v = bad ? nan : __dadd_rn(acc[r][c], comp[r][c]);
                double *out = p.C + row + j * p.ldc;
                const double x = __dmul_rn(p.alpha, v);
                *out = p.beta != 0.0 ? __dadd_rn(*out, x) : x;
            }
        }
    }
}

__global__ void __launch_bounds__(kFbThreads, kFbBlocksPerSm)
native_rows_kernel(const __grid_constant__ NativeParams p, int sms)
{
    dependency_release();
    dependency_wait();
    const int64_t rows = *p.count;
    if (rows == 0) return;
    __shared__ __align__(16) double As[kFbStageDoubles];
    __shared__ __align__(16) double Bs[kFbStageDoubles];
    __shared__ int64_t row_of[32];
    if (small_tiles(rows, p.n, static_cast<int64_t>(kFbBlocksPerSm) * sms)) native_tiles<16>(p, rows, As, Bs, row_of);
    else native_tiles<32>(p, rows, As, Bs, row_of);
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
    const int64_t most = ((m + 15) / 16) * ((n + 15) / 16), cap = static_cast<int64_t>(kFbBlocksPerSm) * sms;
    OZ_CUDA_CHECK(launch(native_rows_kernel, dim3(static_cast<unsigned>(most < cap ? most : cap)), kFbThreads, 0, stream, p, sms));
    count_launch();
    OZ_CUDA_CHECK(cudaGetLastError());
    return OZ_OK;
}

}  // namespace oz
