// Residue GEMMs on the 5th-generation tensor cores (Algorithm 1, the loop over moduli; Sec. 2
// "FP8 variant"; Eq. 8), with the per-modulus combination and `mod m_i` fused into the epilogue.
//
// For every modulus the product of two centred residues is rebuilt from exact plane products:
//   square m = s^2 (planes d0,d1):        d e = d0 e0 + s (d1 e0 + d0 e1)              (mod m)
//   non-square (planes d0,d1,dS=d0+d1):   d e = -15 d0 e0 + 16 dS eS + 240 d1 e1       (Eq. 8)
// so one (modulus, output tile) work item is a short list of "accumulator jobs", each a K-loop
// of tcgen05.mma instructions into one TMEM accumulator:
//   square:      job 0 = D0.E0 (weight 1);  job 1 = [D1|D0].[E0|E1] (two K-loops, weight s)
//   non-square:  job 0 = D0.E0 (-15);  job 1 = DS.ES (16);  job 2 = D1.E1 (240)
//   non-square, merged accumulators (FP8): job 0 = [D0|-16 D1].[E0|E1] (-15); job 1 = DS.ES (16)
//                -- the regrouping discussed under Table "tuples" (N_acc = 2); one TMEM drain
//                fewer per modulus, and the drains are what the epilogue pays for at small k
// Three MMA K-loops per modulus either way (p_mma = 3r); the three of a square run as one loop over its four
// tiles per K chunk, into both accumulator slots (pair_squares).
//
// Split-K inside the kernel: a job whose K range exceeds the exact depth of its accumulator (4097
// or 15420 for the merged job 0, 32768 for every other FP32 accumulator, 2^31 / term size in
// INT32) is cut into segments of whole K chunks; each segment has an accumulator of its own that
// is reduced modulo m_i before it is weighted and added, so the residues are those of the whole K.
//
// The tile is computed transposed: the MMA's M dimension (128 TMEM lanes) runs over 128 columns
// j of C (planes of B), its N dimension (256 TMEM columns) over 256 rows i of C (planes of A).
// An epilogue thread therefore owns one column j and a run of 64 consecutive rows, which is
// contiguous in the column-major residue array; a warp transposes its 32 x 64 block through a
// small swizzled shared-memory buffer so that each store instruction writes whole lines.
//
// Kernel structure (one persistent CTA per SM, 576 threads, up to 96 registers each; launched as
// clusters of two CTAs that share one tcgen05.mma.cta_group::2 unless n pads badly to 256):
//   warp 0       TMA producer: 128-byte-swizzled K-major tiles of B (128 lines) and A (256 lines,
//                or this CTA's half of them in a pair) into a shared-memory ring of 192 KiB
//                (4 stages of 48 KiB, or 6 of 32 KiB in a pair), no multicast
//   warp 1       MMA issuer: an elected lane issues tcgen05.mma (M=128 or 256 across the pair, N=256,
//                K=32); accumulators live in TMEM, two slots of 256 columns used alternately per job
//   warps 2..17  epilogue (4 per TMEM lane quarter, 64 columns each): tcgen05.ld the finished slot,
//                reduce each accumulator modulo m_i in FP32 (all values are integers below 2^24,
//                every step exact), fold it with the job's weight into a per-thread running
//                combination held in registers, release the slot; after the last job reduce once
//                more and store the residues (uint16, or uint8 for the all-byte set)
// so the epilogue of one job overlaps the K-loop of the next, and TMEM never needs the three
// accumulators of a non-square modulus at once.
//
// Exactness: the FP8 route relies on integer-valued partial sums below 2^24 being accumulated
// without rounding (accumulation invariant of Algorithm 2, Lemma 1) and its epilogue works in
// exact FP32; the INT8 routes accumulate in INT32 and their epilogue is integer arithmetic
// (weights by IMAD, `mod m` by a multiply-high division on a biased, non-negative value).
//
// Native INT8 route (all-byte set A only): the centred residue itself is the operand, so a modulus
// is ONE job -- one plane, one K-loop, weight 1 -- and the schedule has r = 15 products; its
// accumulator is loaded straight into the combination registers and the slot released at once.
//
// Every barrier wait is bounded: on expiry the CTA records OZ_ERR_TIMEOUT in the device status
// word, every role leaves its loops, in-flight copies are given a bounded time to land, TMEM is
// freed and the kernel returns.
#include <cuda.h>
#include <atomic>
#include <cstdlib>

#include <cstring>

#include "oz_internal.h"
#include "oz_convert.cuh"

namespace oz {
namespace {

constexpr int BLOCK_M = 128;                       // MMA M: columns j of C (lines of B)
constexpr int BLOCK_N = 256;                       // MMA N: rows i of C (lines of A); NARROW_N where tiles are few
constexpr int NARROW_N = 64;
constexpr int BLOCK_K = 128;                       // bytes = elements (8-bit operands)
constexpr int UMMA_K = 32;                         // 8-bit operands: 32 elements per instruction
constexpr int RING_BYTES = 4 * 49152;              // the shared-memory ring: 192 KiB, whatever a stage holds
constexpr int A_BYTES = BLOCK_M * BLOCK_K;         // 16 KiB: MMA operand a = 128 lines of B's planes per CTA

// CG = 1: one CTA per tile of 128 columns x 256 rows of C.
// CG = 2: a pair of CTAs (cluster of 2) shares one tcgen05.mma.cta_group::2 of M = 256: the tile is
//         256 columns x 256 rows; each CTA loads its own 128 lines of B's planes (operand a) and HALF
//         of the 256 lines of A's planes (operand b), the tensor core reads both halves, and each
//         CTA's TMEM holds the accumulators of its own 128 columns.  Per CTA this halves the
//         shared-memory traffic of operand b and the TMA bytes per MMA.
template <int CG, int BN = BLOCK_N>
struct Tile {
    static constexpr int B_LINES = BN / CG;                     // lines of A's planes loaded per CTA
    static constexpr int B_BYTES = B_LINES * BLOCK_K;            // 32 KiB / 16 KiB
    static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;        // 48 KiB / 32 KiB
    static constexpr int STAGES = RING_BYTES / STAGE_BYTES;      // 4 / 6, narrow tiles 8 / 9
    static constexpr int TILE_J = BLOCK_M * CG;                  // columns of C per work item
};
// Two-plane schedule (SLIM, one tile of columns): a stage holds one of A's planes and the two tiles of B's planes that it
// meets, one per accumulator.  SLIM is the number of lines of B that are loaded: with 64 a fourth stage fits, and the two
// tiles, one behind the other, are the 128 lines of ONE MMA: both accumulators in one slot, the first in TMEM lanes 0 to 63.
template <int SLIM, int BN = BLOCK_N>
struct SlimTile {
    static constexpr int B_BYTES = SLIM * BLOCK_K;
    static constexpr int STAGE_BYTES = 2 * B_BYTES + BN * BLOCK_K;           // 64 or 48 KiB
    static constexpr int STAGES = RING_BYTES / STAGE_BYTES;                  // 3 or 4, narrow tiles 4 or 8
};
constexpr int TMEM_COLS = 512;                     // two accumulator slots of BLOCK_N columns
constexpr int NUM_THREADS = 576;                   // 18 warps, five on one of the schedulers: 96 registers each
constexpr int FIRST_EPI_WARP = 2;                  // warp 0: producer, warp 1: MMA issuer
constexpr int EPI_WARPS = 16;
#ifndef OZ_DRAIN_W
#define OZ_DRAIN_W 16
#endif
constexpr int DRAIN_W = OZ_DRAIN_W;                // accumulator columns per tcgen05.ld of a drain: 64 running
                                                   // values + 16 loaded ones stay inside the 96 registers
constexpr int XPOSE_BYTES = 16 * 128;                // per epilogue warp: 16 lines x 128 bytes
constexpr size_t SMEM_BYTES = RING_BYTES + EPI_WARPS * XPOSE_BYTES + 1024 /*alignment slack*/ + 384 /*barriers*/;

struct ModInfo {
    float m, inv_m;
    uint32_t w[3];        // weight of each job: the bits of a float (FP8), an int (INT8)
    int reduce[3];        // reduce the accumulator modulo m before weighting (0: the exact FP32 range allows skipping it)
    int njobs;            // 2 (square), 3, 1 (native INT8 residues) or 2 (non-square, merged accumulators)
    int kind;             // 0 square, 1 non-square separate, 2 native, 3 non-square merged, 4 / 5 non-square two-plane (SLIM)
    int planeA0, planeB0; // first stored plane of this modulus in A's and in B's plane arrays
    // Split-K inside the kernel: the K range of a job is cut into segments of whole chunks, each with
    // an accumulator of its own that is reduced before the next is added, so that every accumulator
    // stays exact.  nseg / seg_len: job 0 of the merged schedule (depth 4097 or 15420);
    // nseg_all / seg_len_all: every other job (depth 32768 in FP32; 2^31 / term size in INT32).
    int nseg, seg_len;
    int nseg_all, seg_len_all;
    // private residue array
    int store_form;       // kStoredByte, kStoredTen or kStoredPair
    int store_start;      // the byte of a patch where this modulus' residues begin
    float centre;         // (m + 1) / 2 (FP32 epilogue)
    // integer epilogue of the INT8 routes (INT32 accumulators):
    uint32_t mi;          // the modulus
    uint32_t magic;       // floor(2^32 / m)
    uint32_t bias;        // a multiple of m just above 2^31: makes a signed combination non-negative
    // native INT8 residues, one accumulator of at most 2^30 in magnitude (k <= 65536): exact division
    uint32_t magic39;     // ceil(2^39 / m): floor(u / m) = (u * magic39) >> 39 exactly for u < 2^31 + 256, m in (128, 256]
    uint32_t bias30;      // the multiple of m just above 2^30
};
// The parameters travel with every launch, and calls of up to about 128^3 follow one another as fast as launches do: 64^3 13.8 us a call with 112 bytes, 13.4
// with 96.  The order counts too: with the private array's words last the same epilogue takes six registers more, and 8192 x 8192 x 128 464 us instead of 434.
static_assert(sizeof(ModInfo) <= 96, "parameters of a launch");

struct GemmParams {
    int64_t m, n, k;
    int tiles_m, tiles_n, nk;       // tiles of 256 rows / 128 columns of C; nk = K chunks of BLOCK_K
    int vec_store;                  // R rows 16-byte aligned: use vector stores
    int kc_x, plane_z, kc_z;        // TMA coordinates of chunk kc of a plane: x = kc * kc_x, z = plane * plane_z + kc * kc_z
    int pair_squares;               // squares: both jobs in one K-loop
    int stall_producer;             // test hook: the producer issues no copy, so every wait runs out
    int r;
    int patch_bytes;                // private residue array: bytes of a 32 x 64 patch
    int64_t total_items;
    void *R;                        // residues: uint16 (RB = 2) or uint8 (RB = 1, byte moduli)
    int64_t ldr, mod_stride;
    unsigned int *rowmax, *colmax;  // bound product only: one word per row / column, word stride 2
    unsigned int *status;
    ModInfo mod[kMaxR];
};

// ---------------------------------------------------------------- PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
                 : "memory");
}

// cluster-scope acquire: the barriers of the CTA-pair variant are also signalled by the peer CTA
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ uint32_t cluster_ctarank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

// shared::cluster address of the same shared-memory location in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t map_to_cta(uint32_t addr, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}

// Arrivals that hand a drained accumulator back to the MMA issuer.  The TMEM reads they follow have
// already completed (tcgen05.wait::ld) and no memory written by this thread is read by the waiter,
// so the arrive carries no release: a release would first wait for the residue stores in flight.
__device__ __forceinline__ void mbar_arrive_relaxed(uint32_t bar)
{
    asm volatile("mbarrier.arrive.relaxed.cta.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster_relaxed(uint32_t cluster_addr)
{
    asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}

// one lane of the (converged) warp
__device__ __forceinline__ bool elect_one()
{
    uint32_t one;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xFFFFFFFF;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(one));
    return one != 0;
}

// all threads of both CTAs of the pair (no time limit: every thread reaches it on every path)
__device__ __forceinline__ void cluster_sync_all()
{
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ unsigned long long global_timer_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

constexpr unsigned long long kWaitLimitNs = 2000000000ull;   // 2 s per wait

// Bounded wait.  Returns false when the wait ran out or another role already gave up.
// The timer is read only after a long run of failed polls: the common path never touches it.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag,
                                          unsigned int *status)
{
#pragma unroll 1
    for (int it = 0; it < 4096; ++it)
        if (mbar_try_wait(bar, parity)) return true;
    unsigned long long start = global_timer_ns();
    for (;;) {
#pragma unroll 1
        for (int it = 0; it < 256; ++it)
            if (mbar_try_wait(bar, parity)) return true;
        if (*abort_flag) return false;
        if (global_timer_ns() - start > kWaitLimitNs) {
            *abort_flag = 1;
            atomicOr(status, 1u << OZ_ERR_TIMEOUT);
            return false;
        }
    }
}

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap *map, uint32_t bar,
                                            int c0, int c1, int c2)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes "
        "[%0], [%1, {%3, %4, %5}], [%2];"
        ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2)
        : "memory");
}

__device__ __forceinline__ void prefetch_map(const CUtensorMap *map)
{
    asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory");
}

// CTA-pair copy: same as tma_load_3d, but the mbarrier may live in the peer CTA (cluster address)
__device__ __forceinline__ void tma_load_3d_pair(uint32_t dst, const CUtensorMap *map, uint32_t bar_cluster,
                                                 int c0, int c1, int c2)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes "
        "[%0], [%1, {%3, %4, %5}], [%2];"
        ::"r"(dst), "l"(map), "r"(bar_cluster), "r"(c0), "r"(c1), "r"(c2)
        : "memory");
}

// In the CTA-pair variant the same warp of BOTH CTAs executes the allocation / release.
template <int CG>
__device__ __forceinline__ void tmem_alloc(uint32_t dst_smem, uint32_t cols)
{
    if (CG == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    } else {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
}

template <int CG>
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t cols)
{
    if (CG == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
    else
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

template <int SUB, int CG>
__device__ __forceinline__ void umma(uint32_t d_tmem, uint64_t da, uint64_t db, uint32_t idesc,
                                     uint32_t accumulate)
{
#define OZ_UMMA(GROUP, KIND)                                                                      \
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"                              \
                 "tcgen05.mma.cta_group::" GROUP ".kind::" KIND " [%0], %1, %2, %3, p;\n\t}"      \
                 ::"r"(d_tmem), "l"(da), "l"(db), "r"(idesc), "r"(accumulate) : "memory")
    if (SUB == 0 && CG == 1) OZ_UMMA("1", "f8f6f4");
    if (SUB == 0 && CG == 2) OZ_UMMA("2", "f8f6f4");
    if (SUB == 1 && CG == 1) OZ_UMMA("1", "i8");
    if (SUB == 1 && CG == 2) OZ_UMMA("2", "i8");
#undef OZ_UMMA
}

// the same for one CTA, always accumulating, into TMEM lanes 64 to 127 only
template <int SUB>
__device__ __forceinline__ void umma_upper(uint32_t d_tmem, uint64_t da, uint64_t db, uint32_t idesc)
{
#define OZ_UMMA(KIND)                                                                             \
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, 1, 0;\n\t"                               \
                 "tcgen05.mma.cta_group::1.kind::" KIND " [%0], %1, %2, %3, {%4, %4, %5, %5}, p;\n\t}" \
                 ::"r"(d_tmem), "l"(da), "l"(db), "r"(idesc), "r"(0xFFFFFFFFu), "r"(0u) : "memory")
    if (SUB == 0) OZ_UMMA("f8f6f4");
    else OZ_UMMA("i8");
#undef OZ_UMMA
}

// mbarrier arrives once every MMA issued so far by this thread has completed
// (CTA pair: the arrive is delivered to the barrier at this offset in BOTH CTAs)
template <int CG>
__device__ __forceinline__ void umma_commit(uint32_t bar)
{
    if (CG == 1) {
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
    } else {
        const uint16_t both = 3;
        asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                     ::"r"(bar), "h"(both) : "memory");
    }
}

template <int N>
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&v)[N])
{
    static_assert(N == 32, "32 columns");
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
          "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]),
          "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]),
          "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]),
          "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// 16 columns of the warp's 32 lanes, with the wait
template <int N>
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&v)[N])
{
    static_assert(N == 16, "16 columns");
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
          "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]),
          "=r"(v[14]), "=r"(v[15])
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// same load without the wait, into v[OFF .. OFF+31]
template <int OFF>
__device__ __forceinline__ void tmem_ld32_issue(uint32_t taddr, uint32_t (&v)[64])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(v[OFF + 0]), "=r"(v[OFF + 1]), "=r"(v[OFF + 2]), "=r"(v[OFF + 3]), "=r"(v[OFF + 4]),
          "=r"(v[OFF + 5]), "=r"(v[OFF + 6]), "=r"(v[OFF + 7]), "=r"(v[OFF + 8]), "=r"(v[OFF + 9]),
          "=r"(v[OFF + 10]), "=r"(v[OFF + 11]), "=r"(v[OFF + 12]), "=r"(v[OFF + 13]), "=r"(v[OFF + 14]),
          "=r"(v[OFF + 15]), "=r"(v[OFF + 16]), "=r"(v[OFF + 17]), "=r"(v[OFF + 18]), "=r"(v[OFF + 19]),
          "=r"(v[OFF + 20]), "=r"(v[OFF + 21]), "=r"(v[OFF + 22]), "=r"(v[OFF + 23]), "=r"(v[OFF + 24]),
          "=r"(v[OFF + 25]), "=r"(v[OFF + 26]), "=r"(v[OFF + 27]), "=r"(v[OFF + 28]), "=r"(v[OFF + 29]),
          "=r"(v[OFF + 30]), "=r"(v[OFF + 31])
        : "r"(taddr)
        : "memory");
}

// shared-memory matrix descriptor: K-major operand, 128-byte swizzle, 8-row groups 1024 B apart
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr)
{
    uint64_t d = 0;
    d |= static_cast<uint64_t>((addr >> 4) & 0x3FFFu);   // start address / 16
    d |= static_cast<uint64_t>(1) << 16;                 // leading byte offset (unused here) / 16
    d |= static_cast<uint64_t>(1024 >> 4) << 32;         // stride byte offset / 16
    d |= static_cast<uint64_t>(1) << 46;                 // descriptor version of sm_100
    d |= static_cast<uint64_t>(2) << 61;                 // 128-byte swizzle
    return d;
}

// instruction descriptor: D format, A/B formats, K-major both, N/8 at bit 17, M/16 at bit 24
template <int SUB, int CG, int BN = BLOCK_N>
__host__ __device__ constexpr uint32_t instr_desc()
{
    uint32_t cfmt = SUB == 0 ? 1u /*f32*/ : 2u /*s32*/;
    uint32_t abfmt = SUB == 0 ? 0u /*e4m3*/ : 1u /*s8*/;
    return (cfmt << 4) | (abfmt << 7) | (abfmt << 10) | (static_cast<uint32_t>(BN >> 3) << 17) |
           (static_cast<uint32_t>((BLOCK_M * CG) >> 4) << 24);
}

constexpr uint32_t kNegateB = 1u << 14;      // instruction descriptor: the second operand (planes of A) enters negated

// work item -> (modulus, tile_m, tile_n): modulus-major so that one modulus' planes stay in L2;
// inside a modulus, bands of 16 tile rows are swept column by column.
struct Item { int mod, tm, tn; };

__device__ __forceinline__ Item decode_item(int64_t item64, const GemmParams &p)
{
    // the host refuses launches with 2^31 or more items: 32-bit divisions are enough
    constexpr uint32_t BAND = 16;
    const uint32_t item = static_cast<uint32_t>(item64);
    const uint32_t tiles_m = static_cast<uint32_t>(p.tiles_m), tiles_n = static_cast<uint32_t>(p.tiles_n);
    const uint32_t per_mod = tiles_m * tiles_n;
    Item it;
    const uint32_t mod = item / per_mod;
    const uint32_t t = item - mod * per_mod;
    const uint32_t band_size = BAND * tiles_n;
    const uint32_t band = t / band_size;
    const uint32_t in_band = t - band * band_size;
    const uint32_t rows = tiles_m - band * BAND < BAND ? tiles_m - band * BAND : BAND;
    const uint32_t tn = in_band / rows;
    it.mod = static_cast<int>(mod);
    it.tn = static_cast<int>(tn);
    it.tm = static_cast<int>(band * BAND + (in_band - tn * rows));
    return it;
}

// plane pair (A plane, B plane) of K-loop `pair` of job `job`
__device__ __forceinline__ void job_planes(const ModInfo &mi, int job, int pair, int *pa, int *pb)
{
    int oa, ob;
    if (mi.kind == 1) {
        // non-square, stored order d0, d1, dS; jobs d0 e0, dS eS, d1 e1
        oa = ob = job == 0 ? 0 : (job == 1 ? 2 : 1);
    } else if (mi.kind == 3) {
        // non-square merged (A stores d0, -16 d1, dS): job 0 = [d0 | -16 d1] . [e0 | e1] (two K-loops),
        // job 1 = dS eS
        oa = ob = job == 0 ? pair : 2;
    } else if (mi.kind == 0 && job == 1) {
        // square: job 1 = [d1 | d0] . [e0 | e1]
        oa = pair == 0 ? 1 : 0;
        ob = pair == 0 ? 0 : 1;
    } else {
        oa = ob = 0;            // square job 0, native
    }
    *pa = mi.planeA0 + oa;
    *pb = mi.planeB0 + ob;
}

__device__ __forceinline__ int job_pairs(const ModInfo &mi, int job)
{
    return ((mi.kind == 0 && job == 1) || (mi.kind == 3 && job == 0)) ? 2 : 1;
}

// accumulators (K segments) of job `job`
__device__ __forceinline__ int job_segments(const ModInfo &mi, int job)
{
    return (mi.kind == 3 && job == 0) ? mi.nseg : mi.nseg_all;
}

// chunk range [kc0, kc1) of segment `seg`
__device__ __forceinline__ void segment_range(const ModInfo &mi, int job, int seg, int nk, int *kc0, int *kc1)
{
    const int len = (mi.kind == 3 && job == 0) ? mi.seg_len : mi.seg_len_all;
    *kc0 = seg * len;
    *kc1 = min(nk, *kc0 + len);
}

// Two-plane schedule: A's plane h = 0, 1 of a modulus and the planes of B that it is multiplied with, one for each
// accumulator (first: -1 where the plane does not meet the first accumulator):
//   square (kind 0):  d0 with e0 | e1,  d1 with - | e0:              d e = acc0 + s acc1
//   kind 4:           d0 with e0 | e1,  d1 with f0 | f1:             d e = d0 e + d1 f,  f = 16 e mod m
//   kind 5:           d0 with e0 | e1,  -16 d1 with -e0 | -e1:       planes of the merged layouts (kept operands)
// with e = e0 + 16 e1, f = f0 + 16 f1:  d e = acc0 + 16 acc1 (mod m) for the non-squares.
__device__ __forceinline__ void slim_stage(const ModInfo &mi, int h, int *first, int *second)
{
    if (mi.kind == 0) {
        *first = h ? -1 : mi.planeB0;
        *second = h ? mi.planeB0 : mi.planeB0 + 1;
    } else {
        *first = mi.planeB0 + (mi.kind == 4 ? 2 * h : 0);
        *second = *first + 1;
    }
}

// acc - m * rint(acc / m) for a pair of integer-valued floats below 2^24 (exact): rint through the
// 1.5 * 2^23 constant, then one fused multiply-add
__device__ __forceinline__ float2 mod_balanced2(float2 acc, float2 inv_m2, float2 neg_m2)
{
    const float2 big = make_float2(12582912.0f, 12582912.0f), neg_big = make_float2(-12582912.0f, -12582912.0f);
    const float2 quot = __fadd2_rn(__ffma2_rn(acc, inv_m2, big), neg_big);
    return __ffma2_rn(quot, neg_m2, acc);
}

// RB: bytes of one stored residue (2: uint16, 1: uint8 for the all-byte modulus set)
// DIRECT: native INT8 residues -- one accumulator per modulus, loaded straight into the registers
//         that otherwise hold the running combination of several accumulators
// TILED: the residue array is the private, tile-ordered one of the whole-method calls (see
//         ResidueTiling): the 32 columns x 64 rows that an epilogue warp owns form one
//         contiguous patch, [16-byte chunk][lane], so that every store instruction of a warp writes
//         512 consecutive bytes straight from registers -- no transposition through shared memory,
//         which the tensor pipe and the TMA writes need for themselves.  The reconstruction reads
//         the same order.  Without it the public layout R[mod][j][ldr] is written.
//         Sets S and E store 8, 10 or 16 bits a residue (stored_form()): 1.2 instead of 0.5 byte permutations a value, but five
//         16-byte stores a thread and modulus instead of eight.  The FP32 epilogue starts its combination at -centre and adds the
//         centre to the balanced result, which leaves a representative in [0, m + 1] without a comparison.
// BOUND: not a residue product but the magnitude-bound product of the accurate mode (Sec. 2 "The FP8
//         variant", the "+1" pass): one plane per operand, one accumulator per tile, and instead of
//         residues the epilogue reduces the row and column maxima of the tile into p.rowmax / p.colmax.
// BN:      rows of C per tile: 256, or 64 for products with so few tiles that most SMs would be idle (narrow_tiles())
// SLIM:    two-plane schedule of a product with one tile of columns (n <= 128), which reads A's planes from memory once
//         and does little arithmetic with them: d = d0 + 16 d1 of a non-square modulus meets all of e (see kind 4, 5 in
//         slim_stage()), so that dS is never read.  Both accumulators of a modulus fill in one K-loop, per K segment.
template <int SUB, int CG, int RB, bool DIRECT, bool TILED, bool BOUND = false, int SLIM = 0, int BN = BLOCK_N>
__global__ void __launch_bounds__(NUM_THREADS, 1)
residue_gemm_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB,
                    const __grid_constant__ GemmParams p)
{
    static_assert(SLIM == 0 || (CG == 1 && !DIRECT && TILED && !BOUND), "two-plane schedule: whole-method digit products");
    static_assert(BN == BLOCK_N || TILED, "narrow tiles: whole-method products");
    constexpr bool PACKED = TILED && RB == 2 && !BOUND;  // sets S and E in the private array
    constexpr bool BIASED = TILED && SUB == 1 && !DIRECT;        // the combination starts at the bias that makes it non-negative
    using Slim = SlimTile<SLIM ? SLIM : 128, BN>;
    constexpr int STAGES = SLIM ? Slim::STAGES : Tile<CG, BN>::STAGES;
    constexpr int STAGE_BYTES = SLIM ? Slim::STAGE_BYTES : Tile<CG, BN>::STAGE_BYTES;
    constexpr int COLS_PER_WARP = BN / 4;                // four warps share a TMEM lane quarter
    // Both accumulators of a modulus in one slot, one above the other: half the MMAs, which bound a block whose SM is not waiting for
    // memory (a stage of 48 KiB takes 512 cycles instead of 1024), and the other slot free for the next product.  GEMM in us, two MMAs -> one:
    // 10240 x 64 x 10240 482 -> 416 (the last of its 3.24 rounds over the SMs 98 -> 61), 9472 rows (3 rounds) 384 -> 355; calls on kept
    // operands: set E 1104 x 18 x 2754 47.0 -> 36.7, A 1402 x 26 x 7026 125 -> 92.  For it half of the epilogue hands its sums to the other half.
    constexpr bool STACKED = SLIM == 64;
    constexpr int NUM_HANDS = 8;                         // pairs of epilogue warps that hand over the second accumulator
    static_assert(16 * STAGES + 48 + 16 * NUM_HANDS <= 384, "barriers");
    // CTA pair: rank 0 leads (issues the MMAs, owns the `full` and `tmem-empty` barriers that both
    // CTAs signal); work items are dealt to pairs, so both CTAs walk the same item sequence.
    const uint32_t rank = CG == 2 ? cluster_ctarank() : 0u;
    const int64_t first_item = CG == 2 ? (blockIdx.x >> 1) : blockIdx.x;
    const int64_t item_step = CG == 2 ? (gridDim.x >> 1) : gridDim.x;
    extern __shared__ unsigned char smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t tiles = (raw + 1023u) & ~1023u;                     // 1024-byte aligned ring
    const uint32_t bars = tiles + RING_BYTES + EPI_WARPS * XPOSE_BYTES;
    const uint32_t full_bar = bars;                                   // STAGES x 8 bytes
    const uint32_t empty_bar = bars + 8 * STAGES;
    const uint32_t tfull_bar = bars + 16 * STAGES;                    // 2 x 8
    const uint32_t tempty_bar = tfull_bar + 16;                       // 2 x 8
    const uint32_t tmem_slot = tempty_bar + 16;                       // 4 bytes: TMEM base address
    const uint32_t hand_bar = tmem_slot + 16;                         // NUM_HANDS x (written, taken)
    unsigned char *xpose_base = smem_raw + (tiles - raw) + RING_BYTES;
    unsigned char *gen = xpose_base + EPI_WARPS * XPOSE_BYTES;
    volatile uint32_t *tmem_base_ptr = reinterpret_cast<volatile uint32_t *>(gen + 16 * STAGES + 32);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(gen + 16 * STAGES + 40);

    // Broadcast, the warp number and the TMEM base are the same in a warp by construction and need no register of a thread:
    // the epilogue's 64 running values then fit its 96 registers without spills in any of the variants.
    const int warp = __shfl_sync(0xFFFFFFFFu, static_cast<int>(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;

    dependency_release();
    if (threadIdx.x == 0) {
        prefetch_map(&mapA);
        prefetch_map(&mapB);
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(full_bar + 8 * s, 1);
            mbar_init(empty_bar + 8 * s, 1);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(tfull_bar + 8 * s, 1);
            mbar_init(tempty_bar + 8 * s, EPI_WARPS * CG);   // pair: the peer's epilogue warps arrive too
        }
        if constexpr (STACKED)
            for (int s = 0; s < 2 * NUM_HANDS; ++s) mbar_init(hand_bar + 8 * s, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) tmem_alloc<CG>(tmem_slot, TMEM_COLS);
    tc_fence_before();
    __syncthreads();
    if (CG == 2) cluster_sync_all();      // the peer's barriers exist before anything signals them
    tc_fence_after();
    dependency_wait();                    // the planes are there, and the previous readers of the residues are done
    const uint32_t tmem_base = __shfl_sync(0xFFFFFFFFu, *tmem_base_ptr, 0);

    if (warp < FIRST_EPI_WARP) {
        // The whole warp walks the loops of its role and one elected lane issues: with nothing that depends on the thread, what a
        // copy or an MMA takes is computed in uniform registers, where these instructions want it.  A single thread that walks them
        // moves every descriptor over instead and falls behind the tensor cores (us, single threads -> issuer -> both):
        // 8192 x 8192 x 1024 set S FP8 1900 -> 1781 -> 1627, 3000 x 3000 x 500 150 -> 134 -> 123, 6144 x 6144 x 3072 native INT8
        // 1086 -> 1074 -> 994, 10007 x 9973 x 5003 at the power cap 14286 -> 13977 -> 13664.
        const bool leader = elect_one();
        auto wait = [&](uint32_t bar, uint32_t parity) { return __all_sync(0xFFFFFFFFu, mbar_wait(bar, parity, abort_flag, p.status)) != 0; };
        if (warp == 0) {
            // -------------------------------------------------------- TMA producer
            int stage = 0;
            uint32_t phase = 0;
            bool ok = true;
            for (int64_t item = first_item; ok && !p.stall_producer && item < p.total_items; item += item_step) {
                Item it = decode_item(item, p);
                const ModInfo &mi = p.mod[it.mod];
                // one stage: 128 bytes of K of plane pa of A and pb of B
                auto load = [&](int pa, int pb, int kc) {
                    if (!wait(empty_bar + 8 * stage, phase ^ 1u)) return false;
                    uint32_t fb = full_bar + 8 * stage;
                    uint32_t sa = tiles + stage * STAGE_BYTES;
                    if (leader && CG == 1) {
                        mbar_expect_tx(fb, STAGE_BYTES);
                        tma_load_3d(sa, &mapB, fb, kc * p.kc_x, it.tn * BLOCK_M, pb * p.plane_z + kc * p.kc_z);
                        tma_load_3d(sa + A_BYTES, &mapA, fb, kc * p.kc_x, it.tm * BN, pa * p.plane_z + kc * p.kc_z);
                    } else if (leader) {
                        // both CTAs' copies complete on the leader's barrier
                        if (rank == 0) mbar_expect_tx(fb, 2 * STAGE_BYTES);
                        const uint32_t fb_leader = map_to_cta(fb, 0);
                        tma_load_3d_pair(sa, &mapB, fb_leader, kc * p.kc_x,
                                         it.tn * Tile<CG>::TILE_J + static_cast<int>(rank) * BLOCK_M, pb * p.plane_z + kc * p.kc_z);
                        tma_load_3d_pair(sa + A_BYTES, &mapA, fb_leader, kc * p.kc_x,
                                         it.tm * BN + static_cast<int>(rank) * Tile<CG, BN>::B_LINES, pa * p.plane_z + kc * p.kc_z);
                    }
                    if (++stage == STAGES) { stage = 0; phase ^= 1u; }
                    return true;
                };
                if constexpr (SLIM != 0) {
                    for (int kc = 0; ok && kc < p.nk; ++kc)
                        for (int h = 0; ok && h < 2; ++h) {
                            ok = wait(empty_bar + 8 * stage, phase ^ 1u);
                            if (!ok) break;
                            const uint32_t fb = full_bar + 8 * stage, sa = tiles + stage * STAGE_BYTES;
                            int first, second;
                            slim_stage(mi, h, &first, &second);
                            const int x = kc * p.kc_x, z = kc * p.kc_z;
                            if (leader) {
                                mbar_expect_tx(fb, first >= 0 ? STAGE_BYTES : STAGE_BYTES - Slim::B_BYTES);
                                tma_load_3d(sa + 2 * Slim::B_BYTES, &mapA, fb, x, it.tm * BN, (mi.planeA0 + h) * p.plane_z + z);
                                if (first >= 0) tma_load_3d(sa, &mapB, fb, x, it.tn * BLOCK_M, first * p.plane_z + z);
                                tma_load_3d(sa + Slim::B_BYTES, &mapB, fb, x, it.tn * BLOCK_M, second * p.plane_z + z);
                            }
                            if (++stage == STAGES) { stage = 0; phase ^= 1u; }
                        }
                    continue;
                }
                if (!DIRECT && p.pair_squares && mi.kind == 0) {
                    // the two planes of a chunk in two stages, side by side
                    for (int kc = 0; ok && kc < p.nk; ++kc)
                        ok = load(mi.planeA0, mi.planeB0, kc) && load(mi.planeA0 + 1, mi.planeB0 + 1, kc);
                    continue;
                }
                for (int job = 0; ok && job < mi.njobs; ++job)
                for (int seg = 0, nseg = job_segments(mi, job); ok && seg < nseg; ++seg) {
                    int npairs = job_pairs(mi, job), kc0, kc1;
                    segment_range(mi, job, seg, p.nk, &kc0, &kc1);
                    for (int pair = 0; ok && pair < npairs; ++pair) {
                        int pa, pb;
                        job_planes(mi, job, pair, &pa, &pb);
                        for (int kc = kc0; ok && kc < kc1; ++kc) ok = load(pa, pb, kc);
                    }
                }
            }
            if (!ok) {
                // give copies already in flight a bounded time to land before the CTA exits
                unsigned long long t0 = global_timer_ns();
                while (global_timer_ns() - t0 < 2000000ull) { }
            }
        } else if (warp == 1 && rank == 0) {
            // -------------------------------------------------------- MMA issuer (pair: leader CTA only)
            constexpr uint32_t idesc = instr_desc<SUB, CG, BN>();
            int stage = 0;
            uint32_t phase = 0;
            int slot = 0;
            uint32_t slot_phase = 0;   // bit s = phase of slot s
            bool ok = true;
            for (int64_t item = first_item; ok && item < p.total_items; item += item_step) {
                Item it = decode_item(item, p);
                const ModInfo &mi = p.mod[it.mod];
                if constexpr (SLIM != 0) {
                    // kind 5: A's second plane is -16 d1, which the tensor core negates
                    const uint32_t idesc1 = mi.kind == 5 ? idesc | kNegateB : idesc;
                    for (int seg = 0; ok && seg < mi.nseg_all; ++seg) {
                        if constexpr (STACKED) {
                            ok = wait(tempty_bar + 8 * slot, ((slot_phase >> slot) & 1u) ^ 1u);
                        } else {
                            for (int h = 0; ok && h < 2; ++h)
                                ok = wait(tempty_bar + 8 * h, ((slot_phase >> h) & 1u) ^ 1u);
                        }
                        if (!ok) break;
                        tc_fence_after();
                        const uint32_t d_tmem = tmem_base + static_cast<uint32_t>(slot * BLOCK_N);
                        const int kc0 = seg * mi.seg_len_all, kc1 = min(p.nk, kc0 + mi.seg_len_all);
                        for (int st = 0; st < 2 * (kc1 - kc0); ++st) {
                            const int h = st & 1;
                            ok = wait(full_bar + 8 * stage, phase);
                            if (!ok) break;
                            tc_fence_after();
                            const uint32_t sa = tiles + stage * STAGE_BYTES;
                            const uint64_t e0 = smem_desc(sa), e1 = smem_desc(sa + Slim::B_BYTES), a = smem_desc(sa + 2 * Slim::B_BYTES);
                            if (leader) {
#pragma unroll
                                for (int ks = 0; ks < BLOCK_K / UMMA_K; ++ks) {
                                    const uint64_t o = static_cast<uint64_t>(ks * (UMMA_K >> 4));
                                    const uint32_t accumulate = st > 0 || ks > 0 ? 1u : 0u, id = h ? idesc1 : idesc;
                                    if constexpr (STACKED) {
                                        // d1 of a square meets e0 only, in the second accumulator
                                        if (mi.kind != 0 || h == 0) umma<SUB, CG>(d_tmem, e0 + o, a + o, id, accumulate);
                                        else umma_upper<SUB>(d_tmem, e0 + o, a + o, idesc);
                                    } else {
                                        if (mi.kind != 0 || h == 0) umma<SUB, CG>(tmem_base, e0 + o, a + o, id, accumulate);
                                        umma<SUB, CG>(tmem_base + BLOCK_N, e1 + o, a + o, id, accumulate);
                                    }
                                }
                                umma_commit<CG>(empty_bar + 8 * stage);
                            }
                            if (++stage == STAGES) { stage = 0; phase ^= 1u; }
                        }
                        if (!ok) break;
                        if (leader) {
                            umma_commit<CG>(tfull_bar + 8 * slot);
                            if constexpr (!STACKED) umma_commit<CG>(tfull_bar + 8 * (slot ^ 1));
                        }
                        if constexpr (STACKED) { slot_phase ^= 1u << slot; slot ^= 1; }
                        else slot_phase ^= 3u;
                    }
                    continue;
                }
                if (!DIRECT && p.pair_squares && mi.kind == 0) {
                    // d0 e0 into one slot, d1 e0 + d0 e1 into the other, from the four tiles of a chunk: first all that goes into
                    // the first slot, so that it is complete while the last chunk's other products run, and the next product's
                    // can begin in it while the epilogue still empties the second.  That takes longer than one chunk's 4 MMAs, so
                    // a pair starts with those of two chunks.  (Two at a time throughout leave two of the six stages to prefetch
                    // into.)  Both slots waited for and complete together -> in turn: 8192 x 8192 x 512 set E INT8 1003 -> 909 us,
                    // 8192 x 8192 x 1024 set S FP8 1707 -> 1621, 16384 x 16384 x 1024 7510 -> 7100, 4096 x 4096 x 4096
                    // 1596 -> 1578; in turn -> two chunks at the start (two at a time): 955 -> 923 (915), 1721 -> 1691 (1732),
                    // 7182 -> 7036 (7237), 1689 -> 1678 (1691).
                    const uint32_t d0 = tmem_base + static_cast<uint32_t>(slot * BLOCK_N);
                    const uint32_t d1 = tmem_base + static_cast<uint32_t>((slot ^ 1) * BLOCK_N);
                    constexpr int GROUP = CG == 2 ? 2 : 1;           // chunks
                    for (int kc = 0, count; ok && kc < p.nk; kc += count) {
                        const int start = stage;
                        count = kc == 0 ? min(GROUP, p.nk) : 1;
                        const uint32_t start_phase = phase;
                        if (kc == 0) ok = wait(tempty_bar + 8 * slot, ((slot_phase >> slot) & 1u) ^ 1u);
                        for (int c = 0; ok && c < count; ++c) {
                            ok = wait(full_bar + 8 * stage, phase);
                            if (!ok) break;
                            tc_fence_after();
                            const uint32_t t0 = tiles + stage * STAGE_BYTES;
                            const uint64_t e0 = smem_desc(t0), a0 = smem_desc(t0 + A_BYTES);
                            if (leader) {
#pragma unroll
                                for (int ks = 0; ks < BLOCK_K / UMMA_K; ++ks) {
                                    const uint64_t o = static_cast<uint64_t>(ks * (UMMA_K >> 4));
                                    umma<SUB, CG>(d0, e0 + o, a0 + o, idesc, kc > 0 || c > 0 || ks > 0 ? 1u : 0u);
                                }
                            }
                            for (int h = 0; h < 2; ++h)
                                if (++stage == STAGES) { stage = 0; phase ^= 1u; }
                        }
                        if (!ok) break;
                        if (leader && kc + count >= p.nk) umma_commit<CG>(tfull_bar + 8 * slot);
                        if (kc == 0) ok = wait(tempty_bar + 8 * (slot ^ 1), ((slot_phase >> (slot ^ 1)) & 1u) ^ 1u);
                        stage = start;
                        phase = start_phase;
                        for (int c = 0; ok && c < count; ++c) {
                            const int s0 = stage;
                            if (++stage == STAGES) { stage = 0; phase ^= 1u; }
                            ok = wait(full_bar + 8 * stage, phase);
                            if (!ok) break;
                            tc_fence_after();
                            const uint32_t t0 = tiles + s0 * STAGE_BYTES, t1 = tiles + stage * STAGE_BYTES;
                            const uint64_t e0 = smem_desc(t0), a0 = smem_desc(t0 + A_BYTES), e1 = smem_desc(t1), a1 = smem_desc(t1 + A_BYTES);
                            if (leader) {
#pragma unroll
                                for (int ks = 0; ks < BLOCK_K / UMMA_K; ++ks) {
                                    const uint64_t o = static_cast<uint64_t>(ks * (UMMA_K >> 4));
                                    umma<SUB, CG>(d1, e0 + o, a1 + o, idesc, kc > 0 || c > 0 || ks > 0 ? 1u : 0u);
                                    umma<SUB, CG>(d1, e1 + o, a0 + o, idesc, 1u);
                                }
                                umma_commit<CG>(empty_bar + 8 * s0);
                                umma_commit<CG>(empty_bar + 8 * stage);
                            }
                            if (++stage == STAGES) { stage = 0; phase ^= 1u; }
                        }
                    }
                    if (!ok) break;
                    if (leader) umma_commit<CG>(tfull_bar + 8 * (slot ^ 1));
                    slot_phase ^= 3u;
                    continue;
                }
                for (int job = 0; ok && job < mi.njobs; ++job)
                for (int seg = 0, nseg = job_segments(mi, job); ok && seg < nseg; ++seg) {
                    ok = wait(tempty_bar + 8 * slot, ((slot_phase >> slot) & 1u) ^ 1u);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t d_tmem = tmem_base + static_cast<uint32_t>(slot * BLOCK_N);
                    int kc0, kc1;
                    segment_range(mi, job, seg, p.nk, &kc0, &kc1);
                    int steps = job_pairs(mi, job) * (kc1 - kc0);
                    for (int st = 0; st < steps; ++st) {
                        ok = wait(full_bar + 8 * stage, phase);
                        if (!ok) break;
                        tc_fence_after();
                        uint32_t sa = tiles + stage * STAGE_BYTES;
                        uint64_t da = smem_desc(sa), db = smem_desc(sa + A_BYTES);
                        if (leader) {
#pragma unroll
                            for (int ks = 0; ks < BLOCK_K / UMMA_K; ++ks)
                                // advancing K inside the 128-byte swizzle atom: +32 bytes = +2 in the address field
                                umma<SUB, CG>(d_tmem, da + static_cast<uint64_t>(ks * (UMMA_K >> 4)),
                                          db + static_cast<uint64_t>(ks * (UMMA_K >> 4)), idesc, st > 0 || ks > 0 ? 1u : 0u);
                            umma_commit<CG>(empty_bar + 8 * stage);     // frees the stage when these MMAs finish
                        }
                        if (++stage == STAGES) { stage = 0; phase ^= 1u; }
                    }
                    if (!ok) break;
                    if (leader) umma_commit<CG>(tfull_bar + 8 * slot);           // accumulator complete
                    slot_phase ^= 1u << slot;
                    slot ^= 1;
                }
            }
            if (!ok) {
                unsigned long long t0 = global_timer_ns();
                while (global_timer_ns() - t0 < 2000000ull) { }
            }
        }
    } else {
        // ------------------------------------------------------------ epilogue
        const int q = warp & 3;                              // TMEM lane quarter this warp may read
        const int part = (warp - FIRST_EPI_WARP) >> 2;       // which 64 of the tile's 256 TMEM columns (any four
                                                             // consecutive warps cover the four lane quarters)
        // STACKED: warps of lanes 64 to 127 drain the second accumulator and hand it to those of lanes 0 to 63
        const bool second = STACKED && q >= 2;
        uint32_t hand_phase = 0;
        int slot = 0;
        uint32_t slot_phase = 0;   // bit s = phase of slot s
        bool ok = true;
        for (int64_t item = first_item; ok && item < p.total_items; item += item_step) {
            Item it = decode_item(item, p);
            const ModInfo &mi = p.mod[it.mod];
            const float mm = mi.m, inv_m = mi.inv_m;
            const float centre_big = mi.centre + 8388608.0f;     // exact: m < 2^11
            const float2 inv_m2 = make_float2(inv_m, inv_m), neg_m2 = make_float2(-mm, -mm);
            const uint32_t im = mi.mi, imagic = mi.magic, ibias = mi.bias;
            // running combination per element: FP32 (FP8 route) or INT32 (INT8 routes), as raw bits
            uint32_t comb[COLS_PER_WARP];
            if constexpr (!DIRECT) {
                const uint32_t start = second ? 0u : SUB == 0 ? (PACKED ? __float_as_uint(-mi.centre) : 0u) : (BIASED ? ibias : 0u);
#pragma unroll
                for (int c = 0; c < COLS_PER_WARP; ++c) comb[c] = start;
            }
            // SLIM: both jobs of a K segment before the next segment.  (The bound is read where it is compared: in a register of its
            // own it costs the public FP8 pair 72 bytes of spills instead of 40.)
            for (int o = 0; ok && o < (SLIM ? mi.nseg_all : mi.njobs); ++o)
            for (int i = 0, inner = STACKED ? 1 : SLIM ? 2 : job_segments(mi, o); ok && i < inner; ++i) {
                const int job = STACKED ? q >> 1 : SLIM ? i : o;
                // every lane polls for itself; the outcome is made warp-uniform before anything that
                // contains a warp barrier depends on it
                ok = __all_sync(0xFFFFFFFFu, mbar_wait(tfull_bar + 8 * slot, (slot_phase >> slot) & 1u, abort_flag, p.status));
                if (!ok) break;
                tc_fence_after();
                const float wj = __uint_as_float(mi.w[job]);
                const bool reduce_first = mi.reduce[job] != 0;
                const uint32_t taddr = tmem_base + (static_cast<uint32_t>(q * 32) << 16) +
                                       static_cast<uint32_t>(slot * BLOCK_N + part * COLS_PER_WARP);
                if constexpr (DIRECT) {
                    // the only accumulator of this modulus lands in the combination registers as it is
                    if constexpr (COLS_PER_WARP == 64) {
                        tmem_ld32_issue<0>(taddr, comb);
                        tmem_ld32_issue<32>(taddr + 32, comb);
                        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    } else {
                        tmem_ld16(taddr, comb);
                    }
                } else
#pragma unroll
                for (int c0 = 0; c0 < COLS_PER_WARP; c0 += DRAIN_W) {
                    uint32_t v[DRAIN_W];
                    if constexpr (DRAIN_W == 32) tmem_ld32(taddr + c0, v);
                    else tmem_ld16(taddr + c0, v);
                    if constexpr (SUB == 0) {
                        // two values per instruction (packed FP32 pairs): half the issue slots
                        const float2 wj2 = make_float2(wj, wj);
                        if (reduce_first) {
#pragma unroll
                            for (int e = 0; e < DRAIN_W; e += 2) {
                                const float2 acc = make_float2(__uint_as_float(v[e]), __uint_as_float(v[e + 1]));
                                const float2 res = mod_balanced2(acc, inv_m2, neg_m2);       // exact, |res| <= ~m/2
                                const float2 cur = make_float2(__uint_as_float(comb[c0 + e]), __uint_as_float(comb[c0 + e + 1]));
                                const float2 nxt = __ffma2_rn(res, wj2, cur);
                                comb[c0 + e] = __float_as_uint(nxt.x);
                                comb[c0 + e + 1] = __float_as_uint(nxt.y);
                            }
                        } else {
                            // the host has checked that w * acc stays below 2^24 for this k
#pragma unroll
                            for (int e = 0; e < DRAIN_W; e += 2) {
                                const float2 acc = make_float2(__uint_as_float(v[e]), __uint_as_float(v[e + 1]));
                                const float2 cur = make_float2(__uint_as_float(comb[c0 + e]), __uint_as_float(comb[c0 + e + 1]));
                                const float2 nxt = __ffma2_rn(acc, wj2, cur);
                                comb[c0 + e] = __float_as_uint(nxt.x);
                                comb[c0 + e + 1] = __float_as_uint(nxt.y);
                            }
                        }
                    } else {
                        // INT32 accumulators: exact integer arithmetic, no conversions
                        // (modulo 2^32: a combination that starts at its bias, above 2^31, is no int.  Written as comb += ..., k = 128 is 1.5 percent slower.)
                        const uint32_t iwj = mi.w[job];
                        if (reduce_first) {
#pragma unroll
                            for (int e = 0; e < DRAIN_W; ++e) {
                                uint32_t u = v[e] + ibias;                       // non-negative, same residue
                                uint32_t r = u - __umulhi(u, imagic) * im;       // in [0, 2m)
                                r = min(r, r - im);
                                comb[c0 + e] = r * iwj + comb[c0 + e];
                            }
                        } else {
                            // the host has checked that the weighted sum stays inside INT32 for this k
#pragma unroll
                            for (int e = 0; e < DRAIN_W; ++e)
                                comb[c0 + e] = v[e] * iwj + comb[c0 + e];
                        }
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    if (CG == 1) mbar_arrive_relaxed(tempty_bar + 8 * slot);
                    else mbar_arrive_cluster_relaxed(map_to_cta(tempty_bar + 8 * slot, 0));   // the leader's barrier
                }
                slot_phase ^= 1u << slot;
                slot ^= 1;
            }
            if (!ok) break;
            // this thread: column j of C, rows i0 .. i0+63 (contiguous in the residue array)
            const int64_t jw = static_cast<int64_t>(it.tn) * Tile<CG>::TILE_J + rank * BLOCK_M + q * 32;   // first column of the warp
            const int64_t j = jw + lane;
            const int64_t i0 = static_cast<int64_t>(it.tm) * BN + part * COLS_PER_WARP;
            if constexpr (STACKED) {
                // through 4 KiB of shared memory a pair of warps, a word of every lane at a time: no bank conflicts
                constexpr int PIECE = COLS_PER_WARP < 32 ? COLS_PER_WARP : 32;
                const int pair = part * 2 + (q & 1);
                if (i0 < p.m && (q & 1) * 32 < p.n) {
                    uint32_t *box = reinterpret_cast<uint32_t *>(xpose_base + pair * (2 * XPOSE_BYTES)) + lane;
                    const uint32_t written = hand_bar + 16 * pair, taken = written + 8;
#pragma unroll
                    for (int c0 = 0; c0 < COLS_PER_WARP; c0 += PIECE) {
                        ok = ok && __all_sync(0xFFFFFFFFu, mbar_wait(second ? taken : written, second ? hand_phase ^ 1u : hand_phase, abort_flag, p.status));
                        if (ok) {
                            if (second) {
#pragma unroll
                                for (int c = 0; c < PIECE; ++c) box[32 * c] = comb[c0 + c];
                            } else {
#pragma unroll
                                for (int c = 0; c < PIECE; ++c) {
                                    if constexpr (SUB == 0) comb[c0 + c] = __float_as_uint(__uint_as_float(comb[c0 + c]) + __uint_as_float(box[32 * c]));
                                    else comb[c0 + c] += box[32 * c];
                                }
                            }
                            __syncwarp();
                            if (lane == 0) mbar_arrive(second ? written : taken);
                        }
                        hand_phase ^= 1u;
                    }
                    if (!ok) break;
                }
            }
            if (i0 >= p.m || jw >= p.n) continue;                                 // warp-uniform
            if constexpr (BOUND) {
                // The accumulators are non-negative integers held exactly in FP32: their bit patterns
                // order like their values, so the maxima are taken on the raw words.
                uint32_t colv = 0u, keep0 = 0u, keep1 = 0u;
#pragma unroll
                for (int c = 0; c < COLS_PER_WARP; ++c) {
                    colv = max(colv, comb[c]);
                    const uint32_t rowv = __reduce_max_sync(0xFFFFFFFFu, comb[c]);   // over the warp's 32 columns
                    if ((c & 31) == lane) { if (c < 32) keep0 = rowv; else keep1 = rowv; }
                }
                if (j < p.n && colv) atomicMax(p.colmax + 2 * j, colv);
                if (i0 + lane < p.m && keep0) atomicMax(p.rowmax + 2 * (i0 + lane), keep0);
                if (i0 + 32 + lane < p.m && keep1) atomicMax(p.rowmax + 2 * (i0 + 32 + lane), keep1);
            }
            if constexpr (!BOUND) {
            // last reduction of one combination value: the stored residue in the low bits of a word
            auto final_bits = [&](uint32_t cv) -> uint32_t {
                if constexpr (SUB == 0) {
                    float t = __uint_as_float(cv);
                    float quot = fmaf(t, inv_m, 12582912.0f) - 12582912.0f;
                    float res = fmaf(-quot, mm, t);                      // |res| <= ~m/2
                    res = res < 0.0f ? res + mm : res;                   // canonical [0, m) (PACKED: final_bits2)
                    return __float_as_uint(res + 8388608.0f);            // integer in the low mantissa bits
                } else if constexpr (DIRECT) {
                    uint32_t u = cv + mi.bias30;                          // in (0, 2^31 + 256)
                    return u - (__umulhi(u, mi.magic39) >> 7) * im;      // exact quotient: canonical [0, m)
                } else {
                    uint32_t u = BIASED ? cv : cv + ibias;
                    uint32_t r = u - __umulhi(u, imagic) * im;           // in [0, 2m)
                    return __viaddmin_u32(r, 0u - im, r);                // canonical [0, m)
                }
            };
            // same for two values at once; the balanced FP32 form is done with packed pairs
            auto final_bits2 = [&](uint32_t c0v, uint32_t c1v, uint32_t &b0, uint32_t &b1) {
                if constexpr (SUB == 0 && PACKED) {
                    const float2 res = mod_balanced2(make_float2(__uint_as_float(c0v), __uint_as_float(c1v)), inv_m2, neg_m2);
                    const float2 out = __fadd2_rn(res, make_float2(centre_big, centre_big));
                    b0 = __float_as_uint(out.x);
                    b1 = __float_as_uint(out.y);
                } else {
                    b0 = final_bits(c0v);
                    b1 = final_bits(c1v);
                }
            };
            // rows a, a + 1, b and b + 1 of the thread's run -> one (RB = 1) or two (RB = 2) words
            auto pack_rows = [&](int a, int b, uint32_t &w0, uint32_t &w1) {
                uint32_t b0, b1, b2, b3;
                final_bits2(comb[a], comb[a + 1], b0, b1);
                final_bits2(comb[b], comb[b + 1], b2, b3);
                if constexpr (RB == 2) {
                    w0 = __byte_perm(b0, b1, 0x5410);
                    w1 = __byte_perm(b2, b3, 0x5410);
                } else {
                    w0 = __byte_perm(__byte_perm(b0, b1, 0x0040), __byte_perm(b2, b3, 0x0040), 0x5410);
                    w1 = 0u;
                }
            };
            constexpr int NCH = COLS_PER_WARP * RB / 16;     // 16-byte chunks of a thread's run of rows
            if constexpr (TILED) {
                // patch (tile, CTA rank, warp), then modulus: the residues of one 32 x 64 patch of the output lie next to one
                // another, which is how the reconstruction reads them
                const int64_t tile = i0 / BLOCK_N;                   // the layout's tiles have 256 rows, its patches 64
                const int patch = (static_cast<int>(i0 >> 6) & 3) * 4 + q, chunk0 = static_cast<int>(i0 & 63) / 16;
                unsigned char *base = static_cast<unsigned char *>(p.R) +
                    (((tile * p.tiles_n + it.tn) * CG + rank) * EPI_WARPS + patch) * static_cast<int64_t>(p.patch_bytes) + mi.store_start + lane * 16;
                if constexpr (PACKED) {
                    if (mi.store_form == kStoredPair) {
#pragma unroll
                        for (int c = 0; c < COLS_PER_WARP / 8; ++c) {
                            uint4 val;
                            pack_rows(8 * c, 8 * c + 2, val.x, val.y);
                            pack_rows(8 * c + 4, 8 * c + 6, val.z, val.w);
                            *reinterpret_cast<uint4 *>(base + (2 * chunk0 + c) * 512) = val;
                        }
                    } else if (mi.store_form == kStoredTen) {
                        uint32_t high[COLS_PER_WARP / 16];           // bits 8 and 9 of sixteen rows
#pragma unroll
                        for (int g = 0; g < COLS_PER_WARP / 16; ++g) {
                            uint32_t lo[4], hi[4];
#pragma unroll
                            for (int h = 0; h < 4; ++h) {
                                uint32_t w0, w1;
                                pack_rows(16 * g + 2 * h, 16 * g + 2 * h + 8, w0, w1);
                                lo[h] = __byte_perm(w0, w1, 0x6420);
                                hi[h] = __byte_perm(w0, w1, 0x7531);
                                if constexpr (SUB == 0) hi[h] &= 0x03030303u;        // 1024 is 0 modulo 1024
                            }
                            *reinterpret_cast<uint4 *>(base + (chunk0 + g) * 512) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
                            high[g] = (hi[0] + 4u * hi[1]) + 16u * (hi[2] + 4u * hi[3]);
                        }
                        if constexpr (COLS_PER_WARP == 64) *reinterpret_cast<uint4 *>(base + 2048) = make_uint4(high[0], high[1], high[2], high[3]);
                        else *reinterpret_cast<uint32_t *>(base + 2048 + 4 * chunk0) = high[0];
                    } else {
#pragma unroll
                        for (int g = 0; g < COLS_PER_WARP / 16; ++g) {
                            uint32_t lo[4];
#pragma unroll
                            for (int h = 0; h < 4; ++h) {
                                uint32_t b0, b1, b8, b9;
                                final_bits2(comb[16 * g + 2 * h], comb[16 * g + 2 * h + 1], b0, b1);
                                final_bits2(comb[16 * g + 2 * h + 8], comb[16 * g + 2 * h + 9], b8, b9);
                                lo[h] = __byte_perm(__byte_perm(b0, b1, 0x0040), __byte_perm(b8, b9, 0x0040), 0x5410);
                            }
                            *reinterpret_cast<uint4 *>(base + (chunk0 + g) * 512) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
                        }
                    }
                } else {
#pragma unroll
                    for (int c = 0; c < COLS_PER_WARP / 16; ++c) {
                        uint4 val;
                        uint32_t unused;
                        pack_rows(16 * c, 16 * c + 8, val.x, unused);
                        pack_rows(16 * c + 2, 16 * c + 10, val.y, unused);
                        pack_rows(16 * c + 4, 16 * c + 12, val.z, unused);
                        pack_rows(16 * c + 6, 16 * c + 14, val.w, unused);
                        *reinterpret_cast<uint4 *>(base + (chunk0 + c) * 512) = val;
                    }
                }
            } else {
            // residues packed 4 / RB to a word in row order
            uint32_t packed[COLS_PER_WARP * RB / 4];
#pragma unroll
            for (int c = 0; c < COLS_PER_WARP; c += 4) {
                if constexpr (RB == 2) pack_rows(c, c + 2, packed[c >> 1], packed[(c >> 1) + 1]);
                else {
                    uint32_t unused;
                    pack_rows(c, c + 2, packed[c >> 2], unused);
                }
            }
            // all are packed before the first is stored: the unpacked ones in between cost 72 bytes of spills.  (Native residues have none that way and up to 56 bytes
            // packed first: in single CTAs 300^3 12.1 us against 10.8, 200 x 300 x 1000 11.9 against 10.1.)
            if constexpr (!DIRECT) {
#pragma unroll
                for (int c = 0; c < COLS_PER_WARP * RB / 4; ++c) asm volatile("" : "+r"(packed[c]));
            }
            unsigned char *rbase = static_cast<unsigned char *>(p.R) + it.mod * p.mod_stride * RB;
            if (p.vec_store && i0 + COLS_PER_WARP <= p.m) {
                // Transpose through a per-warp shared buffer so that one store instruction writes
                // whole lines of the residue array (128 bytes per column for uint16, 64 for uint8)
                // instead of 32 separate 16-byte pieces.  Chunks are XOR-swizzled by the line
                // number: both the writes and the reads are free of bank conflicts.
                unsigned char *xp = xpose_base + (warp - FIRST_EPI_WARP) * XPOSE_BYTES;
                if constexpr (RB == 2) {
                    // 16 lines x 128 bytes per pass; lane -> line lane/8 + 4t, 16-byte chunk lane%8
#pragma unroll
                    for (int rho = 0; rho < 2; ++rho) {
                        if ((lane >> 4) == rho) {
                            const int lr = lane & 15;
#pragma unroll
                            for (int c = 0; c < 8; ++c)
                                *reinterpret_cast<uint4 *>(xp + lr * 128 + ((c ^ (lr & 7)) << 4)) =
                                    make_uint4(packed[4 * c], packed[4 * c + 1], packed[4 * c + 2], packed[4 * c + 3]);
                        }
                        __syncwarp();
#pragma unroll
                        for (int t = 0; t < 4; ++t) {
                            const int lr = (lane >> 3) + 4 * t, c = lane & 7;
                            uint4 val = *reinterpret_cast<const uint4 *>(xp + lr * 128 + ((c ^ (lr & 7)) << 4));
                            const int64_t jg = jw + 16 * rho + lr;
                            if (jg < p.n) *reinterpret_cast<uint4 *>(rbase + (jg * p.ldr + i0 + 8 * c) * 2) = val;
                        }
                        __syncwarp();
                    }
                } else {
                    // 32 lines x 64 bytes in one pass; lane -> line lane/4 + 8t, 16-byte chunk lane%4
#pragma unroll
                    for (int c = 0; c < NCH; ++c)
                        *reinterpret_cast<uint4 *>(xp + lane * 64 + (((c ^ (lane >> 1)) & 3) << 4)) =
                            make_uint4(packed[4 * c], packed[4 * c + 1], packed[4 * c + 2], packed[4 * c + 3]);
                    __syncwarp();
#pragma unroll
                    for (int t = 0; t < 4; ++t) {
                        const int lr = (lane >> 2) + 8 * t, c = lane & 3;
                        uint4 val = *reinterpret_cast<const uint4 *>(xp + lr * 64 + (((c ^ (lr >> 1)) & 3) << 4));
                        const int64_t jg = jw + lr;
                        if (jg < p.n) *reinterpret_cast<uint4 *>(rbase + jg * p.ldr + i0 + 16 * c) = val;
                    }
                    __syncwarp();
                }
            } else if (j < p.n) {
                unsigned char *dst = rbase + (j * p.ldr + i0) * RB;
#pragma unroll
                for (int c = 0; c < COLS_PER_WARP; ++c)
                    if (i0 + c < p.m) {
                        if constexpr (RB == 2)
                            reinterpret_cast<uint16_t *>(dst)[c] = static_cast<uint16_t>((packed[c >> 1] >> (16 * (c & 1))) & 0xFFFFu);
                        else
                            dst[c] = static_cast<unsigned char>((packed[c >> 2] >> (8 * (c & 3))) & 0xFFu);
                    }
            }
            }   // public layout
            }   // residues
        }
    }

    tc_fence_before();
    __syncthreads();
    if (CG == 2) cluster_sync_all();      // neither CTA leaves while the other may still touch it
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc<CG>(tmem_base, TMEM_COLS);
    }
}

#include "oz_gemm_fused.cuh"

// ---------------------------------------------------------------- host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                  const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                  const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_tiled_fn()
{
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void *sym = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &sym, cudaEnableDefault, &qres) == cudaSuccess &&
            qres == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(sym);
    }
    return fn;
}

// 3-D map over planes[plane][line][kbyte] (private layout: planes[plane * chunks + chunk][line][128 bytes]);
// box = 128 bytes x box_lines lines x 1 plane, 128-byte swizzle, out-of-range elements read as zero.
bool make_plane_map(CUtensorMap *map, const uint8_t *base, int64_t lines, int64_t pitch,
                    int64_t plane_stride, int planes, int box_lines)
{
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return false;
    cuuint64_t dims[3] = {static_cast<cuuint64_t>(pitch), static_cast<cuuint64_t>(lines),
                          static_cast<cuuint64_t>(planes)};
    cuuint64_t strides[2] = {static_cast<cuuint64_t>(pitch), static_cast<cuuint64_t>(plane_stride)};
    cuuint32_t box[3] = {static_cast<cuuint32_t>(BLOCK_K), static_cast<cuuint32_t>(box_lines), 1};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult rc = fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, const_cast<uint8_t *>(base), dims, strides,
                     box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                     CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return rc == CUDA_SUCCESS;
}

// 3-D map over private-layout planes[plane * chunks + chunk][line][128 bytes] for the fused kernel: box = 16 bytes x
// 128 lines x 1 chunk, no swizzle (8 rows x 16 bytes land as one contiguous core matrix), out-of-range
// elements read as zero.
bool make_core_matrix_map(CUtensorMap *map, const uint8_t *base, int64_t lines, int64_t chunks_total)
{
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return false;
    cuuint64_t dims[3] = {static_cast<cuuint64_t>(BLOCK_K), static_cast<cuuint64_t>(lines),
                          static_cast<cuuint64_t>(chunks_total)};
    cuuint64_t strides[2] = {static_cast<cuuint64_t>(BLOCK_K), static_cast<cuuint64_t>(BLOCK_K * lines)};
    cuuint32_t box[3] = {16, 128, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult rc = fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, const_cast<uint8_t *>(base), dims, strides,
                     box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                     CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return rc == CUDA_SUCCESS;
}

template <int SUB, int SET>
oz_status_t launch_fused_variant(const CUtensorMap &mapB, const GemmParams &p, const FusedGemmParams &f, int sms,
                                 cudaStream_t stream)
{
    constexpr int LAYOUT_A = SUB == 0 ? kLayoutMerged : kLayoutMergedI8A;
    auto kernel = fused_gemm_kernel<SUB, SET, LAYOUT_A>;
    constexpr size_t smem = fused_gemm_smem(SET);
    OZ_CUDA_CHECK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem)));
    const int grid = f.tiles < sms ? f.tiles : sms;
    kernel<<<grid, F_THREADS, smem, stream>>>(mapB, p, f);
    count_launch();
    OZ_CUDA_CHECK(cudaGetLastError());
    return OZ_OK;
}

template <int SUB, int CG, int RB, bool DIRECT = false, bool TILED = false, bool BOUND = false, int SLIM = 0, int BN = BLOCK_N>
oz_status_t launch_variant(const CUtensorMap &mapA, const CUtensorMap &mapB, const GemmParams &p, int sms,
                           cudaStream_t stream)
{
    auto kernel = residue_gemm_kernel<SUB, CG, RB, DIRECT, TILED, BOUND, SLIM, BN>;
    static std::atomic<unsigned long long> ready{0};
    OZ_CUDA_CHECK(allow_shared(kernel, SMEM_BYTES, ready));
    int64_t groups = sms / CG;                                    // CTAs, or CTA pairs
    if (p.total_items < groups) groups = p.total_items;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(groups * CG));
    cfg.blockDim = dim3(NUM_THREADS);
    cfg.dynamicSmemBytes = SMEM_BYTES;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CG;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    OZ_CUDA_CHECK(cudaLaunchKernelEx(&cfg, kernel, mapA, mapB, p));
    count_launch();
    OZ_CUDA_CHECK(cudaGetLastError());
    return OZ_OK;
}


// Whole-method products (tile-ordered residues): the variants of one substrate, residue width and tile height
template <int SUB, int RB, bool DIRECT, int BN>
oz_status_t launch_tiled(const CUtensorMap &mapA, const CUtensorMap &mapB, const GemmParams &p, int cg, bool slim, int sms, cudaStream_t stream)
{
    if constexpr (!DIRECT) {
        if (slim)
            return p.n <= 64 ? launch_variant<SUB, 1, RB, false, true, false, 64, BN>(mapA, mapB, p, sms, stream)
                             : launch_variant<SUB, 1, RB, false, true, false, 128, BN>(mapA, mapB, p, sms, stream);
    }
    return cg == 2 ? launch_variant<SUB, 2, RB, DIRECT, true, false, 0, BN>(mapA, mapB, p, sms, stream)
                   : launch_variant<SUB, 1, RB, DIRECT, true, false, 0, BN>(mapA, mapB, p, sms, stream);
}

template <int SUB, int RB, bool DIRECT>
oz_status_t launch_tiled(const CUtensorMap &mapA, const CUtensorMap &mapB, const GemmParams &p, int cg, bool slim, bool narrow, int sms,
                         cudaStream_t stream)
{
    return narrow ? launch_tiled<SUB, RB, DIRECT, NARROW_N>(mapA, mapB, p, cg, slim, sms, stream)
                  : launch_tiled<SUB, RB, DIRECT, BLOCK_N>(mapA, mapB, p, cg, slim, sms, stream);
}

// Tiles of 64 rows instead of 256 where the rounds over the SMs then cost less.  A narrow tile is bound by its operands' way
// from L2 to shared memory, not by its quarter of the products: per K chunk it needs 5/8 of a wide one's bytes in CTA pairs and with
// 128 lines of B in the two-plane schedule (20 of 32, 40 of 64 KiB), half in the other forms (24 of 48).  5/8 serves them all: with
// 4/8 and 6/8 products of 200 to 9000 rows and 16 to 300 columns stayed within 3 percent either way (1300 x 128 x 300: 23.2, 22.6 and 22.6 us).
// (3/8, which takes narrow tiles more often: 53 of 160 drawn products change, to 0.88 to 1.14 of their time, 1.02 in the mean.)
bool narrow_tiles(int64_t m, int64_t tiles_n, int r, int cg, int sms)
{
    const int64_t groups = sms / cg;
    const int64_t wide = (r * tiles_n * ((m + BLOCK_N - 1) / BLOCK_N) + groups - 1) / groups;
    const int64_t narrow = (r * tiles_n * ((m + NARROW_N - 1) / NARROW_N) + groups - 1) / groups;
    return 5 * narrow < 8 * wide;
}

}  // namespace

// Which variant runs: CTA pairs (tcgen05 cta_group::2, tiles of 256 columns) unless that would pad
// the column count noticeably more than 128-column tiles do (n = 128: one half-empty pair tile).
static int cta_group_choice(int64_t n)
{
    const int64_t pad1 = round_up(n, BLOCK_M), pad2 = round_up(n, 2 * BLOCK_M);
    return (pad2 * 20 <= pad1 * 21) ? 2 : 1;
}

// Test hook for the bounded waits, read once when the library is loaded: with
// OZ_TEST_STALL_PRODUCER=once in the environment the first residue-GEMM launch of the process loads
// no operand, every role's wait runs into its time limit, the kernel sets OZ_ERR_TIMEOUT and
// returns cleanly; later launches are normal.  ("1": every launch.)
static std::atomic<int> g_stall_producer{[] {
    const char *env = getenv("OZ_TEST_STALL_PRODUCER");
    if (!env) return 0;
    return env[0] == '1' ? 1 : (env[0] == 'o' ? 2 : 0);
}()};

static int take_stall_flag()
{
    int v = g_stall_producer.load();
    if (v == 2) {
        g_stall_producer.store(0);
        return 1;
    }
    return v;
}

// Per-modulus constants of the epilogue and the accumulator schedule (jobs, weights, which
// accumulators are reduced before they are weighted, K segments) for inner dimension k; p.r and p.nk
// (chunks of BLOCK_K) are set by the caller.  Calls of up to about 128^3 wait for the host: with the starts of the stored residues summed
// anew for every modulus a call kept it for 10.6 us, like this for 10.4.
static void fill_mod_info(GemmParams &p, int set, const Route &rt, int64_t k, bool slim = false)
{
    p.patch_bytes = 0;
    for (int i = 0; i < p.r; ++i) {
        const int mi = modulus(set, i), s = kSetTables.root[set][i];
        p.mod[i].m = static_cast<float>(mi);
        p.mod[i].inv_m = 1.0f / static_cast<float>(mi);
        // Exact range of the running combination.  Digits are bounded by |d0| <= 14 (16 for
        // squares), |d1| <= 16, |d0+d1| <= 22 (Lemma 1), a reduced accumulator by (m+1)/2 <= 545
        // (FP32 path, balanced) or m-1 <= 1088 (integer path, canonical).  A job's accumulator may
        // be weighted without reducing it first while the worst-case sum stays inside the exact
        // range: 2^24 for the FP32 epilogue (minus the centre), 2^31 (minus headroom for the bias) for the integer one.
        const bool integer = rt.substrate != 0;
        const int64_t lim = integer ? (1ll << 31) - 8192 : (1ll << 24) - 546, kk = k > 0 ? k : 1;
        const int64_t red = integer ? 1088 : 545;
        ModInfo &mo = p.mod[i];
        float w[3] = {0.0f, 0.0f, 0.0f};
        mo.mi = static_cast<uint32_t>(mi);
        mo.magic = barrett_magic(static_cast<uint32_t>(mi));
        mo.bias = static_cast<uint32_t>((((1ull << 31) + mi - 1) / mi) * mi);
        mo.magic39 = mi > 128 ? static_cast<uint32_t>(((1ull << 39) + mi - 1) / mi) : 0u;
        mo.bias30 = static_cast<uint32_t>((((1ull << 30) + mi - 1) / mi) * mi);
        mo.store_form = form_of(mi);
        mo.store_start = p.patch_bytes;
        p.patch_bytes += form_bytes(mo.store_form);
        mo.centre = static_cast<float>((mi + 1) / 2);
        mo.planeA0 = kSetTables.first[set][rt.layout(0)][i];
        mo.planeB0 = kSetTables.first[set][rt.layout(1)][i];
        mo.nseg = 1;
        mo.seg_len = p.nk;
        // exact depth of one accumulator, in chunks of BLOCK_K: the largest term is 2 * 16 * 16 (the
        // two-product job of a square), 128 * 128 for native residues
        const int seg_max_all = !integer ? (1 << 24) / 512 / BLOCK_K
                                         : static_cast<int>(((1ll << 31) - 1) / (rt.native() ? 16384 : 512) / BLOCK_K);
        mo.nseg_all = (p.nk + seg_max_all - 1) / seg_max_all;
        mo.seg_len_all = (p.nk + mo.nseg_all - 1) / mo.nseg_all;
        const bool split = mo.nseg_all > 1;       // then every accumulator is reduced before it is weighted
        if (rt.native()) {
            mo.njobs = 1;
            mo.kind = 2;
            w[0] = 1.0f; w[1] = w[2] = 0.0f;
            mo.reduce[0] = split ? 1 : 0;
            mo.reduce[1] = mo.reduce[2] = 1;
        } else if (s) {
            mo.njobs = 2;
            mo.kind = 0;
            w[0] = 1.0f; w[1] = static_cast<float>(s); w[2] = 0.0f;
            const bool skip_all = !split && integer && (256 + 512 * static_cast<int64_t>(s)) * kk <= lim;
            mo.reduce[0] = (skip_all || (!split && 256 * kk + static_cast<int64_t>(s) * red <= lim)) ? 0 : 1;
            mo.reduce[1] = skip_all ? 0 : 1;
            mo.reduce[2] = 1;
        } else if (slim) {
            // d e = acc0 + 16 acc1.  Planes d0, d1 against e and f: terms 8 8 + 16 8 and 8 16 + 16 16.  Planes of the merged
            // layouts, d0 and -16 d1 (Lemma 1: |d0| <= 14, |d1| <= 16 on the 9-bit tail, 8 and 8 on bytes): 14 14 + 256 14 and
            // 14 16 + 256 16, or 8 8 + 128 8 in both, and K segments that keep these exact.
            mo.njobs = 2;
            mo.kind = rt.two_plane() ? 4 : 5;
            w[0] = 1.0f; w[1] = 16.0f; w[2] = 0.0f;
            const int64_t t0 = mo.kind == 4 ? 192 : (mi > 256 ? 3780 : 1088), t1 = mo.kind == 4 ? 384 : (mi > 256 ? 4320 : 1088);
            if (mo.kind == 5) {
                const int seg_max = static_cast<int>((1 << 24) / t1 / BLOCK_K);
                mo.nseg_all = (p.nk + seg_max - 1) / seg_max;
                mo.seg_len_all = (p.nk + mo.nseg_all - 1) / mo.nseg_all;
            }
            const int64_t first = 16 * red * mo.nseg_all;     // the other accumulator's part once it is reduced
            const bool one = mo.nseg_all == 1;
            const bool skip_all = one && (t0 + 16 * t1) * kk <= lim;
            mo.reduce[0] = (skip_all || (one && t0 * kk + first <= lim)) ? 0 : 1;
            mo.reduce[1] = skip_all ? 0 : 1;
            mo.reduce[2] = 1;
        } else if (rt.merged()) {
            // d e = -15 [d0 e0 - 16 d1 e1] + 16 dS eS; merged term <= 4095 (9-bit tail) or 1088 (bytes).
            // INT8 planes hold -d0 and 4*d1, so the accumulator is the NEGATIVE of the bracket (weight
            // +15) and its term is bounded by 4292 for every modulus up to 1089.
            mo.njobs = 2;
            mo.kind = 3;
            w[0] = integer ? 15.0f : -15.0f; w[1] = 16.0f; w[2] = 0.0f;
            // K longer than the exact range of one merged accumulator is cut into equal segments,
            // each drained and reduced on its own (the residues add modulo m).
            const int64_t merged_term = integer ? 4292 : (mi > 256 ? 4095 : 1088);
            const int seg_max = integer ? static_cast<int>(((1ll << 31) - 1) / merged_term / BLOCK_K)
                                        : static_cast<int>(merged_k_limit(set) / BLOCK_K);
            mo.nseg = (p.nk + seg_max - 1) / seg_max;
            if (mo.nseg < 1) mo.nseg = 1;
            mo.seg_len = (p.nk + mo.nseg - 1) / mo.nseg;
            const bool skip_all = !split && mo.nseg == 1 && (15 * merged_term + 16 * 484) * kk <= lim;
            mo.reduce[0] = skip_all ? 0 : 1;
            mo.reduce[1] = (skip_all || (!split && 16 * 484 * kk + 15 * red * mo.nseg <= lim)) ? 0 : 1;
            mo.reduce[2] = 1;
        } else {
            mo.njobs = 3;
            mo.kind = 1;
            w[0] = -15.0f; w[1] = 16.0f; w[2] = 240.0f;
            const bool skip_all = !split && integer && (15 * 196 + 16 * 484 + 240 * 256) * kk <= lim;
            const bool skip01 = skip_all || (!split && (15 * 196 + 16 * 484) * kk + 240 * red <= lim);
            mo.reduce[0] = skip01 ? 0 : 1;
            mo.reduce[1] = skip01 ? 0 : 1;
            mo.reduce[2] = skip_all ? 0 : 1;
        }
        for (int j = 0; j < 3; ++j) {
            const int as_int = static_cast<int>(w[j]);
            if (integer) memcpy(&mo.w[j], &as_int, sizeof(as_int));
            else memcpy(&mo.w[j], &w[j], sizeof(w[j]));
        }
    }
}

bool two_plane_applies(int64_t m, int64_t n, const Route &rt)
{
    return rt.automatic && rt.merged() && !rt.fused && n <= BLOCK_M && m >= n;
}

// Kept operands (planes of the merged layouts): a fifth less of A from memory for a sixth more products, which up to 64 columns both
// accumulators share.  Calls with three planes and with two, us: set S 2126 x 9 x 8360 109 -> 89, 1200 x 64 x 9000 113 -> 87, 3000 x 64 x 30000
// (eight K segments) 457 -> 373; E 1900 x 50 x 20000 247 -> 196; A 800 x 50 x 16000 193 -> 144.  Not with more columns, whose
// accumulators need products of their own: 4000 x 100 x 4000 119 -> 118.
static bool slim_merged(int64_t n) { return n <= 64; }

ResidueTiling residue_tiling(int64_t m, int64_t n, int set)
{
    ResidueTiling t;
    t.cg = cta_group_choice(n);
    t.tile_cols = BLOCK_M * t.cg;
    t.tiles_m = static_cast<int>((m + BLOCK_N - 1) / BLOCK_N);
    t.tiles_n = static_cast<int>((n + t.tile_cols - 1) / t.tile_cols);
    t.mod_stride = static_cast<int64_t>(t.tiles_m) * t.tiles_n * t.tile_cols * BLOCK_N;
    (void)set;
    return t;
}

oz_status_t launch_residue_gemm(int64_t m, int64_t n, int64_t k, const uint8_t *PA, int64_t strideA,
                                int64_t pitchA, const uint8_t *PB, int64_t strideB, int64_t pitchB,
                                int set, const Route &rt, void *R, int64_t ldr,
                                int64_t mod_stride, bool tiled, cudaStream_t stream)
{
    const int cg = cta_group_choice(n);
    GemmParams p{};
    p.m = m; p.n = n; p.k = k;
    p.tiles_n = static_cast<int>((n + BLOCK_M * cg - 1) / (BLOCK_M * cg)); // 128 (256) columns of C per tile
    const int sms = sm_count();
    const bool narrow = tiled && narrow_tiles(m, p.tiles_n, set_r(set), cg, sms);
    const int rows = narrow ? NARROW_N : BLOCK_N;                          // rows of C per tile
    p.tiles_m = static_cast<int>((m + rows - 1) / rows);
    const int rb = residue_bytes(set);
    p.vec_store = ((ldr * rb) % 16 == 0 && (mod_stride * rb) % 16 == 0 && (reinterpret_cast<uintptr_t>(R) & 15u) == 0) ? 1 : 0;
    p.nk = static_cast<int>((k + BLOCK_K - 1) / BLOCK_K);
    if (k == 0) p.nk = 1;   // one all-zero chunk (the planes' padding) gives residues 0
    p.r = set_r(set);
    p.total_items = static_cast<int64_t>(p.r) * p.tiles_m * p.tiles_n;
    if (p.total_items >= 0x7FFFFFFFll) return OZ_ERR_UNSUPPORTED;        // item numbers are 32-bit in the kernel
    p.R = R; p.ldr = ldr; p.mod_stride = mod_stride;
    p.stall_producer = take_stall_flag();
    p.status = device_status_word();
    const bool slim = tiled && cg == 1 && p.tiles_n == 1 && (rt.two_plane() || (rt.merged() && rt.substrate == 0 && slim_merged(n)));
    fill_mod_info(p, set, rt, k, slim);
    // Squares in one K-loop: the products of a square read d0 and e0 twice, so job after job a K chunk costs six tiles;
    // with both accumulators open it costs four.  The drains of the two slots hide behind less of the K-loop than job after
    // job, which costs less than the tiles at every size measured, with the slots still filled and emptied together: 10240 x 64 x 10240 with a kept operator (DRAM) 680 -> 620 us a
    // call, 131072 x 128 x 4096 9159 -> 8801, 16384 x 16384 x 1024 (power) 11.52 -> 11.10 ms, 4096^3 2371 -> 2358 us.  Not
    // with K segments, whose accumulators take the slots in turn.
    p.pair_squares = !rt.native() && p.mod[0].nseg_all == 1;

    CUtensorMap mapA, mapB;
    const int planesA = kSetTables.first[set][rt.layout(0)][p.r], planesB = kSetTables.first[set][rt.layout(1)][p.r];
    bool maps;
    if (tiled) {       // private layout: one 128-byte column of lines per (plane, chunk); both operands have the same pitch
        const int chunks = static_cast<int>(pitchA / BLOCK_K);
        p.kc_x = 0; p.plane_z = chunks; p.kc_z = 1;
        maps = make_plane_map(&mapA, PA, m, BLOCK_K, BLOCK_K * m, planesA * chunks, rows / cg) &&
               make_plane_map(&mapB, PB, n, BLOCK_K, BLOCK_K * n, planesB * chunks, slim && n <= 64 ? 64 : BLOCK_M);
    } else {
        p.kc_x = BLOCK_K; p.plane_z = 1; p.kc_z = 0;
        maps = make_plane_map(&mapA, PA, m, pitchA, strideA, planesA, BLOCK_N / cg) &&
               make_plane_map(&mapB, PB, n, pitchB, strideB, planesB, BLOCK_M);
    }
    if (!maps) return OZ_ERR_CUDA;

    // one accumulator per modulus of at most 128 * 128 * k <= 2^30: the direct drain with the exact division
    const bool direct = rt.native() && p.mod[0].nseg_all == 1 && k <= 65536;
    // substrate 0: FP8 planes; otherwise INT8 planes (two-limb digits or native residues)
    if (tiled) {
#define OZ_TILED(SUB, RB, DIRECT) launch_tiled<SUB, RB, DIRECT>(mapA, mapB, p, cg, slim, narrow, sms, stream)
        if (direct) return OZ_TILED(1, 1, true);
        if (rb == 1) return rt.substrate == 0 ? OZ_TILED(0, 1, false) : OZ_TILED(1, 1, false);
        return rt.substrate == 0 ? OZ_TILED(0, 2, false) : OZ_TILED(1, 2, false);
#undef OZ_TILED
    }
#define OZ_LAUNCH(SUB, RB, DIRECT)                                                                  \
    (cg == 2 ? launch_variant<SUB, 2, RB, DIRECT>(mapA, mapB, p, sms, stream)                      \
             : launch_variant<SUB, 1, RB, DIRECT>(mapA, mapB, p, sms, stream))
    if (direct) return OZ_LAUNCH(1, 1, true);
    if (rb == 1) return rt.substrate == 0 ? OZ_LAUNCH(0, 1, false) : OZ_LAUNCH(1, 1, false);
    return rt.substrate == 0 ? OZ_LAUNCH(0, 2, false) : OZ_LAUNCH(1, 2, false);
#undef OZ_LAUNCH
}

// Whether the fused mode applies: merged schedule on digit planes, all of B in one 128-lane tile, and
// an inner dimension that every accumulator holds exactly without K segments.
bool fused_gemm_applies(int64_t m, int64_t n, int64_t k, int set, const Route &rt)
{
    if (rt.native() || !rt.merged() || n < 1 || n > BLOCK_M || m < 1 || k < 1) return false;
    if ((m + F_LINES - 1) / F_LINES >= 0x7FFFFFFFll) return false;
    // one accumulator per job over all of k: FP32 holds the merged term (4095 on the 9-bit tail of S,
    // 1088 on byte moduli) exactly to 2^24, INT32 the term 4292 far beyond any k taken here; where the
    // epilogue reduces an accumulator before weighting it is decided for this k by fill_mod_info
    const int64_t kmax = rt.substrate == 0 ? merged_k_limit(set) : 262144;
    return k <= kmax;
}

// Residue products with A converted on the fly (storage mode F): A in FP64 with the shifts of its rows,
// B's planes materialised in the layout of side 1 of the route; canonical residues in the public layout
// R[mod][j][ldr], ldr a multiple of 64 and at least m rounded up to 64 (the last tile stores whole).
oz_status_t launch_fused_gemm(int64_t m, int64_t n, int64_t k, const double *A, int64_t lda, const int32_t *shiftA,
                              const uint8_t *PB, int64_t pitchB, int set, const Route &rt, void *R, int64_t ldr,
                              int64_t mod_stride, cudaStream_t stream)
{
    if (!fused_gemm_applies(m, n, k, set, rt)) return OZ_ERR_UNSUPPORTED;
    if (ldr % F_LINES != 0 || ldr < round_up(m, F_LINES) || (reinterpret_cast<uintptr_t>(R) & 15u)) return OZ_ERR_INVALID_ARG;
    GemmParams p{};
    p.m = m; p.n = n; p.k = k;
    p.r = set_r(set);
    p.nk = static_cast<int>((k + BLOCK_K - 1) / BLOCK_K);
    p.R = R; p.ldr = ldr; p.mod_stride = mod_stride;
    p.stall_producer = 0;
    p.status = device_status_word();
    fill_mod_info(p, set, rt, k);
    FusedGemmParams f{};
    f.A = A; f.lda = lda; f.shiftA = shiftA;
    f.lut_global = device_lut(set, rt.substrate);
    f.tz = rt.quant;
    f.tiles = static_cast<int>((m + F_LINES - 1) / F_LINES);
    f.passes = (p.r + F_GROUP - 1) / F_GROUP;
    f.nks = static_cast<int>((k + F_K - 1) / F_K);
    CUtensorMap mapB;
    f.chunksB = static_cast<int>(pitchB / BLOCK_K);
    if (!make_core_matrix_map(&mapB, PB, n, static_cast<int64_t>(p_store(set, rt.layout(1))) * f.chunksB)) return OZ_ERR_CUDA;
    const int sms = sm_count();
#define OZ_FUSED_GEMM(SET_) \
    (rt.substrate == 0 ? launch_fused_variant<0, SET_>(mapB, p, f, sms, stream) : launch_fused_variant<1, SET_>(mapB, p, f, sms, stream))
    if (set == 0) return OZ_FUSED_GEMM(0);
    if (set == 1) return OZ_FUSED_GEMM(1);
    return OZ_FUSED_GEMM(2);
#undef OZ_FUSED_GEMM
}

// The magnitude-bound product of the accurate mode: one E4M3 plane per operand (digits <= 32, terms
// <= 1024, so one FP32 accumulator is exact for k <= 16384), the same tiles, TMA ring and tcgen05
// instructions as the residue products, and an epilogue that keeps only the row and column maxima.
oz_status_t launch_bound_gemm(int64_t m, int64_t n, int64_t k, const uint8_t *GA, int64_t pitchA,
                              const uint8_t *GB, int64_t pitchB, unsigned int *rowmax,
                              unsigned int *colmax, cudaStream_t stream)
{
    if (k > kBoundKMax) return OZ_ERR_UNSUPPORTED;
    const int cg = cta_group_choice(n);
    GemmParams p{};
    p.m = m; p.n = n; p.k = k;
    p.tiles_m = static_cast<int>((m + BLOCK_N - 1) / BLOCK_N);
    p.tiles_n = static_cast<int>((n + BLOCK_M * cg - 1) / (BLOCK_M * cg));
    p.nk = static_cast<int>((k + BLOCK_K - 1) / BLOCK_K);
    if (k == 0) p.nk = 1;
    p.r = 1;
    p.total_items = static_cast<int64_t>(p.tiles_m) * p.tiles_n;
    if (p.total_items >= 0x7FFFFFFFll) return OZ_ERR_UNSUPPORTED;
    p.stall_producer = 0;
    p.kc_x = BLOCK_K; p.plane_z = 1; p.kc_z = 0;
    p.status = device_status_word();
    p.rowmax = rowmax;
    p.colmax = colmax;
    ModInfo &mo = p.mod[0];
    mo.m = 1.0f; mo.inv_m = 1.0f; mo.mi = 1u;
    mo.njobs = 1;
    mo.kind = 2;                       // one plane, one K-loop
    mo.w[0] = 0x3F800000u;             // 1.0f
    mo.reduce[0] = 0;
    mo.planeA0 = mo.planeB0 = 0;
    mo.nseg = mo.nseg_all = 1;
    mo.seg_len = mo.seg_len_all = p.nk;
    CUtensorMap mapA, mapB;
    if (!make_plane_map(&mapA, GA, m, pitchA, m * pitchA, 1, BLOCK_N / cg) ||
        !make_plane_map(&mapB, GB, n, pitchB, n * pitchB, 1, BLOCK_M))
        return OZ_ERR_CUDA;
    const int sms = sm_count();
    return cg == 2 ? launch_variant<0, 2, 2, true, false, true>(mapA, mapB, p, sms, stream)
                   : launch_variant<0, 1, 2, true, false, true>(mapA, mapB, p, sms, stream);
}

}  // namespace oz
