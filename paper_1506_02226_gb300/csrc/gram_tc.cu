// gram_tc.cu — tensor-core Gram form of the pair test (tcgen05, sm_103a).
//
// Section IV-B of the paper rewrites the squared distance as
//   dist(t, p) = |t|^2 + |p|^2 - 2 t.p
// and hoists the per-point terms out of the loop.  For d >= 16 the dot
// products t.p of a 128 x 256 tile of pairs are one dense contraction, so they
// run on the 5th-generation tensor cores: tcgen05.mma with FP16 or BF16
// operands staged in shared memory and an FP32 accumulator in tensor memory.
//
// Exactness.  Coordinates are centred, v = u - 512 in [-512, 511]:
//   FP16 holds every v exactly, products are exact, and for d <= 64 every
//   partial sum of G = v_p . v_q is an integer of magnitude <= 64 * 2^18 =
//   2^24, so FP32 accumulation leaves G exact.  Then, with beta_q = |v_q|^2 and
//   alpha_p = |v_p|^2 - T (both exact integers, |.| <= 2^24 because T < 2^24),
//   w = fma(2, G, -beta_q) rounds at most once, and w >= alpha_p decides
//   D(p,q) <= T exactly: when |2G - beta| > 2^24 the rounded w stays on the
//   same side of alpha.  The stated FP16 band is therefore 0; the diagnostic
//   pass (TC_VERIFY, dbscan_tc_verify) recomputes every pair exactly on the
//   device and reports max |2G - 2G_exact| = 0 and no pair decided wrongly.
//   BF16 (8-bit significand) cannot hold every v, so each is split into two
//   BF16 terms, v = hi + lo with hi = bf16(v) and lo = v - hi in {-1, 0, 1}
//   (both exact), and the MMA sums hi.hi + hi.lo + lo.hi over K, i.e. G minus
//   sum(lo_p lo_q), |sum| <= K.  Its partial sums stay below
//   K (512^2 + 2 * 512) < 2^25, so each of the 3K accumulations beyond 2^24
//   rounds by at most 2: |G_bf16 - G| <= 7K.  With the roundings of w (at most
//   4 each), a pair is decided directly when |w - alpha| > 16K, and rechecked
//   exactly otherwise (rho = sqrt(16K) (1 + 2^-10) per row and column, so that
//   rho_p rho_q covers the band).  The band holds only pairs within 16K
//   squared units of the threshold.
//
// Folded FP16 count.  The count pass multiplies one more 16-column chunk, so
// that the MMA also subtracts the column term: rows carry 1, 2^11, 2^15 and
// columns the negated digits of h_q = ceil(|v_q|^2 / 2) (integers FP16 holds
// exactly), and the accumulator holds G - h_q.  Every term of that sum is an
// integer and their magnitudes add up to at most
// |v_p||v_q| + h_q <= (|v_p|^2 + 2|v_q|^2 + 1) / 2, so when
// 3 max|v|^2 + 1 <= 2^25 every partial sum, in any order of accumulation, is
// an integer of magnitude <= 2^24 and the accumulator is exact.  With f the
// parity of |v_q|^2, D <= T iff G - h_q >= ceil((|v_p|^2 - T - f) / 2); each
// 256-column tile holds its even |v_q|^2 first, so all but one of its groups
// of 32 columns share one threshold per row.  The epilogue then needs one
// saturating add per pair and no column data.  Inputs with larger norms (only
// the extreme corners of the grid reach them at d = 64) run the same pass on G
// alone with the column norms; the pass decides on the device.
//
// Which tile pairs run.  All pairs would be (n / 256)^2 tile pairs.  From
// kSortMinN points on, the points are put in groups first and most tile pairs
// are proved empty:
//   order   each point goes to its nearest of P sampled pivots (a Gram pass
//           against the pivots' tiles) and points are sorted by (class, pivot):
//           the class is the ratio of that distance to eps, so that dense groups
//           come before scattered points, and pivots within 2 eps of one another
//           are neighbours in the order, so the 256 points of a tile lie close
//           together;
//   balls   a tile's points are split in two by their nearer of two seeds, each
//           part with its rounded mean c and the exact largest distance r to it;
//   cull    a Gram pass of the centres against all points gives, per ball and
//           tile, the least distance m of the tile's points to c; when
//           m > r + eps for one tile's points and both balls of the other, the
//           triangle inequality leaves no pair of the two within eps.
// The passes below visit the remaining tile pairs (a bit matrix).  The tests
// are one-sided (m is an underestimate, r + eps an overestimate), so the order
// and the cull change no result, only how much is proved empty: 200,000 x 64
// in 100 blobs plus 15% noise evaluates 2.74e9 pairs instead of 5.70e10 in the
// three passes (1.07 ms a run instead of 8.74; 100,003 x 48 in BF16 0.94 instead
// of 6.87 ms; a burst of 40 served jobs, a third of them at d = 32, 9.7 instead
// of 65.0 ms).  The limit of 32,768 points is where ordering (some 0.2 ms) and
// testing all pairs cost about the same.  Three more rules skip
// work whose outcome is known: the count leaves a row unit once all its rows
// have min_pts neighbours (unless exact counts are asked for), the merge skips
// a tile pair when each tile's core points are known to be one set and the two
// sets are one, and the border takes only rows that are not core and have a
// neighbour at all.
//
// Data layout.  The points of a tile (256 consecutive positions of the order)
// are packed once, in the canonical K-major layout without swizzle: 8 x 8
// core matrices of 128 contiguous bytes, K-adjacent core matrices 128 B apart
// (leading byte offset) and 8-row groups KG * 128 B apart (stride byte
// offset), followed for FP16 by the folded chunk in the same layout.  A
// 128-row A operand, a 256-row A operand or a 256-column B tile is therefore
// one contiguous block, fetched by a single cp.async.bulk (TMA) copy.  The
// union-find forest, counts and core flags are by position, so a tile's
// entries are contiguous too; labels are mapped to point indices at the end.
//
// CTA roles (320 threads for the FP16 count, order, cull and verification
// passes, 576 otherwise; one CTA per SM, persistent over work items of one row
// unit and a chunk of column tiles):
//   warp 0      producer: finds the next work items that are not empty (32 at a
//               time, a lane each), streams their A operands (2 buffers), B
//               tiles (a ring of 2 to 5 stages, freed by the MMA commit of the
//               tile) and, in a ring of their own, the tiles' metadata and what
//               comes next (a column tile, the item's end, no more work)
//   warp 1      TMEM owner (alloc/dealloc of 512 columns) and MMA issuer:
//               K/16 tcgen05.mma (M=128, N=256, K=16) per MMA tile into one of
//               two 256-column accumulators (with two row tiles, each B tile
//               feeds one MMA tile per row tile, one per accumulator);
//               tcgen05.commit signals the epilogue
//   warps 2..   epilogue: tcgen05.ld of the accumulator (one TMEM lane = one
//               row), the exact decision above, and the pass's consumer.
// Every wait is bounded (about two seconds of %globaltimer); on expiry the CTA
// records DB_EBIT_TIMEOUT, stops issuing work, waits for its own copies and
// MMAs, frees its TMEM and returns.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <atomic>
#include <climits>
#include <cmath>
#include <type_traits>

#include "internal.cuh"
#include "tc_items.h"

namespace {

constexpr int TM = 128, TN = 256;
constexpr unsigned FULL = 0xffffffffu;
constexpr int FP16_BAND = 0;  // FP16 Gram products are exact (see above): no band
// BF16 candidate filter: lowering of its threshold that covers the rounding
// difference between the filter score and the rare path's score (below 16).
constexpr float kBf16FilterSlack = 16.f;
// BF16 band in units of w = 2G - |v_q|^2 for padded dimension K (see above).
__host__ __device__ constexpr int bf16_band(int K) { return 16 * K; }
// rho^2 of the band factor, the same for every point (rounded to FP32 once).
__host__ __device__ inline float bf16_rho(int K) { return sqrtf((float)bf16_band(K)) * (1.f + 1.f / 1024.f); }

// TC_ADJ: the merge's first step, the neighbours of each core point among the
// core points of its own tile, as bits.  TC_LINK, TC_ORDER: first pivot within
// twice eps, nearest pivot.  TC_CULL: ball tests.
enum { TC_COUNT = 0, TC_UNION = 1, TC_BORDER = 2, TC_VERIFY = 3, TC_ADJ = 4, TC_ORDER = 5, TC_CULL = 6, TC_LINK = 7 };

// Shape of each pass.  Rows: two row tiles per item (256 rows) for the FP16
// passes with a cheap or no consumer, one (128 rows) otherwise.  Epilogue
// warps: 8 for the FP16 count, order and cull (one warp per lane quadrant and
// row tile, each deciding all 256 columns), 16 for the FP16 border and adjacency
// (two warps per quadrant and row tile), 16 for the merge and the BF16 passes
// (four per quadrant), 8 for the verification.
template <int PASS, bool BF16>
struct Shape {
    static constexpr bool kWide = PASS == TC_ORDER || PASS == TC_CULL || PASS == TC_LINK || (PASS == TC_COUNT && !BF16);
    static constexpr int RTN = kWide || (!BF16 && (PASS == TC_BORDER || PASS == TC_ADJ)) ? 2 : 1;
    static constexpr int EPI = kWide || PASS == TC_VERIFY ? 8 : 16;
    static constexpr int GW = PASS == TC_VERIFY ? 64 : 32;  // columns per group
    static constexpr int THREADS = 32 * (2 + EPI);
};

// Per-tile metadata (256 positions): beta = |v|^2 (1e30 where the pass has no
// point: padding, or a point the pass masks out), the candidate filter's
// column term beta_f (beta for FP16, beta - rho^2 rounded for BF16), the point
// index, and the number of even-norm points, which come first.
struct MetaTile {
    float beta[TN];
    float beta_f[TN];
    int idx[TN];
    int n_even;
    int pad[63];
};
static_assert(sizeof(MetaTile) == 3328, "MetaTile: a multiple of 16 bytes, at most 16 bytes per point");

struct TcArgs {
    const uint16_t *opR;  // packed row operand
    const MetaTile *metaR;
    const uint16_t *opC;  // packed column operand
    const MetaTile *metaC;
    int nR, nC;           // rows, columns (points)
    int K;                // padded dimension (multiple of 16, <= 64)
    int kv;               // stored operand columns per row: K, or 2K (BF16 terms)
    int fold;             // tiles are followed by the folded chunk (TC_COUNT, FP16)
    int tile_r, tile_c;   // operand elements per 256-row tile of opR, opC
    int T;                // threshold (< 2^24)
    int min_pts;          // count: rows stop mattering at this many neighbours (0: exact counts)
    unsigned long long wait_ns;  // budget of every barrier wait
    int stall;                   // test hook: the MMA issuer issues nothing
    int ct_chunk;                // column tiles per work item: 1, 2, 4, 8, 16 or 32
    int rel_lo, rel_hi;          // chunks visited, relative to the one of the row unit's own tile
    int near_lo, near_hi;        // union: column tiles visited, relative to the row unit's own tile
    int rotate;                  // 1: relative chunks wrap around (count, border of sorted points)
    const unsigned *pairs;       // surviving tile pairs, row stride `words` (null: all)
    int words;
    const int *bmax_ptr;  // FP16 count: largest |v|^2 of the input (decides the folded form)
    int *udone;           // count: per row unit, one bit per epilogue warp whose rows are all done
    const int *tag;       // per tile: -2 no core point, -1 core points of several sets, else their common root
    int4 *items;          // work items that are not empty: unit, first tile, tile bits (null: found by the producers)
    int *nlist, *ticket;  // their number, the next to be taken
    unsigned *adj;        // adjacency: 8 words a row, its neighbours in its own tile
    const int *rowneed;   // border: per tile, some row needs the pass
    const int16_t *v16;   // centred units by position, row stride K (exact recheck)
    int *count;
    int *parent;
    int *border;
    unsigned *status;
    unsigned long long *ctr;  // [6] band pairs, [7] verify: disagreements outside the band, [8] max |w - exact|
    int n_piv;                // order: pivots
    const int *prank;         // order: rank of each pivot among the buckets
    int *key, *rank, *hist;   // order: bucket of each point, its rank in it, bucket sizes
    const float *cbeta, *crad;  // cull: per ball |c|^2 and the largest squared distance of its points (-1: none)
    unsigned *near;           // cull: per tile and ball, "some point of the tile may be within r + eps" (bits)
};

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint64_t globaltimer() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// One thread of a converged warp, chosen by the hardware (elect.sync).  The
// compiler knows that a region guarded by it runs in a single thread, so the
// tensor-core and copy instructions in it, whose descriptors live in uniform
// registers, are issued straight; guarded by `lane == 0` each is issued
// through a per-thread loop.  200,000 x 64 FP16 count pass: 5.36 -> 4.67 ms.
__device__ __forceinline__ bool elect_one() {
    uint32_t pr;
    asm volatile("{\n\t.reg .pred P;\n\telect.sync _|P, 0xffffffff;\n\tselp.u32 %0, 1, 0, P;\n\t}" : "=r"(pr));
    return pr != 0;
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// try_wait with a suspend-time hint: a thread whose phase is not complete
// sleeps (issuing nothing) until the phase completes or about 0.5 ms pass.
__device__ __forceinline__ bool mbar_try_wait_sleep(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity), "r"(500000u)
        : "memory");
    return ok != 0;
}

// Bounded wait: about two seconds, or until another role has given up.
// Waiting threads sleep inside try_wait, so they take no issue slots from the
// epilogue warps sharing their SM sub-partition.
__device__ __noinline__ bool mbar_wait_slow(uint64_t *bar, uint32_t parity, volatile int *abort_flag,
                                            unsigned long long budget_ns) {
    const uint64_t t0 = globaltimer();
    while (true) {
        for (int i = 0; i < 8; ++i)
            if (mbar_try_wait_sleep(bar, parity)) return true;
        if (*abort_flag) return false;
        if (globaltimer() - t0 > budget_ns) {
            *abort_flag = 1;
            return false;
        }
    }
}
// The phase is usually complete: tested inline before the out-of-line wait.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, volatile int *abort_flag,
                                          unsigned long long budget_ns) {
    return mbar_try_wait(bar, parity) || mbar_wait_slow(bar, parity, abort_flag, budget_ns);
}
// The same for a whole warp, with one outcome.
__device__ __forceinline__ bool mbar_wait_warp(uint64_t *bar, uint32_t parity, volatile int *abort_flag,
                                               unsigned long long budget_ns) {
    return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag, budget_ns));
}

// Bounded wait that ignores the abort flag: the abort path uses it to let a
// role's own copies or MMAs in flight land before the CTA's memory goes away.
__device__ __noinline__ bool mbar_wait_quiet(uint64_t *bar, uint32_t parity, unsigned long long budget_ns) {
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = globaltimer();
    while (globaltimer() - t0 <= budget_ns)
        if (mbar_try_wait_sleep(bar, parity)) return true;
    return false;
}
constexpr unsigned long long kDrainNs = 100000000ull;  // 100 ms: copies and MMAs land in microseconds

// Packed FP32 pairs (sm_100 and later): two lanes of arithmetic per
// instruction, each rounded exactly as its scalar counterpart.
__device__ __forceinline__ unsigned long long f2_pack(float lo, float hi) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void f2_unpack(unsigned long long v, float &lo, float &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ unsigned long long f2_fma(unsigned long long a, unsigned long long b,
                                                     unsigned long long c) {
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ unsigned long long f2_add(unsigned long long a, unsigned long long b) {
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// Optional pipeline diagnostics (compile with -DDB_TC_WAIT_STATS): cycles each
// role spends blocked on each barrier, summed per pass into the counters
// listed at the end of the kernel.
#ifdef DB_TC_WAIT_STATS
#define TC_WAIT(acc, expr) ({ long long _t0 = clock64(); bool _r = (expr); acc += clock64() - _t0; _r; })
#else
#define TC_WAIT(acc, expr) (expr)
#endif

__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_alloc(uint32_t *dst, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst)),
                 "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

// D[tmem] (+)= A[smem] * B[smem]^T, M=128, N=256, K=16, FP32 accumulate.
__device__ __forceinline__ void mma_f16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                        uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ void mma_commit(uint64_t *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Waits for this thread's TMEM loads; the registers of r pass through the
// statement, so no use of them can be scheduled before the wait.
__device__ __forceinline__ void tmem_wait_ld_dep(uint32_t (&r)[32]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]),
                   "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]),
                   "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]),
                   "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
                 :
                 : "memory");
}

// 32 consecutive accumulator columns of this thread's TMEM lane (no wait).
__device__ __forceinline__ void tmem_ld32_nowait(uint32_t taddr, uint32_t *r) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
}

// Shared-memory matrix descriptor: no swizzle, K-major, LBO = 128 B (next core
// matrix along K), SBO = KG * 128 B (next 8-row group), descriptor version 1.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t sbo_bytes) {
    return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)(128u >> 4) << 16) |
           ((uint64_t)((sbo_bytes >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}

// Instruction descriptor, kind::f16: D = F32, A/B = F16 or BF16, both K-major,
// N = 256 (bits 17..22 hold N/8), M = 128 (bits 24..28 hold M/16).
__host__ __device__ constexpr uint32_t idesc_f16(bool bf16) {
    return (1u << 4) | ((bf16 ? 1u : 0u) << 7) | ((bf16 ? 1u : 0u) << 10) | ((uint32_t)(TN >> 3) << 17) |
           ((uint32_t)(TM >> 4) << 24);
}

// Exact D(p,q) <= T from the centred int16 rows (the recheck of band pairs).
__device__ __noinline__ int exact_sqdist(const int16_t *__restrict__ v16, int K, int p, int q) {
    const int4 *a = reinterpret_cast<const int4 *>(v16 + (size_t)p * K);
    const int4 *b = reinterpret_cast<const int4 *>(v16 + (size_t)q * K);
    int s = 0;
    for (int c = 0; c < K / 8; ++c) {
        int4 x = a[c], y = b[c];
        const int xs[4] = {x.x, x.y, x.z, x.w}, ys[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            int d0 = (int)(int16_t)(xs[h] & 0xffff) - (int)(int16_t)(ys[h] & 0xffff);
            int d1 = (xs[h] >> 16) - (ys[h] >> 16);
            s += d0 * d0 + d1 * d1;
        }
    }
    return s;
}

// 64 consecutive accumulator columns of this thread's TMEM lane (no wait), and
// the wait for them (see tmem_wait_ld_dep).
__device__ __forceinline__ void tmem_ld64_nowait(uint32_t taddr, uint32_t (&r)[64]) {
    tmem_ld32_nowait(taddr, r);
    tmem_ld32_nowait(taddr + 32, r + 32);
}
__device__ __forceinline__ void tmem_wait_ld_dep64(uint32_t (&r)[64]) {
    tmem_wait_ld_dep(*reinterpret_cast<uint32_t(*)[32]>(r));
    tmem_wait_ld_dep(*reinterpret_cast<uint32_t(*)[32]>(r + 32));
}

// Shared memory of one CTA: KC stored operand columns per row, NS stages of B
// tiles, NM events (a tile's metadata and what the event is).  A B stage is
// free again once its MMAs have completed; the epilogue holds only events, so
// the operand ring runs ahead of the MMAs whatever the epilogue's pace.
template <int KV, int KC, int NS, int NM, int RTN, int CR, bool ONES>
struct __align__(16) SmemT {
    static constexpr int NSTAGE = NS;
    static constexpr int NMETA = NM;
    static constexpr int NABUF = 2;
    uint16_t A[2 * RTN][TM * KV];  // 2 buffers of RTN row tiles
    uint16_t B[NS][TN * KC];
    uint16_t ones[ONES ? TM * 16 : 8];  // the folded chunk of every row: 1, 2^11, 2^15, zeros
    MetaTile metaA[2];
    MetaTile metaB[NM];
    uint64_t a_full[2], a_empty[2];
    uint64_t b_full[NS], b_empty[NS];
    uint64_t m_full[NM], m_empty[NM];
    uint64_t t_full[2], t_empty[2];
    uint64_t drain;    // abort path: one more MMA commit, waited for by the issuer
    int ev[NM];        // event: a column tile (>= 0), EV_END or EV_STOP
    int unit[2];       // row unit of the item in each A buffer
    int done[2];       // count: epilogue warps whose rows all have min_pts neighbours (bits)
    uint32_t tmem_base;
    int abort_flag;
    int drain_failed;  // a role's bounded drain wait gave up
    // union pass (CR = 512): hints of the column points' sets, per accumulator
    // buffer and column (shared by the warps of a column range; a buffer is
    // refilled only after all its epilogue warps have released it)
    int colroot[CR];
};
enum { EV_END = -1, EV_STOP = -2 };

// Stages: as many as fit 227 KB.  FP16 tiles are 32 KB (40 KB with the folded
// chunk), BF16 tiles 64 KB.
template <int PASS, bool BF16>
struct TcSmem {
    static constexpr int RTN = Shape<PASS, BF16>::RTN;
    static constexpr bool FOLD = !BF16 && PASS == TC_COUNT;
    using type = SmemT<BF16 ? 128 : 64, BF16 ? 128 : (FOLD ? 80 : 64), BF16 ? 2 : (FOLD ? 3 : (RTN == 2 ? 4 : 5)),
                       FOLD ? 4 : (RTN == 2 ? 5 : 6), RTN, PASS == TC_UNION ? 512 : 1, FOLD>;
    static constexpr size_t bytes = sizeof(type) + 1024;
    static_assert(bytes <= 232448, "shared memory of one CTA");
};

// Union of two members' sets; returns a root the merged set had at some moment
// (out of line: keeps the union-find loop out of the epilogue's registers).
__device__ __noinline__ int unite_sets(int *parent, int x, int y, unsigned *status) {
    return db::uf_unite_root(parent, x, y, status);
}

// Work item w: row unit u and the column tiles of one chunk, as a bit mask of
// tiles c0 .. c0 + 31 that need a visit.  Items are ordered by the chunk's
// distance from the unit's own, so the tiles around the diagonal of all units
// come first: their neighbours settle most counts and unions, and the rules
// below then drop later items.
template <int PASS, int RTN>
__device__ __forceinline__ unsigned item_mask(const TcArgs &a, int64_t w, int units, int nct, int &u, int &c0) {
    const int nchunk = (nct + a.ct_chunk - 1) / a.ct_chunk;
    const tcitems::Item it = tcitems::item(w, units);
    const int rel = a.rel_lo + it.rel;
    u = it.unit;
    const int i = RTN == 2 ? u : u >> 1;  // the unit's tile
    int ch = rel;
    if (PASS == TC_UNION || PASS == TC_ADJ || a.rotate) ch += i / a.ct_chunk;
    if (ch >= nchunk) {
        if (PASS == TC_UNION || PASS == TC_ADJ) return 0u;
        ch -= nchunk;
    }
    c0 = ch * a.ct_chunk;
    const int nt = min(a.ct_chunk, nct - c0);
    unsigned m = nt >= 32 ? FULL : ((1u << nt) - 1u);
    if (PASS == TC_ADJ) return a.tag[i] != -2 ? 1u << (i - c0) : 0u;
    if (PASS == TC_COUNT) {
        if (a.min_pts > 0 && a.udone[u] == (1 << Shape<TC_COUNT, RTN == 1>::EPI) - 1) return 0u;
    }
    if (PASS == TC_UNION) {  // tiles [i + near_lo, i + near_hi]
        if (c0 < i + a.near_lo) m = i + a.near_lo - c0 >= 32 ? 0u : m & ~((1u << (i + a.near_lo - c0)) - 1u);
        if (i + a.near_hi < c0 + 31) m = i + a.near_hi < c0 ? 0u : m & ((2u << (i + a.near_hi - c0)) - 1u);
    }
    if (PASS == TC_BORDER && !a.rowneed[i]) return 0u;
    if (a.pairs) m &= a.pairs[(size_t)i * a.words + (c0 >> 5)] >> (c0 & 31);
    if (PASS == TC_UNION || PASS == TC_BORDER) {
        const int ti = PASS == TC_UNION ? a.tag[i] : -1;
        if (ti == -2) return 0u;
        for (unsigned mm = m; mm; mm &= mm - 1) {
            const int b = __ffs(mm) - 1, tj = a.tag[c0 + b];
            if (tj == -2 || (PASS == TC_UNION && ti >= 0 && tj == ti)) m &= ~(1u << b);
        }
    }
    return m;
}

// The work items that are not empty, in about the order of their numbers, so
// that the pass's CTAs can take them one by one (200,000 x 64: dealt out by
// number, the busiest CTA of the count had 1.4 times the mean work).
template <int PASS, int RTN>
__global__ void __launch_bounds__(256) tc_items_kernel(TcArgs a) {
    db::wait_prior_grid();  // started as a programmatic dependent
    db::allow_next_grid();
    const int units = (a.nR + TM * RTN - 1) / (TM * RTN), nct = (a.nC + TN - 1) / TN;
    const int64_t nitems = tcitems::count(units, a.rel_hi - a.rel_lo);
    const int lane = threadIdx.x & 31;
    const int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int u = 0, c0 = 0;
    const unsigned m = w < nitems ? item_mask<PASS, RTN>(a, w, units, nct, u, c0) : 0u;
    const unsigned on = __ballot_sync(FULL, m != 0);
    int base = 0;
    if (lane == 0 && on) base = atomicAdd(a.nlist, __popc(on));
    base = __shfl_sync(FULL, base, 0);
    if (m) a.items[base + __popc(on & db::lanemask_lt())] = make_int4(u, c0, (int)m, 0);
}

template <int PASS, bool BF16>
__global__ void __launch_bounds__(Shape<PASS, BF16>::THREADS, 1) tc_pass_kernel(TcArgs a) {
    using Sh = Shape<PASS, BF16>;
    constexpr int EPI_WARPS = Sh::EPI, RTN = Sh::RTN, GW = Sh::GW;
    constexpr int TMU = TM * RTN;                       // rows of a unit
    constexpr int TILE_WARPS = EPI_WARPS / RTN;         // epilogue warps that read one MMA tile
    constexpr int WPQ = TILE_WARPS / 4;                 // warps per lane quadrant on one MMA tile
    constexpr int NG = (TN / WPQ) / GW;                 // groups per epilogue warp and tile
    constexpr int DONE_ALL = (1 << EPI_WARPS) - 1;
    constexpr bool FOLDABLE = PASS == TC_COUNT && !BF16;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    // Align by pointer arithmetic on the shared array (not through an integer),
    // so the compiler keeps shared-space loads, stores and atomics.
    const uint32_t pad = (1024u - (smem_u32(smem_raw) & 1023u)) & 1023u;
    using Smem = typename TcSmem<PASS, BF16>::type;
    constexpr int NSTAGE = Smem::NSTAGE, NMETA = Smem::NMETA, NA = Smem::NABUF;
    Smem &S = *reinterpret_cast<Smem *>(smem_raw + pad);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int units = (a.nR + TMU - 1) / TMU, nct = (a.nC + TN - 1) / TN;
    const int64_t nitems = tcitems::count(units, a.rel_hi - a.rel_lo);

    volatile int *abort_flag = &S.abort_flag;
    if (threadIdx.x == 0) {
        for (int i = 0; i < NA; ++i) {
            mbar_init(&S.a_full[i], 1);
            mbar_init(&S.a_empty[i], 1 + EPI_WARPS);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&S.t_full[i], 1);
            mbar_init(&S.t_empty[i], TILE_WARPS);
        }
        for (int i = 0; i < NSTAGE; ++i) {
            mbar_init(&S.b_full[i], 1);
            mbar_init(&S.b_empty[i], 1);  // the MMA commit of the tile
        }
        for (int i = 0; i < NMETA; ++i) {
            mbar_init(&S.m_full[i], 1);
            mbar_init(&S.m_empty[i], 1 + EPI_WARPS);
        }
        mbar_init(&S.drain, 1);
        S.abort_flag = 0;
        S.drain_failed = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if constexpr (FOLDABLE) {
        // every row's folded chunk, in the operand layout: entries 1, 2^11, 2^15, zeros
        for (int e = threadIdx.x; e < TM * 16; e += blockDim.x) {
            const int k = (e & 7) + ((e >> 6) & 1) * 8;
            S.ones[e] = k == 0 ? 0x3C00 : (k == 1 ? 0x6800 : (k == 2 ? 0x7800 : 0));
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        tmem_alloc(&S.tmem_base, 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    db::wait_prior_grid();  // started as a programmatic dependent
    db::allow_next_grid();
    const uint32_t tmem = S.tmem_base;
    const int K = a.K;
    const int KG = a.kv / 8;
    // FP16 count: the column term folded into the MMA when the input's norms
    // keep it exact (3 max|v|^2 + 1 <= 2^25, see the header).
    bool fold = false;
    if constexpr (FOLDABLE) fold = a.fold && 3ll * (long long)*a.bmax_ptr + 1 <= (1ll << 25);
    const uint32_t a_bytes = (uint32_t)(TM * a.kv * 2), bv_bytes = 2 * a_bytes;
    const uint32_t b_bytes = bv_bytes + (fold ? TN * 16 * 2 : 0);

    long long w_prod = 0, w_mma_b = 0, w_mma_t = 0, w_epi = 0, t_start = clock64();
    (void)w_prod, (void)w_mma_b, (void)w_mma_t, (void)w_epi, (void)t_start;
    if (warp == 0) {
        // ---------------- producer ----------------
        int ia = 0, tb = 0, te = 0;  // items, column tiles and events so far
        bool ok = true;
        // One item: unit iu, the column tiles ic + (bits of m).  done: what the
        // unit's udone word was a little earlier.
        auto run = [&](int iu, int ic, unsigned m, int done) {
            const int itile = RTN == 2 ? iu : iu >> 1;
            if (PASS == TC_COUNT && a.min_pts > 0 && done == DONE_ALL) return;
            if (PASS == TC_UNION) {
                // two tiles, each of one set: skipped when the sets are one by now
                const int ti = a.tag[itile];
                if (ti >= 0) {
                    const int tj = ((m >> lane) & 1u) ? a.tag[ic + lane] : -1;
                    const bool same = tj >= 0 && db::uf_find(a.parent, ti) == db::uf_find(a.parent, tj);
                    m &= ~__ballot_sync(FULL, same);
                }
                if (!m) return;
            }
            const int ab = ia % NA;
            if (!(ok = mbar_wait_warp(&S.a_empty[ab], ((ia / NA) & 1) ^ 1, abort_flag, a.wait_ns))) return;
            if (elect_one()) {
                S.unit[ab] = iu;
                S.done[ab] = 0;
                const uint16_t *src = a.opR + (size_t)itile * a.tile_r + (RTN == 1 ? (iu & 1) * (TM * a.kv) : 0);
                mbar_arrive_expect_tx(&S.a_full[ab], RTN * a_bytes + (uint32_t)sizeof(MetaTile));
                bulk_g2s(S.A[ab * RTN], src, RTN * a_bytes, &S.a_full[ab]);
                bulk_g2s(&S.metaA[ab], a.metaR + itile, (uint32_t)sizeof(MetaTile), &S.a_full[ab]);
            }
            __syncwarp();
            ++ia;
            while (m) {
                const int ct = ic + __ffs(m) - 1;
                m &= m - 1;
                // (one lane's reading decides for the warp: epilogue warps write it)
                if (PASS == TC_COUNT && a.min_pts > 0 &&
                    __shfl_sync(FULL, *(volatile int *)&S.done[ab], 0) == DONE_ALL)
                    break;
                const int s = tb % NSTAGE, me = te % NMETA;
                if (!(ok = TC_WAIT(w_prod, mbar_wait_warp(&S.b_empty[s], ((tb / NSTAGE) & 1) ^ 1, abort_flag, a.wait_ns) &&
                           mbar_wait_warp(&S.m_empty[me], ((te / NMETA) & 1) ^ 1, abort_flag, a.wait_ns))))
                    return;
                if (elect_one()) {
                    S.ev[me] = ct;
                    mbar_arrive_expect_tx(&S.m_full[me], (uint32_t)sizeof(MetaTile));
                    bulk_g2s(&S.metaB[me], a.metaC + ct, (uint32_t)sizeof(MetaTile), &S.m_full[me]);
                    mbar_arrive_expect_tx(&S.b_full[s], b_bytes);
                    bulk_g2s(S.B[s], a.opC + (size_t)ct * a.tile_c, b_bytes, &S.b_full[s]);
                }
                __syncwarp();
                ++tb;
                ++te;
            }
            const int me = te % NMETA;
            if (!(ok = mbar_wait_warp(&S.m_empty[me], ((te / NMETA) & 1) ^ 1, abort_flag, a.wait_ns))) return;
            if (elect_one()) {
                S.ev[me] = EV_END;
                mbar_arrive(&S.m_full[me]);
            }
            __syncwarp();
            ++te;
        };
        // A unit's udone word, one lane's reading for the warp (other CTAs write it).
        auto done_of = [&](int iu) {
            return PASS == TC_COUNT && a.min_pts > 0 ? __shfl_sync(FULL, db::ld_relaxed(a.udone + iu), 0) : 0;
        };
        if (a.items) {
            // from the list, one at a time: the claim, the entry and the unit's
            // state are each fetched an item ahead of their use
            const int nlist = *a.nlist;
            auto claim = [&]() {
                int t = 0;
                if (lane == 0) t = atomicAdd(a.ticket, 1);
                return __shfl_sync(FULL, t, 0);
            };
            auto entry = [&](int t) { return t < nlist ? a.items[t] : make_int4(-1, 0, 0, 0); };
            int4 e0 = entry(claim()), e1 = entry(claim());
            int t2 = claim(), d0 = e0.x >= 0 ? done_of(e0.x) : 0;
            while (e0.x >= 0 && ok) {
                const int d1 = e1.x >= 0 ? done_of(e1.x) : 0;
                const int4 e2 = entry(t2);
                t2 = claim();
                run(e0.x, e0.y, (unsigned)e0.z, d0);
                e0 = e1;
                d0 = d1;
                e1 = e2;
            }
        } else {
            for (int64_t base = blockIdx.x; base < nitems && ok; base += tcitems::round((int)gridDim.x)) {
                const int64_t w = tcitems::dealt(base, lane, (int)gridDim.x);
                int u = 0, c0 = 0;
                unsigned mask = 0;
                if (w < nitems) mask = item_mask<PASS, RTN>(a, w, units, nct, u, c0);
                unsigned live = __ballot_sync(FULL, mask != 0);
                while (live && ok) {
                    const int l = __ffs(live) - 1;
                    live &= live - 1;
                    const int iu = __shfl_sync(FULL, u, l), ic = __shfl_sync(FULL, c0, l);
                    const unsigned m = __shfl_sync(FULL, mask, l);
                    run(iu, ic, m, done_of(iu));
                }
            }
        }
        if (ok) {
            const int me = te % NMETA;
            ok = mbar_wait_warp(&S.m_empty[me], ((te / NMETA) & 1) ^ 1, abort_flag, a.wait_ns);
            if (ok && elect_one()) {
                S.ev[me] = EV_STOP;
                mbar_arrive(&S.m_full[me]);
            }
        }
        // On a clean finish every copy has been consumed, so it has landed.
        // After an abort, wait (bounded) until the last copy into each buffer
        // has landed: a buffer holds at most one copy in flight, so the parity
        // of its last phase identifies it.
        if (!ok) {
            bool fine = true;
            for (int s = 0; s < NSTAGE && s < tb; ++s)
                fine &= mbar_wait_quiet(&S.b_full[s], ((tb - 1 - s) / NSTAGE) & 1, kDrainNs);
            for (int m = 0; m < NMETA && m < te; ++m)
                fine &= mbar_wait_quiet(&S.m_full[m], ((te - 1 - m) / NMETA) & 1, kDrainNs);
            for (int ab = 0; ab < NA && ab < ia; ++ab)
                fine &= mbar_wait_quiet(&S.a_full[ab], ((ia - 1 - ab) / NA) & 1, kDrainNs);
            if (!fine) S.drain_failed = 1;
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer ----------------
        // (test hook a.stall: it issues nothing, so the other roles' bounded
        // waits expire and the CTA takes the abort path with no MMA in flight)
        if (!a.stall && elect_one()) {
            const uint32_t idesc = idesc_f16(BF16);
            int ia = 0, tb = 0, te = 0;
            bool clean = true, in_item = false;
            int row0 = 0;
            unsigned long long evaluated = 0;  // pairs of the tiles multiplied
            while (true) {
                const int me = te % NMETA;
                if (!(clean = TC_WAIT(w_mma_b, mbar_wait(&S.m_full[me], (te / NMETA) & 1, abort_flag, a.wait_ns)))) break;
                const int ev = *(volatile int *)&S.ev[me];
                mbar_arrive(&S.m_empty[me]);
                ++te;
                if (ev == EV_STOP) break;
                const int ab = ia % NA;
                if (ev == EV_END) {
                    mma_commit(&S.a_empty[ab]);
                    ++ia;
                    in_item = false;
                    continue;
                }
                if (!in_item) {
                    if (!(clean = TC_WAIT(w_mma_b, mbar_wait(&S.a_full[ab], (ia / NA) & 1, abort_flag, a.wait_ns)))) break;
                    in_item = true;
                    row0 = *(volatile int *)&S.unit[ab] * TMU;
                }
                const int s = tb % NSTAGE;
                if (!(clean = TC_WAIT(w_mma_b, mbar_wait(&S.b_full[s], (tb / NSTAGE) & 1, abort_flag, a.wait_ns)))) break;
                const uint32_t b_addr = smem_u32(S.B[s]);
#pragma unroll
                for (int r = 0; r < RTN; ++r) {
                    // accumulator buffer and its use count: with two row tiles each
                    // buffer serves one of them on every B tile; otherwise the
                    // buffers alternate between tiles
                    const int b = RTN == 2 ? r : (tb & 1), use = RTN == 2 ? tb : (tb >> 1);
                    if (!(clean = TC_WAIT(w_mma_t, mbar_wait(&S.t_empty[b], (use & 1) ^ 1, abort_flag, a.wait_ns)))) break;
                    tc_fence_after();
                    // the RTN row tiles lie back to back (a_bytes each) from the buffer's start
                    const uint32_t a_addr = smem_u32(S.A[ab * RTN]) + (uint32_t)r * a_bytes;
                    // FP16: sum over K of v_p v_q.  BF16: hi.hi + hi.lo + lo.hi, the
                    // lo columns K/16 chunks after the hi ones (256 B per chunk).
                    const int kch = K / 16;
                    for (int kk = 0; kk < kch; ++kk) {
                        const uint64_t ad = smem_desc(a_addr + kk * 256, KG * 128);
                        const uint64_t bd = smem_desc(b_addr + kk * 256, KG * 128);
                        mma_f16(tmem + (uint32_t)(b * TN), ad, bd, idesc, kk > 0 ? 1u : 0u);
                        if (BF16) {
                            const uint64_t bl = smem_desc(b_addr + (kch + kk) * 256, KG * 128);
                            const uint64_t al = smem_desc(a_addr + (kch + kk) * 256, KG * 128);
                            mma_f16(tmem + (uint32_t)(b * TN), ad, bl, idesc, 1u);
                            mma_f16(tmem + (uint32_t)(b * TN), al, bd, idesc, 1u);
                        }
                    }
                    if (FOLDABLE && fold)  // the folded chunk follows the tile's v columns
                        mma_f16(tmem + (uint32_t)(b * TN), smem_desc(smem_u32(S.ones), 256),
                                smem_desc(b_addr + bv_bytes, 256), idesc, 1u);
                    mma_commit(&S.t_full[b]);  // accumulator ready for the epilogue
                    evaluated += (unsigned long long)max(0, min(TM, a.nR - row0 - r * TM)) * min(TN, a.nC - ev * TN);
                }
                if (!clean) break;
                mma_commit(&S.b_empty[s]);  // operands of this stage consumed
                ++tb;
            }
            // Wait for the arrivals of the last commits, so that none lands after
            // the CTA has exited.
            if (clean && !*abort_flag) {
                for (int s = 0; s < NSTAGE && s < tb; ++s)
                    mbar_wait(&S.b_empty[s], ((tb - 1 - s) / NSTAGE) & 1, abort_flag, a.wait_ns);
                for (int ab = 0; ab < NA && ab < ia; ++ab)
                    mbar_wait(&S.a_empty[ab], ((ia - 1 - ab) / NA) & 1, abort_flag, a.wait_ns);
            }
            if ((PASS == TC_COUNT || PASS == TC_UNION || PASS == TC_BORDER || PASS == TC_ADJ) && evaluated)
                atomicAdd(a.ctr + DB_CTR_EVAL + (PASS == TC_ADJ ? TC_UNION : PASS), evaluated);
            if (FOLDABLE && fold && blockIdx.x == 0) a.ctr[DB_CTR_TC_FOLD] = 1ull;
            // After an abort: one more commit, which arrives once every MMA this
            // thread issued has completed, and a bounded wait for it.
            if (*abort_flag && tb + te > 0) {
                mma_commit(&S.drain);
                if (!mbar_wait_quiet(&S.drain, 0, kDrainNs)) S.drain_failed = 1;
            }
        }
    } else {
        // ---------------- epilogue ----------------
        const int ew = warp - 2;                  // 0..EPI_WARPS-1
        const int quad = warp & 3;                // TMEM lane quadrant this warp may access
        const int rsel = RTN == 2 ? ew / TILE_WARPS : 0;     // row tile of the unit this warp serves
        const int colbase = ((ew >> 2) % WPQ) * (TN / WPQ);  // first column of this warp in the tile
        const int r = quad * 32 + lane;           // row within the row tile
        const uint32_t lane_base = (uint32_t)(quad * 32) << 16;
        const float rho2 = BF16 ? bf16_rho(K) * bf16_rho(K) : 0.f;
        (void)rho2;
        int ia = 0, tb = 0, te = 0;
        bool fresh = true;  // the next event begins an item
        unsigned long long band_cnt = 0, bad_cnt = 0;
        unsigned maxerr = 0;
        int p = 0, rbase = 0;  // position of this row, first position of the warp's rows
        bool row_ok = false;
        float beta_p = 0.f, alpha = 0.f, c_even = 0.f, c_odd = 0.f;
        int cnt = 0, prior = 0, bmin = INT_MAX, rootp = -2;
        bool told = false;           // count: this warp's rows are all done and the producer knows
        bool first = true;           // count: no tile of the item seen (its prior counts are still on their way)
        unsigned best = 0;           // order: least squared distance so far (bits, column in the low 8)
        int besti = 0;               // and its pivot
        float reach = 0.f;           // cull: (r + eps)^2, an overestimate
        while (true) {
            const int me = te % NMETA;
            if (!TC_WAIT(w_epi, mbar_wait_warp(&S.m_full[me], (te / NMETA) & 1, abort_flag, a.wait_ns))) break;
            const int ev = *(volatile int *)&S.ev[me];
            ++te;
            if (ev == EV_STOP) break;
            const int ab = ia % NA;
            if (fresh) {
                fresh = false;
                if (!mbar_wait_warp(&S.a_full[ab], (ia / NA) & 1, abort_flag, a.wait_ns)) break;
                const int u = *(volatile int *)&S.unit[ab];
                rbase = u * TMU + rsel * TM + quad * 32;
                p = rbase + lane;
                row_ok = p < a.nR;
                const int rin = RTN == 2 ? rsel * TM + r : (u & 1) * TM + r;  // row within its tile
                if (PASS == TC_CULL) {
                    beta_p = row_ok ? a.cbeta[p] : 0.f;
                    // m > r + eps with m^2 = beta_p + w: everything rounded towards keeping the pair
                    // (radius -1: an empty ball, near nothing)
                    const float r2 = row_ok ? a.crad[p] : -1.f;
                    const float rr = (sqrtf(fmaxf(r2, 0.f)) + sqrtf((float)a.T)) * 1.000001f;
                    reach = r2 < 0.f ? -3.0e38f : rr * rr * 1.000001f + 8.f;
                } else {
                    beta_p = S.metaA[ab].beta[rin];
                }
                if (PASS == TC_LINK) reach = 4.f * (float)a.T;  // twice eps
                alpha = beta_p - (float)a.T;  // |v_p|^2 - T, exact (1e30 for a masked row: never passes)
                if (PASS == TC_COUNT && !BF16) {
                    // folded form: 1 - thr_f for the even (f = 0) and odd (f = 1)
                    // columns, thr_f = ceil((|v_p|^2 - T - f) / 2) = (a_p - f + 1) >> 1
                    const int a_p = row_ok ? (int)beta_p - a.T : 0;
                    c_even = (float)(1 - ((a_p + 1) >> 1));
                    c_odd = (float)(1 - (a_p >> 1));
                }
                cnt = 0;
                if (PASS == TC_COUNT && a.min_pts > 0) {
                    prior = row_ok ? db::ld_relaxed(a.count + p) : a.min_pts;
                    told = false;
                    first = true;
                }
                bmin = INT_MAX;
                // union: a member of p's set (its parent, then the last root seen)
                if (PASS == TC_UNION) rootp = (row_ok && beta_p < 1e29f) ? db::ld_relaxed(a.parent + p) : -2;
                best = 0xffffffffu;
                besti = 0;
            }
            if (ev == EV_END) {
                if (row_ok) {
                    if ((PASS == TC_COUNT || PASS == TC_VERIFY) && cnt) atomicAdd(a.count + p, cnt);
                    if (PASS == TC_BORDER && bmin != INT_MAX) atomicMin(a.border + p, bmin);
                    // (a pivot is within reach of itself, unless rounding says otherwise)
                    if (PASS == TC_LINK) a.key[p] = (int)min(best, (unsigned)p);
                    if (PASS == TC_ORDER) {
                        // class: the ratio of the squared distance to T, in powers of 4
                        const float ratio = __uint_as_float(best & 0x7fffff00u) / (float)max(a.T, 1);
                        int cl = 0;
                        for (float lim = 4.f; cl < 7 && ratio > lim; lim *= 4.f) ++cl;
                        const int key = cl * a.n_piv + a.prank[besti];
                        a.key[p] = key;
                        a.rank[p] = atomicAdd(a.hist + key, 1);
                    }
                }
                if (PASS == TC_COUNT && a.min_pts > 0 && __all_sync(FULL, prior + cnt >= a.min_pts) && lane == 0)
                    atomicOr(a.udone + *(volatile int *)&S.unit[ab], 1 << ew);
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(&S.a_empty[ab]);
                    mbar_arrive(&S.m_empty[me]);
                }
                ++ia;
                fresh = true;
                continue;
            }
            const int ct = ev;
            const int b = RTN == 2 ? rsel : (tb & 1), use = RTN == 2 ? tb : (tb >> 1);
            ++tb;
            if (!TC_WAIT(w_epi, mbar_wait_warp(&S.t_full[b], use & 1, abort_flag, a.wait_ns))) break;
            tc_fence_after();
            const MetaTile &mc = S.metaB[me];
            const uint32_t tb_addr = tmem + lane_base + (uint32_t)(b * TN);
            if constexpr (Sh::kWide) {
                // all 256 columns in four groups of 64: the next group's TMEM load is
                // in flight while this group is decided, and the accumulator goes
                // back to the issuer before the last group is (groups of 32, given
                // back at the end: 385 instead of 353 us for the count of
                // 200,000 x 64, its warps waiting on tensor memory)
                uint32_t ga[64], gb[64];
                auto all_groups = [&](auto &&decide) {
                    tmem_ld64_nowait(tb_addr, ga);
                    tmem_wait_ld_dep64(ga);
#pragma unroll 1
                    for (int h = 0; h < 2; ++h) {
                        tmem_ld64_nowait(tb_addr + (uint32_t)(128 * h + 64), gb);
                        decide(ga, 128 * h);
                        tmem_wait_ld_dep64(gb);
                        if (h == 0) {
                            tmem_ld64_nowait(tb_addr + 128, ga);
                        } else {
                            tc_fence_before();
                            __syncwarp();
                            if (lane == 0) mbar_arrive(&S.t_empty[b]);
                        }
                        decide(gb, 128 * h + 64);
                        if (h == 0) tmem_wait_ld_dep64(ga);
                    }
                };
                if constexpr (PASS == TC_COUNT) {
                    unsigned long long acc[4] = {0ull, 0ull, 0ull, 0ull};  // +0.0f in both halves
                    if (fold) {
                        // Folded form: the accumulator holds G - h_q exactly, with
                        // h_q = ceil(|v_q|^2 / 2) (see the header).  D <= T iff
                        // G - h_q >= thr_f = ceil((|v_p|^2 - T - f) / 2), so
                        // sat(acc + 1 - thr_f) is exactly 1 for a neighbour and 0
                        // otherwise: one saturating add per pair, one packed add per
                        // two pairs, no column data.  f = 0 for the first n_even columns.
                        const int ne = mc.n_even;
                        all_groups([&](uint32_t(&g)[64], int col) {
                            if (ne >= col + 64 || ne <= col) {
                                const float cf = ne <= col ? c_odd : c_even;
#pragma unroll
                                for (int h = 0; h < 32; ++h)
                                    acc[h & 3] =
                                        f2_add(acc[h & 3], f2_pack(__saturatef(__uint_as_float(g[2 * h]) + cf),
                                                                   __saturatef(__uint_as_float(g[2 * h + 1]) + cf)));
                            } else {  // the one group with columns of both parities
                                const int bd = ne - col;
#pragma unroll
                                for (int h = 0; h < 32; ++h)
                                    acc[h & 3] = f2_add(
                                        acc[h & 3],
                                        f2_pack(__saturatef(__uint_as_float(g[2 * h]) + (2 * h < bd ? c_even : c_odd)),
                                                __saturatef(__uint_as_float(g[2 * h + 1]) +
                                                            (2 * h + 1 < bd ? c_even : c_odd))));
                            }
                        });
                    } else {
                        // G alone (exact), so sat(2G - |v_q|^2 + 1 - alpha) is exactly
                        // 1 for a neighbour (T - D + 1 >= 1) and 0 otherwise.  Two
                        // pairs per packed FFMA (w' = |v_q|^2 - 2G, the exact negation
                        // of fma(2, G, -|v_q|^2): round-to-nearest is symmetric), one
                        // saturating subtract per pair (c1 - w' = c1 + w, the same
                        // rounding as before) and one packed add per two pairs.
                        const float c1 = 1.f - alpha;
                        const unsigned long long m2 = f2_pack(-2.f, -2.f);
                        all_groups([&](uint32_t(&g)[64], int col) {
                            const float *bet = mc.beta + col;
#pragma unroll
                            for (int j8 = 0; j8 < 8; ++j8) {
                                const float4 ba = *reinterpret_cast<const float4 *>(bet + 8 * j8);
                                const float4 bb = *reinterpret_cast<const float4 *>(bet + 8 * j8 + 4);
                                const float bq[8] = {ba.x, ba.y, ba.z, ba.w, bb.x, bb.y, bb.z, bb.w};
#pragma unroll
                                for (int h = 0; h < 4; ++h) {
                                    const unsigned long long w = f2_fma(
                                        f2_pack(__uint_as_float(g[8 * j8 + 2 * h]), __uint_as_float(g[8 * j8 + 2 * h + 1])),
                                        m2, f2_pack(bq[2 * h], bq[2 * h + 1]));
                                    float w0, w1;
                                    f2_unpack(w, w0, w1);
                                    acc[h] = f2_add(acc[h], f2_pack(__saturatef(c1 - w0), __saturatef(c1 - w1)));
                                }
                            }
                        });
                    }
                    float sm[8];
#pragma unroll
                    for (int h = 0; h < 4; ++h) f2_unpack(acc[h], sm[2 * h], sm[2 * h + 1]);
                    if (row_ok) cnt += (int)(((sm[0] + sm[1]) + (sm[2] + sm[3])) + ((sm[4] + sm[5]) + (sm[6] + sm[7])));
                } else {
                    const unsigned long long m2 = f2_pack(-2.f, -2.f), bp = f2_pack(beta_p, beta_p);
                    float lo = 3.0e38f;
                    unsigned least = 0xffffffffu;
                    all_groups([&](uint32_t(&g)[64], int col) {
#pragma unroll
                        for (int j4 = 0; j4 < 16; ++j4) {
                            const float4 b4 = *reinterpret_cast<const float4 *>(mc.beta + col + 4 * j4);
                            unsigned long long q01 = f2_pack(b4.x, b4.y), q23 = f2_pack(b4.z, b4.w);
                            if (PASS != TC_CULL) {
                                q01 = f2_add(q01, bp);
                                q23 = f2_add(q23, bp);
                            }
                            float w[4];
                            f2_unpack(f2_fma(f2_pack(__uint_as_float(g[4 * j4]), __uint_as_float(g[4 * j4 + 1])), m2,
                                             q01), w[0], w[1]);
                            f2_unpack(f2_fma(f2_pack(__uint_as_float(g[4 * j4 + 2]), __uint_as_float(g[4 * j4 + 3])),
                                             m2, q23), w[2], w[3]);
                            if (PASS == TC_LINK) {
#pragma unroll
                                for (int h = 0; h < 4; ++h)
                                    if (w[h] <= reach) least = min(least, (unsigned)(ct * TN + col + 4 * j4 + h));
                            } else if (PASS == TC_ORDER) {
                                // squared distances (>= 0, so they order as integers) with
                                // the column in the low 8 bits: the nearest pivot up to 2^-15
                                // of its distance, which is all a sort key needs
                                unsigned k[4];
#pragma unroll
                                for (int h = 0; h < 4; ++h)
                                    k[h] = (__float_as_uint(w[h]) & 0x7fffff00u) | (unsigned)(col + 4 * j4 + h);
                                least = __vimin3_u32(__vimin3_u32(least, k[0], k[1]), k[2], k[3]);
                            } else {
                                lo = fminf(fminf(lo, fminf(w[0], w[1])), fminf(w[2], w[3]));
                            }
                        }
                    });
                    if (PASS == TC_LINK) best = min(best, least);
                    if (PASS == TC_ORDER && least < best) {
                        best = least;
                        besti = ct * TN + (int)(least & 255u);
                    }
                    if (PASS == TC_CULL) {
                        // two balls per tile: a tile is near when either is
                        unsigned m = __ballot_sync(FULL, row_ok && beta_p + lo <= reach);
                        m = (m | (m >> 1)) & 0x55555555u;
                        m = (m | (m >> 1)) & 0x33333333u;
                        m = (m | (m >> 2)) & 0x0f0f0f0fu;
                        m = (m | (m >> 4)) & 0x00ff00ffu;
                        m = (m | (m >> 8)) & 0x0000ffffu;
                        if (lane == 0 && rbase < a.nR)
                            reinterpret_cast<uint16_t *>(a.near + (size_t)ct * a.words)[rbase >> 5] = (uint16_t)m;
                    }
                }
            } else {
                int *colroot = S.colroot + (PASS == TC_UNION ? b * TN : 0);
                bool hints = false;  // union: colroot filled for this tile
                // union: the parents of this warp's GW * NG column points of the
                // tile, loaded now so that their latency hides behind the
                // accumulator loads and scores
                int pr[NG];
                if (PASS == TC_UNION) {
#pragma unroll
                    for (int k = 0; k < NG; ++k) {
                        const int q = ct * TN + colbase + lane + GW * k;
                        pr[k] = q < a.nC ? db::ld_relaxed(a.parent + q) : -1;
                    }
                }
                int hm0 = -3, hm1 = -3;  // union: hints already merged with p's set
#pragma unroll 1
                for (int hc = 0; hc < NG; ++hc) {
                    const int cb = colbase + hc * GW;  // column within the tile
                    uint32_t g[GW];
                    const uint32_t taddr = tb_addr + (uint32_t)cb;
                    tmem_ld32_nowait(taddr, g);
                    if constexpr (GW >= 64) tmem_ld32_nowait(taddr + 32, g + 32);
                    tmem_wait_ld();
                    if (PASS == TC_VERIFY) {
                        if (!row_ok) continue;
#pragma unroll 1
                        for (int j = 0; j < GW; ++j) {
                            const int q = ct * TN + cb + j;
                            if (q >= a.nC) continue;
                            const float gv = __uint_as_float(g[j & (GW - 1)]);
                            const float wv = fmaf(2.f, gv, -mc.beta[cb + j]);
                            const int D = exact_sqdist(a.v16, K, p, q);
                            // 2G exactly, from integers: |v_p|^2 + |v_q|^2 - D (the betas are exact)
                            const long long two_g = (long long)beta_p + (long long)mc.beta[cb + j] - D;
                            const double err = fabs(2.0 * (double)gv - (double)two_g);
                            maxerr = max(maxerr, (unsigned)fmin(err, 4.0e9));
                            const bool nb_exact = D <= a.T;
                            const float del = BF16 ? rho2 : (float)FP16_BAND;
                            const bool in_band = fabsf(wv - alpha) <= del;
                            band_cnt += in_band;
                            if (!in_band && ((wv >= alpha) != nb_exact)) ++bad_cnt;
                            cnt += nb_exact;
                        }
                        continue;
                    }
                    // One FFMA per pair; the maxima of the eight strided column
                    // groups (j mod 8) come from the first three levels of an FMNMX
                    // tree.  Only groups whose maximum can reach the threshold are
                    // rescanned.
                    // Candidate score per pair: 2G - beta_f, computed as the exact
                    // negation beta_f - 2G two pairs per packed FFMA (round-to-nearest
                    // is symmetric), minus its minimum.  FP16: beta_f = |v_q|^2.
                    // BF16: beta_f = |v_q|^2 - rho^2 (rho is the same for every point),
                    // so the score is the rare path's 2G - |v_q|^2 + rho^2 up to a few
                    // units of rounding (at most 2 per rounding at magnitudes below
                    // 2^25, two roundings on each side); the threshold is lowered by
                    // kBf16FilterSlack to cover them, and the rare path decides.
                    const float thr = BF16 ? alpha - kBf16FilterSlack : alpha - (float)FP16_BAND;
                    float mx;
                    float nv[GW];  // after the tree, nv[i] = minimum over the columns j = i (mod 8)
                    {
                        const unsigned long long m2 = f2_pack(-2.f, -2.f);
#pragma unroll
                        for (int j4 = 0; j4 < GW / 4; ++j4) {
                            const float4 b4 = *reinterpret_cast<const float4 *>(&mc.beta_f[cb + 4 * j4]);
                            const unsigned long long w01 =
                                f2_fma(f2_pack(__uint_as_float(g[4 * j4 + 0]), __uint_as_float(g[4 * j4 + 1])), m2,
                                       f2_pack(b4.x, b4.y));
                            const unsigned long long w23 =
                                f2_fma(f2_pack(__uint_as_float(g[4 * j4 + 2]), __uint_as_float(g[4 * j4 + 3])), m2,
                                       f2_pack(b4.z, b4.w));
                            f2_unpack(w01, nv[4 * j4 + 0], nv[4 * j4 + 1]);
                            f2_unpack(w23, nv[4 * j4 + 2], nv[4 * j4 + 3]);
                        }
#pragma unroll
                        for (int w2 = GW / 2; w2 >= 8; w2 >>= 1)
#pragma unroll
                            for (int j = 0; j < w2; ++j) nv[j] = fminf(nv[j], nv[j + w2]);
                        mx = -fminf(fminf(fminf(nv[0], nv[1]), fminf(nv[2], nv[3])),
                                    fminf(fminf(nv[4], nv[5]), fminf(nv[6], nv[7])));
                    }
                    const bool need = row_ok && mx >= thr;
                    if (!__any_sync(FULL, need)) {
                        if (PASS == TC_ADJ && row_ok) a.adj[(size_t)p * 8 + (cb >> 5)] = 0u;
                        continue;
                    }
                    if (PASS == TC_UNION && !hints) {
                        // the parents loaded at the tile's start, for this warp's columns
                        // (the warps of the other lane quadrants that share them write
                        // them too: any value is a member of the column point's set)
#pragma unroll
                        for (int k = 0; k < NG; ++k) colroot[colbase + lane + GW * k] = pr[k];
                        __syncwarp();
                        hints = true;
                    }
                    // Rare path: the lanes that need it build the mask of
                    // possible neighbours (for FP16 exactly the neighbours; masked
                    // columns never pass, their beta is 1e30).  The merge pass also
                    // drops the columns whose set hint equals the row's: those pairs
                    // need no union.
                    // Only the residues j mod 8 whose minimum passes the filter in
                    // some lane of the warp are scanned (warp-uniform branches, so the
                    // column indices stay compile-time constants).
                    unsigned mask = 0;  // possible neighbours
                    unsigned sure = 0;  // BF16: those beyond the rounding band, neighbours without a recheck
                    {
                        unsigned rm = 0;
                        if (need) {
#pragma unroll
                            for (int i = 0; i < 8; ++i) rm |= (unsigned)(-nv[i] >= thr) << i;
                        }
                        const unsigned um = __reduce_or_sync(FULL, rm);
                        const int col_lim = PASS == TC_UNION ? p - ct * TN : -1;  // merge: columns after the row
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            if (!((um >> i) & 1u)) continue;
#pragma unroll
                            for (int u = 0; u < GW / 8; ++u) {
                                const int j = i + 8 * u;
                                const float w1 = fmaf(2.f, __uint_as_float(g[j]), -mc.beta[cb + j]);
                                bool c = need && (BF16 ? (w1 + rho2 >= alpha) : (w1 >= alpha));
                                if (PASS == TC_UNION) c = c && colroot[cb + j] != rootp;
                                c = c && (cb + j) > col_lim;
                                mask |= (unsigned)c << j;
                                if (BF16) sure |= (unsigned)(c && w1 - rho2 >= alpha) << j;
                            }
                        }
                    }
                    unsigned nbm = BF16 ? sure : mask;  // confirmed neighbours among the mask
                    if (BF16)
                        for (unsigned mm = mask & ~sure; mm; mm &= mm - 1) {
                            const int j = __ffs((int)mm) - 1;
                            ++band_cnt;
                            nbm |= (unsigned)(exact_sqdist(a.v16, K, p, ct * TN + cb + j) <= a.T) << j;
                        }
                    if (PASS == TC_COUNT) cnt += __popc(nbm);
                    if (PASS == TC_ADJ && row_ok) a.adj[(size_t)p * 8 + (cb >> 5)] = nbm;
                    if (PASS == TC_BORDER)
                        for (unsigned mm = nbm; mm; mm &= mm - 1) bmin = min(bmin, mc.idx[cb + __ffs((int)mm) - 1]);
                    if (PASS == TC_UNION) {
                        // Skip a neighbour whose set p is known to be in: colroot[j]
                        // holds a member of column j's set (its parent, or the root
                        // of a later union), rootp a member of p's, hm0 and hm1 members
                        // that p's set has been merged with.  Equal members mean one
                        // set, so only pairs from different-looking sets reach the
                        // atomics.  After a union both endpoints point straight at the
                        // returned root (a valid ancestor; never written on the root
                        // itself, whose link another thread may have set), so later
                        // tiles find the forest flat and a converged cluster costs one
                        // shared-memory compare per pair.
                        // Lanes that would join the same two sets leave it to one of
                        // them: a tile pair of two groups is one union a warp.
                        unsigned left = nbm;
                        while (true) {
                            int j = -1, hq = 0;
                            while (left) {
                                const int k = cb + __ffs((int)left) - 1;
                                left &= left - 1;
                                hq = colroot[k];
                                if (hq == rootp || hq == hm0 || hq == hm1) continue;
                                j = k;
                                break;
                            }
                            if (!__any_sync(FULL, j >= 0)) break;
                            const unsigned long long key =
                                j >= 0 ? ((unsigned long long)(unsigned)rootp << 32) | (unsigned)hq : ~(unsigned long long)lane;
                            const int leader = __ffs((int)__match_any_sync(FULL, key)) - 1;
                            int rt = 0;
                            if (j >= 0 && lane == leader) {
                                const int q = ct * TN + j;
                                rt = unite_sets(a.parent, rootp, hq, a.status);
                                if (q != rt) db::st_relaxed(a.parent + q, rt);
                                if (p != rt && rt != rootp) db::st_relaxed(a.parent + p, rt);
                            }
                            rt = __shfl_sync(FULL, rt, leader);
                            if (j >= 0) {
                                hm0 = hq;
                                if (rt != rootp) hm1 = rootp;
                                rootp = rt;
                                colroot[j] = rt;
                            }
                        }
                    }
                }
            }
            if (!Sh::kWide) tc_fence_before();
            if (PASS == TC_COUNT && a.min_pts > 0 && !told) {
                if (!first && __all_sync(FULL, prior + cnt >= a.min_pts)) {
                    told = true;
                    if (lane == 0) atomicOr(&S.done[ab], 1 << ew);
                }
                first = false;
            }
            __syncwarp();
            if (lane == 0) {
                if (!Sh::kWide) mbar_arrive(&S.t_empty[b]);
                mbar_arrive(&S.m_empty[me]);
            }
        }
        if (band_cnt) atomicAdd(a.ctr + 6, band_cnt);
        if (bad_cnt) atomicAdd(a.ctr + 7, bad_cnt);
        if (maxerr) atomicMax(a.ctr + 8, (unsigned long long)maxerr);
    }

#ifdef DB_TC_WAIT_STATS
    // slots 9..13 (count), 20..24 (merge), 25..29 (border): producer, MMA issuer
    // on events and operands, MMA issuer on accumulators, one epilogue warp,
    // issuer total
    if (PASS == TC_COUNT || PASS == TC_UNION || PASS == TC_BORDER) {
        unsigned long long *ws = a.ctr + (PASS == TC_COUNT ? 9 : (PASS == TC_UNION ? 20 : 25));
        if (threadIdx.x == 0) atomicAdd(ws, (unsigned long long)w_prod);
        if (warp == 1 && w_mma_b) {
            atomicAdd(ws + 1, (unsigned long long)w_mma_b);
            atomicAdd(ws + 2, (unsigned long long)w_mma_t);
            atomicAdd(ws + 4, (unsigned long long)(clock64() - t_start));
        }
        if (threadIdx.x == 64) atomicAdd(ws + 3, (unsigned long long)w_epi);
    }
#endif
    // ---------------- teardown ----------------
    tc_fence_before();
    __syncthreads();
    if (S.abort_flag) {
        if (threadIdx.x == 0) atomicOr(a.status, DB_EBIT_TIMEOUT);
        // The producer has waited (bounded) for the last copy into each buffer
        // and the MMA issuer for a final commit that follows all its MMAs, so
        // nothing of this CTA is in flight.  Only if one of those waits gave up
        // does thread 0 also spin 20 ms before the tensor memory is freed.
        if (threadIdx.x == 0 && S.drain_failed) {
            const uint64_t t0 = globaltimer();
            while (globaltimer() - t0 < 20000000ull) {
            }
        }
        __syncthreads();
    }
    tc_fence_after();
    if (warp == 1) tmem_dealloc(tmem, 512);
}

// ---------------- preparation kernels ----------------

__device__ __forceinline__ uint16_t fp16_bits(int v) {
    __half h = __int2half_rn(v);
    return *reinterpret_cast<uint16_t *>(&h);
}
__device__ __forceinline__ uint16_t bf16_bits_rn(int v) {
    __nv_bfloat16 h = __float2bfloat16_rn((float)v);
    return *reinterpret_cast<uint16_t *>(&h);
}
__device__ __forceinline__ int bf16_value(uint16_t bits) {
    return (int)__uint_as_float((uint32_t)bits << 16);  // an integer for every |v| <= 512
}

// Column side of the folded chunk: the digits of h_q = ceil(|v_q|^2 / 2) =
// q0 + 2^11 q1 + 2^22 q2 (q0, q1 < 2^11), negated, as -q0, -q1, -2^7 q2 (then
// zeros) against the rows' 1, 2^11, 2^15; a padding column takes h = 2^24.
// Every entry is an integer FP16 holds exactly, and the chunk's products sum
// to -h_q, so the MMA accumulates G - h_q.
__device__ __forceinline__ int fold_entry(int kk, bool valid, int nrm_q) {
    const int h = valid ? (nrm_q + 1) >> 1 : (1 << 24);
    return kk == 0 ? -(h & 2047) : (kk == 1 ? -((h >> 11) & 2047) : (kk == 2 ? -((h >> 22) << 7) : 0));
}

struct PackArgs {
    const float *x;
    const int *list;  // point of each position (null: identity)
    int n, d, K;
    int n_src;        // > 0: pack n pivots sampled from n_src points
    int bf16;         // two BF16 terms instead of FP16
    int fold;         // even |v|^2 first within the tile, and the folded chunk
    uint16_t *op;
    MetaTile *meta;
    int *perm;        // point of each position as packed (null: not wanted)
    int *inv;         // position of each point (null)
    int *count;       // zeroed by position (null)
    int *udone;       // zeroed, units_per_tile per tile (null)
    int units_per_tile;
    int16_t *v16;     // centred units by position (null)
    int *bmax;        // largest |v|^2 (null; starts at 0)
    uint16_t *cop;    // packed ball centres (null: no balls)
    float *cbeta, *crad;  // two balls per tile
    unsigned *status;
};

// Pivot k of P: a point of the k-th of P equal index ranges.
__device__ __forceinline__ int pivot_point(int k, int P, int n) {
    const int lo = (int)((long long)n * k / P), hi = (int)((long long)n * (k + 1) / P);
    return lo + (int)(((unsigned)k * 2654435761u) % (unsigned)max(1, hi - lo));
}

// One block of 256 threads packs one tile: 256 positions' rows are checked
// against the grid, centred, staged in shared memory (the rows of a tile are
// scattered when they are taken through a list; each is read coalesced, a warp
// per row) and written in the operand layout with their metadata.  Bound by
// the scattered row reads and the coalesced operand writes: 200,000 x 64 (51 MB
// in, 32 MB out).
__global__ void __launch_bounds__(256) tc_pack_kernel(PackArgs a) {
    db::wait_prior_grid();  // started as a programmatic dependent
    db::allow_next_grid();
    __shared__ int16_t rows[TN][66];  // 33 words a row: column reads by consecutive threads hit different banks
    __shared__ int src_s[TN];         // point of each row as loaded
    __shared__ int nrm_s[TN];
    __shared__ short rowat[TN];       // loaded row of each packed row
    __shared__ int wsum[8], wval[8];
    __shared__ int csum[2][4][64];
    __shared__ int cen[2][64];
    __shared__ unsigned long long far_s[8];
    __shared__ uint8_t part_s[TN];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tile = blockIdx.x, base = tile * TN, K = a.K;
    const int pos = base + tid;
    const bool valid = pos < a.n;
    src_s[tid] = !valid ? -1 : (a.n_src ? pivot_point(pos, a.n, a.n_src) : (a.list ? a.list[pos] : pos));
    __syncthreads();
    bool ok = true;
#pragma unroll 1
    for (int r0 = 0; r0 < 32; r0 += 16) {  // 16 rows of the warp in flight
        float f[16][2];
#pragma unroll
        for (int rr = 0; rr < 16; ++rr) {
            const int src = src_s[warp * 32 + r0 + rr];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int k = lane + 32 * h;
                f[rr][h] = k < a.d && src >= 0 ? a.x[(size_t)src * a.d + k] : 0.5f;
            }
        }
#pragma unroll
        for (int rr = 0; rr < 16; ++rr) {
            const int row = warp * 32 + r0 + rr;
            int s = 0;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                int u;
                ok &= db::on_grid(f[rr][h], u);
                const int v = u - 512;  // 0 for the padding
                if (lane + 32 * h < K) rows[row][lane + 32 * h] = (int16_t)v;
                s += v * v;
            }
            s = __reduce_add_sync(FULL, s);
            if (lane == 0) nrm_s[row] = s;
        }
    }
    if (!__all_sync(FULL, ok) && lane == 0) atomicOr(a.status, DB_EBIT_NOT_QUANTISED);
    __syncthreads();
    const int nrm = nrm_s[tid];
    // packed row of each loaded row: as loaded, or even |v|^2 first, then odd, then padding
    const unsigned ev = __ballot_sync(FULL, valid && !(nrm & 1)), va = __ballot_sync(FULL, valid);
    if (lane == 0) {
        wsum[warp] = __popc(ev);
        wval[warp] = __popc(va);
    }
    __syncthreads();
    int e_before = 0, v_before = 0, n_even = 0;
    for (int w = 0; w < 8; ++w) {
        if (w < warp) {
            e_before += wsum[w];
            v_before += wval[w];
        }
        n_even += wsum[w];
    }
    e_before += __popc(ev & db::lanemask_lt());
    v_before += __popc(va & db::lanemask_lt());
    int to = tid;
    if (a.fold && valid) to = (nrm & 1) ? n_even + (v_before - e_before) : e_before;
    rowat[to] = (short)tid;
    if (a.bmax) {
        const int wmax = __reduce_max_sync(FULL, valid ? nrm : 0);
        if (lane == 0 && wmax > 0) atomicMax(a.bmax, wmax);
    }
    {
        MetaTile &m = a.meta[tile];
        const float beta = valid ? (float)nrm : 1e30f;
        const float rho = bf16_rho(K);
        m.beta[to] = beta;
        m.beta_f[to] = valid && a.bf16 ? (float)nrm - rho * rho : beta;
        m.idx[to] = valid ? src_s[tid] : -1;
        if (tid == 0) m.n_even = n_even;
        if (valid) {
            if (a.perm) a.perm[base + to] = src_s[tid];
            if (a.inv) a.inv[src_s[tid]] = base + to;
            if (a.count) a.count[base + to] = 0;
        }
        if (a.udone && tid < a.units_per_tile) a.udone[tile * a.units_per_tile + tid] = 0;
    }
    __syncthreads();
    // operand: one 16-byte piece (a row's 8 columns) per step, in layout order
    const int KV = a.bf16 ? 2 * K : K, KG = KV / 8;
    uint16_t *op = a.op + (size_t)tile * TN * (KV + (a.fold ? 16 : 0));
    auto store8 = [&](uint16_t *dst, const uint16_t *h) {
        uint4 pk;
        pk.x = h[0] | ((uint32_t)h[1] << 16);
        pk.y = h[2] | ((uint32_t)h[3] << 16);
        pk.z = h[4] | ((uint32_t)h[5] << 16);
        pk.w = h[6] | ((uint32_t)h[7] << 16);
        *reinterpret_cast<uint4 *>(dst) = pk;
    };
    for (int e = tid; e < TN * KG; e += TN) {
        const int ri = e & 7, kg = (e >> 3) % KG, rg = (e >> 3) / KG;
        const int row = rowat[rg * 8 + ri];
        const bool lo = kg >= K / 8;  // BF16: the remainder columns
        const int k0 = (lo ? kg - K / 8 : kg) * 8;
        uint16_t h[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int v = rows[row][k0 + k];
            if (!a.bf16) {
                h[k] = fp16_bits(v);
            } else {
                const uint16_t hi = bf16_bits_rn(v);
                h[k] = lo ? bf16_bits_rn(v - bf16_value(hi)) : hi;  // v - hi is -1, 0 or 1: exact
            }
        }
        store8(op + (size_t)e * 8, h);
    }
    if (a.fold) {
        uint16_t *ch = op + (size_t)TN * KV;
        for (int e = tid; e < TN * 2; e += TN) {
            const int ri = e & 7, kg = (e >> 3) & 1, rg = e >> 4;
            const int row = rowat[rg * 8 + ri];
            uint16_t h[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) h[k] = fp16_bits(fold_entry(kg * 8 + k, base + row < a.n, nrm_s[row]));
            store8(ch + (size_t)e * 8, h);
        }
    }
    if (a.v16)
        for (int e = tid; e < TN * K; e += TN) {
            const int r = e / K, k = e - r * K;
            if (base + r < a.n) a.v16[(size_t)(base + r) * K + k] = rows[rowat[r]][k];
        }
    if (a.cop) {
        // The tile's two balls: its points split by which of two seeds they are
        // nearer to (the first point and the point farthest from it), so that a
        // tile where two groups of points meet still has small balls.  A
        // ball's centre is its points' mean, rounded to the grid (an operand row
        // like any other), its radius the largest distance of a point to it.
        auto dist2 = [&](const int16_t *r1, auto &&c) {
            int D = 0;
            for (int j = 0; j < K; ++j) {
                const int df = r1[j] - c[j];
                D += df * df;
            }
            return D;
        };
        const int D0 = valid ? dist2(rows[tid], rows[0]) : -1;
        unsigned long long key = ((unsigned long long)(unsigned)(D0 + 1) << 8) | (unsigned)tid;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long y = __shfl_xor_sync(FULL, key, o);
            key = y > key ? y : key;
        }
        if (lane == 0) far_s[warp] = key;
        __syncthreads();
        for (int w = 0; w < 8; ++w) key = far_s[w] > key ? far_s[w] : key;
        const int part = valid && dist2(rows[tid], rows[key & 255ull]) < D0;
        part_s[tid] = (uint8_t)part;
        const int n1 = __syncthreads_count(part), nv = min(TN, a.n - base), n0 = nv - n1;
        {
            const int k = tid & 63, q4 = tid >> 6;
            int s0 = 0, s1 = 0;
            if (k < K)
                for (int rr = q4 * 64; rr < min(nv, q4 * 64 + 64); ++rr) {
                    const int v = rows[rr][k];
                    s0 += v;
                    s1 += part_s[rr] ? v : 0;
                }
            csum[0][q4][k] = s0 - s1;
            csum[1][q4][k] = s1;
        }
        __syncthreads();
        if (tid < 128) {
            const int b = tid >> 6, k = tid & 63;
            const int t = csum[b][0][k] + csum[b][1][k] + csum[b][2][k] + csum[b][3][k];
            cen[b][k] = k < K ? __float2int_rn((float)t / (float)max(1, b ? n1 : n0)) : 0;
        }
        __syncthreads();
        const int D = valid ? dist2(rows[tid], cen[part]) : -1;
        const int m0 = __reduce_max_sync(FULL, part ? -1 : D), m1 = __reduce_max_sync(FULL, part ? D : -1);
        if (lane == 0) {
            wsum[warp] = m0;
            wval[warp] = m1;
        }
        __syncthreads();
        if (tid < 2) {
            int R = -1, cc = 0;  // -1: no point in this ball
            for (int w = 0; w < 8; ++w) R = max(R, tid ? wval[w] : wsum[w]);
            for (int j = 0; j < K; ++j) cc += cen[tid][j] * cen[tid][j];
            a.crad[2 * tile + tid] = (float)R;
            a.cbeta[2 * tile + tid] = (float)cc;
        }
        const int kgs = K / 8;
        if (tid < 2 * kgs) {
            const int b = tid >= kgs, kg = tid - b * kgs, ball = 2 * tile + b, ct = ball / TN, cr = ball % TN;
            uint16_t h[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) h[j] = fp16_bits(cen[b][kg * 8 + j]);
            store8(a.cop + (size_t)ct * TN * K + ((size_t)((cr >> 3) * kgs + kg) * 64) + (cr & 7) * 8, h);
        }
    }
}

// Rank of each pivot in the order (group, pivot), groups being the trees of
// the links (each pivot to the first one within twice eps): the pivots of one
// group of points, and so their buckets, lie side by side (a bitonic sort by
// one block of P threads).  Also clears the bucket sizes.
__global__ void __launch_bounds__(1024) tc_pivot_rank_kernel(const int *__restrict__ link, int P,
                                                             int *__restrict__ prank, int *__restrict__ hist,
                                                             int nhist) {
    db::wait_prior_grid();  // started as a programmatic dependent
    db::allow_next_grid();
    __shared__ int up[1024];
    __shared__ unsigned s[1024];
    const int t = threadIdx.x;
    for (int e = t; e < nhist; e += (int)blockDim.x) hist[e] = 0;
    up[t] = link[t];
    __syncthreads();
    int r = t;
    while (up[r] < r) r = up[r];  // links point to smaller pivots: ends at the group's first
    s[t] = ((unsigned)r << 10) | (unsigned)t;
    for (int k = 2; k <= P; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            __syncthreads();
            const int y = t ^ j;
            if (y > t) {
                const unsigned a = s[t], b = s[y];
                if ((a > b) == ((t & k) == 0)) {
                    s[t] = b;
                    s[y] = a;
                }
            }
        }
    __syncthreads();
    prank[s[t] & 1023u] = t;
}

__global__ void tc_bucket_scatter_kernel(int n, const int *__restrict__ key, const int *__restrict__ rank,
                                         const int *__restrict__ start, int *__restrict__ list) {
    db::wait_prior_grid();  // started as a programmatic dependent
    db::allow_next_grid();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) list[start[key[i]] + rank[i]] = i;
}

// pairs = near & transpose(near), in place: a warp per 32 x 32 block pair
// (ib, jb) with ib <= jb reads and writes both blocks.
__global__ void __launch_bounds__(256) tc_pairs_kernel(int nt, int words, unsigned *__restrict__ near) {
    db::wait_prior_grid();  // started as a programmatic dependent
    db::allow_next_grid();
    const int lane = threadIdx.x & 31;
    const long long nblk = (long long)words * words;
    const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long w = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < nblk; w += nwarps) {
        const int ib = (int)(w / words), jb = (int)(w - (long long)ib * words);
        if (ib > jb) continue;
        const int i = ib * 32 + lane, j = jb * 32 + lane;
        const unsigned r = i < nt ? near[(size_t)i * words + jb] : 0u;  // row i, columns of jb
        const unsigned c = j < nt ? near[(size_t)j * words + ib] : 0u;  // row j, columns of ib
        unsigned ct = 0, rt = 0;  // transposes: bit k of lane l = bit l of lane k
#pragma unroll
        for (int k = 0; k < 32; ++k) {
            const unsigned bc = __ballot_sync(FULL, (c >> k) & 1u), br = __ballot_sync(FULL, (r >> k) & 1u);
            if (lane == k) {
                ct = bc;
                rt = br;
            }
        }
        if (i < nt) near[(size_t)i * words + jb] = r & ct;
        if (j < nt) near[(size_t)j * words + ib] = c & rt;
    }
}

// Core flags and what follows from them, a block per tile: metadata with the
// non-core points masked out (merge; border columns) and with all but the rows
// the border pass needs masked out (not core, some neighbour: their counts are
// exact, since a row unit is left early only when all its rows are core).
__global__ void __launch_bounds__(256) tc_core_kernel(int n, int min_pts, const int *__restrict__ count,
                                                      uint8_t *__restrict__ core, int *__restrict__ parent,
                                                      int *__restrict__ border, int *__restrict__ least,
                                                      const MetaTile *__restrict__ meta, MetaTile *__restrict__ mcore,
                                                      MetaTile *__restrict__ mneed, int *__restrict__ tag,
                                                      int *__restrict__ rowneed) {
    db::wait_prior_grid();  // started as a programmatic dependent
    db::allow_next_grid();
    const int tile = blockIdx.x, t = threadIdx.x, p = tile * TN + t;
    const int c = p < n ? count[p] : 0;
    const bool is = p < n && c >= min_pts, need = p < n && !is && c > 1;
    if (p < n) {
        core[p] = is;
        parent[p] = p;
        border[p] = DB_NONE;
        least[p] = DB_NONE;
    }
    const float b = meta[tile].beta[t], bf = meta[tile].beta_f[t];
    const int idx = meta[tile].idx[t];
    mcore[tile].beta[t] = is ? b : 1e30f;
    mcore[tile].beta_f[t] = is ? bf : 1e30f;
    mcore[tile].idx[t] = idx;
    mneed[tile].beta[t] = need ? b : 1e30f;
    const int any = __syncthreads_or(is), anyn = __syncthreads_or(need);
    if (t == 0) {
        tag[tile] = any ? -1 : -2;
        rowneed[tile] = anyn;
    }
}

// The core points of a tile joined among themselves, from the adjacency words
// of the tile with itself: every row under its first neighbour, flattened, then
// smaller labels of any neighbour until none is left, in shared memory.  The
// merge then only crosses tiles (200,000 x 64: with each row only hooked under
// its first earlier neighbour some 55 sets a tile were left, and the near tiles
// took 238 us).  A block per tile; sets the tile's tag.
__global__ void __launch_bounds__(256) tc_join_kernel(int n, const uint8_t *__restrict__ core,
                                                      const uint4 *__restrict__ adj, int *__restrict__ parent,
                                                      int *__restrict__ tag) {
    db::wait_prior_grid();  // started as a programmatic dependent
    db::allow_next_grid();
    __shared__ int lab[TN];
    const int tile = blockIdx.x, t = threadIdx.x, p = tile * TN + t;
    const bool is = p < n && core[p];
    if (!__syncthreads_or(is)) return;  // the tag says so already
    unsigned m[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
    if (is) {
        const uint4 x = adj[(size_t)p * 2], y = adj[(size_t)p * 2 + 1];
        m[0] = x.x, m[1] = x.y, m[2] = x.z, m[3] = x.w, m[4] = y.x, m[5] = y.y, m[6] = y.z, m[7] = y.w;
    }
    int l = t;
#pragma unroll
    for (int k = 7; k >= 0; --k)
        if (m[k]) l = 32 * k + __ffs((int)m[k]) - 1;
    lab[t] = min(l, t);
    __syncthreads();
    while (true) {
        l = t;
        while (lab[l] < l) l = lab[l];  // labels point to earlier rows
        __syncthreads();
        lab[t] = l;
        if (__syncthreads_count(is && l == t) <= 1) break;
        int least = l;
#pragma unroll
        for (int k = 0; k < 8; ++k)
            for (unsigned w = m[k]; w; w &= w - 1) least = min(least, lab[32 * k + __ffs((int)w) - 1]);
        const bool moved = least < l;
        if (!__syncthreads_or(moved)) break;
        if (moved) {
            atomicMin(&lab[l], least);  // the group's first row, too
            atomicMin(&lab[t], least);
        }
        __syncthreads();
    }
    if (is) parent[p] = tile * TN + l;
    const int roots = __syncthreads_count(is && l == t);
    if (is && l == t && roots == 1) tag[tile] = p;
}

// Every core point straight under its root, and per tile the root its core
// points share (-1 when they are of several sets), a block per tile.
__global__ void __launch_bounds__(256) tc_tag_kernel(int n, const uint8_t *__restrict__ core, int *parent,
                                                     int *__restrict__ tag) {
    db::wait_prior_grid();  // started as a programmatic dependent
    db::allow_next_grid();
    __shared__ int lo_s[8], hi_s[8];
    const int tile = blockIdx.x, t = threadIdx.x, p = tile * TN + t;
    const bool is = p < n && core[p];
    int root = -1;
    if (is) {
        root = db::uf_find(parent, p);
        if (root != p) db::st_relaxed(parent + p, root);
    }
    const int lo = __reduce_min_sync(FULL, is ? root : INT_MAX), hi = __reduce_max_sync(FULL, root);
    if ((t & 31) == 0) {
        lo_s[t >> 5] = lo;
        hi_s[t >> 5] = hi;
    }
    __syncthreads();
    if (t == 0) {
        int l = INT_MAX, h = -1;
        for (int w = 0; w < 8; ++w) {
            l = min(l, lo_s[w]);
            h = max(h, hi_s[w]);
        }
        if (h >= 0) tag[tile] = l == h ? l : -1;
    }
}

// Root of every core position, and the smallest point index of each set.
__global__ void __launch_bounds__(256) tc_root_kernel(int n, const uint8_t *__restrict__ core,
                                                      const int *__restrict__ perm, int *parent, int *least) {
    db::wait_prior_grid();  // started as a programmatic dependent
    db::allow_next_grid();
    const int p = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
    const bool is = p < n && core[p];
    const int root = is ? db::uf_settle(parent, p) : -1 - lane;
    // one atomic per distinct root of the warp, and none that cannot lower the value
    const unsigned peers = __match_any_sync(FULL, root);
    if (is) {
        const int m = __reduce_min_sync(peers, perm ? perm[p] : p);
        if (lane == __ffs(peers) - 1 && m < db::ld_relaxed(least + root)) atomicMin(least + root, m);
    }
}

// Labels (a core point: the smallest point index of its set; a border point:
// the label of its smallest-index core neighbour; noise: -1), the optional
// counts and core flags, and the run's statistics.
__global__ void __launch_bounds__(256) tc_label_kernel(int n, const uint8_t *__restrict__ core,
                                                       const int *__restrict__ perm, const int *__restrict__ inv,
                                                       const int *__restrict__ parent, const int *__restrict__ border,
                                                       const int *__restrict__ least, const int *__restrict__ count,
                                                       int *__restrict__ labels, int *__restrict__ counts_out,
                                                       uint8_t *__restrict__ core_out, unsigned long long *ctr,
                                                       const unsigned *status, unsigned *status_out) {
    db::wait_prior_grid();  // started as a programmatic dependent
    db::allow_next_grid();
    db::report_status(status, status_out);
    __shared__ int red[4];
    if (threadIdx.x < 4) red[threadIdx.x] = 0;
    __syncthreads();
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    int kind = -1;
    bool root = false;
    if (p < n) {
        const int o = perm[p];
        int lab = -1;
        kind = 2;
        if (core[p]) {
            const int r = parent[p];
            lab = least[r];
            root = r == p;
            kind = 0;
        } else if (border[p] != DB_NONE) {
            lab = least[parent[inv[border[p]]]];
            kind = 1;
        }
        labels[o] = lab;
        if (counts_out) counts_out[o] = count[p];
        if (core_out) core_out[o] = kind == 0;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const unsigned m = __ballot_sync(FULL, k < 3 ? kind == k : root);
        if ((threadIdx.x & 31) == 0 && m) atomicAdd(&red[k], __popc(m));
    }
    __syncthreads();
    if (threadIdx.x < 4 && red[threadIdx.x]) atomicAdd(ctr + 2 + threadIdx.x, (unsigned long long)red[threadIdx.x]);
}

template <int PASS, bool BF16>
cudaError_t launch_pass_t(const TcArgs &a, int sms, cudaStream_t st) {
    // the shared-memory attribute, set once per device (plans may live on
    // several devices of one process; setting it twice is harmless)
    static std::atomic<unsigned long long> attr_set{0};
    int dev = 0;
    cudaGetDevice(&dev);
    const unsigned long long bit = dev < 64 ? 1ull << dev : 0ull;
    if (!(attr_set.load(std::memory_order_relaxed) & bit) || !bit) {
        cudaError_t e = cudaFuncSetAttribute(tc_pass_kernel<PASS, BF16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)TcSmem<PASS, BF16>::bytes);
        if (e) return e;
        attr_set.fetch_or(bit, std::memory_order_relaxed);
    }
    return launch_dependent_smem(tc_pass_kernel<PASS, BF16>, dim3(sms), dim3(Shape<PASS, BF16>::THREADS),
                                 TcSmem<PASS, BF16>::bytes, st, a);
}

template <int PASS>
cudaError_t launch_pass(const TcArgs &a, bool bf16, int sms, cudaStream_t st) {
    return bf16 ? launch_pass_t<PASS, true>(a, sms, st) : launch_pass_t<PASS, false>(a, sms, st);
}

int sm_count() {
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms;
}

// Merge: the tiles after a row unit's own that are taken first.
constexpr int kNearTiles = 2;

// Points from which they are ordered and tile pairs culled (see the header).
constexpr int kSortMinN = 32768;

}  // namespace

// Host launcher of the whole tensor-core all-pairs pipeline.
cudaError_t launch_allpairs_tc(const DbWork &w, const float *x, int64_t n64, int32_t d, int64_t Tc, int32_t min_pts,
                               bool exact, bool bf16, bool stall, int32_t *labels, int32_t *counts_out,
                               uint8_t *core_out, cudaStream_t st) {
    const int n = (int)n64;
    const int K = ((d + 15) / 16) * 16;
    const int nt = (n + TN - 1) / TN, words = (nt + 31) / 32;
    const int sms = sm_count();
    const bool sorted = n >= kSortMinN;
    MetaTile *meta = reinterpret_cast<MetaTile *>(w.metaAll), *mcore = reinterpret_cast<MetaTile *>(w.metaCore),
             *mneed = reinterpret_cast<MetaTile *>(w.metaNon);
    int *bmax = w.tc_lens;
    int *least = w.scan, *perm = w.list_a, *inv = w.list_b;
    cudaError_t e;

    TcArgs a{};
    a.K = K;
    a.T = (int)Tc;
    a.status = w.status;
    a.ctr = w.ctr;
    a.wait_ns = 2000000000ull;  // about two seconds per barrier wait
    a.v16 = w.v16;
    a.count = w.count;
    a.parent = w.parent;
    a.border = w.border;
    a.udone = w.tc_udone;
    a.tag = w.tc_tag;
    a.rowneed = w.tc_rowneed;
    a.cbeta = w.tc_cbeta;
    a.crad = w.tc_crad;
    a.words = words;

    PackArgs pk{};
    pk.x = x;
    pk.n = n;
    pk.d = d;
    pk.K = K;
    pk.status = w.status;
    if ((e = cudaMemsetAsync(bmax, 0, sizeof(int) * 8, st))) return e;
    if (sorted) {
        const int P = n < 65536 ? 256 : (n < 131072 ? 512 : 1024), nhist = 8 * P;
        int *link = w.parent, *prank = w.border, *hist = w.tc_hist, *key = w.count, *rank = w.scan;  // free until later
        PackArgs pp = pk;  // pivots
        pp.n = P;
        pp.n_src = n;
        pp.op = w.opNon;
        pp.meta = mneed;
        launch_dependent(tc_pack_kernel, P / TN, 256, st, pp);
        w.marks->kernel("tc_pack_pivots", st);
        TcArgs o = a;
        o.opR = o.opC = w.opNon;
        o.metaR = o.metaC = mneed;
        o.nR = o.nC = P;
        o.kv = K;
        o.tile_r = o.tile_c = TN * K;
        o.ct_chunk = P / TN;
        o.rel_lo = 0;
        o.rel_hi = 1;
        o.key = link;
        if ((e = launch_pass_t<TC_LINK, false>(o, sms, st))) return e;
        w.marks->kernel("tc_pivot_link", st);
        launch_dependent(tc_pivot_rank_kernel, 1, P, st, link, P, prank, hist, nhist);
        w.marks->kernel("tc_pivot_rank", st);
        PackArgs pu = pk;  // all points in index order
        pu.op = w.opCore;
        pu.meta = mcore;
        launch_dependent(tc_pack_kernel, nt, 256, st, pu);
        w.marks->kernel("tc_prep", st);
        o.opR = w.opCore;
        o.metaR = mcore;
        o.nR = n;
        o.n_piv = P;
        o.prank = prank;
        o.key = key;
        o.rank = rank;
        o.hist = hist;
        if ((e = launch_pass_t<TC_ORDER, false>(o, sms, st))) return e;
        w.marks->kernel("tc_order", st);
        if ((e = launch_bucket_scan(hist, nhist, st))) return e;
        w.marks->kernel("tc_bucket_scan", st);
        launch_dependent(tc_bucket_scatter_kernel, (n + 255) / 256, 256, st, n, key, rank, hist, perm);
        w.marks->kernel("tc_bucket_scatter", st);
        pk.list = perm;
    }
    // The points in their final order, with the balls of their tiles.  BF16
    // plans cull on FP16 operands too (exact), packed into the order pass's buffer.
    pk.perm = perm;
    pk.inv = inv;
    pk.count = w.count;
    pk.udone = w.tc_udone;
    pk.units_per_tile = bf16 ? 2 : 1;
    const int fold = bf16 ? 0 : 1, kv = bf16 ? 2 * K : K, tile = TN * (kv + 16 * fold);
    if (bf16 && sorted) {
        PackArgs pf = pk;
        pf.op = w.opCore;
        pf.meta = mcore;
        pf.cop = w.opNon;
        pf.cbeta = w.tc_cbeta;
        pf.crad = w.tc_crad;
        launch_dependent(tc_pack_kernel, nt, 256, st, pf);
        w.marks->kernel("tc_pack_cull", st);
    }
    pk.op = w.opAll;
    pk.meta = meta;
    pk.bf16 = bf16 ? 1 : 0;
    pk.fold = fold;
    pk.bmax = bmax;
    if (bf16) pk.v16 = w.v16;
    if (sorted && !bf16) {
        pk.cop = w.opNon;
        pk.cbeta = w.tc_cbeta;
        pk.crad = w.tc_crad;
    }
    launch_dependent(tc_pack_kernel, nt, 256, st, pk);
    w.marks->kernel("tc_pack", st);
    if (sorted) {
        TcArgs c = a;
        c.opR = w.opNon;
        c.metaR = mneed;  // copied, not read: the balls' terms come from cbeta and crad
        c.nR = 2 * nt;  // two balls per tile
        c.opC = bf16 ? w.opCore : w.opAll;
        c.metaC = bf16 ? mcore : meta;
        c.nC = n;
        c.kv = K;
        c.tile_r = TN * K;
        c.tile_c = bf16 ? TN * K : tile;
        c.near = w.tc_pairs;
        c.ct_chunk = tcitems::chunk_tiles((2 * nt + 255) / 256, nt, sms);
        c.rel_lo = 0;
        c.rel_hi = (nt + c.ct_chunk - 1) / c.ct_chunk;
        if ((e = launch_pass_t<TC_CULL, false>(c, sms, st))) return e;
        w.marks->kernel("tc_cull", st);
        const int64_t blk = (int64_t)words * words;
        launch_dependent(tc_pairs_kernel, (int)std::min<int64_t>((blk + 7) / 8, 152 * 8), 256, st, nt, words,
                         w.tc_pairs);
        w.marks->kernel("tc_pairs", st);
        a.pairs = w.tc_pairs;
        a.rotate = 1;
    }

    // pass 1: neighbour counts (the stall hook: a 50 ms budget the waits
    // exhaust, since no MMA completes)
    a.opR = a.opC = w.opAll;
    a.metaR = a.metaC = meta;
    a.nR = a.nC = n;
    a.kv = kv;
    a.fold = fold;
    a.tile_r = a.tile_c = tile;
    a.min_pts = exact ? 0 : min_pts;
    a.bmax_ptr = bmax;
    a.stall = stall ? 1 : 0;
    if (stall) a.wait_ns = 50000000ull;
    const int units1 = (n + TM - 1) / TM;  // units of one row tile
    a.ct_chunk = tcitems::chunk_tiles(bf16 ? units1 : nt, nt, sms);
    a.rel_lo = 0;
    a.rel_hi = (nt + a.ct_chunk - 1) / a.ct_chunk;
    // opCore is free from here on: adjacency words, then the item list (when it fits)
    a.adj = reinterpret_cast<unsigned *>(w.opCore);
    int4 *list = reinterpret_cast<int4 *>(w.opCore + (size_t)nt * TN * 16);
    const int64_t list_cap = (w.tc_cap_pad * 64 - (int64_t)nt * TN * 16) / 8;
    int next_list = 1;  // tc_lens[1..6]: length and ticket of up to three lists, cleared above
    auto use_list = [&](auto pass) -> cudaError_t {
        constexpr int PASS = decltype(pass)::value;
        const int64_t units = bf16 || PASS == TC_UNION ? (n + TM - 1) / TM : nt, nit = tcitems::count((int)units, a.rel_hi - a.rel_lo);
        a.items = nullptr;
        if (!sorted || nit > list_cap) return cudaSuccess;
        a.nlist = w.tc_lens + next_list++;
        a.ticket = w.tc_lens + next_list++;
        TcArgs q = a;
        q.items = list;
        const int blocks = (int)((nit + 255) / 256);
        if constexpr (PASS == TC_UNION) launch_dependent(tc_items_kernel<PASS, 1>, blocks, 256, st, q);
        else if (bf16) launch_dependent(tc_items_kernel<PASS, 1>, blocks, 256, st, q);
        else launch_dependent(tc_items_kernel<PASS, 2>, blocks, 256, st, q);
        w.marks->kernel("tc_items", st);
        a.items = list;
        return cudaGetLastError();
    };
    if ((e = use_list(std::integral_constant<int, TC_COUNT>{}))) return e;
    if ((e = launch_pass<TC_COUNT>(a, bf16, sms, st))) return e;
    a.items = nullptr;
    w.marks->kernel("tc_count", st);
    a.stall = 0;
    a.wait_ns = 2000000000ull;
    launch_dependent(tc_core_kernel, nt, 256, st, n, min_pts, w.count, w.core, w.parent, w.border, least, meta, mcore,
                     mneed, w.tc_tag, w.tc_rowneed);
    w.marks->kernel("core_init", st);

    // pass 2: union of core-core neighbours.  First inside every tile; then the
    // near tiles; then the rest, most of which the sets found so far skip.
    a.metaR = a.metaC = mcore;
    a.fold = 0;
    const int ch_union = tcitems::chunk_tiles(units1, nt, sms), nch = (nt + ch_union - 1) / ch_union;
    a.ct_chunk = ch_union;
    a.rel_lo = 0;
    a.rel_hi = 1;
    if ((e = launch_pass<TC_ADJ>(a, bf16, sms, st))) return e;
    w.marks->kernel("tc_adj", st);
    launch_dependent(tc_join_kernel, nt, 256, st, n, w.core, reinterpret_cast<const uint4 *>(a.adj), w.parent,
                     w.tc_tag);
    w.marks->kernel("tc_join", st);
    // (the tiles right after a row unit's own first: they link most of what
    // belongs together, and the tags then skip most of the rest)
    a.near_lo = 0;
    a.near_hi = kNearTiles;
    a.rel_hi = std::min(nch, 1 + (kNearTiles + ch_union - 1) / ch_union);
    if ((e = launch_pass<TC_UNION>(a, bf16, sms, st))) return e;
    w.marks->kernel("tc_union_near", st);
    if (nt > 1 + kNearTiles) {
        launch_dependent(tc_tag_kernel, nt, 256, st, n, w.core, w.parent, w.tc_tag);
        w.marks->kernel("tc_tag", st);
        a.near_lo = 1 + kNearTiles;
        a.near_hi = nt;
        a.rel_lo = 0;
        a.rel_hi = nch;
        if ((e = use_list(std::integral_constant<int, TC_UNION>{}))) return e;
        if ((e = launch_pass<TC_UNION>(a, bf16, sms, st))) return e;
        a.items = nullptr;
        w.marks->kernel("tc_union", st);
    }

    // pass 3: smallest core neighbour of the rows that need one
    a.metaR = mneed;
    a.metaC = mcore;
    a.ct_chunk = tcitems::chunk_tiles(bf16 ? units1 : nt, nt, sms);
    a.rel_lo = 0;
    a.rel_hi = (nt + a.ct_chunk - 1) / a.ct_chunk;
    if ((e = use_list(std::integral_constant<int, TC_BORDER>{}))) return e;
    if ((e = launch_pass<TC_BORDER>(a, bf16, sms, st))) return e;
    w.marks->kernel("tc_border", st);

    launch_dependent(tc_root_kernel, (n + 255) / 256, 256, st, n, w.core, perm, w.parent, least);
    w.marks->kernel("tc_root", st);
    launch_dependent(tc_label_kernel, (n + 255) / 256, 256, st, n, w.core, perm, inv, w.parent, w.border, least,
                     w.count, labels, counts_out, core_out, w.ctr, w.status, w.status_out);
    w.marks->kernel("labels", st);
    return cudaGetLastError();
}

// Diagnostic: the count pass with every pair also decided exactly; records in
// ctr[6] the band pairs, ctr[7] the pairs outside the band whose fast decision
// disagrees with the exact one (must be 0), ctr[8] the largest |2G - exact|.
cudaError_t launch_tc_verify(const DbWork &w, const float *x, int64_t n64, int32_t d, int64_t Tc, bool bf16,
                             cudaStream_t st) {
    const int n = (int)n64;
    const int K = ((d + 15) / 16) * 16;
    const int nt = (n + TN - 1) / TN, sms = sm_count();
    PackArgs pk{};
    pk.x = x;
    pk.n = n;
    pk.d = d;
    pk.K = K;
    pk.status = w.status;
    pk.bf16 = bf16 ? 1 : 0;
    pk.op = w.opAll;
    pk.meta = reinterpret_cast<MetaTile *>(w.metaAll);
    pk.count = w.count;
    pk.v16 = w.v16;
    launch_dependent(tc_pack_kernel, nt, 256, st, pk);
    TcArgs a{};
    a.K = K;
    a.kv = bf16 ? 2 * K : K;
    a.tile_r = a.tile_c = TN * a.kv;
    a.T = (int)Tc;
    a.v16 = w.v16;
    a.count = w.count;
    a.status = w.status;
    a.ctr = w.ctr;
    a.wait_ns = 2000000000ull;
    a.opR = a.opC = w.opAll;
    a.metaR = a.metaC = reinterpret_cast<const MetaTile *>(w.metaAll);
    a.nR = a.nC = n;
    a.ct_chunk = tcitems::chunk_tiles((n + TM - 1) / TM, nt, sms);
    a.rel_lo = 0;
    a.rel_hi = (nt + a.ct_chunk - 1) / a.ct_chunk;
    return launch_pass<TC_VERIFY>(a, bf16, sms, st);
}
