// Tree-masked verification attention over a paged bf16 KV cache (Section 2.2;
// Algorithm 1, the target pass over all tree tokens; Section 3.3 Phase 2), sm_100a:
// the streaming schedule, what its two kernels share: how work is laid out and cut, and the pieces of a CTA.
// tree_attention_rows.cu and tree_attention_alt.cu hold the kernels, tree_attention.cu the dispatch and the C entry points.
//
// Work decomposition.  The N tree nodes x G query heads that share one KV head form
// M = N*G query rows (<= 512).  An *item* is one (layer, sequence, KV head); its work
// is measured in steps of 128 keys (two 64-token pages), its end counts as kItemExtra
// more.  All items are laid end to end and cut into equal ranges, one range per *gang*; a gang is the 1 or 2
// CTAs (one per 256 query rows) that walk the same range side by side, so that the
// second CTA finds the K/V of the first in L2.  A kernel launch is one resident CTA
// per SM that loops over the segments of its range: whole items write their output
// directly, items cut by a range boundary leave unnormalised partial results that
// the merge kernel combines, told by a record per range which item that is.  Nothing waits on another CTA.
//
// Inside a CTA (384 threads): tensor memory holds two slots t of (S_t 128 x 128 fp32 scores,
// O_t 128 x 128 fp32 accumulator): S_t in columns [128t, 128t+128), O_t in [256+128t, 384+128t).
//   TMA      : K and V tiles of a step (2 pages x 2 d-halves) -> 128B-swizzled shared memory, rings of
//              3 K tiles and 2 or 3 V tiles, mbarriers; the query tiles also arrive by TMA
//   tcgen05  : S_t = Q K^T into TMEM, O_t += P_t V with P as the TMEM A operand (V MN-major); one warp
//              issues for both slots, in blocks [P V of an earlier step, scores of a later one]
//   softmax  : one warpgroup per slot, one thread per row: tcgen05.ld S in 32-column chunks,
//              online softmax in fp32 (log2 domain, lazy rescale), P -> bf16 back into TMEM
//              over the first 64 columns of S_t
// The two slots alternate on the tensor pipe: while one's warpgroup runs its softmax, the pipe works on the
// other.  What a slot is depends on the batch's largest tree, which the device works out:
//   tree_attention_rows.cu (more than 128 rows): slot = row tile; every step goes to both slots, K/V enters the SM once.
//   tree_attention_alt.cu (up to 128 rows): both slots belong to the same rows and take the even and the odd steps
//     of a segment, each with its own accumulator and running (reference, sum); combined in the epilogue.
//     (With one slot per row tile the chain scores -> softmax -> P V would be strictly serial.)
// Clocks per K=16 slice, measured (128 rows, N columns): N/2 with the A operand in TMEM; with both in shared memory 32 + N/4 up to
// N = 128, which is what reading them takes, so scores of 64 keys cost 48 and of 128 keys 64: hence the 128-key step.
// All waits are bounded: on expiry the CTA records SAGE_STATUS_TIMEOUT, waits (bounded) for
// its copies and MMAs in flight, frees its TMEM and returns.
#pragma once

#include <cuda.h>

#include <atomic>

#include "sage_common.cuh"

namespace sage {
namespace stream {

constexpr int kRowTile = 128;                  // query rows per MMA tile
constexpr int kRowsPerCta = 2 * kRowTile;
constexpr int kStepKeys = 2 * kPageSize;       // keys per pipeline step
constexpr int kKStages = 3;                    // K tiles in flight
constexpr int kRing = 4;                       // barrier pairs of the copy ring (> ring steps in flight)
constexpr int kPageHalfBytes = kPageSize * 64 * 2;          // one TMA box: 64 keys x 64-wide d-half = 8 KB
constexpr int kTileHalfBytes = kStepKeys * 64 * 2;          // one d-half of a 128-key tile: 16 KB
constexpr int kTileBytes = 2 * kTileHalfBytes;              // K or V tile of one step: 32 KB
constexpr int kQTileBytes = kRowTile * kHeadDim * 2;        // 32 KB
constexpr int kQHalfBytes = kRowTile * 64 * 2;              // one 64-wide d-half of a Q tile: 16 KB
constexpr int kAttnThreads = 384;              // 2 softmax warpgroups + one warpgroup of TMA warp, MMA warp and two idle warps
// A row's step whose probabilities sum to this or more goes through its maximum, to which the reference then moves.  Lower, rows of
// widely spread scores compute many steps twice (one layer, 60 nodes, 16k keys of three times the usual spread: 54.8 us at 2^8,
// 49.2 at 2^10, 44.7 here, 40.5 for the usual); higher, the dominant probability of a row is rounded to bf16 more often where it
// would be exactly 1 (error on growing scores 1.92e-3 of the outputs' norm at 2^8, 1.95e-3 here, 1.98e-3 at 2^14, 2.15e-3 at 2^30).
constexpr float kMaxSum = 4096.f;
// No more ranges than one for so many steps (the extra of ends of items counts, so one may hold fewer).  And where items have no more on
// average, and there is a gang for each, ranges are as many as items: with 147 items of two steps on 148 gangs every boundary cut one into two
// single steps (23.0 us instead of 18.4; 72 items on 74 pairs of CTAs 28.0 instead of 22.2).
constexpr int kMinSteps = 2;
// What an item costs beyond its steps, in steps: the step that holds the tree takes longer, and between two segments lie an epilogue, new
// query rows and a first step.  Without it ranges of equally many steps take as much longer as they hold more ends of items (sixteen
// sequences of 1k to 8k keys: a CTA's 53 steps took 122 us on average, 134 at most).  Measured with 0 / 1 / 2 / 3 / 4, us: those 145.0 / 143.7 /
// 142.8 / 142.1 / 144.6; sixteen of 1k to 4k, 12 nodes 57.7 / 57.0 / 54.1 / 56.1 / 56.6; forty of 64 to 1000 89.9 / 83.8 / 80.0 / 79.4 / 77.6;
// one of 4k, 80 layers 257 / 259 / 256 / 257 / 257.
constexpr int kItemExtra = 2;

// The boundary in front of a CTA's range as the merge kernel needs it: which item it cuts, and which gangs hold the item.
struct __align__(16) Cut {
    int n_rp;                       // CTAs per gang
    int s0;                         // step inside the item that the boundary falls on; 0: between two items, or there is no boundary
    int layer, u, b, n0, N, steps;  // the item
    int k_first, k_last;            // gangs that hold it
    int mid;                        // it begins in the middle of the first one's range
    int pad;
};
struct AttnParams {
    __nv_bfloat16* out;
    // Partial results, one slot per CTA for the head and one for the tail of its range.  Four output columns of
    // consecutive rows lie side by side: a warp (one thread per row) writes 512 contiguous bytes per instruction, where
    // row-major slots took 32 separate lines (an epilogue of 6 000 to 10 000 clocks; now 1 500 to 3 000).
    float4* part_o;    // [CTA][2][32 column quads][256 rows]   unnormalised
    float2* part_ml;   // [CTA][2][256 rows]                    (reference in log2 units, l)
    Cut* cuts;         // [CTA]
    const int32_t* page_table;
    const int32_t* seq_len;
    const int32_t* parent;
    const int32_t* node_offsets;
    int32_t* status;
    int n_layers, batch, sum_nodes, n_pages, max_pages;
    int Hq, Hkv, G, g_shift;   // G = 1 << g_shift query heads per KV head
    int n_ctas, n_rp;          // CTAs of the launch; most CTAs a gang can have (row pairs of the largest possible tree)
    float scale_log2;          // sm_scale * log2(e)
    long long wait_cycles;     // budget of every on-device wait
    int producer_off;          // diagnostics: the TMA warp issues no copies (every consumer wait then runs out)
};

// How a launch's work is laid out (see make_plan).
struct Plan {
    int n_rp;               // CTAs per gang
    int heads_all;          // units that every sequence takes part in; the others are for trees of two row pairs only
    int steps_all, steps_big;   // steps of all sequences, and of those with two row pairs (here and below: with kItemExtra for each item)
    int n_act;              // gangs that get a range (which may turn out empty, see locate)
    int one_tile;           // no tree has more than one row tile
    long long steps_layer, W;   // steps of a layer, of the launch
};
struct Place { int layer, u, b, s0; };     // layer, unit, sequence and step of a position in the launch's work
struct __align__(16) Shared {
    uint64_t kv_full[kRing];   // ring step r: its K tile and its V tile have landed
    uint64_t kv_done[kRing];   // ring step r: every MMA that reads those tiles has finished
    uint64_t s_full[2];        // [slot]: scores of a step are in TMEM
    uint64_t p_full[2];        // [slot]: probabilities of a step are in TMEM
    uint64_t o_full[2];        // [slot]: every MMA of the slot's part of the segment has finished
    uint64_t epi_done;         // alternating: the softmax warps have read both accumulators of the segment
    uint64_t q_free;           // the segment's last score MMAs have read the query tiles
    uint64_t q_ready;          // the query tiles of the segment are in shared memory
    uint64_t drain;            // abort path: everything issued so far has retired
    volatile uint32_t eflag[2][4];     // alternating: [slot][quadrant] segment number whose (reference, sum) this warp has posted
    long long range_begin, range_end;
    Plan plan;
    Place first;               // where the range begins
    int n_rp, heads_all;       // of the plan
    uint32_t tmem_base;
    volatile int abort;
    int parked[8][24];         // alternating: what a softmax warp knows of its segment and need not hold in registers
};
constexpr int kSmemBytes = 1024 /*align*/ + 7 * kTileBytes + (int)sizeof(Shared);
static_assert(kSmemBytes <= 232448, "shared memory budget of one CTA exceeded");

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// ---- mbarrier ---------------------------------------------------------------
__device__ __forceinline__ void mbar_init(uint64_t* bar, int count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
    return ok != 0;
}
// Bounded wait.  Returns false when the CTA is aborting (this wait or another one expired).
template <typename S, typename P>
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, S* sh, const P& p) {
    if (mbar_try(bar, parity)) return true;
    const long long t0 = clock64();
    while (true) {
        // (Not unrolled: left to the compiler, every wait of a kernel held 64 tries, a quarter to a third of its code, and spinning
        // warps ran through it beside those that work.  One row tile: 116 -> 89 KB of code.)
#pragma unroll 1
        for (int i = 0; i < 64; ++i)
            if (mbar_try(bar, parity)) return true;
        if (sh->abort) return false;
        if (clock64() - t0 > p.wait_cycles) {
            sh->abort = 1;
            report_status(p.status, SAGE_STATUS_TIMEOUT);
            return false;
        }
    }
}
// The same for a whole converged warp: every lane polls, so that the warp never splits over the answer.
template <typename S, typename P>
__device__ __forceinline__ bool mbar_wait_warp(uint64_t* bar, uint32_t parity, S* sh, const P& p) {
    if (__all_sync(0xffffffffu, mbar_try(bar, parity))) return true;
    return __all_sync(0xffffffffu, mbar_wait(bar, parity, sh, p));
}
// Used on the abort path only: gives up silently after the budget.
__device__ __forceinline__ void mbar_wait_quiet(uint64_t* bar, uint32_t parity, long long budget) {
    const long long t0 = clock64();
    while (!mbar_try(bar, parity) && clock64() - t0 < budget) {}
}

// ---- TMA ----------------------------------------------------------------------
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, int c0, int c1, int c2, int c3,
                                            uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
        ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void tma_load_5d(uint32_t dst, const CUtensorMap* map, int c0, int c1, int c2, int c3, int c4,
                                            uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, %6}], [%7];"
        ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(smem_u32(bar)) : "memory");
}

// ---- tcgen05 --------------------------------------------------------------------
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// One lane of a converged warp; the same lane every time for a full mask.
__device__ __forceinline__ bool elect_one() {
    uint32_t e;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(e));
    return e != 0;
}
// The helpers below are called by a whole converged warp, so that their operands stay in uniform registers, and
// carry the elected lane as a predicate of the instruction itself: a branch around it (`if (lane == 0)`) makes the
// compiler move every operand back into uniform registers first, 73 to 84 clocks per 128 x 128 x 16 MMA instead of
// the 64 that the tensor pipe needs (measured with eight P V and eight score MMAs per block).
__device__ __forceinline__ void tc_commit(uint32_t leader, uint64_t* bar) {
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %1, 0;\n\t"
                 "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}"
                 ::"r"(smem_u32(bar)), "r"(leader) : "memory");
}
// Shared-memory matrix descriptors are passed as their low word: the high word (kDescHi) is the same everywhere.
// D[tmem] (+)= A[smem desc] * B[smem desc]
template <uint32_t kHi, uint32_t kIdesc>
__device__ __forceinline__ void mma_ss(uint32_t leader, uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t acc) {
    asm volatile("{\n\t.reg .pred p, q;\n\t.reg .b64 da, db;\n\tsetp.ne.b32 p, %5, 0;\n\tsetp.ne.b32 q, %6, 0;\n\t"
                 "mov.b64 da, {%1, %3};\n\tmov.b64 db, {%2, %3};\n\t"
                 "@q tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p;\n\t}"
                 ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "n"(kHi), "n"(kIdesc), "r"(acc), "r"(leader) : "memory");
}
// D[tmem] (+)= A[tmem] * B[smem desc]
template <uint32_t kHi, uint32_t kIdesc>
__device__ __forceinline__ void mma_ts(uint32_t leader, uint32_t d_tmem, uint32_t a_tmem, uint32_t b_lo, uint32_t acc) {
    asm volatile("{\n\t.reg .pred p, q;\n\t.reg .b64 db;\n\tsetp.ne.b32 p, %5, 0;\n\tsetp.ne.b32 q, %6, 0;\n\t"
                 "mov.b64 db, {%2, %3};\n\t"
                 "@q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], db, %4, p;\n\t}"
                 ::"r"(d_tmem), "r"(a_tmem), "r"(b_lo), "n"(kHi), "n"(kIdesc), "r"(acc), "r"(leader) : "memory");
}
// 32 lanes x 32 consecutive 32-bit columns: thread i of the warp gets lane (quadrant*32 + i)
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t* r) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
          "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]),
          "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]),
          "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31]) : "memory");
}
__device__ __forceinline__ void tmem_st2(uint32_t taddr, uint32_t a, uint32_t b) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%0], {%1, %2};" ::"r"(taddr), "r"(a), "r"(b) : "memory");
}
// two columns, waited for
__device__ __forceinline__ void tmem_ld2(uint32_t taddr, uint32_t& a, uint32_t& b) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];" : "=r"(a), "=r"(b) : "r"(taddr) : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
// The wait, tied to the registers that a load filled: what uses them stays behind it, other loads need not.
__device__ __forceinline__ void tmem_wait_ld_of(uint32_t (&r)[32]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]),
                   "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]), "+r"(r[16]),
                   "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]), "+r"(r[24]),
                   "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
                 :: "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ float fast_exp2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}

// Shared-memory matrix descriptor (sm_100 format): start address, leading / stride byte
// offsets in 16-byte units, version 1, 128-byte swizzle.  Low word: address and leading offset;
// high word: stride offset (1024 bytes between 8-row groups everywhere here), version, swizzle.
__device__ __forceinline__ uint32_t desc_lo(uint32_t saddr, uint32_t lbo_bytes) {
    return ((saddr & 0x3FFFFu) >> 4) | ((lbo_bytes >> 4) << 16);
}
constexpr uint32_t kDescHi = (1024u >> 4) | (1u << 14) | (2u << 29);
// Instruction descriptor, kind::f16: D fp32, A and B bf16, M = 128, N as given.
constexpr uint32_t idesc_f16(uint32_t n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((n >> 3) << 17) | ((128u >> 4) << 24);
}
constexpr uint32_t kIdescQK = idesc_f16(kStepKeys);              // S (128 x 128): A, B both K-major
constexpr uint32_t kIdescPV = idesc_f16(kHeadDim) | (1u << 16);  // O (128 x 128): B (= V) MN-major

__device__ __forceinline__ float max3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// ---- packed fp32 pairs (one instruction works on two values) ----
__device__ __forceinline__ uint64_t f2_pack(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void f2_unpack(uint64_t v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t f2_fma(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t f2_add(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// 2^x for a pair of x <= ~8 on the FMA and integer pipes instead of the special-function unit
// (which delivers only 16 results per clock per SM and would otherwise bound the softmax):
// x = n + f with n = round(x), f in [-0.5, 0.5]; 2^f by a cubic fitted to 7.5e-5 relative error
// (well below the 2^-9 rounding of the bf16 probabilities); n goes straight into the exponent bits.
// Inputs are clamped to [-125, 127], so that 2^x never leaves the normal range; -inf does not come here.
__device__ __forceinline__ void exp2_pair_fma(uint64_t x2, float& p0, float& p1) {
    constexpr float kMagic = 12582912.f;             // 1.5 * 2^23: adding it leaves round(x) in the low mantissa bits
    float x0, x1;
    f2_unpack(x2, x0, x1);
    x2 = f2_pack(fminf(fmaxf(x0, -125.f), 127.f), fminf(fmaxf(x1, -125.f), 127.f));
    const uint64_t t2 = f2_add(x2, f2_pack(kMagic, kMagic));
    const uint64_t n2 = f2_add(t2, f2_pack(-kMagic, -kMagic));
    const uint64_t f2 = f2_fma(n2, f2_pack(-1.f, -1.f), x2);
    uint64_t q2 = f2_fma(f2, f2_pack(0.0551716685f, 0.0551716685f), f2_pack(0.2426111251f, 0.2426111251f));
    q2 = f2_fma(q2, f2, f2_pack(0.6932609677f, 0.6932609677f));
    q2 = f2_fma(q2, f2, f2_pack(0.9999280572f, 0.9999280572f));
    float t0, t1, q0, q1;
    f2_unpack(t2, t0, t1);
    f2_unpack(q2, q0, q1);
    p0 = __uint_as_float(__float_as_uint(q0) + (__float_as_uint(t0) << 23));
    p1 = __uint_as_float(__float_as_uint(q1) + (__float_as_uint(t1) << 23));
}

#ifndef SAGE_EXP2_FMA_PAIRS
#define SAGE_EXP2_FMA_PAIRS 1       // of every 8 column pairs, evaluated on the FMA pipe instead of the SFU
#endif

// Maximum of 32 raw scores of one query row, folded into mx.
__device__ __forceinline__ void max_chunk(const uint32_t* sr, float& mx) {
    float m4[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        float mq = max3(__uint_as_float(sr[q * 8]), __uint_as_float(sr[q * 8 + 1]), __uint_as_float(sr[q * 8 + 2]));
        mq = max3(mq, __uint_as_float(sr[q * 8 + 3]), __uint_as_float(sr[q * 8 + 4]));
        mq = max3(mq, __uint_as_float(sr[q * 8 + 5]), __uint_as_float(sr[q * 8 + 6]));
        m4[q] = fmaxf(mq, __uint_as_float(sr[q * 8 + 7]));
    }
    mx = fmaxf(max3(mx, m4[0], m4[1]), fmaxf(m4[2], m4[3]));
}

// 32 score columns of one query row: p = 2^(s * scale + neg_ref) packed to 16 bf16 pairs, and the
// fp32 sums of p in `acc`.  kEmu of every 8 column pairs take the FMA-pipe exp2.  Written in stages
// over the chunk so that neighbouring instructions are independent.
template <int kEmu>
__device__ __forceinline__ void exp_chunk(const uint32_t* sr, float scale, float neg_ref, uint32_t* pk,
                                          uint64_t (&acc)[2]) {
    const uint64_t scale2 = f2_pack(scale, scale), nref2 = f2_pack(neg_ref, neg_ref);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        uint64_t x2[8];
#pragma unroll
        for (int i = 0; i < 8; ++i)
            x2[i] = f2_fma(f2_pack(__uint_as_float(sr[16 * h + 2 * i]), __uint_as_float(sr[16 * h + 2 * i + 1])), scale2, nref2);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            float p0, p1;
            if (i < kEmu) {
                exp2_pair_fma(x2[i], p0, p1);
            } else {
                float x0, x1;
                f2_unpack(x2[i], x0, x1);
                p0 = fast_exp2(x0);
                p1 = fast_exp2(x1);
            }
            x2[i] = f2_pack(p0, p1);
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) acc[i & 1] = f2_add(acc[i & 1], x2[i]);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            float p0, p1;
            f2_unpack(x2[i], p0, p1);
            pk[8 * h + i] = pack_bf16(p0, p1);
        }
    }
}

// Which of 32 keys a row may see, one bit each; jt0: tree slot of the first of them (< 0 = prefix).  Tree slot jt is visible
// iff it is an ancestor of (or is) the row's node, a bit of anc; positions past the tree are never visible.
__device__ __forceinline__ uint32_t visible_keys(int jt0, uint64_t anc) {
    if (jt0 >= 0) return jt0 < 64 ? (uint32_t)(anc >> jt0) : 0u;
    return jt0 <= -32 ? 0xffffffffu : ((1u << -jt0) - 1u) | ((uint32_t)anc << -jt0);
}
// Scores of keys this row may not see become -inf.  (With the test made key by key from the 64-bit set, the step that
// holds the tree took 11 000 to 13 000 clocks instead of 2 000: as much as five other steps, in every segment.)
__device__ __forceinline__ void mask_chunk(uint32_t* sr, int jt0, uint64_t anc) {
    const uint32_t vis = visible_keys(jt0, anc);
#pragma unroll
    for (int i = 0; i < 32; ++i)
        if (!(vis & (1u << i))) sr[i] = 0xff800000u;      // -inf
}

// The 128 scores of a step for one query row, TMEM -> registers: four loads, one wait.
__device__ __forceinline__ void load_scores(uint32_t s_taddr, uint32_t (&sr)[128]) {
    tmem_ld32(s_taddr, *reinterpret_cast<uint32_t(*)[32]>(&sr[0]));
    tmem_ld32(s_taddr + 32, *reinterpret_cast<uint32_t(*)[32]>(&sr[32]));
    tmem_ld32(s_taddr + 64, *reinterpret_cast<uint32_t(*)[32]>(&sr[64]));
    tmem_ld32(s_taddr + 96, *reinterpret_cast<uint32_t(*)[32]>(&sr[96]));
    tmem_wait_ld();
}

// O row *= alpha for the 32 rows of this warp (rare: only when a row maximum grew by more than 2^8).
static __device__ __noinline__ void rescale_o_rows(uint32_t o_taddr, float alpha) {
#pragma unroll 1
    for (int c = 0; c < 4; ++c) {
        uint32_t orr[32];
        tmem_ld32(o_taddr + c * 32, orr);
        tmem_wait_ld();
#pragma unroll
        for (int i = 0; i < 32; ++i) orr[i] = __float_as_uint(__uint_as_float(orr[i]) * alpha);
        tmem_st32(o_taddr + c * 32, orr);
    }
    tmem_wait_st();
}

// 4 x 4 transpose of 16-byte pieces among each four lanes: lane 4a + b gives its piece i to lane 4a + i and ends up with
// piece b of rows 4a .. 4a + 3 in v[0 .. 3].
__device__ __forceinline__ void transpose4(uint4 (&v)[4], int lane) {
    auto swap = [&](uint4& keep_lo, uint4& keep_hi, bool hi, int mask) {      // lanes with `hi` send the first, the others the second
        uint4 mine = hi ? keep_lo : keep_hi;
        mine.x = __shfl_xor_sync(0xffffffffu, mine.x, mask);
        mine.y = __shfl_xor_sync(0xffffffffu, mine.y, mask);
        mine.z = __shfl_xor_sync(0xffffffffu, mine.z, mask);
        mine.w = __shfl_xor_sync(0xffffffffu, mine.w, mask);
        if (hi) keep_lo = mine;
        else keep_hi = mine;
    };
    const bool h1 = lane & 1, h2 = lane & 2;
    swap(v[0], v[1], h1, 1);
    swap(v[2], v[3], h1, 1);
    swap(v[0], v[2], h2, 2);
    swap(v[1], v[3], h2, 2);
}

__device__ __forceinline__ void pack_rows(const uint32_t (&o)[32], float f, uint4 (&v)[4]) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
        v[i] = make_uint4(pack_bf16(__uint_as_float(o[8 * i + 0]) * f, __uint_as_float(o[8 * i + 1]) * f),
                          pack_bf16(__uint_as_float(o[8 * i + 2]) * f, __uint_as_float(o[8 * i + 3]) * f),
                          pack_bf16(__uint_as_float(o[8 * i + 4]) * f, __uint_as_float(o[8 * i + 5]) * f),
                          pack_bf16(__uint_as_float(o[8 * i + 6]) * f, __uint_as_float(o[8 * i + 7]) * f));
}

// ---- schedule: items, ranges, segments ---------------------------------------------------
struct Item { int n0, N, L, steps, rp; };     // steps == 0: the sequence is skipped (and reported); rp: row pairs

__device__ __forceinline__ Item load_item(const AttnParams& p, int b, int* err) {
    Item it;
    it.n0 = p.node_offsets[b];
    it.N = p.node_offsets[b + 1] - it.n0;
    it.L = p.seq_len[b];
    it.steps = 0;
    it.rp = 0;
    if (it.N < 1 || it.N > SAGE_MAX_NODES || it.n0 < 0 || it.n0 + it.N > p.sum_nodes) {
        *err = SAGE_STATUS_BAD_TREE;
        return it;
    }
    if (it.L < 0 || (long long)it.L + it.N > (long long)p.max_pages * kPageSize) {
        *err = SAGE_STATUS_BAD_PAGE;
        return it;
    }
    it.steps = (it.L + it.N + kStepKeys - 1) / kStepKeys;
    it.rp = (it.N * p.G + kRowsPerCta - 1) / kRowsPerCta;
    return it;
}

// The work of a launch, laid end to end in steps: layer by layer, unit by unit, sequence by sequence.  With one CTA per
// gang a unit is a KV head.  With two (some tree of the batch has more than 256 rows) it is a KV head for the trees of
// two row pairs, one per CTA, and two KV heads, one per CTA, for the trees of one: both CTAs always have rows to work on
// (with a head per unit throughout, one of them idled through the small trees of a mixed batch).
// Called by a whole warp; the same answer in every CTA.
__device__ __forceinline__ Plan make_plan(const AttnParams& p, int lane, int* err) {
    Plan pl;
    int mx = 0, all = 0, big = 0;
    for (int b0 = 0; b0 < p.batch; b0 += 32) {
        Item it{0, 0, 0, 0, 0};
        if (b0 + lane < p.batch) it = load_item(p, b0 + lane, err);
        if (it.steps) mx = max(mx, it.N * p.G);
        const int cost = it.steps ? it.steps + kItemExtra : 0;
        all += cost;
        big += it.rp > 1 ? cost : 0;
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    pl.steps_all = __reduce_add_sync(0xffffffffu, all);
    pl.steps_big = __reduce_add_sync(0xffffffffu, big);
    pl.n_rp = mx > kRowsPerCta ? 2 : 1;
    pl.heads_all = pl.n_rp == 2 ? (p.Hkv + 1) / 2 : p.Hkv;
    pl.steps_layer = (long long)pl.heads_all * pl.steps_all + (long long)(p.Hkv - pl.heads_all) * pl.steps_big;
    pl.one_tile = mx <= kRowTile;
    pl.W = pl.steps_layer * p.n_layers;
    const long long a = pl.W / kMinSteps;
    const int gangs = p.n_ctas / pl.n_rp;
    pl.n_act = a < 1 ? 1 : a < gangs ? (int)a : gangs;
    // (the number of items: trees of one and of two row pairs in a batch make it more, skipped sequences less)
    const long long items = (long long)p.n_layers * p.batch * (pl.steps_big == pl.steps_all ? p.Hkv : pl.heads_all);
    if (a > gangs && items < gangs && pl.W <= (kMinSteps + kItemExtra) * items) pl.n_act = (int)items;
    return pl;
}
// Where a gang's range begins, before locate has moved it out of an item's extra.  (32-bit division where the numbers allow it: the 64-bit
// one takes some hundred clocks.)
__device__ __forceinline__ long long gang_begin(const Plan& pl, int gang) {
    if (pl.W < (1 << 23)) return (unsigned)gang * (unsigned)pl.W / (unsigned)pl.n_act;      // gang <= 148 < 2^9
    return (long long)gang * pl.W / pl.n_act;
}
// Gang whose range holds position pos: the largest k with gang_begin(k) <= pos.
__device__ __forceinline__ int gang_of(const Plan& pl, long long pos) { return (int)(((pos + 1) * pl.n_act - 1) / pl.W); }

// Layer, unit, sequence and step inside it of position pos < W; whole warp.  The extra of an item lies behind its steps: a position there
// is moved to the start of the next item (which may be W; the place is then past the last layer).
__device__ __forceinline__ Place locate(const AttnParams& p, const Plan& pl, int lane, long long* position) {
    const long long pos = *position;
    Place at;
    unsigned r;
    if (pl.W < (1ll << 31)) {
        at.layer = (int)((unsigned)pos / (unsigned)pl.steps_layer);
        r = (unsigned)pos % (unsigned)pl.steps_layer;
    } else {
        at.layer = (int)(pos / pl.steps_layer);
        r = (unsigned)(pos % pl.steps_layer);
    }
    const unsigned first = (unsigned)pl.heads_all * (unsigned)pl.steps_all;
    const bool big_only = r >= first;
    if (big_only) r -= first;
    const unsigned per_unit = (unsigned)(big_only ? pl.steps_big : pl.steps_all);
    at.u = (int)(r / per_unit) + (big_only ? pl.heads_all : 0);
    const int off = (int)(r % per_unit);
    int run = 0, err = 0;
    at.b = p.batch;
    at.s0 = 0;
    for (int b0 = 0; b0 < p.batch; b0 += 32) {
        int s = 0;
        if (b0 + lane < p.batch) {
            const Item it = load_item(p, b0 + lane, &err);
            if (it.steps && (!big_only || it.rp > 1)) s = it.steps + kItemExtra;
        }
        int inc = s;
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += v;
        }
        const unsigned hit = __ballot_sync(0xffffffffu, run + inc > off);
        if (hit) {
            const int l = __ffs(hit) - 1;
            const int incl = __shfl_sync(0xffffffffu, inc, l), sl = __shfl_sync(0xffffffffu, s, l);
            at.b = b0 + l;
            at.s0 = off - (run + incl - sl);
            if (at.s0 >= sl - kItemExtra) {
                *position += sl - at.s0;
                at.s0 = 0;
                if (++at.b == p.batch) {
                    at.b = 0;
                    if (++at.u == p.Hkv) { at.u = 0; ++at.layer; }
                }
            }
            break;
        }
        run += __shfl_sync(0xffffffffu, inc, 31);
    }
    return at;
}
// Which 256 rows of a tree of two row pairs a gang member takes: alternates, so that the member with the smaller
// share of one tree (36 and 48 nodes leave 32 and 128 rows) has the larger one of the next.
__device__ __forceinline__ int row_pair_of(int member, int u, int b) { return (member + u + b) & 1; }

struct Seg { int layer, g, b, n0, N, L, s0, s1, steps, row0; bool at_range_begin; };   // g: KV head, row0: first row of this CTA

// Walks the segments of a CTA's range; every thread that needs them runs its own copy.
struct SegIter {
    int remaining;      // of the range, still to hand out (steps, and kItemExtra for each end of an item)
    int layer, u, b, s0;
    int n_rp, heads_all, member;
    bool fresh;         // nothing handed out yet
    __device__ __forceinline__ void init(const Shared* sh) {
        remaining = (int)(sh->range_end - sh->range_begin);
        layer = sh->first.layer;
        u = sh->first.u;
        b = sh->first.b;
        s0 = sh->first.s0;
        n_rp = sh->n_rp;
        heads_all = sh->heads_all;
        member = n_rp == 2 ? (blockIdx.x & 1) : 0;
        fresh = true;
    }
    __device__ __forceinline__ void next_sequence(const AttnParams& p) {
        s0 = 0;
        if (++b == p.batch) {
            b = 0;
            if (++u == p.Hkv) { u = 0; ++layer; }
        }
    }
    // The next segment that has rows for this CTA.  sg: the one before.
    __device__ __forceinline__ bool next(const AttnParams& p, Seg& sg) {
        while (remaining > 0 && layer < p.n_layers) {
            int err = 0;
            Item it;
            if (!fresh && b == sg.b) {                              // the sequence of the segment before: no need to load it
                it = Item{sg.n0, sg.N, sg.L, sg.steps, (sg.N * p.G + kRowsPerCta - 1) / kRowsPerCta};
            } else {
                it = load_item(p, b, &err);
            }
            if (it.steps == 0 || (u >= heads_all && it.rp < 2)) {
                next_sequence(p);
                continue;
            }
            const int s1 = (it.steps - s0 <= remaining) ? it.steps : s0 + remaining;      // (the range may end in the item's extra)
            const bool pair = n_rp == 2 && it.rp == 1;              // two heads of a small tree, one per CTA
            sg.layer = layer; sg.b = b;
            sg.g = pair ? 2 * u + member : u;
            sg.row0 = it.rp == 2 ? row_pair_of(member, u, b) * kRowsPerCta : 0;
            sg.n0 = it.n0; sg.N = it.N; sg.L = it.L;
            sg.s0 = s0; sg.s1 = s1; sg.steps = it.steps;
            sg.at_range_begin = fresh;
            fresh = false;
            remaining -= s1 - s0 + (s1 == it.steps ? kItemExtra : 0);
            if (s1 == it.steps) next_sequence(p);
            else s0 = s1;
            if (sg.g < p.Hkv) return true;
        }
        return false;
    }
};

// Query rows past the tree (one row tile): the tile's box reaches into the next sequence's rows, or into spare capacity.
// Nothing reads what these rows result in, but the tensor cores draw less power on zeros, and long launches run at the power limit:
// nine nodes in arrays of 64, 80 layers x 16k keys, 1035 -> 990 us.  Not for short segments, where it costs more than it saves.
// Called by the whole MMA warp.
constexpr int kClearMinSteps = 32;
__device__ __forceinline__ void clear_query_rows(const AttnParams& p, const Seg& sg, uint8_t* sQ, int live, int lane) {
    if (live >= kRowTile || sg.s1 - sg.s0 < kClearMinSteps || sg.n0 + sg.N >= p.sum_nodes) return;      // (past sum_nodes TMA fills in zeros)
    const uint32_t q = smem_u32(sQ) + ((lane >> 3) & 1) * kQHalfBytes + (lane >> 4) * 128 + (lane & 7) * 16;
#pragma unroll 4
    for (int r = live + (live & 1); r < kRowTile; r += 2)           // two rows a turn (an odd row at the front may stay)
        asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(q + r * 128), "r"(0) : "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");    // generic writes -> visible to the MMA unit
    __syncwarp();
}

// Set-up of a CTA, side by side: warp 0 works out the CTA's range of steps, another warp allocates tensor memory (512
// columns: nothing else is resident), a thread prepares the barriers and fetches the tensor maps.  kOneTile: which trees the
// kernel is for.  Returns false (and holds no tensor memory) when there is nothing to do.
template <bool kOneTile>
__device__ __forceinline__ bool set_up(const AttnParams& p, Shared* sh, int warp, int lane, const CUtensorMap& qmap,
                                       const CUtensorMap& kmap, const CUtensorMap& vmap, uint32_t* tmem_out) {
    if (warp == 0) {
        int err = 0;
        const Plan pl = make_plan(p, lane, &err);
        if (err) report_status(p.status, err);
        const int gang = pl.n_rp == 2 ? blockIdx.x >> 1 : blockIdx.x;
        long long begin = 0, end = 0;
        Place at{0, 0, 0, 0};
        if (pl.W > 0 && gang < pl.n_act && pl.one_tile == (kOneTile ? 1 : 0)) {
            begin = gang_begin(pl, gang);
            end = gang_begin(pl, gang + 1);
            if (end > begin) at = locate(p, pl, lane, &begin);
        }
        if (lane == 0) {
            sh->range_begin = begin; sh->range_end = end;
            if (end <= begin && pl.one_tile == (kOneTile ? 1 : 0)) p.cuts[blockIdx.x] = Cut{pl.n_rp};
            sh->plan = pl;
            sh->first = at;
            sh->n_rp = pl.n_rp; sh->heads_all = pl.heads_all;
        }
    } else if (warp == 8) {
        if (lane == 0) {
            asm volatile("prefetch.tensormap [%0];" ::"l"(&kmap) : "memory");
            asm volatile("prefetch.tensormap [%0];" ::"l"(&vmap) : "memory");
            asm volatile("prefetch.tensormap [%0];" ::"l"(&qmap) : "memory");
            for (int i = 0; i < kRing; ++i) { mbar_init(&sh->kv_full[i], 1); mbar_init(&sh->kv_done[i], 1); }
            for (int t = 0; t < 2; ++t) {
                mbar_init(&sh->s_full[t], 1);
                mbar_init(&sh->p_full[t], 4);               // one arrival per softmax warp
                mbar_init(&sh->o_full[t], 1);
            }
            mbar_init(&sh->epi_done, 8);                    // one arrival per softmax warp
            for (int i = 0; i < 8; ++i) (&sh->eflag[0][0])[i] = 0;
            mbar_init(&sh->q_free, 1);
            mbar_init(&sh->drain, 1);
            mbar_init(&sh->q_ready, 1);
            sh->abort = 0;
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
    } else if (warp == 9) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(&sh->tmem_base)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sh->tmem_base;
    if (sh->range_end <= sh->range_begin) {                 // uniform: nothing to do
        if (warp == 9) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
        return false;
    }
    *tmem_out = tmem;
    if (warp == 11 && lane == 0) {                          // (idle otherwise) what the merge kernel has to know of the range's beginning
        const Plan pl = sh->plan;
        const Place at = sh->first;
        Cut c{pl.n_rp, at.s0, at.layer, at.u, at.b};
        if (at.s0 > 0) {
            int err = 0;
            const Item it = load_item(p, at.b, &err);
            const long long a = sh->range_begin - at.s0;    // position of the item's first step
            c.n0 = it.n0; c.N = it.N; c.steps = it.steps;
            c.k_first = gang_of(pl, a);
            c.k_last = gang_of(pl, a + it.steps - 1);
            c.mid = gang_begin(pl, c.k_first) < a - kItemExtra;      // (more than the extra of the item in front lies before it)
        }
        p.cuts[blockIdx.x] = c;
    }
    return true;
}

// Teardown: every role is past its last TMEM access.
__device__ __forceinline__ void tear_down(uint32_t tmem, int warp) {
    tc_fence_before();
    __syncthreads();
    if (warp == 9) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
}

// The opt-in to large dynamic shared memory is a per-device attribute of a kernel.  Internal linkage: two
// kernels of the same type in different translation units must not share the flags (one such kernel per unit).
template <int kBytes, typename K>
static bool allow_shared_memory(K kernel) {
    static std::atomic<bool> done[64];
    int dev = 0;
    if (!succeeded(cudaGetDevice(&dev)) || dev < 0 || dev >= 64) return false;
    if (!done[dev].load(std::memory_order_acquire)) {
        if (!succeeded(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kBytes))) return false;
        done[dev].store(true, std::memory_order_release);
    }
    return true;
}

}  // namespace stream
}  // namespace sage
