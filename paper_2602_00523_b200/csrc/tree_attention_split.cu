// Tree-masked verification attention over a paged bf16 KV cache (Section 2.2;
// Algorithm 1, the target pass over all tree tokens; Section 3.3 Phase 2), sm_100a:
// the split schedule, used for launches too short to give every SM a long stream of work (single layers,
// short contexts).  tree_attention.cu holds the dispatch.
//
// Flash-decoding layout.  The N tree nodes x G query heads that share one KV head
// form M = N*G query rows (<= 512).  A CTA owns up to two 128-row tiles of them and
// one slice of the context (split-K).  The pipeline step is one 64-token page:
//   TMA      : query tiles; K and V pages -> 128B-swizzled shared memory, two 5-page rings, mbarriers
//   tcgen05  : S_t = Q_t K^T (128 x 64, fp32) into TMEM; one warp per row tile issues, the elected
//              lane being a predicate of each MMA
//   softmax  : one warpgroup per row tile, one thread per row: tcgen05.ld S, online
//              softmax in fp32 (log2 domain, lazy rescale), P -> bf16 back into TMEM
//   tcgen05  : O_t += P_t V with P as the TMEM A operand, V MN-major from shared memory
// Every row tile has two S buffers (even / odd pages), so the tensor pipe computes the
// scores of page j+1 while the warpgroup is busy with page j and never waits for it.
// TMEM map (512 columns): tile t owns S_t,even [128t, 128t+64), S_t,odd [128t+64, 128t+128)
// (P overlays the first 32 columns of its S buffer) and O_t [256+128t, 384+128t).
// Slices are merged by attention_split_merge_kernel.
// These launches are bound by fixed costs, so the way to the first MMA is kept short: tensor maps are fetched while the
// kernel before still runs, then one round of loads (the sequence's offsets and length) beside the allocation of tensor
// memory, the barriers, and the copies start; what is left of the set-up (page ids, ancestors) happens in the roles.  Before, query
// rows went through registers, partial results were written row by row (32 lines per store) and merged one warp per row:
// one layer, 8 KV heads of 8 queries, 60 nodes: 2k keys 23.5 -> 16.3 us, 16k keys 49.7 -> 39.8; 24 nodes, 16k: 37.3 -> 26.1.
// With two row tiles a page costs 1650 clocks, of which the tensor pipe is busy for 1280 (a 64-key score product costs 48
// clocks per K=16 slice where one of 128 keys costs 64); with one row tile HBM is the bound (6 TB/s).
// All waits are bounded: on expiry the CTA records SAGE_STATUS_TIMEOUT, drains its copies, frees its
// TMEM and returns.
#include "attention_stream.cuh"

namespace sage {
namespace split {

using namespace stream;

constexpr int kPageStages = 5;                 // depth of the K ring and of the V ring, in pages
constexpr int kPageBytes = kPageSize * kHeadDim * 2;        // one (page, head) tile: 16 KB
constexpr int kTablePages = 256;               // page tables of up to so many pages are read ahead of the lengths that say which part is needed
constexpr int kSplitThreads = 352;             // 2 softmax warpgroups + TMA warp + one MMA warp per row tile
constexpr uint32_t kIdescPageQK = idesc_f16(kPageSize);     // S (128 x 64): A, B both K-major

struct SplitParams {
    __nv_bfloat16* out;
    float4* part_o;    // [layer][split][32 column quads][sum_nodes*Hq rows]   unnormalised (rows of a KV head: 128 contiguous bytes)
    float2* part_ml;   // [layer][split][sum_nodes*Hq rows]                    (reference in log2 units, l)
    const int32_t* page_table;
    const int32_t* seq_len;
    const int32_t* parent;
    const int32_t* node_offsets;
    int32_t* status;
    int n_layers, batch, sum_nodes, n_pages, max_pages;
    int Hq, Hkv, G, g_shift, n_splits;     // G = 1 << g_shift query heads per KV head
    float scale_log2;  // sm_scale * log2(e)
    long long wait_cycles;     // budget of every on-device wait
    int producer_off;          // diagnostics: the TMA warp issues no copies (every consumer wait then runs out)
};

struct __align__(8) Barriers {
    uint64_t k_full[kPageStages], k_empty[kPageStages];
    uint64_t v_full[kPageStages], v_empty[kPageStages];
    uint64_t s_full[2][2];     // [row tile][page parity]: scores of a page are in TMEM
    uint64_t p_full[2][2];     // [row tile][page parity]: probabilities of a page are in TMEM (an arrival per warp that has rows)
    uint64_t pv_done[2];       // [row tile]: completes once per page, when its P V product has finished
    uint64_t o_full[2];        // [row tile]: every MMA of the tile has finished
    uint64_t q_ready;          // the query tiles are in shared memory
    uint32_t tmem_base;
    volatile int abort;
    int pages[kTablePages];    // the sequence's row of the page table, where that is no longer
};
constexpr int kSplitSmemBytes = 1024 /*align*/ + 2 * kQTileBytes + 2 * kPageStages * kPageBytes + (int)sizeof(Barriers);

// 64 scores of a page for one query row per thread: probabilities (bf16, over the first 32 columns of the S buffer), running
// reference and sum.  The reference works as in the streaming kernels (see softmax_step in tree_attention_alt.cu); pv_done / parity: the P V product of the page before.
__device__ __forceinline__ bool softmax_page(const SplitParams& p, Barriers* bars, uint64_t* pv_done, uint32_t pv_parity, uint32_t s_taddr,
                                             uint32_t o_taddr, bool row_ok, bool first, bool masked, int jt0, uint64_t anc,
                                             float& m_ref, float& l_sum) {
    uint32_t sr[64];
    bool by_max = masked || first, outgrown = false;
    if (!by_max) {
        uint64_t acc[2] = {0ull, 0ull};
        tmem_ld32(s_taddr, *reinterpret_cast<uint32_t(*)[32]>(&sr[0]));
        tmem_ld32(s_taddr + 32, *reinterpret_cast<uint32_t(*)[32]>(&sr[32]));
        tmem_wait_ld();
#pragma unroll
        for (int c = 0; c < 2; ++c) exp_chunk<SAGE_EXP2_FMA_PAIRS>(sr + 32 * c, p.scale_log2, -m_ref, sr + 16 * c, acc);
        float sum_a, sum_b;
        f2_unpack(f2_add(acc[0], acc[1]), sum_a, sum_b);
        const float sum = sum_a + sum_b;
        outgrown = !(sum < kMaxSum);
        by_max = __any_sync(0xffffffffu, row_ok && outgrown);
        if (!by_max) l_sum += sum;
    }
    if (by_max) {
        tmem_ld32(s_taddr, *reinterpret_cast<uint32_t(*)[32]>(&sr[0]));
        tmem_ld32(s_taddr + 32, *reinterpret_cast<uint32_t(*)[32]>(&sr[32]));
        tmem_wait_ld();
        if (masked) {
            mask_chunk(sr, jt0, anc);
            mask_chunk(sr + 32, jt0 + 32, anc);
        }
        float mx = -INFINITY;
        max_chunk(sr, mx);
        max_chunk(sr + 32, mx);
        const float m_cand = mx * p.scale_log2;
        const bool grow = m_cand > m_ref + (outgrown ? 0.f : 8.0f);
        float alpha = 1.0f;
        if (grow) {
            alpha = fast_exp2(m_ref - m_cand);              // 0 when m_ref was -inf
            m_ref = m_cand;
        }
        if (!first && __any_sync(0xffffffffu, grow)) {
            // O_t *= alpha, once the P V product of the page before has finished
            if (!__all_sync(0xffffffffu, mbar_wait(pv_done, pv_parity, bars, p))) return false;
            tc_fence_after();
            rescale_o_rows(o_taddr, alpha);
        }
        const float neg_ref = (m_ref == -INFINITY) ? 0.f : -m_ref;
        uint64_t acc[2] = {0ull, 0ull};
#pragma unroll
        for (int c = 0; c < 2; ++c) exp_chunk<0>(sr + 32 * c, p.scale_log2, neg_ref, sr + 16 * c, acc);   // may hold -inf
        float sum_a, sum_b;
        f2_unpack(f2_add(acc[0], acc[1]), sum_a, sum_b);
        l_sum = l_sum * alpha + (sum_a + sum_b);
    }
    tmem_st32(s_taddr, sr);                                 // P over the first 32 columns of this S buffer
    tmem_wait_st();
    tc_fence_before();
    return true;
}

__global__ void __launch_bounds__(kSplitThreads, 1)
tree_attention_split_kernel(const SplitParams p, const __grid_constant__ CUtensorMap qmap, const __grid_constant__ CUtensorMap kmap,
                            const __grid_constant__ CUtensorMap vmap) {
    extern __shared__ uint8_t smem_raw[];
    // 1024-byte alignment: the 128B swizzle pattern repeats every 1024 bytes of address
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* sQ = smem;                                 // [2 tiles][2 d-halves][128 rows][128 B]
    uint8_t* sK = smem + 2 * kQTileBytes;               // [kPageStages][2 d-halves][64 keys][128 B]
    uint8_t* sV = sK + kPageStages * kPageBytes;        // [kPageStages][2 d-halves][64 keys][128 B]
    Barriers* bars = reinterpret_cast<Barriers*>(sV + kPageStages * kPageBytes);

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int split = blockIdx.x, rpair = blockIdx.y;
    const int g = blockIdx.z % p.Hkv;
    const int b = (blockIdx.z / p.Hkv) % p.batch;
    const int layer = blockIdx.z / (p.Hkv * p.batch);

    // before the kernel in front has finished: nothing here touches global memory
    if (warp == 8 && lane == 0) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(&kmap) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&vmap) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&qmap) : "memory");
    }
    after_previous_kernel();
    // Not earlier: held while this block waits for the kernel in front, the tensor memory would be missing to a block of that
    // kernel (any kernel, of the caller's too) that shares the SM and asks for its own only after it has let this one start.
    if (warp == 9) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(&bars->tmem_base)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    const int n0 = p.node_offsets[b];
    const int N = p.node_offsets[b + 1] - n0;
    const int L = p.seq_len[b];
    // The whole row of the page table in the same round of loads, not the slice's part in a second one once the length is known (one
    // layer of ten nodes at 2k keys 9.18 -> 8.94 us, 60 nodes 16.0 -> 15.8, 15 nodes at 627 keys 9.42 -> 9.02, 24 at 4k 14.8 -> 14.5).  A prefix
    // of 16k keys and any tree have 257 pages: reading 320 ahead instead of 256 measured the same.
    const bool table = p.max_pages <= kTablePages;
    if (warp == 8 && table) {
        const int32_t* pages = p.page_table + (size_t)b * p.max_pages;
        int ids[kTablePages / 32];
#pragma unroll
        for (int i = 0; i < kTablePages / 32; ++i)
            if (lane + 32 * i < p.max_pages) ids[i] = pages[lane + 32 * i];
#pragma unroll
        for (int i = 0; i < kTablePages / 32; ++i)
            if (lane + 32 * i < p.max_pages) bars->pages[lane + 32 * i] = ids[i];
    }
    const bool bad_tree = N < 1 || N > SAGE_MAX_NODES || n0 < 0 || n0 + N > p.sum_nodes;
    const bool bad_page = !bad_tree && (L < 0 || L + N > p.max_pages * kPageSize);
    const int T = L + N;
    const int M = N * p.G;
    const bool live = !bad_tree && !bad_page && rpair * kRowsPerCta < M;
    const int n_rtiles = (M - rpair * kRowsPerCta > kRowTile) ? 2 : 1;
    if (tid == 0) {
        if (bad_tree || bad_page) report_status(p.status, bad_tree ? SAGE_STATUS_BAD_TREE : SAGE_STATUS_BAD_PAGE);
        for (int i = 0; i < kPageStages; ++i) {
            mbar_init(&bars->k_full[i], 1); mbar_init(&bars->k_empty[i], n_rtiles);   // one release per MMA warp
            mbar_init(&bars->v_full[i], 1); mbar_init(&bars->v_empty[i], n_rtiles);
        }
        for (int t = 0; t < 2; ++t) {
            const int warps = max(1, min(4, (M - rpair * kRowsPerCta - t * kRowTile + 31) / 32));      // of the tile, with rows of the tree
            for (int x = 0; x < 2; ++x) { mbar_init(&bars->s_full[t][x], 1); mbar_init(&bars->p_full[t][x], warps); }
            mbar_init(&bars->pv_done[t], 1);
            mbar_init(&bars->o_full[t], 1);
        }
        mbar_init(&bars->q_ready, 1);
        bars->abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = bars->tmem_base;
    if (!live) {                                        // uniform
        if (warp == 9) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
        return;
    }
    // this CTA's slice of the context, in pages
    const int n_pages_seq = (T + kPageSize - 1) / kPageSize;
    const int per_split = (n_pages_seq + p.n_splits - 1) / p.n_splits;
    const int pg_begin = split * per_split;
    const int ns = max(0, min(n_pages_seq, pg_begin + per_split) - pg_begin);        // pipeline steps

    if (warp == 8) {
        // =========================== TMA producer ===========================
        if (lane == 0 && ns > 0 && !p.producer_off) {
            const int32_t* pages = table ? bars->pages + pg_begin : p.page_table + (size_t)b * p.max_pages + pg_begin;
            mbar_expect_tx(&bars->q_ready, n_rtiles * kQTileBytes);
            for (int t = 0; t < n_rtiles; ++t)
                for (int h = 0; h < 2; ++h)
                    tma_load_5d(smem_u32(sQ + t * kQTileBytes + h * kQHalfBytes), &qmap, h * 64, 0, g,
                                n0 + ((rpair * kRowsPerCta + t * kRowTile) >> p.g_shift), layer, &bars->q_ready);
            int issued_k = 0, issued_v = 0;
            int next = pages[0];
            for (int j = 0; j < ns; ++j) {
                const int slot = j % kPageStages, use = j / kPageStages;
                int id = next;                          // (checked: it becomes a TMA coordinate)
                if (j + 1 < ns) next = pages[j + 1];
                if (id < 0 || id >= p.n_pages) {
                    report_status(p.status, SAGE_STATUS_BAD_PAGE);
                    id = 0;
                }
                const int c2 = id * p.Hkv + g;
                if (use > 0 && !mbar_wait(&bars->k_empty[slot], (use - 1) & 1, bars, p)) break;
                mbar_expect_tx(&bars->k_full[slot], kPageBytes);
                for (int h = 0; h < 2; ++h)
                    tma_load_4d(smem_u32(sK + slot * kPageBytes + h * kPageHalfBytes), &kmap, h * 64, 0, c2, layer, &bars->k_full[slot]);
                issued_k = j + 1;
                if (use > 0 && !mbar_wait(&bars->v_empty[slot], (use - 1) & 1, bars, p)) break;
                mbar_expect_tx(&bars->v_full[slot], kPageBytes);
                for (int h = 0; h < 2; ++h)
                    tma_load_4d(smem_u32(sV + slot * kPageBytes + h * kPageHalfBytes), &vmap, h * 64, 0, c2, layer, &bars->v_full[slot]);
                issued_v = j + 1;
            }
            if (bars->abort) {
                // drain: every issued copy must land before the CTA may exit
                mbar_wait_quiet(&bars->q_ready, 0, p.wait_cycles);
                for (int n = max(0, issued_k - kPageStages); n < issued_k; ++n)
                    mbar_wait_quiet(&bars->k_full[n % kPageStages], (n / kPageStages) & 1, p.wait_cycles);
                for (int n = max(0, issued_v - kPageStages); n < issued_v; ++n)
                    mbar_wait_quiet(&bars->v_full[n % kPageStages], (n / kPageStages) & 1, p.wait_cycles);
            }
        }
    } else if (warp >= 9) {
        // =========================== MMA issuers: warp 9 -> row tile 0, warp 10 -> row tile 1 ===========================
        // Broadcasts from lane 0 tell the compiler that these values are warp-uniform.
        const int t = __shfl_sync(0xffffffffu, warp - 9, 0);
        const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
        const int n = __shfl_sync(0xffffffffu, ns, 0);
        const int tiles = __shfl_sync(0xffffffffu, n_rtiles, 0);
        const int first_pos = __shfl_sync(0xffffffffu, pg_begin * kPageSize, 0);
        const uint32_t leader = elect_one() ? 1u : 0u;
        auto wait_all = [&](uint64_t* bar, uint32_t parity) { return mbar_wait_warp(bar, parity, bars, p); };
        // descriptors differ only in their 14-bit start-address field (bytes >> 4); shared memory ends below 256 KB
        const uint32_t dq = desc_lo(smem_u32(sQ) + t * kQTileBytes, 16);
        const uint32_t dk = desc_lo(smem_u32(sK), 16);
        const uint32_t dv = desc_lo(smem_u32(sV), kPageHalfBytes);
        const uint32_t s_tmem = tm + t * 128, o_tmem = tm + 256 + t * 128;
        auto issue_qk = [&](int x, int slot) {
            // S_t,x = Q_t K^T: 8 slices of K = 16 over d = 128 (4 per 64-wide half)
            const uint32_t dks = dk + ((slot * kPageBytes) >> 4);
            const uint32_t d = s_tmem + x * 64;
#pragma unroll
            for (int ks = 0; ks < 8; ++ks)
                mma_ss<kDescHi, kIdescPageQK>(leader, d, dq + (((ks >> 2) * kQHalfBytes + (ks & 3) * 32) >> 4),
                                              dks + (((ks >> 2) * kPageHalfBytes + (ks & 3) * 32) >> 4), ks > 0 ? 1u : 0u);
        };
        auto issue_pv = [&](int x, int slot, bool first) {
            // O_t += P_t,x V: 4 slices of K = 16 keys; P in TMEM (8 columns per slice), V MN-major
            const uint32_t dvs = dv + ((slot * kPageBytes) >> 4);
            const uint32_t a = s_tmem + x * 64;
#pragma unroll
            for (int ks = 0; ks < 4; ++ks)
                mma_ts<kDescHi, kIdescPV>(leader, o_tmem, a + ks * 8, dvs + ((ks * 2048) >> 4), (!first || ks > 0) ? 1u : 0u);
        };
        bool ok = n > 0 && t < tiles;
        if (ok) ok = wait_all(&bars->q_ready, 0);
        // prologue: scores of the first two pages
        for (int j = 0; ok && j < min(2, n); ++j) {
            ok = wait_all(&bars->k_full[j], 0);
            if (!ok) break;
            tc_fence_after();
            issue_qk(j, j);
            tc_commit(leader, &bars->s_full[t][j]);
            tc_commit(leader, &bars->k_empty[j]);
        }
        // The V page of step j and the K page of step j+2 are looked up one step ahead (`stage_inputs`),
        // while the softmax of the previous page is still running, so that only the wait for the
        // probabilities sits between the softmax and the MMAs that depend on it.
        auto stage_inputs = [&](int j) -> bool {
            if (j >= n) return true;
            const int vslot = j % kPageStages;
            if (!wait_all(&bars->v_full[vslot], (j / kPageStages) & 1)) return false;
            const int valid = min(kPageSize, T - first_pos - j * kPageSize);
            if (valid < kPageSize) {
                // rows past the end of the sequence may hold anything: zero them so that 0 * V stays 0
                // (both MMA warps write the same zeros; each orders its own writes before its own MMAs)
                uint8_t* vb = sV + vslot * kPageBytes;
                for (int c = lane; c < (kPageSize - valid) * 16; c += 32) {
                    const int r = valid + c / 16, ch = c % 16;
                    *reinterpret_cast<uint4*>(vb + (ch >> 3) * kPageHalfBytes + r * 128 + ((ch & 7) << 4)) = make_uint4(0, 0, 0, 0);
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
            }
            const int jn = j + 2;
            if (jn < n && !wait_all(&bars->k_full[jn % kPageStages], (jn / kPageStages) & 1)) return false;
            return true;
        };
        if (ok) ok = stage_inputs(0);
        for (int j = 0; ok && j < n; ++j) {
            const int x = j & 1, vslot = j % kPageStages;
            const int jn = j + 2, kslot = jn % kPageStages;
            ok = wait_all(&bars->p_full[t][x], (j >> 1) & 1);
            if (!ok) break;
            tc_fence_after();
            issue_pv(x, vslot, j == 0);
            tc_commit(leader, &bars->pv_done[t]);
            tc_commit(leader, &bars->v_empty[vslot]);
            if (jn < n) {
                // the scores of page j+2 reuse this S buffer: in pipe order after P V of page j
                issue_qk(x, kslot);
                tc_commit(leader, &bars->s_full[t][x]);
                tc_commit(leader, &bars->k_empty[kslot]);
            }
            ok = stage_inputs(j + 1);
        }
        if (t < tiles) tc_commit(leader, &bars->o_full[t]);     // arrives when every MMA of this tile has completed
        // abort: everything this warp has issued must retire before the TMEM and the tiles go away
        if (!ok && t < tiles && lane == 0) mbar_wait_quiet(&bars->o_full[t], 0, p.wait_cycles);
        __syncwarp();
    } else {
        // =========================== softmax warpgroups ===========================
        const int t = warp >> 2;                        // row tile of this warpgroup
        const int r = tid & 127;                        // row inside the tile == TMEM lane
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t s_taddr = tmem + lane_base + t * 128;
        const uint32_t o_taddr = tmem + lane_base + 256 + t * 128;
        const int row0 = rpair * kRowsPerCta + t * kRowTile;
        const int R = row0 + r;
        const bool row_ok = R < M;
        const int node = row_ok ? R >> p.g_shift : 0;
        const bool warp_live = row0 + (warp & 3) * 32 < M;
        uint64_t anc = 0;
        if ((pg_begin + ns) * kPageSize > L && row_ok) {
            // the slice reaches the tree part: this row's ancestor bitset (the G rows of a node walk the same
            // parent chain, at most N - 1 cached loads deep, while the first pages are on their way)
            bool bad = false;
            anc = ancestor_bits(p.parent + n0, N, node, &bad);
            if (bad) { report_status(p.status, SAGE_STATUS_BAD_TREE); anc = 1ull << node; }
        }
        float m_ref = -INFINITY, l_sum = 0.f;
        // A warp none of whose 32 rows exists takes no part: the probabilities of these rows stay what their scores were, and their outputs are never
        // stored.  (Left to keep the barriers going, three such warps polled beside the tile's one and held it up: nine sequences of 1.5k keys, 17
        // nodes x 8 queries 28.6 -> 25.5 us, 24 nodes, two warps of the second tile, 27.8 -> 26.6.)
        bool ok = t < n_rtiles && warp_live;
        for (int j = 0; ok && j < ns; ++j) {
            const int x = j & 1;
            ok = mbar_wait_warp(&bars->s_full[t][x], (j >> 1) & 1, bars, p);
            if (!ok) break;
            if (warp_live) {                                        // (always; told so, the compiler lays the loop out better: short launches 8.5 -> 8.3 us)
                tc_fence_after();
                const int jt0 = (pg_begin + j) * kPageSize - L;     // tree slot of the page's first key
                ok = softmax_page(p, bars, &bars->pv_done[t], (j - 1) & 1, s_taddr + x * 64, o_taddr, row_ok, j == 0, jt0 + kPageSize > 0, jt0, anc,
                                  m_ref, l_sum);
                if (!ok) break;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars->p_full[t][x]);
        }
        // ---- epilogue: O_t / l -> bf16 output, or unnormalised partials for the merge
        if (ok && ns > 0) ok = mbar_wait_warp(&bars->o_full[t], 0, bars, p);
        if (ok && warp_live) {
            tc_fence_after();
            const size_t rows_total = (size_t)p.sum_nodes * p.Hq;
            const size_t row = (size_t)(n0 + node) * p.Hq + g * p.G + (row_ok ? R & (p.G - 1) : 0);
            const size_t part = (size_t)layer * p.n_splits + split;
            const float inv = (l_sum > 0.f) ? 1.0f / l_sum : 0.f;
            if (p.n_splits > 1 && row_ok) p.part_ml[part * rows_total + row] = make_float2(m_ref, l_sum);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                uint32_t o[32];
                if (ns == 0) break;                     // (an empty slice: its l = 0 keeps the merge from reading more)
                tmem_ld32(o_taddr + c * 32, o);
                tmem_wait_ld();
                if (p.n_splits == 1) {
                    uint4 v[4];
                    pack_rows(o, inv, v);
                    transpose4(v, lane);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int Ri = R - lane + (lane & ~3) + i;
                        if (Ri < M) {
                            const size_t orow = (size_t)(n0 + (Ri >> p.g_shift)) * p.Hq + g * p.G + (Ri & (p.G - 1));
                            reinterpret_cast<uint4*>(p.out + ((size_t)layer * rows_total + orow) * kHeadDim + c * 32)[lane & 3] = v[i];
                        }
                    }
                } else if (row_ok) {
                    float4* po = p.part_o + (part * (kHeadDim / 4) + c * 8) * rows_total + row;
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        po[i * rows_total] = make_float4(__uint_as_float(o[4 * i]), __uint_as_float(o[4 * i + 1]), __uint_as_float(o[4 * i + 2]),
                                                         __uint_as_float(o[4 * i + 3]));
                }
            }
        }
    }
    tear_down(tmem, warp);
}

// Merge of the slices.  A block owns 32 rows (one per lane) and 32 of the 128 columns (four per warp): enough warps to
// keep the loads of a few hundred rows in flight on the whole chip.  The partial results are requested before the weights
// are known.  Up to eight slices (many rows, as the chip is then filled by few slices) every thread works out the weights
// of its row itself and the kernel stays small; more are shared among the warps through shared memory.
constexpr int kMaxSplits = 32;
template <int kMaxS>
__global__ void __launch_bounds__(256) attention_split_merge_kernel(const SplitParams p) {
    after_previous_kernel();
    constexpr bool kShare = kMaxS > 8;
    constexpr int kMl = kShare ? kMaxS / 8 : kMaxS;         // weights per thread
    constexpr int kBatch = kMaxS < 16 ? kMaxS : 16;         // slices in flight
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const size_t rows_total = (size_t)p.sum_nodes * p.Hq;
    const size_t row = (size_t)blockIdx.x * 32 + lane;
    const int layer = blockIdx.y, S = p.n_splits, quad = blockIdx.z * 8 + warp;
    const bool ok = row < rows_total && row < (size_t)p.node_offsets[p.batch] * p.Hq;   // rows past the live nodes were never written
    if (!__any_sync(0xffffffffu, ok)) return;               // the same for all warps
    const size_t r = ok ? row : (size_t)blockIdx.x * 32;
    const float2* ml = p.part_ml + (size_t)layer * S * rows_total + r;
    const float4* po = p.part_o + ((size_t)layer * S * (kHeadDim / 4) + quad) * rows_total + r;
    const size_t slice = (kHeadDim / 4) * rows_total;
    float2 m[kMl];
    float4 v[kBatch];
#pragma unroll
    for (int u = 0; u < kMl; ++u) {
        const int s = kShare ? warp + 8 * u : u;
        m[u] = s < S ? ml[(size_t)s * rows_total] : make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < kBatch; ++u)
        if (u < S) v[u] = po[u * slice];
    float mx = -INFINITY, lsum = 0.f;
#pragma unroll
    for (int u = 0; u < kMl; ++u)
        if (m[u].y > 0.f) mx = fmaxf(mx, m[u].x);
    __shared__ float s_max[kShare ? 8 : 1][32], s_sum[kShare ? 8 : 1][32], s_w[kShare ? kMaxS : 1][32];
    if constexpr (kShare) {
        s_max[warp][lane] = mx;
        __syncthreads();
#pragma unroll
        for (int u = 0; u < 8; ++u) mx = fmaxf(mx, s_max[u][lane]);
    }
#pragma unroll
    for (int u = 0; u < kMl; ++u) {
        const float w = m[u].y > 0.f ? exp2f(m[u].x - mx) : 0.f;
        lsum = fmaf(m[u].y, w, lsum);
        if constexpr (kShare) s_w[warp + 8 * u][lane] = w;
        else m[u].x = w;
    }
    if constexpr (kShare) {
        s_sum[warp][lane] = lsum;
        __syncthreads();
        lsum = 0.f;
#pragma unroll
        for (int u = 0; u < 8; ++u) lsum += s_sum[u][lane];
    }
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int s0 = 0; s0 < kMaxS; s0 += kBatch) {
        if (s0 > 0) {
            if (s0 >= S) break;
#pragma unroll
            for (int u = 0; u < kBatch; ++u)
                if (s0 + u < S) v[u] = po[(s0 + u) * slice];
        }
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            if (s0 + u >= S) break;
            float w;
            if constexpr (kShare) w = s_w[s0 + u][lane];
            else w = m[u].x;
            if (w > 0.f) {                                  // (else an empty slice: nothing was written)
                acc.x = fmaf(w, v[u].x, acc.x); acc.y = fmaf(w, v[u].y, acc.y);
                acc.z = fmaf(w, v[u].z, acc.z); acc.w = fmaf(w, v[u].w, acc.w);
            }
        }
    }
    if (!ok) return;
    const float inv = lsum > 0.f ? 1.f / lsum : 0.f;
    *reinterpret_cast<uint2*>(p.out + ((size_t)layer * rows_total + row) * kHeadDim + quad * 4) =
        make_uint2(pack_bf16(acc.x * inv, acc.y * inv), pack_bf16(acc.z * inv, acc.w * inv));
}

static int row_pairs_for(int sum_nodes, int G) {
    const int n = sum_nodes < SAGE_MAX_NODES ? sum_nodes : SAGE_MAX_NODES;      // a tree has at most that many nodes
    return (n * G + kRowsPerCta - 1) / kRowsPerCta;
}

// Slices of the context, down to a page each (512 keys, 60 nodes: 0.6 us less than with two pages at least, now 12.5).  One CTA
// is resident per SM; a wave of them takes what its pages take plus a fixed part (set-up, first copies, drain), worth about
// six pages (four and nine measure the same), and every slice costs the merge a little.
static double wave_cost(int n_sms, long blocks, int pages, int s) {
    return (double)((blocks * s + n_sms - 1) / n_sms) * (6 + (pages + s - 1) / s) + (s > 1 ? 4.0 + 0.25 * s : 0.0);
}
static int pick_splits(int n_sms, int n_layers, int batch, int n_kv_heads, int G, int max_pages, int sum_nodes) {
    const long base = (long)n_layers * batch * n_kv_heads * row_pairs_for(sum_nodes, G);
    const int s_max = max_pages < kMaxSplits ? max_pages : kMaxSplits;
    int best = 1;
    double best_cost = 0.0;
    for (int s = 1; s <= s_max; ++s) {
        const long waves = (base * s + n_sms - 1) / n_sms;
        if (s > 1 && waves > 4) break;                      // (the last wave matters little by then, partial results do)
        const double cost = wave_cost(n_sms, base, max_pages, s);
        if (s == 1 || cost < best_cost - 1e-9) { best_cost = cost; best = s; }
    }
    return best;
}

// What a launch takes, in pages of 64 keys, if its trees are of the average size (blocks for rows that a tree does not have leave at once).
double estimate(int n_sms, int n_layers, int batch, int sum_nodes, int n_q_heads, int n_kv_heads, int max_pages_per_seq) {
    const int G = n_q_heads / n_kv_heads;
    const int S = pick_splits(n_sms, n_layers, batch, n_kv_heads, G, max_pages_per_seq, sum_nodes);
    return wave_cost(n_sms, (long)n_layers * batch * n_kv_heads * (sum_nodes / batch * G > kRowsPerCta ? 2 : 1), max_pages_per_seq, S);
}

int slices(int n_sms, int n_layers, int batch, int sum_nodes, int n_q_heads, int n_kv_heads, int max_pages_per_seq) {
    return pick_splits(n_sms, n_layers, batch, n_kv_heads, n_q_heads / n_kv_heads, max_pages_per_seq, sum_nodes);
}

// Whether the merge is brought up while the split kernel runs.  Its blocks then settle on the multiprocessors that the split grid leaves
// free and do the whole merge there, so that pays only where they are few: with more than two for each such multiprocessor the merge is
// launched in order.  4 sequences of 8 query and 8 KV heads, mixed trees, 0.5k keys (128 split blocks, 168 merge blocks) 11.5 -> 9.9 us; 2 of
// 16 and 8, 24 nodes, 0.75k (96, 192) 11.8 -> 10.6; over 400 launches 0.96 to 0.93 of the time from two to twenty a multiprocessor, 1.02 where
// there is less than one, 0.997 where the split grid has more than one wave (left as it is).
bool merge_overlaps(int n_sms, int n_layers, int batch, int sum_nodes, int n_q_heads, int n_kv_heads, int S) {
    const long long blocks = (long long)S * row_pairs_for(sum_nodes, n_q_heads / n_kv_heads) * n_layers * batch * n_kv_heads;
    const long long merge_blocks = ((long long)sum_nodes * n_q_heads + 31) / 32 * n_layers * 4;
    return blocks > n_sms || merge_blocks <= 2 * (n_sms - blocks);
}

size_t workspace_size(int n_sms, int n_layers, int batch, int sum_nodes, int n_q_heads, int n_kv_heads, int max_pages_per_seq) {
    const int S = pick_splits(n_sms, n_layers, batch, n_kv_heads, n_q_heads / n_kv_heads, max_pages_per_seq, sum_nodes);
    if (S == 1) return 16;
    return (size_t)n_layers * S * sum_nodes * n_q_heads * (kHeadDim + 2) * sizeof(float);
}

// Arguments have been validated by sage_tree_attention.
int launch(int n_sms, int n_layers, int n_pages, const int32_t* page_table, int max_pages_per_seq,
           const int32_t* seq_len, const int32_t* parent, const int32_t* node_offsets, int batch, int sum_nodes,
           int n_q_heads, int n_kv_heads, float sm_scale, void* out, void* ws, int32_t* status, long long wait_cycles,
           int producer_off, const CUtensorMap& qmap, const CUtensorMap& kmap, const CUtensorMap& vmap, cudaStream_t stream) {
    const int G = n_q_heads / n_kv_heads;
    const int S = pick_splits(n_sms, n_layers, batch, n_kv_heads, G, max_pages_per_seq, sum_nodes);
    SplitParams p{};
    p.out = (__nv_bfloat16*)out;
    p.part_o = (float4*)ws;
    p.part_ml = S > 1 ? (float2*)((float*)ws + (size_t)n_layers * S * sum_nodes * n_q_heads * kHeadDim) : nullptr;
    p.page_table = page_table; p.seq_len = seq_len; p.parent = parent; p.node_offsets = node_offsets;
    p.status = status;
    p.n_layers = n_layers; p.batch = batch; p.sum_nodes = sum_nodes; p.n_pages = n_pages;
    p.max_pages = max_pages_per_seq; p.Hq = n_q_heads; p.Hkv = n_kv_heads; p.G = G; p.g_shift = __builtin_ctz(G); p.n_splits = S;
    p.scale_log2 = sm_scale * 1.4426950408889634f;
    p.wait_cycles = wait_cycles;
    p.producer_off = producer_off;
    const dim3 grid(S, row_pairs_for(sum_nodes, G), n_layers * batch * n_kv_heads);
    if (!allow_shared_memory<kSplitSmemBytes>(tree_attention_split_kernel) ||
        !succeeded(sage::launch(tree_attention_split_kernel, grid, kSplitThreads, kSplitSmemBytes, stream, 0, p, qmap, kmap, vmap)))
        return SAGE_ERR_CUDA;
    if (S == 1) return SAGE_OK;
    const size_t rows_total = (size_t)sum_nodes * n_q_heads;
    const dim3 mg((unsigned)((rows_total + 31) / 32), n_layers, 4);
    const auto merge = S <= 4 ? attention_split_merge_kernel<4> : S <= 8 ? attention_split_merge_kernel<8> : attention_split_merge_kernel<kMaxSplits>;
    if (!merge_overlaps(n_sms, n_layers, batch, sum_nodes, n_q_heads, n_kv_heads, S)) return launch_status(launch_in_order(merge, mg, 256, stream, p));
    return launch_status(sage::launch(merge, mg, 256, 0, stream, 0, p));
}

}  // namespace split
}  // namespace sage
