// Streaming schedule of the tree attention for trees of up to 128 query rows per KV head: both slots belong to the same
// rows and take the even and the odd steps of a segment (see attention_stream.cuh); the merge of cut items for both kernels
// of the schedule, and their launch.
#include "attention_stream.cuh"

namespace sage {
namespace stream {

constexpr int kLag = 2;                        // ring step i carries the K tile of step i and the V tile of step i - kLag
constexpr int kVStages = 3;                    // V tiles in flight
constexpr int kDepth = 3;                      // ring steps the copies run ahead of the MMAs

// =========================== TMA producer (one thread) ===========================
__device__ __forceinline__ void produce(const AttnParams& p, Shared* sh, uint8_t* smem, const CUtensorMap& qmap,
                                        const CUtensorMap& kmap, const CUtensorMap& vmap) {
    uint8_t* sQ = smem;
    uint8_t* sK = sQ + kQTileBytes;
    uint8_t* sV = sK + kKStages * kTileBytes;
    SegIter it;
    it.init(sh);
    Seg sg;
    int rc = 0, kslot = 0, vslot = 0, nq = 0;    // ring steps issued, slots of the next K and V tile, query loads issued
    bool ok = !p.producer_off;
    while (ok && it.next(p, sg)) {
        const int32_t* pages = p.page_table + (size_t)sg.b * p.max_pages;
        const int n_pages_seq = (sg.L + sg.N + kPageSize - 1) / kPageSize;
        const int n = sg.s1 - sg.s0;
        // the segment's query tiles, once the previous segment's score MMAs have read theirs
        if (nq > 0 && !mbar_wait(&sh->q_free, (nq - 1) & 1, sh, p)) break;
        mbar_expect_tx(&sh->q_ready, kQTileBytes);
        for (int h = 0; h < 2; ++h)
            tma_load_5d(smem_u32(sQ + h * kQHalfBytes), &qmap, h * 64, 0, sg.g, sg.n0, sg.layer, &sh->q_ready);
        ++nq;
        int ids[kLag + 1][2] = {}, npg[kLag + 1] = {};       // pages of steps i, i - 1, ...
        for (int i = 0; i < n + kLag; ++i) {
            const int j = sg.s0 + i;
#pragma unroll
            for (int d = kLag; d > 0; --d) {
                ids[d][0] = ids[d - 1][0]; ids[d][1] = ids[d - 1][1]; npg[d] = npg[d - 1];
            }
            // page ids of step j (checked: they become TMA coordinates)
            npg[0] = 0;
            if (i < n) {
                npg[0] = (2 * j + 1 < n_pages_seq) ? 2 : 1;
#pragma unroll
                for (int pi = 0; pi < 2; ++pi) {
                    if (pi < npg[0]) {
                        ids[0][pi] = pages[2 * j + pi];
                        if (ids[0][pi] < 0 || ids[0][pi] >= p.n_pages) {
                            report_status(p.status, SAGE_STATUS_BAD_PAGE);
                            ids[0][pi] = 0;
                        }
                    }
                }
            }
            const int npv = i >= kLag ? npg[kLag] : 0;
            // the tiles that ring step rc - kDepth used are free once its MMAs have finished
            if (rc >= kDepth && !mbar_wait(&sh->kv_done[(rc - kDepth) % kRing], ((rc - kDepth) / kRing) & 1, sh, p)) { ok = false; break; }
            uint64_t* full = &sh->kv_full[rc % kRing];
            mbar_expect_tx(full, (npg[0] + npv) * 2 * kPageHalfBytes);
            if (i < n) {
#pragma unroll
                for (int pi = 0; pi < 2; ++pi)
                    if (pi < npg[0])
                        for (int h = 0; h < 2; ++h)
                            tma_load_4d(smem_u32(sK + kslot * kTileBytes + h * kTileHalfBytes + pi * kPageHalfBytes), &kmap, h * 64, 0,
                                        ids[0][pi] * p.Hkv + sg.g, sg.layer, full);
                kslot = kslot == kKStages - 1 ? 0 : kslot + 1;
            }
            if (i >= kLag) {
#pragma unroll
                for (int pi = 0; pi < 2; ++pi)
                    if (pi < npv)
                        for (int h = 0; h < 2; ++h)
                            tma_load_4d(smem_u32(sV + vslot * kTileBytes + h * kTileHalfBytes + pi * kPageHalfBytes), &vmap, h * 64, 0,
                                        ids[kLag][pi] * p.Hkv + sg.g, sg.layer, full);
                vslot = vslot == kVStages - 1 ? 0 : vslot + 1;
            }
            ++rc;
        }
    }
    if (sh->abort) {
        // drain: every issued copy must land before the CTA may exit
        for (int n = max(0, rc - kDepth); n < rc; ++n)
            mbar_wait_quiet(&sh->kv_full[n % kRing], (n / kRing) & 1, p.wait_cycles);
        if (nq > 0) mbar_wait_quiet(&sh->q_ready, (nq - 1) & 1, p.wait_cycles);
    }
}

// =========================== MMA issuer (one warp) ===========================
// One warp issues for both slots, in blocks [P V of step i - kLag, scores of step i] of a slot: a slot's block
// runs on the tensor pipe while the other slot's warpgroup is in its softmax, and the blocks never interleave
// (two issuers would finish both slots' scores at the same moment and leave the pipe idle during both
// softmaxes).  The whole warp walks the loop and the elected lane is a predicate of each MMA (see mma_ss).
__device__ __forceinline__ void issue(const AttnParams& p, Shared* sh, uint8_t* smem, uint32_t tmem, int lane) {
    const uint32_t leader = elect_one() ? 1u : 0u;
    const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);      // (a broadcast: known to be the same in all lanes)
    // descriptors differ only in their 14-bit start-address field (bytes >> 4); shared memory ends below 256 KB
    const uint32_t dq = desc_lo(smem_u32(smem), 16);
    const uint32_t dk = desc_lo(smem_u32(smem + kQTileBytes), 16);
    const uint32_t dv = desc_lo(smem_u32(smem + kQTileBytes + kKStages * kTileBytes), kTileHalfBytes);
    auto issue_qk = [&](int t, int slot) {
        // S_t = Q_t K^T: 8 slices of K = 16 over d = 128 (4 per 64-wide half)
        const uint32_t dks = dk + ((slot * kTileBytes) >> 4);
        const uint32_t s_tmem = tm + t * 128;
#pragma unroll
        for (int ks = 0; ks < 8; ++ks)
            mma_ss<kDescHi, kIdescQK>(leader, s_tmem, dq + (((ks >> 2) * kQHalfBytes + (ks & 3) * 32) >> 4),
                                      dks + (((ks >> 2) * kTileHalfBytes + (ks & 3) * 32) >> 4), ks > 0 ? 1u : 0u);
    };
    auto issue_pv = [&](int t, int slot, bool first) {
        // O_t += P_t V: 8 slices of K = 16 keys; P in TMEM (8 columns per slice), V MN-major
        const uint32_t dvs = dv + ((slot * kTileBytes) >> 4);
        const uint32_t s_tmem = tm + t * 128, o_tmem = tm + 256 + t * 128;
#pragma unroll
        for (int ks = 0; ks < 8; ++ks)
            mma_ts<kDescHi, kIdescPV>(leader, o_tmem, s_tmem + ks * 8, dvs + ((ks * 2048) >> 4), (first && ks == 0) ? 0u : 1u);
    };
    SegIter it;
    it.init(sh);
    Seg sg;
    int rc = 0, kslot = 0, vslot = 0, nseg = 0;     // ring steps consumed, slots of the next K and V tile; segments started
    int np[2] = {0, 0};                             // steps of each slot whose probabilities were consumed
    bool ok = true;
    // The loop holds as few synchronisation instructions as the protocol allows: one wait and one commit
    // per ring step for the tiles, one of each per slot.
    while (ok && it.next(p, sg)) {
        const int n = __shfl_sync(0xffffffffu, sg.s1 - sg.s0, 0);
        ok = mbar_wait_warp(&sh->q_ready, nseg & 1, sh, p);
        if (ok) clear_query_rows(p, sg, smem, sg.N * p.G, lane);
        for (int i = 0; ok && i < n + kLag; ++i) {
            ok = mbar_wait_warp(&sh->kv_full[rc % kRing], (rc / kRing) & 1, sh, p);
            if (!ok) break;
            const int t = i & 1;
            if (i >= kLag) {
                // (the warpgroup zeroed the V rows past the end of the sequence before it arrived)
                ok = mbar_wait_warp(&sh->p_full[t], np[t] & 1, sh, p);
                if (!ok) break;
                ++np[t];
                // the segment's first P V products overwrite both accumulators, which the softmax warps
                // read in the epilogue of the segment before
                if (i == kLag && nseg > 0) {
                    ok = mbar_wait_warp(&sh->epi_done, (nseg - 1) & 1, sh, p);
                    if (!ok) break;
                }
                tc_fence_after();
                issue_pv(t, vslot, i < 2 * kLag);
                if (i >= n) tc_commit(leader, &sh->o_full[t]);          // the slot's last step of the segment
            }
            if (i < n) {
                issue_qk(t, kslot);
                tc_commit(leader, &sh->s_full[t]);
            }
            tc_commit(leader, &sh->kv_done[rc % kRing]);
            ++rc;
            if (i < n) kslot = (kslot == kKStages - 1) ? 0 : kslot + 1;
            if (i >= kLag) vslot = (vslot == kVStages - 1) ? 0 : vslot + 1;
            if (i == n - 1) tc_commit(leader, &sh->q_free);             // the segment's last score MMAs read the query tiles
        }
        ++nseg;
    }
    if (!ok) {
        // abort: everything this warp has issued must retire before the TMEM and the tiles go away
        tc_commit(leader, &sh->drain);
        mbar_wait_quiet(&sh->drain, 0, p.wait_cycles);
    }
    __syncwarp();
}

// =========================== softmax ===========================
// One step of one query row per thread: scores of S_t -> probabilities (bf16, over the first 64 columns of S_t), running
// reference and sum.  first: nothing has been accumulated yet; masked: the step reaches into the tree part (or past
// the end), jt0: tree slot of its first key.  row_ok: the row exists (others, spare rows or the next sequence's, have no say in
// how the rows beside them are computed).
__device__ __forceinline__ void softmax_step(uint32_t s_taddr, uint32_t o_taddr, float scale, bool row_ok, bool first, bool masked,
                                             int jt0, uint64_t anc, float& m_ref, float& l_sum) {
    uint32_t sr[128];
    // Probabilities are taken against the row's reference of the steps before, so a step need not look for its maximum
    // first.  It shows in the step's sum whether the reference still serves; the first step of a segment, steps with
    // masked scores and steps whose sum has grown to kMaxSum go through the maximum.
    bool by_max = masked || first, outgrown = false;
    if (!by_max) {
        uint64_t acc[2] = {0ull, 0ull};
        tmem_ld32(s_taddr, *reinterpret_cast<uint32_t(*)[32]>(&sr[0]));
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            tmem_wait_ld_of(*reinterpret_cast<uint32_t(*)[32]>(&sr[32 * c]));
            if (c < 3) tmem_ld32(s_taddr + 32 * (c + 1), *reinterpret_cast<uint32_t(*)[32]>(&sr[32 * (c + 1)]));
            exp_chunk<SAGE_EXP2_FMA_PAIRS>(sr + 32 * c, scale, -m_ref, sr + 16 * c, acc);
        }
        float sum_a, sum_b;
        f2_unpack(f2_add(acc[0], acc[1]), sum_a, sum_b);
        const float sum = sum_a + sum_b;
        outgrown = !(sum < kMaxSum);
        by_max = __any_sync(0xffffffffu, row_ok && outgrown);
        if (!by_max) l_sum += sum;
    }
    if (by_max) {
        load_scores(s_taddr, sr);
        if (masked) {
#pragma unroll
            for (int c = 0; c < 4; ++c) mask_chunk(sr + 32 * c, jt0 + 32 * c, anc);
        }
        float mx = -INFINITY;
#pragma unroll
        for (int c = 0; c < 4; ++c) max_chunk(sr + 32 * c, mx);
        // the reference moves where the row's sum asked for it, else only when its maximum grew by more than 2^8
        const float m_cand = mx * scale;
        const bool grow = m_cand > m_ref + (outgrown ? 0.f : 8.0f);
        float alpha = 1.0f;
        if (grow) {
            alpha = fast_exp2(m_ref - m_cand);              // 0 when m_ref was -inf
            m_ref = m_cand;
        }
        // O_t *= alpha.  The P V product of the step before has finished: the scores of this step were
        // issued after it, and their completion is what this warp waited for above.
        if (!first && __any_sync(0xffffffffu, grow)) rescale_o_rows(o_taddr, alpha);
        const float neg_ref = (m_ref == -INFINITY) ? 0.f : -m_ref;
        uint64_t acc[2] = {0ull, 0ull};
#pragma unroll
        for (int c = 0; c < 4; ++c) exp_chunk<0>(sr + 32 * c, scale, neg_ref, sr + 16 * c, acc);   // may hold -inf
        float sum_a, sum_b;
        f2_unpack(f2_add(acc[0], acc[1]), sum_a, sum_b);
        l_sum = l_sum * alpha + (sum_a + sum_b);
    }
    // (chunk c of 32 scores has left its 16 words of bf16 pairs at sr[16c ..])
    uint32_t* pk = sr;
    tmem_st32(s_taddr, pk);                 // P over the first 64 columns of S_t
    tmem_st32(s_taddr + 32, pk + 32);
    tmem_wait_st();
    tc_fence_before();
}

// Four lanes exchange the 64 bytes of output that each has of its row, so that a store instruction writes 64 contiguous
// bytes of eight rows instead of 16 bytes of 32.  v: 32 columns of the row as bf16; col: the first one; row0: row of lane 0.
__device__ __forceinline__ void store_rows(const AttnParams& p, const Seg& sg, uint4 (&v)[4], int row0, int M, int col, int lane) {
    transpose4(v, lane);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int R = row0 + (lane & ~3) + i;
        if (R < M) {
            const size_t row = (size_t)(sg.n0 + (R >> p.g_shift)) * p.Hq + sg.g * p.G + (R & (p.G - 1));
            reinterpret_cast<uint4*>(p.out + ((size_t)sg.layer * p.sum_nodes * p.Hq + row) * kHeadDim + col)[lane & 3] = v[i];
        }
    }
}
// 32 columns of a partial result; po: the thread's place in the first column quad.
__device__ __forceinline__ void store_partial(float4* po, const uint32_t (&o)[32]) {
#pragma unroll
    for (int i = 0; i < 8; ++i)
        po[i * kRowsPerCta] = make_float4(__uint_as_float(o[4 * i]), __uint_as_float(o[4 * i + 1]), __uint_as_float(o[4 * i + 2]),
                                          __uint_as_float(o[4 * i + 3]));
}

// The two slots combined, this warpgroup taking the output columns [64t, 64t + 64) of both accumulators.
// Returns false when the CTA is aborting.
__device__ __forceinline__ bool finish_slots(const AttnParams& p, Shared* sh, const Seg& sg, uint32_t tmem, uint32_t lane_base, int t, int q,
                                             int r, int lane, bool has1, uint32_t eseq, float m_ref, float l_sum) {
    const int M = sg.N * p.G;
    // 64 columns of both accumulators, 32 at a time
    const uint32_t o0 = tmem + lane_base + 256 + 64 * t, o1 = o0 + 128;
    uint32_t oa[32], ob[32];
    tmem_ld32(o0, oa);
    if (has1) tmem_ld32(o1, ob);
    tmem_wait_ld();
    // The row's (reference, sum) of this slot goes to the other warpgroup through two columns of O_t
    // that this thread has just read and nobody else reads: columns 64t and 64t + 1.
    tmem_st2(tmem + lane_base + 256 + 128 * t + 64 * t, __float_as_uint(m_ref), __float_as_uint(l_sum));
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    tc_fence_before();
    __syncwarp();
    if (lane == 0) {
        __threadfence_block();
        sh->eflag[t][q] = eseq;
    }
    // bounded wait for the partner warp (same rows, other slot)
    volatile uint32_t* flag = &sh->eflag[1 - t][q];
    bool seen = (*flag == eseq);
    if (!seen) {
        const long long t0 = clock64();
        while (true) {
#pragma unroll 1
            for (int k = 0; k < 64 && !seen; ++k) seen = (*flag == eseq);
            if (seen || sh->abort) break;
            if (clock64() - t0 > p.wait_cycles) {
                sh->abort = 1;
                report_status(p.status, SAGE_STATUS_TIMEOUT);
                break;
            }
        }
    }
    if (!__all_sync(0xffffffffu, seen)) return false;
    tc_fence_after();
    uint32_t pm, pl;
    tmem_ld2(tmem + lane_base + 256 + (1 - t) * 128 + 64 * (1 - t), pm, pl);
    const float m_o = __uint_as_float(pm), l_o = __uint_as_float(pl);
    // weights of the two slots under the common reference (a slot without visible keys has l = 0)
    const float m_all = fmaxf(l_sum > 0.f ? m_ref : -INFINITY, l_o > 0.f ? m_o : -INFINITY);
    const float w_me = l_sum > 0.f ? fast_exp2(m_ref - m_all) : 0.f;
    const float w_ot = l_o > 0.f ? fast_exp2(m_o - m_all) : 0.f;
    const float l_all = l_sum * w_me + l_o * w_ot;
    const bool whole = (sg.s0 == 0 && sg.s1 == sg.steps);
    // factors of O_0 and O_1: the slot weights, and 1 / l for a finished row
    const float inv = whole ? ((l_all > 0.f) ? 1.0f / l_all : 0.f) : 1.0f;
    const float f0 = (t == 0 ? w_me : w_ot) * inv, f1 = has1 ? (t == 0 ? w_ot : w_me) * inv : 0.f;
    const size_t slot = (size_t)blockIdx.x * 2 + (sg.at_range_begin ? 0 : 1);
    float4* po = p.part_o + (slot * (kHeadDim / 4) + 16 * t) * kRowsPerCta + r;
    if (!whole && t == 0 && r < M) p.part_ml[slot * kRowsPerCta + r] = make_float2(m_all, l_all);
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        if (c == 1) {
            tmem_ld32(o0 + 32, oa);
            if (has1) tmem_ld32(o1 + 32, ob);
            tmem_wait_ld();
        }
#pragma unroll
        for (int i = 0; i < 32; ++i) {
            float v = __uint_as_float(oa[i]) * f0;
            if (has1) v = fmaf(__uint_as_float(ob[i]), f1, v);
            oa[i] = __float_as_uint(v);
        }
        if (whole) {
            uint4 v[4];
            pack_rows(oa, 1.0f, v);
            store_rows(p, sg, v, r - lane, M, 64 * t + c * 32, lane);
        } else if (r < M) {
            store_partial(po + c * 8 * kRowsPerCta, oa);
        }
    }
    return true;
}

// Warpgroup t owns slot t; one thread per query row.
__device__ __forceinline__ void softmax(const AttnParams& p, Shared* sh, uint8_t* smem, uint32_t tmem, int t, int q, int r, int lane) {
    uint8_t* sV = smem + kQTileBytes + kKStages * kTileBytes;
    const uint32_t lane_base = (uint32_t)(q * 32) << 16;            // r: row inside the tile == TMEM lane, q: its quadrant
    const uint32_t s_taddr = tmem + lane_base + t * 128;
    const uint32_t o_taddr = tmem + lane_base + 256 + t * 128;
    // A step needs all registers for its scores: where the warp is in its range, and what only the epilogue needs of the
    // segment, waits in shared memory (as spilled registers it went to L2 and back, see the kernel).
    struct Parked { SegIter it; Seg sg; };
    static_assert(sizeof(Parked) <= sizeof(sh->parked[0]), "parked state outgrew its place");
    Parked* parked = reinterpret_cast<Parked*>(sh->parked[t * 4 + q]);
    if (lane == 0) {
        SegIter it;
        it.init(sh);
        parked->it = it;
        parked->sg.b = -1;
    }
    int nsteps = 0, nseg = 0, nseg1 = 0;            // steps this slot has been through; segments; those with work for the slot (for slot 1, alternating)
    int vc0 = 0;                                    // V tiles of the CTA before the current segment
    int anc_b = -1;                                 // the sequence that anc belongs to
    uint64_t anc = 0;
    bool ok = true;
    while (ok) {
        __syncwarp();
        Seg sg = parked->sg;
        {
            SegIter it = parked->it;
            if (!it.next(p, sg)) break;
            __syncwarp();
            if (lane == 0) { parked->it = it; parked->sg = sg; }
            __syncwarp();
        }
        const int M = sg.N * p.G, n = sg.s1 - sg.s0;
        const bool row_ok = r < M;
        const bool warp_live = q * 32 < M;
        if (sg.b != anc_b) {
            anc_b = sg.b;
            anc = 0;
        }
        if (sg.s1 * kStepKeys > sg.L && row_ok && anc == 0) {
            // the segment reaches the tree part: this row's ancestor bitset (the G rows of a node
            // walk the same parent chain, at most N - 1 loads deep; kept for the sequence's next heads and layers)
            const int node = r >> p.g_shift;
            bool bad = false;
            anc = ancestor_bits(p.parent + sg.n0, sg.N, node, &bad);
            if (bad) { report_status(p.status, SAGE_STATUS_BAD_TREE); anc = 1ull << node; }
        }
        float m_ref = -INFINITY, l_sum = 0.f;
        for (int i = t; i < n; i += 2) {
            const int j = sg.s0 + i;
            ok = mbar_wait_warp(&sh->s_full[t], nsteps & 1, sh, p);
            if (!ok) break;
            ++nsteps;
            const int valid = sg.L + sg.N - j * kStepKeys;      // keys of this step that exist
            if (valid < kStepKeys) {
                // V rows past the end of the sequence may hold anything (a missing second page was not even
                // copied): zero them so that 0 * V stays 0.  Each warp of the warpgroup takes a quarter of
                // the rows; the writes are ordered before this warp's arrival, which the P V product waits for.  The V tile of step s0 + i lands with ring
                // step i + kLag of the segment.
                const int rcv = vc0 + (nseg + 1) * kLag + i;    // (a segment of n steps takes n + kLag ring steps)
                ok = mbar_wait_warp(&sh->kv_full[rcv % kRing], (rcv / kRing) & 1, sh, p);
                if (!ok) break;
                uint8_t* vb = sV + ((vc0 + i) % kVStages) * kTileBytes;
                for (int c = q * 32 + lane; c < (kStepKeys - valid) * 16; c += 128) {
                    const int vr = valid + c / 16, ch = c % 16;
                    *reinterpret_cast<uint4*>(vb + (ch >> 3) * kTileHalfBytes + vr * 128 + ((ch & 7) << 4)) = make_uint4(0, 0, 0, 0);
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            }
            // (a warp none of whose 32 rows exists keeps the barrier protocol going and leaves the scores of these
            // rows, which are zero, as they are; their outputs are never stored)
            if (warp_live) {
                tc_fence_after();
                const int jt0 = j * kStepKeys - sg.L;           // tree slot of the step's first key
                softmax_step(s_taddr, o_taddr, p.scale_log2, row_ok, i < 2, jt0 + kStepKeys > 0, jt0, anc, m_ref, l_sum);
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh->p_full[t]);
        }
        if (!ok) break;
        const bool has1 = n >= 2;                   // slot 1 took part in this segment
        ok = mbar_wait_warp(&sh->o_full[0], nseg & 1, sh, p);
        if (ok && has1) ok = mbar_wait_warp(&sh->o_full[1], nseg1 & 1, sh, p);
        ++nseg;
        if (has1) ++nseg1;
        vc0 += n;
        if (!ok) break;
        if (warp_live) {
            tc_fence_after();
            asm volatile("" ::: "memory");
            ok = finish_slots(p, sh, parked->sg, tmem, lane_base, t, q, r, lane, has1, (uint32_t)nseg, m_ref, l_sum);
            if (!ok) break;
        }
        tc_fence_before();                          // the next segment's first P V products overwrite O_0 and O_1
        __syncwarp();
        if (lane == 0) mbar_arrive(&sh->epi_done);
    }
}

__global__ void __launch_bounds__(kAttnThreads, 1)
tree_attention_alt_kernel(const AttnParams p, const __grid_constant__ CUtensorMap qmap,
                          const __grid_constant__ CUtensorMap kmap, const __grid_constant__ CUtensorMap vmap) {
    after_previous_kernel();
    extern __shared__ uint8_t smem_raw[];
    // 1024-byte alignment: the 128B swizzle pattern repeats every 1024 bytes of address
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    // the query tile [2 d-halves][128 rows][128 B], then rings of K and V tiles [2 d-halves][128 keys][128 B]
    Shared* sh = reinterpret_cast<Shared*>(smem + 7 * kTileBytes);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t tmem;
    if (!set_up<true>(p, sh, warp, lane, qmap, kmap, vmap, &tmem)) return;
    // Registers move from the copy / MMA warpgroup (which needs few) to the softmax warpgroups:
    // 4 warps give up 168 - 40 registers per thread, 8 warps take 232 - 168 each.  (With 72 and 216 the softmax
    // warps kept part of a segment's state in local memory, which L1 is too small to hold beside this much shared memory:
    // a segment's epilogue and the way to the next one took 12 000 clocks.  80 layers of 4k keys, 12 nodes: 288 -> 270 us,
    // and 254 with the state that is parked in shared memory.  The kernel for more rows spills nothing with 72 and 216.)
    if (warp >= 8) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");
        if (warp == 8) {
            if (lane == 0) produce(p, sh, smem, qmap, kmap, vmap);
        } else if (warp == 9) {
            issue(p, sh, smem, tmem, lane);
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 232;");
        softmax(p, sh, smem, tmem, warp >> 2, warp & 3, tid & 127, lane);
    }
    tear_down(tmem, warp);
}

// Merge of the items that a range boundary cut into segments.  Only a boundary between two gangs' ranges can cut an
// item, so the grid holds kMergeParts blocks per boundary and CTA of a gang.  A block is told which item its boundary falls into by the
// gang behind it (Cut) and leaves if the boundary coincides with the item's start; the blocks of all boundaries inside the item share
// its output columns, and combine the item's segments: which of a gang's two partial slots holds one follows from the positions.  One
// thread per row.  The kernel is a chain of latencies at the end of a launch, so all that an item of two segments (the usual one) needs is
// asked for at once.  Blocks that made the plan, looked their item up and read the sums first, one after the other, took four times the
// code: sixteen ragged sequences of 1k to 8k keys 151 -> 145 us, sixteen of up to 4k and 12 nodes 62.7 -> 57.7, a layer of forty 98 -> 90.
// (Warps that finish a cut item themselves when the next gang's part is already there: 146, the reading only moves.)
constexpr int kMergeParts = 4;
__global__ void __launch_bounds__(kRowsPerCta, 4) attention_merge_kernel(AttnParams p) {
    after_previous_kernel();
    const int row = threadIdx.x;
    const int n_rp = p.cuts[blockIdx.x].n_rp;
    const Cut c1 = p.cuts[min((int)blockIdx.x + 1, p.n_ctas - 1)], c2 = p.cuts[min((int)blockIdx.x + 2, p.n_ctas - 1)];
    const Cut c = n_rp == 2 ? c2 : c1;
    const int k_cut = blockIdx.x / n_rp + 1;            // boundary between gang k_cut - 1 and gang k_cut
    if ((int)blockIdx.x + n_rp >= p.n_ctas || c.s0 == 0) return;        // no such boundary, or it falls between two items
    const int member = blockIdx.x % n_rp;
    const int part = (k_cut - 1 - c.k_first) * kMergeParts + blockIdx.y, parts = (c.k_last - c.k_first) * kMergeParts;
    if (part >= kHeadDim / 16) return;
    Item it{c.n0, c.N, 0, c.steps, (c.N * p.G + kRowsPerCta - 1) / kRowsPerCta};
    const bool pair = n_rp == 2 && it.rp == 1;
    const int g = pair ? 2 * c.u + member : c.u;
    const int R = row + (it.rp == 2 ? row_pair_of(member, c.u, c.b) * kRowsPerCta : 0);
    if (g >= p.Hkv || R >= it.N * p.G) return;
    auto slot_of = [&](int k) { return (k * n_rp + member) * 2 + (k == c.k_first && c.mid ? 1 : 0); };
    const size_t orow = (size_t)(it.n0 + (R >> p.g_shift)) * p.Hq + g * p.G + (R & (p.G - 1));
    uint4* out = reinterpret_cast<uint4*>(p.out + ((size_t)c.layer * p.sum_nodes * p.Hq + orow) * kHeadDim);
    const bool two = c.k_last == c.k_first + 1;
    float mx = -INFINITY;
    if (!two) {
        for (int k0 = c.k_first; k0 <= c.k_last; k0 += 4) {
            float2 ml[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) ml[u] = p.part_ml[slot_of(min(k0 + u, c.k_last)) * kRowsPerCta + row];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (ml[u].y > 0.f) mx = fmaxf(mx, ml[u].x);
        }
    }
#pragma unroll 1
    for (int q0 = part * 4; q0 < kHeadDim / 4; q0 += parts * 4) {      // 16 output columns
        const float4* po = p.part_o + (size_t)q0 * kRowsPerCta + row;
        float lsum = 0.f;
        float4 acc[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int k0 = c.k_first; k0 <= c.k_last; k0 += 2) {
            float2 ml[2];
            float4 v[2][4];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int slot = slot_of(min(k0 + u, c.k_last));
                ml[u] = p.part_ml[slot * kRowsPerCta + row];
#pragma unroll
                for (int i = 0; i < 4; ++i) v[u][i] = po[((size_t)slot * (kHeadDim / 4) + i) * kRowsPerCta];
            }
            if (two) mx = fmaxf(ml[0].y > 0.f ? ml[0].x : -INFINITY, ml[1].y > 0.f ? ml[1].x : -INFINITY);
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                if (k0 + u <= c.k_last && ml[u].y > 0.f) {
                    const float w = exp2f(ml[u].x - mx);
                    lsum = fmaf(ml[u].y, w, lsum);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        acc[i].x = fmaf(w, v[u][i].x, acc[i].x); acc[i].y = fmaf(w, v[u][i].y, acc[i].y);
                        acc[i].z = fmaf(w, v[u][i].z, acc[i].z); acc[i].w = fmaf(w, v[u][i].w, acc[i].w);
                    }
                }
            }
        }
        const float inv = lsum > 0.f ? 1.f / lsum : 0.f;
#pragma unroll
        for (int h = 0; h < 2; ++h)
            out[q0 / 2 + h] = make_uint4(pack_bf16(acc[2 * h].x * inv, acc[2 * h].y * inv), pack_bf16(acc[2 * h].z * inv, acc[2 * h].w * inv),
                                         pack_bf16(acc[2 * h + 1].x * inv, acc[2 * h + 1].y * inv),
                                         pack_bf16(acc[2 * h + 1].z * inv, acc[2 * h + 1].w * inv));
    }
}

// The kernel for trees of more than one row tile (tree_attention_rows.cu).
bool launch_rows(const AttnParams& p, const CUtensorMap& qmap, const CUtensorMap& kmap, const CUtensorMap& vmap, cudaStream_t stream);

// ---- host side ------------------------------------------------------------------------------
static int row_pairs(int sum_nodes, int G) {
    const int n = sum_nodes < SAGE_MAX_NODES ? sum_nodes : SAGE_MAX_NODES;      // a tree has at most that many nodes
    return (n * G + kRowsPerCta - 1) / kRowsPerCta;
}

// Two partial slots (head and tail of its range) and the boundary in front of it per resident CTA, independent of the problem size.
size_t workspace_size(int n_ctas) { return (size_t)n_ctas * (2 * kRowsPerCta * (kHeadDim + 2) * sizeof(float) + sizeof(Cut)); }

int launch(int n_ctas, int n_layers, int n_pages, const int32_t* page_table, int max_pages_per_seq,
           const int32_t* seq_len, const int32_t* parent, const int32_t* node_offsets, int batch, int sum_nodes,
           int n_q_heads, int n_kv_heads, float sm_scale, void* out, void* ws, int32_t* status, long long wait_cycles,
           int producer_off, const CUtensorMap& qmap, const CUtensorMap& kmap, const CUtensorMap& vmap,
           cudaStream_t stream) {
    const int G = n_q_heads / n_kv_heads;
    AttnParams p{};
    p.n_rp = row_pairs(sum_nodes, G);
    p.n_ctas = (n_ctas / p.n_rp) * p.n_rp;          // whole gangs whatever the gang size turns out to be (1 or 2)
    p.out = (__nv_bfloat16*)out;
    p.part_o = (float4*)ws;
    p.part_ml = (float2*)((float*)ws + (size_t)n_ctas * 2 * kRowsPerCta * kHeadDim);
    p.cuts = (Cut*)(p.part_ml + (size_t)n_ctas * 2 * kRowsPerCta);
    p.page_table = page_table; p.seq_len = seq_len; p.parent = parent; p.node_offsets = node_offsets;
    p.status = status;
    p.n_layers = n_layers; p.batch = batch; p.sum_nodes = sum_nodes; p.n_pages = n_pages;
    p.max_pages = max_pages_per_seq; p.Hq = n_q_heads; p.Hkv = n_kv_heads; p.G = G; p.g_shift = __builtin_ctz(G);
    p.scale_log2 = sm_scale * 1.4426950408889634f;
    p.wait_cycles = wait_cycles;
    p.producer_off = producer_off;
    // Where the host's bound on the tree sizes (the capacity of the node arrays) allows both kernels, both are started and the
    // one that is not meant leaves after its plan; the usually shorter one first, since between the other and the merge it
    // would hold up the chain (69 instead of 63 us for a layer of 60 nodes at 16k).  One kernel with both inside saves
    // less than the compiler loses on the softmax loops (57 -> 61 us; as functions, 80 layers: 2.72 -> 2.80 ms).
    const int most_nodes = sum_nodes < SAGE_MAX_NODES ? sum_nodes : SAGE_MAX_NODES;
    if (!allow_shared_memory<kSmemBytes>(tree_attention_alt_kernel) ||
        !succeeded(sage::launch(tree_attention_alt_kernel, dim3(p.n_ctas), kAttnThreads, kSmemBytes, stream, 0, p, qmap, kmap, vmap)))
        return SAGE_ERR_CUDA;
    if (most_nodes * G > kRowTile && !launch_rows(p, qmap, kmap, vmap, stream)) return SAGE_ERR_CUDA;
    if (p.n_ctas <= 1) return SAGE_OK;
    // (a gang's boundaries and members: as many as CTAs; blocks that find no cut item leave)
    return launch_status(sage::launch(attention_merge_kernel, dim3(p.n_ctas, kMergeParts), kRowsPerCta, 0, stream, 0, p));
}

}  // namespace stream
}  // namespace sage
