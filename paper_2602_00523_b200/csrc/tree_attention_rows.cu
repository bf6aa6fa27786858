// Streaming schedule of the tree attention for trees of more than 128 query rows per KV head: two row tiles per CTA,
// slot = row tile, so that K and V enter the SM once (see attention_stream.cuh).
#include "attention_stream.cuh"

namespace sage {
namespace stream {

constexpr int kVStages = 2;                    // V tiles in flight (ring steps in flight <= 2)

__global__ void __launch_bounds__(kAttnThreads, 1)
tree_attention_rows_kernel(const AttnParams p, const __grid_constant__ CUtensorMap qmap,
                           const __grid_constant__ CUtensorMap kmap, const __grid_constant__ CUtensorMap vmap) {
    after_previous_kernel();
    extern __shared__ uint8_t smem_raw[];
    // 1024-byte alignment: the 128B swizzle pattern repeats every 1024 bytes of address
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* sQ = smem;                                 // [2 tiles][2 d-halves][128 rows][128 B]
    uint8_t* sK = sQ + 2 * kQTileBytes;                 // [kKStages][2 d-halves][128 keys][128 B]
    uint8_t* sV = sK + kKStages * kTileBytes;           // [kVStages][2 d-halves][128 keys][128 B]
    Shared* sh = reinterpret_cast<Shared*>(sV + kVStages * kTileBytes);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t tmem;
    if (!set_up<false>(p, sh, warp, lane, qmap, kmap, vmap, &tmem)) return;

    // Registers move from the copy / MMA warpgroup (which needs few) to the softmax warpgroups:
    // 4 warps give up 168 - 72 registers per thread, 8 warps take 216 - 168 each.
    if (warp >= 8) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 72;");
    if (warp == 8) {
        // =========================== TMA producer ===========================
        if (lane == 0) {
            SegIter it;
            it.init(sh);
            Seg sg;
            // A segment of n steps takes n + 1 ring steps: ring step i carries the K tile of step s0 + i
            // (i < n) and the V tile of step s0 + i - 1 (i > 0), which is what the MMA warp consumes together
            // ([P V of the step before, scores of this step]); both land on one barrier.
            int rc = 0, kc = 0, vc = 0, nq = 0;          // ring steps, K tiles, V tiles, query loads issued so far
            bool ok = !p.producer_off;
            while (ok && it.next(p, sg)) {
                const int M = sg.N * p.G;
                const int n_rt = (M - sg.row0 > kRowTile) ? 2 : 1;
                const int32_t* pages = p.page_table + (size_t)sg.b * p.max_pages;
                const int n_pages_seq = (sg.L + sg.N + kPageSize - 1) / kPageSize;
                const int n = sg.s1 - sg.s0;
                // the segment's query tiles, once the previous segment's score MMAs have read theirs
                if (nq > 0 && !mbar_wait(&sh->q_free, (nq - 1) & 1, sh, p)) break;
                mbar_expect_tx(&sh->q_ready, n_rt * kQTileBytes);
                for (int t = 0; t < n_rt; ++t)
                    for (int h = 0; h < 2; ++h)
                        tma_load_5d(smem_u32(sQ + t * kQTileBytes + h * kQHalfBytes), &qmap, h * 64, 0, sg.g,
                                    sg.n0 + ((sg.row0 + t * kRowTile) >> p.g_shift), sg.layer, &sh->q_ready);
                ++nq;
                int ids_prev[2] = {0, 0}, npg_prev = 0;
                for (int i = 0; i <= n; ++i) {
                    const int j = sg.s0 + i;
                    // page ids of step j (checked: they become TMA coordinates)
                    int ids[2] = {0, 0}, npg = 0;
                    if (i < n) {
                        npg = (2 * j + 1 < n_pages_seq) ? 2 : 1;
                        for (int pi = 0; pi < npg; ++pi) {
                            ids[pi] = pages[2 * j + pi];
                            if (ids[pi] < 0 || ids[pi] >= p.n_pages) {
                                report_status(p.status, SAGE_STATUS_BAD_PAGE);
                                ids[pi] = 0;
                            }
                        }
                    }
                    // the tiles that ring step rc - 2 used are free once its MMAs have finished
                    if (rc >= 2 && !mbar_wait(&sh->kv_done[(rc - 2) % kRing], ((rc - 2) / kRing) & 1, sh, p)) { ok = false; break; }
                    uint64_t* full = &sh->kv_full[rc % kRing];
                    mbar_expect_tx(full, (npg + (i > 0 ? npg_prev : 0)) * 2 * kPageHalfBytes);
                    if (i < n) {
                        const int kslot = kc % kKStages;
                        for (int pi = 0; pi < npg; ++pi)
                            for (int h = 0; h < 2; ++h)
                                tma_load_4d(smem_u32(sK + kslot * kTileBytes + h * kTileHalfBytes + pi * kPageHalfBytes), &kmap,
                                            h * 64, 0, ids[pi] * p.Hkv + sg.g, sg.layer, full);
                        ++kc;
                    }
                    if (i > 0) {
                        const int vslot = vc % kVStages;
                        for (int pi = 0; pi < npg_prev; ++pi)
                            for (int h = 0; h < 2; ++h)
                                tma_load_4d(smem_u32(sV + vslot * kTileBytes + h * kTileHalfBytes + pi * kPageHalfBytes), &vmap,
                                            h * 64, 0, ids_prev[pi] * p.Hkv + sg.g, sg.layer, full);
                        ++vc;
                    }
                    ++rc;
                    ids_prev[0] = ids[0]; ids_prev[1] = ids[1]; npg_prev = npg;
                }
            }
            if (sh->abort) {
                // drain: every issued copy must land before the CTA may exit
                for (int n = max(0, rc - 2); n < rc; ++n)
                    mbar_wait_quiet(&sh->kv_full[n % kRing], (n / kRing) & 1, p.wait_cycles);
                if (nq > 0) mbar_wait_quiet(&sh->q_ready, (nq - 1) & 1, p.wait_cycles);
            }
        }
    } else if (warp == 9) {
        // =========================== MMA issuer ===========================
        // One warp issues for both row tiles, in blocks [P V of step j-1, scores of step j] per tile:
        // a tile's block runs on the tensor pipe while the other tile's warpgroup is in its softmax, and
        // the blocks of the two tiles never interleave (two issuers would finish both tiles' scores at
        // the same moment and leave the pipe idle during both softmaxes).  The whole warp walks the loop and
        // the elected lane is a predicate of each MMA (see mma_ss): 80 layers x 16k keys, 24 nodes: 1349 -> 1257 us.
        const uint32_t leader = elect_one() ? 1u : 0u;
        const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);      // (a broadcast: known to be the same in all lanes)
        // descriptors differ only in their 14-bit start-address field (bytes >> 4); shared memory ends below 256 KB
        const uint32_t dq = desc_lo(smem_u32(sQ), 16);
        const uint32_t dk = desc_lo(smem_u32(sK), 16);
        const uint32_t dv = desc_lo(smem_u32(sV), kTileHalfBytes);
        auto issue_qk = [&](int t, int slot) {
            // S_t = Q_t K^T: 8 slices of K = 16 over d = 128 (4 per 64-wide half)
            const uint32_t dqt = dq + ((t * kQTileBytes) >> 4);
            const uint32_t dks = dk + ((slot * kTileBytes) >> 4);
            const uint32_t s_tmem = tm + t * 128;
#pragma unroll
            for (int ks = 0; ks < 8; ++ks)
                mma_ss<kDescHi, kIdescQK>(leader, s_tmem, dqt + (((ks >> 2) * kQHalfBytes + (ks & 3) * 32) >> 4),
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
        int rc = 0, kslot = 0, vslot = 0, nq = 0;       // ring steps consumed, slots of the next K and V tile; segments started
        int np[2] = {0, 0};                             // steps of each row tile whose probabilities were consumed
        bool ok = true;
        // The loop holds as few synchronisation instructions as the protocol allows: one wait and one commit
        // per ring step for the tiles, one of each per row tile.
        while (ok && it.next(p, sg)) {
            const int n_rt = __shfl_sync(0xffffffffu, (sg.N * p.G - sg.row0 > kRowTile) ? 2 : 1, 0);
            const int n = __shfl_sync(0xffffffffu, sg.s1 - sg.s0, 0);
            ok = mbar_wait_warp(&sh->q_ready, nq & 1, sh, p);
            ++nq;
            // ring step i: the P V products of step i - 1 (when i > 0) and the scores of step i (when i < n)
            for (int i = 0; ok && i <= n; ++i) {
                ok = mbar_wait_warp(&sh->kv_full[rc % kRing], (rc / kRing) & 1, sh, p);
                if (!ok) break;
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                    if (t < n_rt) {
                        if (i > 0) {
                            // (the warpgroup zeroed the V rows past the end of the sequence before it arrived)
                            ok = mbar_wait_warp(&sh->p_full[t], np[t] & 1, sh, p);
                            if (!ok) break;
                            ++np[t];
                            tc_fence_after();
                            issue_pv(t, vslot, i == 1);
                            if (i == n) tc_commit(leader, &sh->o_full[t]);  // every MMA of this tile's segment has been issued
                        }
                        if (i < n) {
                            issue_qk(t, kslot);
                            tc_commit(leader, &sh->s_full[t]);
                        }
                    }
                }
                if (!ok) break;
                tc_commit(leader, &sh->kv_done[rc % kRing]);
                ++rc;
                if (i < n) kslot = (kslot == kKStages - 1) ? 0 : kslot + 1;
                if (i > 0) vslot = (vslot == kVStages - 1) ? 0 : vslot + 1;
                if (i == n - 1) tc_commit(leader, &sh->q_free);             // the segment's last score MMAs read the query tiles
            }
        }
        if (!ok) {
            // abort: everything this warp has issued must retire before the TMEM and the tiles go away
            tc_commit(leader, &sh->drain);
            mbar_wait_quiet(&sh->drain, 0, p.wait_cycles);
        }
        __syncwarp();
    }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 216;");
        // =========================== softmax warpgroups ===========================
        const int t = warp >> 2;                        // row tile of this warpgroup
        const int r = tid & 127;                        // row inside the tile == TMEM lane
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t s_taddr = tmem + lane_base + t * 128;
        const uint32_t o_taddr = tmem + lane_base + 256 + t * 128;
        SegIter it;
        it.init(sh);
        Seg sg;
        int nsteps = 0, nseg = 0;                       // steps / segments this row tile has been through
        int rc0 = 0, vc0 = 0;                           // ring steps / V tiles of the CTA before the current segment
        int anc_b = -1;                                 // the sequence that anc_of (by half of the rows) belongs to
        uint64_t anc_of[2] = {0, 0};
        bool ok = true;
        while (ok && it.next(p, sg)) {
            const int M = sg.N * p.G;
            const int rc_seg = rc0, vc_seg = vc0;       // this segment's first ring step / V tile
            rc0 += sg.s1 - sg.s0 + 1;
            vc0 += sg.s1 - sg.s0;
            if (t == 1 && M - sg.row0 <= kRowTile) continue;
            const int R = sg.row0 + t * kRowTile + r;
            const bool row_ok = R < M;
            const bool warp_live = sg.row0 + t * kRowTile + (warp & 3) * 32 < M;
            if (sg.b != anc_b) {
                anc_b = sg.b;
                anc_of[0] = anc_of[1] = 0;
            }
            uint64_t anc = sg.row0 == 0 ? anc_of[0] : anc_of[1];
            if (sg.s1 * kStepKeys > sg.L && row_ok && anc == 0) {
                // the segment reaches the tree part: this row's ancestor bitset (the G rows of a node walk the same
                // parent chain, at most N - 1 loads deep; kept for the sequence's next heads and layers)
                const int node = R >> p.g_shift;
                bool bad = false;
                anc = ancestor_bits(p.parent + sg.n0, sg.N, node, &bad);
                if (bad) { report_status(p.status, SAGE_STATUS_BAD_TREE); anc = 1ull << node; }
                if (sg.row0 == 0) anc_of[0] = anc;
                else anc_of[1] = anc;
            }
            float m_ref = -INFINITY, l_sum = 0.f;
            for (int j = sg.s0; j < sg.s1; ++j) {
                ok = mbar_wait_warp(&sh->s_full[t], nsteps & 1, sh, p);
                if (!ok) break;
                const int valid = sg.L + sg.N - j * kStepKeys;      // keys of this step that exist
                if (valid < kStepKeys) {
                    // V rows past the end of the sequence may hold anything (a missing second page was not even
                    // copied): zero them so that 0 * V stays 0.  Each warp of the warpgroup takes a quarter of
                    // the rows (both warpgroups write the same zeros); the writes are ordered before this
                    // warp's arrival, which the P V product waits for.  The V tile of step j lands with ring
                    // step j - s0 + 1 of the segment.
                    const int rcv = rc_seg + (j - sg.s0) + 1;
                    ok = mbar_wait_warp(&sh->kv_full[rcv % kRing], (rcv / kRing) & 1, sh, p);
                    if (!ok) break;
                    uint8_t* vb = sV + ((vc_seg + (j - sg.s0)) % kVStages) * kTileBytes;
                    for (int c = (warp & 3) * 32 + lane; c < (kStepKeys - valid) * 16; c += 128) {
                        const int vr = valid + c / 16, ch = c % 16;
                        *reinterpret_cast<uint4*>(vb + (ch >> 3) * kTileHalfBytes + vr * 128 + ((ch & 7) << 4)) = make_uint4(0, 0, 0, 0);
                    }
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                }
                if (!warp_live) {
                    // none of this warp's 32 rows exists (ragged last tile): keep the barrier protocol
                    // going, leave the probabilities of these rows as they are; their outputs are never stored
                    ++nsteps;
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&sh->p_full[t]);
                    continue;
                }
                tc_fence_after();
                const int jt0 = j * kStepKeys - sg.L;            // tree slot of the step's first key
                const bool masked = jt0 + kStepKeys > 0;     // reaches into the tree part (or past the end)
                uint32_t sr[128];
                // Probabilities are taken against the row's reference of the steps before, so a step need not look for its maximum
                // first.  It shows in the step's sum whether the reference still serves; the first step of a segment, steps with
                // masked scores and steps whose sum has grown to kMaxSum go through the maximum (rows that do not exist have no say).
                bool by_max = masked || j == sg.s0, outgrown = false;
                if (!by_max) {
                    uint64_t acc[2] = {0ull, 0ull};
                    tmem_ld32(s_taddr, *reinterpret_cast<uint32_t(*)[32]>(&sr[0]));
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        tmem_wait_ld_of(*reinterpret_cast<uint32_t(*)[32]>(&sr[32 * c]));
                        if (c < 3) tmem_ld32(s_taddr + 32 * (c + 1), *reinterpret_cast<uint32_t(*)[32]>(&sr[32 * (c + 1)]));
                        exp_chunk<SAGE_EXP2_FMA_PAIRS>(sr + 32 * c, p.scale_log2, -m_ref, sr + 16 * c, acc);
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
                    const float m_cand = mx * p.scale_log2;
                    const bool grow = m_cand > m_ref + (outgrown ? 0.f : 8.0f);
                    float alpha = 1.0f;
                    if (grow) {
                        alpha = fast_exp2(m_ref - m_cand);              // 0 when m_ref was -inf
                        m_ref = m_cand;
                    }
                    // O_t *= alpha.  The P V product of the step before has finished: the scores of this step were
                    // issued after it, and their completion is what this warp waited for above.
                    if (j > sg.s0 && __any_sync(0xffffffffu, grow)) rescale_o_rows(o_taddr, alpha);
                    const float neg_ref = (m_ref == -INFINITY) ? 0.f : -m_ref;
                    uint64_t acc[2] = {0ull, 0ull};
#pragma unroll
                    for (int c = 0; c < 4; ++c) exp_chunk<0>(sr + 32 * c, p.scale_log2, neg_ref, sr + 16 * c, acc);   // may hold -inf
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
                ++nsteps;
                __syncwarp();
                if (lane == 0) mbar_arrive(&sh->p_full[t]);
            }
            if (!ok) break;
            // ---- epilogue: O_t / l -> bf16 output, or unnormalised partials for the merge
            ok = mbar_wait_warp(&sh->o_full[t], nseg & 1, sh, p);
            ++nseg;
            if (!ok) break;
            tc_fence_after();
            const bool whole = (sg.s0 == 0 && sg.s1 == sg.steps);
            const float inv = (l_sum > 0.f) ? 1.0f / l_sum : 0.f;
            float4* po = nullptr;
            if (!whole) {
                const size_t slot = (size_t)blockIdx.x * 2 + (sg.at_range_begin ? 0 : 1);
                po = p.part_o + slot * (kHeadDim / 4) * kRowsPerCta + t * kRowTile + r;
                if (row_ok) p.part_ml[slot * kRowsPerCta + t * kRowTile + r] = make_float2(m_ref, l_sum);
            }
            if (warp_live) {
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    uint32_t orr[32];
                    tmem_ld32(o_taddr + c * 32, orr);
                    tmem_wait_ld();
                    if (whole) {
                        // every lane holds 64 bytes of its row; four lanes exchange them, so that a store instruction writes
                        // 64 contiguous bytes of eight rows instead of 16 bytes of 32
                        uint4 v[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            v[i] = make_uint4(pack_bf16(__uint_as_float(orr[8 * i + 0]) * inv, __uint_as_float(orr[8 * i + 1]) * inv),
                                              pack_bf16(__uint_as_float(orr[8 * i + 2]) * inv, __uint_as_float(orr[8 * i + 3]) * inv),
                                              pack_bf16(__uint_as_float(orr[8 * i + 4]) * inv, __uint_as_float(orr[8 * i + 5]) * inv),
                                              pack_bf16(__uint_as_float(orr[8 * i + 6]) * inv, __uint_as_float(orr[8 * i + 7]) * inv));
                        transpose4(v, lane);
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const int Ri = sg.row0 + t * kRowTile + (warp & 3) * 32 + (lane & ~3) + i;
                            if (Ri < M) {
                                const size_t row = (size_t)(sg.n0 + (Ri >> p.g_shift)) * p.Hq + sg.g * p.G + (Ri & (p.G - 1));
                                reinterpret_cast<uint4*>(p.out + ((size_t)sg.layer * p.sum_nodes * p.Hq + row) * kHeadDim + c * 32)[lane & 3] = v[i];
                            }
                        }
                    } else if (row_ok) {
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            po[(c * 8 + i) * kRowsPerCta] =
                                make_float4(__uint_as_float(orr[4 * i]), __uint_as_float(orr[4 * i + 1]),
                                            __uint_as_float(orr[4 * i + 2]), __uint_as_float(orr[4 * i + 3]));
                    }
                }
            }
            tc_fence_before();                          // the next segment's first P V overwrites O_t
        }
    }
    tear_down(tmem, warp);
}

bool launch_rows(const AttnParams& p, const CUtensorMap& qmap, const CUtensorMap& kmap, const CUtensorMap& vmap, cudaStream_t stream) {
    // The two CTAs of a gang are launched as a cluster, which puts them side by side: they read the same K and V.  (Left to
    // itself, the order in which SMs become free behind the kernel before decides, and a gang spread over both dies
    // costs power: 60 nodes, 80 layers x 16k keys at the power limit, 3000 -> 2815 us.)
    return allow_shared_memory<kSmemBytes>(tree_attention_rows_kernel) &&
           succeeded(sage::launch(tree_attention_rows_kernel, dim3(p.n_ctas), kAttnThreads, kSmemBytes, stream, p.n_rp, p, qmap, kmap, vmap));
}

}  // namespace stream
}  // namespace sage
