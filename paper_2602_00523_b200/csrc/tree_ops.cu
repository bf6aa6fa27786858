// Tree-side kernels of the SAGE decode round: template selection, ancestor
// bitsets, draft-token expansion, greedy acceptance and KV compaction.
// All of them are latency-bound (a few hundred bytes to a few MB per round).
#include <atomic>

#include "sage_common.cuh"

namespace sage {

// ---------------------------------------------------------------------------
// alpha -> template (Eq. 10 / Eq. 11, Section 3.2) + optional hand-over of the
// chosen templates' parent/rank arrays for the next round.
// ---------------------------------------------------------------------------
struct SelectParams {
    const float* alpha;
    const int32_t* alpha_row;
    int batch;
    sage_tree_policy pol;
    int32_t* template_id;
    float* depth_cont;
    float* width_cont;
    const int32_t* bank_parent;
    const int32_t* bank_rank;
    const int32_t* bank_n_nodes;
    int32_t* next_parent;
    int32_t* next_rank;
    int32_t* next_node_offsets;
    int32_t* status;
};

__device__ __forceinline__ int pick_template(const SelectParams& p, int b, float* a_out) {
    const int row = p.alpha_row ? p.alpha_row[b] : b;
    const float a = p.alpha[row];
    int t = 0;
    for (int j = 0; j + 1 < p.pol.n_templates; ++j) t += (a < p.pol.alpha_thresholds[j]) ? 1 : 0;
    *a_out = a;
    return t;
}

__global__ void select_tree_kernel(SelectParams p) {
    after_previous_kernel();
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= p.batch) return;
    float a;
    const int t = pick_template(p, b, &a);
    p.template_id[b] = t;
    if (p.depth_cont) p.depth_cont[b] = fmaf(a, p.pol.d_max - p.pol.d_min, p.pol.d_min);
    if (p.width_cont) p.width_cont[b] = fmaf(1.0f - a, p.pol.w_max - p.pol.w_min, p.pol.w_min);
}

// One block: offsets are a running sum over the batch, then every tree is copied.
__global__ void handover_trees_kernel(SelectParams p) {
    after_previous_kernel();
    __shared__ int s_bad;
    if (threadIdx.x == 0) {
        int off = 0, bad = 0;
        for (int b = 0; b < p.batch; ++b) {
            p.next_node_offsets[b] = off;
            int n = p.bank_n_nodes[p.template_id[b]];
            if (n < 1 || n > SAGE_MAX_NODES) { bad = 1; n = 1; }
            off += n;
        }
        p.next_node_offsets[p.batch] = off;
        s_bad = bad;
        if (bad) report_status(p.status, SAGE_STATUS_BAD_TREE);
    }
    __syncthreads();
    if (s_bad) return;
    for (int b = 0; b < p.batch; ++b) {
        const int t = p.template_id[b];
        const int n = p.bank_n_nodes[t];
        const int off = p.next_node_offsets[b];
        for (int i = threadIdx.x; i < n; i += blockDim.x) {
            p.next_parent[off + i] = p.bank_parent[t * SAGE_MAX_NODES + i];
            p.next_rank[off + i] = p.bank_rank[t * SAGE_MAX_NODES + i];
        }
    }
}

// ---------------------------------------------------------------------------
// Ancestor bitsets (Section 2.2; Algorithm 1 TreeAttnMask)
// ---------------------------------------------------------------------------
__global__ void ancestor_mask_kernel(const int32_t* __restrict__ parent, const int32_t* __restrict__ node_offsets,
                                     uint64_t* __restrict__ anc, int32_t* status) {
    after_previous_kernel();
    const int b = blockIdx.x;
    const int n0 = node_offsets[b];
    const int n = node_offsets[b + 1] - n0;
    if (n < 1 || n > SAGE_MAX_NODES) {
        if (threadIdx.x == 0) report_status(status, SAGE_STATUS_BAD_TREE);
        return;
    }
    const int i = threadIdx.x;
    if (i >= n) return;
    bool bad = false;
    const uint64_t a = ancestor_bits(parent + n0, n, i, &bad);
    if (bad) report_status(status, SAGE_STATUS_BAD_TREE);
    anc[n0 + i] = bad ? (1ull << i) : a;
}

// ---------------------------------------------------------------------------
// Greedy acceptance, one warp per tree (Section 2.2, Eq. 5; Section 3.3 Phase 2).
// Node i is accepted iff every non-root node on its root path matches the
// target's argmax at its parent.  With anc(i) as a bitset and `match` the bitset
// of matching nodes this is (anc(i) & ~match) == 0.  Because parent < child, a
// root path read in increasing node index is the path itself, so "longest, then
// lexicographically smallest" is the maximum of (depth, bit-reversed anc(i)).
// A chain of latencies: two rounds of loads (offsets, nodes), the rest in registers and shuffles.  Walking up the parents in memory, a
// node at a time, and looking tokens up behind that took 2.88 us instead of 2.06 (four trees, back to back in a graph).
// ---------------------------------------------------------------------------
__global__ void accept_kernel(const int32_t* __restrict__ parent, const int32_t* __restrict__ draft_token,
                              const int32_t* __restrict__ target_argmax, const int32_t* __restrict__ node_offsets,
                              int batch, int max_path, int32_t* __restrict__ path, int32_t* __restrict__ path_len,
                              int32_t* __restrict__ bonus_token, int32_t* status) {
    after_previous_kernel();
    const int warps_per_block = blockDim.x >> 5;
    const int b = blockIdx.x * warps_per_block + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (b >= batch) return;
    const int n0 = node_offsets[b];
    const int n = node_offsets[b + 1] - n0;
    int32_t* my_path = path + (size_t)b * max_path;
    bool bad_tree = (n < 1 || n > SAGE_MAX_NODES);
    // Everything about the nodes in one round of loads; a parent's part of it comes from the lane that has it.
    const int count = bad_tree ? 0 : n;
    int par[2], draft[2], target[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int i = lane + 32 * u;
        par[u] = i < count ? parent[n0 + i] : -1;
        draft[u] = i < count ? draft_token[n0 + i] : 0;
        target[u] = i < count ? target_argmax[n0 + i] : 0;
    }
    auto of = [](const auto (&v)[2], int node) {
        const auto lo = __shfl_sync(0xffffffffu, v[0], node & 31), hi = __shfl_sync(0xffffffffu, v[1], node & 31);
        return node < 32 ? lo : hi;
    };
    uint64_t anc[2];
    int up[2];
    bool match[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int i = lane + 32 * u;
        if (i < count && (i == 0 ? par[u] != -1 : par[u] < 0 || par[u] >= i)) bad_tree = true;
        up[u] = i < count && i > 0 ? par[u] : 0;
        anc[u] = 1ull << i;
    }
    bad_tree = __any_sync(0xffffffffu, bad_tree);
    if (bad_tree) {
        if (lane == 0) {
            report_status(status, SAGE_STATUS_BAD_TREE);
            path_len[b] = 0;
            bonus_token[b] = -1;
        }
        for (int j = lane; j < max_path; j += 32) my_path[j] = -1;
        return;
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int i = lane + 32 * u, at_parent = of(target, up[u]);
        match[u] = i < n && (i == 0 || draft[u] == at_parent);
    }
    // ancestors by doubling: what a node has collected so far, and how far up that reaches
    while (__any_sync(0xffffffffu, (up[0] | up[1]) != 0)) {
        const uint64_t a0 = of(anc, up[0]), a1 = of(anc, up[1]);
        const int u0 = of(up, up[0]), u1 = of(up, up[1]);
        anc[0] |= a0;
        anc[1] |= a1;
        up[0] = u0;
        up[1] = u1;
    }
    anc[0] |= 1ull;
    anc[1] |= 1ull;
    const uint64_t match_bits = (uint64_t)__ballot_sync(0xffffffffu, match[0]) |
                                ((uint64_t)__ballot_sync(0xffffffffu, match[1]) << 32);
    // best key over accepted nodes: depth first, then bit-reversed ancestor set
    int best_depth = -1;
    uint64_t best_rev = 0, best_anc = 0;
    for (int u = 0; u < 2; ++u) {
        const int i = lane + 32 * u;
        if (i < n && (anc[u] & ~match_bits) == 0) {
            const int len = __popcll(anc[u]);   // nodes on the path = depth + 1
            if (len <= max_path) {
                const uint64_t rev = __brevll(anc[u]);
                if (len > best_depth || (len == best_depth && rev > best_rev)) {
                    best_depth = len; best_rev = rev; best_anc = anc[u];
                }
            }
        }
    }
    for (int off = 16; off > 0; off >>= 1) {
        const int od = __shfl_xor_sync(0xffffffffu, best_depth, off);
        const uint64_t orv = __shfl_xor_sync(0xffffffffu, best_rev, off);
        const uint64_t oan = __shfl_xor_sync(0xffffffffu, best_anc, off);
        if (od > best_depth || (od == best_depth && orv > best_rev)) {
            best_depth = od; best_rev = orv; best_anc = oan;
        }
    }
    // best_anc holds the accepted path (the root alone is always accepted: len 1 <= max_path)
    const int len = __popcll(best_anc);
    for (int j = lane; j < max_path; j += 32) {
        int node = -1;
        if (j < len) {
            uint64_t m = best_anc;
            for (int s = 0; s < j; ++s) m &= m - 1;      // drop the j lowest set bits
            node = __ffsll((long long)m) - 1;
        }
        my_path[j] = node;
    }
    const int bonus = of(target, 63 - __clzll((long long)best_anc));
    if (lane == 0) {
        path_len[b] = len;
        bonus_token[b] = bonus;
    }
}

// ---------------------------------------------------------------------------
// KV compaction (Algorithm 1 cache update), one cluster of blocks per sequence: every
// block works out the moves for itself, thread = one 16-byte column of a K or V row of one
// (layer, kv head).  Destinations L+j never lie above their sources L+path[j] (path[j] >= j
// because parent < child), and sources of later j lie above every earlier destination, so
// walking the moves upwards with "read a batch, then write it" needs no barrier.
// The length advances in the same launch: the cluster's barrier says when every block has
// read the old one.  Latency-bound (a few MB at most): all loads of a batch are in flight
// together, and what an SM can keep in flight limits a sequence: 80 layers, 9 entries, one
// sequence 10.9 us with 8 blocks, 7.5 us with 16; four 11.3 and 8.3 us.  (Two launches, one for the
// length, with one thread planning: 17.3 us for four with the acceptance before it; one launch 15.0.)
// ---------------------------------------------------------------------------
struct CompactParams {
    __nv_bfloat16* k_pool;
    __nv_bfloat16* v_pool;
    int64_t layer_stride;
    int n_layers, n_pages, max_pages, max_path, n_kv_heads;
    int blocks;                                  // per sequence: one cluster
    const int32_t* page_table;
    int32_t* seq_len;
    const int32_t* path;
    const int32_t* path_len;
    int32_t* status;
};

constexpr int kCompactThreads = 512;
constexpr int kCompactCluster = 16;              // blocks of a sequence at most (sm_100a allows 16 on request)
constexpr int kColumns = 3;                      // columns a thread works on at a time
constexpr int kMoves = 4;                        // moves of a batch

__global__ void __launch_bounds__(kCompactThreads) compact_kv_kernel(const CompactParams p) {
    after_previous_kernel();
    __shared__ int64_t s_src[SAGE_MAX_NODES];    // element offsets of the (page, head 0, slot) rows to move
    __shared__ int64_t s_dst[SAGE_MAX_NODES];
    __shared__ int s_moves, s_len;               // s_len: the sequence's new length, -1 if it does not advance
    const int b = blockIdx.x / p.blocks, part = blockIdx.x % p.blocks, tid = threadIdx.x, lane = tid & 31;
    if (tid < 32) {
        // Checks the accepted path and turns it into moves, two entries per lane.  A path or a page id that is not
        // valid leaves the sequence exactly as it is (nothing moves, its length does not advance).
        // (the path's first entries are asked for beside the lengths)
        const int ahead = lane < p.max_path ? p.path[(size_t)b * p.max_path + lane] : SAGE_MAX_NODES;
        const int L = p.seq_len[b];
        const int plen = p.path_len[b];
        const bool whole_bad = plen < 0 || plen > p.max_path || plen > SAGE_MAX_NODES || L < 0;
        bool bad_path = whole_bad, bad_page = false;
        int moves = 0, before = -1;              // before: the last node of the previous 32 entries
        for (int j0 = 0; j0 < (whole_bad ? 0 : plen); j0 += 32) {
            const int j = j0 + lane;
            const int node = j >= plen ? SAGE_MAX_NODES : j0 == 0 ? ahead : p.path[(size_t)b * p.max_path + j];
            int prev = __shfl_up_sync(0xffffffffu, node, 1);
            if (lane == 0) prev = before;
            before = __shfl_sync(0xffffffffu, node, 31);
            int64_t so = 0, dofs = 0;
            bool move = false;
            if (j < plen) {
                if (node <= prev || node < j || node >= SAGE_MAX_NODES || (j == 0 && node != 0)) {
                    bad_path = true;             // a root path starts at 0 and visits increasing indices
                } else if (node != j) {
                    const int s_pos = L + node, d_pos = L + j;
                    if (s_pos / kPageSize >= p.max_pages) {
                        bad_page = true;
                    } else {
                        const int sp = p.page_table[(size_t)b * p.max_pages + s_pos / kPageSize];
                        const int dp = p.page_table[(size_t)b * p.max_pages + d_pos / kPageSize];
                        if (sp < 0 || sp >= p.n_pages || dp < 0 || dp >= p.n_pages) {
                            bad_page = true;
                        } else {
                            so = ((int64_t)sp * p.n_kv_heads * kPageSize + s_pos % kPageSize) * kHeadDim;
                            dofs = ((int64_t)dp * p.n_kv_heads * kPageSize + d_pos % kPageSize) * kHeadDim;
                            move = true;
                        }
                    }
                }
            }
            const unsigned mv = __ballot_sync(0xffffffffu, move);
            if (move) {
                const int at = moves + __popc(mv & ((1u << lane) - 1u));
                s_src[at] = so;
                s_dst[at] = dofs;
            }
            moves += __popc(mv);
        }
        bad_path = __any_sync(0xffffffffu, bad_path);
        bad_page = __any_sync(0xffffffffu, bad_page);
        const int code = bad_path ? SAGE_STATUS_BAD_PATH : (bad_page ? SAGE_STATUS_BAD_PAGE : 0);
        if (lane == 0) {
            s_moves = code ? 0 : moves;
            s_len = code ? -1 : L + plen;
            if (code && part == 0) report_status(p.status, code);
        }
    }
    __syncthreads();
    // this block has read the old length
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    const int moves = s_moves;
    const int per_pool = p.n_kv_heads * 16;      // 16-byte columns of a token's K (or V) across heads
    const int per_layer = 2 * per_pool, total = per_layer * p.n_layers;
    const int stride = p.blocks * kCompactThreads;
    if (moves > 0) {
        for (int c0 = part * kCompactThreads + tid; c0 < total; c0 += kColumns * stride) {
            __nv_bfloat16* col[kColumns];
#pragma unroll
            for (int u = 0; u < kColumns; ++u) {
                const int c = c0 + u * stride;
                const int layer = c / per_layer, r = c % per_layer, cc = r % per_pool;
                col[u] = c < total ? (r < per_pool ? p.k_pool : p.v_pool) + (int64_t)layer * p.layer_stride +
                                         (int64_t)(cc / 16) * kPageSize * kHeadDim + (cc % 16) * 8
                                   : nullptr;
            }
            for (int m0 = 0; m0 < moves; m0 += kMoves) {
                uint4 r[kColumns][kMoves];
#pragma unroll
                for (int u = 0; u < kColumns; ++u)
#pragma unroll
                    for (int m = 0; m < kMoves; ++m)
                        if (col[u] && m0 + m < moves) r[u][m] = *reinterpret_cast<const uint4*>(col[u] + s_src[m0 + m]);
#pragma unroll
                for (int u = 0; u < kColumns; ++u)
#pragma unroll
                    for (int m = 0; m < kMoves; ++m)
                        if (col[u] && m0 + m < moves) *reinterpret_cast<uint4*>(col[u] + s_dst[m0 + m]) = r[u][m];
            }
        }
    }
    asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
    if (part == 0 && tid == 0 && s_len >= 0) p.seq_len[b] = s_len;
}

// Clusters of more than 8 blocks are a per-device opt-in of the kernel.
static bool allow_large_cluster() {
    static std::atomic<bool> done[64];
    int dev = 0;
    if (!succeeded(cudaGetDevice(&dev)) || dev < 0 || dev >= 64) return false;
    if (!done[dev].load(std::memory_order_acquire)) {
        if (!succeeded(cudaFuncSetAttribute(compact_kv_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1))) return false;
        done[dev].store(true, std::memory_order_release);
    }
    return true;
}

// ---------------------------------------------------------------------------
// Dynamic tree construction, one level per launch (Section 3.2: hierarchical width
// decay, Eq. 12, and "Dynamic Tree Construction").  One block per sequence.
// A child of rank r of frontier node u joins the tree iff
// r < W_l and exp(cum_logprob) > theta_l; both tests only ever cut a suffix of the
// (descending) candidate row, so each node contributes a prefix of its ranks, and the
// children are laid out in breadth-first order by a prefix sum.  Decisions are taken
// in fp64 on the fp32 inputs; cumulative log-probabilities are fp32 sums.
// ---------------------------------------------------------------------------
struct GrowParams {
    const int32_t* topk_idx;
    const float* topk_logprob;
    int k;
    const float* alpha;
    const int32_t* alpha_row;
    sage_tree_policy pol;
    int n_max;
    int32_t *parent, *rank, *depth, *token;
    float* cum_logprob;
    int32_t *n_nodes, *frontier_begin;
    const float* d_max_seq;
    int32_t* status;
};

// A launch is one short chain of dependent steps, so the chain is what is kept short: one round of loads for the sequence's
// numbers, one for the nodes and their candidates, and a thread per candidate, 16 to a node, for the fp64 exponentials (one
// thread per node went through up to 16 loads and exponentials in turn).
constexpr int kGrowThreads = 512;                          // 32 frontier nodes at a time
constexpr int kGrowNodes = kGrowThreads / SAGE_MAX_TOPK, kGrowTurns = SAGE_MAX_NODES / kGrowNodes;
static_assert(SAGE_MAX_TOPK == 16 && SAGE_MAX_NODES == 64, "two nodes per warp, two counts per lane");
__global__ void __launch_bounds__(kGrowThreads) grow_tree_kernel(GrowParams p) {
    after_previous_kernel();
    __shared__ int s_count[SAGE_MAX_NODES];
    const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31;
    const int r = tid % SAGE_MAX_TOPK;                     // rank of this thread's candidates
    const int base = b * SAGE_MAX_NODES;
    const int n = p.n_nodes[b], fb = p.frontier_begin[b];
    const double a = (double)p.alpha[p.alpha_row ? p.alpha_row[b] : b];
    const double d_max = p.d_max_seq ? (double)p.d_max_seq[b] : (double)p.pol.d_max;
    if (n < 1 || n > p.n_max || fb < 0 || fb > n) {
        if (tid == 0) report_status(p.status, SAGE_STATUS_BAD_TREE);
        return;
    }
    if (fb == n) return;                                   // nothing left to expand
    const int level = p.depth[base + fb] + 1;
    float cum_u[kGrowTurns], c[kGrowTurns];
    int32_t word[kGrowTurns];
#pragma unroll
    for (int t = 0; t < kGrowTurns; ++t) {
        const int node = fb + t * kGrowNodes + tid / SAGE_MAX_TOPK;
        cum_u[t] = 0.f;
        c[t] = 0.f;
        word[t] = 0;
        if (node < n) {
            cum_u[t] = p.cum_logprob[base + node];
            if (r < p.k) {
                c[t] = p.topk_logprob[(size_t)(base + node) * p.k + r];
                word[t] = p.topk_idx[(size_t)(base + node) * p.k + r];
            }
        }
    }
    // explicit roundings: no fused multiply-add, so that a host check in plain fp64 sees the same D and W
    const double D = __dadd_rn((double)p.pol.d_min, __dmul_rn(a, d_max - (double)p.pol.d_min));
    const double W = __dadd_rn((double)p.pol.w_min, __dmul_rn(1.0 - a, (double)p.pol.w_max - (double)p.pol.w_min));
    if ((double)level > D) {                               // the tree has reached its depth
        if (tid == 0) p.frontier_begin[b] = n;
        return;
    }
    const double theta = 0.1 * (double)level / D;
    int count[kGrowTurns];
#pragma unroll
    for (int t = 0; t < kGrowTurns; ++t) {
        bool in = false;
        if (fb + t * kGrowNodes + tid / SAGE_MAX_TOPK < n && r < p.k) {
            const double w_l = (level == 1) ? W : W / (double)level * (0.5 + exp((double)cum_u[t]));
            c[t] = __fadd_rn(cum_u[t], c[t]);
            in = (double)r < w_l && exp((double)c[t]) > theta;
        }
        // the node's children are its ranks up to the first that fails
        const unsigned out = ~__ballot_sync(0xffffffffu, in) >> (lane & SAGE_MAX_TOPK);
        count[t] = __ffs(out | (1u << SAGE_MAX_TOPK)) - 1;
        if (r == 0) s_count[t * kGrowNodes + tid / SAGE_MAX_TOPK] = count[t];
    }
    __syncthreads();
    const int c0 = s_count[lane], c1 = s_count[lane + 32];
    const int total = __reduce_add_sync(0xffffffffu, c0 + c1);
#pragma unroll
    for (int t = 0; t < kGrowTurns; ++t) {
        // children of the nodes in front of this thread's
        const int first = t * kGrowNodes + tid / 32 * 2;   // the warp's first node
        const int before = __reduce_add_sync(0xffffffffu, (lane < first ? c0 : 0) + (lane + 32 < first ? c1 : 0));
        const int pos = n + before + (lane >= SAGE_MAX_TOPK ? s_count[first] : 0) + r;
        if (r < count[t] && pos < p.n_max) {               // node budget: breadth-first prefix
            p.parent[base + pos] = fb + first + lane / SAGE_MAX_TOPK;
            p.rank[base + pos] = r;
            p.depth[base + pos] = level;
            p.token[base + pos] = word[t];
            p.cum_logprob[base + pos] = c[t];
        }
    }
    if (tid == 0) {
        p.n_nodes[b] = min(n + total, p.n_max);
        p.frontier_begin[b] = n;
    }
}

// ---------------------------------------------------------------------------
// Adaptive history tracking (Section 3.3; window 10, thresholds 2 and 3 in Section 5.1).
// One thread per sequence: push tau = path_len - 1 into the sequence's ring of recent
// acceptance lengths; once `min_samples` values are there, their mean below `lower`
// lowers the sequence's maximum depth by `step`, above `upper` raises it, clamped to
// [d_lo, d_hi].  The mean is an exact integer sum divided in fp64.
// ---------------------------------------------------------------------------
__global__ void update_history_kernel(const int32_t* __restrict__ path_len, int batch, sage_history_policy pol,
                                      int32_t* __restrict__ window_buf, int32_t* __restrict__ count,
                                      float* __restrict__ d_max, int32_t* status) {
    after_previous_kernel();
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= batch) return;
    const int pl = path_len[b];
    const int c = count[b];
    if (pl < 1 || c < 0) {                          // the root is always accepted: path_len >= 1
        report_status(status, SAGE_STATUS_BAD_PATH);
        return;
    }
    int32_t* ring = window_buf + (size_t)b * pol.window;
    ring[c % pol.window] = pl - 1;
    count[b] = c + 1;
    const int n = min(c + 1, pol.window);
    if (n < pol.min_samples) return;
    long long sum = 0;
    for (int i = 0; i < n; ++i) sum += ring[i];
    const double mean = (double)sum / (double)n;
    float d = d_max[b];
    if (mean < (double)pol.lower) d = fmaxf(pol.d_lo, d - pol.step);
    else if (mean > (double)pol.upper) d = fminf(pol.d_hi, d + pol.step);
    d_max[b] = d;
}

}  // namespace sage

using namespace sage;

extern "C" int sage_select_tree(const float* alpha, const int32_t* alpha_row, int batch,
                                const sage_tree_policy* policy, int32_t* template_id, float* depth_cont,
                                float* width_cont, const int32_t* bank_parent, const int32_t* bank_rank,
                                const int32_t* bank_n_nodes, int32_t* next_parent, int32_t* next_rank,
                                int32_t* next_node_offsets, int32_t* status, void* stream) {
    if (!alpha || !policy || !template_id || batch < 0) return SAGE_ERR_INVALID_ARG;
    if (policy->n_templates < 1 || policy->n_templates > SAGE_MAX_TEMPLATES) return SAGE_ERR_INVALID_ARG;
    for (int j = 0; j + 2 < policy->n_templates; ++j)
        if (!(policy->alpha_thresholds[j] >= policy->alpha_thresholds[j + 1])) return SAGE_ERR_INVALID_ARG;
    const bool handover = next_parent != nullptr;
    if (handover && (!bank_parent || !bank_rank || !bank_n_nodes || !next_rank || !next_node_offsets))
        return SAGE_ERR_INVALID_ARG;
    if (batch == 0) return SAGE_OK;
    SelectParams p{alpha, alpha_row, batch, *policy, template_id, depth_cont, width_cont, bank_parent,
                   bank_rank, bank_n_nodes, next_parent, next_rank, next_node_offsets, status};
    const int code = launch_status(launch(select_tree_kernel, dim3((batch + 127) / 128), 128, 0, as_stream(stream), 0, p));
    if (code != SAGE_OK || !handover) return code;
    return launch_status(launch(handover_trees_kernel, dim3(1), 256, 0, as_stream(stream), 0, p));
}

extern "C" int sage_build_ancestor_mask(const int32_t* parent, const int32_t* node_offsets, int batch,
                                        uint64_t* anc, int32_t* status, void* stream) {
    if (!parent || !node_offsets || !anc || batch < 0) return SAGE_ERR_INVALID_ARG;
    if (batch == 0) return SAGE_OK;
    return launch_status(launch(ancestor_mask_kernel, dim3(batch), SAGE_MAX_NODES, 0, as_stream(stream), 0, parent, node_offsets, anc, status));
}

extern "C" int sage_accept(const int32_t* parent, const int32_t* draft_token, const int32_t* target_argmax,
                           const int32_t* node_offsets, int batch, int max_path, int32_t* path,
                           int32_t* path_len, int32_t* bonus_token, int32_t* status, void* stream) {
    if (!parent || !draft_token || !target_argmax || !node_offsets || !path || !path_len || !bonus_token)
        return SAGE_ERR_INVALID_ARG;
    if (batch < 0 || max_path < 1) return SAGE_ERR_INVALID_ARG;
    if (batch == 0) return SAGE_OK;
    const int wpb = 4;
    return launch_status(launch(accept_kernel, dim3((batch + wpb - 1) / wpb), wpb * 32, 0, as_stream(stream), 0, parent, draft_token,
                 target_argmax, node_offsets, batch, max_path, path, path_len, bonus_token, status));
}

extern "C" int sage_compact_kv(void* k_pool, void* v_pool, int64_t layer_stride_elems, int n_layers, int n_pages,
                               const int32_t* page_table, int max_pages_per_seq, int32_t* seq_len,
                               const int32_t* path, const int32_t* path_len, int batch, int max_path,
                               int n_kv_heads, int head_dim, int page_size, int32_t* status, void* stream) {
    if (!k_pool || !v_pool || !page_table || !seq_len || !path || !path_len) return SAGE_ERR_INVALID_ARG;
    if (batch < 0 || n_layers < 1 || n_pages < 1 || max_pages_per_seq < 1 || max_path < 1 || n_kv_heads < 1 ||
        layer_stride_elems < 0)
        return SAGE_ERR_INVALID_ARG;
    if (head_dim != kHeadDim || page_size != kPageSize || n_layers > 65535) return SAGE_ERR_UNSUPPORTED;
    if (((uintptr_t)k_pool | (uintptr_t)v_pool) & 15 || (layer_stride_elems & 7)) return SAGE_ERR_INVALID_ARG;
    if (batch == 0) return SAGE_OK;
    // as many blocks per sequence as have columns, a power of two
    const int64_t columns = (int64_t)n_layers * n_kv_heads * 32;
    if (columns > 0x3fffffff || batch > 0x7fffffff / kCompactCluster) return SAGE_ERR_UNSUPPORTED;
    int blocks = 1;
    while (blocks < kCompactCluster && (int64_t)blocks * kCompactThreads < columns) blocks *= 2;
    CompactParams p{(__nv_bfloat16*)k_pool, (__nv_bfloat16*)v_pool, layer_stride_elems, n_layers, n_pages,
                    max_pages_per_seq, max_path, n_kv_heads, blocks, page_table, seq_len, path, path_len, status};
    if (blocks > 8 && !allow_large_cluster()) return SAGE_ERR_CUDA;
    return launch_status(launch(compact_kv_kernel, dim3((unsigned)(blocks * batch)), kCompactThreads, 0, as_stream(stream), blocks, p));
}

extern "C" int sage_grow_tree(const int32_t* topk_idx, const float* topk_logprob, int k, const float* alpha,
                              const int32_t* alpha_row, int batch, const sage_tree_policy* policy, int n_max,
                              int32_t* parent, int32_t* rank, int32_t* depth, int32_t* token, float* cum_logprob,
                              int32_t* n_nodes, int32_t* frontier_begin, const float* d_max_seq, int32_t* status,
                              void* stream) {
    if (!topk_idx || !topk_logprob || !alpha || !policy || !parent || !rank || !depth || !token || !cum_logprob ||
        !n_nodes || !frontier_begin)
        return SAGE_ERR_INVALID_ARG;
    if (batch < 0 || k < 1 || n_max < 1) return SAGE_ERR_INVALID_ARG;
    if (k > SAGE_MAX_TOPK || n_max > SAGE_MAX_NODES) return SAGE_ERR_UNSUPPORTED;
    if (!(policy->d_max >= policy->d_min) || !(policy->d_min > 0.f) || !(policy->w_max >= policy->w_min) ||
        !(policy->w_min > 0.f))
        return SAGE_ERR_INVALID_ARG;
    if (batch == 0) return SAGE_OK;
    GrowParams p{topk_idx, topk_logprob, k, alpha, alpha_row, *policy, n_max, parent, rank, depth, token,
                 cum_logprob, n_nodes, frontier_begin, d_max_seq, status};
    return launch_status(launch(grow_tree_kernel, dim3(batch), kGrowThreads, 0, as_stream(stream), 0, p));
}

extern "C" int sage_update_history(const int32_t* path_len, int batch, const sage_history_policy* policy,
                                   int32_t* window_buf, int32_t* count, float* d_max, int32_t* status,
                                   void* stream) {
    if (!path_len || !policy || !window_buf || !count || !d_max || batch < 0) return SAGE_ERR_INVALID_ARG;
    if (policy->window < 1 || policy->min_samples < 1 || policy->min_samples > policy->window ||
        !(policy->upper >= policy->lower) || !(policy->d_hi >= policy->d_lo) || !(policy->step >= 0.f))
        return SAGE_ERR_INVALID_ARG;
    if (policy->window > 1024) return SAGE_ERR_UNSUPPORTED;
    if (batch == 0) return SAGE_OK;
    return launch_status(launch(update_history_kernel, dim3((batch + 127) / 128), 128, 0, as_stream(stream), 0, path_len, batch, *policy,
                 window_buf, count, d_max, status));
}

extern "C" const char* sage_status_string(int code) {
    switch (code) {
        case SAGE_OK: return "ok";
        case SAGE_ERR_INVALID_ARG: return "invalid argument";
        case SAGE_ERR_UNSUPPORTED: return "outside the supported envelope";
        case SAGE_ERR_WORKSPACE: return "workspace missing or too small";
        case SAGE_ERR_CUDA: return "CUDA call failed";
        case SAGE_ERR_TOO_LARGE: return "problem is larger than the call without scratch memory takes";
        case SAGE_STATUS_BAD_TREE: return "device: parent array or node count violates the tree rules";
        case SAGE_STATUS_BAD_PAGE: return "device: page id out of range or sequence longer than its page table";
        case SAGE_STATUS_TIMEOUT: return "device: bounded wait expired";
        case SAGE_STATUS_BAD_PATH: return "device: accepted path is not a valid root path";
        default: return "unknown status";
    }
}
