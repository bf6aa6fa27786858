// Fused softmax entropy + top-k over vocabulary-sized fp32 rows (Eq. 4, Eq. 7-9)
// and the draft-token expansion gather, in one launch.
//
// A row belongs to a cluster of CTAs, each of which streams one contiguous chunk of it once from
// HBM.  Every thread copies its own 16-byte pieces asynchronously to shared memory, three batches
// ahead, and is the only one to read them: no barrier in the stream, and 48 KB per CTA in flight
// without registers to hold them.
//  1. Every thread keeps softmax moments (s = sum e^(x-m), t = sum (x-m) e^(x-m), m the largest
//     element so far or larger) in fp32 over its elements: about seven instructions
//     per logit, loads included.
//  2. The K best.  After batches 0, 1, 3, 7, ... the CTA takes a threshold from its threads' largest
//     elements: the q-th largest of the warps' r-th largest thread maxima, q = ceil(K / r), so that at
//     least K elements reach it.  Elements that reach the threshold are appended to the CTA's list, some
//     50 in all; the rest of the stream only compares each thread's largest element of a batch with
//     it.  When the list is full (ascending data, many equal values), the warps' sorted queues take
//     over, whose K-th value raises the threshold for the whole CTA too.  Keys order by value (with -0 == +0) and then by
//     lowest index, so every merge order gives the same answer.
//  3. Moments (in fp64) and the K best keys of every CTA go to the first CTA of the cluster through
//     distributed shared memory; it ranks them, derives lse, entropies, log-probs and alpha, and
//     hands the row's tokens to the children of the row's node.
// What bounds it: HBM for many rows (960 rows x 152064, K = 10: 158 -> 94 us, 6.2 TB/s), the chain
// launch -> load -> select -> merge for few (60 rows: 41 -> 15.7 us; 15 rows x 32000, K = 4: 13 -> 5.4 us).  Rows that are
// constant, or masked with one value, take the same time (600 rows: 63 to 69 us); ascending rows are the worst (884 us).
// The form before this one offered every element to per-warp queues that started empty, 67 thread
// instructions per logit at K = 10, and took two more launches to merge and to gather the tokens.
#include <math.h>

#include <atomic>

#include "sage_common.cuh"

namespace sage {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kMaxChunks = 8;                    // CTAs of a cluster (the portable limit)
constexpr int kBatch = 4;                        // 16-byte pieces of a batch per thread
constexpr int kStages = 3;                       // batches on their way per thread
constexpr int kStreamBytes = kStages * kBatch * kThreads * 16;
constexpr int kCtasPerSm = 4;
constexpr int kListCap = 256;                    // candidates a CTA takes down before its warps' queues take over

__device__ __forceinline__ uint32_t order_key(float x) {
    x += 0.0f;                                   // -0 -> +0
    const uint32_t u = __float_as_uint(x);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float key_value(uint32_t k) {
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}
__device__ __forceinline__ uint64_t make_key(float x, int idx) {
    return ((uint64_t)order_key(x) << 32) | (uint32_t)(0xffffffffu - (uint32_t)idx);
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
__device__ __forceinline__ uint64_t f2_mul(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// e^d through the hardware 2^x (relative error about 2^-22): one multiply and one special-function
// instruction instead of the library routine's range reduction.  The moments built from it are merged
// in fp64; the entropy stays well inside its 1e-5 bound.
__device__ __forceinline__ float ex2(float y) {
    float e;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(y));
    return e;
}
constexpr float kLog2e = 1.4426950408889634f;

// Online softmax moments of one thread: s = sum e^(x - m), t = sum (x - m) e^(x - m).
struct Moments {
    float m;           // reference, -1e30 before the first element
    uint64_t s2, t2;   // (even, odd) partial sums
    __device__ __forceinline__ void init() { m = -1e30f; s2 = 0; t2 = 0; }
    // The reference moves with the largest element, whose e^(x - m) is exactly 1 then (left up to 8 below it, a confident row's
    // log-probability and entropy took the rounding of e^8).  After the first batch, whose maximum the CTA shares,
    // that hardly ever happens: no divergent rescaling.
    __device__ __forceinline__ void rise(float mx) {
        if (mx > m) {
            const float c = expf(m - mx);
            float s0, s1, t0, t1;
            f2_unpack(s2, s0, s1);
            f2_unpack(t2, t0, t1);
            t2 = f2_pack(c * fmaf(m - mx, s0, t0), c * fmaf(m - mx, s1, t1));
            s2 = f2_pack(s0 * c, s1 * c);
            m = mx;
        }
    }
    // The 16 elements of a batch are summed by themselves and then added: a long row's sums then take one rounding per batch at
    // their full size instead of eight (148 rows of 152064 with a peak, error of the entropy against 64 bits, root mean
    // square: 5.1e-7 -> 2.8e-7; 3.3e-7 if a row is cut into 32 chunks instead).
    // kAll: every piece is there, else the first `n` of them.
    template <bool kAll>
    __device__ __forceinline__ void add_batch(const float4 (&v)[kBatch], int n) {
        const uint64_t nm2 = f2_pack(-m, -m);
        uint64_t s = 0, t = 0;
        auto add = [&](float x0, float x1) {
            const uint64_t d2 = f2_add(f2_pack(x0, x1), nm2);
            float y0, y1;
            f2_unpack(f2_mul(d2, f2_pack(kLog2e, kLog2e)), y0, y1);
            const uint64_t e2 = f2_pack(ex2(y0), ex2(y1));
            s = f2_add(s, e2);
            t = f2_fma(d2, e2, t);
        };
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            if (kAll || u < n) {
                add(v[u].x, v[u].y);
                add(v[u].z, v[u].w);
            }
        }
        s2 = f2_add(s2, s);
        t2 = f2_add(t2, t);
    }
    __device__ __forceinline__ void add1(float x) {
        rise(x);
        const float d = x - m, e = expf(d);
        s2 = f2_add(s2, f2_pack(e, 0.f));
        t2 = f2_add(t2, f2_pack(d * e, 0.f));
    }
};

__device__ __forceinline__ float max4(const float4& v) { return fmaxf(fmaxf(v.x, v.y), fmaxf(v.z, v.w)); }

// The K best keys a warp has been offered, lane j < K holding the j-th best (0 = empty).
struct WarpQueue {
    uint64_t q, kth;   // kth: key in lane K-1 (same in all lanes)
    int K;
    __device__ __forceinline__ void init(int k) { q = 0; kth = 0; K = k; }
    // Called by the whole warp with the same key in every lane.
    __device__ __forceinline__ void insert(uint64_t cand, int lane) {
        const unsigned gt = __ballot_sync(0xffffffffu, q > cand);   // lanes >= K hold 0
        const int pos = __popc(gt);
        const uint64_t up = __shfl_up_sync(0xffffffffu, q, 1);
        if (lane < K && lane >= pos) q = (lane == pos) ? cand : up;
        kth = __shfl_sync(0xffffffffu, q, K - 1);
    }
};

// ---- asynchronous copies of a thread's own pieces ----
__device__ __forceinline__ void copy16(uint32_t dst, const float4* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int kPending>
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(kPending) : "memory"); }

// ---- the same shared-memory location in the first CTA of the cluster ----
__device__ __forceinline__ uint32_t lead_addr(const void* ptr) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"((uint32_t)__cvta_generic_to_shared(ptr)));
    return r;
}
__device__ __forceinline__ void st_cluster(uint32_t addr, uint64_t v) {
    asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(addr), "l"(v) : "memory");
}

struct ExpandParams {
    const float* logits;
    int64_t row_stride;
    int rows, vocab, chunk_len, k, k_entropy, K;
    int32_t* topk_idx;
    float *topk_logprob, *entropy_full, *entropy_topk, *alpha, *lse;
    const int32_t *parent, *rank, *node_offsets, *root_token;
    int batch;
    int32_t* draft_token;
    int32_t* status;
    double inv_ln_k;                             // 1 / ln(k_entropy)
};

// A well-formed tree of the batch that row `row` belongs to.
__device__ __forceinline__ bool row_of_tree(const ExpandParams& p, int b, int row, int* n0_out, int* n_out) {
    const int n0 = p.node_offsets[b];
    const int n = p.node_offsets[b + 1] - n0;
    *n0_out = n0;
    *n_out = n;
    if (n < 1 || n > SAGE_MAX_NODES || n0 < 0 || n0 + n > p.rows) {
        if (row == 0) report_status(p.status, SAGE_STATUS_BAD_TREE);
        return false;
    }
    return row >= n0 && row < n0 + n;
}

// draft_token[i] = topk_idx[row(parent(i))][rank(i)] (Section 2.2 "Tree-based Drafting") for the children i of the
// node this row stands for; one warp.  s_idx: the row's candidates.
__device__ __forceinline__ void hand_tokens(const ExpandParams& p, int row, int lane, const int32_t* s_idx) {
    for (int b0 = 0; b0 < p.batch; b0 += 32) {
        int n0 = 0, n = 0;
        unsigned hit = __ballot_sync(0xffffffffu, b0 + lane < p.batch && row_of_tree(p, b0 + lane, row, &n0, &n));
        while (hit) {
            const int src = __ffs(hit) - 1;
            hit &= hit - 1;
            const int t0 = __shfl_sync(0xffffffffu, n0, src), tn = __shfl_sync(0xffffffffu, n, src);
            const int u = row - t0;                      // this row's node
            for (int i = lane; i < tn; i += 32) {
                const int par = p.parent[t0 + i], r = p.rank[t0 + i];
                const bool ok = par >= 0 && par < i && r >= 0 && r < p.k;
                if (i == u) {
                    if (i == 0) {
                        p.draft_token[t0] = p.root_token[b0 + src];
                    } else if (!ok) {
                        report_status(p.status, SAGE_STATUS_BAD_TREE);
                        p.draft_token[t0 + i] = -1;
                    }
                } else if (i > 0 && ok && par == u) {
                    p.draft_token[t0 + i] = s_idx[r];
                }
            }
        }
    }
}

// A threshold that at least K of the CTA's elements reach (see the top of the file), as a value key; 0 lets everything
// pass.  top_key: key of this thread's largest element so far; *most: the largest of the warps' values.  r: the choice that
// lets the fewest elements pass (ten batches of normal data: K = 4, r = 1 / 2: 17 / 24; K = 8, r = 1 / 2 / 3: 76 / 42 / 57;
// K = 10, r = 2 / 3: 52 / 72; K = 16, r = 2 / 3 / 4: 119 / 100 / 98).
__device__ __forceinline__ uint32_t cta_threshold(int K, uint32_t top_key, uint32_t* s_wtop, uint32_t* most, int lane, int warp) {
    const int r_th = K <= 5 ? 1 : K <= 12 ? 2 : 3;
    const int q_th = (K + r_th - 1) / r_th;
    uint32_t wt = __reduce_max_sync(0xffffffffu, top_key);
    for (int n = __popc(__ballot_sync(0xffffffffu, top_key == wt)); n < r_th;) {
        top_key = top_key == wt ? 0u : top_key;
        wt = __reduce_max_sync(0xffffffffu, top_key);
        n += __popc(__ballot_sync(0xffffffffu, top_key == wt));
    }
    if (lane == 0) s_wtop[warp] = wt;
    __syncthreads();
    const uint32_t v = s_wtop[lane & (kWarps - 1)];
    int ge = 0;
    *most = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
        const uint32_t o = s_wtop[w];
        ge += (o >= v) ? 1 : 0;
        *most = max(*most, o);
    }
    return __reduce_max_sync(0xffffffffu, ge >= q_th ? v : 0u);
}

// Number of the n keys (n a multiple of 8, the list padded with 0) above `mine`.
__device__ __forceinline__ int rank_of(const uint64_t* keys, int n, uint64_t mine) {
    int rank = 0;
    for (int j = 0; j < n; j += 8) {
        ulonglong2 k[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) k[u] = *reinterpret_cast<const ulonglong2*>(keys + j + 2 * u);
#pragma unroll
        for (int u = 0; u < 4; ++u) rank += (k[u].x > mine ? 1 : 0) + (k[u].y > mine ? 1 : 0);
    }
    return rank;
}

__global__ void __launch_bounds__(kThreads, kCtasPerSm) expand_topk_kernel(const ExpandParams p) {
    extern __shared__ float4 s_stream[];                         // [kStages][kBatch][kThreads]
    __shared__ uint32_t s_thr;                                   // threshold raised by full queues
    __shared__ uint32_t s_wtop[2][kWarps];
    __shared__ float s_wref[kWarps];
    __shared__ double s_ws[kWarps], s_wt[kWarps];
    __shared__ __align__(16) uint64_t s_list[kListCap + kWarps * SAGE_MAX_TOPK];   // candidates; what the queues hold
    __shared__ int s_n, s_nq;                                    // of both (s_n goes on counting past kListCap)
    // written by every CTA of the cluster in its first CTA
    __shared__ uint64_t s_stat[kMaxChunks][3];                   // moments (M, S, T), as doubles
    __shared__ __align__(16) uint64_t s_ckeys[kMaxChunks * SAGE_MAX_TOPK];     // K best keys of every CTA, 0 where there are fewer
    __shared__ uint64_t s_best[SAGE_MAX_TOPK];
    __shared__ int32_t s_idx[SAGE_MAX_TOPK];
    after_previous_kernel();
    const int chunk = blockIdx.x, row = blockIdx.y, n_chunks = gridDim.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int begin = chunk * p.chunk_len;
    const int end = min(p.vocab, begin + p.chunk_len);
    const float* rowp = p.logits + (int64_t)row * p.row_stride;
    const int n4 = max(0, end - begin) >> 2;                     // 16-byte pieces: `begin` and row_stride are multiples of 4 elements
    const float4* src4 = reinterpret_cast<const float4*>(rowp + begin);
    const int n_tail = max(0, end - begin) & 3;                  // ragged end of the last chunk, one element to each of the first lanes
    // this thread's pieces of batch b (a group even when there are none)
    auto start = [&](int b) {
        const int i0 = b * kBatch * kThreads + tid;
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(s_stream + (b % kStages) * kBatch * kThreads + tid);
#pragma unroll
        for (int u = 0; u < kBatch; ++u)
            if (i0 + u * kThreads < n4) copy16(dst + u * kThreads * 16, src4 + i0 + u * kThreads);
        copy_commit();
    };
#pragma unroll
    for (int b = 0; b < kStages; ++b) start(b);
    // (read and raised after the barrier in the first cta_threshold)
    for (int i = tid; i < kListCap + kWarps * SAGE_MAX_TOPK; i += kThreads) s_list[i] = 0;
    if (tid == 0) { s_n = 0; s_nq = 0; s_thr = 0; }
    if (tid < SAGE_MAX_TOPK) { s_best[tid] = 0; s_idx[tid] = -1; }       // (stays where a row has fewer candidates, all others NaN)
    // (the other half of this barrier, before the first store to the first CTA's memory: that CTA runs by then)
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");

    // ---- 1. and 2.: the stream
    Moments mo;
    mo.init();
    WarpQueue wq;
    wq.init(p.K);
    {
        const int n_batch = (n4 + kBatch * kThreads - 1) / (kBatch * kThreads);
        // Value key that this warp's elements still have to reach: above what K elements in front of them reach already, since
        // of equal values the lowest index counts.
        uint32_t least = 0;
        float top = -INFINITY;                                   // this thread's largest element so far
        for (int b = 0; b < n_batch; ++b) {
            copy_wait<kStages - 1>();
            const int i0 = b * kBatch * kThreads + tid;
            const float4* buf = s_stream + (b % kStages) * kBatch * kThreads;
            float4 v[kBatch];
            float mx4[kBatch];
#pragma unroll
            for (int u = 0; u < kBatch; ++u) {
                v[u] = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
                if (i0 + u * kThreads < n4) v[u] = buf[u * kThreads + tid];
                mx4[u] = max4(v[u]);
            }
            const float mx = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3]));
            top = fmaxf(top, mx);
            uint32_t thr = least;
            if ((b & (b + 1)) == 0) {
                // after batches 0, 1, 3, 7, ...: as many elements pass in each doubling of the stream
                uint32_t most;
                const uint32_t reached = cta_threshold(p.K, top == -INFINITY ? 0u : order_key(top), s_wtop[__popc(b) & 1], &most, lane, warp);
                thr = max(thr, reached);
                least = max(least, reached ? reached + 1 : 0);   // (from the next batch on)
                // threads share their first reference, so that the sums hardly ever need rescaling when they are merged
                if (b == 0 && most) mo.m = fmaxf(mo.m, key_value(most));
            }
            thr = max(thr, *(volatile uint32_t*)&s_thr);
            const float thr_x = thr ? key_value(thr) : -INFINITY;
            if (__any_sync(0xffffffffu, mx >= thr_x)) {
                // this thread's elements that reach the threshold, one bit each
                uint32_t mask = 0;
#pragma unroll
                for (int u = 0; u < kBatch; ++u) {
                    if (i0 + u * kThreads < n4)
                        mask |= ((v[u].x >= thr_x ? 1u : 0u) | (v[u].y >= thr_x ? 2u : 0u) | (v[u].z >= thr_x ? 4u : 0u) |
                                 (v[u].w >= thr_x ? 8u : 0u)) << (4 * u);
                }
                if (__reduce_add_sync(0xffffffffu, __popc(mask)) > 2 * 32) {
                    // Many at a time, equal ones most likely (masked words): of those at the threshold itself only the first K
                    // count, and whole pieces in front of an element, in this warp, tell most of the others.
                    int before = 0;
#pragma unroll
                    for (int u = 0; u < kBatch; ++u) {
                        const unsigned whole = __ballot_sync(0xffffffffu, ((mask >> (4 * u)) & 15u) == 15u);
                        if (before + 4 * __popc(whole & ((1u << lane) - 1u)) >= p.K)
                            mask &= ~(((v[u].x == thr_x ? 1u : 0u) | (v[u].y == thr_x ? 2u : 0u) | (v[u].z == thr_x ? 4u : 0u) |
                                       (v[u].w == thr_x ? 8u : 0u)) << (4 * u));
                        before += 4 * __popc(whole);
                    }
                }
                if (mask) {
                    int at = atomicAdd(&s_n, __popc(mask));
                    for (; mask != 0 && at < kListCap; ++at) {
                        const int e = __ffs(mask) - 1;
                        mask &= mask - 1;
                        const int piece = (e >> 2) * kThreads + tid;
                        s_list[at] = make_key(reinterpret_cast<const float*>(buf + piece)[e & 3],
                                              begin + 4 * (b * kBatch * kThreads + piece) + (e & 3));
                    }
                }
                if (__any_sync(0xffffffffu, mask != 0)) {
                    // The list is full (ascending or masked data, many equal values): the warp's queue takes the rest, the best
                    // of all lanes first, so that a batch costs it K insertions at most.
                    const int at0 = begin + 4 * (b * kBatch * kThreads + tid);
                    auto best_left = [&]() {
                        uint64_t best = 0;
                        for (uint32_t m = mask; m; m &= m - 1) {
                            const int e = __ffs(m) - 1, piece = (e >> 2) * kThreads;
                            const uint64_t key = make_key(reinterpret_cast<const float*>(buf + piece + tid)[e & 3], at0 + 4 * piece + (e & 3));
                            best = key > best ? key : best;
                        }
                        return best;
                    };
                    uint64_t mine = best_left();
                    while (true) {
                        const uint32_t hi = __reduce_max_sync(0xffffffffu, (uint32_t)(mine >> 32));
                        const uint32_t lo = __reduce_max_sync(0xffffffffu, (uint32_t)(mine >> 32) == hi ? (uint32_t)mine : 0u);
                        const uint64_t best = ((uint64_t)hi << 32) | lo;
                        if (best <= wq.kth) break;
                        wq.insert(best, lane);
                        if (mine == best) {
                            const int off = (int)(0xffffffffu - lo) - at0;       // 4 * piece + element
                            mask &= ~(1u << (off / (4 * kThreads) * 4 + (off & 3)));
                            mine = best_left();
                        }
                    }
                    const uint32_t kth = (uint32_t)(wq.kth >> 32);
                    if (kth) least = max(least, kth + 1);
                    if (lane == 0 && kth > thr) atomicMax(&s_thr, kth);
                }
            }
            mo.rise(mx);
            start(b + kStages);                                  // (into the slots just read)
            if ((b + 1) * kBatch * kThreads <= n4) mo.add_batch<true>(v, kBatch);
            else mo.add_batch<false>(v, i0 < n4 ? (n4 - 1 - i0) / kThreads + 1 : 0);
        }
        copy_wait<0>();
        if (warp == 0) {
            for (int j = 0; j < n_tail; ++j) {
                const int i = begin + 4 * n4 + j;
                const float x = rowp[i];
                const uint64_t key = make_key(x, i);
                if (x == x && key > wq.kth) wq.insert(key, lane);
                if (lane == j) mo.add1(x);
            }
        }
        const unsigned have = __ballot_sync(0xffffffffu, wq.q != 0);
        if (have) {
            int at = 0;
            if (lane == 0) at = atomicAdd(&s_nq, __popc(have));
            at = __shfl_sync(0xffffffffu, at, 0);
            if (wq.q != 0) s_list[kListCap + at + lane] = wq.q;
        }
    }
    // the warp's moments, in fp64 under the warp's reference
    {
        float wr = mo.m;
        for (int o = 16; o > 0; o >>= 1) wr = fmaxf(wr, __shfl_xor_sync(0xffffffffu, wr, o));
        float s0, s1, t0, t1;
        f2_unpack(mo.s2, s0, s1);
        f2_unpack(mo.t2, t0, t1);
        double ds = (double)s0 + (double)s1, dt = (double)t0 + (double)t1;
        if (!__all_sync(0xffffffffu, mo.m == wr)) {
            if (ds > 0.0) {
                const double dm = (double)mo.m - (double)wr;
                const double c = exp(dm);
                dt = c * (dt + dm * ds);
                ds *= c;
            }
        }
        for (int o = 16; o > 0; o >>= 1) {
            ds += __shfl_xor_sync(0xffffffffu, ds, o);
            dt += __shfl_xor_sync(0xffffffffu, dt, o);
        }
        if (lane == 0) { s_wref[warp] = wr; s_ws[warp] = ds; s_wt[warp] = dt; }
    }
    __syncthreads();
    // ---- 3. the moments of this CTA (the last warp) and its K best keys (the others) go to the first CTA of the cluster
    asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
    if (warp == kWarps - 1) {
        const int w = lane & (kWarps - 1);
        const float wr = s_wref[w];
        float ref = wr;
        for (int o = kWarps / 2; o > 0; o >>= 1) ref = fmaxf(ref, __shfl_xor_sync(0xffffffffu, ref, o));
        double ds = s_ws[w], dt = s_wt[w];
        if (!__all_sync(0xffffffffu, wr == ref)) {
            if (ds > 0.0) {
                const double dm = (double)wr - (double)ref;
                const double c = exp(dm);
                dt = c * (dt + dm * ds);
                ds *= c;
            }
        }
        for (int o = kWarps / 2; o > 0; o >>= 1) {
            ds += __shfl_xor_sync(0xffffffffu, ds, o);
            dt += __shfl_xor_sync(0xffffffffu, dt, o);
        }
        if (lane < 3)
            st_cluster(lead_addr(&s_stat[chunk][lane]), (uint64_t)__double_as_longlong(lane == 0 ? (double)ref : lane == 1 ? ds : dt));
    } else {
        const int n = min(s_n, kListCap), nq = s_nq;
        const uint32_t keys = lead_addr(&s_ckeys[chunk * SAGE_MAX_TOPK]);
        for (int i = tid; i < n + nq; i += kThreads - 32) {
            const uint64_t mine = s_list[i < n ? i : kListCap + i - n];
            int rank = rank_of(s_list, (n + 7) & ~7, mine);              // keys are unique
            if (nq) rank += rank_of(s_list + kListCap, (nq + 7) & ~7, mine);
            if (rank < p.K) st_cluster(keys + rank * 8, mine);
        }
        if (tid >= min(n + nq, p.K) && tid < SAGE_MAX_TOPK) st_cluster(keys + tid * 8, 0);
    }
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (chunk != 0) return;

    // ---- the row: lse and entropy in warp 0; meanwhile four warps rank every CTA's keys among all, and one of them goes on
    // with the entropy of the best ones, which needs no lse
    if (warp > 4) return;
    if (warp == 0) {
        double lse;
        double Mc = -INFINITY, Sc = 0.0, Tc = 0.0;
        if (lane < n_chunks) {
            Mc = __longlong_as_double((long long)s_stat[lane][0]);
            Sc = __longlong_as_double((long long)s_stat[lane][1]);
            Tc = __longlong_as_double((long long)s_stat[lane][2]);
        }
        double M = Mc;
        for (int o = 4; o > 0; o >>= 1) M = fmax(M, __shfl_xor_sync(0xffffffffu, M, o));
        M = __shfl_sync(0xffffffffu, M, 0);
        double S = 0.0, T = 0.0;
        if (Sc > 0.0) {
            const double dm = Mc - M, c = exp(dm);
            S = c * Sc;
            T = c * (Tc + dm * Sc);
        }
        for (int o = 4; o > 0; o >>= 1) {
            S += __shfl_xor_sync(0xffffffffu, S, o);
            T += __shfl_xor_sync(0xffffffffu, T, o);
        }
        // (lanes 0 .. 7 hold the sums; log-probabilities are needed in up to 16 lanes)
        S = __shfl_sync(0xffffffffu, S, 0);
        T = __shfl_sync(0xffffffffu, T, 0);
        const double lnS = log(S);
        lse = M + lnS;
        if (lane == 0) {
            if (p.lse) p.lse[row] = (float)lse;
            if (p.entropy_full) p.entropy_full[row] = (float)(lnS - T / S);
        }
        asm volatile("bar.sync 1, 160;" ::: "memory");                   // the keys are ranked
        if (lane < p.k && p.topk_logprob)
            p.topk_logprob[(size_t)row * p.k + lane] = (float)((double)key_value((uint32_t)(s_best[lane] >> 32)) - lse);
        return;
    }
    if (tid - 32 < n_chunks * SAGE_MAX_TOPK) {
        const uint64_t mine = s_ckeys[tid - 32];
        if (mine != 0) {
            const int rank = rank_of(s_ckeys, n_chunks * SAGE_MAX_TOPK, mine);
            if (rank < p.K) {
                s_best[rank] = mine;
                s_idx[rank] = (int32_t)(0xffffffffu - (uint32_t)mine);
            }
        }
    }
    asm volatile("bar.arrive 1, 160;" ::: "memory");
    asm volatile("bar.sync 2, 128;" ::: "memory");
    if (warp == 1) {
        if (lane < p.k) p.topk_idx[(size_t)row * p.k + lane] = s_idx[lane];
        if (p.draft_token) hand_tokens(p, row, lane, s_idx);
    } else if (warp == 2 && (p.entropy_topk || p.alpha)) {
        const bool have = lane < p.k_entropy && s_best[lane] != 0;
        const double v = have ? (double)key_value((uint32_t)(s_best[lane] >> 32)) : 0.0;
        const double v1 = __shfl_sync(0xffffffffu, v, 0);
        double w = 0.0, wd = 0.0;                        // w_j = P_j / P_1
        if (have) {
            const double d = v - v1;
            w = exp(d);
            wd = w * d;
        }
        for (int o = 8; o > 0; o >>= 1) {
            w += __shfl_xor_sync(0xffffffffu, w, o);
            wd += __shfl_xor_sync(0xffffffffu, wd, o);
        }
        if (lane == 0) {
            // P~_j = w_j / wsum;  H = -sum P~ ln P~ = ln(wsum) - sum w ln w / wsum
            const double H = log(w) - wd / w;
            if (p.entropy_topk) p.entropy_topk[row] = (float)H;
            if (p.alpha) p.alpha[row] = p.k_entropy > 1 ? (float)fmin(1.0, fmax(0.0, 1.0 - H * p.inv_ln_k)) : 1.0f;
        }
    }
}

// The opt-in to more than 48 KB of shared memory is a per-device attribute of the kernel.
static bool allow_stream_buffer() {
    static std::atomic<bool> done[64];
    int dev = 0;
    if (!succeeded(cudaGetDevice(&dev)) || dev < 0 || dev >= 64) return false;
    if (!done[dev].load(std::memory_order_acquire)) {
        if (!succeeded(cudaFuncSetAttribute(expand_topk_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kStreamBytes))) return false;
        done[dev].store(true, std::memory_order_release);
    }
    return true;
}

// CTAs per row.  Up to 148 rows: as many as fit two to an SM, since two CTAs of an SM take little longer than one and three
// nearly twice as long (clusters of three and more do not pack the SMs quite full).  us at K = 10, 152064 words: 36 rows, 6 / 7 /
// 8 CTAs: 12.8 / 13.1 / 15.9; 56 rows, 4 / 5 / 6: 15.5 / 14.6 / 18.1; 88 rows, 2 / 3 / 4: 21.9 / 19.5 / 22.6; 148 rows, 1 / 2 / 3:
// 27.3 / 22.9 / 26.7.  Beyond that long rows are cut where it makes up for SMs that would wait: 180 rows, 1 / 3: 34.1 /
// 27.2; 400 rows, 1 / 2: 55.1 / 49.0; 560 rows: 59.5 / 62.6; 672 rows, K = 1: 83.2 / 69.1; 800 rows: 85.0 / 86.9.  (Rows of
// 32000 gain nothing there: 180 rows, 1 / 3: 12.7 / 13.7; 640 rows, 1 / 2: 21.9 / 24.3.)
static int pick_chunks(int rows, int vocab) {
    constexpr int kSms = 148;
    const int batch = kBatch * 4 * kThreads;
    for (int c = kMaxChunks; c >= 2; --c) {                      // (a CTA gets more than (c - 1) / c of a batch)
        if ((c - 1) * batch < vocab && (long)c * rows <= (c > 2 ? 272 : 2 * kSms)) return c;
    }
    if (vocab < 16 * batch) return 1;
    if (3 * (long)rows <= 544) return 3;
    return (rows > 2 * kSms && rows <= 3 * kSms) || (rows > 4 * kSms && rows <= 5 * kSms) ? 2 : 1;
}

// Scratch that callers hand in: the size that they were always asked for (24 bytes of moments and SAGE_MAX_TOPK keys
// for each of up to 32 chunks of a row).  Results pass from CTA to CTA in distributed shared memory, the buffer is not
// written.
static size_t workspace_bytes(int rows, int vocab) {
    int c = (592 + rows - 1) / rows;
    const int max_by_len = (vocab + 4095) / 4096;
    if (c > max_by_len) c = max_by_len;
    if (c > 32) c = 32;
    if (c < 1) c = 1;
    return (size_t)rows * c * (3 * sizeof(double) + SAGE_MAX_TOPK * sizeof(uint64_t));
}

static int launch_expand(const ExpandParams& p, cudaStream_t stream) {
    if (!allow_stream_buffer()) return SAGE_ERR_CUDA;
    const int C = pick_chunks(p.rows, p.vocab);
    ExpandParams q = p;
    q.chunk_len = (((p.vocab + C - 1) / C) + 3) & ~3;
    return launch_status(launch(expand_topk_kernel, dim3((unsigned)C, (unsigned)p.rows), kThreads, kStreamBytes, stream, C, q));
}

}  // namespace sage

using namespace sage;

extern "C" size_t sage_expand_topk_workspace_size(int rows, int vocab) {
    if (rows <= 0 || vocab <= 0) return 0;
    return workspace_bytes(rows, vocab);
}

// Checks of the arguments that both entry points share, then the launch.
static int expand_topk(const float* logits, int rows, int vocab, int64_t row_stride, int k, int k_entropy,
                       int32_t* topk_idx, float* topk_logprob, float* entropy_full, float* entropy_topk,
                       float* alpha, float* lse, const int32_t* parent, const int32_t* rank,
                       const int32_t* node_offsets, int batch, const int32_t* root_token,
                       int32_t* draft_token, bool have_ws, int32_t* status, void* stream) {
    if (!logits || !topk_idx || rows < 0 || vocab < 1 || row_stride < vocab) return SAGE_ERR_INVALID_ARG;
    if (k < 1 || k_entropy < 1) return SAGE_ERR_INVALID_ARG;
    if (k > SAGE_MAX_TOPK || k_entropy > SAGE_MAX_TOPK) return SAGE_ERR_UNSUPPORTED;
    const int K = k > k_entropy ? k : k_entropy;
    if (K > vocab) return SAGE_ERR_INVALID_ARG;
    if (((uintptr_t)logits & 15) || (row_stride & 3)) return SAGE_ERR_UNSUPPORTED;
    if (draft_token && (!parent || !rank || !node_offsets || !root_token || batch < 0)) return SAGE_ERR_INVALID_ARG;
    if (rows == 0) return SAGE_OK;
    if (rows > 65535) return SAGE_ERR_UNSUPPORTED;
    if (!have_ws) return SAGE_ERR_WORKSPACE;
    ExpandParams p{logits, row_stride, rows, vocab, 0, k, k_entropy, K, topk_idx, topk_logprob, entropy_full,
                   entropy_topk, alpha, lse, parent, rank, node_offsets, root_token, batch,
                   batch > 0 ? draft_token : nullptr, status, k_entropy > 1 ? 1.0 / log((double)k_entropy) : 0.0};
    return launch_expand(p, as_stream(stream));
}

extern "C" int sage_expand_topk(const float* logits, int rows, int vocab, int64_t row_stride, int k, int k_entropy,
                                int32_t* topk_idx, float* topk_logprob, float* entropy_full, float* entropy_topk,
                                float* alpha, float* lse, const int32_t* parent, const int32_t* rank,
                                const int32_t* node_offsets, int batch, const int32_t* root_token,
                                int32_t* draft_token, void* ws, size_t ws_bytes, int32_t* status, void* stream) {
    const bool have_ws = ws && !((uintptr_t)ws & 15) && ws_bytes >= sage_expand_topk_workspace_size(rows, vocab);
    return expand_topk(logits, rows, vocab, row_stride, k, k_entropy, topk_idx, topk_logprob, entropy_full, entropy_topk,
                       alpha, lse, parent, rank, node_offsets, batch, root_token, draft_token, have_ws, status, stream);
}

// The same without a scratch argument, within the size limit that the header states.
extern "C" int sage_expand_topk_static(const float* logits, int rows, int vocab, int64_t row_stride, int k,
                                       int k_entropy, int32_t* topk_idx, float* topk_logprob, float* entropy_full,
                                       float* entropy_topk, float* alpha, float* lse, const int32_t* parent,
                                       const int32_t* rank, const int32_t* node_offsets, int batch,
                                       const int32_t* root_token, int32_t* draft_token, int32_t* status,
                                       void* stream) {
    if (rows < 0 || vocab < 1) return SAGE_ERR_INVALID_ARG;
    if (rows > 0 && sage_expand_topk_workspace_size(rows, vocab) > (size_t)SAGE_STATIC_SCRATCH_BYTES)
        return SAGE_ERR_TOO_LARGE;
    return expand_topk(logits, rows, vocab, row_stride, k, k_entropy, topk_idx, topk_logprob, entropy_full, entropy_topk,
                       alpha, lse, parent, rank, node_offsets, batch, root_token, draft_token, true, status, stream);
}
