// Tree-masked verification attention over a paged bf16 KV cache (Section 2.2;
// Algorithm 1, the target pass over all tree tokens; Section 3.3 Phase 2), sm_100a:
// the C entry points, the tensor maps and the choice of schedule.  The kernels are in tree_attention_rows.cu and
// tree_attention_alt.cu (streaming schedule, launched from the latter) and tree_attention_split.cu (split schedule).
#include <cuda.h>

#include <mutex>

#include "sage_common.cuh"

namespace sage {

constexpr int kRowTile = 128;                            // query rows per MMA tile
constexpr long long kWaitCyclesDefault = 4000000000ll;   // ~2 s at 2 GHz: far beyond any legitimate wait

// ---- host side ------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* sym = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (succeeded(cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &sym, cudaEnableDefault, &qres)) &&
            qres == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(sym);
    }
    return fn;
}

// Tensor maps depend only on (base pointer, shape); a serving loop calls with the same few buffers
// over and over, so the last few encodings are kept.
struct MapKey {
    const void* base;
    long long a, b, c, d;
    int kind;
    bool operator==(const MapKey& o) const {
        return base == o.base && a == o.a && b == o.b && c == o.c && d == o.d && kind == o.kind;
    }
};
constexpr int kMapCache = 16;
static std::mutex g_map_mu;
static MapKey g_map_key[kMapCache];
static CUtensorMap g_map_val[kMapCache];
static int g_map_used = 0, g_map_next = 0;

template <typename Make>
static bool cached_map(CUtensorMap* out, const MapKey& key, Make make) {
    std::lock_guard<std::mutex> lock(g_map_mu);
    for (int i = 0; i < g_map_used; ++i)
        if (g_map_key[i] == key) { *out = g_map_val[i]; return true; }
    if (!make(out)) return false;
    g_map_key[g_map_next] = key;
    g_map_val[g_map_next] = *out;
    g_map_next = (g_map_next + 1) % kMapCache;
    if (g_map_used < kMapCache) ++g_map_used;
    return true;
}

// Pool viewed as [layer][page*Hkv + head][slot][d]; one box = one 64-wide d-half of one (page, head).
static bool make_pool_map(CUtensorMap* map, const void* pool, int n_layers, int n_pages, int n_kv_heads,
                          int64_t layer_stride_elems) {
    const MapKey key{pool, n_layers, n_pages, n_kv_heads, layer_stride_elems, 0};
    return cached_map(map, key, [&](CUtensorMap* m) {
        EncodeTiledFn fn = encode_fn();
        if (!fn) return false;
        const cuuint64_t page_head_bytes = (cuuint64_t)kPageSize * kHeadDim * 2;
        cuuint64_t dims[4] = {(cuuint64_t)kHeadDim, (cuuint64_t)kPageSize, (cuuint64_t)n_pages * n_kv_heads,
                              (cuuint64_t)n_layers};
        cuuint64_t layer_bytes = n_layers > 1 ? (cuuint64_t)layer_stride_elems * 2 : dims[2] * page_head_bytes;
        cuuint64_t strides[3] = {(cuuint64_t)kHeadDim * 2, page_head_bytes, layer_bytes};
        cuuint32_t box[4] = {64, (cuuint32_t)kPageSize, 1, 1};
        cuuint32_t estr[4] = {1, 1, 1, 1};
        return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(pool), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    });
}

// Queries viewed as [layer][node][kv head][head in group][d]; one box = one 64-wide d-half of the
// 128 query rows (128/G nodes x G heads) of a row tile.  Nodes past sum_nodes read as zero.
static bool make_q_map(CUtensorMap* map, const void* q, int n_layers, int sum_nodes, int n_kv_heads, int G) {
    const MapKey key{q, n_layers, sum_nodes, n_kv_heads, G, 1};
    return cached_map(map, key, [&](CUtensorMap* m) {
        EncodeTiledFn fn = encode_fn();
        if (!fn) return false;
        const cuuint64_t row = (cuuint64_t)kHeadDim * 2;
        cuuint64_t dims[5] = {(cuuint64_t)kHeadDim, (cuuint64_t)G, (cuuint64_t)n_kv_heads, (cuuint64_t)sum_nodes,
                              (cuuint64_t)n_layers};
        cuuint64_t strides[4] = {row, row * G, row * G * n_kv_heads, row * G * n_kv_heads * sum_nodes};
        cuuint32_t box[5] = {64, (cuuint32_t)G, 1, (cuuint32_t)(kRowTile / G), 1};
        cuuint32_t estr[5] = {1, 1, 1, 1, 1};
        return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(q), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    });
}

// One resident CTA per SM (148 when no device can be asked, e.g. a size query on a host without a GPU).
static int resident_ctas() {
    static int cached[64] = {};
    int dev = 0;
    if (!succeeded(cudaGetDevice(&dev)) || dev < 0 || dev >= 64) return 148;
    if (!cached[dev]) {
        int n = 0;
        if (!succeeded(cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev)) || n < 1) return 148;
        cached[dev] = n;
    }
    return cached[dev];
}
static long long g_wait_cycles = kWaitCyclesDefault;
static int g_producer_off = 0;
static int g_schedule = 0;     // 0: chosen per launch, 2: split, else streaming

// The split schedule (tree_attention_split.cu).
namespace split {
double estimate(int n_sms, int n_layers, int batch, int sum_nodes, int n_q_heads, int n_kv_heads, int max_pages_per_seq);
int slices(int n_sms, int n_layers, int batch, int sum_nodes, int n_q_heads, int n_kv_heads, int max_pages_per_seq);
bool merge_overlaps(int n_sms, int n_layers, int batch, int sum_nodes, int n_q_heads, int n_kv_heads, int S);
size_t workspace_size(int n_sms, int n_layers, int batch, int sum_nodes, int n_q_heads, int n_kv_heads, int max_pages_per_seq);
int launch(int n_sms, int n_layers, int n_pages, const int32_t* page_table, int max_pages_per_seq,
           const int32_t* seq_len, const int32_t* parent, const int32_t* node_offsets, int batch, int sum_nodes,
           int n_q_heads, int n_kv_heads, float sm_scale, void* out, void* ws, int32_t* status, long long wait_cycles,
           int producer_off, const CUtensorMap& qmap, const CUtensorMap& kmap, const CUtensorMap& vmap, cudaStream_t stream);
}  // namespace split

// The streaming schedule (tree_attention_alt.cu).
namespace stream {
size_t workspace_size(int n_ctas);
int launch(int n_ctas, int n_layers, int n_pages, const int32_t* page_table, int max_pages_per_seq,
           const int32_t* seq_len, const int32_t* parent, const int32_t* node_offsets, int batch, int sum_nodes,
           int n_q_heads, int n_kv_heads, float sm_scale, void* out, void* ws, int32_t* status, long long wait_cycles,
           int producer_off, const CUtensorMap& qmap, const CUtensorMap& kmap, const CUtensorMap& vmap,
           cudaStream_t stream);
}  // namespace stream

// Which schedule runs a launch.
//   streaming: persistent CTAs that walk equal ranges of 128-key steps, whatever the batch looks like.
//   split: grid over (context slice, row pair, layer x sequence x KV head), 64-key steps: shorter set-up and no plan, for
//     launches too short to give every SM a long stream (single layers, short contexts: fixed costs dominate).
// The line lies where both take the same time (us, split / streaming; steps per SM in brackets; 8 KV heads of 8 queries;
// bursts of a few ms, in longer loops the power limit takes 10 to 20 % off the lead of the split schedule):
//   one sequence, up to one row pair: 24 nodes, 16k keys, 4 layers (28) 71/74, 8 (56) 157/150; 12 nodes, 4k keys, 16 layers (28) 60/62,
//     24 (43) 107/86, 32 (57) 124/106;
//   one sequence whose node arrays have room for two row pairs: 60 nodes, 16k keys, 3 layers (21) 110/121, 4 (28) 155/148; but nine
//     nodes in such arrays, for which half of the split grid is empty, 2 layers (14) 53/52, 4 (28) 93/69;
//   several sequences, long: the split grid is as uneven as their lengths.  1k to 8k keys, 24 to 60 nodes: four sequences (14) 66/48,
//     eight (28) 116/91, sixteen of 24 nodes (56) 138/103; eight of 2k keys, 36 nodes (7) 40/56.
// Above the line, several sequences under narrow page tables: what decides is how full the last wave of the split grid is, a block per item
// and slice.  Both schedules are estimated in pages of 64 keys (split::estimate; streaming: the items' pages and extra over the SMs, and 21
// for plan, first copies and merge), and the split schedule is taken when it is ahead by a twentieth.  8 KV heads of 8 queries, split /
// streaming: 16 sequences of 1.7k keys, 12 nodes 28/43, 24 nodes 34/51, 60 nodes 67/83; 19: 54/51, 58/57, 94/94 (one item too many for a
// wave); 36: 61/70, 79/94, 147/169; 28 of 1k keys 41/52, 45/59; 18 of up to 1.7k, 24 nodes 36/46.
// Narrow: the estimates know the table's width, not the lengths, and if a single sequence fills it while the others are short, a split launch
// takes what the pages of that one take a block of its own (0.7 us each), a streaming one hardly more than its least.  So only as far as
// that is no loss: 16 sequences, one long and the others a tenth of it, 12 nodes, one query head per KV head, 27 pages 23/19, 33
// pages 26/21, 37 pages 29/21 (full tables 24/32, 28/36, 30/38); eight, whose ends of items cost more, 28 pages 24/24, 33 pages 28/25,
// 37 pages 30/26 (full tables 28/43, 32/47, 34/49; the streaming schedule's 25 and 26 were 29 before its ends of items were weighed).
// Below the line the split schedule runs, whatever the estimates say.  They know what a table and the node arrays can hold, not what they
// do hold, and a streaming launch takes 20 us however little there is to do: 27 sequences in tables of 21 pages an eighth full, one KV head of 8
// queries, 3 layers 12/29; twelve chains of nine nodes in arrays of 64 each, 21 full pages 22/32.  (Tight batches may pay for it: twelve
// sequences of 2k keys, 60 nodes 86/74.)
// The host knows the width of the page table, not the lengths, so a wide table takes short sequences across the line, or into
// more slices than they fill: eight sequences of 1k keys 22 us with 17 pages per row, 41 with 512; one of 2k keys, 60 nodes, 16.2
// with 33 pages, 16.1 with 512, 10 nodes 9.4 and 10.7.
static bool use_streaming(int n_layers, int batch, int sum_nodes, int n_q_heads, int n_kv_heads, int max_pages_per_seq) {
    if (g_schedule) return g_schedule != 2;
    const int G = n_q_heads / n_kv_heads;
    const int rows = (sum_nodes < SAGE_MAX_NODES ? sum_nodes : SAGE_MAX_NODES) * G;      // most that a tree can have
    const long long items = (long long)n_layers * batch * n_kv_heads;
    const long long steps = items * ((max_pages_per_seq + 1) / 2);   // upper bound
    const int line = batch > 1 ? 12 : rows > 256 ? 24 : 40;
    if (steps < (long long)line * resident_ctas()) return false;
    const int narrow = G >= 4 ? 33 : 24;
    if (batch == 1 || max_pages_per_seq > narrow || items > 65535) return true;      // (the split schedule's grid ends there)
    const int rows_avg = sum_nodes / batch * G;
    const double streaming = (double)items * (rows_avg > 256 ? 2 : 1) * (max_pages_per_seq + 4) / resident_ctas() + 21.0;
    return streaming < 1.05 * split::estimate(resident_ctas(), n_layers, batch, sum_nodes, n_q_heads, n_kv_heads, max_pages_per_seq);
}

}  // namespace sage

using namespace sage;

extern "C" size_t sage_tree_attention_workspace_size(int n_layers, int batch, int sum_nodes, int n_q_heads,
                                                     int n_kv_heads, int head_dim, int max_pages_per_seq) {
    if (n_layers < 1 || batch < 1 || sum_nodes < 1 || n_q_heads < 1 || n_kv_heads < 1 || max_pages_per_seq < 1 ||
        n_q_heads % n_kv_heads)
        return 0;
    (void)head_dim;
    // streaming: two partial slots (head and tail of its range) per resident CTA, independent of the problem size;
    // split: one partial per context slice.  Either may run, so the larger is asked for.
    const size_t streaming = stream::workspace_size(resident_ctas());
    const size_t split_ws = split::workspace_size(resident_ctas(), n_layers, batch, sum_nodes, n_q_heads, n_kv_heads, max_pages_per_seq);
    return streaming > split_ws ? streaming : split_ws;
}

extern "C" void sage_debug_attention_waits(long long wait_cycles, int producer_off) {
    g_wait_cycles = wait_cycles > 0 ? wait_cycles : kWaitCyclesDefault;
    g_producer_off = producer_off ? 1 : 0;
}

extern "C" void sage_debug_attention_schedule(int schedule) { g_schedule = (schedule >= 1 && schedule <= 3) ? schedule : 0; }

extern "C" int sage_debug_attention_plan(int n_layers, int batch, int sum_nodes, int n_q_heads, int n_kv_heads, int max_pages_per_seq, int* plan) {
    if (n_layers < 1 || batch < 1 || sum_nodes < 1 || n_q_heads < 1 || n_kv_heads < 1 || max_pages_per_seq < 1 || n_q_heads % n_kv_heads || !plan)
        return SAGE_ERR_INVALID_ARG;
    plan[0] = use_streaming(n_layers, batch, sum_nodes, n_q_heads, n_kv_heads, max_pages_per_seq) ? 1 : 2;
    plan[1] = plan[0] == 1 ? 0 : split::slices(resident_ctas(), n_layers, batch, sum_nodes, n_q_heads, n_kv_heads, max_pages_per_seq);
    plan[2] = plan[1] > 1 && split::merge_overlaps(resident_ctas(), n_layers, batch, sum_nodes, n_q_heads, n_kv_heads, plan[1]) ? 1 : 0;
    return SAGE_OK;
}

extern "C" int sage_tree_attention(const void* q, const void* k_pool, const void* v_pool, int64_t layer_stride_elems,
                                   int n_layers, int n_pages, const int32_t* page_table, int max_pages_per_seq,
                                   const int32_t* seq_len, const int32_t* parent, const int32_t* node_offsets,
                                   int batch, int sum_nodes, int n_q_heads, int n_kv_heads, int head_dim,
                                   int page_size, float sm_scale, void* out, void* ws, size_t ws_bytes,
                                   int32_t* status, void* stream) {
    if (!q || !k_pool || !v_pool || !page_table || !seq_len || !parent || !node_offsets || !out)
        return SAGE_ERR_INVALID_ARG;
    if (n_layers < 1 || n_pages < 1 || max_pages_per_seq < 1 || batch < 0 || sum_nodes < 1 || n_q_heads < 1 ||
        n_kv_heads < 1 || layer_stride_elems < 0 || !(sm_scale > 0.f))
        return SAGE_ERR_INVALID_ARG;
    if (head_dim != kHeadDim || page_size != kPageSize) return SAGE_ERR_UNSUPPORTED;
    if (n_q_heads % n_kv_heads) return SAGE_ERR_UNSUPPORTED;
    const int G = n_q_heads / n_kv_heads;
    if (G != 1 && G != 2 && G != 4 && G != 8) return SAGE_ERR_UNSUPPORTED;
    if ((long long)n_layers * batch * n_kv_heads > 0x7fffffffll || max_pages_per_seq > (1 << 24)) return SAGE_ERR_UNSUPPORTED;
    if ((((uintptr_t)q | (uintptr_t)k_pool | (uintptr_t)v_pool | (uintptr_t)out) & 15) || (layer_stride_elems & 7))
        return SAGE_ERR_INVALID_ARG;
    if (n_layers > 1 && layer_stride_elems < (int64_t)n_pages * n_kv_heads * kPageSize * kHeadDim)
        return SAGE_ERR_INVALID_ARG;
    if (batch == 0) return SAGE_OK;
    const size_t need = sage_tree_attention_workspace_size(n_layers, batch, sum_nodes, n_q_heads, n_kv_heads,
                                                           head_dim, max_pages_per_seq);
    if (!ws || ws_bytes < need || ((uintptr_t)ws & 15)) return SAGE_ERR_WORKSPACE;
    const bool streaming = use_streaming(n_layers, batch, sum_nodes, n_q_heads, n_kv_heads, max_pages_per_seq);
    if (!streaming && (long long)n_layers * batch * n_kv_heads > 65535) return SAGE_ERR_UNSUPPORTED;    // grid limit of the split schedule
    CUtensorMap qmap, kmap, vmap;
    if (!make_pool_map(&kmap, k_pool, n_layers, n_pages, n_kv_heads, layer_stride_elems) ||
        !make_pool_map(&vmap, v_pool, n_layers, n_pages, n_kv_heads, layer_stride_elems) ||
        !make_q_map(&qmap, q, n_layers, sum_nodes, n_kv_heads, G))
        return SAGE_ERR_CUDA;
    if (!streaming)
        return split::launch(resident_ctas(), n_layers, n_pages, page_table, max_pages_per_seq, seq_len, parent, node_offsets, batch,
                             sum_nodes, n_q_heads, n_kv_heads, sm_scale, out, ws, status, g_wait_cycles, g_producer_off,
                             qmap, kmap, vmap, as_stream(stream));
    return stream::launch(resident_ctas(), n_layers, n_pages, page_table, max_pages_per_seq, seq_len, parent, node_offsets,
                          batch, sum_nodes, n_q_heads, n_kv_heads, sm_scale, out, ws, status, g_wait_cycles, g_producer_off,
                          qmap, kmap, vmap, as_stream(stream));
}
