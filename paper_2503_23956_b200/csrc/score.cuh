// Shared by the scoring kernels (score.cu, score_cluster.cu): launch parameters, the tensor map over the caller's
// key cache and the load of one key tile through it.
#pragma once

#include "common.cuh"
#include "ptx.cuh"

namespace aircache {

struct ScoreParams {
    const uint16_t *k;
    int64_t s_layer, s_batch, s_head, s_token;
    const uint16_t *qw;  // [L,B,W,Hq,d]
    float *scores;       // [L,B,Nv]
    uint64_t *elite_mask;
    int32_t *row_count;
    int32_t *row_info;
    float *row_coef;
    float2 *row_text;
    float2 *chunk_stats;
    float2 *row_final;   // (max, weight / normaliser) per elite row, written by the last stats CTA of a group
    uint32_t *group_ticket;
    uint32_t *dispatch;     // one-pass scoring: blocks started so far
    float *imp_part;        // one-pass scoring: [L*B*Hkv][Nv] importance of one KV group
    uint16_t *q_block;      // one-pass scoring: [L*B*Hkv][16][d] the first 16 elite query rows, gathered
    int op_chunks;      // numbers (blocks) per KV group in the one-pass grid
    int op_tile_cap;    // most 16-key tiles a warp of the one-pass kernel takes: 16, or fewer when the call is small
    int L, B, Hq, Hkv, G, d, Nv, Nt, W;
    int lb0, n_lb;   // the launch covers regions lb0 .. lb0 + n_lb - 1 (a range of layers)
    int per_head;    // scores are kept apart per KV group: [L,B,Hkv,Nv], Eq. 8 averaged over the group's heads only
    int cap, chunks, chunk_keys;
    float scale, sl2, ln_alpha;
    int keep_all;
    // one stats launch handles the KV groups with rows_lo < elite rows <= rows_hi
    int rows_lo, rows_hi;
    // dense (tcgen05) path: position of the token / head / sequence / layer coordinate in the key tensor map
    int pos_token, pos_head, pos_batch, pos_layer;
    uint32_t *status;
};

constexpr float kNegBig = -1.0e30f;

// 5-D tensor map over the caller's key cache: channels innermost, then token / head / sequence / layer in
// the order of their strides (smallest first); one box = 64 channels x 128 tokens.
inline int make_key_map(CUtensorMap *tm, ScoreParams &p, const aircache_shape_t *s, const aircache_full_t *f) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return AIRCACHE_ERR_CUDA;
    struct Dim { int64_t size, stride; int which; };
    Dim dims[4] = {{(int64_t)s->n_visual + s->n_text, f->stride_token, 0}, {s->n_kv_heads, f->stride_head, 1},
                   {s->batch, f->stride_batch, 2}, {s->n_layers, f->stride_layer, 3}};
    for (int i = 0; i < 4; ++i)
        for (int j = i + 1; j < 4; ++j)
            if (dims[j].stride < dims[i].stride || (dims[j].stride == dims[i].stride && dims[j].size < dims[i].size)) {
                const Dim t = dims[i]; dims[i] = dims[j]; dims[j] = t;
            }
    cuuint64_t gdim[5] = {(cuuint64_t)s->head_dim, 1, 1, 1, 1};
    cuuint64_t gstr[4] = {0, 0, 0, 0};
    cuuint32_t box[5] = {64, 1, 1, 1, 1};
    const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    int pos[4] = {0, 0, 0, 0};
    for (int i = 0; i < 4; ++i) {
        if (dims[i].size > 1 && dims[i].stride == 0) return AIRCACHE_ERR_UNSUPPORTED;   // one copy shared: no tensor map
        gdim[i + 1] = (cuuint64_t)dims[i].size;
        // a dimension of extent 1 never moves; give it the smallest stride the encoder accepts
        gstr[i] = (cuuint64_t)(dims[i].stride > 0 ? dims[i].stride : s->head_dim) * 2;
        pos[dims[i].which] = i + 1;
        if (dims[i].which == 0) box[i + 1] = 128;
    }
    p.pos_token = pos[0]; p.pos_head = pos[1]; p.pos_batch = pos[2]; p.pos_layer = pos[3];
    const CUresult rc = fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void *>(f->k), gdim, gstr, box, estr,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return rc == CUDA_SUCCESS ? AIRCACHE_OK : AIRCACHE_ERR_CUDA;
}

constexpr int kKeySubBytes = 128 * 128;   // 128 keys x 64 channels

#ifdef __CUDACC__
// Coordinates 1 to 4 of a key in that map.  (Selects: an array indexed by position would live in local memory.)
__device__ __forceinline__ int4 key_coords(const ScoreParams &p, int key, int g, int b, int l) {
    auto at = [&](int i) { return p.pos_token == i ? key : p.pos_head == i ? g : p.pos_batch == i ? b : l; };
    return make_int4(at(1), at(2), at(3), at(4));
}
// One tile of 128 keys (D / 64 boxes of 64 channels, 128-byte swizzle) of KV head g of sequence b, layer l.
template <int D>
__device__ __forceinline__ void load_key_tile(uint32_t dst, const CUtensorMap *tm, const ScoreParams &p, int key,
                                              int g, int b, int l, uint32_t bar) {
    const int4 c = key_coords(p, key, g, b, l);
    mbar_expect_tx(bar, D / 64 * kKeySubBytes);
#pragma unroll
    for (int sub = 0; sub < D / 64; ++sub)
        tma_load_5d(dst + sub * kKeySubBytes, tm, sub * 64, c.x, c.y, c.z, c.w, bar);
}
// The same tile asked into L2.
template <int D>
__device__ __forceinline__ void prefetch_key_tile(const CUtensorMap *tm, const ScoreParams &p, int key, int g, int b, int l) {
    const int4 c = key_coords(p, key, g, b, l);
#pragma unroll
    for (int sub = 0; sub < D / 64; ++sub) tma_prefetch_5d(tm, sub * 64, c.x, c.y, c.z, c.w);
}

#endif

// score_cluster.cu: the scoring kernel for sequences that a cluster of up to eight blocks holds (*taken = 1 if it ran).
int launch_score_cluster(ScoreParams &p, const aircache_shape_t *s, const aircache_full_t *f, cudaStream_t st, int *taken);
// score_dense.cu: the two passes for alpha = 0 (*taken = 1 if they ran).
int launch_score_dense(ScoreParams &p, const aircache_shape_t *s, const aircache_full_t *f, cudaStream_t st, int *taken);
// score.cu: Eq. 8 over the KV groups, behind a kernel that wrote the groups' parts.
int launch_group_sum(const ScoreParams &p, cudaStream_t st);

}  // namespace aircache
