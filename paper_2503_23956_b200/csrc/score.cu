// aircache_score: importance of every visual token seen from the elite observation window
// (Section 3.3, Eq. 4-8), all layers and sequences per launch.
//
// Sequences of up to 16384 visual tokens are scored by the cluster kernel of score_cluster.cu, alpha = 0 with 32 window
// rows or more by the passes of score_dense.cu.  Here is the rest: longer sequences, windows too wide for the cluster
// kernel's shared memory (of 128 channels: 128 queries with 8 heads to a group, 110 with 16), many groups of hardly a tile,
// and caches that no tensor map describes.  Kernels on one stream:
//   elite_kernel       one CTA per (layer, sequence, KV head): the W candidate keys and the last text query
//                      are staged in shared memory; Eq. 4 logits as fp64 dot products in element order (so
//                      the Eq. 5 decision does not depend on a summation order), the elite set of each
//                      query head, the table of elite rows (head, window slot) of the KV group, and each
//                      row's softmax statistics over the text keys it may see (elite, causal).
//                      It also leaves a gathered copy of the group's first 16 elite query rows.
//   onepass_kernel     Eq. 7 and Eq. 8 with one read of the visual keys: Q_tk K_v^T on tensor cores (keys on
//   + group_sum_kernel the M axis, elite rows on N), a chunk's logits kept in shared memory between the
//                      statistics and the probabilities; see the comment at the kernel.
//   stats_kernel       the same in two passes, for sequences too long for the one-pass kernel.  Pass one:
//   + importance_kernel running (max, sum of exp2) of every elite row over one chunk of visual keys; the CTA
//                      that finishes a KV group last (ticket) merges the chunks and the text statistics
//                      into one (max, weight / normaliser) pair per row.  Pass two recomputes the same
//                      tiles, turns logits into probabilities and sums the rows of all heads per key with
//                      weight 1 / (|E_h| Hq), KV heads in ascending order by one thread per key.
//
// The mma.sync kernels read the keys straight from global memory into MMA fragments: every key byte is used
// once per CTA, so staging it in shared memory would only add a round trip.
#include <math.h>

#include <mutex>

#include "score.cuh"

namespace aircache {

namespace {

// ---------------------------------------------------------------------------------------------
// Eq. 4-5 and the elite-row table
// ---------------------------------------------------------------------------------------------
// QREG: the row's query is held in registers (64 of them at d = 128, two CTAs per SM) - worth it when a thread
// takes many rows against many text keys, i.e. when every candidate is elite (alpha = 0); otherwise the row is
// re-read from L1 per text key and six CTAs share an SM.
template <int D, bool QREG>
__global__ void __launch_bounds__(128, QREG ? 2 : 6) elite_kernel(ScoreParams p) {
    constexpr int KS = D + 8;   // padded row: 16-byte reads of consecutive rows fall into different banks
    extern __shared__ __align__(16) uint16_t s_dyn[];
    uint16_t *s_k = s_dyn;                 // [W][KS]   candidate keys
    uint16_t *s_ql = s_dyn + p.W * KS;     // [G][KS]   queries of the last text token
    __shared__ float s_logit[kMaxGroup * kMaxWindow];
    __shared__ uint64_t s_mask[kMaxGroup][2];   // candidate w is bit w % 64 of word w / 64
    __shared__ int s_first_row[kMaxGroup + 1];
    const int words = (p.W + 63) >> 6;

    const int grp = p.lb0 * p.Hkv + blockIdx.x;  // (l*B + b)*Hkv + g
    const int g = grp % p.Hkv;
    const int lb = grp / p.Hkv;
    const int l = lb / p.B, b = lb % p.B;
    const int N = p.Nv + p.Nt;
    const uint16_t *k_g = p.k + (int64_t)l * p.s_layer + (int64_t)b * p.s_batch + (int64_t)g * p.s_head;
    const uint16_t *k_cand = k_g + (int64_t)(N - p.W) * p.s_token;
    const uint16_t *q_lb = p.qw + (int64_t)lb * p.W * p.Hq * D;

    if (threadIdx.x == 0) {
        p.group_ticket[grp] = 0;   // the statistics pass counts its chunks here
        if (blockIdx.x == 0) *p.dispatch = 0;
    }
    for (int idx = threadIdx.x; idx < (p.W + p.G) * (D / 8); idx += blockDim.x) {
        const int row = idx / (D / 8), c = idx % (D / 8);
        const uint16_t *src = row < p.W ? k_cand + (int64_t)row * p.s_token
                                        : q_lb + ((int64_t)(p.W - 1) * p.Hq + g * p.G + (row - p.W)) * D;
        *reinterpret_cast<uint4 *>(s_dyn + row * KS + c * 8) = __ldg(reinterpret_cast<const uint4 *>(src) + c);
    }
    __syncthreads();

    // Eq. 4, last row only: logit of candidate w for head hl, fp64 dot product in element order.
    for (int idx = threadIdx.x; idx < p.G * p.W; idx += blockDim.x) {
        const int hl = idx / p.W, w = idx % p.W;
        const uint4 *q = reinterpret_cast<const uint4 *>(s_ql + hl * KS);
        const uint4 *kk = reinterpret_cast<const uint4 *>(s_k + w * KS);
        double acc = 0.0;
#pragma unroll 4
        for (int c = 0; c < D / 8; ++c) {
            const uint4 a = q[c], bb = kk[c];
            const uint32_t av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {bb.x, bb.y, bb.z, bb.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                // a product of two bf16 values is exact in fp64, so the fused form rounds exactly where the
                // separate multiply and add do
                acc = __fma_rn((double)bf16lo(av[e]), (double)bf16lo(bv[e]), acc);
                acc = __fma_rn((double)bf16hi(av[e]), (double)bf16hi(bv[e]), acc);
            }
        }
        s_logit[idx] = __fmul_rn((float)acc, p.scale);
    }
    __syncthreads();

    // Eq. 5: candidates within a factor alpha of the best one (compared in the log domain, fp32).
    if (threadIdx.x < p.G) {
        const int hl = threadIdx.x;
        const float *t = s_logit + hl * p.W;
        float tmax = -INFINITY;
        for (int w = 0; w < p.W; ++w) tmax = fmaxf(tmax, t[w]);
        uint64_t mask[2] = {0, 0};
        for (int w = 0; w < p.W; ++w) {
            const float diff = __fsub_rn(t[w], tmax);
            if (p.keep_all || diff >= p.ln_alpha) mask[w >> 6] |= (uint64_t)1 << (w & 63);
        }
        s_mask[hl][0] = mask[0];
        s_mask[hl][1] = mask[1];
        if (p.elite_mask)
            for (int j = 0; j < words; ++j) p.elite_mask[((int64_t)lb * p.Hq + g * p.G + hl) * words + j] = mask[j];
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int r = 0;
        for (int hl = 0; hl < p.G; ++hl) {
            s_first_row[hl] = r;
            r += __popcll(s_mask[hl][0]) + __popcll(s_mask[hl][1]);
        }
        s_first_row[p.G] = r;
        p.row_count[grp] = r;
    }
    __syncthreads();

    // Row table: elite rows of head hl are consecutive, ascending window slot.
    int32_t *info = p.row_info + (int64_t)grp * p.cap;
    float *coef = p.row_coef + (int64_t)grp * p.cap;
    float2 *text = p.row_text + (int64_t)grp * p.cap;
    for (int idx = threadIdx.x; idx < p.G * p.W; idx += blockDim.x) {
        const int hl = idx / p.W, w = idx % p.W;
        const uint64_t m_lo = s_mask[hl][0], m_hi = s_mask[hl][1];
        auto elite = [&](int j) { return (((j < 64 ? m_lo : m_hi) >> (j & 63)) & 1) != 0; };
        if (!elite(w)) continue;
        // elite candidates in front of w
        const int before = w < 64 ? __popcll(m_lo & (((uint64_t)1 << w) - 1))
                                  : __popcll(m_lo) + __popcll(m_hi & (((uint64_t)1 << (w - 64)) - 1));
        const int r = s_first_row[hl] + before;
        info[r] = (hl << 8) | w;
        coef[r] = 1.0f / ((float)(__popcll(m_lo) + __popcll(m_hi)) * (float)(p.per_head ? p.G : p.Hq));
        // Eq. 6-7, text columns: row w sees the elite text keys w' <= w.  The keys come from shared memory, the
        // query row is re-read for every key (256 bytes that stay in L1) rather than held in 64 registers.
        const uint4 *qq = reinterpret_cast<const uint4 *>(q_lb + ((int64_t)w * p.Hq + g * p.G + hl) * D);
        if (r < 16) {   // the one-pass kernel stages the first 16 rows from this gathered copy
            uint4 *qb = reinterpret_cast<uint4 *>(p.q_block + ((int64_t)grp * 16 + r) * D);
#pragma unroll 4
            for (int c = 0; c < D / 8; ++c) qb[c] = __ldg(qq + c);
        }
        uint4 qr[QREG ? D / 8 : 1];
        if (QREG) {
#pragma unroll
            for (int c = 0; c < D / 8; ++c) qr[c] = __ldg(qq + c);
        }
        float m = kNegBig, z = 0.0f;
        for (int w2 = 0; w2 <= w; ++w2) {
            if (!elite(w2)) continue;
            const uint4 *kk = reinterpret_cast<const uint4 *>(s_k + w2 * KS);
            float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll QREG ? D / 8 : 4
            for (int c = 0; c < D / 8; ++c) {
                const uint4 a = QREG ? qr[c] : __ldg(qq + c), bb = kk[c];
                a0 = fmaf(bf16lo(a.x), bf16lo(bb.x), a0); a1 = fmaf(bf16hi(a.x), bf16hi(bb.x), a1);
                a2 = fmaf(bf16lo(a.y), bf16lo(bb.y), a2); a3 = fmaf(bf16hi(a.y), bf16hi(bb.y), a3);
                a0 = fmaf(bf16lo(a.z), bf16lo(bb.z), a0); a1 = fmaf(bf16hi(a.z), bf16hi(bb.z), a1);
                a2 = fmaf(bf16lo(a.w), bf16lo(bb.w), a2); a3 = fmaf(bf16hi(a.w), bf16hi(bb.w), a3);
            }
            merge_stats(m, z, ((a0 + a1) + (a2 + a3)) * p.sl2, 1.0f);
        }
        text[r] = make_float2(m, z);
    }
}

// ---------------------------------------------------------------------------------------------
// Tensor-core tile shared by both passes.
//
// One warp computes S^T = K_tile (16 keys x d) * Q^T (d x 8*NT elite rows) with mma.m16n8k16.  The
// contraction index is permuted inside each block of 32 channels so that every thread feeds the MMA
// from one 16-byte load: thread t of a quad owns channels 8t..8t+7 of the block, both for the key rows
// (read straight from global memory) and for the query rows (shared memory).  A dot product does not
// depend on the order of its terms' indices as long as both operands use the same order.
// ---------------------------------------------------------------------------------------------
template <int D>
struct KeyFrag {
    uint4 lo[D / 32];  // key row gid
    uint4 hi[D / 32];  // key row gid + 8
};

template <int D>
__device__ __forceinline__ void load_keys(KeyFrag<D> &f, const uint16_t *row_lo, const uint16_t *row_hi, int t) {
#pragma unroll
    for (int kb = 0; kb < D / 32; ++kb) {
        f.lo[kb] = __ldg(reinterpret_cast<const uint4 *>(row_lo + kb * 32 + 8 * t));
        f.hi[kb] = __ldg(reinterpret_cast<const uint4 *>(row_hi + kb * 32 + 8 * t));
    }
}

template <int D>
__device__ __forceinline__ void tile_mma(float (&acc)[4], const KeyFrag<D> &f, const uint16_t *q_row, int t) {
    acc[0] = acc[1] = acc[2] = acc[3] = 0.f;
#pragma unroll
    for (int kb = 0; kb < D / 32; ++kb) {
        const uint4 bq = *reinterpret_cast<const uint4 *>(q_row + kb * 32 + 8 * t);
        mma_bf16_16816(acc, f.lo[kb].x, f.hi[kb].x, f.lo[kb].y, f.hi[kb].y, bq.x, bq.y);
        mma_bf16_16816(acc, f.lo[kb].z, f.hi[kb].z, f.lo[kb].w, f.hi[kb].w, bq.z, bq.w);
    }
}

// The same tile with the contraction split over two accumulators (channels 0..d/2-1 and d/2..d-1) that are
// added at the end: half the dependent-MMA chain, for callers with few row tiles to interleave.
template <int D>
__device__ __forceinline__ void tile_mma_split(float (&acc)[4], const KeyFrag<D> &f, const uint16_t *q_row, int t) {
    constexpr int H = D / 64;
    float lo[4] = {0.f, 0.f, 0.f, 0.f}, hi[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int kb = 0; kb < H; ++kb) {
        const uint4 bq = *reinterpret_cast<const uint4 *>(q_row + kb * 32 + 8 * t);
        const uint4 bq2 = *reinterpret_cast<const uint4 *>(q_row + (kb + H) * 32 + 8 * t);
        mma_bf16_16816(lo, f.lo[kb].x, f.hi[kb].x, f.lo[kb].y, f.hi[kb].y, bq.x, bq.y);
        mma_bf16_16816(hi, f.lo[kb + H].x, f.hi[kb + H].x, f.lo[kb + H].y, f.hi[kb + H].y, bq2.x, bq2.y);
        mma_bf16_16816(lo, f.lo[kb].z, f.hi[kb].z, f.lo[kb].w, f.hi[kb].w, bq.z, bq.w);
        mma_bf16_16816(hi, f.lo[kb + H].z, f.hi[kb + H].z, f.lo[kb + H].w, f.hi[kb + H].w, bq2.z, bq2.w);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[i] = lo[i] + hi[i];
}

// Copies up to 8*NT elite query rows (starting at row0) of one KV group into shared memory, zero padded.
template <int D>
__device__ __forceinline__ void stage_queries(uint16_t *s_q, const ScoreParams &p, int grp, int lb, int g,
                                              int row0, int n_rows_total, int rows_pad,
                                              const int32_t *staged_info = nullptr) {
    constexpr int QS = D + 32;
    // (head, slot) words of the rows: from the caller's copy in shared memory (rows row0.., row0 = 0) if it has one
    const int32_t *info = staged_info ? staged_info - row0 : p.row_info + (int64_t)grp * p.cap;
    const uint16_t *q_lb = p.qw + (int64_t)lb * p.W * p.Hq * D;
    for (int idx = threadIdx.x; idx < rows_pad * (D / 8); idx += blockDim.x) {
        const int r = idx / (D / 8), c = idx % (D / 8);
        uint4 v = make_uint4(0, 0, 0, 0);
        if (row0 + r < n_rows_total) {
            const int in = info[row0 + r];
            const int hl = in >> 8, w = in & 255;
            v = __ldg(reinterpret_cast<const uint4 *>(q_lb + ((int64_t)w * p.Hq + g * p.G + hl) * D) + c);
        }
        *reinterpret_cast<uint4 *>(s_q + r * QS + c * 8) = v;
    }
}

// Eq. 7, pass one.  grid = (chunks, L*B*Hkv), 128 threads.
template <int D, int NT>
__global__ void __launch_bounds__(128) stats_kernel(ScoreParams p) {
    constexpr int QS = D + 32;
    __shared__ __align__(16) uint16_t s_q[NT * 8 * QS];
    __shared__ float2 s_red[4][NT * 8];
    __shared__ int s_is_last;

    const int grp = p.lb0 * p.Hkv + blockIdx.y;
    const int g = grp % p.Hkv;
    const int lb = grp / p.Hkv;
    const int l = lb / p.B, b = lb % p.B;
    const int chunk = blockIdx.x;
    const int key0 = chunk * p.chunk_keys;
    const int key1 = min(p.Nv, key0 + p.chunk_keys);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, gid = lane >> 2, t = lane & 3;
    const uint16_t *k_g = p.k + (int64_t)l * p.s_layer + (int64_t)b * p.s_batch + (int64_t)g * p.s_head;
    const int n_rows = p.row_count[grp];
    if (n_rows <= p.rows_lo || n_rows > p.rows_hi) return;
    float2 *out = p.chunk_stats + ((int64_t)(grp - p.lb0 * p.Hkv) * p.chunks + chunk) * p.cap;

    for (int row0 = 0; row0 < n_rows; row0 += NT * 8) {
        const int nt_used = min(NT, (n_rows - row0 + 7) / 8);
        __syncthreads();
        stage_queries<D>(s_q, p, grp, lb, g, row0, n_rows, nt_used * 8);
        __syncthreads();

        float m[NT][2], z[NT][2];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) { m[nt][0] = m[nt][1] = kNegBig; z[nt][0] = z[nt][1] = 0.f; }

        // software pipeline: the next tile's keys are requested before this tile's MMAs
        auto fetch = [&](KeyFrag<D> &dst, int kt) {
            const int ka = kt + gid, kb = kt + gid + 8;
            load_keys<D>(dst, k_g + (int64_t)(ka < key1 ? ka : key1 - 1) * p.s_token,
                         k_g + (int64_t)(kb < key1 ? kb : key1 - 1) * p.s_token, t);
        };
        KeyFrag<D> f, f_next;
        if (key0 + warp * 16 < key1) fetch(f, key0 + warp * 16);
        for (int kt = key0 + warp * 16; kt < key1; kt += 64) {
            const int ka = kt + gid, kb = kt + gid + 8;
            const bool va = ka < key1, vb = kb < key1;
            if (kt + 64 < key1) fetch(f_next, kt + 64);
            // and the tile after that is asked into L2 (one 128-byte line per lane: 16 rows x D channels)
            if (kt + 128 < key1 && lane < 16 * (D * 2 / 128)) {
                const int kp = min(kt + 128 + lane / (D * 2 / 128), key1 - 1);
                prefetch_l2(k_g + (int64_t)kp * p.s_token + (lane % (D * 2 / 128)) * 64);
            }
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                if (nt < nt_used) {
                    float acc[4];
                    tile_mma<D>(acc, f, s_q + (nt * 8 + gid) * QS, t);
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const float xa = va ? acc[j] * p.sl2 : kNegBig;
                        const float xb = vb ? acc[j + 2] * p.sl2 : kNegBig;
                        const float mn = fmaxf(m[nt][j], fmaxf(xa, xb));
                        const float ea = va ? fast_exp2(xa - mn) : 0.f;
                        const float eb = vb ? fast_exp2(xb - mn) : 0.f;
                        z[nt][j] = z[nt][j] * fast_exp2(m[nt][j] - mn) + (ea + eb);
                        m[nt][j] = mn;
                    }
                }
            }
            if (kt + 64 < key1) f = f_next;
        }
        // combine the eight key lanes of a column, then the four warps, in a fixed order
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            if (nt < nt_used) {
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    float mm = m[nt][j], zz = z[nt][j];
#pragma unroll
                    for (int sh = 4; sh < 32; sh <<= 1) {
                        const float m2 = __shfl_xor_sync(0xffffffffu, mm, sh);
                        const float z2 = __shfl_xor_sync(0xffffffffu, zz, sh);
                        merge_stats(mm, zz, m2, z2);
                    }
                    if (gid == 0) s_red[warp][nt * 8 + 2 * t + j] = make_float2(mm, zz);
                }
            }
        }
        __syncthreads();
        for (int r = threadIdx.x; r < nt_used * 8; r += blockDim.x) {
            float2 a = s_red[0][r];
#pragma unroll
            for (int w2 = 1; w2 < 4; ++w2) merge_stats(a.x, a.y, s_red[w2][r].x, s_red[w2][r].y);
            if (row0 + r < n_rows) __stcg(out + row0 + r, a);
        }
    }

    // The CTA that finishes the group last merges text and chunk statistics, one warp per row: lanes take
    // chunks lane, lane + 32, ... in order, then a fixed xor tree.  (The ticket was zeroed by elite_kernel.)
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        s_is_last = atomicAdd(p.group_ticket + grp, 1u) == (unsigned)p.chunks - 1;
        if (s_is_last) __threadfence();
    }
    __syncthreads();
    if (!s_is_last) return;
    for (int r = warp; r < n_rows; r += 4) {
        float mm = kNegBig, zz = 0.f;
        if (lane == 0) {
            const float2 tx = p.row_text[(int64_t)grp * p.cap + r];
            mm = tx.x; zz = tx.y;
        }
        for (int c = lane; c < p.chunks; c += 32) {
            const float2 cs = __ldcg(p.chunk_stats + ((int64_t)(grp - p.lb0 * p.Hkv) * p.chunks + c) * p.cap + r);
            merge_stats(mm, zz, cs.x, cs.y);
        }
#pragma unroll
        for (int sh = 1; sh < 32; sh <<= 1) {
            const float m2 = __shfl_xor_sync(0xffffffffu, mm, sh);
            const float z2 = __shfl_xor_sync(0xffffffffu, zz, sh);
            merge_stats(mm, zz, m2, z2);
        }
        if (lane == 0) p.row_final[(int64_t)grp * p.cap + r] = make_float2(mm, p.row_coef[(int64_t)grp * p.cap + r] / zz);
    }
}

// Eq. 7 pass two and Eq. 8.  grid = (ceil(Nv / 128), L*B), 128 threads; each warp owns 32 keys.
template <int D, int NT>
__global__ void __launch_bounds__(128) importance_kernel(ScoreParams p) {
    constexpr int QS = D + 32;
    __shared__ __align__(16) uint16_t s_q[NT * 8 * QS];
    __shared__ float2 s_stat[NT * 8];  // (row max, weight / normaliser)
    // the row tables of all KV heads of the sequence, fetched in one go at the start: per head the first NT * 8
    // rows' (head, slot) words and statistics, so that the loop over the heads waits for the query rows only
    constexpr int kMaxKv = 8;
    __shared__ int s_rows[kMaxKv];
    __shared__ int32_t s_info_all[kMaxKv][NT * 8];
    __shared__ float2 s_stat_all[kMaxKv][NT * 8];

    const int lb = p.lb0 + blockIdx.y;
    const int l = lb / p.B, b = lb % p.B;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, gid = lane >> 2, t = lane & 3;
    const int kbase = blockIdx.x * kScoreKeyTile + warp * 32;
    float imp[2][2] = {{0.f, 0.f}, {0.f, 0.f}};  // [m-tile][key gid / gid+8]

    for (int i = threadIdx.x; i < p.Hkv * NT * 8; i += blockDim.x) {
        const int g = i / (NT * 8), r = i % (NT * 8);
        const int64_t at = (int64_t)(lb * p.Hkv + g) * p.cap + r;
        const bool inside = r < p.cap;
        s_info_all[g][r] = inside ? p.row_info[at] : 0;
        s_stat_all[g][r] = inside ? p.row_final[at] : make_float2(0.f, 0.f);
        if (r == 0) s_rows[g] = p.row_count[lb * p.Hkv + g];
    }
    __syncthreads();

    for (int g = 0; g < p.Hkv; ++g) {
        const int grp = lb * p.Hkv + g;
        const uint16_t *k_g = p.k + (int64_t)l * p.s_layer + (int64_t)b * p.s_batch + (int64_t)g * p.s_head;
        const int n_rows = s_rows[g];
        KeyFrag<D> f[2];
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) {
            const int ka = kbase + mt * 16 + gid, kb = ka + 8;
            load_keys<D>(f[mt], k_g + (int64_t)(ka < p.Nv ? ka : p.Nv - 1) * p.s_token,
                         k_g + (int64_t)(kb < p.Nv ? kb : p.Nv - 1) * p.s_token, t);
        }
        for (int row0 = 0; row0 < n_rows; row0 += NT * 8) {
            const int nt_used = min(NT, (n_rows - row0 + 7) / 8);
            __syncthreads();
            stage_queries<D>(s_q, p, grp, lb, g, row0, n_rows, nt_used * 8, row0 == 0 ? s_info_all[g] : nullptr);
            for (int r = threadIdx.x; r < nt_used * 8; r += blockDim.x)
                s_stat[r] = row0 + r >= n_rows ? make_float2(0.f, 0.f)
                            : (row0 == 0 ? s_stat_all[g][r] : p.row_final[(int64_t)grp * p.cap + row0 + r]);
            __syncthreads();
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                if (nt < nt_used) {
                    const float2 s0 = s_stat[nt * 8 + 2 * t], s1 = s_stat[nt * 8 + 2 * t + 1];
#pragma unroll
                    for (int mt = 0; mt < 2; ++mt) {
                        float acc[4];
                        tile_mma<D>(acc, f[mt], s_q + (nt * 8 + gid) * QS, t);
                        imp[mt][0] += fast_exp2(acc[0] * p.sl2 - s0.x) * s0.y + fast_exp2(acc[1] * p.sl2 - s1.x) * s1.y;
                        imp[mt][1] += fast_exp2(acc[2] * p.sl2 - s0.x) * s0.y + fast_exp2(acc[3] * p.sl2 - s1.x) * s1.y;
                    }
                }
            }
        }
        if (p.per_head || g == p.Hkv - 1) {
            // the key's score is complete: of this KV group alone, or summed over all of them
            float *out = p.scores + (p.per_head ? (int64_t)grp : (int64_t)lb) * p.Nv;
#pragma unroll
            for (int mt = 0; mt < 2; ++mt) {
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    float v = imp[mt][j];
                    v += __shfl_xor_sync(0xffffffffu, v, 1);
                    v += __shfl_xor_sync(0xffffffffu, v, 2);
                    const int key = kbase + mt * 16 + gid + 8 * j;
                    if (t == 0 && key < p.Nv) out[key] = v;
                    imp[mt][j] = 0.f;
                }
            }
        }
    }
}

// ---------------------------------------------------------------------------------------------
// Eq. 7 and Eq. 8 in ONE pass over the keys.
//
// The two kernels above read the keys from HBM twice when the cache is larger than L2.  Here a block owns a
// chunk of one KV group's keys and keeps the chunk's logits (fp32 MMA accumulators, up to 16 rows) in shared
// memory: pass one gives the chunk's (max, sum) per row; when all chunks of the group have published theirs,
// every block of the group merges them (same fixed order in every block: equal bits), turns its stored logits
// into probabilities and sums them per key - no second read of the keys, no second contraction.  A chunk is
// 1024 keys for a group of up to 8 elite rows and 512 keys beyond, so the stored logits fill the same 32 KB
// (five blocks per SM); the per-key sums of pass two go into slots of that buffer the warp has already read.
// Rows beyond 16 (wide windows, small alpha) are recomputed from the keys, which are still in L1/L2.
//
// Waiting inside a grid is safe here because a block draws its number from a counter when it STARTS: all
// lower numbers belong to blocks that are running or done.  Numbers are group-major, a group spans
// op_chunks numbers, and the host only takes this path when op_chunks is at most half of the blocks the GPU
// holds at once - so the blocks a waiting block depends on are always resident or next in line, and blocks
// of lower groups, which wait for nothing that has not started, always finish.  The wait is bounded all the same.
//
// The sum over the KV groups of a (layer, sequence) is a second, small kernel (fixed order g = 0, 1, ...).
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t ld_acquire_u32(const uint32_t *ptr) {
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(ptr) : "memory");
    return v;
}

__device__ __forceinline__ int onepass_tiles(int n_rows, int cap) {   // 16-key tiles per warp
    return min(n_rows <= 8 ? 16 : 8, cap);
}

template <int D>
__global__ void __launch_bounds__(128, 5) onepass_kernel(ScoreParams p) {
    constexpr int NT = 2, QS = D + 32;
    extern __shared__ __align__(16) uint16_t s_dyn[];
    float4 *s_S = reinterpret_cast<float4 *>(s_dyn);        // [tile of the warp][row tile][thread]: 2048 x 16 B
    __shared__ __align__(16) uint16_t s_q[NT * 8 * QS];
    __shared__ float2 s_red[4][NT * 8];
    __shared__ float2 s_stat[NT * 8];
    __shared__ int s_flag;

    if (threadIdx.x == 0) s_flag = (int)atomicAdd(p.dispatch, 1u);
    __syncthreads();
    const int vid = s_flag;
    __syncthreads();

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gid = lane >> 2, t = lane & 3;
    const int gi = vid / p.op_chunks, c = vid % p.op_chunks;
    if (gi >= p.n_lb * p.Hkv) return;
    const int grp = p.lb0 * p.Hkv + gi;
    const int g = grp % p.Hkv, lb = grp / p.Hkv, l = lb / p.B, b = lb % p.B;
    const int n_rows = p.row_count[grp];
    const int tpw = onepass_tiles(n_rows, p.op_tile_cap);
    const int KB = 64 * tpw;
    const int chunks_g = (p.Nv + KB - 1) / KB;
    if (c >= chunks_g) return;
    const int nt0 = min(NT, (n_rows + 7) >> 3);
    const uint16_t *k_g = p.k + (int64_t)l * p.s_layer + (int64_t)b * p.s_batch + (int64_t)g * p.s_head;
    const int key0 = c * KB, key1 = min(p.Nv, key0 + KB);
    const int wk0 = key0 + warp * tpw * 16, wk1 = min(key1, wk0 + tpw * 16);
    // the warp's first two tiles are asked into L2 now (HBM latency runs beside the query staging), every later
    // tile two tiles before its turn.  (Asking for the whole chunk at once measured 15 % slower: the burst
    // queues in front of the loads that are waited for.)
    constexpr int kAhead = 2 * 16;
    for (int i = lane; i < min(wk1 - wk0, kAhead) * (D * 2 / 128); i += 32)
        prefetch_l2(k_g + (int64_t)(wk0 + i / (D * 2 / 128)) * p.s_token + (i % (D * 2 / 128)) * 64);

    auto fetch = [&](KeyFrag<D> &dst, int kt) {
        const int ka = kt + gid, kb = kt + gid + 8;
        load_keys<D>(dst, k_g + (int64_t)(ka < wk1 ? ka : wk1 - 1) * p.s_token,
                     k_g + (int64_t)(kb < wk1 ? kb : wk1 - 1) * p.s_token, t);
    };
    // (max, weight / normaliser) of rows row0 .. row0 + n - 1 into s_stat: one thread per row merges the text
    // statistics and then the chunks' statistics in chunk order (all loads of a row are independent, one round
    // trip), the same order in every block
    auto merge_rows = [&](int row0, int n) {
        if (tid < n) {
            const int row = row0 + tid;
            float2 fin = make_float2(0.f, 0.f);
            if (row < n_rows) {
                const float2 *cs = p.chunk_stats + (int64_t)gi * p.op_chunks * p.cap + row;
                const float2 tx = p.row_text[(int64_t)grp * p.cap + row];
                const float coef = p.row_coef[(int64_t)grp * p.cap + row];
                float mm = tx.x, zz = tx.y;
                int cc = 0;
                for (; cc + 4 <= chunks_g; cc += 4) {
                    const float2 c0 = __ldcg(cs + (int64_t)cc * p.cap), c1 = __ldcg(cs + (int64_t)(cc + 1) * p.cap);
                    const float2 c2 = __ldcg(cs + (int64_t)(cc + 2) * p.cap), c3 = __ldcg(cs + (int64_t)(cc + 3) * p.cap);
                    merge_stats(mm, zz, c0.x, c0.y); merge_stats(mm, zz, c1.x, c1.y);
                    merge_stats(mm, zz, c2.x, c2.y); merge_stats(mm, zz, c3.x, c3.y);
                }
                for (; cc < chunks_g; ++cc) {
                    const float2 c0 = __ldcg(cs + (int64_t)cc * p.cap);
                    merge_stats(mm, zz, c0.x, c0.y);
                }
                fin = make_float2(mm, coef / zz);
            }
            s_stat[tid] = fin;
        }
    };

    // ---- pass one: statistics of the chunk, logits of the first 16 rows kept ----
    float2 *out = p.chunk_stats + ((int64_t)gi * p.op_chunks + c) * p.cap;
    for (int row0 = 0; row0 < n_rows; row0 += NT * 8) {
        const int nt_used = min(NT, (n_rows - row0 + 7) / 8);
        KeyFrag<D> f, f_next;
        if (wk0 < wk1) fetch(f, wk0);
        __syncthreads();
        if (row0 == 0) {
            const uint4 *qb = reinterpret_cast<const uint4 *>(p.q_block + (int64_t)grp * 16 * D);
            for (int idx = tid; idx < nt_used * 8 * (D / 8); idx += blockDim.x) {
                const int r = idx / (D / 8), cc = idx % (D / 8);
                *reinterpret_cast<uint4 *>(s_q + r * QS + cc * 8) = r < n_rows ? __ldg(qb + idx) : make_uint4(0, 0, 0, 0);
            }
        } else {
            stage_queries<D>(s_q, p, grp, lb, g, row0, n_rows, nt_used * 8);
        }
        __syncthreads();
        float m[NT][2], z[NT][2];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) { m[nt][0] = m[nt][1] = kNegBig; z[nt][0] = z[nt][1] = 0.f; }
        int slot = tid;   // (tile * nt_used + nt) * 128 + tid
        for (int kt = wk0; kt < wk1; kt += 16) {
            const int ka = kt + gid, kb = kt + gid + 8;
            const bool va = ka < wk1, vb = kb < wk1;
            if (kt + 16 < wk1) fetch(f_next, kt + 16);
            if (kt + kAhead < wk1 && lane < 16 * (D * 2 / 128)) {   // one 128-byte line per lane: 16 rows x d channels
                const int kp = min(kt + kAhead + lane / (D * 2 / 128), wk1 - 1);
                prefetch_l2(k_g + (int64_t)kp * p.s_token + (lane % (D * 2 / 128)) * 64);
            }
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                if (nt < nt_used) {
                    float acc[4];
                    tile_mma_split<D>(acc, f, s_q + (nt * 8 + gid) * QS, t);
                    if (row0 == 0) { s_S[slot] = make_float4(acc[0], acc[1], acc[2], acc[3]); slot += 128; }
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const float xa = va ? acc[j] * p.sl2 : kNegBig;
                        const float xb = vb ? acc[j + 2] * p.sl2 : kNegBig;
                        const float mn = fmaxf(m[nt][j], fmaxf(xa, xb));
                        const float ea = va ? fast_exp2(xa - mn) : 0.f;
                        const float eb = vb ? fast_exp2(xb - mn) : 0.f;
                        z[nt][j] = z[nt][j] * fast_exp2(m[nt][j] - mn) + (ea + eb);
                        m[nt][j] = mn;
                    }
                }
            }
            if (kt + 16 < wk1) f = f_next;
        }
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            if (nt < nt_used) {
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    float mm = m[nt][j], zz = z[nt][j];
#pragma unroll
                    for (int sh = 4; sh < 32; sh <<= 1) {
                        const float m2 = __shfl_xor_sync(0xffffffffu, mm, sh);
                        const float z2 = __shfl_xor_sync(0xffffffffu, zz, sh);
                        merge_stats(mm, zz, m2, z2);
                    }
                    if (gid == 0) s_red[warp][nt * 8 + 2 * t + j] = make_float2(mm, zz);
                }
            }
        }
        __syncthreads();
        for (int r = tid; r < nt_used * 8; r += blockDim.x) {
            float2 a = s_red[0][r];
#pragma unroll
            for (int w2 = 1; w2 < 4; ++w2) merge_stats(a.x, a.y, s_red[w2][r].x, s_red[w2][r].y);
            if (row0 + r < n_rows) __stcg(out + row0 + r, a);
        }
    }

    // ---- publish the chunk, wait until every chunk of the group is published ----
    __syncthreads();
    if (tid == 0) {
        __threadfence();   // the block's statistics (ordered before this by the barrier) before the ticket
        int ok = atomicAdd(p.group_ticket + grp, 1u) + 1u >= (unsigned)chunks_g;
        for (uint32_t i = 0; !ok && i < kSpinLimit; ++i) {
            __nanosleep(i < 64 ? 32 : 1000);
            ok = ld_acquire_u32(p.group_ticket + grp) >= (unsigned)chunks_g;
        }
        if (!ok) atomicExch(p.status, 8u);
        __threadfence();
        s_flag = ok;
    }
    __syncthreads();
    if (!s_flag) return;

    // ---- pass two: probabilities from the kept logits, summed over the rows of the group ----
    merge_rows(0, nt0 * 8);
    __syncthreads();
    {
        int slot = tid;
        float *imp_w = reinterpret_cast<float *>(s_S + warp * 32);   // + tile * nt0 * 512 floats: the warp's own slots of the tile
#pragma unroll 4
        for (int kt = wk0; kt < wk1; kt += 16, imp_w += nt0 * 512) {
            float a0 = 0.f, a1 = 0.f;
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                if (nt < nt0) {
                    const float4 v = s_S[slot]; slot += 128;
                    const float2 s0 = s_stat[nt * 8 + 2 * t], s1 = s_stat[nt * 8 + 2 * t + 1];
                    a0 += fast_exp2(v.x * p.sl2 - s0.x) * s0.y + fast_exp2(v.y * p.sl2 - s1.x) * s1.y;
                    a1 += fast_exp2(v.z * p.sl2 - s0.x) * s0.y + fast_exp2(v.w * p.sl2 - s1.x) * s1.y;
                }
            }
            a0 += __shfl_xor_sync(0xffffffffu, a0, 1); a0 += __shfl_xor_sync(0xffffffffu, a0, 2);
            a1 += __shfl_xor_sync(0xffffffffu, a1, 1); a1 += __shfl_xor_sync(0xffffffffu, a1, 2);
            if (t == 0) { imp_w[gid] = a0; imp_w[gid + 8] = a1; }
        }
    }
    // rows beyond 16: logits recomputed from the keys
    for (int row0 = NT * 8; row0 < n_rows; row0 += NT * 8) {
        const int nt_used = min(NT, (n_rows - row0 + 7) / 8);
        __syncthreads();
        stage_queries<D>(s_q, p, grp, lb, g, row0, n_rows, nt_used * 8);
        merge_rows(row0, nt_used * 8);
        __syncthreads();
        KeyFrag<D> f;
        float *imp_w = reinterpret_cast<float *>(s_S + warp * 32);
        for (int kt = wk0; kt < wk1; kt += 16, imp_w += nt0 * 512) {
            fetch(f, kt);
            float a0 = 0.f, a1 = 0.f;
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                if (nt < nt_used) {
                    float acc[4];
                    tile_mma_split<D>(acc, f, s_q + (nt * 8 + gid) * QS, t);
                    const float2 s0 = s_stat[nt * 8 + 2 * t], s1 = s_stat[nt * 8 + 2 * t + 1];
                    a0 += fast_exp2(acc[0] * p.sl2 - s0.x) * s0.y + fast_exp2(acc[1] * p.sl2 - s1.x) * s1.y;
                    a1 += fast_exp2(acc[2] * p.sl2 - s0.x) * s0.y + fast_exp2(acc[3] * p.sl2 - s1.x) * s1.y;
                }
            }
            a0 += __shfl_xor_sync(0xffffffffu, a0, 1); a0 += __shfl_xor_sync(0xffffffffu, a0, 2);
            a1 += __shfl_xor_sync(0xffffffffu, a1, 1); a1 += __shfl_xor_sync(0xffffffffu, a1, 2);
            if (t == 0) { imp_w[gid] += a0; imp_w[gid + 8] += a1; }
        }
    }
    __syncthreads();

    // ---- Eq. 8: the group's own score, or its part of the sum over the KV groups ----
    const int nkeys = key1 - key0;
    float *dst = (p.per_head ? p.scores : p.imp_part) + (int64_t)grp * p.Nv + key0;
    for (int i = tid; i < nkeys; i += blockDim.x) {
        const int w = i / (tpw * 16), rem = i % (tpw * 16);
        dst[i] = reinterpret_cast<const float *>(s_S + w * 32)[(rem >> 4) * nt0 * 512 + (rem & 15)];
    }
}

// Eq. 8, the mean over all query heads: the KV groups' parts added in the order g = 0, 1, ...  Bound by latency (a launch, a
// load, a store): four loads in flight instead of one behind the other took a one-layer scoring call from 14.6 to 14.3 us.
__global__ void __launch_bounds__(256) group_sum_kernel(ScoreParams p) {
    const int lb = p.lb0 + blockIdx.y;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    // launched ahead of its predecessor's end: nothing is read before the wait
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (i >= p.Nv) return;
    const float *src = p.imp_part + (int64_t)lb * p.Hkv * p.Nv + i;
    float v = 0.f;
#pragma unroll 4
    for (int g = 0; g < p.Hkv; ++g) v += __ldcg(src + (int64_t)g * p.Nv);
    p.scores[(int64_t)lb * p.Nv + i] = v;
}

// Blocks of the one-pass kernel the device holds at once (0 if the kernel cannot run); asked once per device,
// under a lock.
template <int D>
int onepass_resident_blocks() {
    static std::mutex lock;
    static int cached[64];
    static bool have[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    std::lock_guard<std::mutex> guard(lock);
    if (!have[dev]) {
        int per_sm = 0, sms = 0;
        if (cudaFuncSetAttribute(onepass_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, 32768) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, onepass_kernel<D>, 128, 32768) != cudaSuccess ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
            return 0;
        cached[dev] = per_sm * sms;
        have[dev] = true;
    }
    return cached[dev];
}

template <int D>
int launch_onepass(const ScoreParams &p, cudaStream_t st) {
    const int64_t blocks = (int64_t)p.n_lb * p.Hkv * p.op_chunks;
    onepass_kernel<D><<<(unsigned)blocks, 128, 32768, st>>>(p);
    AIRCACHE_LAUNCH_CHECK();
    return p.per_head ? AIRCACHE_OK : launch_group_sum(p, st);
}

template <int D, int NT>
int launch_stats(ScoreParams p, int rows_lo, int rows_hi, cudaStream_t st) {
    p.rows_lo = rows_lo; p.rows_hi = rows_hi;
    stats_kernel<D, NT><<<dim3(p.chunks, (unsigned)((int64_t)p.n_lb * p.Hkv)), 128, 0, st>>>(p);
    AIRCACHE_LAUNCH_CHECK();
    return AIRCACHE_OK;
}

template <int D, int NT>
int launch_importance(const ScoreParams &p, cudaStream_t st) {
    importance_kernel<D, NT><<<dim3((p.Nv + kScoreKeyTile - 1) / kScoreKeyTile, (unsigned)p.n_lb), 128, 0,
                               st>>>(p);
    AIRCACHE_LAUNCH_CHECK();
    return AIRCACHE_OK;
}

// The number of elite rows of a KV group is known on the device only and is small for the paper's
// threshold (a few rows per head), far below the G*W the shape allows.  The statistics pass keeps per-row
// state in registers, so groups with at most 32 rows run in a 4-tile instantiation (more CTAs per SM); if
// the shape allows more rows, a second launch with the wide instantiation picks up the groups beyond 32
// rows and exits at once elsewhere.  The importance pass keeps no per-row state and runs once.
template <int D>
int launch_passes_d(const ScoreParams &p, cudaStream_t st) {
    const int nt_max = (p.G * p.W + 7) / 8;
    const int big = 1 << 30;
    int rc;
    if (nt_max <= 2) {
        if ((rc = launch_stats<D, 2>(p, 0, big, st))) return rc;
        return launch_importance<D, 2>(p, st);
    }
    if ((rc = launch_stats<D, 4>(p, 0, nt_max <= 4 ? big : 32, st))) return rc;
    if (nt_max > 4) {
        rc = nt_max <= 8 ? launch_stats<D, 8>(p, 32, big, st) : launch_stats<D, 16>(p, 32, big, st);
        if (rc) return rc;
    }
    return nt_max <= 4 ? launch_importance<D, 4>(p, st) : launch_importance<D, 8>(p, st);
}

}  // namespace

int launch_group_sum(const ScoreParams &p, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((p.Nv + 255) / 256, (unsigned)p.n_lb);
    cfg.blockDim = dim3(256);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    AIRCACHE_CUDA_TRY(cudaLaunchKernelEx(&cfg, group_sum_kernel, p));
    return AIRCACHE_OK;
}

// Many KV groups of hardly a tile of keys: a cluster then spends its time on a group's elite rows, one unit of 16 after the
// other, with two blocks to an SM; elite_kernel and the one-pass kernel hold six and five.  What there is of it grows with
// the elite rows, of which a low alpha leaves many, and large groups fill the cluster kernel's units better.  Measured
// (older kernels, cluster kernel, the latter when a one-layer call took it 17 us, 13.7 since; us a call):
//   14336 groups of 4 heads, 64 channels, 16 window queries: alpha 0.9, 3 tokens 210, 270; 32 tokens 242, 277; 96 tokens 306,
//   278.  alpha 0.1, 3 tokens 508, 944; 64 tokens 700, 939; 128 tokens 954, 961.  alpha 0.3, 16 tokens 346, 596.
//   3584 groups of 2 heads: alpha 0.9, 32 tokens 64, 79; 128 tokens 92, 90 (alpha 0.5).  14336 groups of 1 head of 128 channels:
//   alpha 0.9, 3 tokens 230, 292; 64 tokens 303, 287.  7168 groups of 7 heads: alpha 0.9, 64 tokens 219, 171.
//   224 groups of 4 heads, alpha 0.1, 3 tokens: 36, 25.
static bool hardly_a_tile(const ScoreParams &p, float alpha, int sms) {
    if ((int64_t)p.n_lb * p.Hkv < 6 * (int64_t)sms || p.keep_all) return false;
    if (alpha < 0.75f) return (int64_t)p.Nv * p.Nv * p.G <= 136 * 136;
    return p.G <= 4 && p.W <= 64 && p.Nv <= 32;
}

int launch_score(const aircache_shape_t *s, const aircache_full_t *f, const void *q_window, float alpha,
                 int layer_begin, int layer_count, float *scores, uint64_t *elite_mask, void *ws, cudaStream_t st) {
    const WsLayout w = ws_layout(s);
    ScoreParams p = {};
    p.k = (const uint16_t *)f->k;
    p.s_layer = f->stride_layer; p.s_batch = f->stride_batch; p.s_head = f->stride_head; p.s_token = f->stride_token;
    p.qw = (const uint16_t *)q_window;
    p.scores = scores;
    p.elite_mask = elite_mask;
    p.row_count = ws_ptr<int32_t>(ws, w.row_count);
    p.row_info = ws_ptr<int32_t>(ws, w.row_info);
    p.row_coef = ws_ptr<float>(ws, w.row_coef);
    p.row_text = ws_ptr<float2>(ws, w.row_text);
    p.chunk_stats = ws_ptr<float2>(ws, w.chunk_stats);
    p.row_final = ws_ptr<float2>(ws, w.row_final);
    p.group_ticket = ws_ptr<uint32_t>(ws, w.group_ticket);
    p.dispatch = ws_ptr<uint32_t>(ws, w.dispatch);
    p.imp_part = ws_ptr<float>(ws, w.imp_part);
    p.q_block = ws_ptr<uint16_t>(ws, w.q_block);
    p.L = s->n_layers; p.B = s->batch; p.Hq = s->n_q_heads; p.Hkv = s->n_kv_heads;
    p.G = s->n_q_heads / s->n_kv_heads; p.d = s->head_dim; p.Nv = s->n_visual; p.Nt = s->n_text; p.W = s->window;
    p.per_head = s->per_kv_head;
    p.lb0 = layer_begin * s->batch;
    p.n_lb = layer_count * s->batch;
    p.cap = score_row_cap(s);
    p.scale = s->scale;
    p.sl2 = s->scale * kLog2e;
    p.keep_all = alpha <= 0.0f;
    p.ln_alpha = p.keep_all ? 0.0f : (float)log((double)alpha);
    p.rows_lo = 0; p.rows_hi = 1 << 30;
    p.pos_token = p.pos_head = p.pos_batch = p.pos_layer = 0;
    p.status = ws_ptr<uint32_t>(ws, w.status);

    // alpha = 0 with at least a cluster's two query blocks keeps the tensor cores and the exponentials busy by itself
    int taken = 0, dev = 0, sms = 0;
    int rc = current_device(&dev, &sms);
    if (rc) return rc;
    if (p.keep_all && p.G * p.W >= 32) rc = launch_score_dense(p, s, f, st, &taken);
    else if (!hardly_a_tile(p, alpha, sms)) rc = launch_score_cluster(p, s, f, st, &taken);
    if (rc || taken) return rc;

    // What the remaining kernels need.  A call over few KV groups (a layer at a time, a single sequence) would leave SMs
    // idle with 512- and 1024-key blocks of the one-pass kernel: while the blocks would fill less than half of the GPU,
    // they take half the tiles per warp, down to 256 keys per block (four sequences of 6272 tokens, a layer at a time, when
    // this kernel still took them: 41 -> 33 us per layer).
    const int resident = s->head_dim == 64 ? onepass_resident_blocks<64>() : onepass_resident_blocks<128>();
    const int64_t groups = (int64_t)p.n_lb * p.Hkv;
    auto numbers_per_group = [&](int cap) { const int k = 64 * (cap < 8 ? cap : 8); return (s->n_visual + k - 1) / k; };
    p.op_tile_cap = 16;
    while (p.op_tile_cap > 4 &&
           groups * ((s->n_visual + 64 * p.op_tile_cap - 1) / (64 * p.op_tile_cap)) * 2 < (int64_t)resident &&
           (int64_t)numbers_per_group(p.op_tile_cap / 2) * 2 <= resident)
        p.op_tile_cap >>= 1;
    p.op_chunks = numbers_per_group(p.op_tile_cap);
    p.chunks = score_chunks(s->n_visual, groups);
    p.chunk_keys = (int)align_up((s->n_visual + p.chunks - 1) / p.chunks, 16);
    const size_t elite_smem = (size_t)(p.W + p.G) * (p.d + 8) * 2;
    if (p.keep_all) {
        if (s->head_dim == 64) elite_kernel<64, true><<<(unsigned)groups, 128, elite_smem, st>>>(p);
        else elite_kernel<128, true><<<(unsigned)groups, 128, elite_smem, st>>>(p);
    } else {
        if (s->head_dim == 64) elite_kernel<64, false><<<(unsigned)groups, 128, elite_smem, st>>>(p);
        else elite_kernel<128, false><<<(unsigned)groups, 128, elite_smem, st>>>(p);
    }
    AIRCACHE_LAUNCH_CHECK();
    // one pass over the keys, if a group's blocks are sure to be resident together
    if ((int64_t)p.op_chunks * 2 <= resident && (int64_t)p.n_lb * p.Hkv * p.op_chunks < ((int64_t)1 << 31))
        return s->head_dim == 64 ? launch_onepass<64>(p, st) : launch_onepass<128>(p, st);
    return s->head_dim == 64 ? launch_passes_d<64>(p, st) : launch_passes_d<128>(p, st);
}

}  // namespace aircache
