// Scoring by thread-block clusters: Eq. 4-8 in one launch with one read of the visual keys, for sequences that a
// cluster of up to eight blocks holds (16384 visual tokens).
//
// A cluster of C blocks works on one KV group (layer, sequence, KV head) at a time, each block on a stretch of the
// visual keys in tiles of 128.  Warp roles inside a block (two blocks share an SM):
//   producer   one thread: key tiles by TMA (128-byte swizzle) through a ring of shared-memory stages
//   tensor     one thread: tcgen05.mma M = 128 keys, N = 16 elite rows, D in a 16-column slot of tensor memory per
//              tile, so the logits of all of a block's tiles stay on chip
//   elite      four warps: Eq. 4-5 of the group (fp64 logits in element order, masks), the table of elite rows,
//              16 query rows at a time into the swizzled operand layout, each row's softmax statistics over the
//              elite text keys it sees.  Every block of the cluster does this for itself, one group ahead.
//   epilogue   four warps, a thread owns a key (tensor-memory lane) of every tile and the 16 rows' values in
//              registers:  e = exp2(logit - reference) as a tile arrives, written back over the logit, and the
//              running sum per row; at the end of the stretch the sums meet (warp, block, then cluster through
//              distributed shared memory), and p = e * F with F = weight / normaliser * exp2(reference - max) per
//              thread and row: one exponential per logit, no reduction across lanes for Eq. 8.
// The reference is the thread's first logit of the row.  It need not be the maximum, only near enough for fp32's
// range: a logit more than 2^24 above it moves it (the stored values of the earlier tiles are rescaled; rare).
//
// More than 16 elite rows: the keys are read again (from L2) for every further 16.  The KV groups of a (layer,
// sequence) either follow one another in the same cluster, each adding to the scores, or - when there are too few
// sequences to fill the GPU that way - go to different clusters and group_sum_kernel adds them, g = 0, 1, ...
//
// What it replaced (elite kernel, one-pass kernel on mma.sync with a wait between blocks, sum kernel) streamed keys
// during half of a block's life and took three launches.  Measured, 28 layers of 28 query and 4 KV heads of 128
// channels: 64 sequences of 2916 tokens 1180 -> 952 us (5.6 TB/s of keys); one of 7290 tokens 75 -> 56 us; four of
// 6272, a call per layer, 33 -> 20 us a call.
//
// With up to eight tiles per block the tensor memory holds two units of work and the tensor core runs ahead of the
// epilogue; with up to sixteen the other block of the SM fills the gap.  All waits are bounded.
#include <math.h>

#include <mutex>

#include "score.cuh"

namespace aircache {

namespace {

constexpr int kRows = 16;             // elite rows per unit of work (the MMA's N)
constexpr int kSlots = 16;            // tensor-memory slots of kRows columns
constexpr int kMaxCluster = 8;
constexpr int kMaxStages = 6;
// Twelve warps: control (producer, tensor core, two idle), elite, epilogue.  (Ten would do, but blocks are given
// registers in fours of warps, and at 96 registers ten warps left room for one block per SM: 1.5 times slower.)
constexpr int kClusterThreads = 384;
constexpr int kEliteThreads = 128, kEpiThreads = 128;
constexpr int kEliteWarp0 = 4, kEpiWarp0 = 8;
constexpr int kSmemPerBlock = (228 * 1024) / 2 - 1024;   // two blocks per SM, 1 KB each is the system's
constexpr float kRescale = 24.f;

struct ClusterSmem {   // small state behind the ring and the query block
    uint64_t full[kMaxStages], empty[kMaxStages];
    uint64_t q_full[2], meta_empty[2], q_free;
    uint64_t acc_full[kSlots], acc_empty[2], exchange[2];
    float2 stats[2][kMaxCluster][kRows];   // (max, sum) of every block of the cluster
    float2 warp_stats[2][4][kRows];
    float2 fin[4][kRows];                  // per epilogue warp: (max, weight / normaliser)
    float2 text[2][kRows];
    float coef[2][kRows];
    int2 meta[2];                          // rows of the unit, last unit of its group
    uint32_t mask[kMaxGroup][4];           // elite candidates, bit w % 32 of word w / 32
    uint32_t tmem;
    int abort;
};

template <int D>
struct ClusterCfg {
    static constexpr int TILE_BYTES = D / 64 * kKeySubBytes;
    static constexpr int Q_SUB = kRows * 128;
    static constexpr int Q_BYTES = D / 64 * Q_SUB;
    static constexpr int KS = D + 8;   // padded row of the staged candidate keys and last queries
    static int tail_bytes(int W, int G) {
        return (int)sizeof(ClusterSmem) + (W + G) * KS * 2 + (G * W * 4 + 15) / 16 * 16;
    }
    static int stages(int W, int G) {
        const int fit = (kSmemPerBlock - Q_BYTES - tail_bytes(W, G)) / TILE_BYTES;
        return fit > kMaxStages ? kMaxStages : fit;
    }
    static int smem_bytes(int W, int G) { return stages(W, G) * TILE_BYTES + Q_BYTES + tail_bytes(W, G); }
};

struct ClusterPlan {
    // bufs units of slots_per_unit tiles fit the tensor memory; part: sums go to the per-group buffer
    int items, groups_per_item, cluster, slots_per_unit, bufs, stages, part;
};

__device__ __forceinline__ void named_bar(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }
// the same, and whether `ok` holds in all of the threads: the warps of a role leave their loop together or not at all
__device__ __forceinline__ bool named_bar_and(int id, int n, bool ok) {
    int r;
    asm volatile(
        "{\n.reg .pred p, q;\nsetp.ne.s32 p, %1, 0;\nbar.red.and.pred q, %2, %3, p;\nselp.s32 %0, 1, 0, q;\n}\n"
        : "=r"(r) : "r"((int)ok), "r"(id), "r"(n) : "memory");
    return r != 0;
}

template <int D>
__global__ void __launch_bounds__(kClusterThreads, 2)
score_cluster_kernel(const __grid_constant__ CUtensorMap tm_k, ScoreParams p, ClusterPlan plan) {
    using C = ClusterCfg<D>;
    extern __shared__ __align__(1024) uint8_t smem[];
    const int S = plan.stages;
    uint8_t *s_ring = smem;
    uint8_t *s_q = smem + S * C::TILE_BYTES;
    ClusterSmem &sm = *reinterpret_cast<ClusterSmem *>(s_q + C::Q_BYTES);
    uint16_t *s_k = reinterpret_cast<uint16_t *>(&sm + 1);   // [W][KS] candidate keys, then [G][KS] last queries
    float *s_logit = reinterpret_cast<float *>(s_k + (p.W + p.G) * C::KS);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t rank = cluster_rank();
    const int n_clusters = gridDim.x / plan.cluster, cid = blockIdx.x / plan.cluster;

    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (tid == 0) {
        for (int i = 0; i < S; ++i) { mbar_init(smem_u32(&sm.full[i]), 1); mbar_init(smem_u32(&sm.empty[i]), 1); }
        for (int i = 0; i < 2; ++i) {
            mbar_init(smem_u32(&sm.q_full[i]), 1);
            mbar_init(smem_u32(&sm.meta_empty[i]), 5);   // producer and four epilogue warps
            mbar_init(smem_u32(&sm.acc_empty[i]), 4);
            mbar_init(smem_u32(&sm.exchange[i]), 1);
        }
        mbar_init(smem_u32(&sm.q_free), 1);
        for (int i = 0; i < kSlots; ++i) mbar_init(smem_u32(&sm.acc_full[i]), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        sm.abort = 0;
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tm_k)) : "memory");
    }
    if (warp == 1) tmem_alloc(smem_u32(&sm.tmem), kSlots * kRows);
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();   // the barriers of every block are ready
    tc_fence_after();
    const uint32_t tmem = sm.tmem;
    volatile int *abort_flag = &sm.abort;

    // this block's tiles of every group
    const int all_tiles = (p.Nv + 127) >> 7;
    const int t0 = all_tiles * (int)rank / plan.cluster, t1 = all_tiles * ((int)rank + 1) / plan.cluster;
    const int T = t1 - t0, key0 = t0 * 128;
    const int first_grp = p.lb0 * p.Hkv;

    asm volatile("griddepcontrol.wait;" ::: "memory");   // nothing above read global memory

    // Units of work, in the same order in every role: item (the cluster's share), KV group of the item, 16 rows.
    if (warp == 0) {
        // ================================ producer ================================
        if (lane == 0) {
            bool ok = true;
            uint32_t u = 0, it = 0;
            for (int item = cid; ok && item < plan.items; item += n_clusters) {
                for (int gi = 0; ok && gi < plan.groups_per_item; ++gi) {
                    const int grp = first_grp + item * plan.groups_per_item + gi;
                    const int g = grp % p.Hkv, lb = grp / p.Hkv, l = lb / p.B, b = lb - l * p.B;
                    for (bool last = false; ok && !last; ++u) {
                        for (int t = 0; t < T; ++t, ++it) {
                            const uint32_t st = it % S;
                            ok = mbar_wait(smem_u32(&sm.empty[st]), ((it / S) & 1) ^ 1, abort_flag, p.status, 20);
                            if (!ok) break;
                            load_key_tile<D>(smem_u32(s_ring + st * C::TILE_BYTES), &tm_k, p, key0 + t * 128, g, b, l,
                                             smem_u32(&sm.full[st]));
                        }
                        ok = ok && mbar_wait(smem_u32(&sm.q_full[u & 1]), (u >> 1) & 1, abort_flag, p.status, 21);
                        if (!ok) break;
                        last = sm.meta[u & 1].y != 0;
                        mbar_arrive(smem_u32(&sm.meta_empty[u & 1]));
                    }
                }
            }
            if (!ok) {   // the loads in flight end before the block does
                for (uint32_t i = it > (uint32_t)S ? it - S : 0; i < it; ++i)
                    for (uint32_t n = 0; n < kSpinLimit && !mbar_test(smem_u32(&sm.full[i % S]), (i / S) & 1); ++n) __nanosleep(40);
            }
        }
    } else if (warp == 1) {
        // ================================ tensor core ================================
        if (lane == 0) {
            bool ok = true;
            uint32_t u = 0, it = 0;
            const uint32_t idesc = umma_idesc_bf16(128, kRows);
            for (int item = cid; ok && item < plan.items; item += n_clusters) {
                for (int gi = 0; ok && gi < plan.groups_per_item; ++gi) {
                    for (bool last = false; ok && !last; ++u) {
                        const uint32_t buf = plan.bufs == 2 ? u & 1 : 0, use = plan.bufs == 2 ? u >> 1 : u;
                        ok = mbar_wait(smem_u32(&sm.q_full[u & 1]), (u >> 1) & 1, abort_flag, p.status, 22) &&
                             mbar_wait(smem_u32(&sm.acc_empty[buf]), (use & 1) ^ 1, abort_flag, p.status, 23);
                        if (!ok) break;
                        last = sm.meta[u & 1].y != 0;
                        tc_fence_after();
                        for (int t = 0; t < T; ++t, ++it) {
                            const uint32_t st = it % S, slot = buf * plan.slots_per_unit + t;
                            ok = mbar_wait(smem_u32(&sm.full[st]), (it / S) & 1, abort_flag, p.status, 24);
                            if (!ok) break;
                            const uint32_t a = smem_u32(s_ring + st * C::TILE_BYTES), bq = smem_u32(s_q);
#pragma unroll
                            for (int kk = 0; kk < D / 16; ++kk)
                                umma_bf16(tmem + slot * kRows, umma_desc_sw128(a + (kk >> 2) * kKeySubBytes + (kk & 3) * 32),
                                          umma_desc_sw128(bq + (kk >> 2) * C::Q_SUB + (kk & 3) * 32), idesc, kk > 0 ? 1u : 0u);
                            umma_commit(smem_u32(&sm.empty[st]));
                            umma_commit(smem_u32(&sm.acc_full[slot]));
                        }
                        umma_commit(smem_u32(&sm.q_free));
                    }
                }
            }
        }
    } else if (warp >= kEliteWarp0 && warp < kEpiWarp0) {
        // ================================ elite rows ================================
        const int et = tid - kEliteWarp0 * 32, ew = warp - kEliteWarp0;
        const int words = (p.W + 31) >> 5;
        bool ok = true;
        uint32_t u = 0;
        for (int item = cid; ok && item < plan.items; item += n_clusters) {
            for (int gi = 0; ok && gi < plan.groups_per_item; ++gi) {
                const int grp = first_grp + item * plan.groups_per_item + gi;
                const int g = grp % p.Hkv, lb = grp / p.Hkv, l = lb / p.B, b = lb - l * p.B;
                const uint16_t *k_cand = p.k + (int64_t)l * p.s_layer + (int64_t)b * p.s_batch + (int64_t)g * p.s_head +
                                         (int64_t)(p.Nv + p.Nt - p.W) * p.s_token;
                const uint16_t *q_lb = p.qw + (int64_t)lb * p.W * p.Hq * D;
                named_bar(2, kEliteThreads);   // the previous group's keys and masks have been used
                for (int idx = et; idx < (p.W + p.G) * (D / 8); idx += kEliteThreads) {
                    const int row = idx / (D / 8), c = idx % (D / 8);
                    const uint16_t *src = row < p.W ? k_cand + (int64_t)row * p.s_token
                                                    : q_lb + ((int64_t)(p.W - 1) * p.Hq + g * p.G + (row - p.W)) * D;
                    *reinterpret_cast<uint4 *>(s_k + row * C::KS + c * 8) = __ldg(reinterpret_cast<const uint4 *>(src) + c);
                }
                named_bar(2, kEliteThreads);
                // Eq. 4, last row only: logit of candidate w for head hl, fp64 dot product in element order
                for (int idx = et; idx < p.G * p.W; idx += kEliteThreads) {
                    const int hl = idx / p.W, w = idx - hl * p.W;
                    const uint4 *q = reinterpret_cast<const uint4 *>(s_k + (p.W + hl) * C::KS);
                    const uint4 *kk = reinterpret_cast<const uint4 *>(s_k + w * C::KS);
                    double acc = 0.0;
#pragma unroll 4
                    for (int c = 0; c < D / 8; ++c) {
                        const uint4 a = q[c], bb = kk[c];
                        const uint32_t av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {bb.x, bb.y, bb.z, bb.w};
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            // a product of two bf16 values is exact in fp64, so the fused form rounds exactly where
                            // the separate multiply and add do
                            acc = __fma_rn((double)bf16lo(av[e]), (double)bf16lo(bv[e]), acc);
                            acc = __fma_rn((double)bf16hi(av[e]), (double)bf16hi(bv[e]), acc);
                        }
                    }
                    s_logit[idx] = __fmul_rn((float)acc, p.scale);
                }
                named_bar(2, kEliteThreads);
                // Eq. 5: candidates within a factor alpha of the best one (log domain, fp32); a warp per head
                for (int hl = ew; hl < p.G; hl += 4) {
                    float top = -INFINITY;
                    for (int w = lane; w < p.W; w += 32) top = fmaxf(top, s_logit[hl * p.W + w]);
                    top = warp_max(top);
                    for (int j = 0; j < 4; ++j) {
                        const int w = j * 32 + lane;
                        const bool elite = w < p.W && (p.keep_all || __fsub_rn(s_logit[hl * p.W + w], top) >= p.ln_alpha);
                        const uint32_t bits = __ballot_sync(0xffffffffu, elite);
                        if (lane == 0) sm.mask[hl][j] = bits;
                    }
                }
                named_bar(2, kEliteThreads);
                if (p.elite_mask && rank == 0 && et < p.G * ((p.W + 63) >> 6)) {
                    const int w64 = (p.W + 63) >> 6, hl = et / w64, j = et - hl * w64;
                    p.elite_mask[((int64_t)lb * p.Hq + g * p.G + hl) * w64 + j] =
                        (uint64_t)sm.mask[hl][2 * j] | ((uint64_t)sm.mask[hl][2 * j + 1] << 32);
                }
                // rows: elite rows of head 0 first, ascending window slot; lane hl holds the rows up to and with head hl
                int count = 0;
                if (lane < p.G)
                    for (int j = 0; j < words; ++j) count += __popc(sm.mask[lane][j]);
                int incl = count;
#pragma unroll
                for (int sh = 1; sh < 16; sh <<= 1) {
                    const int o = __shfl_up_sync(0xffffffffu, incl, sh);
                    if (lane >= sh) incl += o;
                }
                const int n_rows = __shfl_sync(0xffffffffu, incl, kMaxGroup - 1);
                const float head_coef = lane < p.G && count > 0 ? 1.0f / ((float)count * (float)(p.per_head ? p.G : p.Hq)) : 0.f;
                // 8 threads per row of the unit
                const int rr = et >> 3, sub = et & 7, quad = lane >> 3;
                for (int row0 = 0; ok && (row0 == 0 || row0 < n_rows); row0 += kRows, ++u) {
                    int hl = 0;
#pragma unroll
                    for (int q4 = 0; q4 < 4; ++q4) {
                        const int row_q = row0 + ew * 4 + q4;
                        const int before = __popc(__ballot_sync(0xffffffffu, lane < p.G && incl <= row_q));
                        if (quad == q4) hl = before;
                    }
                    const int row = row0 + rr;
                    const bool real = row < n_rows;
                    if (!real) hl = 0;
                    int kth = row - (__shfl_sync(0xffffffffu, incl, hl) - __shfl_sync(0xffffffffu, count, hl));
                    const float coef = __shfl_sync(0xffffffffu, head_coef, hl);
                    int w = 0;
                    uint4 qv[D / 64];
#pragma unroll
                    for (int i = 0; i < D / 64; ++i) qv[i] = make_uint4(0u, 0u, 0u, 0u);
                    if (real) {
                        // the kth elite slot of the head
                        int j = 0;
                        uint32_t m = sm.mask[hl][0];
                        while (kth >= __popc(m)) { kth -= __popc(m); m = sm.mask[hl][++j]; }
                        for (; kth > 0; --kth) m &= m - 1;
                        w = j * 32 + __ffs(m) - 1;
                        const uint4 *src = reinterpret_cast<const uint4 *>(q_lb + ((int64_t)w * p.Hq + g * p.G + hl) * D);
#pragma unroll
                        for (int i = 0; i < D / 64; ++i) qv[i] = __ldg(src + i * 8 + sub);
                    }
                    // Eq. 6-7, text columns: row w sees the elite text keys w' <= w
                    float mm = kNegBig, zz = 0.f;
                    if (real) {
                        const unsigned octet = 0xffu << (quad * 8);
                        for (int j = 0; j <= (w >> 5); ++j) {
                            uint32_t m = sm.mask[hl][j];
                            if (j == (w >> 5)) m &= 0xffffffffu >> (31 - (w & 31));
                            while (m) {
                                const int w2 = j * 32 + __ffs(m) - 1;
                                m &= m - 1;
                                float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll
                                for (int i = 0; i < D / 64; ++i) {
                                    const uint4 kv = *reinterpret_cast<const uint4 *>(s_k + w2 * C::KS + (i * 8 + sub) * 8);
                                    a0 = fmaf(bf16lo(qv[i].x), bf16lo(kv.x), a0); a1 = fmaf(bf16hi(qv[i].x), bf16hi(kv.x), a1);
                                    a2 = fmaf(bf16lo(qv[i].y), bf16lo(kv.y), a2); a3 = fmaf(bf16hi(qv[i].y), bf16hi(kv.y), a3);
                                    a0 = fmaf(bf16lo(qv[i].z), bf16lo(kv.z), a0); a1 = fmaf(bf16hi(qv[i].z), bf16hi(kv.z), a1);
                                    a2 = fmaf(bf16lo(qv[i].w), bf16lo(kv.w), a2); a3 = fmaf(bf16hi(qv[i].w), bf16hi(kv.w), a3);
                                }
                                float dot = (a0 + a1) + (a2 + a3);
                                dot += __shfl_xor_sync(octet, dot, 1);
                                dot += __shfl_xor_sync(octet, dot, 2);
                                dot += __shfl_xor_sync(octet, dot, 4);
                                merge_stats(mm, zz, dot * p.sl2, 1.0f);
                            }
                        }
                    }
                    __syncwarp();
                    // the query block is free when the previous unit's MMAs have completed, the small tables when
                    // the unit before that has been read
                    ok = (u < 1 || mbar_wait(smem_u32(&sm.q_free), (u - 1) & 1, abort_flag, p.status, 25)) &&
                         (u < 2 || mbar_wait(smem_u32(&sm.meta_empty[u & 1]), ((u >> 1) & 1) ^ 1, abort_flag, p.status, 26));
                    if (ok) {
#pragma unroll
                        for (int i = 0; i < D / 64; ++i)
                            *reinterpret_cast<uint4 *>(s_q + i * C::Q_SUB + rr * 128 + ((sub ^ (rr & 7)) << 4)) = qv[i];
                        if (sub == 0) {
                            sm.text[u & 1][rr] = make_float2(mm, real ? zz : 1.f);
                            sm.coef[u & 1][rr] = real ? coef : 0.f;
                        }
                        if (et == 0) sm.meta[u & 1] = make_int2(min(kRows, max(n_rows - row0, 0)), row0 + kRows >= n_rows);
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // read by the tensor core
                    }
                    ok = named_bar_and(2, kEliteThreads, ok);
                    if (et == 0 && ok) mbar_arrive(smem_u32(&sm.q_full[u & 1]));
                }
            }
        }
    } else if (warp >= kEpiWarp0) {
        // ================================ epilogue ================================
        const int et = tid - kEpiWarp0 * 32, ew = warp - kEpiWarp0;
        const int own = (warp & 3) * 32 + lane;   // key of a tile = tensor-memory lane
        const uint32_t taddr = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        bool ok = true, leave = false;   // leave: uniform over the four warps
        uint32_t u = 0;
        for (int item = cid; !leave && item < plan.items; item += n_clusters) {
            for (int gi = 0; !leave && gi < plan.groups_per_item; ++gi) {
                const int grp = first_grp + item * plan.groups_per_item + gi;
                float *out = (plan.part ? p.imp_part : p.scores) +
                             (int64_t)(plan.part || p.per_head ? grp : grp / p.Hkv) * p.Nv;
                bool add = gi > 0;   // the first unit of an item writes, later ones add
                for (bool last = false; !last; ++u, add = true) {
                    const uint32_t par = u & 1, buf = plan.bufs == 2 ? par : 0, use = plan.bufs == 2 ? u >> 1 : u;
                    const uint32_t base = taddr + buf * plan.slots_per_unit * kRows;
                    if (et == 0) mbar_expect_tx(smem_u32(&sm.exchange[par]), plan.cluster * kRows * 8);
                    // (a wait that gave up is carried to the barrier below, where all four warps leave)
                    ok = mbar_wait(smem_u32(&sm.q_full[par]), (u >> 1) & 1, abort_flag, p.status, 27) && ok;
                    __syncwarp();
                    const int2 meta = sm.meta[par];
                    last = meta.y != 0;
                    const int quads = (meta.x + 3) >> 2;   // rows in use, in fours
                    float m[kRows], z[kRows];
#pragma unroll
                    for (int r = 0; r < kRows; ++r) { m[r] = kNegBig; z[r] = 0.f; }

                    // ---- exponentials as the tiles arrive ----
                    for (int t = 0; t < T; ++t) {
                        ok = ok && mbar_wait(smem_u32(&sm.acc_full[buf * plan.slots_per_unit + t]), use & 1, abort_flag,
                                             p.status, 28);
                        __syncwarp();
                        tc_fence_after();
                        float x[kRows];
                        tmem_ld16_issue(base + t * kRows, x);
                        tmem_ld_wait(x);
                        const bool tail = key0 + t * 128 + 128 > p.Nv;
                        const bool valid = key0 + t * 128 + own < p.Nv;
                        if (t == 0) {
#pragma unroll
                            for (int r = 0; r < kRows; ++r) m[r] = valid ? x[r] * p.sl2 : kNegBig;
                        }
                        float top = -INFINITY;
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            if (q < quads) {
#pragma unroll
                                for (int r = 4 * q; r < 4 * q + 4; ++r) {
                                    x[r] = fmaf(x[r], p.sl2, -m[r]);
                                    if (tail && !valid) x[r] = -INFINITY;
                                    top = fmaxf(top, x[r]);
                                }
                            }
                        }
                        if (__any_sync(0xffffffffu, top > kRescale)) {
                            // move the references of the rows that outgrew them and rescale what is stored
                            tmem_st_wait();
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                if (q < quads) {
                                    float fac[4];
#pragma unroll
                                    for (int j = 0; j < 4; ++j) {
                                        const int r = 4 * q + j;
                                        const bool move = x[r] > kRescale;
                                        fac[j] = move ? fast_exp2(-x[r]) : 1.f;
                                        z[r] *= fac[j];
                                        if (move) { m[r] += x[r]; x[r] = 0.f; }
                                    }
#pragma unroll 1
                                    for (int t2 = 0; t2 < t; ++t2) {
                                        float y[4];
                                        tmem_ld4(base + t2 * kRows + 4 * q, y);
#pragma unroll
                                        for (int j = 0; j < 4; ++j) y[j] *= fac[j];
                                        tmem_st4(base + t2 * kRows + 4 * q, y);
                                    }
                                }
                            }
                        }
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            if (q < quads) {
#pragma unroll
                                for (int r = 4 * q; r < 4 * q + 4; ++r) {
                                    x[r] = fast_exp2(x[r]);
                                    z[r] += x[r];
                                }
                            }
                        }
                        tmem_st16(base + t * kRows, x);
                    }

                    // ---- (max, sum) of every row: warp, block, cluster ----
                    float top_mine = kNegBig;   // lanes 2r, 2r + 1 end up with row r
#pragma unroll
                    for (int r = 0; r < kRows; ++r) {
                        if ((r >> 2) < quads) {
                            const float top_r = warp_max(m[r]);
                            z[r] *= fast_exp2(m[r] - top_r);
                            if ((lane >> 1) == r) top_mine = top_r;
                        }
                    }
                    float s8[8], s4[4], s2[2];   // 16 sums over 32 lanes: halves of the rows change hands
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const float mine = lane & 16 ? z[8 + i] : z[i], give = lane & 16 ? z[i] : z[8 + i];
                        s8[i] = mine + __shfl_xor_sync(0xffffffffu, give, 16);
                    }
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float mine = lane & 8 ? s8[4 + i] : s8[i], give = lane & 8 ? s8[i] : s8[4 + i];
                        s4[i] = mine + __shfl_xor_sync(0xffffffffu, give, 8);
                    }
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        const float mine = lane & 4 ? s4[2 + i] : s4[i], give = lane & 4 ? s4[i] : s4[2 + i];
                        s2[i] = mine + __shfl_xor_sync(0xffffffffu, give, 4);
                    }
                    float s1 = (lane & 2 ? s2[1] : s2[0]) + __shfl_xor_sync(0xffffffffu, lane & 2 ? s2[0] : s2[1], 2);
                    s1 += __shfl_xor_sync(0xffffffffu, s1, 1);
                    if ((lane & 1) == 0) sm.warp_stats[par][ew][lane >> 1] = make_float2(top_mine, s1);
                    tmem_st_wait();
                    leave = !named_bar_and(1, kEpiThreads, ok);
                    if (leave) break;
                    if ((et >> 4) < plan.cluster) {
                        const int r = et & 15, peer = et >> 4;
                        float2 a = sm.warp_stats[par][0][r];
#pragma unroll
                        for (int w2 = 1; w2 < 4; ++w2) {
                            const float2 o = sm.warp_stats[par][w2][r];
                            merge_stats(a.x, a.y, o.x, o.y);
                        }
                        st_async_f32x2(peer_smem(smem_u32(&sm.stats[par][rank][r]), peer), a.x, a.y,
                                       peer_smem(smem_u32(&sm.exchange[par]), peer));
                    }
                    ok = mbar_wait_cluster(smem_u32(&sm.exchange[par]), (u >> 1) & 1, abort_flag, p.status, 29);
                    __syncwarp();
                    if (lane < kRows) {
                        float2 a = sm.text[par][lane];
                        for (int c = 0; c < plan.cluster; ++c) {
                            const float2 o = sm.stats[par][c][lane];
                            merge_stats(a.x, a.y, o.x, o.y);
                        }
                        sm.fin[ew][lane] = make_float2(a.x, sm.coef[par][lane] / a.y);
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&sm.meta_empty[par]));
#pragma unroll
                    for (int r = 0; r < kRows; ++r) {
                        const float2 f = sm.fin[ew][r];
                        m[r] = f.y * fast_exp2(m[r] - f.x);
                    }
                    __syncwarp();

                    // ---- Eq. 8: one key per thread and tile ----
                    for (int t = 0; t < T; ++t) {
                        float x[kRows];
                        tmem_ld16_issue(base + t * kRows, x);
                        const int key = key0 + t * 128 + own;
                        const float old = add && key < p.Nv ? out[key] : 0.f;
                        tmem_ld_wait(x);
                        float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            if (q < quads) {
#pragma unroll
                                for (int j = 0; j < 4; ++j) acc[j] = fmaf(x[4 * q + j], m[4 * q + j], acc[j]);
                            }
                        }
                        if (key < p.Nv) out[key] = old + ((acc[0] + acc[1]) + (acc[2] + acc[3]));
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&sm.acc_empty[buf]));
                }
            }
        }
    }

    __syncthreads();
    if (sm.abort) __nanosleep(100000);   // gave up: whatever neighbours still send lands before the block ends
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, kSlots * kRows);
    }
    cluster_sync_all();
}

// Stands in for the kernel above in occupancy queries (same block, same shared memory): the runtime answers one block
// per SM for every kernel that allocates tensor memory, whatever the amount; two blocks with half of it each do run.
__global__ void __launch_bounds__(kClusterThreads, 2) cluster_room_kernel() {}

// What the launch needs to know of a device, asked once: how many clusters of 1, 2, 4 and 8 blocks it holds at once.
template <int D>
const int *clusters_at_once(int smem) {
    static std::mutex lock;
    static int known[kMaxDevices][kMaxStages + 1][4];   // [device][ring stages][log2 cluster size]
    static bool have[kMaxDevices][kMaxStages + 1];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return nullptr;
    const int st = smem / ClusterCfg<D>::TILE_BYTES > kMaxStages ? kMaxStages : smem / ClusterCfg<D>::TILE_BYTES;
    std::lock_guard<std::mutex> guard(lock);
    if (!have[dev][st]) {
        if (cudaFuncSetAttribute(score_cluster_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemPerBlock) != cudaSuccess ||
            cudaFuncSetAttribute(cluster_room_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemPerBlock) != cudaSuccess) {
            cudaGetLastError();
            return nullptr;
        }
        for (int i = 0; i < 4; ++i) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(1024);
            cfg.blockDim = dim3(kClusterThreads);
            cfg.dynamicSmemBytes = smem;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = 1 << i;
            attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            int n = 0;
            if (cudaOccupancyMaxActiveClusters(&n, cluster_room_kernel, &cfg) != cudaSuccess) { cudaGetLastError(); n = 0; }
            known[dev][st][i] = n;
        }
        have[dev][st] = true;
    }
    return known[dev][st];
}

template <int D>
int launch_score_cluster_d(ScoreParams &p, const aircache_shape_t *s, const aircache_full_t *f, cudaStream_t st, int *taken) {
    using C = ClusterCfg<D>;
    *taken = 0;
    const int tiles = (p.Nv + 127) / 128;
    const int stages = C::stages(p.W, p.G);
    if (tiles > kMaxCluster * kSlots || stages < 2) return AIRCACHE_OK;
    const int smem = C::smem_bytes(p.W, p.G);
    const int *at_once = clusters_at_once<D>(smem);
    if (!at_once) return AIRCACHE_OK;
    CUtensorMap tm;
    if (make_key_map(&tm, p, s, f) != AIRCACHE_OK) return AIRCACHE_OK;

    int best = -1, best_gpi = 1;
    int64_t best_cost = 0;
    for (int i = 0; i < 4; ++i) {
        const int c = 1 << i;
        const int per = (tiles + c - 1) / c;
        if (c > tiles || per > kSlots || at_once[i] < 1) continue;
        for (int gpi = p.Hkv; ; gpi = 1) {
            if (!(p.per_head && gpi > 1)) {
                const int64_t items = (int64_t)p.n_lb * p.Hkv / gpi;
                const int64_t rounds = (items + at_once[i] - 1) / at_once[i];
                const int64_t cost = rounds * gpi * (10 * per + 20) + (gpi < p.Hkv && !p.per_head ? 20 : 0);
                if (best < 0 || cost < best_cost) { best = i; best_gpi = gpi; best_cost = cost; }
            }
            if (gpi == 1) break;
        }
    }
    if (best < 0) return AIRCACHE_OK;
    ClusterPlan plan;
    plan.cluster = 1 << best;
    plan.groups_per_item = best_gpi;
    plan.items = (int)((int64_t)p.n_lb * p.Hkv / best_gpi);
    const int per = (tiles + plan.cluster - 1) / plan.cluster;
    plan.bufs = per <= kSlots / 2 ? 2 : 1;
    plan.slots_per_unit = plan.bufs == 2 ? kSlots / 2 : kSlots;
    plan.stages = stages;
    plan.part = best_gpi < p.Hkv && !p.per_head;
    const int clusters = plan.items < at_once[best] ? plan.items : at_once[best];

    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(clusters * plan.cluster));
    cfg.blockDim = dim3(kClusterThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = plan.cluster;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    AIRCACHE_CUDA_TRY(cudaLaunchKernelEx(&cfg, score_cluster_kernel<D>, tm, p, plan));
    *taken = 1;
    return plan.part ? launch_group_sum(p, st) : AIRCACHE_OK;
}

}  // namespace

int launch_score_cluster(ScoreParams &p, const aircache_shape_t *s, const aircache_full_t *f, cudaStream_t st, int *taken) {
    return s->head_dim == 64 ? launch_score_cluster_d<64>(p, s, f, st, taken) : launch_score_cluster_d<128>(p, s, f, st, taken);
}

}  // namespace aircache
