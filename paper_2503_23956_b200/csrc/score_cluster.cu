// Scoring by thread-block clusters: Eq. 4-8 in one launch with one read of the visual keys, for sequences that a
// cluster of up to eight blocks holds (16384 visual tokens) and windows that fit a block beside two ring stages.
//
// A cluster of C blocks works on one KV group (layer, sequence, KV head) at a time, each block on a stretch of the
// visual keys in tiles of 128.  Warp roles inside a block (two blocks share an SM):
//   producer   one thread: key tiles by TMA (128-byte swizzle) through a ring of shared-memory stages
//   tensor     one warp, of which an elected lane issues: tcgen05.mma M = 128 keys, N = 16 elite rows, D in a 16-column
//              slot of tensor memory per tile, so the logits of all of a block's tiles stay on chip
//   elite      four warps: Eq. 4-5 of the group (fp32 logits, and the defining fp64 ones in element order for heads with
//              a candidate at the threshold), the masks, the table of elite rows, 16 query rows at a time into the
//              swizzled operand layout, each row's softmax statistics over the elite text keys it sees.  Every block
//              of the cluster does this for itself, one group ahead.
//   epilogue   four warps, a thread owns a key (tensor-memory lane) of every tile and the 16 rows' values in
//              registers:  e = exp2(logit - reference) as a tile arrives, written back over the logit, and the
//              running sum per row; at the end of the stretch the sums meet (warp, block, then cluster through
//              distributed shared memory), and p = e * F with F = weight / normaliser * exp2(reference - max) per
//              warp and row: one exponential per logit, no reduction across lanes for Eq. 8.
// The reference is the warp's largest logit of the row in its first tile, taken while the next tiles are on their way.  It
// need not be the maximum, only near enough for fp32's range: when a logit is more than 2^24 above it, the warp's largest
// takes its place (the stored values of the earlier tiles are rescaled; rare).  A masked key (a logit of minus infinity) is
// no reference, and scores zero.  A key 2^126 below its warp's reference has a subnormal exponential, taken without the flush
// in the same rare branch, so that a score keeps its bits down to 2^-149 (but for the additions of further units and groups
// in global memory, which flush).
//
// More than 16 elite rows: the keys are read again (from L2) for every further 16.  The KV groups of a (layer,
// sequence) either follow one another in the same cluster, each adding to the scores, or - when there are too few
// sequences to fill the GPU that way - go to different clusters and group_sum_kernel adds them, g = 0, 1, ...
//
// What it replaced (elite kernel, one-pass kernel on mma.sync with a wait between blocks, sum kernel) streamed keys
// during half of a block's life and took three launches.  Measured, 28 layers of 28 query and 4 KV heads of 128
// channels: 64 sequences of 2916 tokens 1196 -> 835 to 870 us by the box (6.2 TB/s of keys: at the memory's rate); one of
// 7290 tokens 75 -> 41 us; four of 6272, a call per layer, 33 -> 13.7 us a call.  A call of one layer is a chain of latencies (us
// behind the wait for what is before it in the stream, when a call took 13.9): 1.2 until the rows of the first query block are
// staged, 4 until the block is ready, 8 until the last tile has been multiplied, 11.5 at the end; then the sum over groups
// and the launches' hand-over, 2.4.  What shortened it from 17: the first rows and tiles are asked into L2 and the addresses worked out ahead of
// the wait, an idle warp's lanes ask for the window's queries (one thread took 1 us for the 16 copies), the text columns'
// statistics and the masks are written behind the query block, which does not need them, and no block waits for its
// cluster at its end: 16.9 -> 15.5 us; image 47.6 -> 45.3.  A reference per warp (below) left no maxima to take behind the
// last tile and the factors to one lane a row, and the first tile's exponentials come back beside the exchange: 14.6; 43.2.
// (The next tile's beside the sums of one: 104 bytes of spills, image 53.)  The bound that decides whether a head needs its
// fp64 sums comes out of the fp32 dot products themselves and no longer from norms taken while the rows were stored: 14.3 ->
// 13.9; 42.4 -> 41.4.  (That bound is 1.08 times the one from norms at normally distributed rows: two chains of 64 products instead
// of four of 32.)  The first tiles asked into L2 once, and not again by the producer: 13.8 -> 13.7; 41.4 -> 41.0.
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
constexpr float kMiddle = 0.5f * (kRescale - 126.f);   // of the exponents that need no care
constexpr float kFarDown = 7.888609052210118e-31f;   // 2^-100
constexpr float kScaleUp = 18446744073709551616.f;   // 2^64
constexpr int kPreloadRows = 128;     // window queries of a group that fit a ring stage
constexpr int kFirstAhead = 5;        // tiles asked into L2 ahead of the wait, behind the first full ring

struct ClusterSmem {   // small state behind the ring and the query block
    uint64_t full[kMaxStages], empty[kMaxStages];
    uint64_t q_full[2], text_full[2], meta_empty[2], q_free, q_all, q_taken;
    uint64_t acc_full[kSlots], acc_empty[2], exchange[2];
    float2 stats[2][kMaxCluster][kRows];   // (max, sum) of every block of the cluster
    alignas(16) float warp_ref[2][4][kRows];
    float warp_sum[2][4][kRows];
    alignas(16) float fin[4][kRows];                   // per epilogue warp: 2^64 times the factor of its rows
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
    // (W more words than the logits and sums take: without them 13 pairs of window and group of 128 channels would have room
    // for a second ring stage and come here from the older kernels, 33 others for one stage more; neither was measured)
    static int tail_bytes(int W, int G) {
        return (int)sizeof(ClusterSmem) + (W + G) * KS * 2 + (G * W * 4 + (W + G) * 4 + 15) / 16 * 16;
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
    float *s_logit = reinterpret_cast<float *>(s_k + (p.W + p.G) * C::KS);   // [G][W], for W > 32
    int *s_size = reinterpret_cast<int *>(s_logit + p.G * p.W);              // [G] largest sum of magnitudes of a head, its bits

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t rank = cluster_rank();
    const int n_clusters = gridDim.x / plan.cluster, cid = blockIdx.x / plan.cluster;

    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (tid == 0) {
        for (int i = 0; i < S; ++i) { mbar_init(smem_u32(&sm.full[i]), 1); mbar_init(smem_u32(&sm.empty[i]), 1); }
        for (int i = 0; i < 2; ++i) {
            mbar_init(smem_u32(&sm.q_full[i]), 1);
            mbar_init(smem_u32(&sm.text_full[i]), kRows);
            mbar_init(smem_u32(&sm.meta_empty[i]), 5);   // producer and four epilogue warps
            mbar_init(smem_u32(&sm.acc_empty[i]), 4);
            mbar_init(smem_u32(&sm.exchange[i]), 1);
        }
        mbar_init(smem_u32(&sm.q_free), 1);
        mbar_init(smem_u32(&sm.q_all), 1);
        mbar_init(smem_u32(&sm.q_taken), 1);
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

    // The block's first group: its rows and first tiles are asked into L2 while the block waits for what is before it in the
    // stream (hints: they consume no value; the blocks of a cluster share the lines of the rows), and the addresses of its
    // rows are worked out.
    const bool preload = p.W * p.G <= kPreloadRows;
    const int n_vec = (p.W + p.G) * (D / 8);   // 16-byte vectors of the candidate keys and the last queries
    const uint4 *first_rows[4];
    {
        const int grp = first_grp + cid * plan.groups_per_item;
        const int g = grp % p.Hkv, lb = grp / p.Hkv, l = lb / p.B, b = lb - l * p.B;
        const uint16_t *k_cand = p.k + (int64_t)l * p.s_layer + (int64_t)b * p.s_batch + (int64_t)g * p.s_head +
                                 (int64_t)(p.Nv + p.Nt - p.W) * p.s_token;
        const uint16_t *q0 = p.qw + ((int64_t)lb * p.W * p.Hq + g * p.G) * D;
        if (warp >= kEliteWarp0 && warp < kEpiWarp0) {
            constexpr int LK = D * 2 / 128;   // 128-byte lines of a key
            const int lines = LK + p.G * LK;  // and of a window slot's queries
            for (int i = (tid - kEliteWarp0 * 32) * plan.cluster + (int)rank; i < p.W * lines; i += kEliteThreads * plan.cluster) {
                const int w = i / lines, c = i - w * lines;
                prefetch_l2(c < LK ? k_cand + (int64_t)w * p.s_token + c * 64 : q0 + (int64_t)w * p.Hq * D + (c - LK) * 64);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int idx = tid - kEliteWarp0 * 32 + i * kEliteThreads, row = idx / (D / 8), c = idx % (D / 8);
                first_rows[i] = reinterpret_cast<const uint4 *>(row < p.W ? k_cand + (int64_t)row * p.s_token
                                                                          : q0 + ((int64_t)(p.W - 1) * p.Hq + row - p.W) * D) + c;
            }
        } else if (tid == 0) {
            for (int t = 0; t < T && t < S + kFirstAhead; ++t) prefetch_key_tile<D>(&tm_k, p, key0 + t * 128, g, b, l);
        }
        asm volatile("griddepcontrol.wait;" ::: "memory");   // no value above came from global memory
        // First unit of the block: all of the window's queries of the group come into the last ring stage at once, since
        // which of them are elite is known two steps later only.
        if (warp == 2 && preload) {
            if (lane == 0) mbar_expect_tx(smem_u32(&sm.q_all), p.W * p.G * D * 2);
            for (int w = lane; w < p.W; w += 32)
                bulk_load(smem_u32(s_ring + (S - 1) * C::TILE_BYTES + w * p.G * D * 2), q0 + (int64_t)w * p.Hq * D, p.G * D * 2,
                          smem_u32(&sm.q_all));
        }
    }

    // Units of work, in the same order in every role: item (the cluster's share), KV group of the item, 16 rows.
    if (warp == 0) {
        // ================================ producer ================================
        // The few rows that the elite warps need first come in before the keys of all blocks.  (Both at once: one-layer calls
        // 15.5 -> 15.7 us, an image 45.3 either way.)
        named_bar(3, kEliteThreads + 32);
        if (lane == 0) {
            bool ok = p.W * p.G > kPreloadRows || mbar_wait(smem_u32(&sm.q_all), 0, abort_flag, p.status, 32);
            uint32_t u = 0, it = 0;
            for (int item = cid; ok && item < plan.items; item += n_clusters) {
                for (int gi = 0; ok && gi < plan.groups_per_item; ++gi) {
                    const int grp = first_grp + item * plan.groups_per_item + gi;
                    const int g = grp % p.Hkv, lb = grp / p.Hkv, l = lb / p.B, b = lb - l * p.B;
                    for (bool last = false; ok && !last; ++u) {
                        for (int t = 0; t < T; ++t, ++it) {
                            const uint32_t st = it % S;
                            ok = mbar_wait(smem_u32(&sm.empty[st]), ((it / S) & 1) ^ 1, abort_flag, p.status, 20) &&
                                 (it != (uint32_t)S - 1 || mbar_wait(smem_u32(&sm.q_taken), 0, abort_flag, p.status, 31));
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
        // The whole warp walks the loop and one elected lane issues: descriptors then stay in uniform registers.  From
        // inside a one-lane branch each instruction cost 67 clocks of moves (0.5 us per tile, whatever N is).
        bool ok = true;
        uint32_t u = 0, it = 0, st = 0;
        const uint32_t idesc = umma_idesc_bf16(128, kRows);
        const uint64_t ring_desc = umma_desc_sw128(smem_u32(s_ring)), q_desc = umma_desc_sw128(smem_u32(s_q));
        for (int item = cid; ok && item < plan.items; item += n_clusters) {
            for (int gi = 0; ok && gi < plan.groups_per_item; ++gi) {
                for (bool last = false; ok && !last; ++u) {
                    const uint32_t buf = plan.bufs == 2 ? u & 1 : 0, use = plan.bufs == 2 ? u >> 1 : u;
                    ok = mbar_wait(smem_u32(&sm.q_full[u & 1]), (u >> 1) & 1, abort_flag, p.status, 22) &&
                         mbar_wait(smem_u32(&sm.acc_empty[buf]), (use & 1) ^ 1, abort_flag, p.status, 23);
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                    last = sm.meta[u & 1].y != 0;
                    tc_fence_after();
                    for (int t = 0; t < T; ++t, ++it) {
                        ok = mbar_wait(smem_u32(&sm.full[st]), (it / S) & 1, abort_flag, p.status, 24);
                        ok = __all_sync(0xffffffffu, ok);
                        if (!ok) break;
                        const uint32_t slot = buf * plan.slots_per_unit + t;
                        const uint64_t a = ring_desc + (uint64_t)(st * (C::TILE_BYTES >> 4));
                        if (elect_one()) {
#pragma unroll
                            for (int kk = 0; kk < D / 16; ++kk)
                                umma_bf16(tmem + slot * kRows, a + (((kk >> 2) * kKeySubBytes + (kk & 3) * 32) >> 4),
                                          q_desc + (((kk >> 2) * C::Q_SUB + (kk & 3) * 32) >> 4), idesc, kk > 0 ? 1u : 0u);
                            umma_commit(smem_u32(&sm.empty[st]));
                            umma_commit(smem_u32(&sm.acc_full[slot]));
                        }
                        __syncwarp();
                        if (++st == (uint32_t)S) st = 0;
                    }
                    if (ok && elect_one()) umma_commit(smem_u32(&sm.q_free));
                    __syncwarp();
                }
            }
        }
    } else if (warp >= kEliteWarp0 && warp < kEpiWarp0) {
        // ================================ elite rows ================================
        const int et = tid - kEliteWarp0 * 32, ew = warp - kEliteWarp0;
        const int words = (p.W + 31) >> 5;
        bool ok = true;
        uint32_t u = 0;
        // four vectors per thread from `base` on: loaded, then stored
        auto load_rows = [&](int grp, int base, uint4 (&v)[4]) {
            const int g = grp % p.Hkv, lb = grp / p.Hkv, l = lb / p.B, b = lb - l * p.B;
            const uint16_t *k_cand = p.k + (int64_t)l * p.s_layer + (int64_t)b * p.s_batch + (int64_t)g * p.s_head +
                                     (int64_t)(p.Nv + p.Nt - p.W) * p.s_token;
            const uint16_t *q_last = p.qw + (((int64_t)lb * p.W + p.W - 1) * p.Hq + g * p.G) * D;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int idx = base + i * kEliteThreads, row = idx / (D / 8), c = idx % (D / 8);
                v[i] = make_uint4(0u, 0u, 0u, 0u);
                if (idx < n_vec)
                    v[i] = __ldg(reinterpret_cast<const uint4 *>(row < p.W ? k_cand + (int64_t)row * p.s_token
                                                                           : q_last + (int64_t)(row - p.W) * D) + c);
            }
        };
        auto store_rows = [&](int base, const uint4 (&v)[4]) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int idx = base + i * kEliteThreads, row = idx / (D / 8), c = idx % (D / 8);
                if (idx < n_vec) *reinterpret_cast<uint4 *>(s_k + row * C::KS + c * 8) = v[i];
            }
        };
        // Eq. 4, last row only: the logit of candidate w for head hl.  The decision of Eq. 5 is defined on fp64 dot
        // products in element order, rounded to fp32.  fp32 dot products settle it wherever the difference to the
        // threshold exceeds what the two can differ by; a head with a candidate closer than that is done again in fp64
        // (about one group in 450).  The fp64 chain alone took 2-4 us of a one-layer call's 19.
        auto logit_fp32 = [&](int hl, int w, float &size) {   // size: the sum of the products' magnitudes
            const uint4 *q = reinterpret_cast<const uint4 *>(s_k + (p.W + hl) * C::KS);
            const uint4 *kk = reinterpret_cast<const uint4 *>(s_k + w * C::KS);
            // (not unrolled: a block passes here first with its instructions still to be fetched, and 7 KB of them took longer
            // than the loop does: an image 43.2 -> 42.6 us)
            float a0 = 0.f, a1 = 0.f, b0 = 0.f, b1 = 0.f;
#pragma unroll 1
            for (int c = 0; c < D / 8; ++c) {
                const uint4 a = q[c], bb = kk[c];
                const uint32_t av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {bb.x, bb.y, bb.z, bb.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float ql = bf16lo(av[e]), qh = bf16hi(av[e]), kl = bf16lo(bv[e]), kh = bf16hi(bv[e]);
                    a0 = fmaf(ql, kl, a0); a1 = fmaf(qh, kh, a1);
                    b0 = fmaf(fabsf(ql), fabsf(kl), b0); b1 = fmaf(fabsf(qh), fabsf(kh), b1);
                }
            }
            size = (b0 + b1) * p.scale;
            return (a0 + a1) * p.scale;
        };
        auto logit_fp64 = [&](int hl, int w) {
            const uint4 *q = reinterpret_cast<const uint4 *>(s_k + (p.W + hl) * C::KS);
            const uint4 *kk = reinterpret_cast<const uint4 *>(s_k + w * C::KS);
            double acc = 0.0;
#pragma unroll 1
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
            return __fmul_rn((float)acc, p.scale);
        };
        // How far (logit - best) can be off in fp32: per logit 66 roundings of the sum and 2 each for the scaled products,
        // relative to the sum of the products' magnitudes, for two logits: 2 * 68 / 2^24 and a margin, of the head's largest such
        // sum.  (Products below fp32's range: their sum is off by 128 * 2^-126 at most.)
        constexpr float kSlack = 9e-6f, kSlackLeast = 1e-30f;

        uint4 ahead[4];   // the first vectors of the next group, on their way while this one is worked on
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            ahead[i] = make_uint4(0u, 0u, 0u, 0u);
            if (et + i * kEliteThreads < n_vec) ahead[i] = __ldg(first_rows[i]);
        }

        for (int item = cid; ok && item < plan.items; item += n_clusters) {
            for (int gi = 0; ok && gi < plan.groups_per_item; ++gi) {
                const int grp = first_grp + item * plan.groups_per_item + gi;
                const int g = grp % p.Hkv, lb = grp / p.Hkv;
                const uint16_t *q_lb = p.qw + (int64_t)lb * p.W * p.Hq * D;
                named_bar(2, kEliteThreads);   // the previous group's keys and masks have been used
                if (p.W > 32 && et < p.G) s_size[et] = 0;
                store_rows(et, ahead);
                if (u == 0) asm volatile("bar.arrive 3, %0;" ::"n"(kEliteThreads + 32) : "memory");
                for (int base = et + 4 * kEliteThreads; base - et < n_vec; base += 4 * kEliteThreads) {
                    load_rows(grp, base, ahead);
                    store_rows(base, ahead);
                }
                {   // the next group of this block, if there is one
                    const int next = gi + 1 < plan.groups_per_item ? grp + 1 : first_grp + (item + n_clusters) * plan.groups_per_item;
                    if (gi + 1 < plan.groups_per_item || item + n_clusters < plan.items) load_rows(next, et, ahead);
                }
                named_bar(2, kEliteThreads);
                // Eq. 5: candidates within a factor alpha of the best one (log domain, fp32)
                if (p.W <= 32 && !p.keep_all) {
                    // a half-warp (or a warp) per head, a lane per candidate: no shared memory, no barrier
                    const int seg = p.W <= 16 ? 16 : 32, per_pass = kEliteThreads / seg;
                    const int w = lane & (seg - 1);
                    for (int h0 = 0; h0 < p.G; h0 += per_pass) {
                        const int hl = h0 + et / seg;
                        const bool in = hl < p.G && w < p.W;
                        float size = 0.f, t = -INFINITY;
                        if (in) t = logit_fp32(hl, w, size);
                        float top = t;
                        for (int sh = 1; sh < seg; sh <<= 1) {
                            top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, sh));
                            size = fmaxf(size, __shfl_xor_sync(0xffffffffu, size, sh));
                        }
                        float diff = __fsub_rn(t, top);
                        const bool near = in && !(fabsf(diff - p.ln_alpha) > fmaf(kSlack, size, kSlackLeast));
                        if (__any_sync(0xffffffffu, near)) {
                            t = in ? logit_fp64(hl, w) : -INFINITY;
                            top = t;
                            for (int sh = 1; sh < seg; sh <<= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, sh));
                            diff = __fsub_rn(t, top);
                        }
                        const uint32_t bits = __ballot_sync(0xffffffffu, in && diff >= p.ln_alpha);
                        if (hl < p.G && w < 4) sm.mask[hl][w] = w > 0 ? 0u : (seg == 32 ? bits : (bits >> (lane & 16)) & 0xffffu);
                    }
                } else if (p.keep_all) {
                    for (int i = et; i < p.G * 4; i += kEliteThreads) {
                        const int left = p.W - (i & 3) * 32;
                        sm.mask[i >> 2][i & 3] = left >= 32 ? 0xffffffffu : (left > 0 ? (1u << left) - 1 : 0u);
                    }
                } else {
                    for (int idx = et; idx < p.G * p.W; idx += kEliteThreads) {
                        float size;
                        s_logit[idx] = logit_fp32(idx / p.W, idx % p.W, size);
                        atomicMax(s_size + idx / p.W, __float_as_int(size));   // (not negative: ordered like the bits)
                    }
                    named_bar(2, kEliteThreads);
                    // a warp per head; a warp that has to look closer does its head again by itself
                    for (int hl = ew; hl < p.G; hl += 4) {
                        const float slack = fmaf(kSlack, __int_as_float(s_size[hl]), kSlackLeast);
                        for (bool again = true, exact = false; again; exact = true) {
                            float top = -INFINITY;
                            for (int w = lane; w < p.W; w += 32) top = fmaxf(top, s_logit[hl * p.W + w]);
                            top = warp_max(top);
                            bool near = false;
                            for (int j = 0; j < 4; ++j) {
                                const int w = j * 32 + lane;
                                const float diff = w < p.W ? __fsub_rn(s_logit[hl * p.W + w], top) : -INFINITY;
                                near = near || (w < p.W && !(fabsf(diff - p.ln_alpha) > slack));
                                const uint32_t bits = __ballot_sync(0xffffffffu, w < p.W && diff >= p.ln_alpha);
                                if (lane == 0) sm.mask[hl][j] = bits;
                            }
                            again = !exact && __any_sync(0xffffffffu, near);
                            if (again) {
                                for (int w = lane; w < p.W; w += 32) s_logit[hl * p.W + w] = logit_fp64(hl, w);
                                __syncwarp();
                            }
                        }
                    }
                }
                named_bar(2, kEliteThreads);
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
                if (preload && u == 0) {
                    ok = mbar_wait(smem_u32(&sm.q_all), 0, abort_flag, p.status, 30);
                    __syncwarp();
                }
                for (int row0 = 0; row0 == 0 || (ok && row0 < n_rows); row0 += kRows, ++u) {
                    int hl = 0;
#pragma unroll
                    for (int q4 = 0; q4 < 4; ++q4) {
                        const int row_q = min(row0 + ew * 4 + q4, n_rows - 1);
                        const int before = __popc(__ballot_sync(0xffffffffu, lane < p.G && incl <= row_q));
                        if (quad == q4) hl = before;
                    }
                    // (the rows that fill the last four are the last one again with weight 0: zeros make NaN of a masked key's
                    // infinities)
                    const bool real = row0 + rr < n_rows;
                    int kth = min(row0 + rr, n_rows - 1) - (__shfl_sync(0xffffffffu, incl, hl) - __shfl_sync(0xffffffffu, count, hl));
                    const float coef = __shfl_sync(0xffffffffu, head_coef, hl);
                    int w = 0;
                    uint4 qv[D / 64];
#pragma unroll
                    for (int i = 0; i < D / 64; ++i) qv[i] = make_uint4(0u, 0u, 0u, 0u);
                    if (n_rows > 0 && row0 + rr < ((n_rows + 3) & ~3)) {
                        // the kth elite slot of the head
                        int j = 0;
                        uint32_t m = sm.mask[hl][0];
                        while (kth >= __popc(m)) { kth -= __popc(m); m = sm.mask[hl][++j]; }
                        for (; kth > 0; --kth) m &= m - 1;
                        w = j * 32 + __ffs(m) - 1;
                        const uint4 *src = reinterpret_cast<const uint4 *>(q_lb + ((int64_t)w * p.Hq + g * p.G + hl) * D);
                        if (preload && u == 0) {
                            const uint4 *kept = reinterpret_cast<const uint4 *>(s_ring + (S - 1) * C::TILE_BYTES) + (w * p.G + hl) * (D / 8);
#pragma unroll
                            for (int i = 0; i < D / 64; ++i) qv[i] = kept[i * 8 + sub];
                        } else {
#pragma unroll
                            for (int i = 0; i < D / 64; ++i) qv[i] = __ldg(src + i * 8 + sub);
                        }
                    }
                    __syncwarp();
                    // the query block is free when the previous unit's MMAs have completed, the small tables when
                    // the unit before that has been read
                    ok = ok && (u < 1 || mbar_wait(smem_u32(&sm.q_free), (u - 1) & 1, abort_flag, p.status, 25)) &&
                         (u < 2 || mbar_wait(smem_u32(&sm.meta_empty[u & 1]), ((u >> 1) & 1) ^ 1, abort_flag, p.status, 26));
                    if (ok) {
#pragma unroll
                        for (int i = 0; i < D / 64; ++i)
                            *reinterpret_cast<uint4 *>(s_q + i * C::Q_SUB + rr * 128 + ((sub ^ (rr & 7)) << 4)) = qv[i];
                        if (sub == 0) sm.coef[u & 1][rr] = real ? coef : 0.f;
                        if (et == 0) sm.meta[u & 1] = make_int2(min(kRows, max(n_rows - row0, 0)), row0 + kRows >= n_rows);
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // read by the tensor core
                    }
                    ok = named_bar_and(2, kEliteThreads, ok);
                    if (et == 0 && ok) {
                        mbar_arrive(smem_u32(&sm.q_full[u & 1]));
                        if (u == 0) mbar_arrive(smem_u32(&sm.q_taken));
                    }
                    if (!ok) break;
                    if (row0 == 0) {
                        if (p.elite_mask && rank == 0 && et < p.G * ((p.W + 63) >> 6)) {
                            const int w64 = (p.W + 63) >> 6, hl = et / w64, j = et - hl * w64;
                            p.elite_mask[((int64_t)lb * p.Hq + g * p.G + hl) * w64 + j] =
                                (uint64_t)sm.mask[hl][2 * j] | ((uint64_t)sm.mask[hl][2 * j + 1] << 32);
                        }
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
                    if (sub == 0) {
                        sm.text[u & 1][rr] = make_float2(mm, real ? zz : 1.f);
                        mbar_arrive(smem_u32(&sm.text_full[u & 1]));
                    }
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
                    float m[kRows], z[kRows];   // minus the reference, and the sum of the row
#pragma unroll
                    for (int r = 0; r < kRows; ++r) { m[r] = -kNegBig; z[r] = 0.f; }

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
                            for (int q = 0; q < 4; ++q) {
                                if (q < quads) {
#pragma unroll
                                    for (int r = 4 * q; r < 4 * q + 4; ++r)   // (a masked key: -inf)
                                        m[r] = -fmaxf(warp_max(valid ? x[r] * p.sl2 : -INFINITY), kNegBig);
                                }
                            }
                        }
                        float top = 0.f;
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            if (q < quads) {
#pragma unroll
                                for (int r = 4 * q; r < 4 * q + 4; r += 2) {
                                    const float2 y = fma2(make_float2(x[r], x[r + 1]), make_float2(p.sl2, p.sl2), make_float2(m[r], m[r + 1]));
                                    x[r] = y.x; x[r + 1] = y.y;
                                    const float2 o = add2(y, make_float2(-kMiddle, -kMiddle));
                                    top = fmaxf(top, fmaxf(fabsf(o.x), fabsf(o.y)));
                                }
                            }
                        }
                        if (tail) {   // (volatile: a branch, and not sixteen selects in every tile)
#pragma unroll
                            for (int r = 0; r < kRows; ++r) {
                                asm volatile("" : "+f"(x[r]));
                                x[r] = valid ? x[r] : -INFINITY;
                            }
                        }
                        // Rare: a reference has to move, or the exponential of a key 2^126 below its warp's reference is a subnormal
                        // number.  One bound covers both: -126 <= x <= 24.  (With a minimum beside the maximum and the products one at a
                        // time an image took 43.4 us; so 41.6, as without the lower bound.)
                        bool rare = __any_sync(0xffffffffu, valid && top > kRescale - kMiddle);
                        if (rare) {   // not for keys that score zero in all rows (a third of the keys masked: 42.6 us, else 47)
                            float most = -INFINITY;
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                if (q < quads) most = fmaxf(most, fmaxf(fmaxf(x[4 * q], x[4 * q + 1]), fmaxf(x[4 * q + 2], x[4 * q + 3])));
                            }
                            rare = __any_sync(0xffffffffu, top > kRescale - kMiddle && most > -150.f);
                        }
                        if (rare) {
                            // Move the references of the rows that outgrew them and rescale what is stored.  The new one is
                            // the warp's largest logit itself, read again: reference plus difference has only the bits that
                            // are left beside the old reference, which may be a masked key's.
                            tmem_st_wait();
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                if (q < quads && __any_sync(0xffffffffu, fmaxf(fmaxf(x[4 * q], x[4 * q + 1]),
                                                                               fmaxf(x[4 * q + 2], x[4 * q + 3])) > kRescale)) {
                                    float fac[4], raw[4];
                                    tmem_ld4(base + t * kRows + 4 * q, raw);
#pragma unroll
                                    for (int j = 0; j < 4; ++j) {
                                        const int r = 4 * q + j;
                                        const bool move = warp_max(x[r]) > kRescale;
                                        const float y = tail && !valid ? -INFINITY : raw[j] * p.sl2, top_r = warp_max(y);
                                        const float mn = move ? top_r : -m[r];
                                        // (a stored value may be 2^24, so a factor below 2^-126 still counts: it is taken 2^100 times
                                        // larger, with a minus for a mark, and these rows go down by that in a second round)
                                        const float below = -m[r] - mn;
                                        fac[j] = !move ? 1.f : below < -100.f ? -fast_exp2(below + 100.f) : fast_exp2(below);
                                        z[r] *= fabsf(fac[j]);
                                        if (fac[j] < 0.f) z[r] *= kFarDown;
                                        // (beside a masked key's 1e29 nothing is left of a difference but the product's rounding)
                                        const float d = fmaf(raw[j], p.sl2, -mn);
                                        if (move) x[r] = y == -INFINITY ? y : (d > 1.f || (d < -1.f && y == mn)) ? 0.f : d;
                                        m[r] = -mn;
                                    }
#pragma unroll 1
                                    while (__any_sync(0xffffffffu, fminf(fminf(fac[0], fac[1]), fminf(fac[2], fac[3])) < 1.f)) {
#pragma unroll 1
                                        for (int t2 = 0; t2 < t; ++t2) {
                                            float o[4];
                                            tmem_ld4(base + t2 * kRows + 4 * q, o);
#pragma unroll
                                            for (int j = 0; j < 4; ++j) o[j] *= fabsf(fac[j]);
                                            tmem_st4(base + t2 * kRows + 4 * q, o);
                                        }
                                        tmem_st_wait();   // what was stored is read again
#pragma unroll
                                        for (int j = 0; j < 4; ++j) fac[j] = fac[j] < 0.f ? kFarDown : 1.f;
                                    }
                                }
                            }
#pragma unroll
                            for (int r = 0; r < kRows; ++r) x[r] = subnormal_exp2(x[r]);
                        } else {
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                if (q < quads) {
#pragma unroll
                                    for (int r = 4 * q; r < 4 * q + 4; ++r) x[r] = fast_exp2(x[r]);
                                }
                            }
                        }
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            if (q < quads) {
#pragma unroll
                                for (int r = 4 * q; r < 4 * q + 4; r += 2) {
                                    const float2 s2 = add2(make_float2(z[r], z[r + 1]), make_float2(x[r], x[r + 1]));
                                    z[r] = s2.x; z[r + 1] = s2.y;
                                }
                            }
                        }
                        tmem_st16(base + t * kRows, x);
                    }

                    // ---- (max, sum) of every row: warp, block, cluster ----
                    if (lane == 0) {
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            reinterpret_cast<float4 *>(sm.warp_ref[par][ew])[q] = make_float4(-m[4 * q], -m[4 * q + 1], -m[4 * q + 2], -m[4 * q + 3]);
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
                    if ((lane & 1) == 0) sm.warp_sum[par][ew][lane >> 1] = s1;
                    tmem_st_wait();
                    leave = !named_bar_and(1, kEpiThreads, ok);
                    if (leave) break;
                    float xa[kRows];   // the exponentials come back beside the exchange
                    tmem_ld16_issue(base, xa);
                    if ((et >> 4) < plan.cluster) {
                        const int r = et & 15, peer = et >> 4;
                        float top = kNegBig, sum = 0.f;
#pragma unroll
                        for (int w2 = 0; w2 < 4; ++w2) top = fmaxf(top, sm.warp_ref[par][w2][r]);
#pragma unroll
                        for (int w2 = 0; w2 < 4; ++w2) sum = fmaf(sm.warp_sum[par][w2][r], fast_exp2(sm.warp_ref[par][w2][r] - top), sum);
                        st_async_f32x2(peer_smem(smem_u32(&sm.stats[par][rank][r]), peer), top, sum,
                                       peer_smem(smem_u32(&sm.exchange[par]), peer));
                    }
                    ok = mbar_wait(smem_u32(&sm.text_full[par]), (u >> 1) & 1, abort_flag, p.status, 33) &&
                         mbar_wait_cluster(smem_u32(&sm.exchange[par]), (u >> 1) & 1, abort_flag, p.status, 29);
                    __syncwarp();
                    if (lane < kRows) {
                        // the largest first, so that the blocks' exponentials do not wait for one another
                        const float2 tx = sm.text[par][lane];
                        const float ref = sm.warp_ref[par][ew][lane];
                        float mx = tx.x;
#pragma unroll 4
                        for (int c = 0; c < plan.cluster; ++c) mx = fmaxf(mx, sm.stats[par][c][lane].x);
                        float sum = tx.y * fast_exp2(tx.x - mx);
#pragma unroll 4
                        for (int c = 0; c < plan.cluster; ++c) {
                            const float2 o = sm.stats[par][c][lane];
                            sum = fmaf(o.y, fast_exp2(o.x - mx), sum);
                        }
                        // 2^64 times the factor: where a warp's reference is 2^126 below the row's maximum, its keys may still be
                        // 2^24 above the reference and their scores in range.  (Exact: powers of two, and the sum in the exponent
                        // loses no bits where it is taken.)
                        const float f = sm.coef[par][lane] / sum * kScaleUp, below = ref - mx;
                        const bool far = below < -100.f;
                        sm.fin[ew][lane] = (far ? f * (1.f / kScaleUp) : f) * fast_exp2(far ? below + 64.f : below);
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&sm.meta_empty[par]));
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float4 f = reinterpret_cast<const float4 *>(sm.fin[ew])[q];
                        m[4 * q] = f.x; m[4 * q + 1] = f.y; m[4 * q + 2] = f.z; m[4 * q + 3] = f.w;
                    }
                    __syncwarp();

                    // ---- Eq. 8: one key per thread and tile, the next tile's values on their way ----
                    auto weigh = [&](const float (&x)[kRows], int t) {
                        const int key = key0 + t * 128 + own;
                        float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            if (q < quads) {
#pragma unroll
                                for (int j = 0; j < 4; ++j) acc[j] = fmaf(x[4 * q + j], m[4 * q + j], acc[j]);
                            }
                        }
                        if (key < p.Nv) {
                            // (added where it lies: one thread owns the key, so the order of the sum is the program's,
                            // and nobody waits for the old value)
                            const float v = ((acc[0] + acc[1]) + (acc[2] + acc[3])) * (1.f / kScaleUp);
                            if (add) asm volatile("red.relaxed.gpu.global.add.f32 [%0], %1;" ::"l"(out + key), "f"(v) : "memory");
                            else out[key] = v;
                        }
                    };
#pragma unroll 1
                    for (int t = 0; t < T; ++t) {
                        tmem_ld_wait(xa);
                        weigh(xa, t);
                        if (t + 1 < T) tmem_ld16_issue(base + (t + 1) * kRows, xa);
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&sm.acc_empty[buf]));
                }
            }
        }
    }

    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, kSlots * kRows);
    }
    // A block that has had its last unit's sums from every other has all that will ever be sent to it, and may end.  One that
    // gave up waits for the others (those that have ended count as arrived): what they still send lands before it ends.
    if (sm.abort) {
        __nanosleep(100000);
        cluster_sync_all();
    }
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
    static std::atomic<uint64_t> allowed[kMaxDevices];
    if (allow_shared_memory((const void *)score_cluster_kernel<D>, kSmemPerBlock, dev, allowed)) {
        cudaGetLastError();
        return nullptr;
    }
    std::lock_guard<std::mutex> guard(lock);
    if (!have[dev][st]) {
        if (cudaFuncSetAttribute(cluster_room_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemPerBlock) != cudaSuccess) {
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

    // Cluster size and groups per item by estimated time (ns).  Measured on a B200, when a one-layer call took 17 us (13.7 since): HBM delivers a tile of 128 keys by
    // 128 channels in 5.3 ns over all SMs; a unit takes a block 0.6 us per tile plus the exchange (4 us where the tensor
    // memory holds one unit only, else hidden), and never less than the elite rows of the next group, 9 us.  A sum over
    // groups in a kernel of its own adds 2.5 us and 3 % of the traffic.
    int best = -1, best_gpi = 1;
    double best_cost = 0;
    for (int i = 0; i < 4; ++i) {
        const int c = 1 << i;
        const int per = (tiles + c - 1) / c;
        if (c > tiles || per > kSlots || at_once[i] < 1) continue;
        for (int gpi = p.per_head ? 1 : p.Hkv; ; gpi = 1) {
            const int64_t items = (int64_t)p.n_lb * p.Hkv / gpi;
            const int64_t rounds = (items + at_once[i] - 1) / at_once[i];
            const double hbm = 5.3 * D / 128 * tiles * p.n_lb * p.Hkv;
            const double stream = 600.0 * per + (per > kSlots / 2 ? 4000.0 : 1000.0);
            const double unit = (stream > 9000.0 ? stream : 9000.0) + 100.0 * per;
            const double busy = unit * rounds * gpi;
            double cost = (hbm > busy ? hbm : busy) + unit;
            if (gpi < p.Hkv && !p.per_head) cost += 2500.0 + 0.03 * hbm;
            if (best < 0 || cost < best_cost) { best = i; best_gpi = gpi; best_cost = cost; }
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
    // as many rounds as the clusters at once need, and no more clusters than fill them evenly
    const int rounds = (plan.items + at_once[best] - 1) / at_once[best];
    const int clusters = (plan.items + rounds - 1) / rounds;

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
