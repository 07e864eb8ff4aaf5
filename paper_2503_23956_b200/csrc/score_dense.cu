// Scoring from the whole window (alpha = 0: every one of the G * W window queries is an elite row, Eq. 7 is a dense
// [G * W x N_v] contraction per KV head), on tcgen05 in two passes over the keys: softmax statistics, then importance.
//
// Both passes are one kernel, one block per SM for the whole pass.  The keys of a KV group are cut into pieces of
// whole tiles of 128 and the blocks take the pieces in turn.  Roles:
//   producer   one thread: key tiles by TMA (128-byte swizzle) through a ring of four stages; blocks of up to 128 query
//              rows, double buffered, by a tensor map over the window queries (row = window slot * G + head)
//   tensor     one warp: tcgen05.mma, M = 128, into four accumulators of 128 tensor-memory columns
//   epilogue   four sets of four warps, a set per accumulator
//   table      two warps, pass two: (reference, weight / normaliser) of the next query rows from pass one's statistics
// Pass one puts the query rows on M, so a thread owns a softmax row and sums along its columns; pass two swaps the
// operands, so a thread owns a key and sums over the rows.  Neither needs a reduction across lanes.
// The window's own keys (the elite text keys, causal) are one more tile of pass one.
//
// What bounds it: the keys, read twice, and the exponentials, two per logit.  28 layers of 28 query heads, 16 window
// queries and 7290 tokens: 36 us a pass without the exponentials (33 at the memory's rate), 24 us a pass for the
// exponentials alone (16 a clock and SM), 48 and 50 us as it is; with what it replaced 189 us a call, now 99 to 102.  (That had
// a kernel for the table of rows, running maxima, sixteen microseconds and a quarter of each pass on merging statistics
// in one block.)  Hence no work per logit but one multiply-add, the exponential and one addition, two logits to an
// instruction: a row's reference is the largest logit of its first columns, and moves only when a sum of 32 passes
// 2^60.  Reading the pieces backwards in pass two found nothing more in L2.
//
// All waits are bounded.
#include <math.h>

#include <atomic>

#include "score.cuh"

namespace aircache {

namespace {

constexpr int kDenseStages = 4;
constexpr int kDenseSets = 4;
constexpr int kEpiThreads = kDenseSets * 128;
constexpr int kDenseThreads = kEpiThreads + 128;
constexpr int kProducerWarp = kEpiThreads / 32, kTensorWarp = kProducerWarp + 1, kTableWarp = kProducerWarp + 2;
constexpr float kTooLarge = 1.152921504606846976e18f;   // 2^60

struct DensePlan {
    int wpb, row_blocks;            // window slots per block of query rows, blocks
    int pieces1, pieces2;           // pieces of a group's tiles in the two passes
    int groups_per_item, part;      // pass two: KV groups summed by one block; part: sums go to the per-group buffer
    int blocks;
};

struct DenseSmem {   // behind the ring and the query blocks
    uint64_t full[kDenseStages], empty[kDenseStages], q_full[2], q_empty[2];
    uint64_t acc_full[kDenseSets], acc_empty[kDenseSets], tab_full[2], tab_empty[2];
    union {
        float2 sums[2][kDenseSets][128];   // pass one: (reference, sum) of every row by set
        struct { float neg_ref[2][128], factor[2][128]; } tab;
    };
    uint32_t tmem;
    int abort;
};

template <int D>
struct DenseCfg {
    static constexpr int TILE_BYTES = D / 64 * kKeySubBytes;
    static constexpr int SMEM = (kDenseStages + 2) * TILE_BYTES + (int)sizeof(DenseSmem);
};

// What a block does, in the same order in every role: pieces of its share; within a piece of pass two the KV groups of
// the item; within these the blocks of query rows.
struct DenseStep {
    int grp, rb;          // KV group, block of query rows
    int t0, n;            // tiles; tile index T of pass one is the window's own keys
    int piece;            // of the group
    bool first;           // first step of its piece
};

template <int PASS, typename F>
__device__ __forceinline__ void for_each_step(const ScoreParams &p, const DensePlan &plan, F &&f) {
    const int tiles = ((p.Nv + 127) >> 7) + (PASS == 1), pieces = PASS == 1 ? plan.pieces1 : plan.pieces2;
    const int gpi = PASS == 1 ? 1 : plan.groups_per_item;
    const int items = p.n_lb * p.Hkv / gpi * pieces;
    for (int at = blockIdx.x; at < items; at += gridDim.x) {
        DenseStep s;
        s.piece = at % pieces;
        s.t0 = tiles * s.piece / pieces;
        s.n = tiles * (s.piece + 1) / pieces - s.t0;
        s.first = true;
        for (int gi = 0; gi < gpi; ++gi) {
            s.grp = p.lb0 * p.Hkv + at / pieces * gpi + gi;
            for (s.rb = 0; s.rb < plan.row_blocks; ++s.rb, s.first = false)
                if (!f(s)) return;
        }
    }
}

__device__ __forceinline__ float2 pair(const uint32_t *x, int j) { return make_float2(__uint_as_float(x[j]), __uint_as_float(x[j + 1])); }
template <int N> struct Int { static constexpr int value = N; };

template <int D, int PASS>
__global__ void __launch_bounds__(kDenseThreads, 1)
dense_kernel(const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_q, ScoreParams p, DensePlan plan) {
    using C = DenseCfg<D>;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint8_t *s_ring = smem, *s_q = smem + kDenseStages * C::TILE_BYTES;
    DenseSmem &sm = *reinterpret_cast<DenseSmem *>(s_q + 2 * C::TILE_BYTES);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int T = (p.Nv + 127) >> 7;

    if (tid == 0) {
        for (int i = 0; i < kDenseStages; ++i) { mbar_init(smem_u32(&sm.full[i]), 1); mbar_init(smem_u32(&sm.empty[i]), 1); }
        for (int i = 0; i < 2; ++i) {
            mbar_init(smem_u32(&sm.q_full[i]), 1);
            mbar_init(smem_u32(&sm.q_empty[i]), 1);
            mbar_init(smem_u32(&sm.tab_full[i]), 2);
            mbar_init(smem_u32(&sm.tab_empty[i]), kEpiThreads / 32);
        }
        for (int i = 0; i < kDenseSets; ++i) { mbar_init(smem_u32(&sm.acc_full[i]), 1); mbar_init(smem_u32(&sm.acc_empty[i]), 4); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        sm.abort = 0;
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tm_k)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tm_q)) : "memory");
    }
    // rows of a query block that no load writes stay zero
    for (int i = tid; i < 2 * C::TILE_BYTES / 16; i += kDenseThreads) reinterpret_cast<uint4 *>(s_q)[i] = make_uint4(0u, 0u, 0u, 0u);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (warp == kTensorWarp) tmem_alloc(smem_u32(&sm.tmem), 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sm.tmem;
    volatile int *abort_flag = &sm.abort;
    // Pass one waits for what is before it in the stream and only then lets pass two start (as its blocks leave): pass
    // two may read keys and queries at once, and waits before it reads statistics or writes.
    if (PASS == 1) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    }

    if (warp == kProducerWarp) {
        // ================================ producer ================================
        if (lane == 0) {
            uint32_t v = 0, it = 0;
            bool ok = true;
            for_each_step<PASS>(p, plan, [&](const DenseStep &s) {
                const int g = s.grp % p.Hkv, lb = s.grp / p.Hkv, l = lb / p.B, b = lb - l * p.B;
                ok = mbar_wait(smem_u32(&sm.q_empty[v & 1]), ((v >> 1) & 1) ^ 1, abort_flag, p.status, 40);
                if (!ok) return false;
                const uint32_t q_dst = smem_u32(s_q + (v & 1) * C::TILE_BYTES), q_bar = smem_u32(&sm.q_full[v & 1]);
                mbar_expect_tx(q_bar, plan.wpb * p.G * D * 2);
                for (int sub = 0; sub < D / 64; ++sub)
                    tma_load_4d(q_dst + sub * kKeySubBytes, &tm_q, sub * 64, g * p.G, s.rb * plan.wpb, lb, q_bar);
                ++v;
                for (int i = 0; i < s.n; ++i, ++it) {
                    const int t = s.t0 + i;
                    const uint32_t st = it % kDenseStages;
                    ok = mbar_wait(smem_u32(&sm.empty[st]), ((it / kDenseStages) & 1) ^ 1, abort_flag, p.status, 41);
                    if (!ok) return false;
                    load_key_tile<D>(smem_u32(s_ring + st * C::TILE_BYTES), &tm_k, p, t < T ? t * 128 : p.Nv + p.Nt - p.W,
                                     g, b, l, smem_u32(&sm.full[st]));
                }
                return true;
            });
            if (!ok) {   // the loads in flight end before the block does
                for (uint32_t i = it > kDenseStages ? it - kDenseStages : 0; i < it; ++i)
                    for (uint32_t n = 0; n < kSpinLimit && !mbar_test(smem_u32(&sm.full[i % kDenseStages]), (i / kDenseStages) & 1); ++n) __nanosleep(40);
                for (uint32_t i = v > 2 ? v - 2 : 0; i < v; ++i)
                    for (uint32_t n = 0; n < kSpinLimit && !mbar_test(smem_u32(&sm.q_full[i & 1]), (i >> 1) & 1); ++n) __nanosleep(40);
            }
        }
    } else if (warp == kTensorWarp) {
        // ================================ tensor core ================================
        uint32_t v = 0, it = 0, base = 0, uses[kDenseSets] = {0, 0, 0, 0};
        const uint64_t ring_desc = umma_desc_sw128(smem_u32(s_ring)), q_desc = umma_desc_sw128(smem_u32(s_q));
        for_each_step<PASS>(p, plan, [&](const DenseStep &s) {
            const int rows = min(plan.wpb, p.W - s.rb * plan.wpb) * p.G;
            const uint32_t idesc = umma_idesc_bf16(128, PASS == 1 ? 128 : (rows + 15) & ~15);
            const uint64_t q0 = q_desc + (uint64_t)((v & 1) * (C::TILE_BYTES >> 4));
            bool ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&sm.q_full[v & 1]), (v >> 1) & 1, abort_flag, p.status, 42));
            for (int i = 0; i < s.n && ok; ++i, ++it) {
                const uint32_t st = it % kDenseStages, a = (base + i) % kDenseSets;
                uint32_t use = 0;
#pragma unroll
                for (int k = 0; k < kDenseSets; ++k)
                    if (a == k) use = uses[k]++;
                ok = mbar_wait(smem_u32(&sm.full[st]), (it / kDenseStages) & 1, abort_flag, p.status, 43) &&
                     mbar_wait(smem_u32(&sm.acc_empty[a]), (use & 1) ^ 1, abort_flag, p.status, 44);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                tc_fence_after();
                const uint64_t k0 = ring_desc + (uint64_t)(st * (C::TILE_BYTES >> 4));
                if (elect_one()) {
#pragma unroll
                    for (int kk = 0; kk < D / 16; ++kk) {
                        const uint32_t off = ((kk >> 2) * kKeySubBytes + (kk & 3) * 32) >> 4;
                        umma_bf16(tmem + a * 128, (PASS == 1 ? q0 : k0) + off, (PASS == 1 ? k0 : q0) + off, idesc, kk > 0 ? 1u : 0u);
                    }
                    umma_commit(smem_u32(&sm.empty[st]));
                    umma_commit(smem_u32(&sm.acc_full[a]));
                    if (i == s.n - 1) umma_commit(smem_u32(&sm.q_empty[v & 1]));
                }
                __syncwarp();
            }
            ++v;
            // pass one: the sets go on in turn; pass two: a tile stays with its set while its piece lasts
            if (PASS == 1) base += s.n;
            return ok;
        });
    } else if (warp >= kTableWarp) {
        if (PASS == 1) {
            // every candidate is elite
            if (p.elite_mask) {
                const int w64 = (p.W + 63) >> 6;
                uint64_t *out = p.elite_mask + (int64_t)p.lb0 * p.Hq * w64;
                for (int64_t i = blockIdx.x * 64 + tid - kTableWarp * 32; i < (int64_t)p.n_lb * p.Hq * w64; i += gridDim.x * 64) {
                    const int left = p.W - (int)(i % w64) * 64;
                    out[i] = left >= 64 ? ~(uint64_t)0 : ((uint64_t)1 << left) - 1;
                }
            }
        } else {
            // ================================ table of rows ================================
            asm volatile("griddepcontrol.wait;" ::: "memory");
            uint32_t v = 0;
            const float coef = 1.0f / ((float)p.W * (float)(p.per_head ? p.G : p.Hq));
            for_each_step<PASS>(p, plan, [&](const DenseStep &s) {
                const int rows = min(plan.wpb, p.W - s.rb * plan.wpb) * p.G;
                const float2 *src = p.chunk_stats + (int64_t)(s.grp - p.lb0 * p.Hkv) * plan.pieces1 * p.cap + s.rb * plan.wpb * p.G;
                const bool ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&sm.tab_empty[v & 1]), ((v >> 1) & 1) ^ 1, abort_flag, p.status, 45));
                if (!ok) return false;
                for (int r = tid - kTableWarp * 32; r < 128; r += 64) {
                    float m = kNegBig, z = 0.f;
                    if (r < rows)
                        for (int k = 0; k < plan.pieces1; ++k) {
                            const float2 o = __ldcg(src + (int64_t)k * p.cap + r);
                            merge_stats(m, z, o.x, o.y);
                        }
                    sm.tab.neg_ref[v & 1][r] = r < rows ? -m : 0.f;
                    sm.tab.factor[v & 1][r] = r < rows ? coef / z : 0.f;
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&sm.tab_full[v & 1]));
                ++v;
                return true;
            });
        }
    } else {
        // ================================ epilogue ================================
        const int set = warp >> 2, row = tid & 127;
        const uint32_t taddr = tmem + set * 128 + ((uint32_t)((warp & 3) * 32) << 16);
        const float2 sl2 = make_float2(p.sl2, p.sl2);
        uint32_t v = 0, base = 0, uses = 0;
        if (PASS == 2) asm volatile("griddepcontrol.wait;" ::: "memory");   // (the scores may have been read by what is before)
        for_each_step<PASS>(p, plan, [&](const DenseStep &s) {
            const int rows = min(plan.wpb, p.W - s.rb * plan.wpb) * p.G;
            bool ok = true;
            auto arrived = [&]() {
                ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&sm.acc_full[set]), uses & 1, abort_flag, p.status, 46));
                tc_fence_after();
                ++uses;
            };
            auto taken = [&]() {   // the accumulator has been read
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&sm.acc_empty[set]));
            };
            if (PASS == 1) {
                const bool work = (warp & 3) * 32 < rows;
                float m = kNegBig, z = 0.f;
                // 32 columns: reference and sum of the thread's row
                auto columns = [&](const uint32_t (&x)[32]) {
                    float2 a0 = make_float2(0.f, 0.f), a1 = a0;
                    const float2 nm = make_float2(-m, -m);
#pragma unroll
                    for (int j = 0; j < 32; j += 4) {
                        const float2 u = fma2(pair(x, j), sl2, nm), w = fma2(pair(x, j + 2), sl2, nm);
                        a0 = add2(a0, make_float2(fast_exp2(u.x), fast_exp2(u.y)));
                        a1 = add2(a1, make_float2(fast_exp2(w.x), fast_exp2(w.y)));
                    }
                    a0 = add2(a0, a1);
                    float sum = a0.x + a0.y;
                    if (!(sum < kTooLarge)) {   // first columns of the row, or far above them
                        float top = __uint_as_float(x[0]);
#pragma unroll
                        for (int j = 1; j < 32; ++j) top = fmaxf(top, __uint_as_float(x[j]));
                        const float mn = fmaxf(m, top * p.sl2);
                        z *= fast_exp2(m - mn);
                        m = mn;
                        sum = 0.f;
#pragma unroll
                        for (int j = 0; j < 32; ++j) sum += fast_exp2(fmaf(__uint_as_float(x[j]), p.sl2, -m));
                    }
                    z += sum;
                };
                for (int i = (set - (int)base) & (kDenseSets - 1); i < s.n; i += kDenseSets) {
                    arrived();
                    if (!ok) break;
                    if (work) {
                        const int t = s.t0 + i;
                        uint32_t x0[32], x1[32];
                        tmem_ld32_issue(taddr, x0);
                        if (t * 128 + 128 <= p.Nv) {
#pragma unroll 1
                            for (int c = 0; c < 128; c += 64) {
                                tmem_ld_wait(x0);
                                tmem_ld32_issue(taddr + c + 32, x1);
                                columns(x0);
                                tmem_ld_wait(x1);
                                if (c == 0) tmem_ld32_issue(taddr + 64, x0);
                                columns(x1);
                            }
                        } else {
                            // the last visual keys, or the window's keys up to the row's own
                            const int valid = t < T ? p.Nv - t * 128 : s.rb * plan.wpb + row / p.G + 1;
#pragma unroll 1
                            for (int c = 0; c < 128; c += 32) {
                                if (c) tmem_ld32_issue(taddr + c, x0);
                                tmem_ld_wait(x0);
#pragma unroll
                                for (int j = 0; j < 32; ++j)
                                    if (c + j >= valid) x0[j] = __float_as_uint(-INFINITY);
                                columns(x0);
                            }
                        }
                    }
                    taken();
                }
                // the sets' sums of a row meet
                sm.sums[v & 1][set][row] = make_float2(m, z);
                int all;
                asm volatile("{\n.reg .pred a, b;\nsetp.ne.s32 a, %1, 0;\nbar.red.and.pred b, 1, %2, a;\nselp.s32 %0, 1, 0, b;\n}\n"
                             : "=r"(all) : "r"((int)ok), "n"(kEpiThreads) : "memory");
                if (!all) return false;
                if (set == (int)(v & 3) && row < rows) {
                    for (int k = 1; k < kDenseSets; ++k) {
                        const float2 o = sm.sums[v & 1][(set + k) & 3][row];
                        merge_stats(m, z, o.x, o.y);
                    }
                    __stcg(p.chunk_stats + ((int64_t)(s.grp - p.lb0 * p.Hkv) * plan.pieces1 + s.piece) * p.cap + s.rb * plan.wpb * p.G + row,
                           make_float2(m, z));
                }
                base += s.n;
            } else {
                float *out = (plan.part ? p.imp_part : p.scores) + (int64_t)(plan.part || p.per_head ? s.grp : s.grp / p.Hkv) * p.Nv;
                ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&sm.tab_full[v & 1]), (v >> 1) & 1, abort_flag, p.status, 47));
                const float4 *nm4 = reinterpret_cast<const float4 *>(sm.tab.neg_ref[v & 1]);
                const float4 *f4 = reinterpret_cast<const float4 *>(sm.tab.factor[v & 1]);
                const int n32 = rows >> 5;               // whole sets of 32 rows; the rest, if any, in up to two of 16
                const bool rest = (rows & 31) != 0, rest2 = (rows & 31) > 16;
                const bool ragged = (rows & 15) != 0;    // rows of zeros fill the last sixteen: NaN beside a masked key's infinities
                float2 a0, a1;
                auto columns = [&](const uint32_t *x, int c, auto n) {
#pragma unroll
                    for (int j = 0; j < decltype(n)::value; j += 4) {
                        const float4 nm = nm4[(c + j) >> 2], f = f4[(c + j) >> 2];
                        float2 xa = pair(x, j), xb = pair(x, j + 2);
                        if (decltype(n)::value == 16 && ragged) {
                            xa = make_float2(c + j < rows ? xa.x : 0.f, c + j + 1 < rows ? xa.y : 0.f);
                            xb = make_float2(c + j + 2 < rows ? xb.x : 0.f, c + j + 3 < rows ? xb.y : 0.f);
                        }
                        const float2 u = fma2(xa, sl2, make_float2(nm.x, nm.y));
                        const float2 w = fma2(xb, sl2, make_float2(nm.z, nm.w));
                        a0 = fma2(make_float2(fast_exp2(u.x), fast_exp2(u.y)), make_float2(f.x, f.y), a0);
                        a1 = fma2(make_float2(fast_exp2(w.x), fast_exp2(w.y)), make_float2(f.z, f.w), a1);
                    }
                };
                for (int i = (set - (int)base) & (kDenseSets - 1); i < s.n && ok; i += kDenseSets) {
                    arrived();
                    if (!ok) break;
                    a0 = a1 = make_float2(0.f, 0.f);
                    uint32_t x0[32], x1[32];
                    tmem_ld32_issue(taddr, x0);   // (beyond the rows the accumulator holds older numbers, unused)
                    int c = 0;
#pragma unroll 1
                    for (; c + 1 < n32; c += 2) {
                        tmem_ld_wait(x0);
                        tmem_ld32_issue(taddr + c * 32 + 32, x1);
                        columns(x0, c * 32, Int<32>());
                        tmem_ld_wait(x1);
                        if (c * 32 + 64 < rows) tmem_ld32_issue(taddr + c * 32 + 64, x0);
                        columns(x1, c * 32 + 32, Int<32>());
                    }
                    tmem_ld_wait(x0);
                    if (c < n32) {
                        if (rest) tmem_ld32_issue(taddr + c * 32 + 32, x1);
                        columns(x0, c * 32, Int<32>());
                        if (rest) {
                            tmem_ld_wait(x1);
                            columns(x1, c * 32 + 32, Int<16>());
                            if (rest2) columns(x1 + 16, c * 32 + 48, Int<16>());
                        }
                    } else if (rest) {
                        columns(x0, c * 32, Int<16>());
                        if (rest2) columns(x0 + 16, c * 32 + 16, Int<16>());
                    }
                    taken();
                    a0 = add2(a0, a1);
                    // the same thread has the key in every step of the piece
                    const int key = (s.t0 + i) * 128 + row;
                    if (key < p.Nv) {
                        if (s.first) out[key] = a0.x + a0.y;
                        else asm volatile("red.relaxed.gpu.global.add.f32 [%0], %1;" ::"l"(out + key), "f"(a0.x + a0.y) : "memory");
                    }
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&sm.tab_empty[v & 1]));
            }
            ++v;
            return ok;
        });
    }

    __syncthreads();
    if (sm.abort) __nanosleep(100000);
    if (warp == kTensorWarp) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

// [L * B][W][Hq][d] window queries; one box = 64 channels x a group's heads x wpb window slots.
int make_query_map(CUtensorMap *tm, const ScoreParams &p, int wpb) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return AIRCACHE_ERR_CUDA;
    const cuuint64_t dim[4] = {(cuuint64_t)p.d, (cuuint64_t)p.Hq, (cuuint64_t)p.W, (cuuint64_t)p.L * p.B};
    const cuuint64_t str[3] = {(cuuint64_t)p.d * 2, (cuuint64_t)p.Hq * p.d * 2, (cuuint64_t)p.W * p.Hq * p.d * 2};
    const cuuint32_t box[4] = {64, (cuuint32_t)p.G, (cuuint32_t)wpb, 1}, one[4] = {1, 1, 1, 1};
    const CUresult rc = fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<uint16_t *>(p.qw), dim, str, box, one,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return rc == CUDA_SUCCESS ? AIRCACHE_OK : AIRCACHE_ERR_CUDA;
}

// Pieces per item, by the longest share of a block: a tile costs tile_ns, a step (a query block, its table, the sets'
// meeting) as much as two tiles.
int choose_pieces(int64_t items, int tiles, int steps, int blocks, int most, double *cost) {
    int best = 1;
    *cost = -1;
    for (int n = 1; n <= most && n <= tiles; ++n) {
        const int64_t rounds = (items * n + blocks - 1) / blocks;
        const double c = (double)rounds * steps * ((tiles + n - 1) / n + 2.0);
        if (*cost < 0 || c < *cost) { *cost = c; best = n; }
    }
    return best;
}

template <int D, int PASS>
int launch_pass(const CUtensorMap &tk, const CUtensorMap &tq, const ScoreParams &p, const DensePlan &plan, int dev, int64_t pieces, cudaStream_t st) {
    static std::atomic<uint64_t> allowed[kMaxDevices];
    const int rc = allow_shared_memory((const void *)dense_kernel<D, PASS>, DenseCfg<D>::SMEM, dev, allowed);
    if (rc) return rc;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(pieces < plan.blocks ? pieces : plan.blocks));
    cfg.blockDim = dim3(kDenseThreads);
    cfg.dynamicSmemBytes = DenseCfg<D>::SMEM;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    AIRCACHE_CUDA_TRY(cudaLaunchKernelEx(&cfg, dense_kernel<D, PASS>, tk, tq, p, plan));
    return AIRCACHE_OK;
}

template <int D>
int launch_score_dense_d(ScoreParams &p, const CUtensorMap &tk, cudaStream_t st, int *taken) {
    *taken = 0;
    int dev = 0, sms = 0;
    int rc = current_device(&dev, &sms);
    if (rc) return rc;
    DensePlan plan;
    plan.blocks = sms;
    plan.row_blocks = (p.W + 128 / p.G - 1) / (128 / p.G);
    plan.wpb = (p.W + plan.row_blocks - 1) / plan.row_blocks;
    CUtensorMap tq;
    if (make_query_map(&tq, p, plan.wpb) != AIRCACHE_OK) return AIRCACHE_OK;
    const int T = (p.Nv + 127) / 128;
    const int64_t groups = (int64_t)p.n_lb * p.Hkv;
    double c1, c2 = 0, c2_all = 0;
    // (the statistics buffer holds onepass_chunks() pieces of every group)
    plan.pieces1 = choose_pieces(groups, T + 1, plan.row_blocks, sms, onepass_chunks(p.Nv), &c1);
    plan.groups_per_item = 1;
    plan.pieces2 = choose_pieces(groups, T, plan.row_blocks, sms, T, &c2);
    if (!p.per_head && p.Hkv > 1) {
        // one block sums the KV groups, or group_sum_kernel does, in the time of some six tiles
        const int all = choose_pieces(p.n_lb, T, plan.row_blocks * p.Hkv, sms, T, &c2_all);
        if (c2_all <= c2 + 6.0) { plan.groups_per_item = p.Hkv; plan.pieces2 = all; }
    }
    plan.part = !p.per_head && plan.groups_per_item < p.Hkv;
    rc = launch_pass<D, 1>(tk, tq, p, plan, dev, groups * plan.pieces1, st);
    if (rc) return rc;
    *taken = 1;
    rc = launch_pass<D, 2>(tk, tq, p, plan, dev, groups / plan.groups_per_item * plan.pieces2, st);
    return rc || !plan.part ? rc : launch_group_sum(p, st);
}

}  // namespace

int launch_score_dense(ScoreParams &p, const aircache_shape_t *s, const aircache_full_t *f, cudaStream_t st, int *taken) {
    *taken = 0;
    CUtensorMap tk;
    if (p.G > kMaxGroup || make_key_map(&tk, p, s, f) != AIRCACHE_OK) return AIRCACHE_OK;
    return s->head_dim == 64 ? launch_score_dense_d<64>(p, tk, st, taken) : launch_score_dense_d<128>(p, tk, st, taken);
}

}  // namespace aircache
