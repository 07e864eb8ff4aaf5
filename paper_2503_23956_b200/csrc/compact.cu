// aircache_compact: per-region top-k of the importance scores and the gather that packs the kept
// visual rows and all text rows into the ragged cache (Algorithm 1, second loop); aircache_append (Eq. 2).
//
//   select_kernel  one CTA per region, or region after region.  The k-th largest score by histograms over an order-preserving integer image
//                  of the fp32 scores: 2048 bins over the range the keys really have, then over the bin that holds
//                  the k-th, until few enough are left to be ranked directly (mostly after one histogram).  Then
//                  the kept token indices in ascending order, duplicates of the threshold value taken from the
//                  lowest indices, by ballots and one scan.
//   gather_kernel  one warp per four output rows [Hkv, d] of K' and of V' (short rows: eight or sixteen): 16-byte loads along
//                  the source rows' head slices, 16-byte stores to the packed rows.  Region of the first row by 32 probes at a time in the
//                  offsets table, of the further ones by walking on.
#include "common.cuh"

namespace aircache {

namespace {

constexpr int kSelBins = 2048;
constexpr int kSelCandidates = 256;   // keys of a bin that are ranked directly
// Order-preserving integer image of a float: a > b as floats <=> key(a) > key(b), a == b <=> equal keys.  The
// two zeros compare equal as floats, so -0.0 takes the key of +0.0 (the lower index then wins among them).
__device__ __forceinline__ uint32_t order_key(float x) {
    uint32_t u = __float_as_uint(x);
    if ((u << 1) == 0u) u = 0u;
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// Exclusive block scan of one unsigned per thread over T threads.
template <int T>
__device__ __forceinline__ uint32_t block_excl_scan(uint32_t v, uint32_t *s_warp) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t incl = v;
#pragma unroll
    for (int sh = 1; sh < 32; sh <<= 1) {
        const uint32_t o = __shfl_up_sync(0xffffffffu, incl, sh);
        if (lane >= sh) incl += o;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    // every warp adds up the warps before it
    const uint32_t w = lane < warp ? s_warp[lane] : 0u;
    const uint32_t before = __reduce_add_sync(0xffffffffu, w);
    __syncthreads();
    return before + incl - v;
}

// A thread keeps PER keys in registers (token kk * T + thread); PER = 0: any number of tokens, read again where needed.
// The chain of latencies is what it costs.  Four 256-bin passes over shared memory took 14 us for 28 regions of 7290
// tokens and 47 us for 1792 of 2916 (512 threads); this takes 6 and 20.
template <int T, int PER>
__device__ __forceinline__ void select_region(int r, const float *__restrict__ scores, const int32_t *__restrict__ budgets,
                                              const int64_t *__restrict__ offsets, int n_visual, int n_text, int slack,
                                              int64_t first_row, int32_t *__restrict__ kept, int64_t kept_cap, uint32_t *status) {
    constexpr int WARPS = T / 32;
    __shared__ uint32_t s_hist[kSelBins];
    __shared__ uint32_t s_warp[32], s_lo[32], s_hi[32];
    __shared__ uint32_t s_cand[kSelCandidates];
    __shared__ uint32_t s_pick[3];   // chosen bin, keys still to be taken from it, keys in it; then threshold, duplicates to take
    __shared__ uint32_t s_n;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    const int k = budgets[r];
    // the region's list starts after the kept rows of the regions before it; budgets and offsets come from
    // device memory, so a pair that does not fit the list buffer is reported instead of followed
    const int64_t start = offsets[r] - first_row - (int64_t)r * (n_text + slack);
    const float *x = scores + (int64_t)r * n_visual;
    uint32_t key[PER > 0 ? PER : 1];
    if (PER > 0) {
        float f[PER > 0 ? PER : 1];
#pragma unroll
        for (int kk = 0; kk < PER; ++kk) f[kk] = kk * T + tid < n_visual ? __ldg(x + kk * T + tid) : 0.f;
#pragma unroll
        for (int kk = 0; kk < PER; ++kk) key[kk] = order_key(f[kk]);
    }
    if (k < 0 || k > n_visual || start < 0 || start + k > kept_cap) {
        if (tid == 0) atomicExch(status, kStatusInconsistent);
        return;
    }
    int32_t *out = kept + start;
    if (k <= 0) return;
    if (k >= n_visual) {
        for (int i = tid; i < n_visual; i += T) out[i] = i;
        return;
    }
    // f(token, key, token exists) for all tokens of the thread; whole warps take part
    auto each = [&](auto &&f) {
        if (PER > 0) {
#pragma unroll
            for (int kk = 0; kk < PER; ++kk)
                if (kk * T + (tid & ~31) < n_visual) f(kk, kk * T + tid, key[kk], kk * T + tid < n_visual);
        } else {
            for (int i = tid; (i & ~31) < n_visual; i += T) f(i / T, i, i < n_visual ? order_key(__ldg(x + i)) : 0u, i < n_visual);
        }
    };

    uint32_t lo = 0xffffffffu, hi = 0u;
    each([&](int, int, uint32_t q, bool in) { if (in) { lo = min(lo, q); hi = max(hi, q); } });
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if (lane == 0) { s_lo[warp] = lo; s_hi[warp] = hi; }
    __syncthreads();
    lo = __reduce_min_sync(0xffffffffu, lane < WARPS ? s_lo[lane] : 0xffffffffu);
    hi = __reduce_max_sync(0xffffffffu, lane < WARPS ? s_hi[lane] : 0u);

    uint32_t thr = lo, need_eq = 0, remaining = (uint32_t)k;
    for (;;) {
        const uint32_t range = hi - lo;
        const int bits = 32 - __clz(range), shift = bits > 11 ? bits - 11 : 0;
        for (int i = tid; i < kSelBins; i += T) s_hist[i] = 0;
        if (tid == 0) s_n = 0;
        __syncthreads();
        each([&](int, int, uint32_t q, bool in) {
            in = in && q >= lo && q <= hi;
            // (scores that share a bin by the warp, zeros above all, are added with one atomic)
            const int bin = in ? (int)((q - lo) >> shift) : -1;
            int same;
            __match_all_sync(0xffffffffu, bin, &same);
            if (same) {
                if (in && lane == 0) atomicAdd(&s_hist[bin], 32u);
            } else if (in) {
                atomicAdd(&s_hist[bin], 1u);
            }
        });
        __syncthreads();
        // bins from the largest down, kSelBins / T to a thread: the one in which `remaining` keys are covered
        constexpr int BPT = kSelBins / T;
        const int top = kSelBins - 1 - tid * BPT;
        uint32_t c[BPT], sum = 0;
#pragma unroll
        for (int i = 0; i < BPT; ++i) { c[i] = s_hist[top - i]; sum += c[i]; }
        uint32_t before = block_excl_scan<T>(sum, s_warp);
        if (before < remaining && remaining <= before + sum) {
#pragma unroll
            for (int i = 0; i < BPT; ++i) {
                if (before < remaining && remaining <= before + c[i]) {
                    s_pick[0] = top - i;
                    s_pick[1] = remaining - before;
                    s_pick[2] = c[i];
                }
                before += c[i];
            }
        }
        __syncthreads();
        const uint32_t count = s_pick[2];
        lo += s_pick[0] << shift;
        hi = min(hi - lo, (1u << shift) - 1) + lo;
        remaining = s_pick[1];
        if (shift == 0) { thr = lo; need_eq = remaining; break; }
        if (count <= kSelCandidates) {
            each([&](int, int, uint32_t q, bool in) { if (in && q >= lo && q <= hi) s_cand[atomicAdd(&s_n, 1u)] = q; });
            __syncthreads();
            for (uint32_t t = tid; t < count; t += T) {
                const uint32_t mine = s_cand[t];
                uint32_t above = 0, equal = 0;
                for (uint32_t j = 0; j < count; ++j) { const uint32_t o = s_cand[j]; above += o > mine; equal += o == mine; }
                if (above < remaining && remaining <= above + equal) { s_pick[0] = mine; s_pick[1] = remaining - above; }
            }
            __syncthreads();
            thr = s_pick[0];
            need_eq = s_pick[1];
            break;
        }
        __syncthreads();   // s_pick has been read by all
    }

    // ---- the kept tokens in ascending order: `need_eq` of those equal to thr (lowest indices first), all above it ----
    const uint32_t lower = (1u << lane) - 1;
    if (PER > 0) {
        // (above, equal) per warp and step, in token order, both in one word: fewer than 65536 tokens
        __syncthreads();
        for (int i = tid; i < PER * WARPS; i += T) s_hist[i] = 0;
        __syncthreads();
        each([&](int kk, int, uint32_t q, bool in) {
            const uint32_t gt = __ballot_sync(0xffffffffu, in && q > thr), eq = __ballot_sync(0xffffffffu, in && q == thr);
            if (lane == 0) s_hist[kk * WARPS + warp] = __popc(gt) | (__popc(eq) << 16);
        });
        __syncthreads();
        uint32_t mine[(PER * WARPS + T - 1) / T > 0 ? (PER * WARPS + T - 1) / T : 1], sum = 0;
        constexpr int EPT = (PER * WARPS + T - 1) / T > 0 ? (PER * WARPS + T - 1) / T : 1;
#pragma unroll
        for (int i = 0; i < EPT; ++i) { mine[i] = tid * EPT + i < PER * WARPS ? s_hist[tid * EPT + i] : 0u; sum += mine[i]; }
        uint32_t before = block_excl_scan<T>(sum, s_warp);
#pragma unroll
        for (int i = 0; i < EPT; ++i) {
            if (tid * EPT + i < PER * WARPS) s_hist[tid * EPT + i] = before;
            before += mine[i];
        }
        __syncthreads();
        each([&](int kk, int i, uint32_t q, bool in) {
            const uint32_t gt = __ballot_sync(0xffffffffu, in && q > thr), eq = __ballot_sync(0xffffffffu, in && q == thr);
            const uint32_t b = s_hist[kk * WARPS + warp];
            const uint32_t eq_before = (b >> 16) + __popc(eq & lower);
            if (in && (q > thr || (q == thr && eq_before < need_eq)))
                out[(b & 0xffffu) + __popc(gt & lower) + min(eq_before, need_eq)] = i;
        });
    } else {
        uint32_t gt_base = 0, eq_base = 0;
        for (int i0 = 0; i0 < n_visual; i0 += T) {
            const int i = i0 + tid;
            const bool in = i < n_visual;
            const uint32_t q = in ? order_key(__ldg(x + i)) : 0u;
            const uint32_t gt = __ballot_sync(0xffffffffu, in && q > thr), eq = __ballot_sync(0xffffffffu, in && q == thr);
            __syncthreads();
            if (lane == 0) s_warp[warp] = __popc(gt) | (__popc(eq) << 16);
            __syncthreads();
            const uint32_t o = lane < WARPS ? s_warp[lane] : 0u;
            const uint32_t b = __reduce_add_sync(0xffffffffu, lane < warp ? o : 0u), all = __reduce_add_sync(0xffffffffu, o);
            const uint32_t eq_before = eq_base + (b >> 16) + __popc(eq & lower);
            if (in && (q > thr || (q == thr && eq_before < need_eq)))
                out[gt_base + (b & 0xffffu) + __popc(gt & lower) + min(eq_before, need_eq)] = i;
            gt_base += all & 0xffffu;
            eq_base += all >> 16;
        }
    }
}

// LOOP: a block takes region after region.  Blocks of 256 threads that take one region have no loop around it: with it they
// spill (76 bytes of loads), 168 regions of 2000 + 16 tokens 34.1 -> 35.9 us a call.  Those of 512 spill without it.
template <int T, int PER, bool LOOP>
__global__ void __launch_bounds__(T, T == 256 ? 5 : T == 512 ? 2 : 1) select_kernel(const float *__restrict__ scores, const int32_t *__restrict__ budgets,
                                                   const int64_t *__restrict__ offsets, int n_regions, int n_visual, int n_text,
                                                   int slack, int64_t first_row, int32_t *__restrict__ kept, int64_t kept_cap,
                                                   uint32_t *status) {
    // What is before in the stream has ended when this kernel lets the gather kernel start: that one copies its text
    // rows by the budgets at once, and waits before it reads the lists.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (!LOOP) {
        select_region<T, PER>(blockIdx.x, scores, budgets, offsets, n_visual, n_text, slack, first_row, kept, kept_cap, status);
        return;
    }
    for (int r = blockIdx.x; r < n_regions; r += gridDim.x) {
        select_region<T, PER>(r, scores, budgets, offsets, n_visual, n_text, slack, first_row, kept, kept_cap, status);
        __syncthreads();   // the shared memory has been read
    }
}

struct GatherParams {
    const uint16_t *k, *v;
    int64_t s_layer, s_batch, s_head, s_token;
    uint16_t *k_out, *v_out;
    const int64_t *offsets;
    const int32_t *budgets;
    const int32_t *kept;
    int text_blocks;   // blocks of text rows; those behind them, or all, take the kept rows
    int64_t total_rows;  // rows the output buffers hold
    int64_t kept_cap;    // entries the kept-list buffer holds
    uint32_t *status;
    int64_t first_row; // rows of the shared buffers in front of this cache's first region
    int L, B, Hkv, d, Nv, Nt, slack;
    int Hc;   // cells per (layer, sequence): 1, or the KV heads in per-KV-head mode (a row then holds one head)
};

constexpr int kGatherThreads = 256;
constexpr int kGatherRows = 4;   // of a lane
// Rows that lie side by side in a warp: a row has heads x channels / 8 vectors of 16 bytes, a power of two from 8 to 128 (1, 2, 4
// or 8 heads of 64 or 128 channels), and one of 8 or 16 leaves lanes to others.
__host__ __device__ inline int gather_rows_abreast(int vec_per_row) { return vec_per_row < 32 ? 32 / vec_per_row : 1; }

// Copies the rows of the ragged cache: for region r first the kept visual rows in ascending token order, then
// the text rows (Algorithm 1's C^l = Concat(K_v[kept], K_t)).  A lane moves a part of four rows at a
// time; short rows (of one head: budgets per KV head) lie side by side in a warp, whose lanes are all at work then: 1280 cells
// of 3000 + 300 tokens, one head of 128 channels 211 -> 148 us a call.
// The text rows need no selection result - their place follows from the budgets alone - so they are copied without a wait
// for the predecessor in the stream (the selection kernel, which releases its dependents when its last block has started):
// that part of the traffic runs beside the selection, which is bound by latency, not by bandwidth.  They have blocks of
// their own, in front, or in small calls are copied by the blocks that take the kept rows afterwards (rule: launch_compact).
// Bound by the memory.
// SHARED: a block copies text rows, then kept rows.  (An instantiation of its own: the others spill 56 bytes with it, 300
// regions of 4097 + 24 tokens 97.2 -> 98.7 us a call.)
template <bool SHARED>
__global__ void __launch_bounds__(kGatherThreads, 4) gather_kernel(GatherParams p) {
    const int lane = threadIdx.x & 31;
    const int n_regions = p.L * p.B * p.Hc;       // cells
    const int row_heads = p.Hc > 1 ? 1 : p.Hkv;   // KV heads in one row of the ragged cache
    const int vec_per_head = p.d / 8;             // 16-byte vectors per head slice
    const int vec_per_row = row_heads * vec_per_head;
    // source offset of token `tok` of cell r (its first head's slice)
    auto src_of = [&](int r, int tok) {
        const int lb = r / p.Hc, g0 = r - lb * p.Hc;
        const int l = lb / p.B, b = lb - l * p.B;
        return (int64_t)l * p.s_layer + (int64_t)b * p.s_batch + (int64_t)g0 * p.s_head + (int64_t)tok * p.s_token;
    };

    const int abreast = gather_rows_abreast(vec_per_row), lanes = 32 / abreast;   // lanes of a row
    const int my_row = lane / lanes;
    const int rows_per_warp = kGatherRows * abreast, rows_per_block = kGatherThreads / 32 * rows_per_warp;

    auto copy_rows = [&](const int64_t (&src_off)[kGatherRows], const int64_t (&dst_row)[kGatherRows]) {
        for (int v0 = lane & (lanes - 1); v0 < vec_per_row; v0 += lanes) {
            const int g = v0 / vec_per_head, c = v0 % vec_per_head;
            uint4 kk[kGatherRows], vv[kGatherRows];
#pragma unroll
            for (int i = 0; i < kGatherRows; ++i) {
                if (dst_row[i] < 0) continue;
                const int64_t so = src_off[i] + (int64_t)g * p.s_head + c * 8;
                kk[i] = __ldg(reinterpret_cast<const uint4 *>(p.k + so));
                vv[i] = __ldg(reinterpret_cast<const uint4 *>(p.v + so));
            }
#pragma unroll
            for (int i = 0; i < kGatherRows; ++i) {
                if (dst_row[i] < 0) continue;
                const int64_t dof = (dst_row[i] * row_heads + g) * p.d + c * 8;
                *reinterpret_cast<uint4 *>(p.k_out + dof) = kk[i];
                *reinterpret_cast<uint4 *>(p.v_out + dof) = vv[i];
            }
        }
    };

    if ((int)blockIdx.x < p.text_blocks) {
        // ---- text rows: row j of region r goes to offsets[r] + budgets[r] + j ----
        const int n_text_rows = n_regions * p.Nt;   // below 2^31: the cache has fewer rows than that
        const int first = (int)blockIdx.x * rows_per_block + (threadIdx.x >> 5) * rows_per_warp;
        int64_t src_off[kGatherRows], dst_row[kGatherRows];
#pragma unroll
        for (int i = 0; i < kGatherRows; ++i) {
            const int idx = first + i * abreast + my_row;
            dst_row[i] = -1;
            src_off[i] = 0;
            if (idx >= n_text_rows) continue;
            const int r = idx / p.Nt, j = idx - r * p.Nt;
            src_off[i] = src_of(r, p.Nv + j);
            const int64_t dst = p.offsets[r] + p.budgets[r] + j;
            if (dst < 0 || dst >= p.total_rows) atomicExch(p.status, kStatusInconsistent);   // not written
            else dst_row[i] = dst;
        }
        copy_rows(src_off, dst_row);
        if (!SHARED) return;
    }

    // ---- kept visual rows: where they go follows from the offsets, what goes there from the selection's lists ----
    const int64_t per = p.Nt + p.slack;   // offsets[r] - first_row - r * per = kept rows of the regions before r
    auto kept_before = [&](int r) { return p.offsets[r] - p.first_row - (int64_t)r * per; };
    int64_t n_kept = kept_before(n_regions);
    if (n_kept < 0 || n_kept > p.kept_cap) {
        if (threadIdx.x == 0) atomicExch(p.status, kStatusInconsistent);
        n_kept = 0;
    }
    const int64_t first = (int64_t)((int)blockIdx.x - (SHARED ? 0 : p.text_blocks)) * rows_per_block + (threadIdx.x >> 5) * rows_per_warp;
    if (first < n_kept) {
        // Largest r with (kept rows before r) <= first (regions without kept rows are passed over), 32 probes at a
        // time; the further rows are found by walking on.  (A binary search per row and behind the wait
        // took 2 to 6 us of a warp's time.)
        int lo = 0, n = n_regions;
        while (n > 1) {
            const int step = (n + 31) >> 5, at = lo + lane * step;
            const bool below = lane * step < n && kept_before(at) <= first;
            const int hits = __popc(__ballot_sync(0xffffffffu, below));   // offsets ascend: the first `hits` probes
            const int next = hits > 0 ? lo + (hits - 1) * step : lo;
            n = min(step, lo + n - next);
            lo = next;
        }
        int region[kGatherRows];
        int64_t src_off[kGatherRows], dst_row[kGatherRows];
        int r = lo;
        int64_t begin = kept_before(r), end = kept_before(r + 1);
#pragma unroll
        for (int i = 0; i < kGatherRows; ++i) {
            const int64_t idx = first + i * abreast + my_row;
            dst_row[i] = -1;
            src_off[i] = 0;
            region[i] = 0;
            if (idx >= n_kept) continue;
            while (r < n_regions - 1 && idx >= end) { ++r; begin = end; end = kept_before(r + 1); }
            region[i] = r;
            dst_row[i] = begin + p.first_row + r * per + (idx - begin);
        }
        asm volatile("griddepcontrol.wait;" ::: "memory");
        int tok[kGatherRows];
#pragma unroll
        for (int i = 0; i < kGatherRows; ++i) tok[i] = first + i * abreast + my_row < n_kept ? p.kept[first + i * abreast + my_row] : 0;
#pragma unroll
        for (int i = 0; i < kGatherRows; ++i) {
            if (first + i * abreast + my_row >= n_kept) continue;
            if (tok[i] < 0 || tok[i] >= p.Nv || dst_row[i] < 0 || dst_row[i] >= p.total_rows) {
                atomicExch(p.status, kStatusInconsistent);   // not copied
                dst_row[i] = -1;
            } else {
                src_off[i] = src_of(region[i], tok[i]);
            }
        }
        copy_rows(src_off, dst_row);
    } else {
        asm volatile("griddepcontrol.wait;" ::: "memory");
    }
}

__global__ void append_kernel(uint16_t *k_out, uint16_t *v_out, const int64_t *offsets, int32_t *lens,
                              const uint16_t *k_new, const uint16_t *v_new, int row_elems) {
    const int r = blockIdx.x;
    const int64_t dst = (offsets[r] + lens[r]) * row_elems;
    const int64_t src = (int64_t)r * row_elems;
    for (int c = threadIdx.x * 8; c < row_elems; c += blockDim.x * 8) {
        *reinterpret_cast<uint4 *>(k_out + dst + c) = *reinterpret_cast<const uint4 *>(k_new + src + c);
        *reinterpret_cast<uint4 *>(v_out + dst + c) = *reinterpret_cast<const uint4 *>(v_new + src + c);
    }
    __syncthreads();
    if (threadIdx.x == 0) lens[r] += 1;
}

struct SelectArgs {
    const float *scores;
    const int32_t *budgets;
    const int64_t *offsets;
    int n_regions, n_visual, n_text, slack;
    int64_t first_row;
    int32_t *kept;
    int64_t kept_cap;
    uint32_t *status;
};

template <int T, int PER, bool LOOP = false>
cudaError_t launch_select(const SelectArgs &a, int blocks, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(T);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, select_kernel<T, PER, LOOP>, a.scores, a.budgets, a.offsets, a.n_regions, a.n_visual, a.n_text, a.slack,
                              a.first_row, a.kept, a.kept_cap, a.status);
}

// Whether the gather kernel's blocks copy text rows and then kept rows, instead of blocks of their own for either.  Separate
// blocks do not keep kept rows waiting behind text rows, and win wherever there are more blocks than start beside the
// selection (28 layers of 7290 + 128 tokens 32.3 -> 30.7 us a pass with the budgets; five sequences of 1000 + 32, 140 regions,
// 21.0 -> 15.9 us a call).  But they put more blocks on some SMs than on others, and a block has an SM's share of the memory
// rate for 1.5 us.  So blocks are shared where all of one kind start beside the selection and not all of both (28 x 8 regions
// of 300 + 32 tokens: 15.9 us apart, 12.8 shared), and where, beside a selection of one block an SM, there is less than a
// text block for every SM that is free, yet one kept block more falls to some of them (28 x 2 of 1000 + 16: 11.7, 10.2).
// Not with rows above 1 KB, whose text rows take twice as long (80 regions of 600 + 64 tokens: 20.3 apart, 23.4 shared).
bool gather_shares_blocks(int64_t text, int64_t kept, int row_bytes, int select_blocks, int blocks_per_sm, int sms) {
    if (row_bytes > 1024) return false;
    // four gather blocks to an SM, fewer beside blocks of the selection
    auto beside = [&](int n) { return n >= blocks_per_sm ? 0 : 4 - (4 * n + blocks_per_sm - 1) / blocks_per_sm; };
    const int each = select_blocks / sms, more = select_blocks % sms;
    const int64_t room = (int64_t)beside(each) * (sms - more) + (int64_t)beside(each + 1) * more;
    if (text + kept > room) return (text > kept ? text : kept) <= room;
    if (blocks_per_sm > 1) return false;
    const int64_t free = sms - select_blocks;
    return text <= free && (text + kept + free - 1) / free > (kept + free - 1) / free;
}

}  // namespace

int launch_compact(const aircache_shape_t *s, const aircache_full_t *f, const float *scores,
                   const int32_t *budgets, double ratio, aircache_ragged_t *out, int32_t *kept_idx, void *ws,
                   cudaStream_t st) {
    const WsLayout w = ws_layout(s);
    const int LB = (int)n_cells(s);
    int32_t *kept = kept_idx ? kept_idx : ws_ptr<int32_t>(ws, w.kept);
    uint32_t *status = ws_ptr<uint32_t>(ws, w.status);
    const int64_t kept_cap = (int64_t)s->batch * kept_per_sequence(s, ratio);
    // At most one region per SM: as many threads as a block has, since the chain of a region is all there is.  More: small
    // blocks, of which an SM holds five (256 threads) or two.
    int dev = 0, sms = 0;
    const int rc = current_device(&dev, &sms);
    if (rc) return rc;
    const SelectArgs a = {scores, budgets, out->offsets, LB, s->n_visual, s->n_text, s->slack, out->first_row, kept, kept_cap, status};
    const bool many = LB > sms;
    // The gather kernel starts when the last block of the selection has.  Where its text rows keep the memory busy for longer
    // than a selection by 512 threads an SM takes (9 us a region), there are no more blocks than that: the rest of the SM
    // copies text rows meanwhile.  64 sequences of 2916 + 256 tokens, 28 layers: 692 -> 652 us a pass with the budgets (for
    // 50 us the memory was idle); with 24 text tokens the selection is what is waited for, and takes 33 us by as many blocks as
    // there are regions and 54 by these.  From twice as many regions on: fewer leave text rows their room anyway, and a
    // second round costs more (300 regions of 4096 + 95 tokens 104.4 us by a block each, 109.8; 300 of 4097 + 140: 118.2, 114.5).
    const double text_us = (double)LB * s->n_text * row_heads_of(s) * s->head_dim * 8 / 6.0e6;
    auto blocks_of = [&](int threads) {
        const int few = sms * (512 / threads);
        return LB >= 2 * few && text_us > 9.0 * ((LB + few - 1) / few) ? few : LB;
    };
    cudaError_t e;
    int blocks_per_sm = 1, select_blocks = LB;   // the most that an SM holds, and how many there are
    if (many && s->n_visual <= 256 * 16) {
        blocks_per_sm = 5;
        select_blocks = blocks_of(256);
        e = select_blocks < LB ? launch_select<256, 16, true>(a, select_blocks, st) : launch_select<256, 16>(a, LB, st);
    } else if (many && s->n_visual <= 512 * 16) {
        blocks_per_sm = 2;
        select_blocks = blocks_of(512);
        e = launch_select<512, 16, true>(a, select_blocks, st);
    } else if (s->n_visual <= 1024 * 8) e = launch_select<1024, 8>(a, LB, st);
    else if (s->n_visual <= 1024 * 16) e = launch_select<1024, 16>(a, LB, st);
    else e = launch_select<1024, 0>(a, LB, st);
    AIRCACHE_CUDA_TRY(e);

    GatherParams p;
    p.k = (const uint16_t *)f->k; p.v = (const uint16_t *)f->v;
    p.s_layer = f->stride_layer; p.s_batch = f->stride_batch; p.s_head = f->stride_head; p.s_token = f->stride_token;
    p.k_out = (uint16_t *)out->k; p.v_out = (uint16_t *)out->v;
    p.offsets = out->offsets; p.budgets = budgets; p.kept = kept;
    p.first_row = out->first_row;
    p.total_rows = out->total_rows;
    p.kept_cap = kept_cap;
    p.status = status;
    p.Hc = cells_of(s);
    p.L = s->n_layers; p.B = s->batch; p.Hkv = s->n_kv_heads; p.d = s->head_dim;
    p.Nv = s->n_visual; p.Nt = s->n_text; p.slack = s->slack;
    // One block per 32 rows, or more short ones (a grid limited to the resident blocks, each striding through the rows, measured
    // 20 % slower on the large configurations).  At least one block waits for the selection.
    const int rows_per_block = kGatherThreads / 32 * kGatherRows * gather_rows_abreast(row_heads_of(s) * s->head_dim / 8);
    const int64_t text = ((int64_t)LB * s->n_text + rows_per_block - 1) / rows_per_block;
    const int64_t kept_blocks = kept_cap > 0 ? (kept_cap + rows_per_block - 1) / rows_per_block : 1;
    p.text_blocks = (int)text;
    const bool shared = gather_shares_blocks(text, kept_blocks, row_heads_of(s) * s->head_dim * 2, select_blocks, blocks_per_sm, sms);
    const int64_t blocks = !shared ? text + kept_blocks : text > kept_blocks ? text : kept_blocks;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(kGatherThreads);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    AIRCACHE_CUDA_TRY(shared ? cudaLaunchKernelEx(&cfg, gather_kernel<true>, p) : cudaLaunchKernelEx(&cfg, gather_kernel<false>, p));
    AIRCACHE_LAUNCH_CHECK();
    return AIRCACHE_OK;
}

int launch_append(const aircache_shape_t *s, aircache_ragged_t *c, const void *k_new, const void *v_new,
                  int32_t appended, cudaStream_t st) {
    (void)appended;
    append_kernel<<<(unsigned)n_cells(s), 64, 0, st>>>((uint16_t *)c->k, (uint16_t *)c->v, c->offsets, c->lens,
                                                       (const uint16_t *)k_new, (const uint16_t *)v_new,
                                                       row_heads_of(s) * s->head_dim);
    AIRCACHE_LAUNCH_CHECK();
    return AIRCACHE_OK;
}

}  // namespace aircache
