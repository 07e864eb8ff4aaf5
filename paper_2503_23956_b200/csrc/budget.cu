// aircache_budget: strength and skewness of every region's importance distribution (Eq. 9-10), the
// layer-wise budget of Eq. 11 turned into integer row counts, and the row offsets of the ragged cache.
//
// One launch.  Every CTA reduces one cell (fp64 block reductions over the fp32 scores, which it keeps in registers:
// sum; then squared and cubed deviations together; one reduction tree for all block sizes).  The
// CTA that finishes a SEQUENCE last (one ticket per sequence in the workspace, put back to zero for the next
// call) runs that sequence's allocation with one warp: sums over the cells taken by one lane in cell order
// and every fp64 operation individually rounded (no fused multiply-add), so that the integer budgets are
// the ones the sequential definition gives; divisions, floors and the ranking of the fractional parts run
// across the lanes.  The CTA that finishes the last sequence scans the region sizes into offsets.
//
// A chain of latencies, most of it fp64.  With 512 threads, three reductions and a division per score it took 17.5 us for
// 28 cells of 7290 scores and 47 us for 1792 of 2916; now 9.3 and 22 us.  (Five blocks of 256 threads to an SM instead of
// four spill registers and gain nothing.)
#include <math.h>

#include <atomic>

#include "common.cuh"

namespace aircache {

namespace {


struct BudgetParams {
    const float *scores;     // [L*B, Nv]
    double *strength, *skewness;  // [L,B]
    int32_t *budgets;        // [L,B]
    int64_t *offsets;        // [L*B+1]
    int32_t *lens;           // [L*B]
    uint32_t *ticket;        // sequences allocated so far; zero between calls
    uint32_t *seq_ticket;    // [B] cells of the sequence reduced so far; zero between calls
    int L, B, Hc, Nv, Nt, slack, mode;   // Hc: cells per (layer, sequence) - the KV heads in per-KV-head mode, else 1
    long long total_kept;    // T per sequence
    long long first_row;     // rows of the shared buffers in front of this cache's first region
};

// The sums run over kSlots slots, token i in slot i % kSlots, whatever the block size T: a thread holds kSlots / T slots
// that lie side by side, and the tree over the slots is the same one (neighbours first), so that a sequence's sums have
// the same bits in a call of its own and in a batch.
constexpr int kSlots = 1024;

// Sums of v[0 .. N-1] over the slots, the same in all threads.  s_part: N * 32 doubles.
template <int T, int N>
__device__ __forceinline__ void block_sums(double (&v)[N][kSlots / T], double (&sum)[N], double (*s_part)[32]) {
    constexpr int S = kSlots / T, LANES = 32 / S;   // lanes that hold 32 slots
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int i = 0; i < N; ++i) {
#pragma unroll
        for (int n = S; n > 1; n >>= 1)
#pragma unroll
            for (int j = 0; j < n / 2; ++j) v[i][j] = __dadd_rn(v[i][2 * j], v[i][2 * j + 1]);
        sum[i] = v[i][0];
    }
#pragma unroll
    for (int sh = 1; sh < LANES; sh <<= 1)
#pragma unroll
        for (int i = 0; i < N; ++i) sum[i] = __dadd_rn(sum[i], __shfl_xor_sync(0xffffffffu, sum[i], sh));
    if (lane % LANES == 0)
#pragma unroll
        for (int i = 0; i < N; ++i) s_part[i][threadIdx.x / LANES] = sum[i];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < N; ++i) sum[i] = s_part[i][lane];
#pragma unroll
    for (int sh = 16; sh > 0; sh >>= 1)
#pragma unroll
        for (int i = 0; i < N; ++i) sum[i] = __dadd_rn(sum[i], __shfl_xor_sync(0xffffffffu, sum[i], sh));
}

__device__ __forceinline__ unsigned ticket_add(uint32_t *t) {   // what the block wrote before it is seen with it
    unsigned v;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(v) : "l"(t) : "memory");
    return v;
}

__device__ __forceinline__ double warp_bcast(double v, int src) {
    return __shfl_sync(0xffffffffu, v, src);
}

// Eq. 11 of one sequence, by one warp: the floors of the cells' shares, and how many rows are left for the largest fractional
// parts (returned; the fractions are in share, -1 for cells outside the split).  st/sk/w/share/bud/act are arrays in shared
// memory over the sequence's cells - its layers, or its (layer, KV head) pairs in per-KV-head mode, layer-major -
// numbered l = 0 .. n - 1; act flags cells that still take part in the proportional split.
__device__ long long split_sequence(const BudgetParams &p, int n, const double *st, const double *sk, double *w,
                                  double *share, unsigned char *act, int *bud) {
    const int L = n, lane = threadIdx.x & 31;
    // across-layer means: one lane, layer order (this fixes the rounding of the sums)
    double mean_t = 0.0, mean_k = 0.0;
    if (lane == 0) {
#pragma unroll 8
        for (int l = 0; l < L; ++l) {
            mean_t = __dadd_rn(mean_t, st[l]);
            const double s = sk[l];
            mean_k = __dadd_rn(mean_k, s > 0.0 ? s : 0.0);
        }
        mean_t = __ddiv_rn(mean_t, (double)L);
        mean_k = __ddiv_rn(mean_k, (double)L);
    }
    mean_t = warp_bcast(mean_t, 0);
    mean_k = warp_bcast(mean_k, 0);
    for (int l = lane; l < L; l += 32) {
        const double t = st[l];
        double s = sk[l];
        if (s < 0.0) s = 0.0;
        const double nt = mean_t > 0.0 ? __ddiv_rn(t, mean_t) : 1.0;
        const double nk = mean_k > 0.0 ? __ddiv_rn(s, mean_k) : 1.0;
        double ww;
        if (p.mode == 0) ww = __dmul_rn(0.5, __dadd_rn(nt, nk));
        else if (p.mode == 1) ww = nt;
        else if (p.mode == 2) ww = nk;
        else ww = 1.0;
        w[l] = ww;
        act[l] = 1;
    }
    __syncwarp();
    long long R = p.total_kept;
    // capped proportional split: a layer whose share reaches Nv keeps everything, the rest re-share
    for (;;) {
        // (a cell that has left the split has weight zero by then: adding it changes nothing)
        double wsum = 0.0;
        if (lane == 0) {
#pragma unroll 8
            for (int l = 0; l < L; ++l) wsum = __dadd_rn(wsum, w[l]);
        }
        int n_active = 0;
        for (int l = lane; l < L; l += 32) n_active += act[l];
        n_active = __reduce_add_sync(0xffffffffu, n_active);
        wsum = warp_bcast(wsum, 0);
        if (n_active == 0) break;
        int moved = 0;
        for (int l = lane; l < L; l += 32) {
            if (!act[l]) continue;
            const double sh = wsum > 0.0 ? __ddiv_rn(__dmul_rn((double)R, w[l]), wsum)
                                         : __ddiv_rn((double)R, (double)n_active);
            share[l] = sh;
            if (sh >= (double)p.Nv) {
                bud[l] = p.Nv;
                act[l] = 0;
                w[l] = 0.0;
                ++moved;
            }
        }
#pragma unroll
        for (int s = 16; s > 0; s >>= 1) moved += __shfl_xor_sync(0xffffffffu, moved, s);
        __syncwarp();
        if (moved == 0) break;
        R -= (long long)moved * p.Nv;
    }
    // floors, then the largest fractional parts (ties to the lower layer) take one more row each
    int given = 0;
    for (int l = lane; l < L; l += 32) {
        if (!act[l]) {
            share[l] = -1.0;
            continue;
        }
        const double sh = share[l];
        const int f = (int)floor(sh);
        bud[l] = f;
        given += f;
        share[l] = __dsub_rn(sh, (double)f);
    }
    long long given_all = given;
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) given_all += __shfl_xor_sync(0xffffffffu, given_all, s);
    return R - given_all;
}

template <int T, int PER>
__global__ void __launch_bounds__(T, 1024 / T) budget_kernel(BudgetParams p) {
    extern __shared__ __align__(16) unsigned char s_dyn[];
    __shared__ double s_part[3][32];
    __shared__ int s_is_last;
    const int tid = threadIdx.x;
    const int LB = p.L * p.B * p.Hc;   // cells

    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // ---------------- Eq. 9 and Eq. 10 of cell blockIdx.x ----------------
    {
        const float *x = p.scores + (int64_t)blockIdx.x * p.Nv;
        const double n = (double)p.Nv;
        constexpr int S = kSlots / T;
        auto token = [&](int k) { return k / S * kSlots + tid * S + k % S; };   // of the thread's k-th score, in slot k % S
        float f[PER];
#pragma unroll
        for (int k = 0; k < PER; ++k) f[k] = token(k) < p.Nv ? __ldg(x + token(k)) : 0.f;
        double slot[1][S] = {}, sum[1];
#pragma unroll
        for (int k = 0; k < PER; ++k) slot[0][k % S] = __dadd_rn(slot[0][k % S], (double)f[k]);
        for (int i = token(PER); i < p.Nv; i += kSlots)   // (more than fit)
#pragma unroll
            for (int j = 0; j < S; ++j)
                if (i + j < p.Nv) slot[0][j] = __dadd_rn(slot[0][j], (double)__ldg(x + i + j));
        block_sums<T, 1>(slot, sum, s_part);
        const double mu = __ddiv_rn(sum[0], n);

        double dslot[2][S] = {}, dev[2];   // sums of the squared and the cubed deviations
        auto add = [&](int j, double xi) {
            const double c = __dsub_rn(xi, mu), c2 = __dmul_rn(c, c);
            dslot[0][j] = __dadd_rn(dslot[0][j], c2);
            dslot[1][j] = __fma_rn(c2, c, dslot[1][j]);
        };
#pragma unroll
        for (int k = 0; k < PER; ++k)
            if (token(k) < p.Nv) add(k % S, (double)f[k]);
        for (int i = token(PER); i < p.Nv; i += kSlots)
#pragma unroll
            for (int j = 0; j < S; ++j)
                if (i + j < p.Nv) add(j, (double)__ldg(x + i + j));
        block_sums<T, 2>(dslot, dev, s_part + 1);
        if (tid == 0) {
            const double sigma = __dsqrt_rn(__ddiv_rn(dev[0], __dsub_rn(n, 1.0)));
            const double pre = __ddiv_rn(n, __dmul_rn(__dsub_rn(n, 1.0), __dsub_rn(n, 2.0)));
            p.strength[blockIdx.x] = sum[0];
            p.skewness[blockIdx.x] = sigma > 0.0 ? __dmul_rn(pre, __ddiv_rn(dev[1], __dmul_rn(__dmul_rn(sigma, sigma), sigma))) : 0.0;
            // cell index = (l * B + b) * Hc + g: the sequence is the middle coordinate
            const int b = (blockIdx.x / p.Hc) % p.B;
            s_is_last = ticket_add(p.seq_ticket + b) == (unsigned)(p.L * p.Hc) - 1;
            if (s_is_last) p.seq_ticket[b] = 0;
        }
        __syncthreads();
        if (!s_is_last) return;
    }

    // ---------------- the sequence's last CTA: its allocation ----------------
    const int b = (blockIdx.x / p.Hc) % p.B;
    const int n = p.L * p.Hc;   // cells of the sequence
    double *st = reinterpret_cast<double *>(s_dyn);
    double *sk = st + n;
    double *w = sk + n;
    double *share = w + n;
    int *bud = reinterpret_cast<int *>(share + n);
    unsigned char *act = reinterpret_cast<unsigned char *>(bud + n);
    // cell l of the sequence sits at ((l / Hc) * B + b) * Hc + l % Hc
    auto at = [&](int l) { return ((l / p.Hc) * p.B + b) * p.Hc + l % p.Hc; };
    for (int l = tid; l < n; l += T) {
        st[l] = __ldcg(p.strength + at(l));
        sk[l] = __ldcg(p.skewness + at(l));
    }
    __syncthreads();
    __shared__ long long s_left;
    if (tid < 32) {
        const long long left = split_sequence(p, n, st, sk, w, share, act, bud);
        if (tid == 0) s_left = left;
    }
    __syncthreads();
    // A cell gets an extra row iff fewer than `left` cells of the split precede it in the order (fraction descending, cell
    // ascending): the same set the one-at-a-time selection picks.  By all of the block: n comparisons a cell, which took one
    // warp 200 us for the 640 cells of a sequence (80 layers, 8 KV heads): 261 -> 62 us a call.
    for (int l = tid; l < n; l += T) {
        const double fr = share[l];
        int rank = 0;
#pragma unroll 4
        for (int l2 = 0; l2 < n; ++l2) {
            const double f2 = share[l2];
            rank += (f2 > fr) || (f2 == fr && l2 < l);
        }
        const int b_l = bud[l] + (act[l] && rank < s_left);
        __stcg(p.budgets + at(l), b_l);
        p.lens[at(l)] = b_l + p.Nt;
    }
    __syncthreads();
    if (tid == 0) {
        s_is_last = p.B == 1 || ticket_add(p.ticket) == (unsigned)p.B - 1;
        if (s_is_last) *p.ticket = 0;
    }
    __syncthreads();
    if (!s_is_last) return;

    // ---------------- the last sequence's CTA: offsets = exclusive scan of (budget + Nt + slack) over the cells ----
    __shared__ long long s_warp[T / 32];
    const int per = (LB + T - 1) / T;
    const int i0 = min(LB, tid * per), i1 = min(LB, i0 + per);
    long long local = 0;
    for (int i = i0; i < i1; ++i) local += __ldcg(p.budgets + i) + p.Nt + p.slack;
    long long incl = local;
    const int lane = tid & 31, warp = tid >> 5;
#pragma unroll
    for (int sh = 1; sh < 32; sh <<= 1) {
        const long long o = __shfl_up_sync(0xffffffffu, incl, sh);
        if (lane >= sh) incl += o;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        long long vv = lane < T / 32 ? s_warp[lane] : 0;
#pragma unroll
        for (int sh = 1; sh < 32; sh <<= 1) {
            const long long o = __shfl_up_sync(0xffffffffu, vv, sh);
            if (lane >= sh) vv += o;
        }
        if (lane < T / 32) s_warp[lane] = vv;
    }
    __syncthreads();
    long long run = p.first_row + incl - local + (warp > 0 ? s_warp[warp - 1] : 0);
    for (int i = i0; i < i1; ++i) {
        p.offsets[i] = run;
        run += __ldcg(p.budgets + i) + p.Nt + p.slack;
    }
    if (tid == T - 1) p.offsets[LB] = p.first_row + s_warp[T / 32 - 1];
}

template <int T, int PER>
int launch_budget_t(const BudgetParams &p, int cells, int dev, cudaStream_t st) {
    static std::atomic<uint64_t> allowed[kMaxDevices];
    const int rc = allow_shared_memory((const void *)budget_kernel<T, PER>, 96 * 1024, dev, allowed);
    if (rc) return rc;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)cells);
    cfg.blockDim = dim3(T);
    cfg.dynamicSmemBytes = (size_t)p.L * p.Hc * (4 * 8 + 4 + 1) + 16;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    AIRCACHE_CUDA_TRY(cudaLaunchKernelEx(&cfg, budget_kernel<T, PER>, p));
    return AIRCACHE_OK;
}

}  // namespace

int launch_budget(const aircache_shape_t *s, const float *scores, double ratio, int32_t mode, int32_t *budgets,
                  double *strength, double *skewness, aircache_ragged_t *layout, void *ws, cudaStream_t st) {
    const WsLayout w = ws_layout(s);
    const int LB = (int)n_cells(s);
    BudgetParams p;
    p.scores = scores;
    p.strength = strength ? strength : ws_ptr<double>(ws, w.mom_strength);
    p.skewness = skewness ? skewness : ws_ptr<double>(ws, w.mom_skew);
    p.budgets = budgets;
    p.offsets = layout->offsets;
    p.lens = layout->lens;
    p.ticket = ws_ptr<uint32_t>(ws, w.status) + 2;   // second word pair of the status block
    // one ticket per sequence: the decode kernel's split-K tickets, which every user leaves at zero (calls that
    // share a workspace are ordered on one stream)
    p.seq_ticket = ws_ptr<uint32_t>(ws, w.tickets);
    p.L = s->n_layers; p.B = s->batch; p.Hc = cells_of(s); p.Nv = s->n_visual; p.Nt = s->n_text; p.slack = s->slack; p.mode = mode;
    p.total_kept = kept_per_sequence(s, ratio);
    p.first_row = layout->first_row;
    // as in the selection: all threads a block can have for few cells, small blocks for many
    int dev = 0, sms = 0;
    const int rc = current_device(&dev, &sms);
    if (rc) return rc;
    const bool many = LB > 2 * sms;
    if (many && s->n_visual <= 256 * 16) return launch_budget_t<256, 16>(p, LB, dev, st);
    if (many) return launch_budget_t<512, 16>(p, LB, dev, st);
    return launch_budget_t<1024, 8>(p, LB, dev, st);
}

}  // namespace aircache
