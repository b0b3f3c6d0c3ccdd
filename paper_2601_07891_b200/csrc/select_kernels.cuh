// Fixed-budget selection (Ablations, "Threshold-based pruning": top-k per head, or per layer as in
// AdaKV, the alternatives thresholding is compared with).  Both are reduced to the path that already
// exists: find the cut value tau*[b,h] -- the k-th largest candidate score of list (b,h), or the
// (H*k)-th largest over all heads of sequence b -- and then run the usual window + threshold mask and
// compaction with that per-list threshold.  Candidates are the positions outside the window; scores
// equal to the cut value are all kept; NaN scores are never candidates.
//
// The cut value comes from a radix select over order-preserving 32-bit keys in three passes of 11, 11 and
// 10 bits: pass p histograms the p-th digit (from the top) of every candidate key that matches the digits
// already fixed.  Histograms of all passes live in global memory; they are zero between calls (the
// compaction that follows the selection clears them).  Each CTA re-derives the digits fixed so far from
// the earlier passes' histograms, so a pass is one launch and no kernel waits for another; in the last
// pass the CTA of a selection that is done last finishes it and writes the cut value.
// What bounds it is the latency of that chain of dependent launches, so there are as few of them as
// possible, a CTA counts one head only (2048 bins instead of 8 x 256 of four passes), and the scores of a
// later pass are loaded before the wait for the pass ahead.  32k tokens x 8 heads, from the first launch to
// the cut values: 35.5 us with four passes of 8 bits, a memset ahead and a launch for the cut values
// behind them, 17.6 us now.  That serves cut values per layer and very long sequences; others take one launch of clusters
// (select_cluster_kernel).
#pragma once

#include "score_kernel.cuh"

namespace kvzap {

constexpr int kSelectThreads = 256;
constexpr int kSelectTokens = 4 * kSelectThreads;      // tokens that a CTA counts at a time, one head
constexpr int kSelectPasses = 3;
constexpr int kSelectBins = 2048;                      // bins stored per pass (the last pass uses half of them)
// Sequences whose selections run at once: the histograms (kSelectPasses * kSelectBins words per sequence and head) are
// then at most 50 MB at 8 heads.  A context has room for kSelectSeqsFirst of them from the start.
constexpr int kSelectSeqs = 256;
constexpr int kSelectSeqsFirst = 8;
// CTAs of a launch per SM, at most: the host does not know how long each sequence is, and a CTA for every block of the whole
// input in every sequence is mostly CTAs with nothing to do (64 x 1000 tokens: 32256 of them a pass, the call 163 us; now
// 75 us).  Two launches' worth of resident CTAs, so up to a few sequences every block still has one of its own.
constexpr int kSelectCtasPerSm = 16;

__host__ __device__ constexpr int select_shift(int pass) { return pass == 0 ? 21 : pass == 1 ? 10 : 0; }
__host__ __device__ constexpr int select_bits(int pass) { return pass == 2 ? 10 : 11; }

// larger score <-> larger key; -0 sorts below +0, NaN is never turned into a key
__device__ __forceinline__ uint32_t score_key(float v)
{
    const uint32_t u = __float_as_uint(v);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float key_score(uint32_t k)
{
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

// The bins of one selection and pass that a thread looks after: 8 consecutive ones (all 2048 by the CTA; the upper
// half is zero in the last pass).
struct SelectBins {
    uint32_t c[8];
};
__device__ __forceinline__ SelectBins load_bins(const uint32_t *hist)
{
    SelectBins b;
    const uint4 x = __ldcg(reinterpret_cast<const uint4 *>(hist) + 2 * threadIdx.x);
    const uint4 y = __ldcg(reinterpret_cast<const uint4 *>(hist) + 2 * threadIdx.x + 1);
    b.c[0] = x.x; b.c[1] = x.y; b.c[2] = x.z; b.c[3] = x.w;
    b.c[4] = y.x; b.c[5] = y.y; b.c[6] = y.z; b.c[7] = y.w;
    return b;
}

// Whole CTA: walking the bins from the top, the one that holds the k-th key (k >= 1); `above` = keys in higher bins.
// Returns kSelectBins when all bins together hold fewer than k keys.  `scratch`: kSelectThreads / 32 + 2 words.
__device__ __forceinline__ uint32_t select_bin(const SelectBins &b, uint32_t k, uint32_t &above, uint32_t *scratch)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int kWarps = kSelectThreads / 32;
    uint32_t mine = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) mine += b.c[i];
    uint32_t incl = mine;                 // becomes the count in this thread's bins and those of all higher lanes
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_down_sync(0xffffffffu, incl, o);
        if (lane + o < 32) incl += y;
    }
    __syncthreads();                      // scratch may still be read by the selection before
    if (lane == 0) scratch[warp] = incl;
    if (threadIdx.x == 0) scratch[kWarps] = kSelectBins;
    __syncthreads();
    uint32_t higher = incl - mine;
#pragma unroll
    for (int w = 0; w < kWarps; ++w)
        if (w > warp) higher += scratch[w];
    if (higher < k && k <= higher + mine) {              // exactly one thread, if any
        uint32_t run = higher, bin = kSelectBins, ab = 0u;
#pragma unroll
        for (int i = 7; i >= 0; --i) {
            if (bin == kSelectBins) {
                if (run + b.c[i] >= k) { bin = 8u * threadIdx.x + i; ab = run; }
                else run += b.c[i];
            }
        }
        scratch[kWarps] = bin;
        scratch[kWarps + 1] = ab;
    }
    __syncthreads();
    above = scratch[kWarps + 1];
    return scratch[kWarps];
}

__device__ __forceinline__ uint32_t select_budget(float keep_ratio, int64_t n_cand, int per_layer, int n_heads, bool &too_many)
{
    const double k = ceil(static_cast<double>(keep_ratio) * static_cast<double>(n_cand));
    const double total = per_layer ? k * n_heads : k;
    too_many = total > 4294967295.0;
    return too_many ? 0xffffffffu : static_cast<uint32_t>(total);
}

// grid (n, n_heads, n_seqs), the sequences being cu_seqlens[0 .. n_seqs]: CTA x of a sequence counts its blocks of kSelectTokens
// tokens x, x + n, x + 2n, ... (kStrided: n may be less than the blocks of the input; the loop over them alone costs 1 us a
// call where it is not needed); hist [kSelectPasses][n_seqs][n_sel][kSelectBins], n_sel =
// per_layer ? 1 : n_heads; arrive [n_seqs][n_sel], zero between launches; the last pass writes tau_list [n_seqs][n_heads].
template <bool kStrided>
__global__ void __launch_bounds__(kSelectThreads)
select_pass_kernel(const float *__restrict__ scores, int64_t n_tokens, int n_heads, const int32_t *__restrict__ cu_seqlens,
                   int n_seqs, int window, float keep_ratio, int per_layer, int pass, uint32_t *__restrict__ hist,
                   uint32_t *__restrict__ arrive, float *__restrict__ tau_list, int32_t *__restrict__ status)
{
    __shared__ uint32_t sh[kSelectBins];
    __shared__ uint32_t scratch[kSelectThreads / 32 + 2];
    __shared__ int last_s;
    // The first pass waits for the scores, and lets the second start once it has: later passes find them complete and
    // wait for the pass ahead only where they need its histogram.
    if (pass == 0) griddep_wait();
    griddep_launch_dependents();
    const int h = blockIdx.y, b = blockIdx.z, tid = threadIdx.x;
    const int64_t t0 = cu_seqlens ? cu_seqlens[b] : 0, t1 = cu_seqlens ? cu_seqlens[b + 1] : n_tokens;
    const int64_t n_cand = t1 - t0 - window > 0 ? t1 - t0 - window : 0;
    const int64_t c0 = static_cast<int64_t>(blockIdx.x) * kSelectTokens;
    bool too_many;
    const uint32_t k = select_budget(keep_ratio, n_cand, per_layer, n_heads, too_many);
    const bool last_pass = pass == kSelectPasses - 1;
    if (c0 >= n_cand || k == 0u) {
        if (pass > 0) griddep_wait();
        if (last_pass && blockIdx.x == 0) {               // nothing to select: the cut value is +inf whatever the scores
            if (tid == 0 && k == 0u) tau_list[b * n_heads + h] = INFINITY;
        }
        return;
    }
    float v[4];
    auto load = [&](int64_t c) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int64_t i = c + j * kSelectThreads + tid;
            v[j] = i < n_cand ? __ldcg(scores + (t0 + i) * n_heads + h) : __uint_as_float(0x7fffffffu);      // NaN: no candidate
        }
    };
    load(c0);
    for (int i = tid; i < kSelectBins; i += kSelectThreads) sh[i] = 0u;
    if (pass > 0) griddep_wait();
    const int n_sel = per_layer ? 1 : n_heads, sel = b * n_sel + (per_layer ? 0 : h);
    const int64_t pass_stride = static_cast<int64_t>(n_seqs) * n_sel * kSelectBins;
    uint32_t *mine = hist + static_cast<int64_t>(sel) * kSelectBins;
    // the digits fixed by the passes before this one
    uint32_t prefix = 0u, k_rem = k, above;
    bool dead = false;                                    // fewer candidates than the budget: the cut value is -inf
    {
        SelectBins bins[kSelectPasses - 1];
#pragma unroll
        for (int q = 0; q < kSelectPasses - 1; ++q)
            if (q < pass) bins[q] = load_bins(mine + q * pass_stride);
#pragma unroll
        for (int q = 0; q < kSelectPasses - 1; ++q) {
            if (q >= pass || dead) continue;
            const uint32_t bin = select_bin(bins[q], k_rem, above, scratch);
            if (bin == kSelectBins) { dead = true; continue; }
            prefix = (prefix << select_bits(q)) | bin;
            k_rem -= above;
        }
    }
    __syncthreads();
    if (!dead) {
        const int shift = select_shift(pass), bits = select_bits(pass);
        auto count = [&]() {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (v[j] != v[j]) continue;
                const uint32_t key = score_key(v[j]);
                if (pass == 0 || (key >> (shift + bits)) == prefix) atomicAdd(&sh[(key >> shift) & ((1u << bits) - 1u)], 1u);
            }
        };
        count();
        if constexpr (kStrided) {
            const int64_t stride = static_cast<int64_t>(gridDim.x) * kSelectTokens;
            for (int64_t c = c0 + stride; c < n_cand; c += stride) {
                load(c);
                count();
            }
        }
    }
    __syncthreads();
    uint32_t *out = mine + pass * pass_stride;
    for (int i = tid; i < kSelectBins; i += kSelectThreads) {
        const uint32_t n = sh[i];
        if (n) atomicAdd(out + i, n);
    }
    if (!last_pass) return;
    // the selection's CTA that is done last takes the last digit
    __threadfence();
    __syncthreads();
    if (tid == 0) {
        if (too_many) atomicCAS(status, 0, 2 /* KVZAP_ERR_UNSUPPORTED */);
        uint32_t n_ctas = static_cast<uint32_t>((n_cand + kSelectTokens - 1) / kSelectTokens);
        if constexpr (kStrided) n_ctas = min(n_ctas, gridDim.x);
        if (per_layer) n_ctas *= n_heads;
        last_s = atomicAdd(arrive + sel, 1u) + 1u == n_ctas;
        if (last_s) arrive[sel] = 0u;
        __threadfence();
    }
    __syncthreads();
    if (!last_s) return;
    float tau = -INFINITY;
    if (!dead) {
        const uint32_t bin = select_bin(load_bins(out), k_rem, above, scratch);
        if (bin != kSelectBins) tau = key_score((prefix << select_bits(kSelectPasses - 1)) | bin);
    }
    if (per_layer) {
        if (tid < n_heads) tau_list[b * n_heads + tid] = tau;
    } else if (tid == 0) {
        tau_list[b * n_heads + h] = tau;
    }
}

// The same selection in one launch, for cut values per head: a cluster of gridDim.x CTAs (a power of two, at most 16) per
// (sequence, head), each with an equal share of the candidates, of which a thread keeps the first kSelectKept in registers
// and reads the others again in every pass.  A pass counts its digit in shared memory, adds what there is to the bins of
// the CTA that owns them (2048 / gridDim.x each, in distributed shared memory), and after one cluster barrier every CTA
// reads all bins and takes the digit itself: no global memory, no launch and no grid-wide meeting between the passes.  The
// pruning behind it reads its first scores before it waits for the cut values.  32k tokens x 8 heads, a quarter kept, the
// whole call: 38.8 us with three launches, 36.5 us with this one, 35.8 us with the early scores as well (4 x 8192 tokens 43.1 and
// 39 us); a first pass on new inputs 74 -> 65 us.  (Bins owned in turn, so that neighbouring ones, which most keys share, spread over the CTAs: 65 us, a thread's
// eight bins then come from eight CTAs.)
constexpr int kSelectKept = 8;
constexpr int kSelectMaxCluster = 16;
// Tokens of an average sequence up to which it is taken.  The whole call, us: one sequence of 300 tokens 23.4 -> 17.8, 16000
// tokens 29.9 -> 26.0, 32768 tokens 38.3 -> 35.8, but 65536 tokens 55.9 -> 57.4, 131072 tokens 87.5 -> 91.8 (16 CTAs a head are
// too few for the counting); 4 x 32768 tokens 99 -> 88, 7 x 4681 tokens 49.2 -> 42.7.  Batches have a bound of their own as well (select_ctas).
constexpr int64_t kSelectClusterTokens = 40960;

__global__ void __launch_bounds__(kSelectThreads)
select_cluster_kernel(const float *__restrict__ scores, int64_t n_tokens, int n_heads, const int32_t *__restrict__ cu_seqlens,
                      int window, float keep_ratio, float *__restrict__ tau_list)
{
    __shared__ uint32_t sh[kSelectBins];
    __shared__ __align__(16) uint32_t all[kSelectPasses][kSelectBins];      // of every pass, the bins that this CTA owns
    __shared__ uint32_t scratch[kSelectThreads / 32 + 2];
    griddep_wait();
    griddep_launch_dependents();
    const int h = blockIdx.y, b = blockIdx.z, tid = threadIdx.x;
    const int64_t t0 = cu_seqlens ? cu_seqlens[b] : 0, t1 = cu_seqlens ? cu_seqlens[b + 1] : n_tokens;
    const int64_t n_cand = t1 - t0 - window > 0 ? t1 - t0 - window : 0;
    bool too_many;
    const uint32_t k = select_budget(keep_ratio, n_cand, 0, n_heads, too_many);      // n_cand < 2^32: never too many
    if (k == 0u) {                                        // the whole cluster
        if (blockIdx.x == 0 && tid == 0) tau_list[b * n_heads + h] = INFINITY;
        return;
    }
    const int64_t share = (n_cand + gridDim.x - 1) / gridDim.x;
    const int64_t lo = blockIdx.x * share, hi = lo + share < n_cand ? lo + share : n_cand;
    const float *mine = scores + t0 * n_heads + h;
    float v[kSelectKept];
#pragma unroll
    for (int j = 0; j < kSelectKept; ++j) {
        const int64_t i = lo + j * kSelectThreads + tid;
        v[j] = i < hi ? __ldcg(mine + i * n_heads) : __uint_as_float(0x7fffffffu);      // NaN: no candidate
    }
    for (int i = tid; i < kSelectBins; i += kSelectThreads) {
        sh[i] = 0u;
#pragma unroll
        for (int q = 0; q < kSelectPasses; ++q) all[q][i] = 0u;
    }
    cluster_sync_all();                                   // everybody's bins are zero
    const int own_bits = 11 - (31 - __clz(static_cast<int>(gridDim.x)));      // log2 of the bins that a CTA owns
    uint32_t prefix = 0u, k_rem = k, above;
    bool dead = false;                                    // fewer candidates than the budget: the cut value is -inf
#pragma unroll
    for (int pass = 0; pass < kSelectPasses; ++pass) {
        const int shift = select_shift(pass), bits = select_bits(pass);
        auto count = [&](float x) {
            if (x != x) return;
            const uint32_t key = score_key(x);
            if (pass == 0 || (key >> (shift + bits)) == prefix) atomicAdd(&sh[(key >> shift) & ((1u << bits) - 1u)], 1u);
        };
#pragma unroll
        for (int j = 0; j < kSelectKept; ++j) count(v[j]);
        for (int64_t base = lo + kSelectKept * kSelectThreads; base < hi; base += 4 * kSelectThreads) {
            float x[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int64_t i = base + j * kSelectThreads + tid;
                x[j] = i < hi ? __ldcg(mine + i * n_heads) : __uint_as_float(0x7fffffffu);
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) count(x[j]);
        }
        __syncthreads();
        const uint32_t bins_addr = smem_u32(&all[pass][0]);
        for (int i = tid; i < kSelectBins; i += kSelectThreads) {
            const uint32_t n = sh[i];
            if (n) {
                sh[i] = 0u;
                red_shared_cluster_add(map_to_cta(bins_addr + 4 * i, static_cast<uint32_t>(i) >> own_bits), n);
            }
        }
        cluster_sync_all();
        SelectBins bins;                                  // 8 consecutive ones belong to one CTA
        const uint32_t at = map_to_cta(bins_addr + 32 * tid, static_cast<uint32_t>(8 * tid) >> own_bits);
        ld_shared_cluster_v4(at, bins.c[0], bins.c[1], bins.c[2], bins.c[3]);
        ld_shared_cluster_v4(at + 16, bins.c[4], bins.c[5], bins.c[6], bins.c[7]);
        const uint32_t bin = select_bin(bins, k_rem, above, scratch);
        if (bin == kSelectBins) { dead = true; break; }   // in the first pass, and the same in every CTA
        prefix = (prefix << bits) | bin;
        k_rem -= above;
    }
    if (blockIdx.x == 0 && tid == 0) tau_list[b * n_heads + h] = dead ? -INFINITY : key_score(prefix);
    cluster_sync_all();                                   // nobody leaves while its bins may still be read
}

}  // namespace kvzap
