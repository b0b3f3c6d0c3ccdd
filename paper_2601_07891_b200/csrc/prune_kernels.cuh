// Threshold/window mask, per-head prefix sums and ordered K/V compaction
// (Algorithm 1: the window, threshold and gather steps).  Everything here is integer / byte work and must
// be bit-exact.
//
// Data flow (all on one stream, no CTA ever waits for another):
//   mask words  [H][n_words]    one keep bit per (head, packed token), 32 tokens per word,
//                               written either by the scoring epilogue or by mask_kernel
//   compact_dense_kernel        the compaction of every entry point that has a context: a CTA owns a
//                               run of 128-token blocks of one head, counts the rows kept before them
//                               straight from the mask words, ranks its kept rows with popc and copies
//                               whole K and V rows with 16-byte accesses to their slot in the (b,h)
//                               list (dense-ragged) or in the list's pages (paged)
//   scan_kernel                 paged output only: lengths[b,h] and the first page of every list
//                               (an exclusive scan over all lists, the one step that needs them all)
//   compact_kernel              the older one-CTA-per-(block, head) compaction behind scan_kernel's
//                               block prefix; still used by the allocation-free entry point
#pragma once

#include "score_kernel.cuh"

namespace kvzap {

constexpr int kBlockTokens = 128;     // tokens per mask block = 4 words (same as the scoring tile)

// ---------------------------------------------------------------------------
// keep[h,t] = in_window(t) || scores[t,h] >= tau, as 32-token ballot words.
// One warp per 32 tokens; 4 warps per CTA = one 128-token block.
// tau_list != nullptr: a threshold per list, tau_list[b * n_heads + h] (fixed-budget selection), instead of tau.
__global__ void __launch_bounds__(128)
mask_kernel(const float *__restrict__ scores, int64_t n_tokens, int n_heads,
            const int32_t *__restrict__ cu_seqlens, int n_seqs, float tau, int window, int window_keep,
            uint32_t *__restrict__ maskbits, int64_t n_words, const float *__restrict__ tau_list)
{
    // may be queued with early start behind the kernels that produce the per-list thresholds
    griddep_launch_dependents();
    griddep_wait();
    const int lane = threadIdx.x & 31;
    const int64_t word = static_cast<int64_t>(blockIdx.x) * 4 + (threadIdx.x >> 5);
    const int64_t t = word * 32 + lane;
    const bool valid = t < n_tokens;
    float s[kMaxHeads], tau_h[kMaxHeads];
#pragma unroll
    for (int h = 0; h < kMaxHeads; ++h) { s[h] = 0.0f; tau_h[h] = tau; }
    bool in_window = false;
    if (valid) {
        const float *src = scores + t * n_heads;
        if (n_heads == kMaxHeads) {
            const float4 a = __ldg(reinterpret_cast<const float4 *>(src));
            const float4 b = __ldg(reinterpret_cast<const float4 *>(src) + 1);
            s[0] = a.x; s[1] = a.y; s[2] = a.z; s[3] = a.w;
            s[4] = b.x; s[5] = b.y; s[6] = b.z; s[7] = b.w;
        } else {
#pragma unroll
            for (int h = 0; h < kMaxHeads; ++h)
                if (h < n_heads) s[h] = __ldg(src + h);
        }
        int64_t seq_end = n_tokens;
        int b = 0;
        if (cu_seqlens != nullptr && n_seqs > 1) {
            b = seq_of_token(cu_seqlens, n_seqs, t);
            seq_end = __ldg(cu_seqlens + b + 1);
        }
        in_window = t >= seq_end - static_cast<int64_t>(window);
        if (tau_list != nullptr) {
            // thresholds written by the kernel ahead in the stream: plain loads
#pragma unroll
            for (int h = 0; h < kMaxHeads; ++h)
                if (h < n_heads) tau_h[h] = __ldcg(tau_list + b * n_heads + h);
        }
    }
    uint32_t my_word = 0;
#pragma unroll
    for (int h = 0; h < kMaxHeads; ++h) {
        const bool keep = valid && (in_window ? window_keep != 0 : s[h] >= tau_h[h]);
        const uint32_t w = __ballot_sync(0xffffffffu, keep);
        if (lane == h) my_word = w;
    }
    if (lane < n_heads) maskbits[static_cast<int64_t>(lane) * n_words + word] = my_word;
}

// Number of kept tokens of head h among packed tokens [0, t), given the block prefix.
__device__ __forceinline__ int32_t kept_before(const uint32_t *__restrict__ maskbits, int64_t n_words,
                                               const int32_t *__restrict__ blockprefix, int64_t n_blocks, int h,
                                               int64_t t)
{
    const int64_t blk = t / kBlockTokens;
    int32_t n = blockprefix[static_cast<int64_t>(h) * (n_blocks + 1) + blk];
    if (blk < n_blocks) {
        const uint32_t *w = maskbits + static_cast<int64_t>(h) * n_words + blk * 4;
        const int r = static_cast<int>(t - blk * kBlockTokens);       // 0..127 bits of this block
        for (int i = 0; i < 4; ++i) {
            const int lo = i * 32;
            if (r >= lo + 32) n += __popc(__ldcg(w + i));
            else if (r > lo) n += __popc(__ldcg(w + i) & ((1u << (r - lo)) - 1u));
        }
    }
    return n;
}

// Where list idx (= b * n_heads + h) of a call lives in the caller's per-list arrays (lengths, page tables): at
// idx itself, or -- appending a batch of prompts to a cache, whose lists are ordered (sequence slot, layer, head) --
// at list_map[b] + h, list_map [n_seqs] naming the list of head 0 of each of the call's sequences.
__device__ __forceinline__ int64_t list_at(const int64_t *__restrict__ list_map, int idx, int n_heads)
{
    return list_map != nullptr ? __ldcg(list_map + idx / n_heads) + idx % n_heads : static_cast<int64_t>(idx);
}

// ---------------------------------------------------------------------------
// Page assignment of the paged output, by all NT threads of one CTA: list idx (= b * n_heads + h) needs
// ceil(lengths[idx] / page_tokens) pages (less those it owns already when appending); list_page0 receives the
// exclusive scan of the needs plus first_page, *n_pages_used the total; a pool or table that is too small
// sets the status word, marks every list with list_page0 = -1 and (append) restores the old lengths.
// fill_table != 0: the page numbers are also entered into page_table here; otherwise the caller does
// that (fill_page_table), e.g. spread over many CTAs.  Arguments as scan_lists.
template <int NT, int kKnown>
__device__ __forceinline__ void
assign_pages(int n_heads, int n_seqs, int32_t *__restrict__ lengths, int page_tokens, int32_t first_page,
             int64_t n_pages_pool, int max_pages, int32_t *__restrict__ list_page0, int32_t *__restrict__ page_table,
             int32_t *__restrict__ n_pages_used, int32_t *__restrict__ page_cursor, int32_t *__restrict__ status, int append,
             int32_t *__restrict__ list_base, const int32_t *__restrict__ free_stack, int32_t *__restrict__ free_top,
             int fill_table, const int64_t *__restrict__ list_map = nullptr)
{
    __shared__ int32_t warp_sums[32];
    __shared__ int32_t carry_s;
    __shared__ int32_t fail_s;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    auto block_scan = [&](int32_t v, int32_t &total) -> int32_t {   // inclusive scan over the CTA
        int32_t x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        __syncthreads();
        if (lane == 31) warp_sums[warp] = x;
        __syncthreads();
        if (warp == 0) {
            int32_t w = lane < NT / 32 ? warp_sums[lane] : 0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int32_t y = __shfl_up_sync(0xffffffffu, w, o);
                if (lane >= o) w += y;
            }
            warp_sums[lane] = w;
        }
        __syncthreads();
        total = warp_sums[31];
        return x + (warp > 0 ? warp_sums[warp - 1] : 0);
    };
    // paged output: exclusive scan of the per-list page counts in (b,h) order.  What a list's thread knows of it stays in
    // shared memory for the table (of the first kKnown lists; the others are looked up again).
    constexpr int kSlots = kKnown > 0 ? kKnown : 1;
    __shared__ int32_t s_page0[kSlots], s_have[kSlots], s_need[kSlots];
    __shared__ int64_t s_list[kSlots];
    int32_t n_free = 0;                                                 // asked for ahead of the scan
    if (page_cursor != nullptr && free_top != nullptr) n_free = __ldcg(free_top);
    __syncthreads();
    if (tid == 0) { carry_s = 0; fail_s = 0; }
    __syncthreads();
    const int n_lists = n_heads * n_seqs;
    for (int base = 0; base < n_lists; base += NT) {
        const int idx = base + tid;
        int32_t need = 0, have = 0;
        int64_t li = 0;
        if (idx < n_lists) {
            li = list_at(list_map, idx, n_heads);
            need = (__ldcg(lengths + li) + page_tokens - 1) / page_tokens;
            if (need > max_pages) fail_s = 1;
            if (append) have = (__ldcg(list_base + idx) + page_tokens - 1) / page_tokens;     // pages the list already owns
            need -= have;
        }
        int32_t total;
        const int32_t incl = block_scan(need, total);
        const int32_t carry = carry_s;
        if (idx < n_lists) {
            list_page0[idx] = first_page + carry + incl - need;
            if (idx < kKnown) {
                s_page0[idx] = first_page + carry + incl - need;
                s_have[idx] = have;
                s_need[idx] = need;
                s_list[idx] = li;
            }
        }
        __syncthreads();
        if (tid == 0) carry_s = carry + total;
        __syncthreads();
    }
    const int32_t used = carry_s;
    if (n_free < 0) n_free = 0;
    const int32_t from_stack = used < n_free ? used : n_free;
    // a cache (page_cursor): what comes from the stack, or an append that needs no page, fits wherever the cursor stands
    const bool fits = static_cast<int64_t>(first_page) + (used - from_stack) <= n_pages_pool ||
                      (page_cursor != nullptr && used == from_stack);
    const bool fail = fail_s != 0 || !fits;
    if (fail) {
        for (int idx = tid; idx < n_lists; idx += NT) {
            list_page0[idx] = -1;
            if (append) lengths[list_at(list_map, idx, n_heads)] = __ldcg(list_base + idx);
        }
        if (tid == 0) {
            atomicCAS(status, 0, 4 /* KVZAP_ERR_OOM_PAGES */);
            if (n_pages_used != nullptr) *n_pages_used = 0;
        }
        return;
    }
    __syncthreads();      // every thread has read the cursor and the stack height
    if (tid == 0) {
        if (n_pages_used != nullptr) *n_pages_used = used;
        if (page_cursor != nullptr) *page_cursor = first_page + used - from_stack;
        if (from_stack > 0) *free_top = n_free - from_stack;
    }
    __syncthreads();      // list_page0 and lengths of all lists are final
    if (!fill_table) return;
    for (int idx = warp; idx < n_lists; idx += NT / 32) {            // a warp per list
        int32_t p0, have, need;
        int64_t li;
        if (idx < kKnown) {
            p0 = s_page0[idx];
            have = s_have[idx];
            need = s_need[idx];
            li = s_list[idx];
        } else {
            p0 = list_page0[idx];
            have = append ? (__ldcg(list_base + idx) + page_tokens - 1) / page_tokens : 0;
            li = list_at(list_map, idx, n_heads);
            need = (__ldcg(lengths + li) + page_tokens - 1) / page_tokens - have;
        }
        for (int32_t i = lane; i < need; i += 32) {
            const int32_t j = p0 - first_page + i;            // ordinal among the pages assigned by this call
            page_table[li * max_pages + have + i] =
                j < from_stack ? __ldcg(free_stack + n_free - 1 - j) : first_page + (j - from_stack);
        }
    }
}



// ---------------------------------------------------------------------------
// One CTA of NT threads (all of them call it).  blockprefix [H][n_blocks+1], seqbase [H][n_seqs+1] (both nullptr when only the
// lengths and the page assignment are wanted: the lists are then counted directly), lengths [n_seqs][H].
// Paged output (page_tokens > 0): list (b,h) gets
// ceil(len/page_tokens) pages numbered contiguously from first_page in (b,h)
// order; list_page0 [n_seqs*H] receives each list's first page and page_table
// [n_seqs*H][max_pages] its page numbers; *n_pages_used the total.  A pool or
// table that is too small sets the status word and marks every list with
// list_page0 = -1 so that the compaction writes nothing.
// append != 0 (paged only): the lists already hold lengths[] rows in the pages their tables name; the
// kept rows are added behind them.  lengths becomes old + kept (unchanged on failure), only the pages
// beyond the old ones are assigned and entered into the table, and list_base receives the old length.
// With a cursor (a cache's allocator) the new pages are taken from the stack of released pages first
// (free_stack / free_top, may be nullptr), then from the cursor: the pages of a list are then not
// consecutive numbers and the compaction finds them through the table; list_page0 is the ordinal of
// the list's first new page among the pages this call assigns (plus first_page), or -1.
template <int NT>
__device__ __forceinline__ void
scan_lists(const uint32_t *__restrict__ maskbits, int64_t n_words, int64_t n_blocks, int n_heads,
            const int32_t *__restrict__ cu_seqlens, int n_seqs, int64_t n_tokens,
            int32_t *__restrict__ blockprefix, int32_t *__restrict__ seqbase, int32_t *__restrict__ lengths,
            int page_tokens, int32_t first_page, int64_t n_pages_pool, int max_pages,
            int32_t *__restrict__ list_page0, int32_t *__restrict__ page_table, int32_t *__restrict__ n_pages_used,
            int32_t *__restrict__ page_cursor, int32_t *__restrict__ status, int append,
            int32_t *__restrict__ list_base, const int32_t *__restrict__ free_stack, int32_t *__restrict__ free_top,
            const int64_t *__restrict__ list_map = nullptr)
{
    // page_cursor != nullptr: the first page comes from (and the pages used are added to) a device-side
    // allocator cursor instead of the first_page argument
    if (page_tokens > 0 && page_cursor != nullptr) first_page = *page_cursor;
    __shared__ int32_t warp_sums[32];
    __shared__ int32_t carry_s;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    auto block_scan = [&](int32_t v, int32_t &total) -> int32_t {   // inclusive scan over the CTA
        int32_t x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        __syncthreads();
        if (lane == 31) warp_sums[warp] = x;
        __syncthreads();
        if (warp == 0) {
            int32_t w = lane < NT / 32 ? warp_sums[lane] : 0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int32_t y = __shfl_up_sync(0xffffffffu, w, o);
                if (lane >= o) w += y;
            }
            warp_sums[lane] = w;
        }
        __syncthreads();
        total = warp_sums[31];
        return x + (warp > 0 ? warp_sums[warp - 1] : 0);
    };

    if (blockprefix == nullptr) {
        // Only the lengths are wanted (the compaction counts its own prefixes): every list's kept rows are
        // counted straight from the mask words of its token range, a group of threads per list.
        const int n_lists_all = n_heads * n_seqs;
        int per_list = NT;
        while (per_list > 32 && NT / per_list < n_lists_all) per_list >>= 1;
        const int n_groups = NT / per_list, grp = tid / per_list, gt = tid % per_list;
        __shared__ int32_t group_sum[32];
        for (int idx0 = 0; idx0 < n_lists_all; idx0 += n_groups) {
            if (tid < 32) group_sum[tid] = 0;
            __syncthreads();
            const int idx = idx0 + grp;
            int32_t cnt = 0;
            if (idx < n_lists_all) {
                const int b = idx / n_heads, h = idx % n_heads;
                const int64_t t_lo = cu_seqlens != nullptr ? static_cast<int64_t>(cu_seqlens[b]) : 0;
                const int64_t t_hi = cu_seqlens != nullptr ? static_cast<int64_t>(cu_seqlens[b + 1]) : n_tokens;
                const uint32_t *wh = maskbits + static_cast<int64_t>(h) * n_words;
                for (int64_t wi = t_lo / 32 + gt; wi * 32 < t_hi; wi += per_list) {
                    uint32_t w = __ldcg(wh + wi);
                    if (wi * 32 < t_lo) w &= ~0u << static_cast<int>(t_lo - wi * 32);               // bits below the sequence
                    if (wi * 32 + 32 > t_hi) w &= (1u << static_cast<int>(t_hi - wi * 32)) - 1u;    // bits above it
                    cnt += __popc(w);
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
            if (lane == 0 && cnt) atomicAdd(&group_sum[grp], cnt);
            __syncthreads();
            if (gt == 0 && idx < n_lists_all) {
                const int64_t li = list_at(list_map, idx, n_heads);
                const int32_t old = append ? lengths[li] : 0;
                if (append) list_base[idx] = old;
                lengths[li] = old + group_sum[grp];
            }
            __syncthreads();
        }
    } else {
    for (int h = 0; h < n_heads; ++h) {
        if (tid == 0) carry_s = 0;
        __syncthreads();
        for (int64_t base = 0; base < n_blocks; base += NT) {
            const int64_t blk = base + tid;
            int32_t cnt = 0;
            if (blk < n_blocks) {
                const uint4 w = __ldcg(reinterpret_cast<const uint4 *>(maskbits + static_cast<int64_t>(h) * n_words + blk * 4));
                cnt = __popc(w.x) + __popc(w.y) + __popc(w.z) + __popc(w.w);
            }
            int32_t total;
            const int32_t incl = block_scan(cnt, total);
            const int32_t carry = carry_s;
            if (blk < n_blocks) blockprefix[static_cast<int64_t>(h) * (n_blocks + 1) + blk] = carry + incl - cnt;
            __syncthreads();
            if (tid == 0) carry_s = carry + total;
            __syncthreads();
        }
        if (tid == 0) blockprefix[static_cast<int64_t>(h) * (n_blocks + 1) + n_blocks] = carry_s;
    }
    __syncthreads();      // blockprefix written by this CTA is visible to it from here on

    for (int idx = tid; idx < n_heads * (n_seqs + 1); idx += NT) {
        const int h = idx / (n_seqs + 1), b = idx % (n_seqs + 1);
        const int64_t t = cu_seqlens != nullptr ? static_cast<int64_t>(cu_seqlens[b]) : (b == 0 ? 0 : n_tokens);
        seqbase[idx] = kept_before(maskbits, n_words, blockprefix, n_blocks, h, t);
    }
    __syncthreads();
    for (int idx = tid; idx < n_heads * n_seqs; idx += NT) {
        const int b = idx / n_heads, h = idx % n_heads;
        const int64_t li = list_at(list_map, idx, n_heads);
        const int32_t old = append ? lengths[li] : 0;
        if (append) list_base[idx] = old;
        lengths[li] = old + seqbase[h * (n_seqs + 1) + b + 1] - seqbase[h * (n_seqs + 1) + b];
    }
    }
    if (page_tokens <= 0) return;
    __syncthreads();
    assign_pages<NT, 128>(n_heads, n_seqs, lengths, page_tokens, first_page, n_pages_pool, max_pages, list_page0, page_table,
                     n_pages_used, page_cursor, status, append, list_base, free_stack, free_top, 1, list_map);
}

// The page assignment as a kernel of its own: one CTA of 1024 threads (behind the fused scoring kernels
// and for appending to a cache's lists).
__global__ void __launch_bounds__(1024)
scan_kernel(const uint32_t *__restrict__ maskbits, int64_t n_words, int64_t n_blocks, int n_heads,
            const int32_t *__restrict__ cu_seqlens, int n_seqs, int64_t n_tokens,
            int32_t *__restrict__ blockprefix, int32_t *__restrict__ seqbase, int32_t *__restrict__ lengths,
            int page_tokens, int32_t first_page, int64_t n_pages_pool, int max_pages,
            int32_t *__restrict__ list_page0, int32_t *__restrict__ page_table, int32_t *__restrict__ n_pages_used,
            int32_t *__restrict__ page_cursor, int32_t *__restrict__ status, int append,
            int32_t *__restrict__ list_base, const int32_t *__restrict__ free_stack, int32_t *__restrict__ free_top,
            const int64_t *__restrict__ list_map)
{
    // may be placed before the kernel that writes the mask has finished; waits for it here
    griddep_launch_dependents();
    griddep_wait();
    scan_lists<1024>(maskbits, n_words, n_blocks, n_heads, cu_seqlens, n_seqs, n_tokens, blockprefix, seqbase, lengths,
                     page_tokens, first_page, n_pages_pool, max_pages, list_page0, page_table, n_pages_used, page_cursor,
                     status, append, list_base, free_stack, free_top, list_map);
}

// ---------------------------------------------------------------------------
// One CTA per (128-token block, head).  Rows are row_bytes = 2*D bytes, moved
// as 16-byte units by 16-lane groups; up to kRowsInFlight rows of K and of V
// are loaded before any is stored.
constexpr int kCompactThreads = 256;
constexpr int kRowsInFlight = 4;

template <bool kPaged>
__global__ void __launch_bounds__(kCompactThreads)
compact_kernel(const uint4 *__restrict__ K, const uint4 *__restrict__ V, uint4 *__restrict__ K_out,
               uint4 *__restrict__ V_out, const uint32_t *__restrict__ maskbits, int64_t n_words, int64_t n_blocks,
               const int32_t *__restrict__ blockprefix, const int32_t *__restrict__ seqbase,
               const int32_t *__restrict__ cu_seqlens, int n_seqs, int64_t n_tokens, int n_heads, int row_units,
               int page_tokens, const int32_t *__restrict__ list_page0)
{
    __shared__ int32_t src_tok[kBlockTokens];     // packed token index of the i-th kept row of this block
    __shared__ int64_t dst_row[kBlockTokens];     // its destination row (dense: within head h; paged: pool row)
    const int64_t blk = blockIdx.x;
    const int h = blockIdx.y;
    const int tid = threadIdx.x;
    const uint32_t *words = maskbits + static_cast<int64_t>(h) * n_words + blk * 4;
    const uint32_t w0 = words[0], w1 = words[1], w2 = words[2], w3 = words[3];
    const int cnt = __popc(w0) + __popc(w1) + __popc(w2) + __popc(w3);
    if (cnt == 0) return;
    if (tid < kBlockTokens) {
        const int wi = tid >> 5, bit = tid & 31;
        const uint32_t w = wi == 0 ? w0 : wi == 1 ? w1 : wi == 2 ? w2 : w3;
        if ((w >> bit) & 1u) {
            int r = __popc(w & ((1u << bit) - 1u));
            if (wi > 0) r += __popc(w0);
            if (wi > 1) r += __popc(w1);
            if (wi > 2) r += __popc(w2);
            const int64_t t = blk * kBlockTokens + tid;
            const int32_t before = blockprefix[static_cast<int64_t>(h) * (n_blocks + 1) + blk] + r;
            int b = 0;
            int64_t seq_start = 0;
            if (cu_seqlens != nullptr && n_seqs > 1) {
                b = seq_of_token(cu_seqlens, n_seqs, t);
                seq_start = cu_seqlens[b];
            }
            const int64_t n = before - seqbase[h * (n_seqs + 1) + b];     // rank inside list (b,h)
            int64_t dst;
            if constexpr (kPaged) {
                const int32_t p0 = list_page0[b * n_heads + h];
                dst = p0 < 0 ? -1 : static_cast<int64_t>(p0) * page_tokens + n;                 // pages in a row
            } else {
                dst = static_cast<int64_t>(h) * n_tokens + seq_start + n;
            }
            src_tok[r] = static_cast<int32_t>(t - blk * kBlockTokens);
            dst_row[r] = dst;
        }
    }
    __syncthreads();

    const int group = tid >> 4, gl = tid & 15;            // 16 groups of 16 lanes
    constexpr int kGroups = kCompactThreads / 16;
    const int64_t head_row0 = static_cast<int64_t>(h) * n_tokens + blk * kBlockTokens;
    for (int i0 = group; i0 < cnt; i0 += kGroups * kRowsInFlight) {
        for (int u0 = gl; u0 < row_units; u0 += 16) {
            uint4 kv[kRowsInFlight], vv[kRowsInFlight];
#pragma unroll
            for (int j = 0; j < kRowsInFlight; ++j) {
                const int i = i0 + j * kGroups;
                if (i < cnt) {
                    const int64_t src = (head_row0 + src_tok[i]) * row_units + u0;
                    kv[j] = __ldg(K + src);
                    vv[j] = __ldg(V + src);
                }
            }
#pragma unroll
            for (int j = 0; j < kRowsInFlight; ++j) {
                const int i = i0 + j * kGroups;
                if (i < cnt) {
                    const int64_t d = dst_row[i];
                    if (d >= 0) {
                        K_out[d * row_units + u0] = kv[j];
                        V_out[d * row_units + u0] = vv[j];
                    }
                }
            }
        }
    }
}

// ---------------------------------------------------------------------------
// Dense-ragged compaction without a separate scan pass.  Grid (chunks, H): a CTA owns
// `blocks_per_cta` consecutive 128-token blocks of one head.  It first counts, straight from the
// mask words, the rows kept before its first block (and before the start of the sequence that is
// in progress there), then walks its blocks keeping a running count, so that every kept row's
// slot in its (sequence, head) list is known without any other CTA's help.  lengths[b,h] is
// written by the thread that handles the last token of sequence b; empty sequences by chunk 0.
constexpr int kDenseThreads = 128;     // = kBlockTokens: one thread ranks one token; small enough to sit beside a scoring CTA
constexpr int kDenseThreadsShort = 256; // short inputs (one block per CTA): twice the rows in flight, one round of row loads

// bits of the block's four words below in-block position r (0..128)
__device__ __forceinline__ int popc_below(uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3, int r)
{
    int n = 0;
    const uint32_t w[4] = {w0, w1, w2, w3};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int lo = i * 32;
        if (r >= lo + 32) n += __popc(w[i]);
        else if (r > lo) n += __popc(w[i] & ((1u << (r - lo)) - 1u));
    }
    return n;
}

// Paged output of a short input: every CTA counts all lists from the mask words and works out all first pages itself,
// instead of a launch of one CTA ahead of the compaction (777 tokens: 8.6 -> 5.5 us from the end of the scoring launch to
// the end of the compaction).  On contexts that trust their producers, where the compaction runs beside the next scoring; elsewhere
// compact_short_kernel.  The counting is H * n_words words per CTA, hence the limits: at 8192 tokens x 8 heads it
// takes the 256 threads 8 loads each.
struct PageAssign {
    int32_t enabled;
    int32_t first_page, max_pages;
    int64_t n_pages_pool;
    int32_t *page_table, *n_pages_used, *status;
};
constexpr int kAssignLists = 256;
constexpr int64_t kAssignWords = 2048;

template <int kThreads>
__device__ __forceinline__ void
assign_pages_locally(const PageAssign &a, const uint32_t *__restrict__ maskbits, int64_t n_words, const int32_t *__restrict__ cu_seqlens,
                     int n_seqs, int64_t n_tokens, int n_heads, int page_tokens, int32_t *__restrict__ lengths, int32_t *s_page0)
{
    __shared__ int32_t s_len[kAssignLists];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n_lists = n_heads * n_seqs;
    const bool multi = cu_seqlens != nullptr && n_seqs > 1;
    for (int i = tid; i < n_lists; i += kThreads) s_len[i] = 0;
    __syncthreads();
    const int total_words = static_cast<int>(n_words) * n_heads;
    for (int i = tid; i < total_words; i += kThreads) {
        uint32_t w = __ldcg(maskbits + i);
        const int h = i / static_cast<int>(n_words), t0 = (i - h * static_cast<int>(n_words)) * 32;
        if (w == 0u) continue;
        if (!multi) {
            atomicAdd(&s_len[h], __popc(w));
            continue;
        }
        int b = seq_of_token(cu_seqlens, n_seqs, t0);
        while (w != 0u) {                                     // the sequences that the word's tokens belong to
            const int end = cu_seqlens[b + 1] - t0;           // bits below it are sequence b's
            const uint32_t mine = end >= 32 ? w : end <= 0 ? 0u : w & ((1u << end) - 1u);
            if (mine) atomicAdd(&s_len[b * n_heads + h], __popc(mine));
            w &= ~mine;
            ++b;
        }
    }
    __syncthreads();
    if (warp == 0) {
        int32_t carry = 0;
        bool fail = false;
        for (int base = 0; base < n_lists; base += 32) {
            const int idx = base + lane;
            const int32_t need = idx < n_lists ? (s_len[idx] + page_tokens - 1) / page_tokens : 0;
            fail = fail || need > a.max_pages;
            int32_t incl = need;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int32_t y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            if (idx < n_lists) s_page0[idx] = a.first_page + carry + incl - need;
            carry += __shfl_sync(0xffffffffu, incl, 31);
        }
        fail = __any_sync(0xffffffffu, fail) || static_cast<int64_t>(a.first_page) + carry > a.n_pages_pool;
        const bool first_cta = blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0;
        if (fail) {
            for (int idx = lane; idx < n_lists; idx += 32) s_page0[idx] = -1;
            if (first_cta && lane == 0) atomicCAS(a.status, 0, 4 /* KVZAP_ERR_OOM_PAGES */);
        }
        if (first_cta) {
            if (lane == 0 && a.n_pages_used != nullptr) *a.n_pages_used = fail ? 0 : carry;
            for (int idx = lane; idx < n_lists; idx += 32) lengths[idx] = s_len[idx];
        }
    }
    __syncthreads();
    if (blockIdx.x == 0 && blockIdx.z == 0)                   // the tables of this CTA's head, a warp per list
        for (int b = warp; b < n_seqs; b += kThreads / 32) {
            const int idx = b * n_heads + blockIdx.y;
            const int32_t p0 = s_page0[idx];
            const int32_t need = p0 < 0 ? 0 : (s_len[idx] + page_tokens - 1) / page_tokens;
            for (int32_t i = lane; i < need; i += 32) a.page_table[static_cast<int64_t>(idx) * a.max_pages + i] = p0 + i;
        }
}

// kThreads = 128, or 256 for short inputs (one block per CTA: all kept rows of the block in flight at once).
// At most 64 registers per thread (eight 128-thread CTAs per SM by registers): two of these CTAs then fit into the
// register-file quarters that the MLP scoring kernel's ten warps leave free, so the compaction of layer
// l runs beside the scoring of layer l + 1 at full width; at 72 registers only one fits and the layer
// period of the fused path grows by ~10 us.
// kAlone: the launch that runs beside nothing (a context that does not trust its producers: the scoring behind it waits
// for it); see launch_compaction.  It assigns no pages: the inputs short enough for that take compact_short_kernel.  gridDim.z CTAs share the kept rows of a block.
template <int kThreads, bool kAlone>
__global__ void __launch_bounds__(kThreads, 1024 / kThreads)
compact_dense_kernel(const uint4 *__restrict__ K, const uint4 *__restrict__ V, uint4 *__restrict__ K_out,
                     uint4 *__restrict__ V_out, const uint32_t *__restrict__ maskbits, int64_t n_words,
                     int64_t n_blocks, int blocks_per_cta, const int32_t *__restrict__ cu_seqlens, int n_seqs,
                     int64_t n_tokens, int n_heads, int row_units, int32_t *__restrict__ lengths, int page_tokens,
                     const int32_t *__restrict__ list_page0, int64_t in_stride_h, int64_t in_stride_t,
                     const int32_t *__restrict__ list_base, const int32_t *__restrict__ page_table, int max_pages,
                     const int64_t *__restrict__ list_map, const PageAssign assign)
{
    // list_base != nullptr (paged): list (b,h) already holds list_base[] rows; kept rows go behind them,
    // into the pages that page_table [list][max_pages] names (the scan has entered the new ones); the table
    // of list (b,h) is row b * H + h of page_table, or row list_map[b] + h (see list_at).
    // Row (h, t) of the inputs starts at row index h * in_stride_h + t * in_stride_t: (n_tokens, 1) for
    // the head-major cache layout [H][T][D], (1, H) for the K/V projection's own output [T][H][D].
    // page_tokens > 0: paged output.  K_out / V_out are the page pools, list (b,h) starts at page
    // list_page0[b * H + h] (-1 = nothing may be written), and lengths come from the scan kernel.
    const bool paged = page_tokens > 0;
    __shared__ int32_t src_tok[kBlockTokens];
    __shared__ int64_t dst_row[kBlockTokens];
    __shared__ int32_t red[2][kThreads / 32];
    __shared__ int32_t base_next_s;
    __shared__ int32_t s_page0[kAlone ? 1 : kAssignLists];
    const int h = blockIdx.y;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t blk0 = static_cast<int64_t>(blockIdx.x) * blocks_per_cta;
    const int64_t blk1 = blk0 + blocks_per_cta < n_blocks ? blk0 + blocks_per_cta : n_blocks;
    const bool multi = cu_seqlens != nullptr && n_seqs > 1;
    const uint32_t *words = maskbits + static_cast<int64_t>(h) * n_words;

    // This grid is small enough to be resident all at once: the next kernel in the stream may be
    // placed as soon as it is; the mask itself is read only after the kernel ahead has completed.
    griddep_launch_dependents();
    griddep_wait();

    const int z = blockIdx.z, nz = gridDim.z;
    if (blockIdx.x == 0 && z == 0 && cu_seqlens != nullptr && !paged)   // empty sequences have no last token to write for them
        for (int b = tid; b < n_seqs; b += kThreads)
            if (cu_seqlens[b + 1] == cu_seqlens[b]) lengths[b * n_heads + h] = 0;
    const bool assigned = !kAlone && assign.enabled;
    if constexpr (!kAlone)
        if (assigned) assign_pages_locally<kThreads>(assign, maskbits, n_words, cu_seqlens, n_seqs, n_tokens, n_heads, page_tokens, lengths, s_page0);
    if (blk0 >= n_blocks) return;

    // rows kept before this CTA's first token, and before the start of the sequence in progress there
    const int64_t t0 = blk0 * kBlockTokens;
    int64_t s0 = 0;
    if (multi) s0 = cu_seqlens[seq_of_token(cu_seqlens, n_seqs, t0)];
    int32_t total = 0, before_s0 = 0;
    // the first block's own words are fetched together with the words before it (one round trip, not two)
    uint4 wv_next = __ldcg(reinterpret_cast<const uint4 *>(words + blk0 * 4));
    for (int64_t i = tid; i < blk0 * 4; i += kThreads) {
        const uint32_t w = __ldcg(words + i);     // not a read-only-data load: it must stay behind griddep_wait()
        const int c = __popc(w);
        total += c;
        const int64_t lo = i * 32;
        if (lo + 32 <= s0) before_s0 += c;
        else if (lo < s0) before_s0 += __popc(w & ((1u << static_cast<int>(s0 - lo)) - 1u));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        total += __shfl_xor_sync(0xffffffffu, total, o);
        before_s0 += __shfl_xor_sync(0xffffffffu, before_s0, o);
    }
    if (lane == 0) { red[0][warp] = total; red[1][warp] = before_s0; }
    __syncthreads();
    int32_t running = 0, base_cur = 0;       // kept before the current block / before the sequence in progress at its start
#pragma unroll
    for (int i = 0; i < kThreads / 32; ++i) { running += red[0][i]; base_cur += red[1][i]; }

    const int group = tid >> 4, gl = tid & 15;
    constexpr int kGroups = kThreads / 16;
    for (int64_t blk = blk0; blk < blk1; ++blk) {
        const uint4 wv = wv_next;
        if (blk + 1 < blk1) wv_next = __ldcg(reinterpret_cast<const uint4 *>(words + (blk + 1) * 4));
        const uint32_t w0 = wv.x, w1 = wv.y, w2 = wv.z, w3 = wv.w;
        const int cnt = __popc(w0) + __popc(w1) + __popc(w2) + __popc(w3);
        const int64_t blk_start = blk * kBlockTokens;
        if (tid < kBlockTokens) {
            const int64_t t = blk_start + tid;
            if (t < n_tokens) {
                int b = 0;
                int64_t s = 0, e = n_tokens;
                if (multi) {
                    b = seq_of_token(cu_seqlens, n_seqs, t);
                    s = cu_seqlens[b];
                    e = cu_seqlens[b + 1];
                }
                // kept rows before the start of this token's sequence
                const int32_t base = s >= blk_start ? running + popc_below(w0, w1, w2, w3, static_cast<int>(s - blk_start))
                                                    : base_cur;
                const int r = popc_below(w0, w1, w2, w3, tid);
                const uint32_t w = tid < 32 ? w0 : tid < 64 ? w1 : tid < 96 ? w2 : w3;
                const bool keep = (w >> (tid & 31)) & 1u;
                if (keep) {
                    src_tok[r] = tid;
                    const int64_t n = running + r - base;                  // rank inside list (b,h)
                    if (paged) {
                        const int32_t p0 = assigned ? s_page0[b * n_heads + h] : __ldcg(list_page0 + b * n_heads + h);
                        if (list_base == nullptr) {
                            dst_row[r] = p0 < 0 ? -1 : static_cast<int64_t>(p0) * page_tokens + n;      // pages in a row
                        } else {
                            const uint32_t nn = static_cast<uint32_t>(__ldcg(list_base + b * n_heads + h) + static_cast<int32_t>(n));
                            const uint32_t pi = nn / static_cast<uint32_t>(page_tokens);
                            if (p0 < 0) {
                                dst_row[r] = -1;
                            } else {
                                const int64_t trow = list_map != nullptr ? __ldcg(list_map + b) + h : static_cast<int64_t>(b * n_heads + h);
                                const int64_t page = __ldcg(page_table + trow * max_pages + pi);
                                dst_row[r] = page * page_tokens + (nn - pi * static_cast<uint32_t>(page_tokens));
                            }
                        }
                    } else {
                        dst_row[r] = static_cast<int64_t>(h) * n_tokens + s + n;
                    }
                }
                if (t + 1 == e && !paged && z == 0) lengths[b * n_heads + h] = running + r + (keep ? 1 : 0) - base;
                if (tid == kBlockTokens - 1 || t + 1 == n_tokens) {
                    // base of the sequence in progress at the next block's first token
                    int32_t nb = base;
                    if (multi && t + 1 == e) nb = running + cnt;      // a new sequence starts exactly there
                    base_next_s = nb;
                }
            }
        }
        __syncthreads();
        const int64_t head_row0 = static_cast<int64_t>(h) * in_stride_h + blk_start * in_stride_t;
        for (int i0 = group + z * kGroups; i0 < cnt; i0 += nz * kGroups * kRowsInFlight) {
            for (int u0 = gl; u0 < row_units; u0 += 16) {
                uint4 kv[kRowsInFlight], vv[kRowsInFlight];
#pragma unroll
                for (int j = 0; j < kRowsInFlight; ++j) {
                    const int i = i0 + j * nz * kGroups;
                    if (i < cnt) {
                        const int64_t src = (head_row0 + src_tok[i] * in_stride_t) * row_units + u0;
                        kv[j] = __ldg(K + src);
                        vv[j] = __ldg(V + src);
                    }
                }
#pragma unroll
                for (int j = 0; j < kRowsInFlight; ++j) {
                    const int i = i0 + j * nz * kGroups;
                    if (i < cnt && dst_row[i] >= 0) {
                        const int64_t d = dst_row[i] * row_units + u0;
                        K_out[d] = kv[j];
                        V_out[d] = vv[j];
                    }
                }
            }
        }
        running += cnt;
        base_cur = base_next_s;
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// The compaction of a short input (mask words and lists as for assign_pages_locally) that runs beside nothing: behind the scoring of
// a default context, or of a chunk.  There the launch is a chain of round trips, and this kernel has as few as there are: mask words,
// sequence offsets, old lengths and the page cursor together; then the rows' loads, for which a CTA needs only its own block's
// words, go out before the lists are counted and pages found; then the stores.  Grid (blocks + n_books, H, z): z CTAs share the rows
// of a block, and the last x do the bookkeeping of a head's lists (lengths, tables, for a chunk also the ring's scores), which no
// row waits for.  A chunk has one of them to as many sequences as a CTA has warps: with one for all, 256 sequences of 200 tokens, one head,
// took 181 us in two chunks, 130 with the launches that this one replaces, now 101.  An append finds the pages of new rows itself, from the cursor and the stack as the launch ahead left them (`taken`).
// Scoring and this, us a call of several layers: 8 x 777 tokens into pages 146.6 -> 136.4, 4 x 5 x 300 93.3 -> 82.1, 4 x 3000 118.6 -> 110.6, dense
// 4 x 777 67.5 -> 63.5; 5120 -> 640 -> 8, 4 x 2000 dense 90.3 -> 86.0.  Chunks, whose launch ahead had spent 7 us on counting and a one-CTA page
// assignment behind the scoring: four prompts in two chunks of 500 tokens, 4 layers, 274.3 -> 224.3, eight of 64 in three 304.9 -> 268.7.
// Two rows in flight per lane group and four CTAs to a block rather than four rows and two CTAs (3000 tokens 110.5 and 117.4).
struct ShortCompact {
    const uint4 *K, *V;
    uint4 *K_out, *V_out;
    const uint32_t *maskbits;         // [H][n_words]
    const int32_t *cu_seqlens;
    int32_t *lengths;                 // [n_lists]; append: of all lists of the cache
    int64_t n_tokens, in_stride_h, in_stride_t;
    int32_t n_words, n_blocks, n_seqs, n_heads, row_units;
    int32_t n_books;                  // bookkeeping CTAs per head
    int32_t page_tokens;              // 0: dense-ragged output
    int32_t page_shift;               // its logarithm, or -1: a division takes some 150 cycles of a chain
    int32_t first_page, max_pages;
    int64_t n_pages_pool;
    int32_t *page_table, *n_pages_used, *status;
    // append (list_base != nullptr)
    const int32_t *list_base;         // [n_lists] rows that a list holds now
    const int64_t *list_map;          // [n_seqs] list of head 0 of each sequence
    int32_t *page_cursor;
    const int32_t *free_stack;
    int32_t *free_top;
    const int32_t *taken;             // page cursor and height of the stack, as copied by the launch ahead
    // the ring's scores: those of the last min(length, window) tokens of each sequence
    const float *scores;
    float *score_ring;
    const int32_t *n_tokens_list;     // tokens of each list, these included
    int32_t window;
    // keep bits from given scores (kFromScores): threshold, or one per list, and the order with the launches around this one
    // as in PruneParams; `scores` as above
    float tau;
    const float *tau_list;
    int32_t wait_first;
    uint4 *clear;
    int64_t clear_units;
};
constexpr int kShortRows = 2;         // rows of K and of V in flight per lane group
__host__ inline bool short_input(int64_t n_words, int n_heads, int64_t n_seqs)
{
    return n_words * n_heads <= kAssignWords && n_seqs * n_heads <= kAssignLists;
}

// seq_of_token over offsets in shared memory
__device__ __forceinline__ int seq_of_shared(const int32_t *cu, int n_seqs, int32_t t)
{
    int lo = 0, hi = n_seqs;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (cu[mid] <= t) lo = mid; else hi = mid;
    }
    return lo;
}

enum ShortKind { kShortDense, kShortPaged, kShortAppend };
// Where the keep bits come from: mask words, or given scores (the pruning calls).  Then every CTA makes the words that it needs
// itself: dense, those of its head up to its block; paged, all of them, a token of all heads per load.
// In place of prune_onepass_kernel, whose CTAs look sequences up in memory one after the other, and whose paged form meets at an arrival
// counter, a page assignment and a flag; us a call: 3 x 500 tokens 8.6 -> 5.8, 800 7.4 -> 4.1, 2200 10.3 -> 5.2, 4000 10.2 -> 7.3; paged 300 12.1 -> 5.0,
// 2 x 450 14.9 -> 8.8, 1500 13.4 -> 11.0.  Up to which sizes: short_prune.
enum ShortSource { kFromWords, kFromScores };
template <ShortKind kKind, ShortSource kFrom>
__global__ void __launch_bounds__(kDenseThreadsShort, 4)
compact_short_kernel(const ShortCompact a)
{
    constexpr int kThreads = kDenseThreadsShort, kWarps = kThreads / 32;
    constexpr bool kPages = kKind != kShortDense, kAppend = kKind == kShortAppend;
    __shared__ uint32_t s_words[kAssignWords];        // dense: of this CTA's head, else of all heads
    __shared__ int32_t s_cu[kAssignLists + 1], s_len[kAssignLists], s_base[kPages ? kAssignLists : 1], s_page0[kPages ? kAssignLists : 1];
    __shared__ int64_t s_list[kPages ? kAssignLists : 1];      // [n_seqs] this head's lists among those of the table
    __shared__ int32_t s_last[kAppend ? kAssignLists : 1];     // [n_seqs] ... the pages that they end in now
    __shared__ float s_tau[kFrom == kFromScores && !kPages ? kAssignLists : 1];
    __shared__ int32_t src_tok[kBlockTokens];
    __shared__ int64_t dst_row[kBlockTokens];
    __shared__ int32_t running_s, before_s, cursor_s, free_s, stack_s;
    const int h = blockIdx.y, H = a.n_heads, z = blockIdx.z, nz = gridDim.z;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int blk = blockIdx.x;
    const bool books = blk >= a.n_blocks;
    if constexpr (kFrom == kFromWords) {
        griddep_launch_dependents();
        griddep_wait();
    } else {
        if (a.wait_first < 2) griddep_launch_dependents();
        if (a.wait_first > 0) {
            griddep_wait();
            if (a.wait_first == 2) griddep_launch_dependents();
        }
    }
    if (books && z != 0) return;

    const int n_lists = a.n_seqs * H, n_words = a.n_words;
    const bool multi = a.cu_seqlens != nullptr && a.n_seqs > 1;
    {
        // all loads before the first store: one round trip
        constexpr int kWordsEach = kAssignWords / kThreads;
        const int total = kPages ? n_words * H : n_words;
        const uint32_t *words = a.maskbits + (kPages ? 0 : static_cast<int64_t>(h) * n_words);
        uint32_t w[kWordsEach];
        constexpr int kScoresEach = kPages ? 4 : 8;               // tokens per thread whose scores are loaded together
        constexpr int kHeadsEach = kPages ? kMaxHeads : 1;
        float sc[kFrom == kFromWords ? 1 : kScoresEach][kHeadsEach];
        // tokens whose scores this CTA needs
        const int32_t n_scores = kPages || books || (blk + 1) * kBlockTokens > a.n_tokens ? static_cast<int32_t>(a.n_tokens) : (blk + 1) * kBlockTokens;
        if constexpr (kFrom == kFromWords) {
#pragma unroll
            for (int k = 0; k < kWordsEach; ++k) w[k] = tid + k * kThreads < total ? __ldcg(words + tid + k * kThreads) : 0u;
        }
        auto load_scores = [&](int32_t t0) {
#pragma unroll
            for (int k = 0; k < kScoresEach; ++k) {
                const int32_t t = t0 + tid + k * kThreads;
                const float *src = a.scores + static_cast<int64_t>(t) * H;
                if constexpr (kPages) {
                    if (H == kMaxHeads && t < n_scores) {
                        const float4 x = __ldcg(reinterpret_cast<const float4 *>(src)), y = __ldcg(reinterpret_cast<const float4 *>(src) + 1);
                        sc[k][0] = x.x; sc[k][1] = x.y; sc[k][2] = x.z; sc[k][3] = x.w;
                        sc[k][4] = y.x; sc[k][5] = y.y; sc[k][6] = y.z; sc[k][7] = y.w;
                    } else {
#pragma unroll
                        for (int i = 0; i < kHeadsEach; ++i) sc[k][i] = i < H && t < n_scores ? __ldcg(src + i) : 0.0f;
                    }
                } else {
                    sc[k][0] = t < n_scores ? __ldcg(src + h) : 0.0f;
                }
            }
        };
        if constexpr (kFrom == kFromScores) load_scores(0);
        int32_t start = 0, end = static_cast<int32_t>(a.n_tokens), base = 0, cursor = a.first_page, top = 0;
        int64_t list0 = static_cast<int64_t>(tid) * H;
        if (multi && tid < a.n_seqs) start = __ldg(a.cu_seqlens + tid);
        if (multi && tid == 0) end = __ldg(a.cu_seqlens + a.n_seqs);
        if constexpr (kAppend) {
            if (tid < n_lists) base = __ldcg(a.list_base + tid);
            if (tid < a.n_seqs) list0 = __ldcg(a.list_map + tid);
            if (tid == 0) {
                cursor = __ldcg(a.taken);
                top = __ldcg(a.taken + 1);
            }
        }
        if constexpr (kFrom == kFromWords) {
#pragma unroll
            for (int k = 0; k < kWordsEach; ++k)
                if (tid + k * kThreads < total) s_words[tid + k * kThreads] = w[k];
        }
        float tau = a.tau;
        if constexpr (kFrom == kFromScores && !kPages)
            if (a.tau_list != nullptr && tid < a.n_seqs) tau = __ldcg(a.tau_list + tid * H + h);
        if constexpr (kFrom == kFromScores && !kPages)
            if (tid < a.n_seqs) s_tau[tid] = tau;
        if (tid < a.n_seqs) s_cu[tid] = start;
        if (tid == 0) s_cu[a.n_seqs] = end;
        if constexpr (kPages) {
            if (tid < n_lists) s_base[tid] = base;
            if (tid < a.n_seqs) s_list[tid] = list0 + h;
            if (tid == 0) { cursor_s = cursor; free_s = top > 0 ? top : 0; }
        }
        if constexpr (kFrom == kFromScores) {
            __syncthreads();
            for (int32_t t0 = 0;;) {
#pragma unroll
                for (int k = 0; k < kScoresEach; ++k) {
                    const int32_t t = t0 + tid + k * kThreads, word = t / 32;
                    if (word * 32 >= n_scores) break;               // the whole warp: no token of it is wanted
                    const int b = multi ? seq_of_shared(s_cu, a.n_seqs, t) : 0;
                    const bool valid = t < n_scores, in_window = t >= s_cu[b + 1] - a.window;
#pragma unroll
                    for (int i = 0; i < kHeadsEach; ++i) {
                        const uint32_t bits = __ballot_sync(0xffffffffu, valid && (in_window || sc[k][i] >= (kPages ? a.tau : s_tau[b])));
                        if (lane == 0 && (!kPages || i < H)) s_words[(kPages ? i * n_words : 0) + word] = bits;
                    }
                }
                t0 += kScoresEach * kThreads;
                if (t0 >= n_scores) break;
                load_scores(t0);
            }
            // the words of a last block that are all past the end
            for (int i = (n_scores + 31) / 32 + tid; i < (n_scores + kBlockTokens - 1) / kBlockTokens * 4; i += kThreads)
                for (int j = 0; j < (kPages ? H : 1); ++j) s_words[j * n_words + i] = 0u;
        }
    }
    __syncthreads();
    const uint32_t *mine = s_words + (kPages ? h * n_words : 0);
    auto whole_pages = [&](int32_t rows) -> int32_t { return a.page_shift >= 0 ? rows >> a.page_shift : rows / a.page_tokens; };
    auto pages_of = [&](int32_t rows) -> int32_t { return whole_pages(rows + a.page_tokens - 1); };
    auto seq_at = [&](int64_t t) -> int { return multi ? seq_of_shared(s_cu, a.n_seqs, static_cast<int32_t>(t)) : 0; };
    // set bits of head words `w` for tokens [lo, hi), by a whole warp
    auto count = [&](const uint32_t *w, int32_t lo, int32_t hi) -> int32_t {
        int32_t n = 0;
        for (int i = lo / 32 + lane; i * 32 < hi; i += 32) {
            uint32_t v = w[i];
            if (i * 32 < lo) v &= ~0u << (lo - i * 32);
            if (i * 32 + 32 > hi) v &= (1u << (hi - i * 32)) - 1u;
            n += __popc(v);
        }
        return __reduce_add_sync(0xffffffffu, n);
    };

    // the rows of this block: which they are needs nothing but its words, so their loads go out first
    const int group = tid >> 4, gl = tid & 15;
    constexpr int kGroups = kThreads / 16;
    const int blk_start = blk * kBlockTokens, first = group + z * kGroups, step = nz * kGroups;
    uint32_t w0 = 0, w1 = 0, w2 = 0, w3 = 0;
    int cnt = 0, rank = 0;
    bool keep = false;
    uint4 kv[kShortRows], vv[kShortRows];
    const int64_t head_row0 = static_cast<int64_t>(h) * a.in_stride_h + blk_start * a.in_stride_t;
    auto load_rows = [&](int i0, int u0) {
#pragma unroll
        for (int j = 0; j < kShortRows; ++j) {
            const int i = i0 + j * step;
            if (i < cnt && u0 < a.row_units) {
                const int64_t src = (head_row0 + src_tok[i] * a.in_stride_t) * a.row_units + u0;
                kv[j] = __ldg(a.K + src);
                vv[j] = __ldg(a.V + src);
            }
        }
    };
    if (!books) {
        w0 = mine[blk * 4]; w1 = mine[blk * 4 + 1]; w2 = mine[blk * 4 + 2]; w3 = mine[blk * 4 + 3];
        cnt = __popc(w0) + __popc(w1) + __popc(w2) + __popc(w3);
        if (tid < kBlockTokens) {
            rank = popc_below(w0, w1, w2, w3, tid);
            const uint32_t w = tid < 32 ? w0 : tid < 64 ? w1 : tid < 96 ? w2 : w3;
            keep = (w >> (tid & 31)) & 1u;
            if (keep) src_tok[rank] = tid;
        }
        __syncthreads();
        load_rows(first, gl);
        if (warp == kWarps - 1) {
            // kept rows before the block, and before the start of the sequence in progress there
            const int32_t s0 = s_cu[seq_at(blk_start)];
            const int32_t before = count(mine, 0, s0 < blk_start ? s0 : blk_start), rest = s0 < blk_start ? count(mine, s0, blk_start) : 0;
            if (lane == 0) { before_s = before; running_s = before + rest; }
        }
    }
    if constexpr (kAppend) {
        if (tid < a.n_seqs) {
            const int32_t have = pages_of(s_base[tid * H + h]);
            s_last[tid] = have > 0 ? __ldcg(a.page_table + s_list[tid] * a.max_pages + have - 1) : 0;
        }
    }
    // kept rows of every list (dense: of this head's, and only for the bookkeeping), by as many threads per list as there are
    if (kPages || books) {
        const int lists = kPages ? n_lists : a.n_seqs;
        int each = 32;
        while (each * lists > kThreads) each >>= 1;
        const int i = tid / each, sub = tid & (each - 1);
        int32_t n = 0;
        if (i < lists) {
            const int b = kPages ? i / H : i;
            const uint32_t *w = s_words + (kPages ? (i - b * H) * n_words : 0);
            const int32_t lo = s_cu[b], hi = s_cu[b + 1];
            for (int j = lo / 32 + sub; j * 32 < hi; j += each) {
                uint32_t v = w[j];
                if (j * 32 < lo) v &= ~0u << (lo - j * 32);
                if (j * 32 + 32 > hi) v &= (1u << (hi - j * 32)) - 1u;
                n += __popc(v);
            }
        }
        for (int o = each >> 1; o > 0; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
        if (i < lists && sub == 0) s_len[i] = n;
    }
    __syncthreads();
    if constexpr (kPages) {
        if (warp == 0) {
            // pages in list order: those that a list needs beside the ones it has; all or nothing
            int32_t carry = 0;
            bool fail = false;
            for (int base = 0; base < n_lists; base += 32) {
                const int idx = base + lane;
                int32_t need = 0;
                if (idx < n_lists) {
                    const int32_t pages = pages_of(s_base[idx] + s_len[idx]);
                    fail = fail || pages > a.max_pages;
                    need = pages - pages_of(s_base[idx]);
                }
                int32_t incl = need;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int32_t y = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += y;
                }
                if (idx < n_lists) s_page0[idx] = carry + incl - need;       // ordinal of its first new page
                carry += __shfl_sync(0xffffffffu, incl, 31);
            }
            const int32_t from_stack = carry < free_s ? carry : free_s;
            // an append that needs no page but released ones fits wherever the cursor stands
            const bool fits = static_cast<int64_t>(cursor_s) + (carry - from_stack) <= a.n_pages_pool || (kAppend && carry == from_stack);
            fail = __any_sync(0xffffffffu, fail) || !fits;
            const bool first_cta = blk == a.n_blocks && h == 0;
            if (fail) {
                for (int idx = lane; idx < n_lists; idx += 32) s_page0[idx] = -1;
                if (first_cta && lane == 0) atomicCAS(a.status, 0, 4 /* KVZAP_ERR_OOM_PAGES */);
            }
            if (lane == 0) {
                stack_s = from_stack;
                if (first_cta && a.n_pages_used != nullptr) *a.n_pages_used = fail ? 0 : carry;
            }
            if (kAppend && first_cta && lane == 0 && !fail) {
                *a.page_cursor = cursor_s + carry - from_stack;
                if (from_stack > 0) *a.free_top = free_s - from_stack;
            }
        }
        __syncthreads();
    }
    auto page_at = [&](int32_t ordinal) -> int32_t {
        if (kAppend && ordinal < stack_s) return __ldcg(a.free_stack + free_s - 1 - ordinal);
        return cursor_s + ordinal - (kAppend ? stack_s : 0);
    };

    // given scores: this launch completes after the one ahead of it, whose scratch it clears
    auto finish = [&]() {
        if constexpr (kFrom == kFromScores) {
            griddep_wait();
            if (a.clear != nullptr) {
                const int64_t n_ctas = (static_cast<int64_t>(a.n_blocks) * nz + 1) * H;
                const int64_t cta = books ? n_ctas - H + h : (static_cast<int64_t>(blk) * nz + z) * H + h;
                for (int64_t i = cta * kThreads + tid; i < a.clear_units; i += n_ctas * kThreads) a.clear[i] = make_uint4(0u, 0u, 0u, 0u);
            }
        }
    };
    if (books) {
        for (int b = (blk - a.n_blocks) * kWarps + warp; b < a.n_seqs; b += a.n_books * kWarps) {
            const int64_t li = kPages ? s_list[b] : static_cast<int64_t>(b) * H + h;
            const int32_t kept = s_len[kPages ? b * H + h : b];
            if constexpr (kPages) {
                const int idx = b * H + h;
                const int32_t p0 = s_page0[idx], have = pages_of(s_base[idx]);
                const int32_t need = p0 < 0 ? 0 : pages_of(s_base[idx] + kept) - have;
                for (int32_t i = lane; i < need; i += 32) a.page_table[li * a.max_pages + have + i] = page_at(p0 + i);
                // an append that found no room leaves its lists as they were; a paged call says how long they would be
                if (lane == 0) a.lengths[li] = kAppend ? s_base[idx] + (p0 < 0 ? 0 : kept) : kept;
            } else {
                if (lane == 0) a.lengths[li] = kept;
            }
            if constexpr (kAppend) {
                const int32_t m = s_cu[b + 1] - s_cu[b], n_win = m < a.window ? m : a.window;
                const int32_t n_now = __ldcg(a.n_tokens_list + li);
                constexpr int kEach = 4;                          // scores per lane on their way together
                for (int32_t i0 = lane; i0 < n_win; i0 += 32 * kEach) {
                    float sc[kEach];
#pragma unroll
                    for (int k = 0; k < kEach; ++k) {
                        const int32_t i = i0 + 32 * k;
                        sc[k] = i < n_win ? __ldcg(a.scores + (static_cast<int64_t>(s_cu[b + 1]) - n_win + i) * H + h) : 0.0f;
                    }
#pragma unroll
                    for (int k = 0; k < kEach; ++k) {
                        const int32_t i = i0 + 32 * k;
                        if (i < n_win) a.score_ring[li * a.window + (n_now - n_win + i) % a.window] = sc[k];
                    }
                }
            }
        }
        finish();
        return;
    }
    if (keep) {
        const int64_t t = blk_start + tid;
        const int b = seq_at(t);
        const int32_t s = s_cu[b];
        // its rank in its list: kept rows before it less those before the start of its sequence
        const int32_t n = running_s + rank - (s >= blk_start ? running_s + popc_below(w0, w1, w2, w3, s - blk_start) : before_s);
        if constexpr (kPages) {
            const int idx = b * H + h;
            const int32_t p0 = s_page0[idx], nn = s_base[idx] + n, pi = whole_pages(nn), have = pages_of(s_base[idx]);
            int64_t page = -1;
            if (p0 >= 0) page = kAppend && pi < have ? s_last[b] : page_at(p0 + pi - have);
            dst_row[rank] = p0 < 0 ? -1 : page * a.page_tokens + (nn - pi * a.page_tokens);
        } else {
            dst_row[rank] = static_cast<int64_t>(h) * a.n_tokens + s + n;
        }
    }
    __syncthreads();
    for (int i0 = first; i0 < cnt; i0 += kShortRows * step)
        for (int u0 = gl; u0 < a.row_units; u0 += 16) {
            if (i0 != first || u0 != gl) load_rows(i0, u0);
#pragma unroll
            for (int j = 0; j < kShortRows; ++j) {
                const int i = i0 + j * step;
                if (i < cnt && dst_row[i] >= 0) {
                    const int64_t d = dst_row[i] * a.row_units + u0;
                    a.K_out[d] = kv[j];
                    a.V_out[d] = vv[j];
                }
            }
        }
    finish();
}

}  // namespace kvzap
