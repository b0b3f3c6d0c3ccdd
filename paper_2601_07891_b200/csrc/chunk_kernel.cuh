// Chunked prefill into a cache, the window side of one chunk of prompt tokens and the page assignment for its rows.
#pragma once

#include "decode_kernels.cuh"
#include "prune_kernels.cuh"

namespace kvzap {

// The sequence slots of a call, by value (so that no copy runs ahead of the kernels); more than kMaxChunkSeqs of them:
// n = 0 and list_map, already in device memory, names the list of head 0 of every sequence.
constexpr int kMaxChunkSeqs = 128;
struct ChunkSeqs {
    int32_t n;
    int32_t slot[kMaxChunkSeqs];
};

constexpr int kChunkThreads = 256;

// For every list (sequence of the call, head) of one layer, one CTA each (grid (H, n_seqs)), after the chunk has been
// scored and its tokens outside the window have been thresholded into mask words:
//   1. the tokens of the present window that the chunk pushes out (positions below n_old + m - w) are
//      decided by their buffered scores, oldest first, and the kept ones appended to the list's paged
//      prefix (pages from the cache's allocator) -- what m decode steps would have done;
//   2. the chunk's last min(m, w) tokens (rows of K, V [H][n_total][D], scores [n_total][H]) take the ring slots of
//      their absolute positions n_old + chunk index;
//   3. n_tokens advances by m; the prefix length becomes what the list will hold once the compaction behind this
//      launch has appended the chunk's own kept rows, list_base remembers what it holds now;
// and the CTA that is done last assigns pages for all lists' new rows (assign_pages, all or nothing), which the
// compaction reads.  assign == 0 (chunks short enough for compact_short_kernel): counting, prefix lengths, pages and the ring's scores are
// left to that launch, and all that this one does behind the scoring is end.  Sequence b's chunk is tokens cu_seqlens[b] .. cu_seqlens[b+1] of the packed buffers (cu_seqlens ==
// nullptr: all of them).
// What bounds it is a chain of round trips to memory (counts, scores, pages, rows, arrival, assignment).  Most of it
// depends on nothing that the scoring computes: with `beside` != 0 the launch ahead is a scoring kernel that lets this one
// start once everything ahead of IT has completed, and 1 and the rows of 2 run beside it; the CTAs are small enough to
// share an SM with its CTAs.  Only the counting of the chunk's kept rows, its scores and the page assignment are left for
// the time after it.  4 prompts x 8 heads, a window of 128 pushed out, from the end of the scoring launch: 24.5 us page by
// page with a launch of its own for the assignment, 16 us as one launch of 1024 threads per list behind the scoring,
// 7.7 us beside it.  Rows of the kept exits only, four in flight, and 32-bit quotients: the window side beside the scoring ended 3 us behind
// it, now with it.
__global__ void __launch_bounds__(kChunkThreads, 4)      // 64 registers: see compact_dense_kernel
chunk_ring_kernel(const CacheView c, const __grid_constant__ ChunkSeqs seqs, int layer, int64_t *__restrict__ list_map,
                  const float *__restrict__ scores, const uint4 *__restrict__ K, const uint4 *__restrict__ V, int64_t n_total, float tau,
                  const int32_t *__restrict__ cu_seqlens, const uint32_t *__restrict__ maskbits, int64_t n_words,
                  int32_t *__restrict__ list_base, int32_t *__restrict__ list_page0, uint32_t *__restrict__ arrive,
                  int32_t *__restrict__ status, int beside, int assign, int32_t *__restrict__ taken)
{
    __shared__ int64_t exit_src[128];       // ring row of an exiting token that is kept
    __shared__ int64_t exit_dst[128];       // its pool row, -1 = no page left for it
    __shared__ int32_t new_pages[128];
    __shared__ int64_t len_s;
    __shared__ int ok_s, kept_s, last_s, cursor_s, moved_s;
    if (!beside) griddep_wait();
    const int h = blockIdx.x, b = blockIdx.y, H = c.n_heads;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t list0 = seqs.n > 0 ? (static_cast<int64_t>(seqs.slot[b]) * c.n_layers + layer) * H : __ldcg(list_map + b);
    const int64_t li = list0 + h;
    const int64_t tok0 = cu_seqlens != nullptr ? static_cast<int64_t>(cu_seqlens[b]) : 0;
    const int32_t m = static_cast<int32_t>(cu_seqlens != nullptr ? static_cast<int64_t>(cu_seqlens[b + 1]) - tok0 : n_total);
    K += tok0 * c.row_units;                // row (h, i) of the chunk is row h * n_total + tok0 + i of the buffers
    V += tok0 * c.row_units;
    scores += tok0 * H;
    // positions and lengths are 32-bit counts (n_tokens): their quotients by window and page size are in every chain below
    const int32_t n_old = __ldcg(c.n_tokens + li);
    const uint32_t window = static_cast<uint32_t>(c.window), page_tokens = static_cast<uint32_t>(c.page_tokens);
    if (tid == 0) { len_s = __ldcg(c.prefix_len + li); kept_s = 0; }
    __syncthreads();
    const int32_t in_ring = n_old < c.window ? n_old : c.window;
    const int32_t first = n_old - in_ring;                         // oldest position still in the window
    const int32_t exit_end = m > c.window ? n_old : n_old + (m - c.window);      // positions below it leave the window
    const int32_t n_exit = m > 0 && exit_end > first ? exit_end - first : 0;      // an empty chunk leaves its list as it is
    int32_t *table = c.page_table + li * c.max_pages;
    const int group = tid >> 4, gl = tid & 15;
    constexpr int kGroups = kChunkThreads / 16, kRows = 4;         // 16 lanes per row, four rows per lane group in flight
    for (int32_t base = 0; base < n_exit; base += 128) {
        if (warp == 0) {
            const uint32_t len = static_cast<uint32_t>(len_s);
            uint32_t kept[4];
            float sc4[4];                                          // the buffered scores of the batch, loaded together
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint32_t pos = static_cast<uint32_t>(first + base + 32 * j + lane);
                sc4[j] = base + 32 * j + lane < n_exit ? __ldcg(c.score_ring + li * c.window + pos % window) : 0.0f;
            }
            int total = 0;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                kept[j] = __ballot_sync(0xffffffffu, base + 32 * j + lane < n_exit && sc4[j] >= tau);
                total += __popc(kept[j]);
            }
            // pages for all of them; what does not fit is dropped, oldest rows first served
            const int32_t have = static_cast<int32_t>((len + page_tokens - 1) / page_tokens);
            int32_t want = static_cast<int32_t>((len + total + page_tokens - 1) / page_tokens);
            bool ok = true;
            if (want > c.max_pages) {
                want = c.max_pages > have ? c.max_pages : have;
                ok = false;
                if (lane == 0) atomicCAS(status, 0, 4 /* KVZAP_ERR_OOM_PAGES */);
            }
            const int n_new = want - have;
            const int got = cache_take_pages(c, status, n_new, new_pages, lane);
            if (got < n_new) ok = false;
            __syncwarp();
            for (int i = lane; i < got; i += 32) table[have + i] = new_pages[i];
            const uint32_t room = static_cast<uint32_t>(have + got) * page_tokens;
            int before = 0;                                        // the kept ones, in order; their rows alone are moved
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint32_t pos = static_cast<uint32_t>(first + base + 32 * j + lane);
                if ((kept[j] >> lane) & 1u) {
                    const int at = before + __popc(kept[j] & ((1u << lane) - 1u));
                    const uint32_t nn = len + static_cast<uint32_t>(at);
                    int64_t dst = -1;
                    if (nn < room) {
                        const int32_t pi = static_cast<int32_t>(nn / page_tokens);
                        const int64_t page = pi < have ? __ldcg(table + pi) : new_pages[pi - have];
                        dst = page * c.page_tokens + (nn - static_cast<uint32_t>(pi) * page_tokens);
                    }
                    exit_src[at] = li * c.window + pos % window;
                    exit_dst[at] = dst;
                }
                before += __popc(kept[j]);
            }
            if (lane == 0) {
                len_s = static_cast<int64_t>(len + total < room ? len + total : room);
                ok_s = ok;
                moved_s = total;
            }
        }
        __syncthreads();
        const bool more = ok_s != 0;        // read between two barriers: all threads leave the loop together
        const int n_batch = moved_s;
        for (int i0 = group; i0 < n_batch; i0 += kRows * kGroups) {
            for (int u = gl; u < c.row_units; u += 16) {
                uint4 kr[kRows], vr[kRows];
#pragma unroll
                for (int j = 0; j < kRows; ++j) {
                    const int i = i0 + kGroups * j;
                    if (i < n_batch && exit_dst[i] >= 0) {
                        kr[j] = __ldcg(c.k_ring + exit_src[i] * c.row_units + u);
                        vr[j] = __ldcg(c.v_ring + exit_src[i] * c.row_units + u);
                    }
                }
#pragma unroll
                for (int j = 0; j < kRows; ++j) {
                    const int i = i0 + kGroups * j;
                    if (i < n_batch && exit_dst[i] >= 0) {
                        c.k_pool[exit_dst[i] * c.row_units + u] = kr[j];
                        c.v_pool[exit_dst[i] * c.row_units + u] = vr[j];
                    }
                }
            }
        }
        __syncthreads();
        if (!more) break;                   // no page left: the exits behind these are dropped
    }
    // the chunk's last min(m, w) tokens into the ring (the slots they take were read above)
    const int32_t n_win = m < c.window ? m : c.window;
    for (int32_t i0 = group; i0 < n_win; i0 += kRows * kGroups) {
        for (int u = gl; u < c.row_units; u += 16) {
            uint4 kr[kRows], vr[kRows];
#pragma unroll
            for (int j = 0; j < kRows; ++j) {
                const int32_t i = i0 + kGroups * j;
                if (i < n_win) {
                    const int64_t src = (static_cast<int64_t>(h) * n_total + m - n_win + i) * c.row_units + u;
                    kr[j] = __ldg(K + src);
                    vr[j] = __ldg(V + src);
                }
            }
#pragma unroll
            for (int j = 0; j < kRows; ++j) {
                const int32_t i = i0 + kGroups * j;
                if (i < n_win) {
                    const int64_t slot = li * c.window + static_cast<uint32_t>(n_old + (m - n_win) + i) % window;
                    c.k_ring[slot * c.row_units + u] = kr[j];
                    c.v_ring[slot * c.row_units + u] = vr[j];
                }
            }
        }
    }
    if (!assign && tid == 0) {
        // compact_short_kernel counts the chunk's own rows and finds their pages; whoever takes a page here last leaves it the
        // allocator as it is then
        if (seqs.n > 0 && h == 0) list_map[b] = list0;
        list_base[b * H + h] = static_cast<int32_t>(len_s);
        c.n_tokens[li] = static_cast<int32_t>(n_old + m);
        if (h == 0 && m > 0) c.active[li / (static_cast<int64_t>(c.n_layers) * H)] = 1;     // the slot holds a sequence again
        if (arrive_last(arrive, gridDim.x * gridDim.y)) {
            taken[0] = __ldcg(c.page_cursor);
            taken[1] = c.free_top != nullptr ? __ldcg(c.free_top) : 0;
        }
    }
    if (beside) griddep_wait();
    griddep_launch_dependents();
    if (!assign) return;
    // the chunk's own kept rows; the scores of those in the ring
    {
        const uint32_t *words = maskbits + static_cast<int64_t>(h) * n_words;
        int cnt = 0;
        for (int64_t wi = tok0 / 32 + tid; wi * 32 < tok0 + m; wi += kChunkThreads) {
            uint32_t w = __ldcg(words + wi);
            if (wi * 32 < tok0) w &= ~0u << static_cast<int>(tok0 - wi * 32);                    // bits below the chunk
            if (wi * 32 + 32 > tok0 + m) w &= (1u << static_cast<int>(tok0 + m - wi * 32)) - 1u; // bits above it
            cnt += __popc(w);
        }
        cnt = __reduce_add_sync(0xffffffffu, cnt);
        if (lane == 0 && cnt) atomicAdd(&kept_s, cnt);
    }
    for (int32_t i = tid; i < n_win; i += kChunkThreads) {
        const int32_t ci = m - n_win + i;                          // index inside the chunk
        c.score_ring[li * c.window + static_cast<uint32_t>(n_old + ci) % window] = __ldcg(scores + static_cast<int64_t>(ci) * H + h);
    }
    __syncthreads();
    if (tid == 0) {
        const int32_t len = static_cast<int32_t>(len_s);
        if (seqs.n > 0 && h == 0) list_map[b] = list0;             // for the page assignment and the compaction
        list_base[b * H + h] = len;
        c.prefix_len[li] = len + kept_s;
        c.n_tokens[li] = static_cast<int32_t>(n_old + m);
        if (h == 0 && m > 0) c.active[li / (static_cast<int64_t>(c.n_layers) * H)] = 1;     // the slot holds a sequence again
        __threadfence();
        last_s = atomicAdd(arrive, 1u) + 1u == gridDim.x * gridDim.y;
        if (last_s) *arrive = 0u;                                  // ready for the next launch
        __threadfence();
        cursor_s = __ldcg(c.page_cursor);
    }
    __syncthreads();
    if (!last_s) return;
    assign_pages<kChunkThreads, 128>(H, gridDim.y, c.prefix_len, c.page_tokens, cursor_s, c.n_pages_pool, c.max_pages, list_page0,
                                c.page_table, nullptr, c.page_cursor, status, 1, list_base, c.free_stack, c.free_top, 1, list_map);
}

// no window: only the token count advances (one block per sequence of the call)
__global__ void tokens_add_kernel(const CacheView c, const __grid_constant__ ChunkSeqs seqs, int layer, int64_t *__restrict__ list_map,
                                  int64_t n_total, const int32_t *__restrict__ cu_seqlens)
{
    const int b = blockIdx.x;
    const int64_t li0 = seqs.n > 0 ? (static_cast<int64_t>(seqs.slot[b]) * c.n_layers + layer) * c.n_heads : list_map[b];
    if (seqs.n > 0 && threadIdx.x == 0) list_map[b] = li0;         // for the page assignment and the compaction
    const int64_t m = cu_seqlens != nullptr ? cu_seqlens[b + 1] - cu_seqlens[b] : n_total;
    if (m <= 0) return;
    if (threadIdx.x < c.n_heads) c.n_tokens[li0 + threadIdx.x] += static_cast<int32_t>(m);
    if (threadIdx.x == 0) c.active[li0 / (static_cast<int64_t>(c.n_layers) * c.n_heads)] = 1;
}

}  // namespace kvzap
