// Attention of the new token over the pruned cache (Introduction, Criterion 3; Discussion,
// "Implementation Challenges": per-head list lengths differ, so the attention kernel has to take
// variable-length lists).  One CTA per (sequence, layer, KV head) list; the G query heads that share
// the KV head (grouped-query attention) are processed together, so every K and V row is read from
// HBM exactly once per step.  The kernel is bound by those reads.
//
// A list is its paged prefix (prefix_len rows in pages of page_tokens rows) plus the valid slots of
// its window ring; softmax attention does not depend on the order of the rows, so the two parts are
// simply walked one after the other in tiles of 16 rows.  Warp w of the CTA takes tiles w, w + W,
// w + 2W, ... with its own online-softmax state and its own ring of shared-memory stages: lane 0
// issues the TMA loads of a tile (K and V, 128-byte swizzle, two 64-element halves per row when
// D = 128) onto the stage's mbarrier, the warp waits for it, and nothing is shared between warps
// until the end, when the partial (max, sum, output) triples are merged through shared memory.
// When a call has too few lists to keep every SM busy to the end (one layer of a moderate batch, or
// a few long sequences), each list is cut into n_parts equal runs of tiles, one CTA each; the parts
// leave their triples in global memory and the part that arrives last (a counter per list) merges
// them in part order, so the result does not depend on which one that was.
// Of a call of many lists the last ones may have more parts than the others: the device takes CTAs in order, and a long list among the
// last would be worked on when all others are done.  The CTAs that this takes are the last of the launch: of a list that turns out
// short they have nothing to do, and pass through slots that the others have left.
// With fewer lists than resident CTAs (a small batch, layer by layer) there is one wave, and it lasts as
// long as its longest part: equal parts of lists whose lengths spread over 1 : 7 (contexts of one batch x
// what each head keeps) leave most of it idle.  There the CTAs share the lists out themselves (attn_unit):
// every CTA reads all list lengths, finds the shortest part length (of at least four tiles a warp) for which
// all parts fit the grid, and takes the part of its index.  8 sequences x 8 heads, 2176 rows on average: 26.0 -> 20.4 us per call.
//
// Layer by layer a small batch is a chain of two launches of about the same length, the step (round trips to memory on a
// fifth of the SMs) and this one (round trips, then rows).  On a context that trusts its producers they run beside one another
// (kBeside): the step behind an attention scores beside it and only its stores to the cache wait, and the attention behind
// that step reads all rows that the lists held before it while it runs; what the step changes (the prefix's last tile, the
// window) is read when it has completed, and so are the queries, once more -- if they are not what they were, the CTA starts
// again.  36 layers x 8 sequences x 2176 rows 1235 -> 855 to 900 us, 4 layers x 128 sequences x 4736 rows 1600 -> 1500 to 1545 us.
// A warp waits for the step, and lets the next one start, while tiles are in flight (behind all of them the copies ran dry, and the
// chain step - wait - next step was the longer by the time of two tiles; when it does: kWaitBase), the new lengths and the second look at the queries share a round trip, and the parts of a list are counted in by one
// release instead of two fences: 36 layers x 8 sequences x 2176 rows 808 -> 740 us, 12 x 4 201 -> 193, 12 x 8 8-bit 279 -> 265, 12 x 32 8-bit
// 419 -> 392 (with the steps of score_split_kernel's kFew on both sides).  (Each pair here and below is of one GPU; from one GPU to another the
// same code differs by up to a tenth, most over 8-bit rows.)
//
// Math per tile, on the warp-level tensor-core path (the work is HBM-bound; 16-row MMAs are enough):
//   S[16 x 16]  = Q[16 x D] K^T      m16n8k16, Q rows 0..G-1 real, the rest zero
//   P           = exp2(S * scale * log2(e) - running max), rows beyond the list's end masked
//   O[16 x D]  += P[16 x 16] V
// Rows of a partly filled tile that lie past the end are excluded from the softmax, and their V
// rows are zeroed in shared memory first (stale pool memory may hold NaN bit patterns).
//
// 8-bit rows (Related work, "Quantization": pruning and quantisation of the cache compose).  A cache whose
// rows are D E4M3 codes followed by a 16-byte trailer (the row's fp32 scale, then 12 unused bytes) is walked
// by the same kernel with kFp8 = true: a tile is 16 whole rows, contiguous in memory, brought in by one
// unswizzled TMA box of full 128-byte lines per K and V, the codes are widened to f16 in registers (one exact conversion per pair) and the MMAs take f16
// operands.  Everything that is not a code is kept inside f16's range by factors applied around the MMAs: a
// query row is divided by the power of two of its largest element (exact; bf16's mantissa fits f16's) and the
// K row scales join that factor on the logits, logit = scale * 2^e * ks_i * (q 2^-e . K8_i); P is multiplied by
// vs_i / vref, vref the largest V scale met so far (the accumulator is rescaled when it grows, together with the
// online softmax's own rescaling, and multiplied by vref at the end), so the second operand lies in [0, 1] and
// is rounded to f16 (11 bits) where the bf16 path rounds P to 8.  The MMA's summation index and the
// output columns may be numbered freely as long as both operands agree, so each lane reads whole 16- or 32-byte
// pieces of a row: for Q K^T lane (n, c) owns bytes [c D/4, (c+1) D/4) of K rows n and n + 8, k-step ks taking
// four of them; the second product is computed transposed, O^T += V^T P^T (P, as the softmax leaves it, is the
// B operand; no accumulator row is wasted on the padding of the query heads to 16), lane (n', c) owning bytes
// [n' D/8, (n'+1) D/8) of V rows 2c, 2c+1, 2c+8, 2c+9.  With rows 144 (or 80) bytes apart these reads have no
// bank conflicts.  Four CTAs fit an SM (128 registers, 56 KB of stages).
#pragma once

#include <cuda_fp16.h>

#include "decode_kernels.cuh"
#include "ptx.cuh"

namespace kvzap {

constexpr int kAttnWarps = 4;
// Stages of a warp's ring.  bf16 rows: two, so that three CTAs fit an SM (168 registers, 66 KB) -- the same bytes in flight as
// two CTAs with three stages, but the serial parts of a CTA (counts, pages, first tiles, merge: some 3 us) run beside two
// others: 128 sequences x 4 layers, layer by layer, 1553 -> 1527 us; 80 x 8 layers 1245 -> 1175 us.  Rows of 64 elements (122
// registers, half the bytes a stage): two or three make 0 to 5 % either way (8 sequences x 2000 rows 13.6 / 14.3 us, 64 x
// 300 12.9 / 13.3, 128 x 4000 169.8 / 169.6, 512 x 200 50.2 / 49.2), so they have two as well.  8-bit rows: three, four CTAs
// fit either way.
__host__ __device__ constexpr int attn_stages(bool fp8) { return fp8 ? 3 : 2; }
constexpr int kAttnTileRows = 16;
constexpr int kAttnThreads = kAttnWarps * 32;
constexpr int kAttnMaxGroup = 8;                 // query heads per KV head (rows 0..7 of the 16-row MMA)
constexpr uint32_t kAttnHalfBytes = kAttnTileRows * 128;   // 16 rows x 64 bf16

struct AttnParams {
    CacheView c;
    int32_t layer0, n_layers_call;
    int32_t group;              // G = query heads per KV head, 1..8
    float scale_log2e;          // softmax scale times log2(e)
    const uint16_t *q;          // [n_layers_call][B][H * G][D] bf16
    uint16_t *out;              // same shape
    int32_t *status;
    int32_t n_parts;            // CTAs per list (1 = the CTA writes the output itself); 0 = by length, see attn_unit
    float *part_scratch;        // [unit] { m[8], l[8], O[8][D] }: the parts of a list are consecutive units; n_parts == 0: unit = CTA
    uint32_t *part_arrive;      // [list - list0] parts that have stored their triple; back to 0 after the launch
    // n_parts > 0: CTAs [0, extra0) are the parts of all lists; behind them the lists from head_lists on have tail_parts - n_parts
    // more each, of which as many take part as leave a part kAttnTailTiles tiles
    int32_t extra0, head_lists, tail_parts;
    int32_t tail_unit0, list0;  // unit of the first part of list head_lists; first list with several parts
    int32_t tiles_shift;        // logarithm of the tiles per page, or -1
    int32_t beside_ctas;        // kBeside: CTAs [0, beside_ctas) run beside the step, as many as find room
    int32_t beside_tiles;       // n_parts == 0: with more tiles than this in all lists all CTAs wait for the step
};

// The lists of a call, of lengths[0 .. n) tiles, cut into at most n_units (>= n) parts: a list of t tiles has
// ceil(t / target) parts, or one if it is empty, with a target from a few steps of bisection between an equal share of
// all tiles and the longest list.  Whole warp, the same result in every warp of the launch (the quotients are taken in
// fp32: whatever their rounding, every warp rounds alike).  Returns the number of parts of the list that `unit` falls
// into, 0 if there is no such unit; `list` and `part` say which.
constexpr int kAttnListsPerLane = 20;       // n <= 32 * this
constexpr float kAttnMinPart = 16.0f;       // tiles
// Beside a step, in one wave: cycles from a CTA's start to its wait for that step, with it the start of the next one, as a base and by
// its tiles of 128 elements.  The step is over by then, and the next one, its launch and the next attention's first CTAs (on the SMs
// that the steps use) are there when this launch ends; earlier the wait would be one, later the memory idles between the two.  Us, 12
// layers, waiting at the last known tile / at this time / a quarter of the tiles' share earlier / later: 16 sequences x 2176 rows 402 /
// 359 / 361 / 356, 32 x 2176 765 / 636 / 643 / 639, 12 x 1628 263 / 247 / 248 / 248, 4 x 7628 346 / 322 / 326 / 320; 8-bit 32 x 1152 402 / 357 / 363 /
// 365, 16 x 2176 349 / 317 / 314 / 328, 30 x 2378 619 / 533 / 551 / 540, 8 x 2176 260 / 263 / 263 / 261; 36 layers, 8 x 2176 730 / 698 / 698 / 702.
// (When half of the tiles are issued, whatever the clock: 361, 640, 248, 323; 366, 321, 542, 257; 693.)  Not with several waves: 512 lists
// of 1128 rows 263 / 271.  Cycles of the SM's clock, at the 1.75 to 1.97 GHz that it has in such calls, which wait for memory: slower, and the wait comes later, at
// the latest with the last known tile.
constexpr int kWaitBase = 12000, kWaitTile = 270, kWaitTile8 = 400;
constexpr int kAttnTailTiles = 40;          // a part of the lists at the end of a launch of many, at least
__device__ __forceinline__ int attn_unit(const int32_t *lengths, int n, int n_units, int unit, int lane, int &list, int &part)
{
    // lane l owns lists [l * per, (l + 1) * per), in registers
    const int per = (n + 31) / 32, first = lane * per;
    float len[kAttnListsPerLane];
    int sum = 0, longest = 1, own = 0;
#pragma unroll
    for (int i = 0; i < kAttnListsPerLane; ++i) {
        if (i >= per) break;
        const int t = first + i < n ? lengths[first + i] : 0;
        if (first + i < n) own = i + 1;
        len[i] = static_cast<float>(t);
        sum += t;
        longest = max(longest, t);
    }
    sum = __reduce_add_sync(0xffffffffu, sum);
    longest = __reduce_max_sync(0xffffffffu, longest);
    auto parts_of = [&](int i, float inv) { return max(1, __float2int_ru(len[i] * inv)); };
    auto lane_parts = [&](float inv) {
        int parts = 0;
#pragma unroll
        for (int i = 0; i < kAttnListsPerLane; ++i) {
            if (i >= per) break;
            if (i < own) parts += parts_of(i, inv);
        }
        return parts;
    };
    float lo = fmaxf(kAttnMinPart, static_cast<float>(sum) / static_cast<float>(n_units)), hi = fmaxf(lo, static_cast<float>(longest));
    if (n * 2 <= n_units) hi = fminf(hi, 2.02f * lo);       // at most sum / hi + n parts
    constexpr float kDown = 1.0f - 1.0f / (1 << 20);        // a list of exactly the target length is one part
    float inv = kDown / hi;                                 // fits: one part each, or half of the units plus one each
    for (int step = 0; step < 6; ++step) {
        const float mid = 0.5f * (lo + hi), inv_mid = kDown / mid;
        const bool fits = __reduce_add_sync(0xffffffffu, lane_parts(inv_mid)) <= n_units;
        if (fits) { hi = mid; inv = inv_mid; } else lo = mid;
    }
    const int mine = lane_parts(inv);
    int incl = mine;                                        // the running number of parts finds the unit's list
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    int at = incl - mine, found = -1, parts = 0;
    if (unit >= at && unit < incl) {
#pragma unroll
        for (int i = 0; i < kAttnListsPerLane; ++i) {
            if (i >= per) break;
            if (found >= 0) continue;
            parts = parts_of(i, inv);
            if (unit < at + parts) found = first + i; else at += parts;
        }
    }
    const uint32_t who = __ballot_sync(0xffffffffu, found >= 0);
    if (who == 0u) return 0;
    const int src = __ffs(who) - 1;
    list = __shfl_sync(0xffffffffu, found, src);
    part = unit - __shfl_sync(0xffffffffu, at, src);
    return __shfl_sync(0xffffffffu, parts, src);
}

constexpr int kAttnTrailerBytes = 16;            // 8-bit rows: fp32 scale + 12 unused bytes behind the codes
__host__ __device__ constexpr uint32_t attn_stage_bytes(int head_dim, bool fp8 = false)
{
    return fp8 ? 2u * kAttnTileRows * (head_dim + kAttnTrailerBytes) : 2u * (head_dim / 64) * kAttnHalfBytes;
}
__host__ __device__ constexpr uint32_t attn_smem_bytes(int head_dim, bool fp8 = false)
{
    return kAttnWarps * attn_stages(fp8) * attn_stage_bytes(head_dim, fp8) + (fp8 ? 128u : 1024u) /* alignment */ + 256u /* barriers */;
}

// four E4M3 codes (a 32-bit word, lowest byte first) -> two packed f16 pairs (exact: f16 holds every E4M3 value)
__device__ __forceinline__ void e4m3x4_to_f16(uint32_t w, uint32_t &lo, uint32_t &hi)
{
    asm("{\n\t.reg .b16 a, b;\n\tmov.b32 {a, b}, %2;\n\tcvt.rn.f16x2.e4m3x2 %0, a;\n\tcvt.rn.f16x2.e4m3x2 %1, b;\n\t}"
        : "=r"(lo), "=r"(hi) : "r"(w));
}
__device__ __forceinline__ float bf16_lo(uint32_t pair) { return __uint_as_float(pair << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t pair) { return __uint_as_float(pair & 0xffff0000u); }

__device__ __forceinline__ void attn_add(float4 &num, const float4 &o, float f)
{
    num.x += o.x * f; num.y += o.y * f; num.z += o.z * f; num.w += o.w * f;
}
// four output elements as bf16; zeros when nothing was summed
__device__ __forceinline__ void attn_store(uint16_t *out, const float4 &num, float den)
{
    const bool some = den > 0.0f;
    const uint2 v = make_uint2(pack_bf16x2(some ? num.x / den : 0.0f, some ? num.y / den : 0.0f),
                               pack_bf16x2(some ? num.z / den : 0.0f, some ? num.w / den : 0.0f));
    *reinterpret_cast<uint2 *>(out) = v;
}

// kBeside: the launch may run beside the step ahead of it; a kernel of its own, since what that takes (the rest of a list learnt
// late, queries read twice, more code) costs a launch 2 to 5 us where nothing runs beside it: behind other work of the caller.
template <int kD, bool kFp8, bool kBeside>
__global__ void __launch_bounds__(kAttnThreads, kFp8 ? 4 : 3)
decode_attn_kernel(const __grid_constant__ CUtensorMap tmap_kpool, const __grid_constant__ CUtensorMap tmap_vpool,
                   const __grid_constant__ CUtensorMap tmap_kring, const __grid_constant__ CUtensorMap tmap_vring,
                   const AttnParams p)
{
    constexpr int kHalves = kD / 64;
    constexpr int kAttnStages = attn_stages(kFp8);
    constexpr uint32_t kStageBytes = attn_stage_bytes(kD, kFp8);
    constexpr int kRowBytes8 = kD + kAttnTrailerBytes;              // 8-bit rows
    constexpr uint32_t kTileBytes8 = kAttnTileRows * kRowBytes8;
    // accumulator tiles: 16 x 8 pieces of O (rows = query heads, half of them unused) for bf16 rows,
    // 16 x 8 pieces of O^T (rows = elements, columns = query heads) for 8-bit rows
    constexpr int kNTiles = kFp8 ? kD / 16 : kD / 8;
    constexpr uint32_t kAlign = kFp8 ? 128u : 1024u;            // swizzled tiles need 1024-byte alignment
    extern __shared__ uint8_t attn_smem_raw[];
    const uint32_t raw_addr = smem_u32(attn_smem_raw);
    const uint32_t pad = (kAlign - (raw_addr & (kAlign - 1u))) & (kAlign - 1u);
    uint8_t *smem = attn_smem_raw + pad;
    const uint32_t smem_base = raw_addr + pad;
    const uint32_t bars = smem_base + kAttnWarps * kAttnStages * kStageBytes;      // [warp][stage] mbarriers
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + kAttnWarps * kAttnStages * kStageBytes + 8 * kAttnWarps * kAttnStages);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const CacheView &c = p.c;
    const int H = c.n_heads, B = c.n_seqs;
    const uint32_t started = kBeside ? static_cast<uint32_t>(clock()) : 0u;       // differences are right across its wrap

    __shared__ int queries_s;               // kBeside: warps that are done with the queries in memory
    if (threadIdx.x == 0) {
        for (int i = 0; i < kAttnWarps * kAttnStages; ++i) mbar_init(bars + 8 * i, 1);
        *abort_flag = 0;
        queries_s = 0;
        fence_mbar_init();
        prefetch_tensormap(&tmap_kpool);
        prefetch_tensormap(&tmap_vpool);
        prefetch_tensormap(&tmap_kring);
        prefetch_tensormap(&tmap_vring);
    }
    __syncthreads();
    // Started while the kernel ahead may still be running: nothing of the caller's or of the cache is read before that has
    // completed.  kBeside: that is the step which appends the newest rows, and nothing else that writes the cache is still
    // running (the host knows, see attention_impl); every whole tile of rows that a list held before it is taken beside it.
    // How long the lists were before the step, by which the CTAs of a launch share them out, all read in c.before: it does
    // not change while this launch runs.  CTAs that find no room beside the step wait for it first.
    bool beside = kBeside && static_cast<int>(blockIdx.x) < p.beside_ctas;
    if (!beside) griddep_wait();

    int list, part, n_parts = p.n_parts;
    int32_t n_before = 0;                   // kBeside: prefix rows that nothing ahead of this launch still touches
    int32_t n_prefix = 0, n_total = 0;      // rows and tokens now; beside the step not known yet
    const int32_t *before = kBeside ? c.before : c.prefix_len;
    auto cache_list = [&](int i) {          // list i of the call among the cache's lists
        return (static_cast<int64_t>((i / H) % B) * c.n_layers + p.layer0 + i / (H * B)) * H + i % H;
    };
    if (n_parts > 0) {
        const int extra = static_cast<int>(blockIdx.x) - p.extra0;
        if (extra < 0) {
            list = static_cast<int>(blockIdx.x) / n_parts;
            part = static_cast<int>(blockIdx.x) - list * n_parts;
        } else {
            const int each = p.tail_parts - n_parts;
            list = p.head_lists + extra / each;
            part = n_parts + extra % each;
        }
        if (kBeside) n_before = min(__ldcg(before + cache_list(list)), __ldcg(c.prefix_len + cache_list(list)));
        if (!beside) {
            n_total = __ldcg(c.n_tokens + cache_list(list));
            n_prefix = __ldcg(c.prefix_len + cache_list(list));
        }
        if (list >= p.head_lists) {
            const int tiles = ((kBeside ? n_before : n_prefix) + min(kBeside ? c.window : n_total, c.window)) / kAttnTileRows;
            // as many as the other lists have, or more; a list that is over in 16 tiles has one
            n_parts = tiles < 16 ? 1 : max(n_parts, min(p.tail_parts, tiles / kAttnTailTiles));
            if (part >= n_parts) {                                 // the whole CTA
                if (beside) griddep_wait();
                return;
            }
        }
    } else {
        // over the stages, not in use yet: [list] tiles, then [list] (prefix rows, tokens); kBeside: the window counts in full
        const int n_lists = p.n_layers_call * B * H;
        int32_t *lengths = reinterpret_cast<int32_t *>(smem);
        int2 *counts = reinterpret_cast<int2 *>(smem + 4 * 32 * kAttnListsPerLane);
        for (int i = threadIdx.x; i < n_lists; i += kAttnThreads) {
            int2 n = make_int2(__ldcg(before + cache_list(i)), beside ? 0 : __ldcg(c.n_tokens + cache_list(i)));
            if (kBeside) n.x = min(n.x, __ldcg(c.prefix_len + cache_list(i)));      // it never is less, nor may it be
            counts[i] = n;
            lengths[i] = (n.x + kAttnTileRows - 1) / kAttnTileRows + ((kBeside ? c.window : min(n.y, c.window)) + kAttnTileRows - 1) / kAttnTileRows;
        }
        __syncthreads();
        // One wave: beside the step, on the SMs that it leaves, if what that adds to the wave's time is less than the step's;
        // else on all of them, behind it.
        int n_units = gridDim.x;
        if constexpr (kBeside) {
            int sum = 0;
            for (int i = lane; i < n_lists; i += 32) sum += lengths[i];
            sum = __reduce_add_sync(0xffffffffu, sum);
            if (n_lists <= p.beside_ctas && sum <= p.beside_tiles) {
                n_units = p.beside_ctas;
            } else if (beside) {
                griddep_wait();
                beside = false;
                for (int i = threadIdx.x; i < n_lists; i += kAttnThreads) counts[i].y = __ldcg(c.n_tokens + cache_list(i));
                __syncthreads();
            }
        }
        n_parts = attn_unit(lengths, n_lists, n_units, blockIdx.x, lane, list, part);
        if (n_parts == 0) {                                        // the whole CTA: more CTAs than parts
            griddep_wait();
            return;
        }
        n_before = n_prefix = counts[list].x;
        n_total = counts[list].y;
        if (kBeside && !beside) n_prefix = __ldcg(c.prefix_len + cache_list(list));
        fence_proxy_async_smem();                                  // the copies below write where these were read
        __syncthreads();
    }

    // This CTA's tiles are its run [s_first, n_tiles) of the list's, the prefix's and then the window's.  kBeside: numbered s = 0, 1,
    // ... n_tiles - 1, [t_first, t_first + n_early) of the prefix's whole tiles, which are there for good, and behind those every
    // n_parts-th of the others (the end of the prefix, the window), known only when the kernel ahead has completed (learn_rest).
    const int tiles_per_page = c.page_tokens / kAttnTileRows;
    const int32_t *pages = c.page_table + cache_list(list) * c.max_pages;
    const int32_t ring_row0 = kBeside ? 0 : static_cast<int32_t>(cache_list(list) * c.window);
    int t_first, n_tiles, n_early = 0;
    int32_t n_ring = 0;
    int n_pt = 0;
    {
        n_ring = c.window > 0 ? (n_total < c.window ? n_total : c.window) : 0;
        n_pt = (n_prefix + kAttnTileRows - 1) / kAttnTileRows;
        const int n_run = kBeside ? n_before / kAttnTileRows : n_pt + (n_ring + kAttnTileRows - 1) / kAttnTileRows;
        t_first = static_cast<int>(static_cast<int64_t>(n_run) * part / n_parts);
        n_tiles = static_cast<int>(static_cast<int64_t>(n_run) * (part + 1) / n_parts);
        if (kBeside) n_early = n_tiles -= t_first;
    }
    const int s_first = kBeside ? 0 : t_first;
    // kBeside, per warp, in shared memory for want of registers: what the main loop seldom needs
    // rows of the prefix's end and of the window; the list among the cache's; the rest as above.  What can be looked up here is not
    // worked out again: code that is run once is waited for (ncu: of a warp's cycles per instruction here 3.9 went by for want of
    // the next instruction, 1.8 for memory).  With page numbers by a shift where that can be, us: 36 layers x 8 sequences x 2176 rows 705 -> 693,
    // 12 x 32 x 1152 8-bit rows 356 -> 339, x 30 x 2378 531 -> 497; 12 layers in one call x 64 x 1664 507 -> 495
    enum { kTail, kRing, kCacheList, kList, kPart, kParts, kFull, kKept };
    __shared__ volatile int32_t kept_s[kAttnWarps][kKept];
    bool waited = !beside;
    auto learn_rest = [&](int32_t tokens, int32_t rows) {          // whole warp, once
        const int32_t tail = rows - kept_s[warp][kFull] * kAttnTileRows;
        const int32_t ring = c.window > 0 ? (tokens < c.window ? tokens : c.window) : 0;
        if (lane == 0) { kept_s[warp][kTail] = tail; kept_s[warp][kRing] = ring; }
        __syncwarp();
        const int n_rest = (tail + kAttnTileRows - 1) / kAttnTileRows + (ring + kAttnTileRows - 1) / kAttnTileRows;
        const int mine = kept_s[warp][kPart], all = kept_s[warp][kParts];
        n_tiles = n_early + (n_rest > mine ? (n_rest - mine + all - 1) / all : 0);
        waited = true;
    };
    // tile s >= n_early: its first row in the prefix's end or in the window, rows left there; true in the window
    auto rest_tile = [&](int s, int32_t &row, int32_t &left) -> bool {
        const int32_t tail = kept_s[warp][kTail];
        const int t = kept_s[warp][kPart] + (s - n_early) * kept_s[warp][kParts], tail_tiles = (tail + kAttnTileRows - 1) / kAttnTileRows;
        const bool ring = t >= tail_tiles;
        row = (ring ? t - tail_tiles : t) * kAttnTileRows;
        left = (ring ? kept_s[warp][kRing] : tail) - row;
        return ring;
    };
    if constexpr (kBeside) {
        if (lane == 0) {
            kept_s[warp][kList] = list;
            kept_s[warp][kCacheList] = static_cast<int32_t>(cache_list(list));
            kept_s[warp][kPart] = part;
            kept_s[warp][kParts] = n_parts;
            kept_s[warp][kFull] = n_before / kAttnTileRows;
        }
        __syncwarp();
        if (!beside) learn_rest(n_total, n_prefix);
    }

    const uint32_t my_stages = smem_base + warp * kAttnStages * kStageBytes;
    const uint32_t my_bars = bars + 8 * warp * kAttnStages;
    const uint64_t policy = l2_policy_evict_first();

    // Tile s: its number among the prefix's tiles, or -1 - its first row in the rings; kBeside only
    auto tile_at = [&](int s) -> int32_t {
        if (s < n_early) return t_first + s;
        int32_t row, left;
        if (rest_tile(s, row, left)) return -1 - (kept_s[warp][kCacheList] * c.window + row);
        return kept_s[warp][kFull] + row / kAttnTileRows;
    };
    // the page that a prefix tile is in, and its first row (in its tensor map) from there; apart, so that the loads of several
    // tiles go out together
    auto page_index = [&](int32_t t) -> int32_t { return p.tiles_shift >= 0 ? t >> p.tiles_shift : t / tiles_per_page; };
    auto page_of = [&](int32_t t) -> int32_t { return t >= 0 ? __ldcg(pages + page_index(t)) : 0; };
    auto row_of = [&](int32_t t, int32_t page) {
        return t >= 0 ? page * c.page_tokens + (t - page_index(t) * tiles_per_page) * kAttnTileRows : t;
    };
    // first row (in its tensor map) of tile s; needs the page number for prefix tiles.  kBeside: rows of the rings as -1 - row
    auto tile_row = [&](int s) -> int32_t {
        if constexpr (kBeside) {
            const int32_t t = tile_at(s);
            return row_of(t, page_of(t));
        } else {
            if (s < n_pt) {
                const int32_t pi = page_index(s), page = __ldcg(pages + pi);
                return page * c.page_tokens + (s - pi * tiles_per_page) * kAttnTileRows;
            }
            return ring_row0 + (s - n_pt) * kAttnTileRows;
        }
    };
    auto issue = [&](int s, int32_t row, int stage) {
        const uint32_t dst = my_stages + stage * kStageBytes;
        const uint32_t bar = my_bars + 8 * stage;
        const bool prefix = kBeside ? row >= 0 : s < n_pt;
        if (kBeside && !prefix) row = -1 - row;
        mbar_arrive_expect_tx(bar, kStageBytes);
        if constexpr (kFp8) {
            // a tile of 8-bit rows is one contiguous piece of memory: coordinates (0, 0, tile)
            tma_load_3d(dst, prefix ? &tmap_kpool : &tmap_kring, bar, 0, 0, row / kAttnTileRows, policy);
            tma_load_3d(dst + kTileBytes8, prefix ? &tmap_vpool : &tmap_vring, bar, 0, 0, row / kAttnTileRows, policy);
        } else {
#pragma unroll
            for (int hf = 0; hf < kHalves; ++hf) {
                tma_load_2d(dst + hf * kAttnHalfBytes, prefix ? &tmap_kpool : &tmap_kring, bar, hf * 64, row, policy);
                tma_load_2d(dst + (kHalves + hf) * kAttnHalfBytes, prefix ? &tmap_vpool : &tmap_vring, bar, hf * 64, row, policy);
            }
        }
    };

    // Fills the stages, all free, from tile s_issue on, the pages of all of them looked up together; row_next belongs to the
    // first tile not yet issued.
    int s_issue = 0;
    int32_t row_next = 0;
    auto fill = [&](int first_stage) {
        int32_t rows[kAttnStages + 1];
        if constexpr (kBeside) {
            int32_t t[kAttnStages + 1], page[kAttnStages + 1];
#pragma unroll
            for (int i = 0; i <= kAttnStages; ++i) t[i] = s_issue + i * kAttnWarps < n_tiles ? tile_at(s_issue + i * kAttnWarps) : -1;
#pragma unroll
            for (int i = 0; i <= kAttnStages; ++i) page[i] = page_of(t[i]);
#pragma unroll
            for (int i = 0; i <= kAttnStages; ++i) rows[i] = row_of(t[i], page[i]);
        } else {
#pragma unroll
            for (int i = 0; i <= kAttnStages; ++i) rows[i] = s_issue + i * kAttnWarps < n_tiles ? tile_row(s_issue + i * kAttnWarps) : 0;
        }
#pragma unroll
        for (int i = 0; i < kAttnStages; ++i)
            if (s_issue < n_tiles) {
                if (lane == 0) issue(s_issue, rows[i], (first_stage + i) % kAttnStages);
                s_issue += kAttnWarps;
            }
        row_next = rows[kAttnStages];
    };

    // the query rows of this KV head as A fragments: row g = lane / 4 (real for g < G), two packed
    // elements at columns 16 ks + 2 (lane % 4) and the same + 8.  8-bit rows: the summation index is renumbered, this lane's
    // k-step ks covers columns c D/4 + 4 ks ..+3
    const int g = lane >> 2, qc = (lane & 3) * 2;
    auto query_row = [&]() {                // of the list's first query head, in `q` and `out`
        return static_cast<int64_t>(kBeside ? static_cast<int>(kept_s[warp][kList]) : list) * p.group;
    };
    // kBeside has no registers to keep it in
    const int64_t row0 = kBeside ? 0 : query_row();
    auto load_query = [&](const uint16_t *qrow, int ks, uint32_t &lo, uint32_t &hi) {
        lo = hi = 0u;
        if (g < p.group) {
            const uint32_t *at = reinterpret_cast<const uint32_t *>(kFp8 ? qrow + (lane & 3) * (kD / 4) + ks * 4 : qrow + ks * 16 + qc);
            lo = kBeside ? __ldcg(at) : __ldg(at);                      // kBeside: read again later, past the L1
            hi = kBeside ? __ldcg(at + (kFp8 ? 1 : 4)) : __ldg(at + (kFp8 ? 1 : 4));
        }
    };
    // 8-bit rows: query rows in f16, divided by the power of two of their largest element, which is returned
    auto query_to_f16 = [&](uint32_t (&q)[kD / 16][2]) -> float {
        float qmax = 0.0f;
#pragma unroll
        for (int ks = 0; ks < kD / 16; ++ks)
            qmax = fmaxf(fmaxf(qmax, fmaxf(fabsf(bf16_lo(q[ks][0])), fabsf(bf16_hi(q[ks][0])))),
                         fmaxf(fabsf(bf16_lo(q[ks][1])), fabsf(bf16_hi(q[ks][1]))));
        qmax = fmaxf(qmax, __shfl_xor_sync(0xffffffffu, qmax, 1));
        qmax = fmaxf(qmax, __shfl_xor_sync(0xffffffffu, qmax, 2));       // the four lanes of a row hold all its elements
        uint32_t e = __float_as_uint(qmax) >> 23;                        // biased exponent (qmax >= 0)
        e = e > 253u ? 253u : e;
        const float down = __uint_as_float((254u - e) << 23);            // 2^-(e - 127)
#pragma unroll
        for (int ks = 0; ks < kD / 16; ++ks) {
            q[ks][0] = pack_f16x2(bf16_lo(q[ks][0]) * down, bf16_hi(q[ks][0]) * down);
            q[ks][1] = pack_f16x2(bf16_lo(q[ks][1]) * down, bf16_hi(q[ks][1]) * down);
        }
        return __uint_as_float(e << 23);                                 // 2^(e - 127); zero for a zero row
    };
    uint32_t qa[kD / 16][2];
    float logit_scale;                     // 8-bit rows: times the power of two taken out of this lane's query row
    auto take_query = [&]() {
        const uint16_t *qrow = p.q + ((kBeside ? query_row() : row0) + g) * kD;
#pragma unroll
        for (int ks = 0; ks < kD / 16; ++ks) load_query(qrow, ks, qa[ks][0], qa[ks][1]);
        logit_scale = p.scale_log2e;
        if constexpr (kFp8) logit_scale *= query_to_f16(qa);
    };
    // Whether the queries are no longer what they were when they were read beside the kernel ahead (the caller only promises
    // them in stream order): read again once it has completed.  Whole warp.
    auto query_changed = [&]() -> bool {
        const uint16_t *qrow = p.q + (query_row() + g) * kD;
        uint32_t diff = 0u;
        if constexpr (kFp8) {
            uint32_t q[kD / 16][2];
#pragma unroll
            for (int ks = 0; ks < kD / 16; ++ks) load_query(qrow, ks, q[ks][0], q[ks][1]);
            const float scale = p.scale_log2e * query_to_f16(q);
            diff = __float_as_uint(scale) ^ __float_as_uint(logit_scale);
#pragma unroll
            for (int ks = 0; ks < kD / 16; ++ks) diff |= (q[ks][0] ^ qa[ks][0]) | (q[ks][1] ^ qa[ks][1]);
        } else {
#pragma unroll
            for (int ks = 0; ks < kD / 16; ++ks) {
                uint32_t lo, hi;
                load_query(qrow, ks, lo, hi);
                diff |= (lo ^ qa[ks][0]) | (hi ^ qa[ks][1]);
            }
        }
        return __any_sync(0xffffffffu, diff != 0u);
    };

    // The launch behind may start when every CTA is here: everything ahead of this launch is complete and no query is read
    // any more (what follows may reuse their memory); it still finds this launch running, reading the cache and storing `out`.
    auto queries_taken = [&]() {            // whole warp, once
        uint32_t seen = 0u;
#pragma unroll
        for (int ks = 0; ks < kD / 16; ++ks) seen |= qa[ks][0] | qa[ks][1];
        seen = __reduce_or_sync(0xffffffffu, seen);                      // every lane's loads have returned
        asm volatile("" ::"r"(seen) : "memory");
        if (lane == 0 && atomicAdd(&queries_s, 1) == kAttnWarps - 1) griddep_launch_dependents();
    };
    float o[kNTiles][4];
    float m_run = 0.0f, l_run = 0.0f;
    float vref = 0.0f;                     // 8-bit rows: the largest V scale met so far; o is in units of it

    bool ok = true, again = true;          // again: from the first tile on
    int s = 0, stage = 0;
    uint32_t parity = 0;
    auto wait_for_rest = [&]() {            // whole warp: the end of the kernel ahead, and what it has left to be read
        griddep_wait();
        const int32_t li = kept_s[warp][kCacheList];
        const int32_t tokens = __ldcg(c.n_tokens + li), rows = __ldcg(c.prefix_len + li);      // on their way beside the queries
        again = query_changed();           // then all of them once more
        if (!again) queries_taken();
        learn_rest(tokens, rows);
    };
    for (;;) {
    // no copies of this warp are in flight here
    if (again) s = s_issue = s_first + warp;
    if (!kFp8 && again) take_query();      // on their way beside the page numbers
    fill(stage);
    if (again) {
        if (kFp8) take_query();
        if (kBeside && waited) queries_taken();
#pragma unroll
        for (int i = 0; i < kNTiles; ++i) o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.0f;
        m_run = -INFINITY;
        l_run = vref = 0.0f;
        again = false;
    }
    for (; s < n_tiles; s += kAttnWarps) {
        if (kBeside && !waited && s_issue < n_tiles &&
            (s_issue + kAttnWarps >= n_tiles ||
             (p.n_parts == 0 && static_cast<uint32_t>(clock()) - started > static_cast<uint32_t>(kWaitBase + (kFp8 ? kWaitTile8 : kWaitTile) * kD / 128 * n_early)))) {
            // time for the next step to start (see kWaitBase), or the last of the tiles known beside the kernel ahead is about to
            // be issued: what comes next is learnt while those in flight are worked on
            wait_for_rest();
            if (again) {                                  // no copy may be in flight then
                for (int d = s; ok && d < s_issue; d += kAttnWarps) {
                    ok = __all_sync(0xffffffffu, mbar_wait(my_bars + 8 * stage, parity, abort_flag));
                    if (++stage == kAttnStages) { stage = 0; parity ^= 1u; }
                }
                break;
            }
        }
        if (!__all_sync(0xffffffffu, mbar_wait(my_bars + 8 * stage, parity, abort_flag))) {
            ok = false;
            break;
        }
        const uint32_t sK = my_stages + stage * kStageBytes;
        const uint32_t sV = sK + (kFp8 ? kTileBytes8 : kHalves * kAttnHalfBytes);
        int32_t valid = kAttnTileRows;                    // rows of the tile, >= 1 (more than a tile's: all of them)
        if constexpr (!kBeside) {
            valid = s < n_pt ? n_prefix - s * kAttnTileRows : n_ring - (s - n_pt) * kAttnTileRows;
        } else if (s >= n_early) {
            int32_t row;
            rest_tile(s, row, valid);
        }
        if (valid < kAttnTileRows) {
            // zero the V rows past the end of the list (8-bit rows: codes and scale)
            if constexpr (kFp8) {
                const int n_units = (kAttnTileRows - valid) * (kRowBytes8 / 16);
                for (int i = lane; i < n_units; i += 32)
                    *reinterpret_cast<uint4 *>(smem + (sV - smem_base) + valid * kRowBytes8 + i * 16) = make_uint4(0u, 0u, 0u, 0u);
            } else {
                const int n_units = (kAttnTileRows - valid) * kHalves * 8;
                for (int i = lane; i < n_units; i += 32) {
                    const int r = valid + i / (kHalves * 8), rem = i % (kHalves * 8);
                    *reinterpret_cast<uint4 *>(smem + (sV - smem_base) + (rem >> 3) * kAttnHalfBytes + r * 128 + ((rem & 7) << 4)) =
                        make_uint4(0u, 0u, 0u, 0u);
                }
            }
            fence_proxy_async_smem();
            __syncwarp();
        }

        // ---- S = Q K^T: two 8-row column tiles
        float s0[4] = {0.0f, 0.0f, 0.0f, 0.0f}, s1[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        if constexpr (kFp8) {
            // rows n = lane / 4 and n + 8 of the tile, this lane's D/4 bytes of each
            const uint8_t *kt = smem + (sK - smem_base);
            const uint32_t *r0 = reinterpret_cast<const uint32_t *>(kt + g * kRowBytes8 + (lane & 3) * (kD / 4));
            const uint32_t *r1 = reinterpret_cast<const uint32_t *>(kt + (g + 8) * kRowBytes8 + (lane & 3) * (kD / 4));
            uint32_t w0[kD / 16], w1[kD / 16];
#pragma unroll
            for (int i = 0; i < kD / 64; ++i) {
                const uint4 a = reinterpret_cast<const uint4 *>(r0)[i], b = reinterpret_cast<const uint4 *>(r1)[i];
                w0[4 * i] = a.x; w0[4 * i + 1] = a.y; w0[4 * i + 2] = a.z; w0[4 * i + 3] = a.w;
                w1[4 * i] = b.x; w1[4 * i + 1] = b.y; w1[4 * i + 2] = b.z; w1[4 * i + 3] = b.w;
            }
#pragma unroll
            for (int ks = 0; ks < kD / 16; ++ks) {
                uint32_t k0, k1, k2, k3;
                e4m3x4_to_f16(w0[ks], k0, k1);
                e4m3x4_to_f16(w1[ks], k2, k3);
                mma_f16_16816(s0, qa[ks][0], 0u, qa[ks][1], 0u, k0, k1);
                mma_f16_16816(s1, qa[ks][0], 0u, qa[ks][1], 0u, k2, k3);
            }
            // the K rows' scales: this lane holds columns (rows of the tile) qc, qc + 1 of both column tiles
            s0[0] *= *reinterpret_cast<const float *>(kt + qc * kRowBytes8 + kD);
            s0[1] *= *reinterpret_cast<const float *>(kt + (qc + 1) * kRowBytes8 + kD);
            s1[0] *= *reinterpret_cast<const float *>(kt + (8 + qc) * kRowBytes8 + kD);
            s1[1] *= *reinterpret_cast<const float *>(kt + (9 + qc) * kRowBytes8 + kD);
        } else {
            const int mi = lane >> 3, r8 = lane & 7;
            const int krow = (mi >> 1) * 8 + r8;
#pragma unroll
            for (int ks = 0; ks < kD / 16; ++ks) {
                const int chunk = 2 * ks + (mi & 1);
                const uint32_t addr = sK + (chunk >> 3) * kAttnHalfBytes + krow * 128 + (((chunk & 7) ^ (krow & 7)) << 4);
                uint32_t k0, k1, k2, k3;
                ldmatrix_x4(addr, k0, k1, k2, k3);
                mma_bf16_16816(s0, qa[ks][0], 0u, qa[ks][1], 0u, k0, k1);
                mma_bf16_16816(s1, qa[ks][0], 0u, qa[ks][1], 0u, k2, k3);
            }
        }
        // ---- online softmax for row g: this lane holds columns qc, qc + 1 of both column tiles
        float v00 = s0[0] * logit_scale, v01 = s0[1] * logit_scale;
        float v10 = s1[0] * logit_scale, v11 = s1[1] * logit_scale;
        if (valid < kAttnTileRows) {
            if (qc >= valid) v00 = -INFINITY;
            if (qc + 1 >= valid) v01 = -INFINITY;
            if (8 + qc >= valid) v10 = -INFINITY;
            if (9 + qc >= valid) v11 = -INFINITY;
        }
        float mx = fmaxf(fmaxf(v00, v01), fmaxf(v10, v11));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
        const float m_new = fmaxf(m_run, mx);             // finite: row 0 of a tile is always valid
        const float alpha = fast_ex2(m_run - m_new);      // 0 on the first tile
        const float p00 = fast_ex2(v00 - m_new), p01 = fast_ex2(v01 - m_new);
        const float p10 = fast_ex2(v10 - m_new), p11 = fast_ex2(v11 - m_new);
        l_run = l_run * alpha + ((p00 + p01) + (p10 + p11));
        m_run = m_new;
        uint32_t pa0, pa2;
        if constexpr (kFp8) {
            // the V rows' scales (zero for rows past the end), relative to the largest one so far
            const uint8_t *vt = smem + (sV - smem_base);
            const float vs00 = *reinterpret_cast<const float *>(vt + qc * kRowBytes8 + kD);
            const float vs01 = *reinterpret_cast<const float *>(vt + (qc + 1) * kRowBytes8 + kD);
            const float vs10 = *reinterpret_cast<const float *>(vt + (8 + qc) * kRowBytes8 + kD);
            const float vs11 = *reinterpret_cast<const float *>(vt + (9 + qc) * kRowBytes8 + kD);
            float vmax = fmaxf(fmaxf(fabsf(vs00), fabsf(vs01)), fmaxf(fabsf(vs10), fabsf(vs11)));
            vmax = fmaxf(vmax, __shfl_xor_sync(0xffffffffu, vmax, 1));
            vmax = fmaxf(vmax, __shfl_xor_sync(0xffffffffu, vmax, 2));
            const float vref_new = fmaxf(vref, vmax);
            const float rinv = vref_new > 0.0f ? 1.0f / vref_new : 0.0f;
            const float alpha_o = alpha * (vref * rinv);
            vref = vref_new;
            // the accumulator tiles hold O^T: this lane's columns are query heads qc and qc + 1
            const float a_lo = __shfl_sync(0xffffffffu, alpha_o, qc * 4), a_hi = __shfl_sync(0xffffffffu, alpha_o, qc * 4 + 4);
#pragma unroll
            for (int i = 0; i < kNTiles; ++i) { o[i][0] *= a_lo; o[i][1] *= a_hi; o[i][2] *= a_lo; o[i][3] *= a_hi; }
            pa0 = pack_f16x2(p00 * (vs00 * rinv), p01 * (vs01 * rinv));
            pa2 = pack_f16x2(p10 * (vs10 * rinv), p11 * (vs11 * rinv));
        } else {
#pragma unroll
            for (int i = 0; i < kNTiles; ++i) { o[i][0] *= alpha; o[i][1] *= alpha; }
            pa0 = pack_bf16x2(p00, p01);
            pa2 = pack_bf16x2(p10, p11);
        }

        // ---- O += P V: two 8-column output tiles per ldmatrix
        if constexpr (kFp8) {
            // O^T[D x 8] += V^T[D x 16] P^T[16 x 8]: P as it comes out of the softmax is the B operand (k = row of the
            // tile, n = query head), V^T is the A operand.  V rows 2c, 2c+1 (k = 2c, 2c+1) and 2c+8, 2c+9 of the tile,
            // this lane's D/8 bytes of each; accumulator tile i takes bytes 2i (MMA rows 0..7) and 2i+1 (rows 8..15)
            const uint8_t *vt = smem + (sV - smem_base) + g * (kD / 8);
            uint32_t ra[kD / 32], rb[kD / 32], rc[kD / 32], rd[kD / 32];
            if constexpr (kD == 128) {
                const uint4 a = *reinterpret_cast<const uint4 *>(vt + qc * kRowBytes8);
                const uint4 b = *reinterpret_cast<const uint4 *>(vt + (qc + 1) * kRowBytes8);
                const uint4 cc = *reinterpret_cast<const uint4 *>(vt + (qc + 8) * kRowBytes8);
                const uint4 d = *reinterpret_cast<const uint4 *>(vt + (qc + 9) * kRowBytes8);
                ra[0] = a.x; ra[1] = a.y; ra[2] = a.z; ra[3] = a.w;
                rb[0] = b.x; rb[1] = b.y; rb[2] = b.z; rb[3] = b.w;
                rc[0] = cc.x; rc[1] = cc.y; rc[2] = cc.z; rc[3] = cc.w;
                rd[0] = d.x; rd[1] = d.y; rd[2] = d.z; rd[3] = d.w;
            } else {
                const uint2 a = *reinterpret_cast<const uint2 *>(vt + qc * kRowBytes8);
                const uint2 b = *reinterpret_cast<const uint2 *>(vt + (qc + 1) * kRowBytes8);
                const uint2 cc = *reinterpret_cast<const uint2 *>(vt + (qc + 8) * kRowBytes8);
                const uint2 d = *reinterpret_cast<const uint2 *>(vt + (qc + 9) * kRowBytes8);
                ra[0] = a.x; ra[1] = a.y; rb[0] = b.x; rb[1] = b.y;
                rc[0] = cc.x; rc[1] = cc.y; rd[0] = d.x; rd[1] = d.y;
            }
#pragma unroll
            for (int i = 0; i < kNTiles; ++i) {
                const uint32_t sel = (i & 1) ? 0x7362u : 0x5140u;       // bytes k, k+1 of both rows, interleaved (k = 0 or 2)
                uint32_t a0, a1, a2, a3;
                e4m3x4_to_f16(__byte_perm(ra[i >> 1], rb[i >> 1], sel), a0, a1);
                e4m3x4_to_f16(__byte_perm(rc[i >> 1], rd[i >> 1], sel), a2, a3);
                mma_f16_16816(o[i], a0, a1, a2, a3, pa0, pa2);
            }
        } else {
            const int mi = lane >> 3, r8 = lane & 7;
            const int krow = (mi & 1) * 8 + r8;
#pragma unroll
            for (int ndp = 0; ndp < kD / 16; ++ndp) {
                const int chunk = 2 * ndp + (mi >> 1);
                const uint32_t addr = sV + (chunk >> 3) * kAttnHalfBytes + krow * 128 + (((chunk & 7) ^ (krow & 7)) << 4);
                uint32_t v0, v1, v2, v3;
                ldmatrix_x4_trans(addr, v0, v1, v2, v3);
                mma_bf16_16816(o[2 * ndp], pa0, 0u, pa2, 0u, v0, v1);
                mma_bf16_16816(o[2 * ndp + 1], pa0, 0u, pa2, 0u, v2, v3);
            }
        }
        __syncwarp();                                     // all lanes are done with this stage
        if (s_issue < n_tiles) {
            if (lane == 0) issue(s_issue, row_next, stage);
            s_issue += kAttnWarps;
            row_next = s_issue < n_tiles ? tile_row(s_issue) : 0;
        }
        if (++stage == kAttnStages) { stage = 0; parity ^= 1u; }
    }
    if (!kBeside || !ok || (waited && !again)) break;
    if (!waited) wait_for_rest();          // out of the tiles known beside the kernel ahead
    }
    if (!waited) griddep_wait();                          // only if a wait ran out
    if (!ok) {
        // a wait ran out: report it, give the copies already in flight a fixed time to land, merge nothing
        if (lane == 0) {
            atomicCAS(p.status, 0, 5 /* KVZAP_ERR_TIMEOUT */);
            const long long t0 = clock64();
            while (clock64() - t0 < 2000000LL) { }
        }
        __syncwarp();
    }

    // ---- merge the warps' partial results: [warp] { m[8], l[8], O[8][kD] } in the warp's own stages
    l_run += __shfl_xor_sync(0xffffffffu, l_run, 1);
    l_run += __shfl_xor_sync(0xffffffffu, l_run, 2);
    {
        float *mine = reinterpret_cast<float *>(smem + warp * kAttnStages * kStageBytes);
        if ((lane & 3) == 0) { mine[g] = m_run; mine[8 + g] = l_run; }
#pragma unroll
        for (int i = 0; i < kNTiles; ++i) {
            if constexpr (kFp8) {           // O^T: rows are elements g D/8 + 2i (+1), columns query heads qc, qc+1; back from units of vref
                mine[16 + qc * kD + g * (kD / 8) + 2 * i] = o[i][0] * vref;
                mine[16 + (qc + 1) * kD + g * (kD / 8) + 2 * i] = o[i][1] * vref;
                mine[16 + qc * kD + g * (kD / 8) + 2 * i + 1] = o[i][2] * vref;
                mine[16 + (qc + 1) * kD + g * (kD / 8) + 2 * i + 1] = o[i][3] * vref;
            } else {
                mine[16 + g * kD + i * 8 + qc] = o[i][0];
                mine[16 + g * kD + i * 8 + qc + 1] = o[i][1];
            }
        }
    }
    __syncthreads();
    const bool failed = *abort_flag != 0;
    const int64_t out_row0 = kBeside ? query_row() : row0;
    if constexpr (kBeside) {
        list = kept_s[warp][kList];
        part = kept_s[warp][kPart];
        n_parts = kept_s[warp][kParts];
    }
    constexpr int kUnit = 16 + kAttnMaxGroup * kD;
    // the list's first unit
    const int unit0 = p.n_parts == 0 ? static_cast<int>(blockIdx.x) - part
                      : list >= p.head_lists ? p.tail_unit0 + (list - p.head_lists) * p.tail_parts : list * p.n_parts;
    float *unit = n_parts > 1 ? p.part_scratch + static_cast<int64_t>(unit0 + part) * kUnit : nullptr;
    // four elements of one query head per thread
    for (int idx = threadIdx.x; idx < p.group * (kD / 4); idx += kAttnThreads) {
        const int gq = idx / (kD / 4), d = idx % (kD / 4) * 4;
        float m_all = -INFINITY;
#pragma unroll
        for (int w = 0; w < kAttnWarps; ++w)
            m_all = fmaxf(m_all, reinterpret_cast<const float *>(smem + w * kAttnStages * kStageBytes)[gq]);
        float4 num = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        float den = 0.0f;
#pragma unroll
        for (int w = 0; w < kAttnWarps; ++w) {
            const float *wp = reinterpret_cast<const float *>(smem + w * kAttnStages * kStageBytes);
            if (wp[gq] > -INFINITY) {                       // a warp that saw no tile contributes nothing
                const float f = fast_ex2(wp[gq] - m_all);
                attn_add(num, *reinterpret_cast<const float4 *>(wp + 16 + gq * kD + d), f);
                den += wp[8 + gq] * f;
            }
        }
        if (n_parts == 1) {
            attn_store(p.out + (out_row0 + gq) * kD + d, num, failed ? 0.0f : den);      // an empty list gives zeros
        } else {
            __stcg(reinterpret_cast<float4 *>(unit + 16 + gq * kD + d), num);
            if (d == 0) {
                __stcg(unit + gq, failed ? -INFINITY : m_all);
                __stcg(unit + 8 + gq, failed ? 0.0f : den);
            }
        }
    }
    if (n_parts == 1) return;

    // ---- several CTAs per list: the one that arrives last merges all parts, in part order
    __shared__ int last_s;
    __syncthreads();
    if (threadIdx.x == 0) last_s = arrive_last(p.part_arrive + (list - p.list0), static_cast<uint32_t>(n_parts));
    __syncthreads();
    if (!last_s) return;
    const float *units = p.part_scratch + static_cast<int64_t>(unit0) * kUnit;
    constexpr int kBatch = 8;               // parts whose values are loaded together: one round trip to memory
    for (int idx = threadIdx.x; idx < p.group * (kD / 4); idx += kAttnThreads) {
        const int gq = idx / (kD / 4), d = idx % (kD / 4) * 4;
        float m_all = -INFINITY, den = 0.0f;
        float4 num = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        for (int i0 = 0; i0 < n_parts; i0 += kBatch) {
            float mv[kBatch], dv[kBatch];
            float4 nv[kBatch];
#pragma unroll
            for (int j = 0; j < kBatch; ++j) {
                const float *u = units + static_cast<int64_t>(i0 + j) * kUnit;
                const bool in = i0 + j < n_parts;
                mv[j] = in ? __ldcg(u + gq) : -INFINITY;
                dv[j] = in ? __ldcg(u + 8 + gq) : 0.0f;
                nv[j] = in ? __ldcg(reinterpret_cast<const float4 *>(u + 16 + gq * kD + d)) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            }
            float m_new = m_all;
#pragma unroll
            for (int j = 0; j < kBatch; ++j) m_new = fmaxf(m_new, mv[j]);
            if (m_all > -INFINITY && m_new > m_all) {
                const float f = fast_ex2(m_all - m_new);
                num.x *= f; num.y *= f; num.z *= f; num.w *= f;
                den *= f;
            }
            m_all = m_new;
#pragma unroll
            for (int j = 0; j < kBatch; ++j) {                          // summed in part order
                const float f = mv[j] > -INFINITY ? fast_ex2(mv[j] - m_all) : 0.0f;      // a part without tiles adds nothing
                attn_add(num, nv[j], f);
                den += dv[j] * f;
            }
        }
        attn_store(p.out + (out_row0 + gq) * kD + d, num, den);
    }
}

}  // namespace kvzap
