// MLP surrogate scoring for FEW tokens per layer (the decode step: one new token per sequence,
// Method, "KVzap" and the caption of Algorithm 1), where one 128-token tile per layer would leave
// most SMs idle and every byte of W1 has to come from HBM.
//
// n_split * k_split CTAs share one 128-token tile.  The hidden units are cut into n_split slices of
// Ns = hidden / n_split; a slice is computed by a cluster of k_split CTAs (1, 2, 4 or 8).  Each CTA of a
// cluster runs its part of the K range (so every byte of W1 is read once, and an X tile once per slice),
// and the partial pre-activation tiles are combined before the GELU: a CTA owns Ns / k_split columns of
// the slice, sends each of the others the columns of its accumulator which that one owns through
// distributed shared memory (into the receiver's pipeline stages, idle by then) and finishes its own:
// the parts in rank order, bias, GELU, its part of the second layer.  The 8 partial sums per token go to
// the cluster's first CTA (distributed shared memory, one cluster barrier).
//
// The slices of a tile meet in global memory: the first CTA of every cluster stores its 128 x 8 partial
// sums, a warp 32 rows, and counts them in; the warp that arrives last adds the parts in slice order (so the sum
// does not depend on who was last) plus b2 and writes the scores (and, if asked for, the keep bits).  Counted per warp with one
// release-and-acquire, and with all loads behind it in one round trip, what follows the last barrier of a cluster is
// one barrier less and one to two round trips less than with one arrival per cluster between two fences: 8 layers of 777 tokens, default
// context, 149.1 -> 145.9 us; four prompts in two chunks, 4 layers, 275.8 -> 273.9 us.
// How many CTAs share a tile is the host's choice by the number of tiles (see SplitLayout): what a launch
// of few tiles costs is the time in which one CTA pulls its part of X and W1, so it takes the widest layout
// whose clusters are all resident at once.  Many tiles (36 layers x 2 slices) keep clusters of two: those
// fill the machine at once, whereas clusters of four do not all find four free SMs in one GPC and leave a
// second wave.  W1 is the context's own copy, so its first tiles are fetched before the wait for the work
// ahead in the stream.
//
// Warp roles as in score_kernel: warp 0 TMA producer, warp 1 MMA issuer / TMEM owner, warps 2..9
// epilogue (TMEM lane quarter = warp % 4; the two warps of a quarter take eight columns in turn; kFew: see below).
#pragma once

#include "decode_kernels.cuh"
#include "score_kernel.cuh"

namespace kvzap {

// Decode step fused into the scoring launch (enabled != 0): while the MMAs run, the epilogue warps
// of a cluster do the cache update of the cluster's own lists -- 128 sequences x H heads of one layer,
// an equal part per CTA -- exactly as decode_update_kernel does (the token that leaves the window is
// judged by its buffered score, so nothing here needs the new scores); the cluster's first CTA puts
// the new scores into the score buffer at the very end (the last cluster of the tile to arrive).
// Consecutive steps may overlap in time (the next launch starts as SMs become free): `done[cluster]`
// counts the steps a cluster has completed, and a cluster touches the cache only after all clusters of
// its tile have published the number of the step before.  Which step a CTA is working on it learns on the
// device: it draws a ticket from a counter of its own (tile, slice, rank) before it lets the next launch be
// placed, so the CTAs that serve the same slice in consecutive launches draw consecutive numbers whatever the
// host knows -- a captured CUDA graph of steps can be replayed.
struct DecodeFuse {
    int32_t enabled;
    int32_t *ticket;                // [n_layers * tiles_per_layer][n_split][k_split]: steps started, per (slice, rank in the cluster)
    CacheView c;
    const uint4 *K_new, *V_new;     // [n_layers_call][B][H][D] bf16
    float tau;
    int32_t *done;                  // [n_layers * tiles_per_layer][n_split]
    int64_t wait_limit;             // cycles a cluster waits for the step before to be published
};

struct SplitSmemLayout {
    uint32_t a_bytes, stage_bytes, stages_end, w2s, b1s, w1s, part, recv, xpart, bars, total;
};
// The parts received from the other CTAs of the cluster ([k_split - 1][own / 4][128 rows] float4) lie over the
// stages, idle by then, and behind them the sums that the cluster's CTAs leave with its first one ([k_split][128][8]).
// b_rows: rows of W1 that a CTA stages, ns or, for CTA pairs, half of them.  x_rows (kFew; else 0): a stage holds only so many
// rows of X, and what the CTAs send one another ([k_split][x_rows][own + 4] and [k_split][x_rows][8]) has a place of its own.
// The MMAs read 128 rows all the same: those behind the staged ones are whatever lies there, within the block (see total), and
// so are their results.
__host__ __device__ inline SplitSmemLayout split_smem_layout(int ns, int n_stages, int k_split, int b_rows, int x_rows = 0)
{
    SplitSmemLayout L;
    const uint32_t own = static_cast<uint32_t>(ns / k_split), k = static_cast<uint32_t>(k_split);
    L.a_bytes = x_rows > 0 ? static_cast<uint32_t>(x_rows) * 128u : kATileBytes;
    L.stage_bytes = L.a_bytes + static_cast<uint32_t>(b_rows) * kBlockK * 2;
    L.stages_end = L.stage_bytes * n_stages;
    L.w2s = L.stages_end;
    L.b1s = L.w2s + static_cast<uint32_t>(ns) * kMaxHeads * 4;
    L.w1s = L.b1s + static_cast<uint32_t>(ns) * 4;            // first-layer row scales (8-bit inputs)
    L.part = L.w1s + static_cast<uint32_t>(ns) * 4;
    if (x_rows > 0) {
        L.recv = L.part;
        L.xpart = L.recv + k * static_cast<uint32_t>(x_rows) * (own + 4) * 4;
        L.bars = L.xpart + k * static_cast<uint32_t>(x_rows) * kMaxHeads * 4;
    } else {
        L.recv = 0;
        L.xpart = own * (k - 1) * kTileM * 4;
        L.bars = L.part + kTileM * kMaxHeads * 4;
    }
    L.total = L.bars + 256;
    const uint32_t last_read = L.stages_end - L.stage_bytes + kATileBytes;
    if (L.total < last_read) L.total = last_read;
    return L;
}
__host__ inline bool split_smem_fits(int ns, int n_stages, int k_split, int b_rows, int budget, int x_rows = 0)
{
    const SplitSmemLayout L = split_smem_layout(ns, n_stages, k_split, b_rows, x_rows);
    return static_cast<int>(L.total) <= budget &&
           (x_rows > 0 || L.xpart + static_cast<uint32_t>(k_split) * kTileM * kMaxHeads * 4 <= L.stages_end);
}

// p.group_w = p.chunk_n = Ns (the MMA's N); p.n_chunks = 1; p.acc_bufs = 1; p.n_tiles = 128-token tiles
// over all layers of the call; cluster dimension k_split, gridDim.x = n_split * k_split * p.n_tiles.
// A CTA ends up owning Ns / k_split hidden units.
// kFp8: hidden states and W1 are E4M3 bytes (K blocks of 128 codes, tcgen05.mma kind::f8f6f4); the scales
// x_scale[token] * w1_scale[hidden unit] multiply the summed pre-activation before the bias.
// kStepKind: none; or the decode step, a kernel of its own, so that the scoring of prompts and chunks carries none of its code;
// or the step directly behind an attention over the cache, which may still be running and reads it: the stores of the cache
// update wait for it, nothing before them does, and the next launch, an attention that runs beside this step, starts once the
// lists' present prefix lengths are in c.before.  That too is a kernel of its own: asked for at run time it cost the other
// steps 1 to 2 % (2 layers x 4 sequences 12.97 -> 12.70 us, 12 x 2 18.0 -> 17.8).
// kPair (prompts, not the fused step): two blocks of 128 tokens share every W1 tile.  A work tile is a pair of blocks, the
// cluster has 2 * k_split CTAs, CTA 2 r + i holds block i's rows of K part r and half of the slice's W1 rows, and its first
// one issues the MMAs of both (cta_group::2, as in score_kernel); everything behind the accumulators is per block, as without
// pairs.  A CTA then loads (128 + Ns / 2) rows per K element instead of 128 + Ns, which is what bounds this kernel.
// kFew (steps of up to kFewTokens tokens a layer): what bounds such a step is a chain of round trips and barriers, and code that is
// fetched to be run once.  A stage holds x_rows rows of X instead of 128, so that in the layouts of few layers all of a CTA's loads
// are out at once; the receive buffers lie beside the stages (no barrier before the exchange); GELU and second layer are shared out
// over all epilogue warps, a pair of hidden units of one token per thread, where one warp had 16 units of all tokens; and
// the last slice to arrive is found per warp, which then needs one round trip for partial sums, bias and ring slots.
// 4096 -> 512 -> 8, one layer a call, calls in a row, us: 1 sequence 11.7 -> 7.7, 8 12.4 -> 8.4, 16 12.7 -> 8.6, 32 13.2 -> 9.3; 8-bit, 8
// sequences 12.6 -> 8.5; 36 layers a call, 8 sequences 33.3 -> 29.3, 32 38.2 -> 35.3.  32 tokens are one lane quarter of the accumulator; more
// would need the exchange's other quarters, and their X fills the stages again.
enum SplitStep { kNoStep, kStep, kStepBehindAttention };
constexpr int kFewTokens = 32;
constexpr int kTileWarps = 4;           // arrival counters of a tile: one per lane quarter
constexpr int kFewWarps = 8;            // ... of steps of few tokens: one per four tokens
template <bool kFp8, bool kPair, SplitStep kStepKind, bool kFew>
__global__ void __maxnreg__(128)
score_split_kernel(const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ CUtensorMap tmap_w,
                   const ScoreParams p, const int n_split, const int k_split, const DecodeFuse f)
{
    constexpr int kElems = kFp8 ? 2 * kBlockK : kBlockK;         // elements per 128-byte K block
    constexpr int kCtas = kPair ? 2 : 1;
    constexpr bool kFused = kStepKind != kNoStep, kBehind = kStepKind == kStepBehindAttention;
    __shared__ int64_t fuse_dst[kFused ? 256 : 1];       // fused decode step: page row of the evicted token (-1 = dropped)
    __shared__ int64_t fuse_ring[kFused ? 256 : 1];      //                     ring row of the list's current slot (-1 = no list)
    __shared__ int32_t fuse_step;           //                     number of the step this CTA works on (its ticket)
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw_addr = smem_u32(smem_raw);
    const uint32_t pad = (1024u - (raw_addr & 1023u)) & 1023u;
    uint8_t *smem = smem_raw + pad;
    const uint32_t smem_base = raw_addr + pad;
    const int ns = p.chunk_n;
    const int n_ctas = n_split * k_split;
    static_assert(!kFew || (kFused && !kPair), "few tokens: decode steps only");
    const SplitSmemLayout L = split_smem_layout(ns, p.n_stages, k_split, ns / kCtas, kFew ? p.x_rows : 0);

    ulonglong2 *w2p = reinterpret_cast<ulonglong2 *>(smem + L.w2s);
    float *w2f = reinterpret_cast<float *>(smem + L.w2s);
    float *b1s = reinterpret_cast<float *>(smem + L.b1s);
    float *w1s = reinterpret_cast<float *>(smem + L.w1s);
    float *part = reinterpret_cast<float *>(smem + L.part);
    float *xpart = reinterpret_cast<float *>(smem + L.xpart);
    float *recv_few = reinterpret_cast<float *>(smem + L.recv);           // kFew: [k_split][x_rows][own + 4]
    const uint32_t bars = smem_base + L.bars;
    const uint32_t bar_full = bars;                      // [kMaxStages] TMA -> MMA
    const uint32_t bar_empty = bars + 8 * kMaxStages;    // [kMaxStages] MMA -> TMA
    const uint32_t bar_tfull = bars + 16 * kMaxStages;   // MMA -> epilogue
    const uint32_t bar_done = bar_tfull + 8;             // abort path only
    const uint32_t bar_pfull = bar_done + 8;             // second warp of a lane quarter -> first
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(smem + L.bars + 16 * kMaxStages + 32);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + L.bars + 16 * kMaxStages + 36);

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const uint32_t cta = cluster_cta_rank();
    const uint32_t half = cta % kCtas;                   // which block of the pair
    const uint32_t rank = cta / kCtas;                   // 0 .. k_split - 1
    const int kh = static_cast<int>(rank);               // which part of the K range
    const int nh = (static_cast<int>(blockIdx.x) / (kCtas * k_split)) % n_split;   // which slice of the hidden units
    const int pos = nh * k_split + kh;                   // this CTA among the n_ctas of its block
    const int tile = static_cast<int>(blockIdx.x) / (kCtas * n_ctas);
    const int l_rel = tile / p.tiles_per_layer;
    const int m_tile = (tile - l_rel * p.tiles_per_layer) * kCtas + static_cast<int>(half) + p.block0;
    const int part_tile = tile * kCtas + static_cast<int>(half);        // among all blocks of the launch
    const int layer = p.layer0 + l_rel;
    if constexpr (kFused) {
        // the step number, drawn before any thread of this CTA lets the next launch be placed: a CTA of that launch
        // starts only after every CTA of this one has passed the instruction below, hence after this draw
        if (threadIdx.x == 0)
            fuse_step = atomicAdd(f.ticket + ((layer * p.tiles_per_layer + m_tile) * n_split + nh) * k_split + kh, 1);
        __syncthreads();
    }
    if (!p.late_trigger && !kBehind) griddep_launch_dependents();
    if constexpr (kFew) cluster_arrive();                // waited for before the first store to another CTA: it runs by then
    const int own_n = ns / k_split;                      // accumulator columns this CTA finishes
    const int own_c0 = kh * own_n;                       // the first of them
    const int j_first = nh * ns + own_c0;                // = first hidden unit of this CTA

    if (threadIdx.x == 0) {
        for (int s = 0; s < kMaxStages; ++s) {
            mbar_init(bar_full + 8 * s, 1);
            mbar_init(bar_empty + 8 * s, 1);
        }
        mbar_init(bar_tfull, 1);
        mbar_init(bar_done, 1);
        mbar_init(bar_pfull, 4);
        *abort_flag = 0;
        fence_mbar_init();
        prefetch_tensormap(&tmap_x);
        prefetch_tensormap(&tmap_w);
    }
    const int k_blocks = p.d_model / kElems / k_split;   // K blocks of this CTA
    const int kb_first = kh * k_blocks;
    const uint64_t pol_x = l2_policy_evict_last();        // the other CTAs of the cluster read the same X tile
    const uint64_t pol_w = l2_policy_evict_first();       // every W1 byte is read once per step
    const int w_row = layer * p.w_rows + nh * ns + static_cast<int>(half) * (ns / kCtas);
    const int row0 = m_tile * kTileM;
    const int n_pre = k_blocks < p.n_stages ? k_blocks : p.n_stages;
    // The first loads go out before the CTA-wide barrier below (TMEM allocation, the other warps): the
    // stages are empty and their barriers were initialised by this warp's lane 0 just above (a pair: those of its first
    // CTA, which count the copies of both).  W1 is the context's own copy and is not written by anything that may still be
    // running ahead of this launch.
    if constexpr (kPair) cluster_sync_all();
    uint32_t full0 = bar_full;                           // the barriers that this CTA's copies complete on
    if constexpr (kPair) full0 = map_to_cta(bar_full, cta - half);
    auto load_w = [&](uint32_t st, uint32_t sa, int kb) {
        if constexpr (kPair) {
            if (half == 0) mbar_arrive_expect_tx(bar_full + 8 * st, 2u * L.stage_bytes);
            tma_load_3d_pair(sa + L.a_bytes, &tmap_w, full0 + 8 * st, 0, w_row, kb_first + kb, pol_w);
        } else {
            mbar_arrive_expect_tx(bar_full + 8 * st, L.stage_bytes);
            tma_load_3d(sa + L.a_bytes, &tmap_w, bar_full + 8 * st, 0, w_row, kb_first + kb, pol_w);
        }
    };
    auto load_x = [&](uint32_t st, uint32_t sa, int kb) {
        if constexpr (kPair) tma_load_3d_pair(sa, &tmap_x, full0 + 8 * st, (kb_first + kb) * kElems, row0, l_rel, pol_x);
        else tma_load_3d(sa, &tmap_x, bar_full + 8 * st, (kb_first + kb) * kElems, row0, l_rel, pol_x);
    };
    if (warp == 0) {
        __syncwarp();
        if (elect_one())
            for (int kb = 0; kb < n_pre; ++kb) load_w(static_cast<uint32_t>(kb), smem_base + kb * L.stage_bytes, kb);
        __syncwarp();
    }
    if (warp == 1) {
        if constexpr (kPair) {
            tmem_alloc_pair(smem_u32(const_cast<uint32_t *>(tmem_slot)), static_cast<uint32_t>(p.tmem_cols));
            tmem_relinquish_pair();
        } else {
            tmem_alloc(smem_u32(const_cast<uint32_t *>(tmem_slot)), static_cast<uint32_t>(p.tmem_cols));
            tmem_relinquish();
        }
    }
    // unless the caller vouches for the producers of its inputs, nothing of them is read before the work
    // ahead in the stream has completed (every thread waits: the loads below are issued by several warps)
    if (p.wait_before_load) griddep_wait();
    if (p.late_trigger) griddep_launch_dependents();     // whatever starts now finds all work ahead of this launch complete
    if (kBehind && warp >= 2) {
        // the present length of this CTA's lists (those of the cache update below), in memory before the next launch starts
        const CacheView &c = f.c;
        const int etid = threadIdx.x - 64;
        const int64_t seqs_left = static_cast<int64_t>(c.n_seqs) - static_cast<int64_t>(m_tile) * kTileM;
        const int tile_seqs = seqs_left < kTileM ? static_cast<int>(seqs_left) : kTileM;
        const int rows_per_cta = (tile_seqs + n_ctas - 1) / n_ctas;
        const int b_loc = pos * rows_per_cta + etid / kMaxHeads, h = etid % kMaxHeads;
        if (etid < rows_per_cta * kMaxHeads && b_loc < tile_seqs && h < c.n_heads) {
            const int64_t li = ((static_cast<int64_t>(m_tile) * kTileM + b_loc) * c.n_layers + layer) * c.n_heads + h;
            c.before[li] = __ldcg(c.prefix_len + li);
            __threadfence();
        }
        named_barrier_sync(1, 256);
        if (etid == 0) griddep_launch_dependents();
    }
    if (warp == 0) {
        __syncwarp();
        if (elect_one())
            for (int kb = 0; kb < n_pre; ++kb) load_x(static_cast<uint32_t>(kb), smem_base + kb * L.stage_bytes, kb);
        __syncwarp();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = *tmem_slot;

    if (warp == 0) {
        // ------------------------------------------------------------ TMA producer (from the stage after those)
        const bool elected = elect_one();
        uint32_t st = n_pre == p.n_stages ? 0u : static_cast<uint32_t>(n_pre);
        uint32_t st_par = n_pre == p.n_stages ? 0u : 1u;
        uint32_t sa = smem_base + st * L.stage_bytes;
        bool ok = true;
        for (int kb = n_pre; kb < k_blocks; ++kb) {
            if (!__all_sync(0xffffffffu, mbar_wait(bar_empty + 8 * st, st_par, abort_flag))) {
                ok = false;
                break;
            }
            if (elected) {
                load_w(st, sa, kb);
                load_x(st, sa, kb);
            }
            __syncwarp();
            sa += L.stage_bytes;
            if (++st == static_cast<uint32_t>(p.n_stages)) { st = 0; st_par ^= 1u; sa = smem_base; }
        }
        if (!ok && lane == 0) {
            // abort path: give the copies already in flight a fixed time to land before the CTA exits
            const long long t0 = clock64();
            while (clock64() - t0 < 2000000LL) { }
        }
    } else if (warp == 1 && half == 0) {
        // ------------------------------------------------------------ MMA issuer (a pair: its first CTA)
        const uint32_t idesc = kFp8 ? umma_idesc_e4m3_f32(kTileM * kCtas, static_cast<uint32_t>(ns))
                                    : umma_idesc_bf16_f32(kTileM * kCtas, static_cast<uint32_t>(ns));
        const uint16_t both = static_cast<uint16_t>(3u << cta);
        const uint64_t desc0 = umma_desc_k_major_sw128(smem_base);
        const uint32_t desc_hi = static_cast<uint32_t>(desc0 >> 32);
        const uint32_t desc_lo0 = static_cast<uint32_t>(desc0);
        const uint32_t stage_units = L.stage_bytes >> 4;
        const bool elected = elect_one();
        uint32_t st = 0, st_par = 0, a_lo = desc_lo0;
        bool ok = true;
        for (int kb = 0; kb < k_blocks; ++kb) {
            if (!__all_sync(0xffffffffu, mbar_wait(bar_full + 8 * st, st_par, abort_flag))) {
                ok = false;
                break;
            }
            tc_fence_after_sync();
            if (elected) {
                issue_k_block<kPair, 1, kFp8>(tmem_base, a_lo, a_lo + (L.a_bytes >> 4), desc_hi, 0, 0, idesc, kb == 0);
                if constexpr (kPair) umma_commit_pair(bar_empty + 8 * st, both);
                else umma_commit(bar_empty + 8 * st);
            }
            __syncwarp();
            a_lo += stage_units;
            if (++st == static_cast<uint32_t>(p.n_stages)) { st = 0; st_par ^= 1u; a_lo = desc_lo0; }
        }
        if (ok && elected) {
            if constexpr (kPair) umma_commit_pair(bar_tfull, both);
            else umma_commit(bar_tfull);
        }
        __syncwarp();
        if (!ok && elected) {
            if constexpr (kPair) umma_commit_pair(bar_done, static_cast<uint16_t>(1u << cta));
            else umma_commit(bar_done);
            const long long t0 = clock64();
            while (!mbar_try_wait(bar_done, 0))
                if (clock64() - t0 > KVZAP_WAIT_LIMIT_CYCLES / 16) break;
        }
    }

    // ------------------------------------------------------------ epilogue (warps 2..9)
    const bool epi = warp >= 2;
    const int q = warp & 3;                 // TMEM lane quarter
    const int hsel = (warp - 2) >> 2;       // which of the two warps of that quarter
    const int row = q * 32 + lane;
    const uint32_t t_row = tmem_base + (static_cast<uint32_t>(q * 32) << 16);
    bool ok = true;
    // ---- the cache update of this CTA's lists: what moves where, then the rows
    int64_t li = -1;
    int32_t n_list = 0, prefix = 0, page = -1;
    int rows_per_cta = 0;
    auto update_plan = [&]() {
        if constexpr (kFused) {
            const CacheView &c = f.c;
            const int etid = threadIdx.x - 64;
            const int cid = layer * p.tiles_per_layer + m_tile;
            if (etid < n_split) {
                const long long t0 = clock64();
                const int32_t expect = fuse_step;
                while (ld_acquire_gpu(f.done + cid * n_split + etid) != expect) {
                    if (clock64() - t0 > f.wait_limit) { *abort_flag = 1; break; }
                }
            }
            named_barrier_sync(1, 256);
            const bool go = *abort_flag == 0;
            const int64_t seqs_left = static_cast<int64_t>(c.n_seqs) - static_cast<int64_t>(m_tile) * kTileM;
            const int tile_seqs = seqs_left < kTileM ? static_cast<int>(seqs_left) : kTileM;
            rows_per_cta = (tile_seqs + n_ctas - 1) / n_ctas;
            // one thread per list: which row leaves, where it goes, which slot the new token takes
            {
                const int b_loc = pos * rows_per_cta + etid / kMaxHeads, h = etid % kMaxHeads;
                const int64_t b = static_cast<int64_t>(m_tile) * kTileM + b_loc;
                int64_t dst = -1, ring = -1;
                int32_t n = 0, idx = 0;
                if (go && etid < rows_per_cta * kMaxHeads && b_loc < tile_seqs && h < c.n_heads && c.active[b] != 0) {
                    li = (b * c.n_layers + layer) * c.n_heads + h;
                    // two round trips to memory instead of four: both counters first, then the score of
                    // the slot's old token and the page the prefix ends in, whether or not it will be needed
                    n = __ldcg(c.n_tokens + li);
                    idx = __ldcg(c.prefix_len + li);
                    const int slot = n % c.window;
                    ring = li * c.window + slot;
                    const int page_i = idx / c.page_tokens, in_page = idx % c.page_tokens;
                    const bool full = n >= c.window;
                    const float s_old = full ? __ldcg(c.score_ring + ring) : 0.0f;
                    const int32_t page_old =
                        full && in_page != 0 && page_i < c.max_pages ? __ldcg(c.page_table + li * c.max_pages + page_i) : -1;
                    if (full && s_old >= f.tau) {
                        if (page_i >= c.max_pages) {
                            atomicCAS(p.status, 0, 4 /* KVZAP_ERR_OOM_PAGES */);
                        } else if (in_page == 0) {
                            page = cache_take_page(c, p.status);
                        } else {
                            page = page_old;
                        }
                        if (page >= 0) dst = static_cast<int64_t>(page) * c.page_tokens + in_page;
                    }
                }
                n_list = n;
                prefix = idx;
                fuse_dst[etid] = dst;
                fuse_ring[etid] = ring;
            }
            named_barrier_sync(1, 256);
        }
    };
    auto update_rows = [&]() {
        if constexpr (kFused) {
            const CacheView &c = f.c;
            const int etid = threadIdx.x - 64;
            bool counted = false;                            // every thread, once, before its first store to the cache
            auto count = [&]() {
                if (kBehind) griddep_wait();
                if (li >= 0) {
                    if (page >= 0) {
                        if (prefix % c.page_tokens == 0) c.page_table[li * c.max_pages + prefix / c.page_tokens] = page;
                        c.prefix_len[li] = prefix + 1;
                    }
                    c.n_tokens[li] = n_list + 1;
                }
                counted = true;
            };
            // rows: 16 lanes per list, kLists lists at a time; a lane loads the (old row, new row) pairs of all
            // of them before it stores any of them, so that their round trips to memory overlap
            {
                constexpr int kLists = 2;
                const int grp = etid >> 4, l16 = etid & 15;
                const int n_lists = rows_per_cta * kMaxHeads;
                for (int j0 = grp; j0 < n_lists; j0 += 16 * kLists) {
                    int64_t ring[kLists], dst[kLists], src[kLists];
#pragma unroll
                    for (int i = 0; i < kLists; ++i) {
                        const int j = j0 + 16 * i;
                        ring[i] = j < n_lists ? fuse_ring[j] : -1;
                        dst[i] = j < n_lists ? fuse_dst[j] : -1;
                        const int b_loc = pos * rows_per_cta + j / kMaxHeads, h = j % kMaxHeads;
                        const int64_t b = static_cast<int64_t>(m_tile) * kTileM + b_loc;
                        src[i] = ((static_cast<int64_t>(l_rel) * c.n_seqs + b) * c.n_heads + h) * c.row_units;
                        ring[i] *= c.row_units;           // stays negative where there is no list
                        dst[i] *= c.row_units;
                    }
                    for (int u = l16; u < c.row_units; u += 16) {
                        uint4 ko[kLists], vo[kLists], kn[kLists], vn[kLists];
#pragma unroll
                        for (int i = 0; i < kLists; ++i) {
                            if (ring[i] >= 0 && dst[i] >= 0) {
                                ko[i] = __ldcg(c.k_ring + ring[i] + u);
                                vo[i] = __ldcg(c.v_ring + ring[i] + u);
                            }
                            if (ring[i] >= 0) {
                                kn[i] = __ldg(f.K_new + src[i] + u);
                                vn[i] = __ldg(f.V_new + src[i] + u);
                            }
                        }
                        if (!counted) count();
#pragma unroll
                        for (int i = 0; i < kLists; ++i) {
                            if (ring[i] >= 0 && dst[i] >= 0) {
                                c.k_pool[dst[i] + u] = ko[i];
                                c.v_pool[dst[i] + u] = vo[i];
                            }
                            if (ring[i] >= 0) {
                                c.k_ring[ring[i] + u] = kn[i];
                                c.v_ring[ring[i] + u] = vn[i];
                            }
                        }
                    }
                }
            }
            if (!counted) count();
        }
    };
    if (epi) {
        // this CTA's slice of b1 and W2 (pairs of hidden units, see mlp_columns)
        const int etid = threadIdx.x - 64;
        const float *w2g = p.w2t + (static_cast<int64_t>(layer) * p.n_hidden + j_first) * kMaxHeads;
        const float *b1g = p.b1 + static_cast<int64_t>(layer) * p.n_hidden + j_first;
        for (int i = etid; i < own_n * kMaxHeads; i += 256) {
            const int j = i >> 3, h = i & 7;
            w2f[kFew ? i : (((j >> 1) * kMaxHeads + h) << 1) + (j & 1)] = __ldg(w2g + i);
        }
        for (int i = etid; i < own_n; i += 256) b1s[i] = __ldg(b1g + i);
        if constexpr (kFp8)
            for (int i = etid; i < own_n; i += 256) w1s[i] = __ldg(p.w1_scale + static_cast<int64_t>(layer) * p.n_hidden + j_first + i);
        named_barrier_sync(1, 256);
        // under the MMAs; the rows of a step behind an attention, for which they wait, when all else of this CTA is done (kFew)
        update_plan();
        if constexpr (!(kFew && kBehind)) update_rows();
        ok = mbar_wait(bar_tfull, 0, abort_flag);
        tc_fence_after_sync();
    }
    const int n16 = own_n >> 4;             // 16-column chunks this CTA owns (and as many it sends to each of the others)
    if constexpr (kFew) {
        // all tokens lie in the first lane quarter: its two warps send every CTA of the cluster, this one too, its columns
        const int x_rows = p.x_rows, pitch = own_n + 4;
        cluster_wait();
        if (epi && q == 0 && ok) {
            for (int i = hsel; i < k_split * n16; i += 2) {
                const uint32_t c = static_cast<uint32_t>(i % n16);
                const uint32_t to = (rank + static_cast<uint32_t>(i / n16)) % static_cast<uint32_t>(k_split);
                uint32_t r[16];
                tmem_ld_x16(t_row + to * own_n + c * 16, r);
                tmem_wait_ld();
                reg_fence16(r);
                const uint32_t dst = map_to_cta(smem_base + L.recv + ((rank * x_rows + lane) * pitch + c * 16) * 4, to);
                if (lane < x_rows) {
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        st_shared_cluster_v4(dst + 16 * j, __uint_as_float(r[4 * j]), __uint_as_float(r[4 * j + 1]),
                                             __uint_as_float(r[4 * j + 2]), __uint_as_float(r[4 * j + 3]));
                }
            }
        }
        tc_fence_before_sync();
        cluster_sync_all();                                     // every part has arrived
        const int token = (warp - 2) * 4 + (lane >> 3), pair = lane & 7;
        if (epi && (warp - 2) * 4 < x_rows) {
            float acc[kMaxHeads];
#pragma unroll
            for (int h = 0; h < kMaxHeads; ++h) acc[h] = 0.0f;
            float sx = 1.0f;
            if constexpr (kFp8)
                if (p.x_scale != nullptr && token < p.n_tokens) sx = __ldg(p.x_scale + static_cast<int64_t>(l_rel) * p.n_tokens + token);
#pragma unroll 1
            for (int j = 2 * pair; ok && j < own_n; j += 16) {
                float z0 = 0.0f, z1 = 0.0f;                     // the parts in rank order
#pragma unroll 4
                for (int part_i = 0; part_i < k_split; ++part_i) {
                    const float2 o = *reinterpret_cast<const float2 *>(recv_few + (part_i * x_rows + token) * pitch + j);
                    z0 += o.x;
                    z1 += o.y;
                }
                const float2 b = *reinterpret_cast<const float2 *>(b1s + j);
                if constexpr (kFp8) {
                    const float2 sw = *reinterpret_cast<const float2 *>(w1s + j);
                    z0 = fmaf(z0, sw.x * sx, b.x);
                    z1 = fmaf(z1, sw.y * sx, b.y);
                } else {
                    z0 += b.x;
                    z1 += b.y;
                }
                float g0, g1;
                f2_unpack(gelu_pair(f2_pack(z0, z1)), g0, g1);
                const float4 *w = reinterpret_cast<const float4 *>(w2f + j * kMaxHeads);
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const float4 wa = w[i], wb = w[2 + i];
                    acc[4 * i] = fmaf(g1, wb.x, fmaf(g0, wa.x, acc[4 * i]));
                    acc[4 * i + 1] = fmaf(g1, wb.y, fmaf(g0, wa.y, acc[4 * i + 1]));
                    acc[4 * i + 2] = fmaf(g1, wb.z, fmaf(g0, wa.z, acc[4 * i + 2]));
                    acc[4 * i + 3] = fmaf(g1, wb.w, fmaf(g0, wa.w, acc[4 * i + 3]));
                }
            }
            // the sums over a token's eight lanes; lane h of them ends up with head h
#pragma unroll
            for (int half_n = 4; half_n > 0; half_n >>= 1) {
                const bool up = pair & half_n;
#pragma unroll
                for (int i = 0; i < half_n; ++i) {
                    const float got = __shfl_xor_sync(0xffffffffu, up ? acc[i] : acc[half_n + i], half_n);
                    acc[i] = (up ? acc[half_n + i] : acc[i]) + got;
                }
            }
            st_shared_cluster_u32(map_to_cta(smem_base + L.xpart + ((rank * x_rows + token) * kMaxHeads + pair) * 4, 0), __float_as_uint(acc[0]));
        }
        if (epi && kBehind) update_rows();
    } else {
        // lanes of a warp whose 32 tokens all lie past the input take no part in the exchange and the second layer
        const bool rows_live = ok && static_cast<int64_t>(row0) + q * 32 < p.n_tokens;
        float4 *recv = reinterpret_cast<float4 *>(smem);          // [k_split - 1][own_n / 4][128 rows] float4, over the idle stages
        if (k_split > 1) {
            // every CTA's MMAs are complete once all have passed this barrier: the stages may be overwritten
            tc_fence_before_sync();
            cluster_sync_all();
            if (epi && rows_live) {
                for (int i = hsel; i < (k_split - 1) * n16; i += 2) {
                    const uint32_t c = static_cast<uint32_t>(i % n16);
                    const uint32_t to = (rank + 1u + static_cast<uint32_t>(i / n16)) % static_cast<uint32_t>(k_split);
                    const uint32_t slot = rank < to ? rank : rank - 1u;         // the receiver's parts in rank order, itself left out
                    const uint32_t dst0 = map_to_cta(smem_base, to * kCtas + half) + (slot * (static_cast<uint32_t>(own_n) >> 2) + c * 4) * kTileM * 16;
                    uint32_t r[16];
                    tmem_ld_x16(t_row + to * own_n + c * 16, r);
                    tmem_wait_ld();
                    reg_fence16(r);
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        st_shared_cluster_v4(dst0 + (static_cast<uint32_t>(j) * kTileM + row) * 16,
                                             __uint_as_float(r[4 * j]), __uint_as_float(r[4 * j + 1]),
                                             __uint_as_float(r[4 * j + 2]), __uint_as_float(r[4 * j + 3]));
                }
            }
            cluster_sync_all();                                     // the others' parts have arrived
        }
        // adds what the other CTAs of the cluster sent for 8-column piece c of this CTA's columns
        auto add_received = [&](uint32_t (&r)[8], int c) {
#pragma unroll 1
            for (int part_i = 0; part_i < k_split - 1; ++part_i) {
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const float4 o = recv[(part_i * (own_n >> 2) + c * 2 + i) * kTileM + row];
                    r[4 * i] = __float_as_uint(__uint_as_float(r[4 * i]) + o.x);
                    r[4 * i + 1] = __float_as_uint(__uint_as_float(r[4 * i + 1]) + o.y);
                    r[4 * i + 2] = __float_as_uint(__uint_as_float(r[4 * i + 2]) + o.z);
                    r[4 * i + 3] = __float_as_uint(__uint_as_float(r[4 * i + 3]) + o.w);
                }
            }
        };
        if (epi) {
            uint64_t acc[kMaxHeads];
#pragma unroll
            for (int h = 0; h < kMaxHeads; ++h) acc[h] = 0ull;
            if (rows_live) {
                // the two warps of a lane quarter take eight columns in turn; not unrolled: what is run once per launch waits for
                // its instructions (chunks of four prompts, 4 layers, 245.5 -> 241.9 us; two prompts of 4000 tokens 113.0 -> 110.7)
                uint32_t r[8];
                uint64_t sx2 = 0ull;                                   // 8-bit inputs: this row's token scale, twice
                if constexpr (kFp8) {
                    float sx = 1.0f;
                    if (p.x_scale != nullptr && row0 + row < p.n_tokens)
                        sx = __ldg(p.x_scale + static_cast<int64_t>(l_rel) * p.n_tokens + row0 + row);
                    sx2 = f2_pack(sx, sx);
                }
#pragma unroll 1
                for (int c = hsel; c < 2 * n16; c += 2) {
                    tmem_ld_x8(t_row + own_c0 + c * 8, r);
                    tmem_wait_ld();
                    reg_fence8(r);
                    add_received(r, c);
                    if constexpr (kFp8) mlp_columns_scaled<8>(r, c * 8, b1s, w1s, sx2, w2p, acc);
                    else mlp_columns<8>(r, c * 8, b1s, w2p, acc);
                }
            }
            float s[kMaxHeads];
#pragma unroll
            for (int h = 0; h < kMaxHeads; ++h) {
                float lo, hi;
                f2_unpack(acc[h], lo, hi);
                s[h] = lo + hi;
            }
            if (hsel == 1) {
                float4 *dst = reinterpret_cast<float4 *>(part + row * kMaxHeads);
                dst[0] = make_float4(s[0], s[1], s[2], s[3]);
                dst[1] = make_float4(s[4], s[5], s[6], s[7]);
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_pfull);
            } else {
                mbar_wait(bar_pfull, 0, abort_flag);
                const float4 *src = reinterpret_cast<const float4 *>(part + row * kMaxHeads);
                const float4 pa = src[0], pb = src[1];
                s[0] += pa.x; s[1] += pa.y; s[2] += pa.z; s[3] += pa.w;
                s[4] += pb.x; s[5] += pb.y; s[6] += pb.z; s[7] += pb.w;
                // hand this CTA's partial sums to its cluster's first CTA: xpart[rank][row][8]
                const uint32_t dst = map_to_cta(smem_base + L.xpart + (rank * kTileM + row) * kMaxHeads * 4, half);
                st_shared_cluster_v4(dst, s[0], s[1], s[2], s[3]);
                st_shared_cluster_v4(dst + 16, s[4], s[5], s[6], s[7]);
            }
        }
    }

    tc_fence_before_sync();
    // every thread of every CTA of the cluster arrives here (all waits above are bounded); after it the
    // partial sums of all CTAs are visible in the first CTA's shared memory
    cluster_sync_all();
    if (threadIdx.x == 0 && *abort_flag) atomicCAS(p.status, 0, 5 /* KVZAP_ERR_TIMEOUT */);
    if (warp == 1) {
        tc_fence_after_sync();
        if constexpr (kPair) tmem_dealloc_pair(tmem_base, static_cast<uint32_t>(p.tmem_cols));
        else tmem_dealloc(tmem_base, static_cast<uint32_t>(p.tmem_cols));
    }
    // If this launch was allowed to start before the kernel ahead of it had finished (consecutive decode
    // steps), it still completes after it: every thread waits here.
    griddep_wait();
    if constexpr (kFew) {
        // ---------------------------------------------------------- first CTA of the cluster: the slice's sums, a (token, head) per thread
        if (rank != 0 || warp < 2) return;
        const int w8 = warp - 2, token = w8 * 4 + (lane >> 3), head = lane & 7;
        const int done_i = layer * n_split + nh;
        if (w8 * 4 < p.x_rows) {
            float sum = 0.0f;
            for (int r = 0; r < k_split; ++r) sum += xpart[(r * p.x_rows + token) * kMaxHeads + head];
            bool last = true;
            const float *parts = p.split_part + static_cast<int64_t>(part_tile) * n_split * kTileM * kMaxHeads + token * kMaxHeads + head;
            if (n_split > 1) {
                // whichever slice brings a warp's tokens in last finishes them
                __stcg(const_cast<float *>(parts) + static_cast<int64_t>(nh) * kTileM * kMaxHeads, sum);
                last = arrive_last_warp(p.split_arrive + part_tile * kFewWarps + w8, static_cast<uint32_t>(n_split));
            }
            const CacheView &c = f.c;
            if (last && token < p.n_tokens && head < c.n_heads) {
                // all slices have arrived, so every CTA of the tile has counted its lists: one round trip for all of it
                const int64_t list = (static_cast<int64_t>(token) * c.n_layers + layer) * c.n_heads + head;
                const int32_t n = __ldcg(c.n_tokens + list);
                const bool live = c.active[token] != 0;
                float v = __ldg(p.b2 + layer * kMaxHeads + head);
                if (n_split > 1) {
                    sum = 0.0f;                                 // in slice order, whoever was last
#pragma unroll 4
                    for (int r = 0; r < n_split; ++r) sum += __ldcg(parts + static_cast<int64_t>(r) * kTileM * kMaxHeads);
                }
                v += sum;
                if (*abort_flag == 0 && live) c.score_ring[list * c.window + (n - 1) % c.window] = v;
                if (p.scores != nullptr) p.scores[(static_cast<int64_t>(l_rel) * p.n_tokens + token) * p.n_heads + head] = v;
            }
        }
        named_barrier_sync(1, 256);
        if (threadIdx.x == 64 && *abort_flag == 0) st_release_gpu(f.done + done_i, fuse_step + 1);
        return;
    }
    if (rank != 0 || warp < 2 || warp >= 6 || m_tile >= p.blocks_per_layer) return;

    // ------------------------------------------------------------ first CTA of the cluster: the slice's sums
    {
        float s[kMaxHeads];
#pragma unroll
        for (int h = 0; h < kMaxHeads; ++h) s[h] = 0.0f;
        for (int r = 0; r < k_split; ++r) {
            const float4 *src = reinterpret_cast<const float4 *>(xpart + (r * kTileM + row) * kMaxHeads);
            const float4 pa = src[0], pb = src[1];
            s[0] += pa.x; s[1] += pa.y; s[2] += pa.z; s[3] += pa.w;
            s[4] += pb.x; s[5] += pb.y; s[6] += pb.z; s[7] += pb.w;
        }
        const int64_t t = static_cast<int64_t>(m_tile) * kTileM + row;
        const bool valid = t < p.n_tokens;
        bool last = true;
        float4 *parts = reinterpret_cast<float4 *>(p.split_part + (static_cast<int64_t>(part_tile) * n_split * kTileM + row) * kMaxHeads);
        constexpr int kSlice = kTileM * kMaxHeads / 4;
        if (n_split > 1) {
            // the slices meet in global memory; of each quarter of the rows, whoever brings it in last finishes it
            __stcg(parts + static_cast<int64_t>(nh) * kSlice, make_float4(s[0], s[1], s[2], s[3]));
            __stcg(parts + static_cast<int64_t>(nh) * kSlice + 1, make_float4(s[4], s[5], s[6], s[7]));
            last = arrive_last_warp(p.split_arrive + part_tile * kTileWarps + q, static_cast<uint32_t>(n_split));
        }
        // the new token's scores go into the slot it took: n_tokens was advanced by the list's CTA, and those of the tile have all
        // arrived.  All loads before the first use of one: one round trip
        int32_t n_new[kMaxHeads];
        bool live = false;
        if constexpr (kFused) {
            const CacheView &c = f.c;
            if (last && valid) {
                live = c.active[t] != 0;
#pragma unroll
                for (int h = 0; h < kMaxHeads; ++h)
                    n_new[h] = h < c.n_heads ? __ldcg(c.n_tokens + (t * c.n_layers + layer) * c.n_heads + h) : 1;
            }
        }
        if (last && n_split > 1) {
#pragma unroll
            for (int h = 0; h < kMaxHeads; ++h) s[h] = 0.0f;
            for (int r = 0; r < n_split; ++r) {                 // in slice order, whoever was last
                const float4 pa = __ldcg(parts + static_cast<int64_t>(r) * kSlice), pb = __ldcg(parts + static_cast<int64_t>(r) * kSlice + 1);
                s[0] += pa.x; s[1] += pa.y; s[2] += pa.z; s[3] += pa.w;
                s[4] += pb.x; s[5] += pb.y; s[6] += pb.z; s[7] += pb.w;
            }
        }
#pragma unroll
        for (int h = 0; h < kMaxHeads; ++h) s[h] += __ldg(p.b2 + layer * kMaxHeads + h);
        if constexpr (kFused) {
            const CacheView &c = f.c;
            if (live && *abort_flag == 0) {
                const int64_t li0 = (t * c.n_layers + layer) * c.n_heads;
#pragma unroll
                for (int h = 0; h < kMaxHeads; ++h)
                    if (h < c.n_heads) c.score_ring[(li0 + h) * c.window + (n_new[h] - 1) % c.window] = s[h];
            }
            // this cluster's part of the step is complete
            named_barrier_sync(2, 128);
            if (threadIdx.x == 64 && *abort_flag == 0)
                st_release_gpu(f.done + (layer * p.tiles_per_layer + m_tile) * n_split + nh, fuse_step + 1);
        }
        if (!last) return;
        if (valid && p.scores != nullptr) {
            float *dst = p.scores + (static_cast<int64_t>(l_rel) * p.n_tokens + t) * p.n_heads;
            if (p.n_heads == kMaxHeads) {
                reinterpret_cast<float4 *>(dst)[0] = make_float4(s[0], s[1], s[2], s[3]);
                reinterpret_cast<float4 *>(dst)[1] = make_float4(s[4], s[5], s[6], s[7]);
            } else {
#pragma unroll
                for (int h = 0; h < kMaxHeads; ++h)
                    if (h < p.n_heads) dst[h] = s[h];
            }
        }
        if (p.maskbits != nullptr) {
            bool in_window = false;
            if (valid) {
                int64_t seq_end = p.n_tokens;
                if (p.cu_seqlens != nullptr && p.n_seqs > 1)
                    seq_end = __ldg(p.cu_seqlens + seq_of_token(p.cu_seqlens, p.n_seqs, t) + 1);
                in_window = t >= seq_end - static_cast<int64_t>(p.window);
            }
            uint32_t my_word = 0;
#pragma unroll
            for (int h = 0; h < kMaxHeads; ++h) {
                const bool keep = valid && (in_window ? p.window_keep != 0 : s[h] >= p.tau);
                const uint32_t word = __ballot_sync(0xffffffffu, keep);
                if (lane == h) my_word = word;
            }
            if (lane < p.n_heads)
                p.maskbits[(static_cast<int64_t>(l_rel) * p.n_heads + lane) * p.n_words +
                           static_cast<int64_t>(m_tile) * 4 + q] = my_word;
        }
    }
}

}  // namespace kvzap
