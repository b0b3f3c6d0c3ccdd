"""The kernel for short inputs, at the edges of what it takes (2048 mask words over all heads, 256 lists; of given scores 32 to 56 blocks by
the sequences, paged 12 or 16) and just beyond: prompts of contexts that do not trust their producers and the pruning of given scores against the oracle,
chunks against the selection by score of their whole streams."""
import numpy as np
import pytest
import torch

from paper_2601_07891_b200 import binding, synth
from tests import parity

pytestmark = pytest.mark.gpu

TAU, W = 0.05, 16


def _case(T, B, H, D, seed, trusted=False):
    ctx = binding.Kvzap(128, 64, H, D, 1, max_tokens=T, max_seqs=B, trusted_producers=trusted)
    ctx.set_weights(0, *synth.mlp_weights(128, 64, H, seed, "cuda", 0.1))
    rng = np.random.default_rng(seed)
    ends = np.sort(rng.integers(0, T + 1, B - 1))           # empty sequences among them
    cu = torch.from_numpy(np.concatenate([[0], ends, [T]]).astype(np.int32)).cuda() if B > 1 else None
    return ctx, synth.hidden_states(T, 128, seed, "cuda"), cu


@pytest.mark.parametrize("T,B,H,D", [(1, 1, 8, 64), (129, 3, 8, 128), (300, 1, 8, 64), (2048, 2, 8, 64), (2049, 7, 8, 64), (8192, 1, 8, 64),
                                     (8192, 32, 8, 40), (8193, 1, 8, 64), (2000, 33, 8, 64), (65536, 5, 1, 64), (5000, 255, 1, 64),
                                     (4000, 7, 3, 512), (3001, 2, 5, 72), (7168, 1, 8, 64), (7169, 1, 8, 64), (6144, 2, 4, 64), (5121, 8, 8, 64),
                                     (4096, 9, 8, 64), (1536, 9, 8, 64), (1537, 9, 8, 64), (1024, 4, 8, 64), (1025, 4, 8, 64)])
@pytest.mark.parametrize("how", ["head major", "token major", "given scores", "given scores, trusted"])
def test_prompts(oracle, T, B, H, D, how):
    ctx, X, cu = _case(T, B, H, D, T + B, "trusted" in how)
    K, V = synth.keys_values(H, T, D, 3, "cuda")
    tok_major = how == "token major"
    Ki, Vi = (x.transpose(0, 1).contiguous() if tok_major else x for x in (K, V))
    P, first = 16, 2
    pages, max_pages = H * (T // P + B + 1), T // P + 2
    s = torch.randn(T, H, generator=torch.Generator(device="cuda").manual_seed(T), device="cuda")
    Ko, Vo = parity.poison_like(K), parity.poison_like(V)
    n = torch.full((B, H), -1, dtype=torch.int32, device="cuda")
    Kp, Vp = (torch.full((pages, P, D), -5.0, dtype=torch.bfloat16, device="cuda") for _ in range(2))
    table, n_paged, used = torch.full((B * H, max_pages), -1, dtype=torch.int32, device="cuda"), n.clone(), torch.zeros(1, dtype=torch.int32, device="cuda")
    h = ctx.handle
    if how.startswith("given"):
        binding.kvzap_prune_prefill(h, K, V, s, cu, B, TAU, W, Ko, Vo, n)
        binding.kvzap_prune_prefill_paged(h, K, V, s, cu, B, TAU, W, Kp, Vp, P, first, table, n_paged, used)
    else:
        (binding.kvzap_prefill_write if tok_major else binding.kvzap_prefill_fused)(h, 0, X, Ki, Vi, cu, B, TAU, W, Ko, Vo, n, s)
        (binding.kvzap_prefill_write_paged if tok_major else binding.kvzap_prefill_fused_paged)(
            h, 0, X, Ki, Vi, cu, B, TAU, W, Kp, Vp, P, first, table, n_paged, used, s)
    torch.cuda.synchronize()
    assert ctx.poll_status() == 0
    cu_np = cu.cpu().numpy() if cu is not None else None
    keep, _ = parity.check_compaction(oracle, K, V, s.cpu().numpy(), TAU, W, cu_np, Ko, Vo, n)
    fill = int(synth.bits(torch.tensor([-5.0], dtype=torch.bfloat16))[0])
    want = oracle.compact_paged(synth.bits(K), synth.bits(V), keep, P, pages, max_pages, cu_seqlens=cu_np, first_page=first, fill=fill)
    for got, ref in zip((synth.bits(Kp), synth.bits(Vp), table.cpu().numpy(), n_paged.cpu().numpy()), want[:4]):
        np.testing.assert_array_equal(got, ref)
    assert int(used) == want[4]
    ctx.close()


# the last three: pages whose size is no power of two, and more sequences than a bookkeeping CTA has warps
@pytest.mark.parametrize("T,B,H,D,P", [(500, 4, 8, 128, 16), (8192, 3, 8, 64, 16), (8300, 3, 8, 64, 16), (3000, 32, 8, 64, 16), (3000, 33, 8, 64, 16),
                                       (40, 6, 2, 40, 16), (700, 3, 8, 64, 24), (2100, 100, 2, 40, 7), (5000, 255, 1, 64, 5)])
def test_chunks(T, B, H, D, P):
    C = 3
    ctx, _, _ = _case(T, B, H, D, T + B)
    max_pages = C * T // P + 2
    pool = [torch.zeros(B * H * (C * T // P // B + 4) + C * T * H // P, P, D, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    cache = binding.kvzap_cache_create(ctx.handle, B + 2, W, P, *pool, max_pages)
    slots = [(5 * b + 1) % (B + 2) if (B + 2) % 5 else b + 1 for b in range(B)]
    streams = [[] for _ in range(B)]
    for first in (True, False):                              # the second time from released pages
        streams = [[] for _ in range(B)]
        for b in slots:
            binding.kvzap_cache_release_seq(ctx.handle, cache, b)
        for c in range(C):
            _, X, cu = _case(T, B, H, D, 10 * c + T)
            K, V = synth.keys_values(H, T, D, 50 + c, "cuda")
            s = torch.zeros(T, H, device="cuda")
            binding.kvzap_prefill_to_cache_batch(ctx.handle, cache, 0, slots, cu, X, K, V, TAU, s)
            torch.cuda.synchronize()
            at = cu.tolist()
            for b in range(B):
                streams[b].append((K[:, at[b]:at[b + 1]], V[:, at[b]:at[b + 1]], s[at[b]:at[b + 1]]))
        assert ctx.poll_status() == 0
    lengths = torch.zeros(B + 2, 1, H, dtype=torch.int32, device="cuda")
    binding.kvzap_cache_lengths(ctx.handle, cache, lengths)
    out = [torch.zeros(C * T, D, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    n = torch.zeros(1, dtype=torch.int32, device="cuda")
    for b in range(B):
        keep = torch.cat([x[2] for x in streams[b]]) >= TAU
        if len(keep):
            keep[-W:] = True
        assert torch.equal(lengths[slots[b], 0].long(), keep.sum(0))
        for h in range(H) if b < 4 else ():
            binding.kvzap_cache_export(ctx.handle, cache, slots[b], 0, h, *out, n)
            for i in range(2):
                want = torch.cat([x[i][h] for x in streams[b]])[keep[:, h]]
                assert torch.equal(out[i][:int(n)].view(torch.int16), want.view(torch.int16))
    binding.kvzap_cache_destroy(cache)
    ctx.close()
