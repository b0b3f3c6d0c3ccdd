"""The window side of chunked prefill: more sequences than fit a launch's arguments, windows of several batches of exits,
released pages taken in batches next to fresh ones, with the launch beside the scoring kernel (default contexts, few
tokens) and behind it (trusted producers, no window).  Every list checked is the selection by score of its whole stream."""
import numpy as np
import pytest
import torch

from paper_2601_07891_b200 import binding, synth

pytestmark = pytest.mark.gpu

D_MODEL, HIDDEN, H, D, TAU = 128, 128, 8, 64, 0.1


@pytest.mark.parametrize("trusted", [False, True])
@pytest.mark.parametrize("n_seqs,window,P,rounds", [
    (130, 16, 4, [9, 30, 2]), (128, 16, 16, [20, 20]), (3, 272, 4, [150, 290, 300, 7]), (2, 128, 1, [128, 128, 1, 400]), (5, 0, 16, [33, 50])])
def test_chunks_against_selection(trusted, n_seqs, window, P, rounds):
    rng = np.random.default_rng(n_seqs)
    top = 2 * max(rounds) + 2
    ctx = binding.Kvzap(D_MODEL, HIDDEN, H, D, 2, max_tokens=n_seqs * top, max_seqs=n_seqs, trusted_producers=trusted)
    for l in range(2):
        ctx.set_weights(l, *[x.cuda() for x in synth.mlp_weights(D_MODEL, HIDDEN, H, 9 + l, "cpu", 0.3)])
    total = 2 * sum(rounds) + 10
    n_pool = n_seqs * H * 2 * (total // P + 2)
    pools = [torch.zeros(n_pool, P, D, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    cache = binding.kvzap_cache_create(ctx.handle, n_seqs + 1, window, P, pools[0], pools[1], total // P + 2)
    slots = [int(s) for s in rng.permutation(n_seqs + 1)[:n_seqs]]
    check = sorted(set([0, n_seqs // 2, n_seqs - 1]))
    for life in range(2):                      # the second life takes the pages that the first one gave back, then fresh ones
        streams = [[[] for _ in range(2)] for _ in check]
        calls = []
        for r, m in enumerate(rounds):
            lens = [int(x) for x in rng.integers(0, 2 * m + 1, n_seqs)]
            lens[0] = max(1, lens[0])
            cu, n = synth.cu_seqlens(lens), sum(lens)
            for l in range(2):
                X = synth.hidden_states(n, D_MODEL, seed=life * 100 + r * 2 + l).cuda()
                K, V = (t.cuda() for t in synth.keys_values(H, n, D, seed=1000 + life * 100 + r * 2 + l))
                s = torch.zeros(n, H, dtype=torch.float32, device="cuda")
                calls.append((l, torch.from_numpy(cu).cuda(), X, K, V, s, cu))
        torch.cuda.synchronize()
        for l, cu_dev, X, K, V, s, _ in calls:         # enqueued back to back
            binding.kvzap_prefill_to_cache_batch(ctx.handle, cache, l, slots, cu_dev, X, K, V, TAU, s)
        torch.cuda.synchronize()
        assert ctx.poll_status() == 0
        for l, _, X, K, V, s, cu in calls:
            for j, b in enumerate(check):
                at = slice(int(cu[b]), int(cu[b + 1]))
                streams[j][l].append((K[:, at], V[:, at], s[at]))
        out = [torch.zeros(total, D, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
        n = torch.zeros(1, dtype=torch.int32, device="cuda")
        for j, b in enumerate(check):
            for l in range(2):
                K, V = (torch.cat([c[i] for c in streams[j][l]], dim=1) for i in range(2))
                keep = torch.cat([c[2] for c in streams[j][l]]) >= TAU
                if window and keep.shape[0]:
                    keep[-window:] = True
                for h in range(H):
                    binding.kvzap_cache_export(ctx.handle, cache, slots[b], l, h, *out, n)
                    torch.cuda.synchronize()
                    idx = keep[:, h].nonzero()[:, 0]
                    assert int(n) == idx.numel()
                    for x, o in zip((K, V), out):
                        assert torch.equal(o[:idx.numel()].view(torch.int16), x[h, idx].view(torch.int16))
        for s in slots:
            binding.kvzap_cache_release_seq(ctx.handle, cache, s)
    binding.kvzap_cache_destroy(cache)
    ctx.close()


@pytest.mark.parametrize("trusted", [False, True])
@pytest.mark.parametrize("max_pages,pool_pages,second", [(40, 4000, 260), (40, 4000, 300), (100, 700, 260), (100, 1, 200)])
def test_pages_run_out_among_several_batches_of_exits(trusted, max_pages, pool_pages, second):
    """A window of 272 tokens pushed out in batches of 128 until the table (160 rows) or the pool is full: a list holds the
    exits that found a page, oldest first, and its window the newest tokens, in every repetition."""
    n_seqs, window, P = 3, 272, 4
    ctx = binding.Kvzap(D_MODEL, HIDDEN, H, D, 1, max_tokens=n_seqs * 400, max_seqs=n_seqs, trusted_producers=trusted)
    ctx.set_weights(0, *[x.cuda() for x in synth.mlp_weights(D_MODEL, HIDDEN, H, 9, "cpu", 0.3)])
    pools = [torch.zeros(pool_pages, P, D, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    lens = [[window] * n_seqs, [second] * n_seqs]
    inputs = []
    for r in range(2):
        n = sum(lens[r])
        inputs.append((torch.from_numpy(synth.cu_seqlens(lens[r])).cuda(), synth.hidden_states(n, D_MODEL, seed=r).cuda(),
                       *(t.cuda() for t in synth.keys_values(H, n, D, seed=10 + r)), torch.zeros(n, H, device="cuda")))
    out = [torch.zeros(max_pages * P + window, D, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    n = torch.zeros(1, dtype=torch.int32, device="cuda")
    for _ in range(4):
        cache = binding.kvzap_cache_create(ctx.handle, n_seqs, window, P, *pools, max_pages)
        for cu, X, K, V, s in inputs:
            binding.kvzap_prefill_to_cache_batch(ctx.handle, cache, 0, list(range(n_seqs)), cu, X, K, V, float("-inf"), s)
        torch.cuda.synchronize()
        assert ctx.poll_status() == 4                  # KVZAP_ERR_OOM_PAGES
        owned = 0
        for b in range(n_seqs):
            stream = [torch.cat([inputs[r][i][:, b * lens[r][b]:(b + 1) * lens[r][b]] for r in range(2)], dim=1) for i in (2, 3)]
            for h in range(H):
                binding.kvzap_cache_export(ctx.handle, cache, b, 0, h, *out, n)
                prefix = int(n) - window
                owned += (prefix + P - 1) // P
                assert 0 <= prefix <= second and (prefix == 160 or max_pages != 40)
                for x, o in zip(stream, out):
                    want = torch.cat([x[h, :prefix], x[h, -window:]])
                    assert torch.equal(o[:int(n)].view(torch.int16), want.view(torch.int16))
        if max_pages != 40:
            assert owned == pool_pages         # every page of the pool went to a list
        binding.kvzap_cache_destroy(cache)
    ctx.close()
