"""8-bit decode steps of more tiles than the one-launch step takes: layer after layer through the scoring of short prompts, then
the update of the cache, which on a default context moves its rows beside the last scoring.  Steps back to back against the
same steps with the GPU waited for behind each, bit for bit: scores, lengths and lists."""
import pytest
import torch

from paper_2601_07891_b200 import binding, synth

pytestmark = pytest.mark.gpu

H, D, P, TAU = 8, 64, 16, 0.1


@pytest.mark.parametrize("trusted", [False, True])
@pytest.mark.parametrize("d_model,hidden,B,L,w", [(256, 128, 5, 45, 8), (256, 128, 140, 20, 16), (1024, 512, 8, 40, 32), (256, 128, 5, 45, 0)])
def test_back_to_back(d_model, hidden, B, L, w, trusted):
    n_steps = w + 40
    weights = []
    for l in range(L):
        W1, b1, W2, b2 = synth.mlp_weights(d_model, hidden, H, 60 + l, "cuda", 0.3)
        weights.append(synth.quantize_e4m3(W1) + (b1, W2, b2))
    inputs = []
    for k in range(5):
        x8, xs = synth.quantize_e4m3(synth.hidden_states(L * B, d_model, 100 + k, "cuda"))
        K, V = (t.view(L, B, H, D) for t in synth.keys_values(L * B, H, D, 200 + k, "cuda"))
        inputs.append((x8.view(L, B, d_model), xs.view(L, B), K, V))
    results = []
    for wait in (False, True):
        ctx = binding.Kvzap(d_model, hidden, H, D, L, max_tokens=max(B, 128), trusted_producers=trusted)
        for l, (w8, ws, b1, W2, b2) in enumerate(weights):
            binding.kvzap_set_weights_fp8(ctx.handle, l, w8, ws, b1, W2, b2)
        pages = B * L * H * (n_steps // P + 2)
        K_pool, V_pool = (torch.zeros(pages, P, D, dtype=torch.bfloat16, device="cuda") for _ in range(2))
        cache = binding.kvzap_cache_create(ctx.handle, B, w, P, K_pool, V_pool, n_steps // P + 2)
        scores = torch.zeros(n_steps, L, B, H, dtype=torch.float32, device="cuda")
        torch.cuda.synchronize()
        before = ctx.launch_count()
        for s in range(n_steps):
            x8, xs, K, V = inputs[s % 5]
            binding.kvzap_decode_step_fp8(ctx.handle, cache, 0, L, x8, xs, K, V, TAU, scores[s])
            if wait:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        assert ctx.launch_count() - before == n_steps * (L + 1)
        assert ctx.poll_status() == 0
        lengths = torch.zeros(B, L, H, dtype=torch.int32, device="cuda")
        binding.kvzap_cache_lengths(ctx.handle, cache, lengths)
        lists = []
        for b, l, h in [(0, 0, 0), (B - 1, L - 1, H - 1), (B // 2, L // 2, 3), (0, L - 1, 5), (B - 1, 0, 2)]:
            out = [torch.zeros(n_steps + 1, D, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
            n = torch.zeros(1, dtype=torch.int32, device="cuda")
            binding.kvzap_cache_export(ctx.handle, cache, b, l, h, *out, n)
            lists += out + [n]
        results.append([scores, lengths] + lists)
        torch.cuda.synchronize()
        binding.kvzap_cache_destroy(cache)
        ctx.close()
    for a, b in zip(*results):
        assert torch.equal(a.view(torch.uint8), b.view(torch.uint8))
    assert 0 < int(results[0][1].sum()) < n_steps * B * L * H
