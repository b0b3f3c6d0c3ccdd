"""KVzap-Linear prompts of contexts that do not trust their producers around the sizes where the launch changes (one and two CTAs of the
four-CTAs-per-tile kernel per SM, the persistent kernel): scores and lists against the oracle."""
import pytest
import torch

from paper_2601_07891_b200 import binding, synth
from tests import parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,B", [(1, 1), (127, 1), (4096, 1), (4736, 1), (4737, 1), (4737, 3), (8192, 2), (8193, 1), (8321, 1), (9500, 2)])
def test_linear_prompts(oracle, T, B):
    d_model, H, D, tau, w = 256, 8, 64, 0.3, 16
    ctx = binding.Kvzap(d_model, 0, H, D, 1, max_tokens=T, max_seqs=B)
    weights = synth.linear_weights(d_model, H, T, "cpu", 0.3)
    ctx.set_weights(0, *[parity.dev(x) for x in weights])
    X, (K, V) = synth.hidden_states(T, d_model, T), synth.keys_values(H, T, D, 6, "cuda")
    cu = synth.cu_seqlens([T // B] * (B - 1) + [T - T // B * (B - 1)]) if B > 1 else None
    cu_dev = torch.from_numpy(cu).cuda() if B > 1 else None
    for _ in range(2):
        s = torch.zeros(T, H, device="cuda")
        Ko, Vo = parity.poison_like(K), parity.poison_like(V)
        n = torch.full((B, H), -1, dtype=torch.int32, device="cuda")
        binding.kvzap_prefill_fused(ctx.handle, 0, parity.dev(X), K, V, cu_dev, B, tau, w, Ko, Vo, n, s)
        torch.cuda.synchronize()
        assert ctx.poll_status() == 0
        _, err = parity.check_scores(oracle, s, X, weights)
        assert err < 1e-4                                    # fp32 sums of 256 products of order one
        parity.check_compaction(oracle, K, V, s.cpu().numpy(), tau, w, cu, Ko, Vo, n)
    ctx.close()
