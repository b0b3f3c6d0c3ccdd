"""Prompts of every number of 128-token blocks at which the MLP scoring changes its launches: single CTAs or CTA pairs per
block, odd numbers of blocks, and whole waves of CTA pairs with the blocks they leave over in a launch of their own.

Scores against a product in 64 bits.  Products of bf16 or E4M3 values are exact in fp32; a pre-activation sums 1024 of them,
2^-24 * sqrt(1024) of about one each at worst of a few standard deviations: 1e-5; the second layer sums up to 640 such times
|W2| < 0.2, and GELU adds 5e-7 each: 1e-4 covers it.  Masks, lengths and rows are then those of the GPU's own scores, bit for
bit.
"""
import numpy as np
import pytest
import torch

from paper_2601_07891_b200 import synth

pytestmark = pytest.mark.gpu

H, D, D_MODEL, TAU, W = 8, 64, 1024, 0.2, 32
WAVE = 148


@pytest.fixture(scope="module")
def binding():
    from paper_2601_07891_b200 import binding as b
    b.load()
    return b


def _inputs(hidden, n, fp8, seed):
    W1, b1, W2, b2 = synth.mlp_weights(D_MODEL, hidden, H, seed, "cuda", 0.1)
    X = synth.hidden_states(n, D_MODEL, seed + 1, "cuda")
    if not fp8:
        return (W1, b1, W2, b2), X, None, W1.double(), X.double()
    w8, ws = synth.quantize_e4m3(W1)
    x8, xs = synth.quantize_e4m3(X)
    return ((w8, ws, b1, W2, b2), x8, xs, w8.view(torch.float8_e4m3fn).double() * ws.double()[:, None],
            x8.view(torch.float8_e4m3fn).double() * xs.double()[:, None])


def _check(binding, hidden, n, fp8, trusted, seqs):
    weights, X, xs, w1, x = _inputs(hidden, n, fp8, n % 1000 + hidden)
    b1, W2, b2 = (t.double() for t in weights[-3:])
    want = torch.nn.functional.gelu(x @ w1.t() + b1) @ W2.t() + b2
    cuts = [0] + sorted(np.random.default_rng(n).choice(np.arange(1, n), seqs - 1, replace=False).tolist()) + [n]
    cu = None if seqs == 1 else torch.tensor(cuts, dtype=torch.int32, device="cuda")
    K, V = synth.keys_values(H, n, D, 5, "cuda")
    ctx = binding.Kvzap(D_MODEL, hidden, H, D, 1, max_tokens=n, max_seqs=seqs, trusted_producers=trusted)
    if fp8:
        binding.kvzap_set_weights_fp8(ctx.handle, 0, *weights)
    else:
        ctx.set_weights(0, *weights)
    for rep in range(2):                                     # back to back: flags and counters of the call before
        K_out, V_out = torch.zeros_like(K), torch.zeros_like(V)
        lengths = torch.zeros(seqs, H, dtype=torch.int32, device="cuda")
        scores = torch.zeros(n, H, dtype=torch.float32, device="cuda")
        torch.cuda.synchronize()
        if fp8:
            binding.prepare_prefill_fused_fp8(ctx.handle, 0, X, xs, K, V, cu, seqs, TAU, W, K_out, V_out, lengths, scores)()
        else:
            binding.prepare_prefill_fused(ctx.handle, 0, X, K, V, cu, seqs, TAU, W, K_out, V_out, lengths, scores)()
        torch.cuda.synchronize()
        assert ctx.poll_status() == 0
        assert float((scores.double() - want).abs().max()) <= 1e-4
        keep = scores >= TAU
        for b in range(seqs):
            keep[max(cuts[b], cuts[b + 1] - W):cuts[b + 1]] = True
        assert torch.equal(lengths, torch.stack([keep[cuts[b]:cuts[b + 1]].sum(0) for b in range(seqs)]).int())
        for b in range(seqs):
            for h in range(H):
                rows = torch.nonzero(keep[cuts[b]:cuts[b + 1], h])[:, 0] + cuts[b]
                at = slice(cuts[b], cuts[b] + rows.numel())
                assert torch.equal(K_out[h, at].view(torch.int16), K[h, rows].view(torch.int16)), (rep, b, h)
                assert torch.equal(V_out[h, at].view(torch.int16), V[h, rows].view(torch.int16)), (rep, b, h)
    ctx.close()


@pytest.mark.parametrize("fp8", [False, True])
@pytest.mark.parametrize("hidden,n", [
    (512, 129), (512, 256), (512, 257), (512, 777), (512, 128 * 9), (512, 128 * 17 + 3), (512, 128 * 18 + 1), (512, 128 * 37),
    (512, 128 * 38 + 5), (512, 128 * 73 + 1), (512, 128 * 74), (512, 128 * 74 + 1),
    (640, 300), (640, 128 * 13 + 64), (640, 128 * 36 + 1), (256, 128 * 20), (256, 128 * 50 + 9),
])
@pytest.mark.parametrize("trusted", [False, True])
def test_short_prompts(binding, hidden, n, fp8, trusted):
    _check(binding, hidden, n, fp8, trusted, 1 if n % 2 else 3)


@pytest.mark.parametrize("fp8", [False, True])
@pytest.mark.parametrize("hidden,blocks,extra", [
    (512, WAVE, 0), (512, WAVE, 1), (512, WAVE + 8, 77), (512, WAVE + 37, 0), (512, WAVE + 74, -5), (512, WAVE + 75, 0),
    (512, 2 * WAVE, 0), (512, 2 * WAVE, 1), (640, WAVE + 1, -127), (640, 2 * WAVE + 100, 3),
])
@pytest.mark.parametrize("seqs", [1, 4])
def test_whole_waves_and_the_rest(binding, hidden, blocks, extra, fp8, seqs):
    _check(binding, hidden, 128 * blocks + extra, fp8, False, seqs)
