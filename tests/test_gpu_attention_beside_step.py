"""Attention directly behind a decode step of a context that trusts its producers.

There the attention reads the rows that every list held before the step while that step is still running, and the rest
(the tile the step may append to, the window) after it.  The same steps on a default context, whose attention reads nothing
before the step has completed, give the reference: the lists are the same, and the outputs differ by rounding only --
probabilities are rounded to bf16 against the running maximum of the warp that met the row, 2 * 2^-9 of the values' size
(below 5 here), and the results once each: 2e-2 + 2^-8 |o|.  A row that is missed or counted twice moves an output by
about |v| / rows: the lists start short, where that is far more.
"""
import numpy as np
import pytest
import torch

from paper_2601_07891_b200 import synth
from tests.test_gpu_foreign_producer import producer  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

H, P = 8, 16


@pytest.fixture(scope="module")
def binding():
    from paper_2601_07891_b200 import binding as b
    b.load()
    return b


class _Side:
    """One context and cache with imported prefixes; the same for both sides but for the trust in the producers."""

    def __init__(self, binding, trusted, d_model, hidden, D, L, B, w, prefix, grow, fp8, P=P):
        self.b, self.fp8 = binding, fp8
        row = (D + synth.E4M3_ROW_TRAILER) // 2 if fp8 else D
        self.ctx = binding.Kvzap(d_model, hidden, H, row, L, max_tokens=max(B, 128), trusted_producers=trusted)
        for l in range(L):
            W1, b1, W2, b2 = synth.mlp_weights(d_model, hidden, H, 40 + l, "cuda", 0.3)
            if fp8:
                codes, scale = synth.quantize_e4m3(W1)
                binding.kvzap_set_weights_fp8(self.ctx.handle, l, codes, scale, b1, W2, b2)
            else:
                self.ctx.set_weights(l, W1, b1, W2, b2)
        pages = (prefix + P - 1) // P
        first = np.concatenate([[0], np.cumsum(pages)[:-1]])
        n_pages = int(pages.sum()) + grow * prefix.size
        max_pages = int(pages.max()) + grow
        self.pools = [self._rows((n_pages, P), D, s) for s in (1, 2)]
        table = torch.from_numpy((first[:, None] + np.arange(max_pages)[None, :]).astype(np.int32)).cuda()
        self.cache = binding.kvzap_cache_create(self.ctx.handle, B, w, P, *self.pools, max_pages)
        binding.kvzap_cache_import(self.ctx.handle, self.cache, torch.from_numpy(prefix.astype(np.int32)).cuda(), table,
                                   int(pages.sum()))

    def _rows(self, shape, D, seed):
        g = torch.Generator(device="cuda").manual_seed(seed)
        x = torch.empty(*shape, D, dtype=torch.float32, device="cuda").normal_(generator=g).clamp_(-4.9, 4.9)
        return synth.pack_rows_e4m3(x.view(-1, D)).view(*shape, -1) if self.fp8 else x.to(torch.bfloat16)

    def step(self, l0, l1, X, scale, K, V, tau, scores):
        if self.fp8:
            self.b.kvzap_decode_step_fp8(self.ctx.handle, self.cache, l0, l1, X, scale, K, V, tau, scores)
        else:
            self.b.kvzap_decode_step(self.ctx.handle, self.cache, l0, l1, X, K, V, tau, scores)

    def attend(self, l0, l1, Q, O):
        (self.b.kvzap_decode_attention_fp8 if self.fp8 else self.b.kvzap_decode_attention)(
            self.ctx.handle, self.cache, l0, l1, Q, 0.1, O)

    def close(self):
        self.b.kvzap_cache_destroy(self.cache)
        self.ctx.close()


def _close(got, want):
    d = (got.float() - want.float()).abs()
    return bool((d <= 2e-2 + 2.0 ** -8 * want.float().abs()).all()) and bool(torch.isfinite(got.float()).all())


# A step of hidden 512 takes 32 CTAs per layer and 128 sequences, one of hidden 128 eight: up to six tiles leave room beside it.
@pytest.mark.parametrize("D,G,B,L,group,w,longest,fp8,hidden,beside", [
    (128, 4, 3, 3, 1, 16, 70, False, 512, True),         # short lists, every tile remainder, layer by layer
    (128, 4, 8, 2, 1, 128, 3000, False, 512, True),      # parts by length
    (128, 4, 8, 2, 1, 16, 26000, False, 512, True),      # so long that all CTAs wait for the step
    (128, 8, 70, 2, 1, 32, 200, False, 512, True),       # more lists than CTAs of a wave
    (128, 2, 64, 2, 1, 32, 2700, False, 512, True),      # ... in two parts each
    (64, 4, 5, 4, 2, 48, 500, False, 128, True),         # rows of 64 elements, two layers a call
    (64, 4, 5, 3, 1, 48, 500, False, 512, True),
    (64, 2, 60, 2, 1, 16, 90, False, 128, True),
    (128, 1, 130, 2, 1, 16, 90, False, 128, True),       # two tiles of sequences per layer
    (128, 4, 4, 3, 1, 16, 900, True, 512, True),         # 8-bit rows
    (128, 4, 70, 2, 1, 16, 300, True, 128, True),        # ... of as many lists as find room beside the step
    (128, 4, 60, 2, 1, 16, 100, True, 512, False),       # ... and of more
    (128, 4, 50, 2, 1, 16, 100, False, 512, True),
    (64, 8, 9, 3, 3, 16, 60, True, 128, True),
    (64, 8, 9, 3, 1, 16, 60, True, 512, True),
    (128, 4, 8, 3, 2, 16, 60, False, 512, False),        # steps on too many SMs
    (128, 4, 70, 2, 1, 32, 1900, False, 512, True),      # more lists than CTAs of a wave, whole, the last ones in two parts
    (128, 4, 80, 2, 1, 16, 1900, True, 128, True),       # ... of 8-bit rows
    (64, 2, 60, 2, 1, 16, 2900, False, 128, True),       # ... the last ones in three
])
@pytest.mark.parametrize("page", [P, 48])
def test_outputs_are_those_of_a_context_that_waits(binding, D, G, B, L, group, w, longest, fp8, hidden, beside, page):
    d_model, steps = 1024, w + 40
    rng = np.random.default_rng(D + B)
    prefix = rng.integers(0, longest, size=B * L * H)
    prefix[:6] = [0, 1, 15, 16, 17, longest]
    sides = [_Side(binding, t, d_model, hidden, D, L, B, w, prefix, steps // P + 2, fp8, page) for t in (True, False)]
    outs = [[], []]
    row = sides[0].pools[0].shape[-1]
    inputs = []
    for k in range(7):
        X, scale = synth.hidden_states(L * B, d_model, 100 + k, "cuda"), None
        if fp8:
            X, scale = synth.quantize_e4m3(X)
            scale = scale.view(L, B)
        K, V = (sides[0]._rows((L, B, H), D, 200 + 2 * k + i) for i in (0, 1))
        inputs.append((X.view(L, B, d_model), scale, K.view(L, B, H, row), V.view(L, B, H, row)))
    Q7 = [synth.hidden_states(L * B * H * G, D, seed=7 + k, device="cuda").view(L, B, H * G, D) for k in range(7)]
    for side, out in zip(sides, outs):
        for k in range(steps):
            Q = Q7[k % 7]
            X, scale, K, V = inputs[k % 7]
            O = torch.full((L, B, H * G, D), 7.0, dtype=torch.bfloat16, device="cuda")
            scores = torch.zeros(L, B, H, dtype=torch.float32, device="cuda")
            for l in range(0, L, group):
                e = min(L, l + group)
                side.step(l, e, X[l:e], None if scale is None else scale[l:e], K[l:e], V[l:e], -0.1, scores[l:e])
                side.attend(l, e, Q[l:e], O[l:e])
            out.append((O, scores))
        torch.cuda.synchronize()
        assert side.ctx.poll_status() == 0
    # all attentions but the first, whose step has none ahead of it; a last call of fewer layers has steps small enough
    calls = [e - l for _ in range(steps) for l in range(0, L, group) for e in [min(L, l + group)]]
    assert binding.kvzap_beside_count(sides[1].ctx.handle) == 0
    assert binding.kvzap_beside_count(sides[0].ctx.handle) == sum(beside or n < group for n in calls[1:])
    n = [torch.empty(B, L, H, dtype=torch.int32, device="cuda") for _ in sides]
    for side, ln in zip(sides, n):
        binding.kvzap_cache_lengths(side.ctx.handle, side.cache, ln)
    assert torch.equal(n[0], n[1]) and int(n[0].sum()) > int(prefix.sum()) + B * L * H * w
    for k, (a, b) in enumerate(zip(*outs)):
        assert torch.equal(a[1], b[1]), k
        assert _close(a[0], b[0]), k
    for side in sides:
        side.close()


# A warp has two tiles in flight (of 8-bit rows three), a CTA four warps.  Up to 700 rows a list, in parts of 16 tiles or more: warps whose tiles
# are all in flight, which wait behind them, and warps with one or two more, which learn of new queries when the last is about to be
# issued.  From 9000 rows: some 35 tiles a warp, and the wait comes at its time, in the middle of them.
@pytest.mark.parametrize("shortest,longest", [(0, 700), (9000, 9400)])
@pytest.mark.parametrize("D,fp8", [(128, False), (128, True), (64, False), (64, True)])
def test_queries_written_between_step_and_attention(binding, producer, D, fp8, shortest, longest):  # noqa: F811
    """The kernel between the two signals before it stores the queries: they are read again once it has completed."""
    G, B, L, w, d_model, hidden = 4, 6, 2, 16, 1024, 128
    prefix = np.random.default_rng(3).integers(shortest, longest, size=B * L * H)
    sides = [_Side(binding, t, d_model, hidden, D, L, B, w, prefix, 4, fp8) for t in (True, False)]
    row = sides[0].pools[0].shape[-1]
    for k in range(6):
        X, scale = synth.hidden_states(L * B, d_model, 300 + k, "cuda"), None
        if fp8:
            X, scale = synth.quantize_e4m3(X)
            scale = scale.view(L, B)
        K, V = (sides[0]._rows((L, B, H), D, 400 + 2 * k + i).view(L, B, H, row) for i in (0, 1))
        old, new = (synth.hidden_states(L * B * H * G, D, seed=500 + 2 * k + i, device="cuda").view(L, B, H * G, D) for i in (0, 1))
        new[:, ::2] = old[:, ::2]                                # some lists keep their queries
        got = []
        for side in sides:
            Q, O = old.clone(), torch.full_like(old, 7.0)
            scores, O0 = torch.zeros(L, B, H, dtype=torch.float32, device="cuda"), torch.empty_like(O)
            torch.cuda.synchronize()
            side.attend(0, L, old, O0)                           # for the step to start behind
            side.step(0, L, X.view(L, B, d_model), scale, K, V, -0.1, scores)
            producer(new, Q)
            side.attend(0, L, Q, O)
            torch.cuda.synchronize()
            assert side.ctx.poll_status() == 0
            got.append(O)
        assert _close(got[0], got[1]), k
    assert binding.kvzap_beside_count(sides[0].ctx.handle) == 6
    for side in sides:
        side.close()


@pytest.mark.parametrize("B,L,w,longest", [(3, 4, 16, 200), (40, 3, 32, 400), (8, 2, 128, 4000)])
def test_any_order_of_calls(binding, B, L, w, longest):
    """Steps, attention, releases and prompts over random layers, back to back: a step started beside an attention is no
    link of a chain of steps, and a step behind a release or a prompt leaves nothing stale to the attention behind it."""
    D, G, d_model, hidden, n_ops = 128, 4, 1024, 512, 160
    rng = np.random.default_rng(B)
    prefix = rng.integers(0, longest, size=B * L * H)
    sides = [_Side(binding, t, d_model, hidden, D, L, B, w, prefix, 24, False) for t in (True, False)]
    X = synth.hidden_states(L * B, d_model, 1, "cuda").view(L, B, d_model)
    K, V = (sides[0]._rows((L, B, H), D, 2 + i) for i in (0, 1))
    Xp = synth.hidden_states(100, d_model, 5, "cuda")
    Kp, Vp = (sides[0]._rows((H, 100), D, 6 + i) for i in (0, 1))
    Sp = torch.zeros(100, H, dtype=torch.float32, device="cuda")
    Q = synth.hidden_states(L * B * H * G, D, seed=7, device="cuda").view(L, B, H * G, D)
    ops = []
    for _ in range(n_ops):
        l0 = int(rng.integers(0, L))
        l1 = int(rng.integers(l0 + 1, L + 1))
        kind = rng.choice(["step", "attend", "both", "prompt"], p=[0.25, 0.25, 0.45, 0.05])
        ops += [("step", l0, l1), ("attend", l0, l1)] if kind == "both" else [(kind, l0, l1)]
    outs = [[], []]
    for side, out in zip(sides, outs):
        # outputs and scores of their own for every call: nothing else orders the launches
        O = torch.full((len(ops), L, B, H * G, D), 7.0, dtype=torch.bfloat16, device="cuda")
        S = torch.zeros(len(ops), L, B, H, dtype=torch.float32, device="cuda")
        torch.cuda.synchronize()
        for i, (kind, l0, l1) in enumerate(ops):
            if kind == "step":
                side.step(l0, l1, X[l0:l1], None, K[l0:l1], V[l0:l1], 0.0, S[i, l0:l1])
            elif kind == "attend":
                side.attend(l0, l1, Q[l0:l1], O[i, l0:l1])
            else:
                binding.kvzap_cache_release_seq(side.ctx.handle, side.cache, (l0 * 7 + l1) % B)
                for l in range(L):
                    binding.kvzap_prefill_to_cache(side.ctx.handle, side.cache, l, (l0 * 7 + l1) % B, Xp, Kp, Vp, 0.0, Sp)
        torch.cuda.synchronize()
        assert side.ctx.poll_status() == 0
        out += [O, S]
    n = [torch.empty(B, L, H, dtype=torch.int32, device="cuda") for _ in sides]
    for side, ln in zip(sides, n):
        binding.kvzap_cache_lengths(side.ctx.handle, side.cache, ln)
    assert torch.equal(*n)
    assert torch.allclose(outs[0][1], outs[1][1], atol=1e-5, rtol=0)
    assert _close(outs[0][0], outs[1][0])
    for side in sides:
        side.close()
