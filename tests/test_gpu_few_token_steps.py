"""Decode steps of up to 32 sequences and just beyond, at the edges of the eights in which the kernel stages hidden states and of
the fours in which its warps take tokens: scores against fp64, lists against the selection by score of their whole streams."""
import pytest
import torch

from paper_2601_07891_b200 import binding, synth
from tests import test_gpu_step_order as order

pytestmark = pytest.mark.gpu


# d_model 512, 8 heads.  Slices x CTAs along K: hidden 512 4 x 8, of many layers a call 2 x 2; 128 4 x 2; 64 2 x 2; 640 5 x 8; 1024 8 x 8; the
# last two of many layers a call 4 x 1, without a cluster
@pytest.mark.parametrize("B,L,hidden,group,trusted,fp8", [
    (1, 2, 512, 1, True, False), (4, 3, 512, 1, False, False), (5, 2, 512, 2, True, True), (8, 12, 512, 12, True, False),
    (9, 2, 512, 1, True, False), (16, 2, 640, 1, True, False), (17, 2, 512, 1, True, True), (24, 3, 128, 1, False, False),
    (25, 36, 512, 36, True, False), (31, 2, 1024, 1, True, False), (32, 2, 512, 1, True, False), (32, 30, 512, 30, True, True),
    (33, 2, 512, 1, True, False), (33, 2, 512, 2, True, True), (7, 2, 64, 1, True, False),
    (8, 36, 640, 36, True, False), (32, 30, 1024, 30, True, False), (5, 30, 1024, 30, False, True)])
def test_steps_of_few_sequences(B, L, hidden, group, trusted, fp8):
    _steps(B, L, hidden, group, trusted, fp8)


@pytest.mark.parametrize("heads", [1, 2, 5, 7])
@pytest.mark.parametrize("B,L,hidden,group,trusted,fp8", [(9, 2, 512, 1, True, False), (32, 12, 512, 12, False, False), (3, 2, 512, 1, True, True)])
def test_fewer_heads(monkeypatch, heads, B, L, hidden, group, trusted, fp8):
    monkeypatch.setattr(order, "H", heads)
    _steps(B, L, hidden, group, trusted, fp8)


def _steps(B, L, hidden, group, trusted, fp8):
    H = order.H
    n = order.W + 24
    s = order._Server(hidden, B, L, trusted, n + 2, fp8)
    for _ in range(n):
        for a in range(0, L, group):
            s.step(a, min(L, a + group))
    made = [s._inputs(L * B)[0].view(L, B, order.D_MODEL)]
    X, scale = made[0], None
    if fp8:
        x8, sx = synth.quantize_e4m3(X.view(L * B, order.D_MODEL))
        X, scale = x8.view(L, B, -1), sx.view(L, B)
    K, V = (t.view(L, B, H, order.D) for t in synth.keys_values(L * B, H, order.D, 77, "cuda"))
    scores = torch.full((L, B, H), float("nan"), dtype=torch.float32, device="cuda")
    for a in range(0, L, group):
        e = min(L, a + group)
        args = (X[a:e],) + ((scale[a:e],) if fp8 else ()) + (K[a:e], V[a:e], order.TAU, scores[a:e])
        call = binding.kvzap_decode_step_fp8 if fp8 else binding.kvzap_decode_step
        s.calls.append(lambda a=a, e=e, args=args: call(s.ctx.handle, s.cache, a, e, *args))
        for b in range(B):
            for l in range(a, e):
                s.events.append(("rows", b, l, K[l, b][:, None], V[l, b][:, None], scores[l, b][None]))
    s.check()
    for l in range(L):
        W1, b1, W2, b2 = synth.mlp_weights(order.D_MODEL, hidden, H, 70 + l, "cuda", 0.3)
        W1, x = W1.double(), X[l].double() if not fp8 else X[l].view(torch.float8_e4m3fn).double() * scale[l].double()[:, None]
        if fp8:
            codes, sw = synth.quantize_e4m3(W1.bfloat16())
            W1 = codes.view(torch.float8_e4m3fn).double() * sw.double()[:, None]
        want = torch.nn.functional.gelu(x @ W1.t() + b1.double()) @ W2.double().t() + b2.double()
        # fp32 sums of 512 products of order 1, GELU to 5e-7, hidden of its products summed in fp32: well below 1e-4
        assert (scores[l].double() - want).abs().max() < 1e-4
