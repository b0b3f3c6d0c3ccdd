"""Pruning and prefill calls back to back on a context that trusts its producers, in every order.

Calls of very different lengths, each form of pruning and the prefill, over a few buffers that they use again as outputs and,
some of them, as inputs: a launch that takes part in a chain may start beside the ones ahead, one that follows a waiting
launch may not meet what was ahead of that.  Every buffer has to end up as when the GPU is waited for behind each call, bit for
bit.  (The rule itself is checked without a GPU in test_inflight.)
"""
import numpy as np
import pytest
import torch

from paper_2601_07891_b200 import synth

pytestmark = pytest.mark.gpu

H, D, P, TAU, W, D_MODEL = 8, 128, 16, 0.3, 64, 512
N_MAX = 30000


@pytest.fixture(scope="module")
def binding():
    from paper_2601_07891_b200 import binding as b
    b.load()
    return b


class _Buffers:
    def __init__(self, n_out):
        new = lambda n, dtype: torch.zeros(n, dtype=dtype, device="cuda")              # noqa: E731
        self.rows = [(new(H * N_MAX * D, torch.bfloat16), new(H * N_MAX * D, torch.bfloat16)) for _ in range(n_out)]
        self.lengths = [new(4 * H, torch.int32) for _ in range(n_out)]
        self.scores = [new(N_MAX * H, torch.float32) for _ in range(n_out)]
        self.tau = [new(4 * H, torch.float32) for _ in range(n_out)]
        self.table = [new(4 * H * (N_MAX // P + 1), torch.int32) for _ in range(n_out)]
        self.used = [new(1, torch.int32) for _ in range(n_out)]

    def all(self):
        return [t for pair in self.rows for t in pair] + self.lengths + self.scores + self.tau + self.table + self.used


@pytest.mark.parametrize("hidden", [0, 256])
@pytest.mark.parametrize("n_out", [1, 2, 3, 5])
@pytest.mark.parametrize("kinds", ["prune", "paged", "prune budget", "prune paged budget prefill", "prune prefill"])
def test_outputs_of_calls_in_a_row(binding, hidden, n_out, kinds):
    rng = np.random.default_rng(n_out + len(kinds) + hidden)
    ctx = binding.Kvzap(D_MODEL, hidden, H, D, 1, max_tokens=N_MAX, max_seqs=4, trusted_producers=True)
    ctx.set_weights(0, *(synth.mlp_weights(D_MODEL, hidden, H, 3, "cuda", 0.2) if hidden else synth.linear_weights(D_MODEL, H, 3, "cuda", 0.2)))
    X = [synth.hidden_states(N_MAX, D_MODEL, 10 + i, "cuda") for i in range(2)]
    rows = [tuple(t.view(-1) for t in synth.keys_values(H, N_MAX, D, 20 + i, "cuda")) for i in range(2)]
    scores = [torch.randn(N_MAX * H, device="cuda", generator=torch.Generator("cuda").manual_seed(30 + i)) for i in range(2)]
    sizes = [40, 300, 1000, 8192, N_MAX]
    cus = {n: torch.tensor([0, n // 7, n // 2, n], dtype=torch.int32, device="cuda") for n in sizes}
    plan = []
    for i in range(60):
        n = int(rng.choice(sizes, p=[0.3, 0.3, 0.2, 0.1, 0.1]))
        # inputs: the callers' own, or rows that a call of at least two calls ago made
        plan.append((str(rng.choice(kinds.split())), n, int(rng.integers(0, 2)), bool(rng.random() < 0.2), int(rng.integers(0, n_out)),
                     bool(rng.random() < 0.4), i % n_out if rng.random() < 0.5 else int(rng.integers(0, n_out))))

    def call(buf, kind, n, src, chained, frm, several, to):
        rows_in = buf.rows[frm] if chained and frm != to else rows[src]
        K, V = (t[:H * n * D].view(H, n, D) for t in rows_in)
        s = scores[src][:n * H].view(n, H)
        cu, B = (cus[n], 3) if several else (None, 1)
        K_out, V_out = buf.rows[to]
        dense = [t[:H * n * D].view(H, n, D) for t in (K_out, V_out)]
        lengths = buf.lengths[to][:B * H].view(B, H)
        if kind == "prune":
            binding.prepare_prune_prefill(ctx.handle, K, V, s, cu, B, TAU, W, *dense, lengths)()
        elif kind == "budget":
            binding.kvzap_prune_prefill_topk(ctx.handle, K, V, s, cu, B, 0.3, W, src == 1, *dense, lengths, buf.tau[to][:B * H].view(B, H))
        elif kind == "paged":
            pools = [t.view(-1, P, D) for t in (K_out, V_out)]
            table = buf.table[to][:B * H * (N_MAX // P + 1)].view(B * H, -1)
            binding.prepare_prune_prefill_paged(ctx.handle, K, V, s, cu, B, TAU, W, *pools, P, 0, table, lengths, buf.used[to])()
        else:
            binding.prepare_prefill_fused(ctx.handle, 0, X[src][:n], K, V, cu, B, TAU, W, *dense, lengths,
                                          buf.scores[to][:n * H].view(n, H))()

    got, want = _Buffers(n_out), _Buffers(n_out)
    for buf, wait in ((got, False), (want, True)):
        torch.cuda.synchronize()
        for at in plan:
            call(buf, *at)
            if wait:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
    assert ctx.poll_status() == 0
    for a, b in zip(got.all(), want.all()):
        assert torch.equal(a.view(torch.uint8), b.view(torch.uint8))
    ctx.close()
