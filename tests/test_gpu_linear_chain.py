"""Short linear prompts back to back on a context that trusts its producers, outputs reused in every pattern.

A call whose outputs are still in use by one of the calls ahead goes ahead up to its stores; one that reads what a call ahead
writes waits before it reads.  Every buffer has to end up with what its last call gives alone, bit for bit.
"""
import numpy as np
import pytest
import torch

from paper_2601_07891_b200 import synth

pytestmark = pytest.mark.gpu

H, D, TAU, W = 8, 128, 0.3, 64


@pytest.fixture(scope="module")
def binding():
    from paper_2601_07891_b200 import binding as b
    b.load()
    return b


@pytest.mark.parametrize("n", [40, 129, 1000, 4096, 8192])
@pytest.mark.parametrize("pattern", ["one", "two", "five", "random", "contexts", "rows_of_the_call_before"])
def test_outputs_of_calls_in_a_row(binding, n, pattern):
    d_model, n_calls, n_in = 1024, 50, 4
    rng = np.random.default_rng(n)
    ctxs = []
    for i in range(3 if pattern == "contexts" else 1):
        c = binding.Kvzap(d_model, 0, H, D, 1, max_tokens=n, trusted_producers=True)
        c.set_weights(0, *synth.linear_weights(d_model, H, 3, "cuda", 0.2))
        ctxs.append(c)
    X = [synth.hidden_states(n, d_model, 10 + i, "cuda") for i in range(n_in)]
    KV = [synth.keys_values(H, n, D, 20 + i, "cuda") for i in range(n_in)]

    def outputs():
        return (torch.zeros(H, n, D, dtype=torch.bfloat16, device="cuda"), torch.zeros(H, n, D, dtype=torch.bfloat16, device="cuda"),
                torch.zeros(1, H, dtype=torch.int32, device="cuda"), torch.zeros(n, H, dtype=torch.float32, device="cuda"))

    def call(ctx, x, k, v, out):
        return binding.prepare_prefill_fused(ctx.handle, 0, x, k, v, None, 1, TAU, W, out[0], out[1], out[2], out[3])

    sets = {"one": 1, "two": 2, "five": 5, "random": 3, "contexts": 3, "rows_of_the_call_before": 2}[pattern]
    order = [(int(rng.integers(0, n_in)), int(rng.integers(0, sets)) if pattern == "random" else i % sets) for i in range(n_calls)]
    got, want = [outputs() for _ in range(sets)], [outputs() for _ in range(sets)]
    for side, wait in ((got, False), (want, True)):
        calls = []
        for i, (src, to) in enumerate(order):
            k, v = KV[src]
            if pattern == "rows_of_the_call_before" and i > 0:
                k, v = side[order[i - 1][1]][:2]
            calls.append(call(ctxs[i % len(ctxs)], X[src], k, v, side[to]))
        torch.cuda.synchronize()
        for c in calls:
            c()
            if wait:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
    for c in ctxs:
        assert c.poll_status() == 0
    for a, b in zip(got, want):
        for x, y in zip(a, b):
            assert torch.equal(x.view(torch.uint8), y.view(torch.uint8))
    for c in ctxs:
        c.close()
