"""GPU parity of the few-token scoring kernel over the layouts it chooses by the number of 128-token tiles: scores at
the sizes where one layout gives way to the next, and decode steps of one cache that change layout from call to call
(all layers in one call, then layer by layer), against the CPU oracle."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest
import torch

from paper_2601_07891_b200 import binding, synth
from tests import parity

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))

# An fp32 pre-activation is a chain of at most d_model / 16 + 8 additions of partial sums below 6 in magnitude, each off
# by at most 2^-23 of it; the second layer adds up |w2| of `hidden` of them: 0.8 sqrt(hidden) * 6 * 2^-23 * 72 at
# d_model = 1024 and hidden = 1024 is 1.3e-3.
ATOL = 2e-3


@pytest.mark.parametrize("hidden", [128, 512, 640, 1024])
@pytest.mark.parametrize("T", [1, 33, 128, 129, 513, 1153, 2305, 4737])
def test_scores_of_every_layout(oracle, hidden, T):
    d_model, H = 1024, 8
    ctx = binding.Kvzap(d_model, hidden, H, 64, 2, max_tokens=T)
    X = synth.hidden_states(T, d_model, seed=T + hidden)
    for layer in range(2):
        wts = synth.mlp_weights(d_model, hidden, H, 40 + layer, "cpu", 0.3)
        ctx.set_weights(layer, *[parity.dev(x) for x in wts])      # the call behind this one may not start early
        scores = torch.full((T, H), 7.0, dtype=torch.float32, device="cuda")
        ctx.score(layer, parity.dev(X), out=scores)
        again = torch.full_like(scores, 7.0)
        ctx.score(layer, parity.dev(X), out=again)
        torch.cuda.synchronize()
        assert ctx.poll_status() == 0
        rows = np.unique(np.concatenate([np.arange(min(T, 160)), np.arange(max(0, T - 160), T)]))
        _, err = parity.check_scores(oracle, scores, X, wts, rows)
        assert err <= ATOL
        assert torch.equal(scores, again)
    ctx.close()


@pytest.mark.parametrize("B,L,trusted", [(5, 20, True), (5, 20, False), (130, 3, True)])
def test_decode_steps_that_change_layout(oracle, B, L, trusted):
    d_model, hidden, H, D, w, P, tau, n_steps = 512, 512, 8, 64, 4, 4, 0.1, 12
    ctx = binding.Kvzap(d_model, hidden, H, D, L, max_tokens=max(B, 128), trusted_producers=trusted)
    for l in range(L):
        ctx.set_weights(l, *[parity.dev(x) for x in synth.mlp_weights(d_model, hidden, H, 60 + l, "cpu", 0.3)])
    n_pool = B * L * H * (n_steps // P + 2)
    K_pool = torch.zeros(n_pool, P, D, dtype=torch.bfloat16, device="cuda")
    V_pool = torch.zeros_like(K_pool)
    cache = binding.kvzap_cache_create(ctx.handle, B, w, P, K_pool, V_pool, n_steps // P + 2)
    dec = oracle.DecodeOracle(B, L, H, D, w)
    steps, scores = [], []
    for step in range(n_steps):
        X = synth.hidden_states(L * B, d_model, seed=300 + step).view(L, B, d_model)
        K, V = (t.view(L, B, H, D) for t in synth.keys_values(L * B, H, D, seed=400 + step))
        steps.append([parity.dev(t) for t in (X, K, V)])
        scores.append(torch.empty(L, B, H, dtype=torch.float32, device="cuda"))
    torch.cuda.synchronize()
    for step, (X, K, V) in enumerate(steps):         # enqueued back to back
        cuts = [0, L] if step % 3 == 0 else list(range(L + 1)) if step % 3 == 1 else [0, 1, L]
        for a, b in zip(cuts[:-1], cuts[1:]):
            binding.kvzap_decode_step(ctx.handle, cache, a, b, X[a:b], K[a:b], V[a:b], tau, scores[step][a:b])
    torch.cuda.synchronize()
    assert ctx.poll_status() == 0
    for (X, K, V), s in zip(steps, scores):
        s, Kb, Vb = s.cpu().numpy(), synth.bits(K.cpu()), synth.bits(V.cpu())
        for l in range(L):
            for b in range(B):
                dec.append(b, l, s[l, b], Kb[l, b], Vb[l, b], tau)
    lengths = torch.zeros(B, L, H, dtype=torch.int32, device="cuda")
    binding.kvzap_cache_lengths(ctx.handle, cache, lengths)
    ln = lengths.cpu().numpy()
    out = [torch.zeros(n_steps, D, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    n = torch.zeros(1, dtype=torch.int32, device="cuda")
    for b in range(B):
        for l in range(L):
            for h in range(H):
                assert ln[b, l, h] == dec.length(b, l, h)
                if b in (0, 3, 4, 127, 128, 129) and l in (0, 1, L - 1):
                    _, Kd, Vd = dec.logical(b, l, h)
                    binding.kvzap_cache_export(ctx.handle, cache, b, l, h, *out, n)
                    torch.cuda.synchronize()
                    m = int(n.item())
                    assert m == len(Kd)
                    np.testing.assert_array_equal(synth.bits(out[0])[:m], Kd)
                    np.testing.assert_array_equal(synth.bits(out[1])[:m], Vd)
    binding.kvzap_cache_destroy(cache)
    ctx.close()


@pytest.fixture(scope="module")
def arrivals():
    lib = os.path.join(HERE, "_build", "libarrivals.so")
    os.makedirs(os.path.dirname(lib), exist_ok=True)
    subprocess.run([shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc", "-gencode", "arch=compute_100a,code=sm_100a", "-O2",
                    "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-o", lib, os.path.join(HERE, "helpers", "arrivals.cu")],
                   check=True)
    return ctypes.CDLL(lib)


@pytest.mark.parametrize("n", [2, 4, 5, 8])
def test_arrivals_of_the_slices_do_not_add_up_over_launches(arrivals, n):
    """Every n-th arrival is the last of its launch and leaves the counter at zero, so that no number of launches wraps it."""
    launch = arrivals.launch_arrivals
    launch.argtypes = [ctypes.c_void_p, ctypes.c_uint, ctypes.c_int] + 3 * [ctypes.c_void_p]
    rounds = 7
    counter = torch.zeros(1, dtype=torch.int32, device="cuda")
    last, after = (torch.full((rounds * n,), -1, dtype=torch.int32, device="cuda") for _ in range(2))
    for _ in range(2):
        assert launch(counter.data_ptr(), n, rounds, last.data_ptr(), after.data_ptr(), torch.cuda.current_stream().cuda_stream) == 0
        torch.cuda.synchronize()
        assert last.tolist() == ([0] * (n - 1) + [1]) * rounds
        assert after.tolist() == (list(range(1, n)) + [0]) * rounds


@pytest.mark.parametrize("n", [1, 2, 5, 8, 148])
def test_every_lane_of_the_last_warp_sees_what_all_lanes_stored(arrivals, n):
    launch = arrivals.launch_warp_arrivals
    launch.argtypes = [ctypes.c_void_p, ctypes.c_uint, ctypes.c_void_p, ctypes.c_int] + 3 * [ctypes.c_void_p]
    counter, lasts = (torch.zeros(1, dtype=torch.int32, device="cuda") for _ in range(2))
    parts, sums = torch.full((n * 32,), -1, dtype=torch.int32, device="cuda"), torch.zeros(50, 32, dtype=torch.int32, device="cuda")
    for i in range(50):
        assert launch(counter.data_ptr(), n, parts.data_ptr(), 1000 * i, sums[i].data_ptr(), lasts.data_ptr(),
                      torch.cuda.current_stream().cuda_stream) == 0
    torch.cuda.synchronize()
    assert int(lasts) == 50 * 32 and int(counter) == 0       # all lanes of one warp a launch
    lane = (torch.arange(32) * 5 + 7) % 32
    for i in range(50):
        assert torch.equal(sums[i].cpu().long(), n * (1000 * i + lane) + 32 * n * (n - 1) // 2)


@pytest.mark.parametrize("hidden", [256, 512, 640, 1024])
@pytest.mark.parametrize("T", [1, 128, 129, 300, 640, 777, 2305])
def test_scores_of_the_layouts_that_leave_room_for_other_launches(oracle, hidden, T):
    """Contexts that trust their producers take narrower layouts for prompts: layers back to back, each its own buffers."""
    d_model, H, L = 1024, 8, 3
    ctx = binding.Kvzap(d_model, hidden, H, 64, L, max_tokens=T, trusted_producers=True)
    X = synth.hidden_states(T, d_model, seed=T + hidden)
    wts = [synth.mlp_weights(d_model, hidden, H, 50 + l, "cpu", 0.3) for l in range(L)]
    for l in range(L):
        ctx.set_weights(l, *[parity.dev(x) for x in wts[l]])
    Xd = parity.dev(X)
    scores = [torch.full((T, H), 7.0, dtype=torch.float32, device="cuda") for _ in range(L)]
    torch.cuda.synchronize()
    for l in range(L):
        ctx.score(l, Xd, out=scores[l])
    torch.cuda.synchronize()
    assert ctx.poll_status() == 0
    rows = np.unique(np.concatenate([np.arange(min(T, 160)), np.arange(max(0, T - 160), T)]))
    for l in range(L):
        _, err = parity.check_scores(oracle, scores[l], X, wts[l], rows)
        assert err <= ATOL
    ctx.close()
