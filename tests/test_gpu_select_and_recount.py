"""Pruning of given scores where the selection and the counting change their form: short inputs on both sides of the size
up to which a CTA counts what lies before it by itself, ragged batches with empty sequences, and the fixed budget's
cut values for scores whose digits differ only at the top, only at the bottom, or not at all.  Exact, against numpy."""
import numpy as np
import pytest
import torch

from paper_2601_07891_b200 import binding

pytestmark = pytest.mark.gpu

H, D = 8, 64


def _scores(kind, T, rng):
    if kind == "normal":
        s = rng.standard_normal((T, H))
    elif kind == "same":
        s = np.full((T, H), 0.25)
    elif kind == "low bits":                       # keys that differ in the last digit only
        s = (np.float32(1.0).view(np.uint32) + rng.integers(0, 700, (T, H)).astype(np.uint32)).view(np.float32)
    elif kind == "mid bits":
        s = (np.float32(-3.0).view(np.uint32) + (rng.integers(0, 2000, (T, H)) << 10).astype(np.uint32)).view(np.float32)
    else:                                          # infinities, NaN, signed zeros, subnormals, the largest values
        pool = np.array([np.inf, -np.inf, np.nan, 0.0, -0.0, 1e-42, -1e-42, 3.4e38, -3.4e38, 1.0], dtype=np.float32)
        s = pool[rng.integers(0, pool.size, (T, H))]
    return s.astype(np.float32)


def _key(x):
    u = x.view(np.uint32).astype(np.int64)
    return np.where(u & 0x80000000, ~u & 0xffffffff, u | 0x80000000)


def _check(K, V, scores, lens, window, keep, got):
    cu = np.concatenate([[0], np.cumsum(lens)])
    K_out, V_out, lengths = got
    for b in range(len(lens)):
        for h in range(H):
            idx = torch.from_numpy(np.flatnonzero(keep[cu[b]:cu[b + 1], h]) + cu[b]).cuda()
            assert int(lengths[b, h]) == idx.numel()
            for x, o in ((K, K_out), (V, V_out)):
                assert torch.equal(o[h, int(cu[b]):int(cu[b]) + idx.numel()].view(torch.int16), x[h, idx].view(torch.int16))


@pytest.fixture(scope="module", params=[False, True])
def ctx(request):
    c = binding.Kvzap(256, 0, H, D, 1, max_tokens=20000, max_seqs=7, trusted_producers=request.param)
    yield c
    c.close()


def _inputs(T, lens, kind):
    rng = np.random.default_rng(T + len(kind))
    g = torch.Generator(device="cuda").manual_seed(T)
    K, V = (torch.empty(H, T, D, dtype=torch.bfloat16, device="cuda").normal_(generator=g) for _ in range(2))
    cu = None if len(lens) == 1 else torch.tensor(np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)).cuda()
    out = [torch.zeros_like(K), torch.zeros_like(V), torch.full((len(lens), H), -1, dtype=torch.int32, device="cuda")]
    return _scores(kind, T, rng), K, V, cu, out


@pytest.mark.parametrize("lens,window", [
    ([1], 0), ([127], 16), ([129], 200), ([2176], 128), ([2177], 128), ([2305], 0), ([500, 501, 500], 128), ([3, 0, 700, 0, 1, 900, 128], 16),
    ([128, 128, 256], 128), ([1000, 1176], 64), ([1000, 1305], 64), ([3000], 128), ([4097], 128), ([4200], 16), ([9000], 128),
    ([20000], 128)])
@pytest.mark.parametrize("kind", ["normal", "special"])
def test_threshold(ctx, lens, window, kind):
    T, tau = sum(lens), 0.5
    s, K, V, cu, out = _inputs(T, lens, kind)
    dev = torch.from_numpy(s).cuda()
    for _ in range(2):
        binding.kvzap_prune_prefill(ctx.handle, K, V, dev, cu, len(lens), tau, window, *out)
    torch.cuda.synchronize()
    assert ctx.poll_status() == 0
    keep = s >= np.float32(tau)
    for e, n in zip(np.cumsum(lens), lens):
        keep[max(e - n, e - window):e] = True
    _check(K, V, s, lens, window, keep, out)


@pytest.mark.parametrize("lens,window", [([1], 0), ([130], 128), ([1024], 0), ([1153], 128), ([5000], 16), ([300, 0, 1025, 2500], 128), ([20000], 128)])
@pytest.mark.parametrize("kind", ["normal", "same", "low bits", "mid bits", "special"])
@pytest.mark.parametrize("ratio,per_layer", [(0.25, False), (0.37, True), (1.0, False), (0.0, True)])
def test_fixed_budget(ctx, lens, window, kind, ratio, per_layer):
    T = sum(lens)
    s, K, V, cu, out = _inputs(T, lens, kind)
    cut = torch.zeros(len(lens), H, dtype=torch.float32, device="cuda")
    dev = torch.from_numpy(s).cuda()
    for _ in range(2):                             # the second call finds the histograms as the first one left them
        binding.kvzap_prune_prefill_topk(ctx.handle, K, V, dev, cu, len(lens), ratio, window, per_layer, *out, cut)
    torch.cuda.synchronize()
    assert ctx.poll_status() == 0
    keep = np.zeros((T, H), dtype=bool)
    start = 0
    for b, n in enumerate(lens):
        n_cand = max(0, n - window)
        k = int(np.ceil(float(np.float32(ratio)) * n_cand))
        cand = s[start:start + n_cand]
        for h in range(H):
            x = cand.reshape(-1) if per_layer else cand[:, h]
            x = x[~np.isnan(x)]
            kk = k * H if per_layer else k
            if kk == 0:
                tau = np.float32(np.inf)
            elif kk > x.size:
                tau = np.float32(-np.inf)
            else:
                order = np.sort(_key(x))[::-1]
                key = np.uint32(order[kk - 1])
                tau = np.array([key & 0x7fffffff if key & 0x80000000 else ~key], dtype=np.uint32).view(np.float32)[0]
            assert np.float32(cut[b, h].item()).view(np.uint32) == tau.view(np.uint32)
            keep[start:start + n_cand, h] = cand[:, h] >= tau
        keep[start + n_cand:start + n] = True
        start += n
    _check(K, V, s, lens, window, keep, out)


def test_scratch_grows_with_the_calls_not_with_max_seqs():
    """A context made for many sequences starts small, takes calls of ever more sequences, and still takes small ones."""
    free = torch.cuda.mem_get_info()[0]
    c = binding.Kvzap(256, 0, H, D, 1, max_tokens=20000, max_seqs=4096)
    assert free - torch.cuda.mem_get_info()[0] < 64 << 20
    rng = np.random.default_rng(4)
    for n_seqs in (3, 9, 255, 256, 257, 700, 2):
        lens = [int(x) for x in rng.integers(0, 40 if n_seqs > 9 else 900, n_seqs)]
        test_fixed_budget(c, lens, 4, "normal", 0.25, n_seqs % 2 == 0)
    c.close()


def test_few_blocks_in_flight_per_sequence():
    """So many sequences that a long one's blocks are counted by fewer CTAs than it has blocks, one after the other."""
    c = binding.Kvzap(256, 0, H, D, 1, max_tokens=40000, max_seqs=400)
    for n_seqs, longest in ((60, 9000), (150, 5121), (400, 17000)):
        rng = np.random.default_rng(n_seqs)
        lens = [int(x) for x in rng.integers(0, 30, n_seqs)]
        lens[n_seqs // 2], lens[7] = longest, 2048 + 16
        for per_layer in (False, True):
            test_fixed_budget(c, lens, 16, "normal", 0.25, per_layer)
        test_fixed_budget(c, lens, 16, "low bits", 0.37, False)
    c.close()
