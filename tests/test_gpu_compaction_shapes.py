"""The compaction of the fused calls in the shapes it is launched in: beside the next layer's scoring (trusted producers)
and alone (default contexts), over blocks shared by several CTAs, several blocks per CTA, ragged batches with empty
sequences, both K/V layouts, dense and paged, row lengths that are not a power of two.  Both contexts give the same bits,
and the rows are those of a plain selection by the scores."""
import numpy as np
import pytest
import torch

from paper_2601_07891_b200 import binding, synth

pytestmark = pytest.mark.gpu

D_MODEL, HIDDEN, H, TAU = 128, 64, 8, 0.1


def _run(trusted, T, lens, D, proj, paged, window, P=16):
    B = len(lens)
    ctx = binding.Kvzap(D_MODEL, HIDDEN, H, D, 1, max_tokens=T, max_seqs=B, trusted_producers=trusted)
    ctx.set_weights(0, *[x.cuda() for x in synth.mlp_weights(D_MODEL, HIDDEN, H, 5, "cpu", 0.3)])
    X = synth.hidden_states(T, D_MODEL, seed=T).cuda()
    g = torch.Generator(device="cuda").manual_seed(T + D)
    shape = (T, H, D) if proj else (H, T, D)
    K, V = (torch.empty(*shape, dtype=torch.bfloat16, device="cuda").normal_(generator=g) for _ in range(2))
    cu = None if B == 1 else torch.from_numpy(synth.cu_seqlens(lens)).cuda()
    lengths = torch.full((B, H), -1, dtype=torch.int32, device="cuda")
    scores = torch.zeros(T, H, dtype=torch.float32, device="cuda")
    if paged:
        n_pages = H * (T // P + 2 * B) + 3
        out = [torch.full((n_pages, P, D), 7.0, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
        table = torch.full((B * H, T // P + 2), -1, dtype=torch.int32, device="cuda")
        used = torch.zeros(1, dtype=torch.int32, device="cuda")
        call = binding.kvzap_prefill_write_paged if proj else binding.kvzap_prefill_fused_paged
        call(ctx.handle, 0, X, K, V, cu, B, TAU, window, *out, P, 3, table, lengths, used, scores)
        extra = [table, used]
    else:
        out = [torch.full((H, T, D), 7.0, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
        call = binding.kvzap_prefill_write if proj else binding.kvzap_prefill_fused
        call(ctx.handle, 0, X, K, V, cu, B, TAU, window, *out, lengths, scores)
        extra = []
    torch.cuda.synchronize()
    assert ctx.poll_status() == 0
    ctx.close()
    return (K, V, scores), [x.view(torch.int16) for x in out] + [lengths, scores] + extra


@pytest.mark.parametrize("T,lens,D,proj,paged,window", [
    (1, [1], 128, False, False, 16), (5, [5], 64, True, True, 0), (128, [128], 128, False, True, 128),
    (129, [100, 0, 29], 128, False, False, 16), (777, [777], 128, True, True, 128), (777, [300, 477], 128, True, False, 64),
    (2061, [500, 516, 517, 528], 128, False, True, 128), (2500, [2500], 96, False, False, 16),
    (9001, [9001], 128, False, False, 128), (9001, [4000, 1, 5000], 64, False, True, 16),
    (33333, [33333], 64, False, False, 128), (40001, [13001, 27000], 64, True, True, 128)])
def test_alone_and_beside_scoring(T, lens, D, proj, paged, window):
    (K, V, scores), got = _run(False, T, lens, D, proj, paged, window)
    _, beside = _run(True, T, lens, D, proj, paged, window)
    for a, b in zip(got, beside):
        assert torch.equal(a, b)
    cu = np.concatenate([[0], np.cumsum(lens)])
    keep = scores >= TAU
    for b in range(len(lens)):
        keep[max(cu[b], cu[b + 1] - window):cu[b + 1]] = True
    page = 3
    for b in range(len(lens)):
        at = slice(int(cu[b]), int(cu[b + 1]))
        for h in range(H):
            idx = keep[at, h].nonzero()[:, 0] + int(cu[b])
            n = idx.numel()
            assert int(got[2][b, h]) == n
            for x, o in zip((K, V), got[:2]):
                want = (x[idx, h] if proj else x[h, idx]).view(torch.int16)
                if paged:
                    assert torch.equal(o.reshape(-1, D)[page * 16:page * 16 + n], want)
                else:
                    assert torch.equal(o[h, int(cu[b]):int(cu[b]) + n], want)
            if paged:
                k = (n + 15) // 16
                assert got[4][b * H + h, :k].tolist() == list(range(page, page + k))
                page += k
    if paged:
        assert int(got[5]) == page - 3


@pytest.mark.parametrize("T,n_pages,max_pages", [(777, 40, 60), (777, 4000, 5), (9001, 40, 700)])
@pytest.mark.parametrize("trusted", [False, True])
def test_paged_pool_or_table_too_small(T, n_pages, max_pages, trusted):
    """Pages assigned inside the compaction (short) and by a launch of its own (long): the status word says so, the lengths
    are there, no page is used and nothing is written."""
    ctx = binding.Kvzap(D_MODEL, HIDDEN, H, 64, 1, max_tokens=T, trusted_producers=trusted)
    ctx.set_weights(0, *[x.cuda() for x in synth.mlp_weights(D_MODEL, HIDDEN, H, 5, "cpu", 0.3)])
    X = synth.hidden_states(T, D_MODEL, seed=T).cuda()
    K, V = (t.cuda() for t in synth.keys_values(H, T, 64, seed=3))
    out = [torch.full((n_pages, 16, 64), 7.0, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    table = torch.full((H, max_pages), -1, dtype=torch.int32, device="cuda")
    used, lengths = torch.full((1,), 9, dtype=torch.int32, device="cuda"), torch.zeros(1, H, dtype=torch.int32, device="cuda")
    scores = torch.zeros(T, H, dtype=torch.float32, device="cuda")
    binding.kvzap_prefill_fused_paged(ctx.handle, 0, X, K, V, None, 1, TAU, 128, *out, 16, 0, table, lengths, used, scores)
    torch.cuda.synchronize()
    assert ctx.poll_status() == 4                       # KVZAP_ERR_OOM_PAGES
    keep = scores >= TAU
    keep[-128:] = True
    assert torch.equal(lengths[0], keep.sum(0).int())
    assert int(used) == 0 and (table == -1).all() and all((x == 7.0).all() for x in out)
    ctx.close()
