"""Attention over few lists of very unequal length, where the CTAs share the lists out by their lengths: on both sides of
the number of resident CTAs at which that rule ends, empty lists, one list that holds nearly all rows, a layer range, both
row formats.  Against softmax attention in fp64 over the rows that were imported."""
import numpy as np
import pytest
import torch

from paper_2601_07891_b200 import binding, synth
from tests import parity

pytestmark = pytest.mark.gpu

ATTN_ATOL = 2e-2        # as in test_gpu_attention.py: probabilities and outputs of order one rounded to bf16
H, G, P = 8, 2, 16


def _lengths(kind, n, rng):
    if kind == "one":
        x = np.zeros(n, dtype=np.int64)
        x[n // 2] = 9001
        return x
    if kind == "equal":
        return np.full(n, 333, dtype=np.int64)
    return np.floor(np.exp(rng.uniform(0, np.log(3000), n))).astype(np.int64) - 1       # 0 .. 2999, mostly short


@pytest.mark.parametrize("fp8,D", [(False, 128), (False, 64), (True, 128)])
@pytest.mark.parametrize("B,L,layers,kind", [(1, 1, (0, 1), "one"), (1, 1, (0, 1), "equal"), (3, 2, (1, 2), "log"), (19, 1, (0, 1), "log"),
                                             (36, 1, (0, 1), "log"), (37, 1, (0, 1), "log"), (37, 1, (0, 1), "one"),
                                             (73, 1, (0, 1), "log"), (75, 1, (0, 1), "equal")])
def test_attention_over_unequal_lists(fp8, D, B, L, layers, kind):
    rng = np.random.default_rng(B * 10 + L)
    row = (D + synth.E4M3_ROW_TRAILER) // 2 if fp8 else D
    ctx = binding.Kvzap(256, 0, H, row, L, max_tokens=128)
    n_lists = B * L * H
    prefix = _lengths(kind, n_lists, rng)
    pages = (prefix + P - 1) // P
    first = np.concatenate([[0], np.cumsum(pages)[:-1]])
    n_pages = int(pages.sum()) + 1
    g = torch.Generator(device="cuda").manual_seed(B)
    kv = [torch.empty(n_pages * P, D, dtype=torch.float32, device="cuda").normal_(generator=g) for _ in range(2)]
    kv = [synth.pack_rows_e4m3(x) if fp8 else x.bfloat16() for x in kv]
    rows = []
    for x in kv:
        if fp8:
            raw = x.view(torch.uint8)
            rows.append(raw[:, :D].contiguous().view(torch.float8_e4m3fn).float().double() *
                        raw[:, D:D + 4].contiguous().view(torch.float32).double())
        else:
            rows.append(x.double())
    for x in kv:                            # rows past a list's end hold NaN patterns
        for f, n, p in zip(first, prefix, pages):
            x[f * P + n:(f + p) * P] = float("nan")
    pools = [x.view(n_pages, P, row) for x in kv]
    max_pages = int(pages.max()) + 1
    cache = binding.kvzap_cache_create(ctx.handle, B, 16, P, pools[0], pools[1], max_pages)
    table = (first[:, None] + np.arange(max_pages)[None, :]).clip(0, n_pages - 1).astype(np.int32)
    binding.kvzap_cache_import(ctx.handle, cache, torch.from_numpy(prefix.astype(np.int32)).cuda(),
                               torch.from_numpy(table).cuda(), n_pages)
    a, e = layers
    Q = synth.hidden_states((e - a) * B * H * G, D, seed=B).view(e - a, B, H * G, D).cuda()
    O = torch.full_like(Q, 7.0)
    attend = binding.kvzap_decode_attention_fp8 if fp8 else binding.kvzap_decode_attention
    for _ in range(2):                      # the arrival counts are back at zero after the first call
        attend(ctx.handle, cache, a, e, Q, 1.0 / np.sqrt(D), O)
    torch.cuda.synchronize()
    assert ctx.poll_status() == 0
    want = torch.zeros(Q.shape, dtype=torch.float64, device="cuda")
    for l in range(a, e):
        for b in range(B):
            for h in range(H):
                li = (b * L + l) * H + h
                at = slice(int(first[li]) * P, int(first[li]) * P + int(prefix[li]))
                if prefix[li]:
                    q = Q[l - a, b, h * G:(h + 1) * G].double()
                    want[l - a, b, h * G:(h + 1) * G] = torch.softmax(q @ rows[0][at].t() / np.sqrt(D), 1) @ rows[1][at]
    assert float((O.double() - want).abs().max()) <= ATTN_ATOL
    binding.kvzap_cache_destroy(cache)
    ctx.close()


@pytest.mark.parametrize("fp8,D", [(False, 128), (False, 64), (True, 128), (True, 64)])
@pytest.mark.parametrize("kind", ["log", "equal", "one"])
@pytest.mark.parametrize("past", [0, 1])
def test_attention_where_sharing_by_length_ends(fp8, D, kind, past):
    """The largest batch with fewer lists than resident CTAs (three per SM, four of the 8-bit kernel's at 128), and the next."""
    slots = torch.cuda.get_device_properties(0).multi_processor_count * (4 if fp8 and D == 128 else 3)
    test_attention_over_unequal_lists(fp8, D, (slots - 1) // H + past, 1, (0, 1), kind)
