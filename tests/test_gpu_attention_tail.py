"""Attention calls of so many lists that the last ones are cut finer than the others: outputs against fp64 over the pages' rows, with
lists of all lengths on both sides of where the finer parts begin."""
import numpy as np
import pytest
import torch

from paper_2601_07891_b200 import binding, synth

pytestmark = pytest.mark.gpu

H = 8


@pytest.mark.parametrize("B,L,D,G,fp8,longest,room,P", [
    (80, 1, 128, 4, False, 2000, 2000, 16),     # one part a list, then two
    (75, 1, 128, 4, True, 2800, 2800, 16),      # 8-bit rows: 600 lists of which half are cut
    (60, 2, 64, 2, False, 3700, 3700, 16),      # 960 lists in three parts, then four
    (77, 1, 128, 8, False, 1700, 1700, 16),     # no list long enough for a second part
    (230, 1, 64, 1, True, 1900, 1900, 16),      # 1840 lists
    (60, 1, 128, 4, False, 700, 32768, 16),     # short lists where there is room for long ones: seven parts each, none more
    (61, 1, 64, 4, True, 12000, 32768, 16),     # ... and some long ones
    (80, 1, 128, 4, False, 2000, 2016, 48),     # pages of three tiles
    (9, 2, 128, 4, True, 2500, 2500, 80),       # ... of five, the lists shared out by their lengths
])
def test_many_lists(B, L, D, G, fp8, longest, room, P):
    rng = np.random.default_rng(B)
    prefix = rng.integers(0, longest, size=B * L * H)
    edges = [n for n in (0, 1, 15, 16, 17, 639, 640, 641, 1279, 1280, 1281, longest) if n <= longest]
    prefix[:len(edges)] = edges
    prefix[-2 * len(edges)::2] = edges
    pages = (prefix + P - 1) // P
    first = np.concatenate([[0], np.cumsum(pages)[:-1]])
    max_pages = room // P + 1
    row = (D + synth.E4M3_ROW_TRAILER) // 2 if fp8 else D
    g = torch.Generator(device="cuda").manual_seed(B)
    raw = [torch.empty(int(pages.sum()) * P, D, device="cuda").normal_(generator=g).to(torch.bfloat16) for _ in range(2)]
    pools = [(synth.pack_rows_e4m3(x.float()) if fp8 else x).view(-1, P, row) for x in raw]
    table = torch.from_numpy(np.minimum(first[:, None] + np.arange(max_pages)[None, :], int(pages.sum()) - 1).astype(np.int32)).cuda()
    ctx = binding.Kvzap(128, 64, H, row, L, max_tokens=max(B, 128))
    cache = binding.kvzap_cache_create(ctx.handle, B, 16, P, *pools, max_pages)
    binding.kvzap_cache_import(ctx.handle, cache, torch.from_numpy(prefix.astype(np.int32)).cuda(), table, int(pages.sum()))
    Q = torch.empty(L, B, H * G, D, device="cuda").normal_(generator=g).to(torch.bfloat16)
    O = torch.full_like(Q, 7.0)
    for _ in range(2):                                       # the arrival counters are back where they were
        (binding.kvzap_decode_attention_fp8 if fp8 else binding.kvzap_decode_attention)(ctx.handle, cache, 0, L, Q, 0.1, O)
    torch.cuda.synchronize()
    assert ctx.poll_status() == 0

    def rows(pool, i):
        x = pool.view(-1, row)[int(first[i]) * P:int(first[i]) * P + int(prefix[i])]
        if not fp8:
            return x.double()
        b = x.contiguous().view(torch.uint8)
        return b[:, :D].contiguous().view(torch.float8_e4m3fn).double() * b[:, D:D + 4].contiguous().view(torch.float32).double()

    look = sorted(set(range(0, B * L * H, 7)) | set(range(len(edges))) | set(range(B * L * H - 3 * len(edges), B * L * H)))
    for i in look:
        b, l, h = i // (L * H), i // H % L, i % H
        got = O[l, b, h * G:(h + 1) * G].double()
        if prefix[i] == 0:
            assert (got == 0).all()
            continue
        k, v = rows(pools[0], i), rows(pools[1], i)
        want = torch.softmax(Q[l, b, h * G:(h + 1) * G].double() @ k.t() * 0.1, dim=1) @ v
        # probabilities and outputs rounded to bf16 once each, values below 5
        assert ((got - want).abs() <= 2e-2 + 2.0 ** -8 * want.abs()).all(), (i, prefix[i])
    binding.kvzap_cache_destroy(cache)
    ctx.close()
