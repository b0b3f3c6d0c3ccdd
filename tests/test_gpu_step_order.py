"""Decode steps enqueued, without a synchronisation anywhere, behind work that they must not run beside: a prompt chunk's
page assignment and compaction, a release, a step in another layout.  In one launch: the step directly behind is followed
by steps of other layers of the same layout, on grids large enough to overlap.  In two launches (more tiles than the
few-token kernel takes; linear surrogate; 8-bit inputs without a few-token layout): the update moves rows beside the
scoring.  Every list is compared with the selection by score of its whole stream, and no page is owned twice."""
import numpy as np
import pytest
import torch

from paper_2601_07891_b200 import binding, synth

pytestmark = pytest.mark.gpu

D_MODEL, H, D, W, P, TAU = 512, 8, 64, 32, 4, 0.1


class _Server:
    """A cache, its streams of tokens per (slot, layer), and calls that are made only when all inputs are there."""

    def __init__(self, hidden, B, L, trusted, n_rows, fp8=False):
        self.B, self.L, self.fp8 = B, L, fp8
        self.ctx = binding.Kvzap(D_MODEL, hidden, H, D, L, max_tokens=512, trusted_producers=trusted)
        for l in range(L):
            w = synth.mlp_weights(D_MODEL, hidden, H, 70 + l, "cuda", 0.3) if hidden else synth.linear_weights(D_MODEL, H, 70 + l, "cuda", 0.3)
            if fp8:
                binding.kvzap_set_weights_fp8(self.ctx.handle, l, *synth.quantize_e4m3(w[0]), *w[1:])
            else:
                self.ctx.set_weights(l, *w)
        self.max_pages = n_rows // P + 2
        self.n_pool = B * L * H * self.max_pages
        self.pools = [torch.zeros(self.n_pool, P, D, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
        self.cache = binding.kvzap_cache_create(self.ctx.handle, B, W, P, *self.pools, self.max_pages)
        self.calls, self.events, self.n_rows = [], [], n_rows
        self.active = [True] * B
        self.seed = 0

    def _inputs(self, n):
        self.seed += 1
        return (synth.hidden_states(n, D_MODEL, self.seed, "cuda"),) + tuple(synth.keys_values(H, n, D, 5000 + self.seed, "cuda"))

    def prompt(self, slot, n):
        for l in range(self.L):
            X, K, V = self._inputs(n)
            s = torch.zeros(n, H, dtype=torch.float32, device="cuda")
            self.calls.append(lambda l=l, X=X, K=K, V=V, s=s: binding.kvzap_prefill_to_cache(
                self.ctx.handle, self.cache, l, slot, X, K, V, TAU, s))
            self.events.append(("rows", slot, l, K, V, s))
        self.active[slot] = True

    def release(self, slot):
        self.calls.append(lambda: binding.kvzap_cache_release_seq(self.ctx.handle, self.cache, slot))
        self.events.append(("release", slot))
        self.active[slot] = False

    def step(self, a, e):
        n, B = e - a, self.B
        X = self._inputs(n * B)[0].view(n, B, D_MODEL)
        K, V = (t.view(n, B, H, D) for t in synth.keys_values(n * B, H, D, 9000 + self.seed, "cuda"))
        s = torch.zeros(n, B, H, dtype=torch.float32, device="cuda")
        if self.fp8:
            x, scale = synth.quantize_e4m3(X.view(n * B, D_MODEL))
            x, scale = x.view(n, B, D_MODEL), scale.view(n, B)
            self.calls.append(lambda: binding.kvzap_decode_step_fp8(self.ctx.handle, self.cache, a, e, x, scale, K, V, TAU, s))
        else:
            self.calls.append(lambda: binding.kvzap_decode_step(self.ctx.handle, self.cache, a, e, X, K, V, TAU, s))
        for b in range(B):
            if self.active[b]:
                for l in range(a, e):
                    self.events.append(("rows", b, l, K[l - a, b][:, None], V[l - a, b][:, None], s[l - a, b][None]))

    def check(self):
        torch.cuda.synchronize()
        for call in self.calls:
            call()
        torch.cuda.synchronize()
        assert self.ctx.poll_status() == 0
        streams = [[[] for _ in range(self.L)] for _ in range(self.B)]
        for e in self.events:
            if e[0] == "release":
                streams[e[1]] = [[] for _ in range(self.L)]
            else:
                streams[e[1]][e[2]].append(e[3:])
        lengths = torch.zeros(self.B, self.L, H, dtype=torch.int32, device="cuda")
        binding.kvzap_cache_lengths(self.ctx.handle, self.cache, lengths)
        lengths = lengths.cpu().numpy()
        out = [torch.zeros(self.n_rows, D, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
        n = torch.zeros(1, dtype=torch.int32, device="cuda")
        rng = np.random.default_rng(1)
        for b in range(self.B):
            for l in range(self.L):
                if not streams[b][l]:
                    assert (lengths[b, l] == 0).all()
                    continue
                keep = torch.cat([c[2] for c in streams[b][l]]) >= TAU
                keep[-W:] = True
                np.testing.assert_array_equal(lengths[b, l], keep.sum(0).cpu().numpy())
                if rng.random() < 0.1 or (b < 3 and l in (0, self.L - 1)):
                    kv = [torch.cat([c[i] for c in streams[b][l]], dim=1) for i in range(2)]
                    for h in range(H):
                        binding.kvzap_cache_export(self.ctx.handle, self.cache, b, l, h, *out, n)
                        for x, o in zip(kv, out):
                            assert torch.equal(o[:int(lengths[b, l, h])].view(torch.int16), x[h, keep[:, h]].view(torch.int16))
        prefix = torch.zeros(self.B * self.L * H, dtype=torch.int32, device="cuda")
        table = torch.zeros(prefix.numel(), self.max_pages, dtype=torch.int32, device="cuda")
        cursor = torch.zeros(1, dtype=torch.int32, device="cuda")
        binding.kvzap_cache_snapshot(self.ctx.handle, self.cache, prefix, table, cursor)
        pages = (prefix.cpu().numpy() + P - 1) // P
        owned = np.concatenate([t[:k] for t, k in zip(table.cpu().numpy(), pages)])
        assert len(np.unique(owned)) == len(owned) and owned.min() >= 0 and owned.max() < int(cursor) <= self.n_pool
        binding.kvzap_cache_destroy(self.cache)
        self.ctx.close()


@pytest.mark.parametrize("trusted", [True, False])
@pytest.mark.parametrize("B,L,group", [(6, 20, 10), (8, 6, 3), (130, 10, 5)])
def test_steps_of_layer_groups_behind_other_work(B, L, group, trusted):
    srv = _Server(512, B, L, trusted, 320)

    def groups(n):
        for _ in range(n):
            for a in range(0, L, group):
                srv.step(a, a + group)

    for b in range(3):
        srv.prompt(b, 70 + 30 * b)
    for r in range(5):
        srv.prompt(r % 3, 41)               # the last layer's chunk, then the steps
        groups(2)
        srv.release((r + 1) % 3)            # pages come back, the steps behind take some
        groups(2)
        srv.prompt((r + 1) % 3, 60)
        srv.step(0, L)                      # in another layout than its groups
        groups(3)
    srv.check()


@pytest.mark.parametrize("trusted", [True, False])
@pytest.mark.parametrize("hidden,B,L", [(512, 130, 20), (512, 6, 40), (0, 130, 20), (64, 6, 38)])
def test_steps_in_two_launches_behind_other_work(hidden, B, L, trusted):
    srv = _Server(hidden, B, L, trusted, 320)
    for b in range(3):
        srv.prompt(b, 70 + 30 * b)
    for r in range(5):
        srv.prompt(r % 3, 41)
        for _ in range(3):                  # behind the chunk, then behind one another
            srv.step(0, L)
        srv.release((r + 1) % 3)
        for _ in range(3):
            srv.step(0, L)
        srv.prompt((r + 1) % 3, 60)
    srv.check()


@pytest.mark.parametrize("trusted", [True, False])
def test_eight_bit_steps_in_two_launches_behind_a_release(trusted):
    srv = _Server(512, 130, 20, trusted, 320, fp8=True)
    for b in range(12):
        for _ in range(6):                  # from the 33rd step on rows leave the window and take pages
            srv.step(0, 20)
        srv.release(b)
    srv.step(0, 20)
    srv.check()
