"""The fp32 backward pass of several chunks at a time (small problems): edges of its clusters, tiles and groups, against the
float64 oracle's gradients."""
import pytest
import torch

from paper_2406_05317_b200 import workloads as wl
from tests.helpers import to_device, to_host
from tests.test_gpu_backward import check_backward, check_gradients

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,heads,d,M,B,L,k,c_mult,per_head,bias", [
    (1, 1, 64, 17, 33, 150, 7, 1, False, True),       # CTAs of one and of two slots; a last chunk of 18
    (2, 3, 64, 48, 100, 403, 5, 1, True, True),       # a last chunk of three tokens, shorter than a tile of anything
    (1, 2, 64, 40, 20, 130, 63, 1, True, False),      # padding wider than a chunk: the first compress step ends inside it
    (1, 2, 128, 20, 7, 45, 9, 2, False, True),        # two fill steps, then a partly filled cache
    (5, 32, 64, 16, 16, 50, 5, 1, False, False),      # more units than SMs: a CTA per unit
    (1, 16, 128, 48, 512, 5632, 3, 1, False, True),   # a group's sizes, but its units would wait for one another: a step at a time
    (1, 8, 128, 48, 512, 10752, 3, 1, False, True),   # more than one group of chunks
    (1, 1, 64, 2, 300, 700, 1, 1, True, True),        # one tap, two slots, a first step without cache and padding
])
def test_grouped_backward(batch, heads, d, M, B, L, k, c_mult, per_head, bias):
    w = wl.Workload("grouped", 38, batch=batch, heads=heads, d=d, M=M, B=B, k=k, L=L, dtype="f32", weights_per_head=per_head, qkv_scale=1.0,
                    g_std=0.05, c_in_mult=c_mult)
    check_backward(w, bias=bias)


@pytest.mark.parametrize("batch,heads,d,M,B,L,k,c_mult,groups", [
    (1, 1, 64, 17, 33, 150, 7, 1, 1),
    (2, 3, 64, 48, 100, 403, 5, 1, 1),
    (1, 2, 64, 40, 20, 130, 63, 1, 1),
    (1, 2, 128, 20, 7, 45, 9, 2, 1),
    (5, 32, 64, 16, 16, 50, 5, 1, 1),
    (1, 16, 128, 48, 512, 5632, 3, 1, 0),
    (1, 8, 128, 48, 512, 10752, 3, 1, 2),
    (1, 1, 64, 2, 300, 700, 1, 1, 1),
    (1, 1, 64, 40, 30, 60, 5, 1, 0),                  # a fill step and one compress step: no chain
])
def test_which_calls_go_in_groups(batch, heads, d, M, B, L, k, c_mult, groups):
    # The way that the calls above are there for: five launches per group behind that of delta, or two and four per step.
    t = Training(wl.Workload("grouped_way", 38, batch=batch, heads=heads, d=d, M=M, B=B, k=k, L=L, dtype="f32", weights_per_head=True, qkv_scale=1.0,
                             g_std=0.05, c_in_mult=c_mult))
    launches = t.backward(torch.empty(t.scratch_bytes, dtype=torch.uint8, device="cuda"))[1]
    compress = [min(M, n * B) + min(B, L - n * B) > M for n in range(-(-L // B))]
    assert launches == (1 + 5 * groups if groups else 2 + sum(4 if x else 2 for x in compress))


class Training:
    """A forward pass with its snapshots; backward passes of it with a scratch of the test's own."""

    def __init__(self, w):
        from paper_2406_05317_b200 import api
        self.w, self.ctx = w, api.Lococo(w.batch, w.heads, w.d, w.M, w.k, w.B, dtype=torch.float32, c_in=w.c_in, weights_per_head=w.weights_per_head)
        self.G, self.bias = wl.make_weights(w, with_bias=True)
        self.ctx.set_weights(to_device(self.G, "f32"), to_device(self.bias, "f32"))
        self.host = (*wl.make_qkv(w), *wl.make_loss_projections(w))
        self.Q, self.K, self.V, self.PO, self.PK, self.PV = (to_device(x, "f32") for x in self.host)
        self.O = torch.empty_like(self.Q)
        caches = [torch.zeros(w.batch, w.heads, w.M, w.d, device="cuda") for _ in range(2)]
        self.saved = torch.empty(self.ctx.saved_bytes(w.L, w.B), dtype=torch.uint8, device="cuda")
        self.ctx.process_sequence(self.Q, self.K, self.V, w.B, self.O, *caches, 0, self.saved)
        self.scratch_bytes = self.ctx.backward_scratch_bytes(w.L, w.B)

    def backward(self, scratch, in_place=False):
        """Gradients, and how many launches they took. in_place: those of K and V take the place of K and V."""
        grads = [torch.empty_like(self.Q), self.K, self.V] if in_place else [torch.empty_like(self.Q) for _ in range(3)]
        dG, dbias = torch.zeros(self.G.shape, device="cuda"), torch.zeros(self.bias.shape, device="cuda")
        before = self.ctx.launch_count()
        self.ctx.process_sequence_backward(self.Q, self.K, self.V, self.O, self.w.B, self.saved, self.PO, self.PK, self.PV, *grads, dG, dbias, scratch)
        torch.cuda.synchronize()
        return dict(zip(("dQ", "dK", "dV", "dG", "dbias"), map(to_host, (*grads, dG, dbias)))), self.ctx.launch_count() - before

    def check(self, got, n, h):
        """Unit (n, h) against the oracle: with a weight set per head and one sequence all of its gradients are its own."""
        from oracle import lococo_oracle as orc
        assert self.w.weights_per_head and self.w.batch == 1
        Q, K, V, PO, PK, PV = (x[n, h] for x in self.host)
        ref = orc.process_sequence_grad(Q, K, V, self.G[h], self.w.B, PO, PK, PV, bias=self.bias[h])
        check_gradients(self.w, {"dQ": got["dQ"][n, h], "dK": got["dK"][n, h], "dV": got["dV"][n, h], "dG": got["dG"][h], "dbias": got["dbias"][h]},
                        dict(zip(("dQ", "dK", "dV", "dG", "dbias"), ref)))


def test_a_shorter_last_group_stays_inside_the_scratch():
    # 111 chunks in groups of 28, 28, 28 and 27: the tiles of 27 are few enough for two partial sums of the convolution each, those of 28 are not.
    w = wl.Workload("grouped_rest", 39, batch=1, heads=16, d=128, M=16, B=200, k=5, L=22200, dtype="f32", weights_per_head=True, qkv_scale=1.0, g_std=0.05)
    t = Training(w)
    room = torch.full((t.scratch_bytes + (16 << 20),), 0x5A, dtype=torch.uint8, device="cuda")
    got, launches = t.backward(room[:t.scratch_bytes])
    assert launches == 1 + 4 * 5
    assert bool((room[t.scratch_bytes:] == 0x5A).all())
    t.check(got, 0, 0)
    t.check(got, 0, 15)


def test_less_scratch():
    # Groups of as many chunks as the scratch holds; with what one chunk takes, and nothing more, a chunk at a time.
    units, d, M, B, L = 8, 64, 48, 64, 777
    t = Training(wl.Workload("grouped_less", 40, batch=1, heads=units, d=d, M=M, B=B, k=5, L=L, dtype="f32", weights_per_head=True, qkv_scale=1.0, g_std=0.05))
    one = units * (M + B) * 2 * d                                   # a gradient of all rows of [cache; chunk]
    least = sum((4 * n + 255) // 256 * 256 for n in (units * M * d, units * M * d, units * L, one * (1 + M // 16), units * M * (M + B)))
    assert least < t.scratch_bytes
    launches = []
    for size in (t.scratch_bytes, t.scratch_bytes // 2, t.scratch_bytes // 4, least):
        room = torch.full((size + (8 << 20),), 0x5A, dtype=torch.uint8, device="cuda")
        got, n = t.backward(room[:size])
        assert bool((room[size:] == 0x5A).all())
        t.check(got, 0, 5)
        launches.append(n)
    assert launches[0] == 1 + 5 and launches[0] < launches[1] < launches[2] and launches[3] == 2 + 4 * 13


def test_gradients_in_the_place_of_keys_and_values():
    # stacked input: dG reads both
    w = wl.Workload("grouped_place", 41, batch=1, heads=4, d=64, M=32, B=50, k=7, L=333, dtype="f32", weights_per_head=True, qkv_scale=1.0, g_std=0.05,
                    c_in_mult=2)
    t = Training(w)
    scratch = torch.empty(t.scratch_bytes, dtype=torch.uint8, device="cuda")
    assert t.backward(scratch)[1] == 1 + 5
    got, launches = t.backward(scratch, in_place=True)
    assert launches == 2 + 4 * 7
    for h in range(4):
        t.check(got, 0, h)
