"""fp32 sequences small enough for the single-launch chunk loop (a cluster of 1 to 16 CTAs per unit): edges of its tiles and clusters, both
head sizes, stacked input, protected slots, a resumed cache, snapshots for the backward pass. Against the float64 oracle."""
import numpy as np
import pytest
import torch

from paper_2406_05317_b200 import workloads as wl
from tests.helpers import assert_close, loop_plan, to_device, to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,M,B,L,k,c_mult,per_head,bias,prot,cut", [
    (64, 16, 16, 256, 5, 1, False, False, 0, 0),
    (64, 1, 2, 9, 1, 1, False, False, 0, 0),
    (64, 13, 7, 50, 3, 2, True, True, 3, 0),          # nothing a multiple of four, a fill step, a short last chunk
    (128, 17, 18, 93, 3, 1, True, False, 0, 40),      # two calls, the second from a full cache
    (128, 8, 5, 64, 5, 2, False, True, 8, 0),         # every slot protected
])
def test_small_loop(d, M, B, L, k, c_mult, per_head, bias, prot, cut):
    from oracle import lococo_oracle as orc
    from paper_2406_05317_b200 import api
    w = wl.Workload("small_loop", 62, batch=2, heads=2, d=d, M=M, B=B, k=k, L=L, dtype="f32", weights_per_head=per_head,
                    qkv_scale=1.0, g_std=0.05, c_in_mult=c_mult)
    ctx = api.Lococo(w.batch, w.heads, d, M, k, B, dtype=torch.float32, c_in=w.c_in, weights_per_head=per_head)
    G, bvec = wl.make_weights(w, with_bias=bias)
    ctx.set_weights(to_device(G, "f32"), None if bvec is None else to_device(bvec, "f32"))
    ctx.set_protected_slots(prot)
    Q, K, V = wl.make_qkv(w)
    dQ, dK, dV = (to_device(x, "f32") for x in (Q, K, V))
    O = torch.empty_like(dQ)
    Kc = torch.zeros(w.batch, w.heads, M, d, device="cuda")
    Vc = torch.zeros_like(Kc)
    c, launches = 0, ctx.launch_count()
    for a, z in ((0, cut), (cut, L)) if cut else ((0, L),):
        sl = slice(a, z)
        c = ctx.process_sequence(dQ[:, :, sl], dK[:, :, sl], dV[:, :, sl], B, O[:, :, sl], Kc, Vc, c)
    assert ctx.launch_count() - launches == (2 if cut else 1)
    torch.cuda.synchronize()
    outs = []
    for n in range(w.batch):
        for h in range(w.heads):
            cache, parts = None, []
            for a, z in ((0, cut), (cut, L)) if cut else ((0, L),):      # chunk borders move with the cut
                o, *cache = orc.process_sequence(Q[n, h, a:z], K[n, h, a:z], V[n, h, a:z], G[h if per_head else 0], B,
                                                 bias=None if bvec is None else bvec[h if per_head else 0],
                                                 cache=cache, protected=prot)[:4]
                parts.append(o)
            outs.append((np.vstack(parts), cache[0], cache[1], cache[2]))
    Or, Kr, Vr = (np.stack(x).reshape(w.batch, w.heads, *x[0].shape) for x in list(zip(*outs))[:3])
    cr = outs[0][3]
    assert c == cr
    assert_close(to_host(O), Or, "f32", "O")
    assert_close(to_host(Kc)[:, :, :c], Kr[:, :, :c], "f32", "K cache")
    assert_close(to_host(Vc)[:, :, :c], Vr[:, :, :c], "f32", "V cache")


def test_the_loop_is_timed_on_request():
    from paper_2406_05317_b200 import api
    ctx = api.Lococo(1, 2, 64, 16, 5, 16, dtype=torch.float32)
    x = torch.randn(1, 2, 100, 64, device="cuda")
    ctx.set_weights(0.05 * torch.randn(1, 16, 64, 5, device="cuda"))
    O, Kc, Vc = torch.empty_like(x), torch.zeros(1, 2, 16, 64, device="cuda"), torch.zeros(1, 2, 16, 64, device="cuda")
    ctx.profile(True)
    ctx.process_sequence(x, x, x, 16, O, Kc, Vc, 0)
    ms, launches = ctx.profile_read(3)
    ctx.profile(False)
    assert launches == 1 and 0 < ms < 100


@pytest.mark.parametrize("batch,heads,d,M,B,L,k,c_mult,prot", [
    (1, 1, 64, 17, 33, 150, 7, 1, 0),         # wide clusters: CTAs of one and of two slots, of two and of three queries
    (1, 1, 64, 3, 40, 130, 9, 2, 1),          # fewer slots than CTAs would fit
    (3, 4, 64, 30, 21, 104, 5, 1, 5),         # CTAs with and without protected slots
    (2, 20, 128, 13, 9, 48, 3, 1, 0),         # clusters of a few CTAs; fill steps first
    (5, 30, 64, 18, 26, 120, 5, 1, 0),        # a CTA per unit
    (1, 2, 64, 65, 30, 190, 11, 1, 0),        # tiles of 8 positions; fill steps whose chunks several CTAs read
])
def test_small_loop_clusters(batch, heads, d, M, B, L, k, c_mult, prot):
    # Snapshots on (the gradients' inputs), so that what every CTA holds of the cache is seen after every chunk.
    from oracle import lococo_oracle as orc
    from paper_2406_05317_b200 import api
    w = wl.Workload("small_loop_clusters", 63, batch=batch, heads=heads, d=d, M=M, B=B, k=k, L=L, dtype="f32", weights_per_head=True,
                    qkv_scale=1.0, g_std=0.05, c_in_mult=c_mult)
    ctx = api.Lococo(batch, heads, d, M, k, B, dtype=torch.float32, c_in=w.c_in, weights_per_head=True)
    G, bias = wl.make_weights(w, with_bias=True)
    ctx.set_weights(to_device(G, "f32"), to_device(bias, "f32"))
    ctx.set_protected_slots(prot)
    Q, K, V = wl.make_qkv(w)
    dQ, dK, dV = (to_device(x, "f32") for x in (Q, K, V))
    O, Kc, Vc = torch.empty_like(dQ), torch.zeros(batch, heads, M, d, device="cuda"), torch.zeros(batch, heads, M, d, device="cuda")
    saved = torch.zeros(ctx.saved_bytes(L, B), dtype=torch.uint8, device="cuda")
    launches = ctx.launch_count()
    c = ctx.process_sequence(dQ, dK, dV, B, O, Kc, Vc, 0, saved)
    assert ctx.launch_count() - launches == 1
    torch.cuda.synchronize()
    chunks, step = -(-L // B), batch * heads * M * d
    size = (chunks * step * 4 + 255) // 256 * 256
    snaps = [saved[i * size:].view(torch.float32)[:chunks * step].view(chunks, batch, heads, M, d).cpu().numpy() for i in range(2)]
    for u in (0, batch * heads // 2, batch * heads - 1):
        n, h = divmod(u, heads)
        Or, Kr, Vr, cr, _, sK, sV, sc = orc.process_sequence(Q[n, h], K[n, h], V[n, h], G[h], B, bias=bias[h], protected=prot, want_snapshots=True)
        assert c == cr
        assert_close(to_host(O)[n, h], Or, "f32", "O")
        assert_close(to_host(Kc)[n, h], Kr, "f32", "K cache")
        assert_close(to_host(Vc)[n, h], Vr, "f32", "V cache")
        for i in range(chunks):
            for got, want in zip(snaps, (sK, sV)):
                if sc[i]:
                    assert_close(got[i, n, h, :sc[i]], want[i, :sc[i]], "f32", f"cache before chunk {i}")


def test_one_chunk_calls_back_to_back():
    # Three launches per call, and the next call's first one may not take its places while this call's last blends run: two of its blocks
    # on one SM take half as long again. The same calls as graphs start with an empty chip.
    from paper_2406_05317_b200 import api
    ctx = api.Lococo(1, 8, 128, 96, 21, 4, dtype=torch.float32)
    ctx.set_weights(0.02 * torch.randn(1, 96, 128, 21, device="cuda"))
    x = torch.randn(1, 8, 4, 128, device="cuda")
    outs, stream = [torch.empty_like(x) for _ in range(2)], torch.cuda.Stream()
    Kc, Vc = torch.randn(1, 8, 96, 128, device="cuda"), torch.randn(1, 8, 96, 128, device="cuda")
    stream.wait_stream(torch.cuda.current_stream())

    def call_us(buffers):                      # (one buffer: replayed from the third call on)
        best = float("inf")
        with torch.cuda.stream(stream):
            for _ in range(6):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record(stream)
                for i in range(40):
                    ctx.process_sequence(x, x, x, 4, outs[i % buffers], Kc, Vc, 96)
                b.record(stream)
                torch.cuda.synchronize()
                best = min(best, a.elapsed_time(b) * 1e3 / 40)
        return best

    assert call_us(2) < 1.25 * call_us(1)


@pytest.mark.parametrize("batch,heads,d,M,B,L,k,c_mult,prot,ctas,tile", [
    (1, 1, 64, 17, 33, 150, 7, 1, 0, range(9, 17), 3),       # (the cases above: what they say they cover)
    (1, 1, 64, 3, 40, 130, 9, 2, 1, range(2, 4), 2),
    (3, 4, 64, 30, 21, 104, 5, 1, 5, range(4, 17), 2),
    (2, 20, 128, 13, 9, 48, 3, 1, 0, range(2, 5), 2),
    (5, 30, 64, 18, 26, 120, 5, 1, 0, [1], 1),
    (1, 2, 64, 65, 30, 190, 11, 1, 0, range(9, 17), 2),
    (1, 1, 64, 16, 90, 363, 3, 1, 3, [16], 2),               # and the widest cluster, a slot each
    (1, 8, 64, 64, 90, 275, 3, 1, 0, range(8, 17), 0),       # tiles of four slots
    (5, 15, 64, 15, 45, 183, 3, 2, 2, [1, 2], None),
])
def test_small_loop_plans(batch, heads, d, M, B, L, k, c_mult, prot, ctas, tile):
    from paper_2406_05317_b200 import api
    plan = loop_plan(api.Lococo(batch, heads, d, M, k, B, dtype=torch.float32, c_in=c_mult * d), L, B)
    assert plan[0] in ctas and (tile is None or plan[2] == tile), plan
    test_small_loop_clusters(batch, heads, d, M, B, L, k, c_mult, prot)
