"""The generation-stage kernel (one token per step, in place) in each of its forms: a cluster of four or two CTAs per unit, a
CTA per unit, two units per CTA; narrow and wide kernels, weights per head, protected slots, views with
strides. Against the float64 oracle."""
import numpy as np
import pytest
import torch

from paper_2406_05317_b200 import workloads as wl
from tests.helpers import assert_close, to_device, to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,heads,k,per_head,prot", [
    (1, 1, 1, False, 0),       # one unit, one tap: three CTAs of the cluster have none
    (2, 16, 21, True, 4),      # 32 units: clusters of four
    (3, 12, 21, False, 0),     # 36 units: clusters of two, of four they would take two rounds
    (5, 8, 5, False, 0),       # 40 units: clusters of two
    (5, 16, 27, True, 0),      # 80 units: a CTA each, the widest kernel
    (5, 31, 3, False, 2),      # 155 units: pairs, an odd unit over
    (5, 32, 21, True, 0),      # pairs of one head, an odd sequence over
])
def test_generation_kernel(batch, heads, k, per_head, prot):
    from oracle import lococo_oracle as orc
    from paper_2406_05317_b200 import api
    M, d, steps = 128, 128, 3
    w = wl.Workload("gen", 63, batch=batch, heads=heads, d=d, M=M, B=1, k=k, L=M + steps, dtype="bf16", weights_per_head=per_head,
                    qkv_scale=0.0884, g_std=0.02)
    G, _ = wl.make_weights(w)
    # (a positive bias keeps the rows of Eq. 7 away from zero sums, where it is discontinuous)
    bvec = wl.round_to_bf16(np.full((heads if per_head else 1, M), 0.05, dtype=np.float32))
    Q, K, V = wl.make_qkv(w)
    # buffers with room between the sequences and the heads; the first M tokens are the cache to start from
    def strided(x):
        t = torch.zeros(batch, heads + 1, x.shape[2] + 3, d, dtype=torch.bfloat16, device="cuda")[:, :heads, :x.shape[2]]
        t.copy_(to_device(x, "bf16"))
        return t
    dQ, dK, dV = (strided(x[:, :, M:]) for x in (Q, K, V))
    Kc, Vc = strided(K[:, :, :M]), strided(V[:, :, :M])
    O = torch.zeros_like(dQ)
    ctx = api.Lococo(batch, heads, d, M, k, 1, weights_per_head=per_head)
    ctx.set_weights(to_device(G, "bf16"), to_device(bvec, "bf16"))
    ctx.set_protected_slots(prot)
    saved = torch.empty(ctx.saved_bytes(steps, 1), dtype=torch.uint8, device="cuda")
    before = ctx.launch_count()
    assert ctx.process_sequence(dQ[:, :, :1], dK[:, :, :1], dV[:, :, :1], 1, O[:, :, :1], Kc, Vc, M) == M
    assert ctx.launch_count() - before == 1                       # one kernel: nothing is copied back
    assert ctx.process_sequence(dQ[:, :, 1:], dK[:, :, 1:], dV[:, :, 1:], 1, O[:, :, 1:], Kc, Vc, M, saved) == M
    torch.cuda.synchronize()
    assert ctx.device_status() == api.OK
    for n in range(batch):
        for h in range(0, heads, max(1, heads // 4)):
            g = h if per_head else 0
            Or, Kr, Vr, _, _ = orc.process_sequence(Q[n, h, M:], K[n, h, M:], V[n, h, M:], G[g], 1, bias=bvec[g],
                                                    cache=(K[n, h, :M], V[n, h, :M], M), protected=prot)
            assert_close(to_host(O[n, h]), Or, "bf16", f"O {n} {h}")
            assert_close(to_host(Kc[n, h]), Kr, "bf16", f"K cache {n} {h}")
            assert_close(to_host(Vc[n, h]), Vr, "bf16", f"V cache {n} {h}")


def test_no_second_round_of_clusters():
    # A step of 33 to 37 units takes about as long as one of 32: as clusters of four these do not all run at the same time (the
    # groups of SMs that a cluster lies within are no multiples of four), and a second round would double the step.
    from paper_2406_05317_b200 import api

    def step_us(units, steps=50):
        g = torch.Generator(device="cuda").manual_seed(units)
        new = lambda *s: (0.1 * torch.randn(*s, device="cuda", generator=g)).to(torch.bfloat16)
        ctx = api.Lococo(1, units, 128, 128, 21, 1)
        ctx.set_weights(new(1, 128, 128, 21))
        Q, K, V, Kc, Vc = new(1, units, 1, 128), new(1, units, 1, 128), new(1, units, 1, 128), new(1, units, 128, 128), new(1, units, 128, 128)
        O, stream = torch.empty_like(Q), torch.cuda.Stream()
        stream.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(stream):
            ctx.process_sequence(Q, K, V, 1, O, Kc, Vc, 128)
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=stream):
                for _ in range(steps):
                    ctx.process_sequence(Q, K, V, 1, O, Kc, Vc, 128)
            best = float("inf")
            for _ in range(6):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record(stream)
                graph.replay()
                b.record(stream)
                torch.cuda.synchronize()
                best = min(best, a.elapsed_time(b) * 1e3 / steps)
        assert ctx.device_status() == api.OK
        return best

    assert max(step_us(34), step_us(37)) < 1.4 * step_us(32)


@pytest.mark.parametrize("batch,heads,k,per_head,prot", [
    (1, 149, 1, False, 0),     # the fewest units that share SMs; one tap: fewer weight pieces than ring stages
    (3, 99, 27, True, 3),      # one unit more than run at the same time; the most taps
    (7, 43, 5, False, 128),    # 301 units; every slot kept
])
def test_two_ctas_per_sm(batch, heads, k, per_head, prot):
    test_generation_kernel(batch, heads, k, per_head, prot)
