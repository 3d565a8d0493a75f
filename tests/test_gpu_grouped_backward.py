"""The fp32 backward pass of several chunks at a time (small problems): edges of its clusters, tiles and groups, against the
float64 oracle's gradients."""
import pytest

from paper_2406_05317_b200 import workloads as wl
from tests.test_gpu_backward import check_backward

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
