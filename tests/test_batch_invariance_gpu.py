"""A token's logits, experts, gates and output are the same bits alone and in a batch of any size: every sum over the model width
runs in one order, whichever form of a kernel the number of tokens selects."""
import pytest
import torch

from paper_2608_00916_b200.binding import FLAG_ROUTER_FP32, MoELayer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,E,k,f,T,flags", [
    (512, 128, 8, 64, 20000, 0),                # 32, 64 and 128 tokens of a tile to a CTA of the router
    (320, 136, 4, 64, 20000, 0),                # two lanes' columns: an accumulator for each 128 experts
    (128, 24, 2, 64, 20000, FLAG_ROUTER_FP32),  # the three terms of an fp32 router weight
    (192, 12, 3, 64, 9000, 0),                  # the router for expert counts that are not a multiple of 8
    (2048, 128, 8, 512, 9000, 0),               # row GEMMs on tokens, on pairs and on one-CTA tiles
    (1024, 32, 4, 1536, 9000, 0),               # the down GEMM as well
])
def test_a_token_alone_and_in_a_batch(d, E, k, f, T, flags):
    g = torch.Generator(device="cuda")
    g.manual_seed(d + E)
    n = lambda *s: torch.empty(*s, device="cuda").normal_(generator=g)
    W_r = n(d, E) / d**0.5
    if not flags & FLAG_ROUTER_FP32:
        W_r = W_r.bfloat16()
    x = n(T, d).bfloat16()
    W = [(0.05 * n(E, *s)).bfloat16() for s in ((d, f), (d, f), (f, d))]
    layer = MoELayer(d, E, f, k, flags)
    names = ("logits", "idx", "gates", "y")
    batch = layer.forward(x, W_r, *W, want_logits=True)
    for t0, t1 in ((0, 1), (7, 40), (100, 700), (1000, 6000), (0, T - 9)):
        part = layer.forward(x[t0:t1], W_r, *W, want_logits=True)
        layer.poll()
        for name in names:
            assert torch.equal(part[name], batch[name][t0:t1]), (name, t0, t1)
