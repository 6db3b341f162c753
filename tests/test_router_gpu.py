"""The tensor-core router at the sizes where it changes form: the number of CTAs that share a token tile, the columns a lane
holds, and token counts around the tokens of a CTA and of a tile."""
import numpy as np
import pytest
import torch

from paper_2608_00916_b200 import synth
from gpu_util import Run, oracle_run
from test_gpu_parity import check_all, check_routing
from test_routing_nonfinite import check_picks

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,d,E,k", [
    (1, 512, 128, 8), (31, 512, 128, 8), (33, 512, 128, 8),        # four CTAs to a tile, 32 tokens each, most of them idle
    (129, 512, 64, 6), (2047, 512, 128, 16),
    (200, 64, 16, 2), (200, 128, 16, 2), (200, 192, 24, 4),        # one to three K blocks
    (33, 512, 256, 32), (300, 512, 136, 8),                        # two groups of four columns to a lane
    (4736, 512, 40, 3), (4737, 512, 40, 3),                        # 148 SMs: two CTAs to a tile
    (18944, 128, 16, 2), (18945, 128, 16, 2),                      # one: as many as SMs, more
    (4737, 256, 200, 4), (9473, 256, 136, 2),                      # more than 128 experts: two CTAs to a tile
    (4096, 256, 40, 3), (4097, 256, 40, 3),                        # four CTAs to a tile, two
    (9472, 128, 40, 3), (9473, 128, 40, 3),                        # two, one
    (4096, 128, 16, 2), (4097, 128, 16, 2),                        # fewer than 32 experts: four, one
    (500, 256, 16, 2), (500, 320, 16, 2), (500, 448, 136, 2),      # four chains of one K block, of one or two
])
def test_routing_in_every_form(T, d, E, k):
    inp = synth.make_inputs(synth.MoEShape(T, d, E, k, 64), 300 + T % 97, x_std=1.0)
    ofw, obw = oracle_run(inp, k, 0.05)
    check_all(Run(inp, k), ofw, obw, 0.05, stages=T < 3000)


@pytest.mark.parametrize("T,d", [(40, 64), (40, 192), (700, 512), (5000, 128), (10000, 192)])
def test_fp32_router_weight_splits_over_its_terms(T, d):
    """The K blocks of an fp32 weight's three terms are shared out like those of one."""
    from paper_2608_00916_b200.binding import FLAG_ROUTER_FP32, MoELayer
    E, k, f = 32, 4, 64
    g = torch.Generator(device="cuda")
    g.manual_seed(d)
    n = lambda *s: torch.empty(*s, device="cuda").normal_(generator=g)
    x, W_r = n(T, d).bfloat16(), n(d, E) / d**0.5
    Wg, Wu, Wd = ((0.1 * n(E, *s)).bfloat16() for s in ((d, f), (d, f), (f, d)))
    layer = MoELayer(d, E, f, k, FLAG_ROUTER_FP32)
    out = layer.forward(x, W_r, Wg, Wu, Wd, want_logits=True)
    layer.poll()
    ref = x.double() @ W_r.double()
    # Each of the 3 d / 16 steps of the tensor cores drops up to a last place, 2^-23, of a partial sum of about 1 / 2, and 3 d / 64 of
    # them follow one another: 2^-24 * 3 d / 64 = 1.4e-6 at d 512 if all dropped that much.  Measured rms 0.07e-6 (d 64) to 0.45e-6
    # (d 512); the bound stands between that and the 2.4e-6 that a lost third term costs.
    rms = lambda e: e.pow(2).mean().sqrt().item()
    assert rms(out["logits"].double() - ref) <= 1e-6
    # what that would miss: without its third term, or the second, the weight is off by much more
    hi = W_r.bfloat16()
    mid = (W_r - hi.float()).bfloat16()
    assert rms(x.double() @ (hi.double() + mid.double()) - ref) > 2e-6
    check_picks(out, k, E)


def test_small_and_large_clusters_agree_on_ties():
    """Tokens with exactly equal logits (two equal columns of W_r, repeated) take the lowest index in every form."""
    d, E, k = 512, 128, 8
    for T in (16, 5000, 20000):
        inp = synth.make_inputs(synth.MoEShape(T, d, E, k, 64), 5, x_std=1.0, guard=False)
        inp["W_r"][:, 64:] = inp["W_r"][:, :64]
        r = Run(inp, k)
        fw = r.forward()
        logits, idx = fw["logits"].cpu().numpy(), fw["idx"].cpu().numpy()
        assert np.array_equal(logits[:, :64], logits[:, 64:])
        assert np.array_equal(idx, np.argsort(-logits, axis=1, kind="stable")[:, :k])


@pytest.mark.parametrize("E,k", [(16, 2), (136, 4)])
@pytest.mark.parametrize("offset", [1, 2, 3])
def test_a_bias_anywhere_in_a_parameter_buffer(E, k, offset):
    """A view into a flat buffer of fp32 parameters is aligned to 4 bytes only: same results as from an aligned bias, through the
    plain, forward-only, adapter and expert-parallel calls."""
    from paper_2608_00916_b200 import ep
    T, d, f, r = 300, 128, 64, 8
    g = torch.Generator(device="cuda")
    g.manual_seed(E)
    n = lambda *s: torch.empty(*s, device="cuda").normal_(generator=g)
    x, W_r = n(T, d).bfloat16(), (n(d, E) / d**0.5).bfloat16()
    W = [(0.1 * n(E, *s)).bfloat16() for s in ((d, f), (d, f), (f, d))]
    lora = {m: (0.1 * n(E, *s)).bfloat16() for m, s in
            (("A1", (d, r)), ("B1_gate", (r, f)), ("B1_up", (r, f)), ("A2", (f, r)), ("B2", (r, d)))}
    aligned = n(E)
    flat = torch.zeros(E + 4, device="cuda")
    view = flat[offset:offset + E]
    view.copy_(aligned)
    from paper_2608_00916_b200.binding import MoELayer

    def calls(b_r):
        layer = MoELayer(d, E, f, k)
        outs = [layer.forward(x, W_r, *W, b_r=b_r, want_logits=True), layer.forward(x, W_r, *W, b_r=b_r, inference=True),
                layer.lora_forward(x, W_r, *W, lora, 2.0, b_r=b_r)]
        layer.poll()
        rank = ep.EPRank(d, E, f, k, 1, 0, T * k)
        rank.set_peers([rank.own_ws.data_ptr()])
        return outs + [rank.route(x, W_r, b_r)]

    for want, got in zip(calls(aligned), calls(view)):
        for name in want:
            assert want[name] is None or torch.equal(want[name], got[name]), name


@pytest.mark.parametrize("d,E,k,other", [(64, 16, 16, 2), (64, 256, 32, 4)])
def test_layers_that_share_a_form_of_the_router(d, E, k, other):
    """The shared-memory limit of a kernel belongs to the device, not to a layer: one that needs less leaves room for the other."""
    T, f = 20000, 64
    inp = synth.make_inputs(synth.MoEShape(T, d, E, k, f), 9, x_std=1.0, guard=False)
    large, small = Run(inp, k), Run(inp, other)
    first = {n: t.clone() for n, t in large.forward().items() if t is not None}
    small.forward()
    again = large.forward()
    assert all(torch.equal(first[n], again[n]) for n in first)


@pytest.mark.parametrize("E,k", [(16, 2), (136, 4), (12, 2)])
@pytest.mark.parametrize("offset", [1, 2, 3])
def test_fp32_and_int32_outputs_anywhere_in_a_buffer(E, k, offset):
    """C entry points: logits, gates, indices, counts, order, aux loss and dW_r that are aligned to 4 bytes only."""
    import ctypes as C
    T, d, f = 300, 128, 64
    inp = synth.make_inputs(synth.MoEShape(T, d, E, k, f), 11, x_std=1.0, guard=False)
    r = Run(inp, k)
    fw = r.forward()
    bw = r.backward(0.05)
    shapes = {"idx": (T, k), "gates": (T, k), "counts": (E,), "perm": (T * k,), "aux": (1,), "logits": (T, E), "dW_r": (d, E)}
    flat, out = {}, {}
    for n, s in shapes.items():
        want = fw[n] if n in fw else bw[n]
        flat[n] = torch.full((want.numel() + 8,), 7, dtype=want.dtype, device="cuda")
        out[n] = flat[n][offset:offset + want.numel()].view(s)
    y, layer, v = torch.empty_like(fw["y"]), r.layer, r.dev
    p = lambda t: C.c_void_p(t.data_ptr())
    stream = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert layer.lib.moe_forward(layer.h, T, p(v["x"]), p(v["W_r"]), None, None, p(v["W_gate"]), p(v["W_up"]), p(v["W_down"]), p(y),
                                 p(out["idx"]), p(out["gates"]), p(out["counts"]), p(out["perm"]), p(out["aux"]), p(out["logits"]),
                                 p(layer.ws), layer.ws.numel(), stream) == 0
    layer.backward(v["dy"], 0.05, grads={"dW_r": out["dW_r"]})
    layer.poll()
    for n in shapes:
        want = fw[n] if n in fw else bw[n]
        if n == "dW_r":  # partial sums instead of one slice of the tokens
            assert (out[n] - want).norm().item() <= 1e-5 * want.norm().item()
        else:
            assert torch.equal(out[n].reshape(want.shape), want), n
        assert (flat[n][:offset] == 7).all() and (flat[n][offset + want.numel():] == 7).all(), n
