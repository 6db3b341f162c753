"""dW_r on both sides of the token count up to which it comes from one slice, written and added."""
import pytest
import torch

from paper_2608_00916_b200 import synth
from gpu_util import Run, oracle_run, rel_fro
from test_gpu_parity import TOL

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [1, 63, 512, 513])
@pytest.mark.parametrize("E,offset", [(8, 0), (136, 0), (40, 1)])
def test_router_weight_gradient(T, E, offset):
    """offset: an output that is not 16-byte aligned takes the partial sums at any size."""
    d, f, k = 192, 64, 2
    inp = synth.make_inputs(synth.MoEShape(T, d, E, k, f), 500 + T, x_std=1.0)
    _, obw = oracle_run(inp, k, 0.05)
    r = Run(inp, k)
    r.forward()
    flat = torch.full((d * E + 4,), 7.0, device="cuda")
    dW_r = flat[offset:offset + d * E].view(d, E)
    r.layer.backward(r.dev["dy"], 0.05, grads={"dW_r": dW_r})
    r.layer.poll()
    assert rel_fro(dW_r.cpu().numpy(), obw["dW_r"]) <= TOL
    assert (flat[:offset] == 7.0).all() and (flat[offset + d * E:] == 7.0).all()
    acc = {n: torch.zeros(s, device="cuda") for n, s in (("dW_gate", (E, d, f)), ("dW_up", (E, d, f)), ("dW_down", (E, f, d)))}
    once = dW_r.clone()
    r.forward()
    r.layer.backward_accumulate(r.dev["dy"], 0.05, {"dW_r": dW_r, **acc})
    r.layer.poll()
    assert torch.equal(dW_r, once + once)  # the same sums, added once
