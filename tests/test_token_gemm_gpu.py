"""Row GEMMs with the tokens as the N operand: stage-by-stage parity at the sizes where the cut of an expert's rows into tiles
changes, for widths that leave a weight tile partly empty, forward-only calls and adapters."""
import pytest
import torch

from paper_2608_00916_b200 import synth
from gpu_util import Run, oracle_run
from test_gpu_parity import check_all
from test_gpu_parity import test_expert_lora_against_the_oracle as lora_against_the_oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,d,E,k,f", [
    (5, 2048, 16, 2, 512),       # experts with a row or none: 16 tokens
    (60, 2048, 8, 2, 512),       # about 15 and 16 rows
    (250, 2112, 8, 2, 512),      # about 62; the second weight tile holds 64 features
    (500, 2048, 8, 2, 576),      # about 125; three weight tiles, half of the last one empty
    (515, 2048, 8, 2, 768),     # about 129
    (1030, 2048, 8, 2, 832),     # about 257: one tile of 256 or two of 144
    (1900, 2048, 8, 2, 512),     # about 475: two tiles, the last one shorter
])
def test_parity(T, d, E, k, f):
    inp = synth.make_inputs(synth.MoEShape(T, d, E, k, f), 400 + T, x_std=1.0)
    ofw, obw = oracle_run(inp, k, 0.05)
    check_all(Run(inp, k), ofw, obw, 0.05)


@pytest.mark.parametrize("T,d,E,k,f", [(5, 2048, 16, 2, 512), (450, 2112, 8, 2, 832), (1030, 2048, 16, 2, 512), (2000, 2048, 8, 2, 512)])
def test_forward_only_call_reads_and_writes_no_pad_rows(T, d, E, k, f):
    """With a workspace full of NaN patterns the result is bitwise that of the training forward."""
    inp = synth.make_inputs(synth.MoEShape(T, d, E, k, f), 85, x_std=1.0)
    train = Run(inp, k).forward()
    r = Run(inp, k)
    v = r.dev
    r.layer._ensure_ws(T, inference=True)
    r.layer.ws.fill_(0xFF)
    got = r.layer.forward(v["x"], v["W_r"], v["W_gate"], v["W_up"], v["W_down"], inference=True)
    r.layer.poll()
    assert torch.equal(got["y"], train["y"]) and torch.isfinite(got["y"].float()).all()


@pytest.mark.parametrize("T,d,E,k,f,rank,seed", [(70, 2048, 8, 2, 512, 16, 95), (1030, 2112, 8, 2, 832, 8, 96), (520, 2048, 8, 2, 512, 64, 97)])
def test_adapters(T, d, E, k, f, rank, seed):
    lora_against_the_oracle(T, d, E, k, f, rank, seed)


def test_one_expert_takes_every_token():
    """Loads of 0, a few and all tokens side by side."""
    inp = synth.make_inputs(synth.MoEShape(700, 2048, 16, 2, 512), 7, x_std=1.0, skew=True)
    ofw, obw = oracle_run(inp, 2, 0.1)
    check_all(Run(inp, 2), ofw, obw, 0.1)
