"""Row GEMMs with the tokens as the N operand: stage-by-stage parity at the sizes where the cut of an expert's rows into tiles
changes, for widths that leave a weight tile partly empty, forward-only calls and adapters."""
import numpy as np
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


def forms(layer, T=None, inference=False):
    """Which form each row GEMM of a layer's last step took: "one" CTA tiles, CTA "pairs" or "tokens" as N (from the CTAs that
    MOE_GEMM_TIMERS counts, one of each pair, apart for the two kinds of operands).  With T, before the step: clears the counters."""
    if T is not None:
        layer._ensure_ws(T, inference)
        layer.ws.zero_()
        return None
    ctas = layer.buffer("timers", torch.int64).view(2, 8, 8)[:, :, 7].cpu().tolist()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    out = {}
    for i, name in ((0, "F3"), (1, "F4"), (2, "B2"), (4, "B4")):
        rows, tokens = ctas[0][i], ctas[1][i]
        assert (rows, tokens) in ((sms, 0), (sms // 2, 0), (0, sms // 2)), (name, rows, tokens)
        out[name] = "tokens" if tokens else "pairs" if rows == sms // 2 else "one"
    return out


def step_forms(T, d, E, k, f):
    g = torch.Generator(device="cuda")
    g.manual_seed(T)
    n = lambda *s: torch.empty(*s, device="cuda").normal_(0, 0.05, generator=g).bfloat16()
    from paper_2608_00916_b200.binding import MoELayer
    layer = MoELayer(d, E, f, k)
    forms(layer, T)
    layer.forward(n(T, d), n(d, E), n(E, d, f), n(E, d, f), n(E, f, d))
    grads = layer.backward(n(T, d), 0.01)
    layer.poll()
    return forms(layer), grads["dx"]


@pytest.mark.parametrize("d,f,T,tokens", [
    (512, 512, 383, {"B2"}), (512, 512, 384, set()),                                 # 96 rows: dgrad-down at a narrow width
    (1024, 512, 479, {"B2"}), (1024, 512, 480, {"B2", "B4"}),                        # 120: dgrad gate/up
    (1024, 1024, 479, {"B2", "B4"}), (2048, 768, 400, {"F3", "B2", "B4"}),           # wider: below that as well; so gate/up
    (2048, 512, 191, {"F3", "B2", "B4"}), (2048, 512, 192, {"B2", "B4"}),            # 48: gate/up otherwise
    (3072, 1536, 319, {"B2", "B4"}), (3072, 1536, 320, {"B2"}),                      # 80: dgrad gate/up from d 3072 on
    (3072, 1536, 479, {"B2"}), (3072, 1536, 480, {"F3", "F4", "B2", "B4"}),          # 120
    (2048, 768, 479, {"F3", "B2", "B4"}), (2048, 768, 480, {"F3", "F4", "B2", "B4"}),          # 120: down,
    (1024, 1536, 479, {"B2", "B4"}), (1024, 1536, 480, {"F4", "B2", "B4"}),                    # also where f is wide,
    (1536, 1024, 480, {"B2", "B4"}), (2048, 512, 480, {"F3", "B2", "B4"}),                     # not where d or f is less
    (2048, 1536, 2559, {"F3", "F4", "B2", "B4"}), (2048, 1536, 2560, {"F3", "B2", "B4"}),      # 640: down
    (3136, 512, 2559, {"F3", "B2", "B4"}), (3136, 512, 2560, {"F3", "B2"}),          # 640: dgrad gate/up above d 3072
    (2048, 512, 12287, {"F3", "B2", "B4"}), (2048, 512, 12288, {"B2"}),              # 3072
    (2048, 1600, 6143, {"F3", "B2", "B4"}), (2048, 1600, 6144, {"B2", "B4"}),        # 1536: gate/up above f 1536
    (1024, 3136, 6143, {"B2", "B4"}), (1024, 3136, 6144, {"B4"}),                    # 1536: dgrad-down above f 3072
])
def test_form_of_each_row_gemm(d, f, T, tokens, monkeypatch):
    """Both sides of every line of the rule (8 experts, top-2: T / 4 rows per expert)."""
    monkeypatch.setenv("MOE_GEMM_TIMERS", "1")
    chosen, _ = step_forms(T, d, 8, 2, f)
    assert {n for n, form in chosen.items() if form == "tokens"} == tokens


@pytest.mark.parametrize("T,d,E,k,f", [
    (200, 2048, 20, 2, 1664),    # gate/up: 13 column tiles, so that row tiles are walked 16 at a time, the last group short; small tiles
    (1300, 2048, 20, 2, 1664),   # the same, pairs of blocks
    (300, 3136, 20, 2, 512),     # dgrad gate/up; small tiles
    (2300, 3136, 8, 2, 1536),    # down and dgrad gate/up, about 24 tiles of 192
    (250, 1024, 24, 2, 3136),    # dgrad-down
])
def test_tiles_walked_in_groups(T, d, E, k, f):
    inp = synth.make_inputs(synth.MoEShape(T, d, E, k, f), 600 + T, x_std=1.0)
    ofw, obw = oracle_run(inp, k, 0.05, dtype=np.float32)
    check_all(Run(inp, k), ofw, obw, 0.05, stages=False)


# Long K loops of the down GEMM, which runs with the tokens as N from f 1536 on.
LONG = [(500, 1024, 8, 2, 1536), (1030, 1088, 8, 2, 1600), (1900, 2048, 8, 2, 1536)]


@pytest.mark.parametrize("T,d,E,k,f", LONG)
def test_down_parity(T, d, E, k, f):
    test_parity(T, d, E, k, f)


@pytest.mark.parametrize("T,d,E,k,f", LONG)
def test_down_of_a_forward_only_call(T, d, E, k, f):
    test_forward_only_call_reads_and_writes_no_pad_rows(T, d, E, k, f)


@pytest.mark.parametrize("rank", [8, 16, 64])
def test_down_with_adapters(rank):
    lora_against_the_oracle(1030, 1088, 8, 2, 1600, rank, 98)


def test_measurement_switches_act_on_every_form(monkeypatch):
    """MOE_B4_PAIR puts dgrad gate/up on one-CTA tiles or pairs where the rule would take the tokens as N; the order in which
    MOE_ROW_GROUP walks the tiles changes no bit."""
    monkeypatch.setenv("MOE_GEMM_TIMERS", "1")
    chosen, dx = step_forms(1000, 2048, 8, 2, 1536)  # 250 rows per expert
    assert set(chosen.values()) == {"tokens"}
    for value, form in (("0", "one"), ("1", "pairs")):
        monkeypatch.setenv("MOE_B4_PAIR", value)
        forced, other = step_forms(1000, 2048, 8, 2, 1536)
        assert forced == {**chosen, "B4": form}
        assert torch.equal(other, dx)
    monkeypatch.delenv("MOE_B4_PAIR")
    for value in ("2", "5"):
        monkeypatch.setenv("MOE_ROW_GROUP", value)
        grouped, other = step_forms(1000, 2048, 8, 2, 1536)
        assert grouped == chosen and torch.equal(other, dx)
