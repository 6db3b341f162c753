"""Stage-by-stage parity at the sizes where the choice of tile shape changes (and that it does change there), and where
a staging unit of the GEMM epilogues (32 rows x 64 columns) is only partly inside the output."""
import pytest
import torch

from paper_2608_00916_b200 import synth
from gpu_util import Run, oracle_run, rel_fro
from test_gpu_parity import TOL, check_all
from test_gpu_parity import test_expert_lora_against_the_oracle as lora_against_the_oracle

pytestmark = pytest.mark.gpu


# The expert GEMMs in the order of their counters: with MOE_GEMM_TIMERS set a launch counts its CTAs (one of each pair).
KINDS = ("F3", "F4", "B2", "B3", "B4", "B5")
ROW = {"F3", "F4", "B4"}  # gate/up, down, dgrad gate/up; B2 is dgrad-down, B3 and B5 are the weight gradients


@pytest.fixture
def on_pairs(monkeypatch):
    """GEMMs of the last step of a layer that ran on CTA pairs.  Call once with the layer and T before the step, to clear
    the counters, and without T after it."""
    monkeypatch.setenv("MOE_GEMM_TIMERS", "1")

    def read(layer, T=None, lora=False):
        if T is not None:
            layer._ensure_ws(T)
            if lora:
                layer.ws = torch.empty(int(layer.lib.moe_lora_workspace_bytes(layer.h, T)), dtype=torch.uint8, device="cuda")
            layer.ws.zero_()
            return None
        ctas = layer.buffer("timers", torch.int64).view(16, 8)[:6, 7].cpu().tolist()
        sms = torch.cuda.get_device_properties(0).multi_processor_count
        assert all(c in (0, sms // 2, sms) for c in ctas)
        return {n for n, c in zip(KINDS, ctas) if c == sms // 2}

    return read


@pytest.mark.parametrize("T,pairs", [
    (520, set()), (524, ROW),            # 130 and 131 rows per expert: the expected tiles of the two shapes cross,
    (1048, ROW), (1052, set()),          # 262, 263: again,
    (1468, set()), (1472, ROW),          # 367, 368: and again
    (1532, ROW), (1536, ROW | {"B3", "B5"}),                          # 383, 384: weight gradients
    (3068, ROW | {"B3", "B5"}), (3072, ROW | {"B2", "B3", "B5"}),     # 767, 768: dgrad-down
])
def test_tile_shape_of_each_gemm(T, pairs, on_pairs):
    """The shape the rule selects on both sides of each of its lines, and the layer's parity there."""
    inp = synth.make_inputs(synth.MoEShape(T, 128, 8, 2, 128), 70, x_std=1.0)
    ofw, obw = oracle_run(inp, 2, 0.05)
    r = Run(inp, 2)
    on_pairs(r.layer, T)
    check_all(r, ofw, obw, 0.05)
    assert on_pairs(r.layer) == pairs


@pytest.mark.parametrize("T,pairs", [(1536, ROW), (2812, ROW), (2816, ROW | {"B3", "B5"})])
def test_tile_shape_of_accumulating_gemms(T, pairs, on_pairs):
    """384, 703 and 704 rows per expert: weight gradients that accumulate change shape later than those that do not; twice the
    same micro-batch on buffers of zeros gives twice the oracle's gradient."""
    d, E, k, f = 128, 8, 2, 192
    inp = synth.make_inputs(synth.MoEShape(T, d, E, k, f), 70, x_std=1.0)
    _, obw = oracle_run(inp, k, 0.05)
    r = Run(inp, k)
    acc = {"dW_r": torch.zeros(d, E, device="cuda"), "dW_gate": torch.zeros(E, d, f, device="cuda"),
           "dW_up": torch.zeros(E, d, f, device="cuda"), "dW_down": torch.zeros(E, f, d, device="cuda")}
    for _ in range(2):
        on_pairs(r.layer, T)
        r.forward()
        r.layer.backward_accumulate(r.dev["dy"], 0.05, acc)
        r.layer.poll()
        assert on_pairs(r.layer) == pairs
    for n in acc:
        assert rel_fro(acc[n].cpu().numpy(), 2.0 * obw[n]) <= TOL, n


@pytest.mark.parametrize("T,pairs", [(520, set()), (524, ROW), (1048, ROW), (1052, set()), (1468, set()), (1472, ROW),
                                     (3072, ROW | {"B2"})])
def test_tile_shape_of_the_adapted_gemms(T, pairs, on_pairs):
    """The large GEMMs of an adapter step take the shapes of the plain layer; both shapes give the same bits."""
    d, E, k, f = 128, 8, 2, 128
    inp = synth.make_inputs(synth.MoEShape(T, d, E, k, f), 70, x_std=1.0)
    lo = {n: torch.empty(*s, dtype=torch.bfloat16, device="cuda").normal_(0, 0.05) for n, s in (
        ("A1", (E, d, 16)), ("B1_gate", (E, 16, f)), ("B1_up", (E, 16, f)), ("A2", (E, f, 16)), ("B2", (E, 16, d)))}

    def step(flags):
        r = Run(inp, k, flags=flags)
        v = r.dev
        on_pairs(r.layer, T, lora=True)
        y = r.layer.lora_forward(v["x"], v["W_r"], v["W_gate"], v["W_up"], v["W_down"], lo, 2.0)["y"]
        g = r.layer.lora_backward(v["dy"], 0.02)
        r.layer.poll()
        return on_pairs(r.layer), {"y": y, **g}

    chosen, out = step(0)
    assert chosen == pairs
    for flags in (1, 2):  # forced: CTA pairs, one-CTA tiles
        forced, other = step(flags)
        assert forced == (ROW | {"B2"} if flags == 1 else set())
        for n in out:
            assert torch.equal(out[n], other[n]), n


@pytest.mark.parametrize("T,d,E,k,f,seed", [
    (640, 192, 8, 2, 320, 71),    # 160 rows per expert: row GEMMs on pairs, weight gradients not
    (1024, 128, 8, 2, 192, 72),   # 256: the same
    (1532, 192, 8, 2, 64, 73),    # 383: the last size with one-CTA weight gradients
    (1540, 320, 8, 2, 192, 74),   # 385: weight gradients on pairs, output rows and columns beyond the last full tile
    (1750, 128, 8, 2, 320, 75),   # 437: the same
    (3080, 192, 8, 2, 128, 76),   # 770: dgrad-down on pairs as well
])
def test_tile_shape_boundaries(T, d, E, k, f, seed):
    inp = synth.make_inputs(synth.MoEShape(T, d, E, k, f), seed, x_std=1.0)
    ofw, obw = oracle_run(inp, k, 0.05)
    check_all(Run(inp, k), ofw, obw, 0.05)


@pytest.mark.parametrize("T,E", [(40960, 8), (40961, 8), (65536 - 127, 8), (65536, 8), (65537, 8), (65536, 32), (65537, 32)])
def test_permutation_on_both_sides_of_its_token_limit(T, E):
    """320 tiles of 128 tokens (512 from 32 experts on) are placed by one kernel, more by a scan and a scatter: same routing,
    same layer."""
    inp = synth.make_inputs(synth.MoEShape(T, 64, E, 2, 64), 77, x_std=1.0)
    ofw, obw = oracle_run(inp, 2, 0.05)
    check_all(Run(inp, 2), ofw, obw, 0.05)


@pytest.mark.parametrize("T,d,E,k,f,seed,flags", [
    (5, 64, 16, 2, 64, 81, 0),       # experts with one row or none
    (150, 192, 16, 2, 320, 82, 0),   # about 19 rows: one group of 32 per tile
    (1030, 128, 16, 2, 192, 83, 1),  # about 129 rows on pairs: the second half empty or nearly so
    (770, 256, 16, 2, 256, 84, 2),   # about 96 rows: the last group of 32 just used or just not
    (2000, 128, 8, 2, 128, 85, 0),   # about 500 rows
])
def test_scoring_never_uses_pad_rows(T, d, E, k, f, seed, flags):
    """A forward-only call neither clears nor stores the pad rows of its buffers: with a workspace full of NaN bit
    patterns its result is bitwise that of the training forward, which does."""
    inp = synth.make_inputs(synth.MoEShape(T, d, E, k, f), seed, x_std=1.0)
    train = Run(inp, k, flags=flags).forward()
    r = Run(inp, k, flags=flags)
    v = r.dev
    r.layer._ensure_ws(T, inference=True)
    r.layer.ws.fill_(0xFF)
    got = r.layer.forward(v["x"], v["W_r"], v["W_gate"], v["W_up"], v["W_down"], inference=True)
    r.layer.poll()
    assert torch.equal(got["y"], train["y"])
    assert torch.isfinite(got["y"].float()).all()


@pytest.mark.parametrize("T,d,E,k,f,rank,seed", [
    (640, 192, 8, 2, 320, 16, 91),    # 160 rows per expert: gate/up, down and dgrad gate/up on pairs
    (1024, 128, 8, 2, 192, 8, 92),    # 256: pairs whose second half is often empty
    (3080, 192, 8, 2, 128, 64, 93),   # 770: dgrad-down on pairs as well, largest rank
])
def test_adapters_on_pairs(T, d, E, k, f, rank, seed):
    lora_against_the_oracle(T, d, E, k, f, rank, seed)
