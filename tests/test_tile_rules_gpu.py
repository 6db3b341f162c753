"""Stage-by-stage parity at the sizes where the choice of tile shape changes and where a staging unit of the GEMM
epilogues (32 rows x 64 columns) is only partly inside the output."""
import pytest
import torch

from paper_2608_00916_b200 import synth
from gpu_util import Run, oracle_run
from test_gpu_parity import check_all
from test_gpu_parity import test_expert_lora_against_the_oracle as lora_against_the_oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,d,E,k,f,seed", [
    (640, 192, 8, 2, 320, 71),    # 160 rows per expert: row GEMMs on pairs, weight gradients not
    (1024, 128, 8, 2, 192, 72),   # 256: row GEMMs on one-CTA tiles
    (1532, 192, 8, 2, 64, 73),    # 383: the last size with one-CTA weight gradients
    (1540, 320, 8, 2, 192, 74),   # 385: weight gradients on pairs, output rows and columns beyond the last full tile
    (1750, 128, 8, 2, 320, 75),   # 437: row GEMMs on pairs again
    (3080, 192, 8, 2, 128, 76),   # 770: dgrad-down on pairs as well
])
def test_tile_shape_boundaries(T, d, E, k, f, seed):
    inp = synth.make_inputs(synth.MoEShape(T, d, E, k, f), seed, x_std=1.0)
    ofw, obw = oracle_run(inp, k, 0.05)
    check_all(Run(inp, k), ofw, obw, 0.05)


@pytest.mark.parametrize("T", [65536 - 127, 65536, 65537])
def test_permutation_on_both_sides_of_its_token_limit(T):
    """512 tiles of 128 tokens are placed by one kernel, more by a scan and a scatter: same routing, same layer."""
    inp = synth.make_inputs(synth.MoEShape(T, 64, 8, 2, 64), 77, x_std=1.0)
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
