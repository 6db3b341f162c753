"""The order in which the tiles of the expert GEMMs are walked: every tile once, whatever the loads and the group size."""
import numpy as np
import pytest
import torch

from paper_2608_00916_b200 import synth
from paper_2608_00916_b200.binding import MoELayer
from gpu_util import Run, oracle_run
from test_gpu_parity import check_all

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flags", [0, 1, 2])  # the default rule, CTA pairs, one-CTA tiles
@pytest.mark.parametrize("T,d,E,k,f", [(900, 1088, 8, 2, 640), (1500, 320, 5, 2, 704), (2600, 576, 2, 1, 320)])
def test_group_size_changes_no_bit(T, d, E, k, f, flags, monkeypatch):
    """Experts with no rows, a few and up to 21 row tiles; groups that do not divide them, ragged last tiles in both directions."""
    g = torch.Generator(device="cuda")
    g.manual_seed(T)
    n = lambda *s: torch.empty(*s, device="cuda").normal_(0, 0.05, generator=g).bfloat16()
    x, W, dy = n(T, d), (n(d, E), n(E, d, f), n(E, d, f), n(E, f, d)), n(T, d)
    b_r = torch.linspace(-2.0, 2.0, E, device="cuda")

    def step():
        layer = MoELayer(d, E, f, k, flags)
        out = layer.forward(x, *W, b_r=b_r)
        grads = layer.backward(dy, 0.01)
        layer.poll()
        return [out["y"]] + [grads[m] for m in ("dx", "dW_gate", "dW_up", "dW_down")]

    plain = step()
    for group in ("2", "3", "7", "40"):
        monkeypatch.setenv("MOE_ROW_GROUP", group)
        assert all(torch.equal(a, b) for a, b in zip(step(), plain)), group


@pytest.mark.parametrize("T,d,E,k,f", [(1200, 2048, 4, 2, 1664), (4400, 2112, 2, 1, 2176)])
def test_pairs_that_keep_step(T, d, E, k, f, monkeypatch):
    """Tiles of 32 K blocks of wide experts, the second shape with weight gradients of 34 K blocks over 25 MB: the pairs wait for one
    another.  The same bits without (a group of one row tile), and when the counters are those of an earlier backward pass.  A pair
    counts every tile once."""
    g = torch.Generator(device="cuda")
    g.manual_seed(T)
    n = lambda *s: torch.empty(*s, device="cuda").normal_(0, 0.05, generator=g).bfloat16()
    x, W, dy = n(T, d), (n(d, E), n(E, d, f), n(E, d, f), n(E, f, d)), n(T, d)
    steps = []
    for group in (None, "1"):
        if group:
            monkeypatch.setenv("MOE_ROW_GROUP", group)
        layer = MoELayer(d, E, f, k, 1)
        for _ in range(2):
            out = layer.forward(x, *W)
            for _ in range(2):
                grads = layer.backward(dy, 0.01)
                steps.append([out["y"]] + [grads[m] for m in ("dx", "dW_gate", "dW_up", "dW_down")])
        layer.poll()
        counted = layer.buffer("pace", torch.int32).view(6, -1).sum(1).tolist()
        if group:
            assert not any(counted)
        else:
            pairs = int(((out["counts"] + 255) // 256).sum())
            wide = {0: pairs * -(-f // 128)}  # gate/up: more than 12 column tiles
            if T == 4400:
                wide[5] = 2 * E * -(-d // 256) * -(-f // 128)  # wgrad gate/up, of two backward passes
            assert {kind: c for kind, c in enumerate(counted) if c} == wide
    assert all(torch.equal(a, b) for s in steps[1:] for a, b in zip(s, steps[0]))


def test_more_rounds_than_pace_counters(monkeypatch):
    """134 column tiles x 36 pairs of row tiles on 74 pairs of CTAs: 66 rounds or more, so that counters are used again."""
    T, d, E, k, f = 9000, 2048, 2, 1, 17152
    g = torch.Generator(device="cuda")
    g.manual_seed(7)
    n = lambda *s: torch.empty(*s, device="cuda").normal_(0, 0.05, generator=g).bfloat16()
    x, W = n(T, d), (n(d, E), n(E, d, f), n(E, d, f), n(E, f, d))
    acts = []
    for group in (None, "1"):
        if group:
            monkeypatch.setenv("MOE_ROW_GROUP", group)
        layer = MoELayer(d, E, f, k, 1)
        out = layer.forward(x, *W)
        layer.poll()
        acts.append((layer.buffer("act", torch.int16).clone(), out["y"]))
        rounds = layer.buffer("pace", torch.int32).view(6, -1)[0].tolist()
        if group:
            assert not any(rounds)
        else:
            workers = torch.cuda.get_device_properties(0).multi_processor_count // 2
            tiles = int(((out["counts"] + 255) // 256).sum()) * (f // 128)
            assert sum(rounds) == tiles > 64 * workers
            assert rounds[0] == 2 * workers and min(rounds) >= workers, rounds
    assert torch.equal(acts[0][0], acts[1][0]) and torch.equal(acts[0][1], acts[1][1])


def test_weight_gradient_of_a_wide_expert():
    """2800 rows, 17 column tiles: by its own rule gate/up walks the three row tiles (the last one short) inside a column tile."""
    inp = synth.make_inputs(synth.MoEShape(22400, 576, 8, 1, 2176), 31, x_std=1.0)
    ofw, obw = oracle_run(inp, 1, 0.05, dtype=np.float32)
    check_all(Run(inp, 1), ofw, obw, 0.05, stages=False)
