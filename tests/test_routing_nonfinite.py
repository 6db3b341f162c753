"""Routing of tokens whose logits are NaN or -inf: k distinct experts in [0, E) whatever the logits, a NaN counts as -inf,
the lowest index wins among equals."""
import numpy as np
import pytest
import torch

INF, NAN = np.float32(np.inf), np.float32(np.nan)


def expected_picks(logits, k):
    v = np.fmax(logits.astype(np.float32), -INF)  # fmax drops NaN
    return np.argsort(-v, axis=1, kind="stable")[:, :k].astype(np.int32)


def tournament(row, k):
    """The selection of the routing epilogue for E <= 128, step by step in float32: groups of four, supers of four groups,
    taken columns and columns beyond E at -inf, the lowest untaken index once nothing larger is left."""
    E = row.size
    v = np.full(128, -INF, np.float32)
    v[:E] = row
    v = v.reshape(8, 4, 4)
    picks = []
    for _ in range(k):
        groups = np.fmax.reduce(v, axis=2)
        supers = np.fmax.reduce(groups, axis=1)
        best = np.fmax.reduce(supers)
        if best > -INF:
            s = int(np.argmax(supers == best))
            g = int(np.argmax(groups[s] == best))
            c = int(np.argmax(v[s, g] == best))
            v[s, g, c] = -INF
            picks.append(16 * s + 4 * g + c)
        else:
            picks.append(min(set(range(k)) - set(picks)))
    return picks


def awkward_rows(rng, E, n):
    """Rows of logits with every mix of numbers, ties, -inf and NaN, all-NaN and all -inf rows among them."""
    rows = rng.choice(np.array([-2, -1, 0, 1, 2], np.float32), (n, E))
    share = rng.random((n, 1))
    rows = np.where(rng.random((n, E)) < share, rng.choice(np.array([NAN, -INF], np.float32), (n, E)), rows)
    rows[0], rows[1] = NAN, -INF
    rows[2, 1:] = NAN
    rows[3, : E - 1] = -INF
    return rows.astype(np.float32)


@pytest.mark.parametrize("E,k", [(8, 8), (40, 6), (128, 8), (128, 16)])
def test_tournament_rule_on_nan_and_inf_rows(E, k):
    rows = awkward_rows(np.random.default_rng(E + k), E, 300)
    got = np.array([tournament(r, k) for r in rows], np.int32)
    assert np.array_equal(got, expected_picks(rows, k))


def check_picks(out, k, E):
    idx, logits = out["idx"].cpu().numpy(), out["logits"].cpu().numpy()
    assert idx.min() >= 0 and idx.max() < E
    assert np.array_equal(idx, expected_picks(logits, k))  # distinct by construction
    flat = idx.reshape(-1)
    assert np.array_equal(out["counts"].cpu().numpy(), np.bincount(flat, minlength=E))
    assert np.array_equal(out["perm"].cpu().numpy(), np.argsort(flat, kind="stable"))


@pytest.mark.gpu
@pytest.mark.parametrize("given", [False, True])
@pytest.mark.parametrize("T,d,E,k", [
    (300, 128, 128, 8),   # tournament, all 128 columns in use
    (150, 64, 40, 16),    # tournament, columns beyond E
    (140, 64, 256, 6),    # passes over tensor memory
    (130, 64, 64, 32),    # the same because of k
    (70, 64, 5, 5),       # one warp per token (E not a multiple of 8), every expert taken
])
def test_every_token_gets_distinct_experts(T, d, E, k, given):
    from paper_2608_00916_b200.binding import MoELayer
    g = torch.Generator(device="cuda")
    g.manual_seed(E)
    n = lambda *s: torch.empty(*s, device="cuda").normal_(generator=g)
    x, W_r = n(T, d).bfloat16(), (0.1 * n(d, E)).bfloat16()
    Wg, Wu, Wd = ((0.1 * n(E, *s)).bfloat16() for s in ((d, 64), (d, 64), (64, d)))
    layer = MoELayer(d, E, 64, k)
    if given:
        li = torch.from_numpy(awkward_rows(np.random.default_rng(E), E, T)).cuda()
        check_picks(layer.forward(x, W_r, Wg, Wu, Wd, logits_in=li, want_logits=True), k, E)
        layer.poll()
        return
    clean = layer.forward(x, W_r, Wg, Wu, Wd, want_logits=True)
    check_picks(clean, k, E)
    bad = x.clone()
    bad[3, 5] = float("nan")   # all logits of one token
    bad[T - 1] = float("nan")
    out = layer.forward(bad, W_r, Wg, Wu, Wd, want_logits=True)
    layer.poll()
    check_picks(out, k, E)
    ok = torch.ones(T, dtype=torch.bool, device="cuda")
    ok[3] = ok[T - 1] = False
    assert torch.equal(out["y"][ok], clean["y"][ok])  # the other tokens do not notice
    assert torch.equal(out["idx"][ok], clean["idx"][ok]) and torch.equal(out["gates"][ok], clean["gates"][ok])
    assert out["y"][~ok].isnan().all() and out["aux"].isnan().all()
    # fewer finite columns than picks, and a router column of NaN
    b = torch.full((E,), float("-inf"), device="cuda")
    b[1::3] = 0.0
    W_nan = W_r.clone()
    W_nan[:, 1] = float("nan")
    for inference in (False, True):
        check_picks(layer.forward(x, W_nan, Wg, Wu, Wd, b_r=b, want_logits=True, inference=inference), k, E)
    layer.poll()
