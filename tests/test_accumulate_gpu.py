"""fp32 accumulation of the weight gradients: exactly old + gradient, rounded once, over the whole range of fp32."""
import pytest
import torch

from paper_2608_00916_b200.binding import MoELayer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,flags", [
    (300, 1),   # CTA pairs: reductions
    (300, 2),   # one-CTA tiles: loads, additions, stores
    (1700, 0),  # 425 rows per expert: one-CTA tiles by the default rule
    (2900, 0),  # 725: pairs
])
@pytest.mark.parametrize("exponent", [0, -85, -95, -103, -112])
def test_accumulation_rounds_once_over_the_whole_range(T, flags, exponent):
    """dy is scaled so that the gradients lie around 2^exponent or far below it; the buffers start from subnormals, zeros of
    both signs, values that nearly cancel the gradient and ordinary ones.  Exactly what an fp32 addition gives."""
    d, E, k, f = 192, 8, 2, 320
    g = torch.Generator(device="cuda")
    g.manual_seed(7)
    n = lambda *s: torch.empty(*s, device="cuda").normal_(generator=g)
    x, W_r = n(T, d).bfloat16(), (0.1 * n(d, E)).bfloat16()
    Wg, Wu, Wd = ((0.1 * n(E, *s)).bfloat16() for s in ((d, f), (d, f), (f, d)))
    dy = torch.ldexp(n(T, d), torch.tensor(exponent - 5, device="cuda")).bfloat16()
    layer = MoELayer(d, E, f, k, flags)
    names = {"dW_gate": Wg, "dW_up": Wu, "dW_down": Wd}

    def accumulate(start):
        acc = {"dW_r": torch.zeros(d, E, device="cuda"), **{m: start[m].cuda() for m in names}}
        layer.forward(x, W_r, Wg, Wu, Wd)
        layer.backward_accumulate(dy, 0.0, acc)
        layer.poll()
        return {m: acc[m].cpu() for m in names}

    grad = accumulate({m: torch.zeros(w.shape) for m, w in names.items()})
    h = torch.Generator().manual_seed(8)
    start = {}
    for m, v in grad.items():
        kind = torch.randint(0, 6, v.shape, generator=h)
        r = torch.randn(v.shape, generator=h)
        subnormal = torch.randint(-(1 << 23), 1 << 23, v.shape, generator=h).double().mul(2.0 ** -149).float()
        near = -v * (1 + torch.randint(-4, 5, v.shape, generator=h) * 2.0 ** -23)
        options = (subnormal, torch.zeros_like(v), -torch.zeros_like(v), near, r * 2.0 ** -125, r * 2.0 ** exponent)
        start[m] = torch.stack(options).gather(0, kind[None])[0]
    got = accumulate(start)
    for m, v in grad.items():
        want = start[m] + v  # on the host, where fp32 additions keep subnormals
        assert torch.equal(got[m], want), m
        if exponent == -112:
            assert ((want != 0) & (want.abs() < 2.0 ** -126)).any()
