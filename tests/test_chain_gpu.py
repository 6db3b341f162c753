"""Kernels of a call that run beside one another: the same bits as with CUDA events between them, from steps that follow one another
without a pause on one workspace and on alternating inputs (a read that came too early would see the other batch's rows)."""
import pytest
import torch

from paper_2608_00916_b200.binding import FLAG_ROUTER_FP32, STAGE_NAMES, MoELayer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,d,E,k,f,flags", [
    (256, 256, 8, 2, 512, 0),              # dW_r from one slice
    (700, 1024, 16, 2, 512, 0),            # tokens as N; partial sums of dW_r
    (700, 320, 12, 3, 192, 0),             # E no multiple of 8: the kernels without tensor cores
    (1500, 512, 8, 2, 640, 1),             # CTA pairs
    (1500, 512, 8, 2, 640, 16),            # pairs, then leftover blocks
    (3000, 2048, 8, 2, 768, FLAG_ROUTER_FP32),
    (40, 64, 64, 2, 64, 0),                # most experts without rows
    (2303, 512, 8, 2, 640, 0),             # the last size at which the large GEMMs overlap
    (2304, 512, 8, 2, 640, 0),             # the first at which only the small kernels run beside them
])
@pytest.mark.parametrize("mode", ["train", "accumulate", "grouped", "lora"])
def test_same_bits_with_and_without_events_between_the_kernels(T, d, E, k, f, flags, mode):
    if mode == "lora" and flags & FLAG_ROUTER_FP32:
        pytest.skip("adapters take a bf16 router weight")
    g = torch.Generator(device="cuda")
    g.manual_seed(T)
    n = lambda *s: torch.empty(*s, device="cuda").normal_(0, 0.05, generator=g).bfloat16()
    batches = [(20 * n(T, d), 20 * n(T, d)) for _ in range(2)]
    W_r = n(d, E).float() if flags & FLAG_ROUTER_FP32 else n(d, E)
    W = (W_r, n(E, d, f), n(E, d, f), n(E, f, d))
    shapes = {"A1": (E, d, 16), "B1_gate": (E, 16, f), "B1_up": (E, 16, f), "A2": (E, f, 16), "B2": (E, 16, d)}
    adapters = {m: n(*s) for m, s in shapes.items()}
    layer = MoELayer(d, E, f, k, flags)

    def step(i):
        x, dy = batches[i % 2]
        if mode == "lora":
            out = layer.lora_forward(x, *W, adapters, 2.0)
            grads = layer.lora_backward(dy, 0.01)
        else:
            out = layer.forward(x, *W)
            if mode == "train":
                grads = layer.backward(dy, 0.01, want_db=True)
            else:
                acc = {m: torch.ones(w.shape, device="cuda") for m, w in zip(("dW_r", "dW_gate", "dW_up", "dW_down"), W)}
                acc["db_r"] = torch.ones(E, device="cuda")
                events = [torch.cuda.Event() for _ in range(6)] if mode == "grouped" else None  # three ranges of experts
                grads = {"dx": layer.backward_accumulate(dy, 0.01, acc, group_events=events), **acc}
        return {"y": out["y"], **grads}

    layer.set_profiling(True)
    apart = [step(i) for i in range(2)]
    layer.poll()
    layer.set_profiling(False)
    together = [step(i) for i in range(8)]
    layer.poll()
    for i, got in enumerate(together):
        for name, v in apart[i % 2].items():
            if v is not None:
                assert torch.equal(got[name], v), (i, name)


@pytest.mark.parametrize("E", [16, 12])  # the router's gradient on tensor cores, and without
def test_every_stage_of_a_step_is_timed(E):
    T, d, k, f = 700, 512, 2, 256
    g = torch.Generator(device="cuda")
    g.manual_seed(E)
    n = lambda *s: torch.empty(*s, device="cuda").normal_(0, 0.05, generator=g).bfloat16()
    x, W, dy = n(T, d), (n(d, E), n(E, d, f), n(E, d, f), n(E, f, d)), n(T, d)
    layer = MoELayer(d, E, f, k)
    layer.set_profiling(True)
    for _ in range(2):
        layer.forward(x, *W)
        layer.backward(dy, 0.01)
    stages, steps = layer.stage_times()
    assert steps == 2 and len(STAGE_NAMES) == 14
    assert all(ms > 0 for ms in stages[:14]) and not any(stages[14:]), stages
