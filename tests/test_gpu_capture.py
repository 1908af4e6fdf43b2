"""Steps captured into CUDA graphs, between eager steps on other streams."""
import pytest
import torch

from paper_2403_03507_b200 import binding as gb

pytestmark = pytest.mark.gpu

DT = {"f32": torch.float32, "bf16": torch.bfloat16}


def _call(kind, dtype, m=256, n=640, r=32):
    """A function that makes one call on the current stream, and the weights it updates."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(3)
    rand = lambda *s: torch.randn(*s, generator=gen, device="cuda")
    P = torch.linalg.qr(rand(m, r))[0].contiguous()
    Ws, Gs = [rand(m, n).to(DT[dtype]) for _ in range(2)], [rand(m, n).to(DT[dtype]) for _ in range(2)]
    if kind == "static":
        M, V = torch.zeros(r, n, device="cuda"), torch.zeros(r, n, device="cuda")
        return (lambda: gb.galore_step_static(P, M, V, Ws[0], Gs[0], 1e-2, completed_steps=3, want_flags=False)), Ws[0]
    layers = [gb.Layer(gb.make_config(m, n, r, w_dtype=dtype, g_dtype=dtype, auto_refresh=False)) for _ in range(2)]
    for l in layers:
        l.set_projector(P)
    if kind == "step":
        call = lambda: layers[0].galore_step(Ws[0], Gs[0], 1e-2)
    else:
        batch = gb.Batch(layers, Ws, Gs)
        call = lambda: batch.galore_step_batch(1e-2)

    def at_step_three():                # a captured call keeps the bias correction it was captured with
        for l in layers:
            l.step_count = 3
        call()
    return at_step_three, Ws[0]


def _on(stream, call):
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        call()
    stream.synchronize()


@pytest.mark.parametrize("kind,dtype", [("static", "f32"), ("step", "f32"), ("step", "bf16"), ("batch", "f32"), ("batch", "bf16")])
def test_captured_step_between_eager_ones(kind, dtype):
    first, second, third = (torch.cuda.Stream() for _ in range(3))
    call, W = _call(kind, dtype)
    for _ in range(4):
        _on(first, call)
    want = W.clone()
    call, W = _call(kind, dtype)
    _on(first, call)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=second):
        call()
    graph.replay()
    torch.cuda.synchronize()
    _on(third, call)
    _on(first, call)
    assert torch.equal(W, want)         # one eager call, one replay, two eager calls
    del graph
