"""fp32 moments that travel through the projection's ring in pieces of 32 x 64: at the edges of the pieces, their boxes of 32
columns and the 16-byte units of a row, against the stand-alone Adam kernel on the same products."""
import pytest
import torch

from paper_2403_03507_b200 import binding as gb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("long", [264, 287, 289, 319, 321, 513, 1000])
# multiples of 8 (others do not run on the tensor path) on either side of the pieces; from 256 on two CTAs share a tile
@pytest.mark.parametrize("rank", [8, 24, 40, 72, 136, 248, 256, 264])
@pytest.mark.parametrize("left", [True, False])
def test_moments_and_weights_equal_those_of_the_stand_alone_kernel(long, rank, left):
    short = 264
    m, n = (short, max(long, short)) if left else (max(long, short), short)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(long * 1000 + rank)
    ld = (n + 15) // 16 * 16
    draw = lambda: torch.randn(m, ld, generator=gen, device="cuda").to(torch.bfloat16)[:, :n]
    W0, Gs = [draw() for _ in range(4)], [[draw() for _ in range(4)] for _ in range(2)]
    out, launches = [], []
    for place in (gb.ADAM_IN_PROJECTION, gb.ADAM_OWN_KERNEL):
        layers = [gb.Layer(gb.make_config(m, n, rank, w_dtype="bf16", g_dtype="bf16", auto_refresh=False, adam_place=place)) for _ in range(4)]
        gen.manual_seed(5)
        for l in layers:
            l.set_projector(torch.linalg.qr(torch.randn(short, rank, generator=gen, device="cuda"))[0].cpu())
        Ws = [torch.empty(m, ld, device="cuda", dtype=torch.bfloat16)[:, :n].copy_(w) for w in W0]
        assert all(l.uses_tensor_path for l in layers)
        batch = gb.Batch(layers, Ws, Gs[0])
        before = gb.galore_launch_count()
        for G in Gs:
            batch.rebind(Ws, G)
            batch.galore_step_batch(1e-2)
        launches.append(gb.galore_launch_count() - before)
        out.append((Ws, [l.get_moments() for l in layers], [l.device_status() for l in layers]))
    assert launches == [4, 6]           # two steps: projection with Adam, update; projection, Adam, update
    (Wa, Ma, Sa), (Wb, Mb, Sb) = out
    # four layers are not cut into K slices: both ways see the same fp32 sums and do the same arithmetic on them
    assert Sa == Sb == [0] * 4
    for a, b in zip(Wa, Wb):
        assert torch.equal(a, b)
    for (ma, va), (mb, vb) in zip(Ma, Mb):
        assert torch.equal(ma, mb) and torch.equal(va, vb)
