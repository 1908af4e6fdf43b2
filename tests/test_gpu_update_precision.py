"""The weight update of operands held in fp32 (three bf16 planes each) against the product in 64 bits: no further from it than
a chain of fp32 fused multiply-adds, and no loss of one sign."""
import pytest
import torch

from paper_2403_03507_b200 import binding as gb

pytestmark = pytest.mark.gpu


# both sides; one to thirty-two blocks of 64, odd numbers of them, a ragged last one; tiles of a CTA pair, tiles of one CTA
# (few of them, or rows of W off the 16-byte boundaries)
@pytest.mark.parametrize("m,n,r,pad", [(1024, 2048, 512, 0), (2048, 2048, 1024, 0), (2304, 2560, 2048, 0), (2560, 2304, 2048, 0),
                                       (512, 1376, 65, 0), (512, 1376, 192, 0), (4096, 5461, 512, 3), (4096, 4104, 1000, 0)])
@pytest.mark.parametrize("count", [1, 2])
def test_update_keeps_fp32_precision_at_every_rank(m, n, r, pad, count):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(m + r)
    rand = lambda *s: torch.randn(*s, generator=gen, device="cuda")
    layers, Ws, Gs = [], [], []
    for _ in range(count):
        # Adafactor: its first moment is N itself, so the operands of the product are known exactly
        layers.append(gb.Layer(gb.make_config(m, n, r, w_dtype="f32", g_dtype="f32", state_fmt="adafactor", auto_refresh=False)))
        layers[-1].set_projector(torch.linalg.qr(rand(layers[-1].proj_rows, r))[0])
        Ws.append(torch.zeros(m, n + pad, device="cuda")[:, :n])
        Gs.append(rand(m, n))
    if count == 1:
        layers[0].galore_step(Ws[0], Gs[0], 1.0)
    else:
        gb.Batch(layers, Ws, Gs).galore_step_batch(1.0)
    for layer, W in zip(layers, Ws):
        assert layer.device_status() == 0
        P, N = layer.get_projector().double(), layer.get_adafactor_state()[0].double()
        want = -0.25 * (P @ N if layer.side == gb.SIDE_LEFT else N @ P.T)       # W was zero, lr alpha is a power of two
        W = W.double()
        # A chain of r fused multiply-adds: r roundings of at most 2^-24 of a partial sum, which after k of them is about
        # sqrt(k / r) of the result; the root of the sum of (2^-24 / sqrt 3)^2 k / r is 0.41 2^-24 sqrt(r) at most, and 0.30 of
        # that unit is what an FMA kernel shows.
        assert float((W - want).norm() / want.norm()) <= max(0.3 * r ** 0.5, 2.2) * 2 ** -24
        # The tensor core cuts off up to a unit of 2^-23 of its accumulator per 16 products, eight times before it is
        # drained.  (An accumulator of the whole rank shows 4.1e-7 at 512 and 1.8e-6 at 2048.)
        assert abs(float((W * want).sum() / (want * want).sum()) - 1) <= 2e-7


# bf16 W in groups: tiles of pairs or of single CTAs by the waves of each, but by the old line up to eight blocks of products
# (rank 64 and below); ragged sizes of both sides in one call
@pytest.mark.parametrize("r", [64, 65, 200])
@pytest.mark.parametrize("count", [3, 16, 28])
def test_grouped_updates_of_bf16_weights_are_rounded_products(r, count):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(r + count)
    rand = lambda *s: torch.randn(*s, generator=gen, device="cuda")
    layers, Ws, Gs = [], [], []
    for i in range(count):
        m, n = [(448, 1200), (448, 448), (1194, 450)][i % 3]
        layers.append(gb.Layer(gb.make_config(m, n, r, w_dtype="bf16", g_dtype="f32", state_fmt="adafactor", auto_refresh=False)))
        layers[-1].set_projector(torch.linalg.qr(rand(layers[-1].proj_rows, r))[0])
        Ws.append(torch.zeros(m, (n + 7) // 8 * 8, device="cuda", dtype=torch.bfloat16)[:, :n])
        Gs.append(rand(m, n))
    gb.Batch(layers, Ws, Gs).galore_step_batch(1.0)
    for layer, W in zip(layers, Ws):
        assert layer.device_status() == 0
        P, N = layer.get_projector().double(), layer.get_adafactor_state()[0].double()
        want = -0.25 * (P @ N if layer.side == gb.SIDE_LEFT else N @ P.T)
        # half a unit of bf16 in the last place, and fp32's error of the product (4e-6 of the largest entry is far above it)
        assert bool(((W.double() - want).abs() <= 2.0 ** -8 * want.abs() + 4e-6 * want.abs().max()).all())


# Tiles with one piece of W (the last columns of a row of tiles, or matrices narrower than a piece) between tiles with several: either
# set of epilogue warps takes pieces that its tiles leave out now and then.  Rows of W off the 16-byte boundaries and on them, pair
# tiles and single ones; the same inputs over again, as a wait that ends too early shows only now and then.
@pytest.mark.parametrize("w,pad", [("bf16", 0), ("bf16", 8), ("f32", 8)])
@pytest.mark.parametrize("shapes,count,r", [([(665, 665)] * 4 + [(665, 1408)] * 2 + [(1408, 665)], 28, 39), ([(2048, 40)] * 3 + [(40, 2049)], 24, 33),
                                            ([(1024, 1281), (1153, 897)], 12, 200), ([(512, 1409), (300, 130)], 2, 72)])
def test_tiles_of_few_pieces_among_tiles_of_many(shapes, count, r, w, pad):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(r)
    rand = lambda *s: torch.randn(*s, generator=gen, device="cuda")
    dt = torch.float32 if w == "f32" else torch.bfloat16
    layers, Ws, Gs = [], [], []
    for i in range(count):
        m, n = shapes[i % len(shapes)]
        layers.append(gb.Layer(gb.make_config(m, n, r, w_dtype=w, g_dtype="f32", state_fmt="adafactor", auto_refresh=False)))
        layers[-1].set_projector(torch.linalg.qr(rand(layers[-1].proj_rows, r))[0])
        Ws.append(torch.zeros(m, n if pad == 0 else (n + 7) // 8 * 8, device="cuda", dtype=dt)[:, :n])
        Gs.append(rand(m, n))
    batch = gb.Batch(layers, Ws, Gs)
    for _ in range(6):
        old = [W.double() for W in Ws]
        batch.galore_step_batch(1.0)
        for layer, W, W0 in zip(layers, Ws, old):
            assert layer.device_status() == 0
            P, N = layer.get_projector().double(), layer.get_adafactor_state()[0].double()
            want = W0 - 0.25 * (P @ N if layer.side == gb.SIDE_LEFT else N @ P.T)
            # half a unit of W's type in the last place, and fp32's error of the product
            half = 2.0 ** -24 if w == "f32" else 2.0 ** -8
            assert bool(((W.double() - want).abs() <= half * want.abs() + 4e-6 * (want - W0).abs().max()).all())
