"""The step with fp32 operands, or operands whose rows TMA cannot address, against fp64 products."""
import pytest
import torch

from paper_2403_03507_b200 import binding as gb

pytestmark = pytest.mark.gpu

DT = {"f32": torch.float32, "bf16": torch.bfloat16}


def _matrix(x, dtype, pad):
    """x in rows of `pad` more elements, the padding NaN."""
    buf = torch.full((x.shape[0], x.shape[1] + pad), float("nan"), device="cuda", dtype=DT[dtype])
    buf[:, :x.shape[1]] = x
    return buf[:, :x.shape[1]]


# edges of the 128 x 128 tiles and of the 64-wide K blocks, single elements, both sides, several K slices
@pytest.mark.parametrize("m,n,r", [(1, 1, 1), (64, 128, 64), (65, 129, 63), (127, 255, 127), (129, 257, 128), (257, 128, 17),
                                   (700, 3, 2), (1000, 2049, 33)])
@pytest.mark.parametrize("g,w,pad", [("f32", "f32", 0), ("f32", "bf16", 1), ("bf16", "bf16", 0), ("bf16", "f32", 3)])
def test_products_of_split_operands_are_fp32_products(m, n, r, g, w, pad):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(m * 7919 + n)
    rand = lambda *s: torch.randn(*s, generator=gen, device="cuda")
    layer = gb.Layer(gb.make_config(m, n, r, w_dtype=w, g_dtype=g, auto_refresh=False, path=gb.PATH_FP32))
    layer.set_projector(torch.linalg.qr(rand(layer.proj_rows, r))[0])
    P = layer.get_projector().double()
    G, W = _matrix(rand(m, n), g, pad), _matrix(0.02 * rand(m, n), w, pad)
    W0 = W.double()
    layer.galore_step(W, G, 1e-2)
    assert layer.device_status() == 0
    left = layer.side == gb.SIDE_LEFT
    R = P.T @ G.double() if left else G.double() @ P
    M, V = (t.double() for t in layer.get_moments())
    # M = 0.1 R and V = 0.001 R^2 from zero moments, each rounded a few times to fp32; R itself is an fp32 sum of K terms
    # whose error relative to the root mean square of R stays below sqrt(K) 2^-24 (1e-6 for K = 257, 3e-6 for 2049)
    K = m if left else n
    tol = 2 ** -24 * (8 + K ** 0.5)
    assert float((M / 0.1 - R).norm() / R.norm()) <= tol
    # the update from the moments the layer stores: fp32 products again, Eq. 15 through approximate roots (2 ulp each),
    # and the rounding of W: half the spacing 2^(e-7) of bf16 (2^(e-23) of fp32) at 2^e <= |W|, at most 2^-8 (2^-24) of |W|
    N = (M / 0.1) / ((V / 0.001).sqrt() + 1e-8)
    dW = -1e-2 * 0.25 * (P @ N if left else N @ P.T)
    slack = (2 ** -8 if w == "bf16" else 2 ** -24) * float((W0.abs() + dW.abs()).max())
    # N is +-1 at the first step except where R is so small that fp32 flushes its square: allow 1e-6 of the update's scale
    assert float((W.double() - W0 - dW).abs().max()) <= slack + 1e-5 * float(dW.abs().max()) + 1e-12
    if pad:
        assert torch.isnan(W._base[:, n:]).all()


# groups around the line between the 128 x 128 tiles and the 256 x 256 tiles of CTA pairs (which 1000 x 1999 and 5460 x 2050 take): ragged tiles
# on both sides, blocks of K cut off, several K slices (one matrix), rows padded to 16 bytes; the largest rank takes two tiles along the rank
@pytest.mark.parametrize("m,n,r,count,pad", [(769, 2052, 256, 12, 0), (2052, 770, 260, 12, 2), (96, 8200, 64, 20, 0), (1000, 1999, 388, 8, 1), (2048, 5460, 512, 1, 0),
                                             (5460, 2050, 512, 1, 2)])
def test_products_of_large_groups_are_fp32_products(m, n, r, count, pad):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(m * 7919 + n)
    rand = lambda *s: torch.randn(*s, generator=gen, device="cuda")
    layers, Ws, Gs = [], [], []
    for _ in range(count):
        layers.append(gb.Layer(gb.make_config(m, n, r, w_dtype="bf16", g_dtype="f32", auto_refresh=False)))
        layers[-1].set_projector(torch.linalg.qr(rand(layers[-1].proj_rows, r))[0])
        Ws.append(_matrix(0.02 * rand(m, n), "bf16", pad))
        Gs.append(_matrix(rand(m, n), "f32", pad))
    if count == 1:
        layers[0].galore_step(Ws[0], Gs[0], 1e-2)
    else:
        gb.Batch(layers, Ws, Gs).galore_step_batch(1e-2)
    for layer, G in zip(layers, Gs):
        assert layer.device_status() == 0
        P = layer.get_projector().double()
        R = P.T @ G.double() if layer.side == gb.SIDE_LEFT else G.double() @ P
        M = layer.get_moments()[0].double()
        # as above: an fp32 sum of K terms; the accumulators of 32 of K lose at most a unit of 2^-23 of one sign per 16 products
        assert float((M / 0.1 - R).norm() / R.norm()) <= 2 ** -24 * (8 + (m if layer.side == gb.SIDE_LEFT else n) ** 0.5)
        assert abs(float((M / 0.1 * R).sum() / (R * R).sum()) - 1) <= 2e-7


# bf16 rows that TMA cannot address, in products long enough for a copy of G on 16-byte rows; tiles of one CTA and of pairs in
# the update (its rows go through shared memory in 16-byte units).  off: columns of W and G in front of the matrix, in the same rows
@pytest.mark.parametrize("m,n,r,off,pad", [(2048, 2051, 512, 0, 0), (2051, 1031, 264, 0, 0), (1000, 2049, 320, 1, 2), (1500, 3001, 128, 3, 0), (4097, 1003, 64, 5, 1),
                                           (1030, 5461, 512, 7, 4), (2048, 2048, 512, 0, 3),
                                           # rows on 4-byte boundaries: from registers; tiles cut off below 32 columns, one and several waves, pairs
                                           (518, 518, 184, 0, 0), (130, 1346, 40, 2, 4), (2051, 34, 16, 4, 0), (2500, 2502, 128, 0, 0), (2500, 2498, 640, 2, 2)])
@pytest.mark.parametrize("state", ["f32", "q8"])
def test_packed_bf16_rows_keep_fp32_precision(m, n, r, off, pad, state):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(m * 31 + n)
    rand = lambda *s: torch.randn(*s, generator=gen, device="cuda")
    layer = gb.Layer(gb.make_config(m, n, r, w_dtype="bf16", g_dtype="bf16", state_fmt=state, auto_refresh=False))
    layer.set_projector(torch.linalg.qr(rand(layer.proj_rows, r))[0])
    P = layer.get_projector().double()
    bufs = []
    for x in (rand(m, n), 0.02 * rand(m, n)):
        buf = torch.full((m, off + n + pad), float("nan"), device="cuda", dtype=torch.bfloat16)
        buf[:, off:off + n] = x
        bufs.append(buf)
    G, W = (b[:, off:off + n] for b in bufs)
    G0, W0 = G.clone(), W.double()
    layer.galore_step(W, G, 1e-2)
    assert layer.device_status() == 0
    left = layer.side == gb.SIDE_LEFT
    R = P.T @ G.double() if left else G.double() @ P
    if state == "f32":
        M, V = (t.double() for t in layer.get_moments())
        # an fp32 sum of K terms, as above; the accumulator of a k-block loses at most a unit of 2^-23 of one sign per 16 products
        assert float((M / 0.1 - R).norm() / R.norm()) <= 2 ** -24 * (8 + (m if left else n) ** 0.5)
        assert abs(float((M / 0.1 * R).sum() / (R * R).sum()) - 1) <= 2e-7
    # the first step: N = +-1 (with 8-bit moments it is worked out before they are rounded), but for an R that fp32 flushes
    N = R / (R.abs() + 1e-8)
    dW = -1e-2 * 0.25 * (P @ N if left else N @ P.T)
    slack = 2 ** -8 * float((W0.abs() + dW.abs()).max())
    # an R within the fp32 rounding of zero may come out on the other side: its N is off by 2
    flips = 2 * 1e-2 * 0.25 * float(P.abs().max()) * float((R.abs() <= 1e-6 * R.square().mean().sqrt()).any())
    assert float((W.double() - W0 - dW).abs().max()) <= slack + 1e-5 * float(dW.abs().max()) + flips
    assert torch.equal(G, G0)
    for buf in bufs:
        assert torch.isnan(buf[:, :off]).all() and torch.isnan(buf[:, off + n:]).all()


def _off_by_one(x):
    """x in rows one element off the 16-byte boundaries: CTA pairs do not take it."""
    buf = torch.zeros(x.shape[0], (x.shape[1] + 4) // 4 * 4, device="cuda", dtype=x.dtype)
    out = buf[:, 1:1 + x.shape[1]]
    out.copy_(x)
    return out


# Groups that take the tiles of CTA pairs: both sides (the operands' majors change from one unit of a pair to the next), sums of 3 to 10
# blocks of 64 (the corrections are added after every eight), decoder layers.  The same gradients off the 16-byte boundaries take the
# tiles of one CTA, whose leading products and corrections are both added after every block.
@pytest.mark.parametrize("shapes,count,r", [([(188, 2304)], 8, 188), ([(448, 2304)], 8, 256), ([(2304, 512)], 8, 256), ([(513, 2304)], 8, 256),
                                            ([(2304, 577)], 8, 256), ([(449, 2300), (2300, 449)], 16, 256), ([(600, 2300), (2300, 520)], 16, 252),
                                            ([(768, 768)] * 4 + [(768, 2048)] * 2 + [(2048, 768)], 14, 256), ([(768, 768)] * 4 + [(768, 2048)] * 2 + [(2048, 768)], 28, 256),
                                            ([(1024, 2816)], 20, 256), ([(3000, 3000)], 8, 512)])
def test_pair_tiles_are_no_further_from_64_bits_than_single_ones(shapes, count, r):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(r + count)
    rand = lambda *s: torch.randn(*s, generator=gen, device="cuda")
    sizes = [shapes[i % len(shapes)] for i in range(count)]
    P = [torch.linalg.qr(rand(min(s), r))[0] for s in sizes]
    G = [rand(m, n) for m, n in sizes]
    err, bias, moments = [], [], []
    for place in (lambda g: _matrix(g, "f32", -g.shape[1] % 4), _off_by_one):
        layers = [gb.Layer(gb.make_config(m, n, r, w_dtype="bf16", g_dtype="f32", auto_refresh=False)) for m, n in sizes]
        for layer, p in zip(layers, P):
            layer.set_projector(p)
        gb.Batch(layers, [torch.zeros(m, (n + 7) // 8 * 8, device="cuda", dtype=torch.bfloat16)[:, :n] for m, n in sizes], [place(g) for g in G]).galore_step_batch(1e-2)
        assert max(layer.device_status() for layer in layers) == 0
        moments.append([layer.get_moments()[0] for layer in layers])
        off, rel = 0.0, 0.0
        for layer, p, g, M in zip(layers, P, G, moments[-1]):
            R = p.double().T @ g.double() if layer.side == gb.SIDE_LEFT else g.double() @ p.double()
            # an fp32 sum of K terms, see above
            e = float((M.double() / 0.1 - R).norm() / R.norm())
            assert e <= 2 ** -24 * (8 + p.shape[0] ** 0.5)
            off, rel = off + e * e / count, rel + float((M.double() / 0.1 * R).sum() / (R * R).sum() - 1) / count
        err.append(off ** 0.5)
        bias.append(abs(rel))
    assert not all(torch.equal(a, b) for a, b in zip(*moments))       # two kernels ran
    assert err[0] <= err[1] and bias[0] <= bias[1] + 1e-9, (err, bias)


# A layer's own step takes slices by their time and adds accumulators to fp32 sums where the slices that fill the machine would end: no
# further from 64 bits than those, which a batch of one takes.  Both sides, tiles of 128 columns, of 256 and of CTA pairs
@pytest.mark.parametrize("m,n,r", [(6368, 2656, 80), (11008, 4096, 128), (4096, 4600, 120), (2104, 4800, 168), (1920, 2272, 256), (1536, 3264, 272), (3840, 2432, 632),
                                   (1600, 4288, 600)])
def test_drained_sums_are_no_further_from_64_bits_than_slices(m, n, r):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(m + r)
    rand = lambda *s: torch.randn(*s, generator=gen, device="cuda")
    P, G = torch.linalg.qr(rand(min(m, n), r))[0], rand(m, n).bfloat16()
    err, bias = [], []
    for batch in (False, True):
        layer = gb.Layer(gb.make_config(m, n, r, w_dtype="bf16", g_dtype="bf16", auto_refresh=False, adam_place=gb.ADAM_OWN_KERNEL))
        assert layer.uses_tensor_path
        layer.set_projector(P)
        W = torch.zeros(m, n, device="cuda", dtype=torch.bfloat16)
        if batch:
            gb.Batch([layer], [W], [G]).galore_step_batch(1e-2)
        else:
            layer.galore_step(W, G, 1e-2)
        assert layer.device_status() == 0
        p = layer.get_projector().double()
        R = p.T @ G.double() if layer.side == gb.SIDE_LEFT else G.double() @ p
        M = layer.get_moments()[0].double() / 0.1
        err.append(float((M - R).norm() / R.norm()))
        bias.append(abs(float((M * R).sum() / (R * R).sum() - 1)))
    # an accumulator loses up to a unit of 2^-23 of one sign per 16 products, four times a block of 64: 32 blocks lose 1.5e-5 at most
    assert err[0] <= err[1] and bias[0] <= bias[1] + 1e-9 and err[0] <= 128 * 2 ** -23, (err, bias)
