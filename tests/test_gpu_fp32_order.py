"""Layers with fp32 W, G and Adam moments: the projection is one chain of fused multiply-adds over k (slice after slice), bit for bit,
on every entry point, so that a run repeats what earlier releases of the library gave."""
import pytest
import torch

from paper_2403_03507_b200 import binding as gb

pytestmark = pytest.mark.gpu


def _fma(a, b, c):
    """fp32 a * b + c rounded once: the product is exact in fp64; the sum is rounded to odd there (its last bit is set
    when anything was cut off), which makes the second rounding to 24 bits the right one."""
    p, c = a.double() * b.double(), c.double()
    s = p + c
    t = s - p
    cut = (p - (s - t)) + (c - t)
    bits = s.view(torch.int64)
    # towards zero by one unit where the rounding went away from it, then the odd bit
    away = (cut != 0) & ((cut > 0) != (s > 0))
    odd = torch.where(cut != 0, (bits - away.long()) | 1, bits)
    return odd.view(torch.float64).float()


def _chain(A, B, slices):
    """A (M x K) B (K x N) as the library sums it."""
    K = A.shape[1]
    chunk = max(16, -(-(-(-K // slices)) // 16) * 16)
    total = None
    for k0 in range(0, K, chunk):
        acc = torch.zeros(A.shape[0], B.shape[1], device="cuda")
        for k in range(k0, min(K, k0 + chunk)):
            acc = _fma(A[:, k:k + 1], B[k:k + 1, :], acc)
        total = acc if total is None else total + acc
    return total


def _slices(rows, cols, K):
    tile = 64 if rows * cols < 128 * 128 * 96 else 128
    tiles = -(-rows // tile) * -(-cols // tile)
    want = min(min(16, max(1, -(-296 // tiles))), max(1, K // 64))
    chunk = max(16, -(-(-(-K // want)) // 16) * 16)
    return -(-K // chunk)


def _problem(m, n, r, pad, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    rand = lambda *s: torch.randn(*s, generator=gen, device="cuda")
    layer = gb.Layer(gb.make_config(m, n, r, w_dtype="f32", g_dtype="f32", auto_refresh=False))
    P = torch.linalg.qr(rand(layer.proj_rows, r))[0].contiguous()
    layer.set_projector(P)
    G = rand(m, n + pad)[:, :n]
    return layer, P, 0.02 * rand(m, n), G


def _expected(layer, P, G, slices):
    R = _chain(P.T, G, slices) if layer.side == gb.SIDE_LEFT else _chain(G, P, slices)
    return torch.tensor(1.0 - 0.9, dtype=torch.float32, device="cuda") * R      # M after one step from zero


# tile edges of 64 and 128, remainders of the 16-wide K blocks, both sides, one and many slices, rows off 16 bytes
SIZES = [(512, 1376, 128, 0), (1376, 512, 128, 0), (65, 129, 17, 1), (129, 64, 63, 3), (1, 1, 1, 0), (1000, 1200, 300, 0), (1100, 5461, 300, 3)]


@pytest.mark.parametrize("m,n,r,pad", SIZES)
def test_moment_is_the_chain_of_fused_multiply_adds(m, n, r, pad):
    layer, P, W, G = _problem(m, n, r, pad, m + n)
    layer.galore_step(W, G, 1e-2)
    assert torch.equal(layer.get_moments()[0], _expected(layer, P, G, _slices(*layer.state_shape, min(m, n))))


@pytest.mark.parametrize("count", [2, 8])
def test_batches_and_host_batches_sum_in_the_same_order(count):
    shapes = [SIZES[i % 4] for i in range(count)]
    probs = [_problem(*s, 31 + i) for i, s in enumerate(shapes)]
    gb.Batch([p[0] for p in probs], [p[2] for p in probs], [p[3] for p in probs]).galore_step_batch(1e-2)
    for (m, n, r, _), (layer, P, W, G) in zip(shapes, probs):
        slices = 1 if count >= 8 else _slices(*layer.state_shape, min(m, n))       # eight layers fill the machine unsliced
        assert torch.equal(layer.get_moments()[0], _expected(layer, P, G, slices))
    probs = [_problem(*s, 31 + i) for i, s in enumerate(shapes)]
    Ws, Gs = [p[2].cpu().pin_memory() for p in probs], [p[3].contiguous().cpu().pin_memory() for p in probs]
    gb.HostBatch([p[0] for p in probs], Ws, Gs).galore_step_host_batch(1e-2)
    torch.cuda.synchronize()
    for (m, n, r, _), (layer, P, W, G) in zip(shapes, probs):
        assert torch.equal(layer.get_moments()[0], _expected(layer, P, G, _slices(*layer.state_shape, min(m, n))))


@pytest.mark.parametrize("m,n,r,pad", SIZES[:4] + [(1024, 4001, 256, 3)])
def test_static_step_sums_in_the_same_order(m, n, r, pad):
    layer, P, W, G = _problem(m, n, r, pad, m)
    M, V = torch.zeros(layer.state_shape, device="cuda"), torch.zeros(layer.state_shape, device="cuda")
    assert gb.galore_step_static(P, M, V, W, G, 1e-2, completed_steps=0) == 0
    assert torch.equal(M, _expected(layer, P, G, _slices(*layer.state_shape, min(m, n))))


# Operands that are copied to shared memory ahead (rows along the tile, or G's along the sum; 16-byte boundaries) and those that
# are not give the same sums: tiles of 64 and of 128, ragged ends, fewer steps of 16 than stages and many, slices
@pytest.mark.parametrize("side", [gb.SIDE_LEFT, gb.SIDE_RIGHT])
@pytest.mark.parametrize("m,n,r", [(5, 9, 4), (16, 70, 12), (40, 200, 36), (300, 515, 64), (513, 1377, 128), (1100, 3001, 260)])
def test_copied_operands_give_the_bits_of_loaded_ones(m, n, r, side):
    if side == gb.SIDE_RIGHT:
        m, n = n, m
    K = min(m, n)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(m + n)
    P = torch.linalg.qr(torch.randn(K, r, generator=gen, device="cuda"))[0]
    G = torch.randn(m, n, generator=gen, device="cuda")
    got = []
    for pitch in ((n + 3) // 4 * 4, (n + 3) // 4 * 4 + 1):       # rows of G on 16-byte boundaries, and off them
        layer = gb.Layer(gb.make_config(m, n, r, w_dtype="f32", g_dtype="f32", auto_refresh=False, side=side))
        layer.set_projector(P)
        g = torch.full((m, pitch), float("nan"), device="cuda")[:, :n]
        g.copy_(G)
        layer.galore_step(torch.zeros(m, n, device="cuda"), g, 1e-2)
        assert layer.device_status() == 0
        got.append(layer.get_moments())
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
    R = P.double().T @ G.double() if side == gb.SIDE_LEFT else G.double() @ P.double()
    # a chain of K fused multiply-adds: at most 2^-24 sqrt(K) of the root mean square of R in the norm
    assert float((got[0][0].double() / 0.1 - R).norm() / R.norm()) <= 2 ** -24 * (8 + K ** 0.5)
