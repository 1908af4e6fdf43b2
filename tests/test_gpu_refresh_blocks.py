"""Refreshes whose block has a size at the edges of the factorisation's 64-wide tiles, with and without Chebyshev pairs."""
import pytest
import torch

from paper_2403_03507_b200 import binding as gb

pytestmark = pytest.mark.gpu


# block = rank + oversample columns; a slowly falling spectrum takes Chebyshev pairs, a gapped one plain steps
@pytest.mark.parametrize("rank,over", [(20, 42), (20, 43), (20, 44), (20, 45), (40, 24), (40, 25), (64, 64), (64, 65), (100, 221), (128, 512)])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("gapped", [False, True])
def test_refresh_is_orthonormal_and_spans_the_top_subspace(rank, over, dtype, gapped):
    m, n = 700, 900
    gen = torch.Generator(device="cuda")
    gen.manual_seed(rank * 1000 + over)
    rand = lambda *s: torch.randn(*s, generator=gen, device="cuda", dtype=torch.float64)
    u, v = torch.linalg.qr(rand(m, m))[0], torch.linalg.qr(rand(n, m))[0]
    i = torch.arange(m, device="cuda", dtype=torch.float64)
    s = torch.where(i < rank, 3.0 - i / rank, 0.5 / (1 + i / m)) if gapped else 2.0 * 0.995 ** i
    G = ((u * s) @ v.T).to(torch.float32 if dtype == "f32" else torch.bfloat16)
    layer = gb.Layer(gb.make_config(m, n, rank, w_dtype="bf16", g_dtype=dtype, auto_refresh=False, refresh_oversample=over, seed=7))
    st, info = layer.galore_refresh_projector(G)
    assert st == gb.OK and layer.device_status() == 0, info.as_dict()
    P = layer.get_unrounded_projector()
    # fp64 CholeskyQR and rotations: orthonormal to a small multiple of 2^-53 times the block's size
    assert float((P.T @ P - torch.eye(rank, device="cuda", dtype=torch.float64)).abs().max()) <= 1e-9
    U = torch.linalg.svd(G.double(), full_matrices=False)[0][:, :rank]
    # sine of the largest principal angle: the refresh stops at a predicted 1e-4 (the project's bound is 1e-3)
    assert float(torch.linalg.matrix_norm(P - U @ (U.T @ P), 2)) <= 1e-3


# The fp64 products read every layer's gradient where it lies; tiles of 32 and of 64, and groups that change from one to the other
@pytest.mark.parametrize("m,n,rank,count", [(96, 200, 17, 2), (200, 96, 17, 3), (520, 700, 120, 3), (1000, 640, 129, 8)])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_grouped_layers_with_gradients_of_different_strides_match_single_refreshes(m, n, rank, count, dtype):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(m + count)
    make = lambda i: gb.Layer(gb.make_config(m, n, rank, w_dtype="bf16", g_dtype=dtype, p_dtype="f32", auto_refresh=False, seed=3 + i))
    tdt = torch.float32 if dtype == "f32" else torch.bfloat16
    Gs = []
    for i in range(count):
        wide = torch.randn(m, n + 8 * i, generator=gen, device="cuda", dtype=torch.float32).to(tdt)
        Gs.append(wide[:, :n])                        # leading dimension n + 8 i
    grouped, single = [make(i) for i in range(count)], [make(i) for i in range(count)]
    need = max(gb.galore_refresh_query_bytes(l) for l in grouped)
    gb.galore_refresh_batch(grouped, Gs, workspace=torch.empty(count * need, dtype=torch.uint8, device="cuda"))
    for a, b, G in zip(grouped, single, Gs):
        b.galore_refresh_projector(G)
        # every element is summed in the same order, alone or grouped: the same bits
        assert torch.equal(a.get_projector(), b.get_projector())


# The eigen-solver computes its angles in single precision, scaled by each pair's own size: a gradient times a power of two has the
# same projector, whatever the power; few blocks of 32 rows and many, one matrix and a group
@pytest.mark.parametrize("m,n,rank,over", [(96, 130, 24, 20), (200, 330, 30, 34), (512, 700, 96, 96), (700, 520, 150, 171)])
@pytest.mark.parametrize("count", [1, 3])
def test_projector_does_not_depend_on_the_scale_of_the_gradient(m, n, rank, over, count):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(m + over)
    Gs = [0.1 * torch.randn(m, n, generator=gen, device="cuda") + torch.randn(m, 1, generator=gen, device="cuda") * torch.randn(1, n, generator=gen, device="cuda")
          for _ in range(count)]
    got = []
    for e in (0, 30, -25):
        layers = [gb.Layer(gb.make_config(m, n, rank, w_dtype="f32", g_dtype="f32", auto_refresh=False, refresh_oversample=over, seed=5 + i)) for i in range(count)]
        scaled = [G * 2.0 ** e for G in Gs]
        if count == 1:
            layers[0].galore_refresh_projector(scaled[0])
        else:
            need = gb.galore_refresh_query_bytes(layers[0])
            gb.galore_refresh_batch(layers, scaled, workspace=torch.empty(count * need, dtype=torch.uint8, device="cuda"))
        assert max(l.device_status() for l in layers) == 0
        got.append([l.get_projector().double() for l in layers])
    for i in range(count):
        for other in got[1:]:
            # every operation scales exactly (no value leaves the normal range), up to columns' signs
            assert float((got[0][i].abs() - other[i].abs()).abs().max()) <= 1e-6
