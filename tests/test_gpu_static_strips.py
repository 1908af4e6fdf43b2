"""galore_step_static on layers whose intermediates do not fit the built-in array at once (done in strips)."""
import pytest
import torch

from paper_2403_03507_b200 import binding as gb

pytestmark = pytest.mark.gpu


# near the limit of 8 bytes per element of R, both sides, a ragged last strip; a tall P (its planes go in ranges of rows)
@pytest.mark.parametrize("m,n,r,side", [(1024, 4001, 512, gb.SIDE_AUTO), (4001, 1024, 512, gb.SIDE_AUTO), (4100, 2000, 1000, gb.SIDE_LEFT)])
def test_strips_equal_the_regular_step(m, n, r, side):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(m + r)
    rand = lambda *s: torch.randn(*s, generator=gen, device="cuda")
    layer = gb.Layer(gb.make_config(m, n, r, w_dtype="f32", g_dtype="f32", auto_refresh=False, side=side))
    P = torch.linalg.qr(rand(layer.proj_rows, r))[0].contiguous()
    layer.set_projector(P)
    W = 0.02 * rand(m, n)
    W_ref, G = W.clone(), rand(m, n)
    M, V = torch.zeros(layer.state_shape, device="cuda"), torch.zeros(layer.state_shape, device="cuda")
    W0 = W.clone()
    assert gb.galore_step_static(P, M, V, W, G, 1e-2, completed_steps=0, side=side) == 0
    layer.galore_step(W_ref, G, 1e-2)
    M_ref, V_ref = layer.get_moments()
    # the K slices of the regular step, whatever the strips: the same bits
    assert torch.equal(M, M_ref) and torch.equal(V, V_ref)
    # the same N through other tiles of the update: fp32 sums of at most 1000 terms
    assert float((W - W_ref).norm() / (W_ref - W0).norm()) <= 4e-6
