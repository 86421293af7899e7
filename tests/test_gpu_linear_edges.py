"""rc_linear at the edges of its row tiles and waves, single CTAs and CTA
pairs, into a matrix that is 16-byte but not 32-byte aligned, against float64;
rows past the last are not written."""
import pytest
import torch

from paper_2608_29809_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def model():
    from paper_2608_29809_gb300 import build as B
    B.build()
    from paper_2608_29809_gb300 import regioncache
    d = synth.Dims(hidden=128, heads=2, mlp=128, layers=1, grid_h=4, grid_w=4, timesteps=1)
    m = regioncache.Model(d, synth.make_weights(d, 1, device="cuda"))
    yield regioncache, m
    m.close()


@pytest.mark.parametrize("rows,n,k", [
    (1, 128, 64), (31, 384, 64), (129, 1152, 1152), (1500, 4608, 128), (2047, 128, 4608),
    (2048, 1152, 128), (2177, 8192, 64), (9001, 3456, 64), (20001, 256, 64)])
@pytest.mark.parametrize("bias", [True, False])
def test_linear_edges(model, rows, n, k, bias):
    R, m = model
    x = synth.randn((rows, k), synth.tensor_seed(1, rows, k), "cuda", 1.0, torch.bfloat16)
    W = synth.randn((n, k), synth.tensor_seed(2, n, k), "cuda", k ** -0.5, torch.bfloat16)
    b = synth.randn((n,), synth.tensor_seed(3, n), "cuda") if bias else None
    buf = torch.full((rows * n + 4 + 2 * n,), 7.0, device="cuda")
    y = buf[4:4 + rows * n].view(rows, n)
    assert y.data_ptr() % 32 == 16
    R.rc_linear(m.ctx, x, W, b, y, rows, n, k)
    R.rc_sync(m.ctx)
    want = x.double() @ W.double().t() + (b.double() if bias else 0.0)
    assert float((y.double() - want).abs().max()) <= 1e-4 * (1.0 + float(want.abs().max()))
    assert bool((buf[:4] == 7.0).all()) and bool((buf[4 + rows * n:] == 7.0).all())
