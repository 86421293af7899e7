"""The dirty-query attention at the edges of its tiles, key blocks and plans
(one or two query tiles a unit, whole or shared keys, one or several waves),
and with scores that make it raise its softmax reference, against float64."""
import numpy as np
import pytest
import torch

from paper_2608_29809_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    from paper_2608_29809_gb300 import build as B
    B.build()
    from paper_2608_29809_gb300 import regioncache
    return regioncache


@pytest.fixture(scope="module")
def models(R):
    made = {}

    def get(heads, dh):
        if (heads, dh) not in made:
            d = synth.Dims(hidden=heads * dh, heads=heads, mlp=256, layers=1, grid_h=4, grid_w=4,
                           timesteps=1)
            made[heads, dh] = R.Model(d, synth.make_weights(d, 1, device="cuda"))
        return made[heads, dh]

    yield get
    for m in made.values():
        m.close()


def _check(R, m, heads, dh, q, k, v, pad=0):
    """O of the library against float64: relative L2 1e-2 and per element
    2^-7 |want| + 2e-2 RMS (bf16 output and bf16 softmax weights)."""
    nq, nk, h = len(q), len(k), heads * dh
    buf = [torch.full((n, h + pad), 3.0, dtype=torch.bfloat16, device="cuda") for n in (nq, nk, nk)]
    for b, x in zip(buf, (q, k, v)):
        b[:, :h] = x
    out = torch.full((nq, h + pad), 7.0, dtype=torch.bfloat16, device="cuda")
    for _ in range(2):  # (twice: whatever a launch leaves behind serves the next)
        R.rc_attention(m.ctx, buf[0], h + pad, buf[1], buf[2], h + pad, nq, nk, out, h + pad)
    R.rc_sync(m.ctx)
    hd = lambda x: x[:, :h].double().view(len(x), heads, dh).transpose(0, 1)  # noqa: E731
    want = torch.softmax(hd(buf[0]) @ hd(buf[1]).transpose(1, 2) / dh ** 0.5, -1) @ hd(buf[2])
    want = want.transpose(0, 1).reshape(nq, h)
    err = (out[:, :h].double() - want).abs()
    rms = want.norm() / want.numel() ** 0.5
    assert float(err.norm() / want.norm()) <= 1e-2
    assert bool((err <= 2.0 ** -7 * want.abs() + 2e-2 * rms).all())
    assert bool((out[:, h:] == 7.0).all())


def _rand(seed, n, h):
    return synth.randn((n, h), synth.tensor_seed(seed, n, h), "cuda", 1.0, torch.bfloat16)


@pytest.mark.parametrize("nq,nk", [
    (1, 129), (1, 1300), (127, 160), (128, 161), (129, 239), (256, 240), (257, 241), (300, 4095),
    (128, 4097), (640, 2000), (1300, 700), (1217, 512), (2433, 130), (1500, 1024), (2600, 3000)])
@pytest.mark.parametrize("heads,dh", [(16, 72), (2, 64)])
def test_tile_block_and_plan_edges(R, models, heads, dh, nq, nk):
    h = heads * dh
    _check(R, models(heads, dh), heads, dh, _rand(1, nq, h), _rand(2, nk, h), _rand(3, nk, h),
           pad=8 if nq % 2 else 0)


@pytest.mark.parametrize("nq,nk", [(130, 900), (60, 900), (520, 4096)])
@pytest.mark.parametrize("scale", [30.0, 300.0])
def test_scores_that_outgrow_the_reference(R, models, nq, nk, scale):
    """Keys get longer from block to block, so that later scores exceed the
    first block's by far more than the exponentials' range."""
    heads, dh = 16, 72
    h = heads * dh
    k = _rand(5, nk, h).float() * torch.linspace(0.1, scale, nk, device="cuda")[:, None]
    _check(R, models(heads, dh), heads, dh, _rand(4, nq, h), k.bfloat16(), _rand(6, nk, h))
    _check(R, models(heads, dh), heads, dh, _rand(4, nq, h), k.flip(0).bfloat16(), _rand(6, nk, h))


def test_keys_past_the_last_are_not_read_into_the_result(R, models):
    """The values after the last key may hold anything (a multiple of 16 keys)."""
    heads, dh, nq, nk = 16, 72, 200, 4096 - 16
    h = heads * dh
    m = models(heads, dh)
    kv = torch.stack([_rand(7, 4096, h), _rand(8, 4096, h)])
    q, out = _rand(9, nq, h), [torch.zeros(nq, h, dtype=torch.bfloat16, device="cuda")
                               for _ in range(2)]
    for o in out:
        R.rc_attention(m.ctx, q, h, kv[0], kv[1], h, nq, nk, o, h)
        R.rc_sync(m.ctx)
        kv[:, nk:] = float("nan")
    assert np.array_equal(out[0].float().cpu().numpy(), out[1].float().cpu().numpy())
