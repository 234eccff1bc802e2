"""The U-Net's passes between convolutions, and the convolution variants, where
their grids wrap: more pixels than one sweep of a reduction's blocks, more
patches than two CTAs per SM take at once, scratch that limits the blocks."""
import numpy as np
import pytest

from oracle import unet_ref as R

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2201_04565_gb300 import build, nn
    build.build()
    nn.lib()
    return torch, nn


@pytest.mark.parametrize("H,W", [(8, 8), (24, 40), (104, 264)])
def test_batch_gradient_is_the_mean_of_the_images_gradients(env, H, W):
    """Loss and gradient of a batch of four against the images one by one: the
    forward pass is the same per image and the output gradients differ by the
    factor 4 exactly, so only the order of the FP32 sums over pixels differs
    (about 100 terms a thread; 2e-4 allows for cancellation by 100)."""
    torch, nn = env
    B = 4
    gen = torch.Generator().manual_seed(H)
    x = torch.zeros((B, H, W, 32))
    x[..., :4] = torch.randn((B, H, W, 4), generator=gen)
    x = x.to(torch.bfloat16).cuda()
    t = torch.randn((B, H, W, 2), generator=gen).cuda()
    net = nn.UNet(H, W, B, seed=1)
    loss, grad = net.gradients(x, t, B)
    one = [net.gradients(x[b].contiguous(), t[b].contiguous(), 1) for b in range(B)]
    assert loss == pytest.approx(np.mean([o[0] for o in one]), rel=1e-5)
    mean = np.mean([np.asarray(o[1], np.float64) for o in one], axis=0)
    wo, bo, hw, hb, n = R.layout()
    blocks = [(wo[q], bo[q]) for q in range(14)] + [(bo[q], bo[q] + R.CONVS[q][1]) for q in range(14)]
    for a, b in blocks + [(hw, hw + 64), (hb, hb + 2)]:
        assert np.linalg.norm(grad[a:b] - mean[a:b]) <= 2e-4 * np.linalg.norm(mean[a:b]), (a, b)


@pytest.mark.parametrize("cout,B,H,W", [(32, 1, 8, 16), (32, 3, 250, 110), (96, 2, 160, 199)])
def test_two_ctas_per_sm_forward(env, cout, B, H, W):
    """32 input channels, 32-channel tiles: the halo variant with two CTAs on
    an SM, one patch up to several per CTA, ragged patches."""
    torch, nn = env
    rng = np.random.default_rng(W)
    x = R.bf16(rng.standard_normal((B, H, W, 32)))
    Wt = R.bf16(0.2 * rng.standard_normal((cout, 9, 32)))
    out = torch.zeros((B, H, W, cout), dtype=torch.bfloat16, device="cuda")
    tx, tw = (torch.from_numpy(a.astype(np.float32)).to(torch.bfloat16).cuda() for a in (x, Wt))
    nn.check(nn.lib().lsm_nn_conv_forward(nn.ptr(tx), 32, 0, 32, nn.ptr(tw), None, nn.ptr(out), cout, 0, cout, B, H, W,
                                          9, 0, None))
    ref = R.bf16(R.conv(x, Wt.reshape(cout, 3, 3, 32), np.zeros(cout)))
    err = np.abs(out.float().cpu().numpy().astype(np.float64) - ref)
    assert np.all(err <= 2 ** -7 * np.abs(ref) + 1e-6 * np.abs(ref).max())


@pytest.mark.parametrize("C,M", [(32, 1), (32, 100000), (288, 5000), (64, 77825)])
def test_bias_gradient_with_little_scratch(env, C, M):
    """The bias sums with only the scratch that one weight block needs (32 C
    floats), from one pixel to several sweeps of the blocks."""
    torch, nn = env
    gen = torch.Generator().manual_seed(C + M)
    g = torch.randn((M, C), generator=gen).to(torch.bfloat16).cuda()
    x = torch.zeros((M, 32), dtype=torch.bfloat16, device="cuda")
    n = 32 * C
    ws = torch.full((n + 64,), 7.0, device="cuda")
    dW, db = torch.zeros(n, device="cuda"), torch.zeros(C, device="cuda")
    nn.check(nn.lib().lsm_nn_conv_wgrad(nn.ptr(g), C, nn.ptr(x), 32, 0, 32, 1, 1, M, 1, nn.ptr(dW), nn.ptr(db),
                                        nn.ptr(ws), n, None))
    ref, mag = g.double().sum(0), g.double().abs().sum(0)
    # chains of at most M / 64 + 64 terms (one block), each rounding 2^-24 of a partial sum
    assert bool(torch.all((db.double() - ref).abs() <= 2.0 ** -24 * (M / 64 + 64) * mag))
    assert bool(torch.all(ws[n:] == 7.0))
