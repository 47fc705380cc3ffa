"""Weight and bias gradients of the surrogate at the sizes where their kernels can go wrong.

The convolution weight gradient (k_wgrad_win) streams 64-position chunks
through a ring that tiles read at any row, split over at most 152 blocks; the
bias sums and the reduction of the partials depend on the number of positions
too.  Widths at both ends of the allowed range, one tile and many, ragged last
tiles, more tiles than blocks.  On exact-structure networks (one unit weight per
output channel: all activations and activation gradients exact), so gradients
differ from the FP64 oracle's by FP32 summation alone: the 1e-5 of
test_gpu_surrogate.py's structure case, here held per layer.
"""
import numpy as np
import pytest
import torch

from oracle import surrogate as S
from test_gpu_surrogate import _net, _perm_params, _rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W,B,n", [(8, 8, 1, 1), (8, 176, 1, 1), (176, 8, 1, 1), (16, 136, 3, 2), (64, 24, 5, 5),
                                     (72, 128, 2, 2)])
def test_layer_gradients_match_oracle(H, W, B, n):
    ic, oc = 2, 12
    ps = _perm_params(ic, oc, (True, False, True))
    r = np.random.default_rng(H * W + B)
    x = S.bf16(r.uniform(0.05, 1, (n, H, W, ic)))
    dy = S.bf16(r.standard_normal((n, H, W, oc)))
    net = _net(H, W, ic, oc, B)
    net.set_params(S.flatten(ps).astype(np.float32))
    y = net.forward(torch.tensor(x, dtype=torch.float32, device="cuda:0")).cpu().numpy()
    net.backward(torch.tensor(dy, dtype=torch.float32, device="cuda:0"))
    got = S.unflatten(net.grads().cpu().numpy().astype(np.float64), ic, oc)
    net.check()
    y0, cache = S.forward(ps, x, rounding=True)
    want, _ = S.backward(ps, cache, dy)
    assert np.array_equal(y, y0)
    for (name, *_), (gw, gb), (ww, wb) in zip(S.layer_table(ic, oc), got, want):
        assert _rel(gw, ww) < 1e-5, name
        assert _rel(gb, wb) < 1e-5, name


@pytest.mark.parametrize("n", [1, 700, 1 << 18])
def test_loss_is_the_mean_square(n):
    H = W = 8
    net = _net(H, W, 1, 1, (n + 63) // 64)
    g = torch.Generator(device="cuda:0").manual_seed(n)
    b = (n + 63) // 64
    y, t = (torch.randn((b, H, W, 1), generator=g, device="cuda:0") for _ in range(2))
    loss, dy = net.mse(y, t)
    d = (y - t).double()
    assert abs(loss.item() - (d * d).mean().item()) < 1e-6 * (d * d).mean().item()
    assert _rel(dy.cpu().numpy(), (2 * d / d.numel()).cpu().numpy()) < 1e-6


@pytest.mark.parametrize("seed", [0, 1])
def test_gradients_of_many_positions_are_sound_and_repeat(seed):
    """64 copies of one 128 x 128 sample: every block of k_wgrad_win streams a hundred tiles through its rings, so a
    dY tile whose slot is refilled before the bias sums have read it shows, as bits that differ from pass to pass
    and as bias entries off by 1e-3.  Exact-structure network as above, so a layer's bias gradient is 64 times the
    sample's FP64 sum of the layer's output gradient: 480 FP32 additions deep over values that cancel, about 1e-7
    relative, held to 1e-6; the weights to 5e-5 (an accumulator in tensor memory takes 448 steps of 2^-24 at most,
    2.7e-5, then 23 more additions)."""
    ic, oc, H, W, B = 1, 24, 128, 128, 64
    ps = _perm_params(ic, oc, (True, False, True))
    r = np.random.default_rng(seed)
    x = S.bf16(r.uniform(0.05, 1, (1, H, W, ic)))
    dy = S.bf16(r.standard_normal((1, H, W, oc)))
    net = _net(H, W, ic, oc, B)
    net.set_params(S.flatten(ps).astype(np.float32))
    net.forward(torch.tensor(x, dtype=torch.float32, device="cuda:0").expand(B, -1, -1, -1))
    d = torch.tensor(dy, dtype=torch.float32, device="cuda:0").expand(B, -1, -1, -1).contiguous()
    net.backward(d)
    first = net.grads()
    for k in range(100):
        net.backward(d)
        assert torch.equal(net.grads().view(torch.int32), first.view(torch.int32)), k
    net.check()
    want, _ = S.backward(ps, S.forward(ps, x, rounding=True)[1], dy)
    got = S.unflatten(first.cpu().numpy().astype(np.float64), ic, oc)
    for (name, *_), (gw, gb), (ww, wb) in zip(S.layer_table(ic, oc), got, want):
        assert _rel(gb, B * wb) < 1e-6, name
        assert _rel(gw, B * ww) < 5e-5, name
