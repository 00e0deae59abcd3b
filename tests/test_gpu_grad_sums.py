"""GPU: how exactly the network's weight and bias gradients are summed.

The parameters make every activation a constant and pass the output gradient G on
unchanged (identity centre taps; G is constant in cells of 2 x 2 x 2 voxels, so that
the half-size layers get 8 G exactly), so each gradient looked at is a sum of G times
a small integer over the voxels whose tap lies inside the volume, which FP64 gives
exactly.  All G are of one sign, their sizes spread over a factor of 256.

Tolerances, relative to the sum, with u = 2^-24.  Weights: tensor cores cut off what
lies below a sum's last place, so s products of 16 voxels one after the other lose up
to half a last place of the sum each, s u; s is a CTA's bricks times 8, at most 1024.
To it come, as for the bias, the FP32 additions of up to n partial sums into one value,
whose errors add up like a random walk: 4 sqrt(n) u with n = 152 CTAs (1216 in the
first layer).  The bias has nothing else: the threads' sums are exact to u."""
import numpy as np
import pytest

from oracle import unet as OU
from test_gpu_unet import P  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

U = 2.0 ** -24
MAX_STEPS = 1024


def constant_params():
    """(theta, offsets of (weights, bias) per convolution)."""
    parts, offs, off = [], [], 0
    shapes = list(OU.param_shapes())
    for i in range(0, 20, 2):
        w = np.zeros(shapes[i], np.float32).reshape(shapes[i][0], 27, -1)  # [out][tap][in]
        layer = i // 2
        if layer in (1, 7, 9):
            w[np.arange(w.shape[0]), 13, np.arange(w.shape[0])] = 1.0
        if layer == 8:  # the upsampled part and the skip
            w[np.arange(32), 13, np.arange(32)] = 1.0
            w[np.arange(32), 13, 64 + np.arange(32)] = 1.0
        b = np.ones(w.shape[0], np.float32)
        offs.append((off, off + w.size))
        off += w.size + b.size
        parts += [w.ravel(), b]
    head = np.zeros((3, 32), np.float32)
    head[0] = 1.0
    return np.concatenate(parts + [head.ravel(), np.zeros(3, np.float32)]), offs


def tap_sums(G):
    """Sum of G over the voxels whose neighbour at each of the 27 taps is inside."""
    out = []
    for dz in (-1, 0, 1):
        for dy in (-1, 0, 1):
            for dx in (-1, 0, 1):
                s = [slice(max(0, -d), n + min(0, -d)) for d, n in zip((dz, dy, dx), G.shape[1:])]
                out.append(G[:, s[0], s[1], s[2]].sum().item())
    return np.array(out)


@pytest.mark.parametrize("shape", [(4, 32, 32, 32), (3, 12, 20, 36), (1, 128, 96, 64), (1, 256, 256, 128)])
def test_sums_of_one_sign(P, shape):  # noqa: F811
    theta, offs = constant_params()
    V = int(np.prod(shape))
    v = torch.ones(shape, device="cuda")
    zero = torch.zeros(shape, device="cuda")
    # prediction 1 + 32 * 6 (d1b = 6); errors e between 2^-8 and 1
    cells = tuple([shape[0]] + [n // 2 for n in shape[1:]])
    e = torch.exp2(-8.0 * torch.rand(cells, device="cuda", generator=torch.Generator("cuda").manual_seed(1)))
    for ax in (1, 2, 3):
        e = e.repeat_interleave(2, ax)
    tu = (193.0 - e).contiguous()
    grad = torch.empty(theta.size, device="cuda")
    with P.WarmStartNet(0) as net:
        net.set_params(theta)
        net.gradient(v, tu, zero, zero, grad=grad)
    inv_n = torch.tensor(1.0 / (3.0 * V), dtype=torch.float32, device="cuda")
    G = ((2.0 * (193.0 - tu)) * inv_n).to(torch.bfloat16).double()
    S, H = tap_sums(G), tap_sums(8.0 * G[:, ::2, ::2, ::2])
    g = grad.cpu().numpy().astype(np.float64)
    # layer: (sums, input channels, activation, CTAs adding into one value)
    layers = {0: (S, 1, 1, 1216), 1: (S, 32, 1, 152), 6: (H, 192, 1, 152), 7: (H, 64, 1, 152), 8: (S, 96, 2, 152),
              9: (S, 32, 5, 152)}
    worst = {}
    for layer, (sums, cin, act, n) in layers.items():
        w, b = offs[layer]
        ref = sums[None, :, None] * act
        dw = g[w:b].reshape(-1, 27, cin)[:32]
        worst[layer] = (np.abs(dw / ref - 1).max(), np.abs(g[b:b + 32] / sums[13] - 1).max(), 4 * n ** 0.5 * U)
    print("SUMS", shape, {k: f"{x[0]:.2e} {x[1]:.2e}" for k, x in worst.items()})
    for layer, (ew, eb, walk) in worst.items():
        assert eb <= walk, (layer, eb)
        assert ew <= MAX_STEPS * U + walk, (layer, ew)
