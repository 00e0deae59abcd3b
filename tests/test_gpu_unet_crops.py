"""GPU: the network on volumes whose planes do not fill a tile of 8 x 16 voxels, which
share tiles (mosaics of volumes or of chunks of planes): against the FP64 oracle, a
batch against its members alone, and their time against that of larger crops.

Tolerances: those of tests/test_gpu_unet.py against the oracle; batch against single is
exact, every voxel sums the same products in the same order."""
import time

import numpy as np
import pytest

from oracle import unet as OU
from test_gpu_unet import GRAD_TOL, H_TOL, P, bf16_params, inputs, rel  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# one volume; more volumes than a mosaic takes; one row of pieces, one column; planes cut
# into chunks; sides of 1, 2, 3 and 5 at the coarser levels
SHAPES = [(7, 4, 4, 4), (1, 32, 4, 12), (5, 8, 4, 20), (6, 4, 24, 4), (23, 8, 8, 8), (9, 4, 12, 12)]


@pytest.mark.parametrize("shape", SHAPES)
def test_small_crops_match_oracle(P, shape):  # noqa: F811
    theta = bf16_params(31)
    v, tgt = inputs(shape, 32)
    with P.WarmStartNet(0) as net:
        net.set_params(torch.from_numpy(theta).cuda())
        u, s, t = (x.cpu().numpy() for x in net.forward(torch.from_numpy(v).cuda()))
        loss, g = net.gradient(*(torch.from_numpy(x).cuda() for x in (v,) + tgt))
    ou, os_, ot = OU.forward(theta.astype(np.float64), v.astype(np.float64))
    assert rel(np.stack([u - v, s, t]), np.stack([ou - v, os_, ot])) <= H_TOL
    oloss, og = OU.loss_and_grad(theta.astype(np.float64), v.astype(np.float64), tgt)
    assert abs(loss - oloss) <= H_TOL * oloss
    off = 0
    for shp in OU.param_shapes():
        n = int(np.prod(shp))
        assert rel(g[off:off + n], og[off:off + n]) <= GRAD_TOL, shp
        off += n


@pytest.mark.parametrize("shape,batch", [((4, 4, 4), 1500), ((8, 8, 8), 700), ((16, 4, 12), 350), ((12, 20, 4), 300)])
def test_batch_of_small_crops_equals_single(P, shape, batch):  # noqa: F811
    v = torch.rand((batch,) + shape, generator=torch.Generator().manual_seed(3)).cuda()
    with P.WarmStartNet(0) as net:
        net.set_params(torch.from_numpy(bf16_params(33)).cuda())
        together = net.forward(v)
        for i in (0, 1, 2, batch // 3, batch // 2 + 1, batch - 2, batch - 1):
            for a, b in zip(together, net.forward(v[i].contiguous())):
                assert torch.equal(a[i], b), i


def test_small_crops_cost(P):  # noqa: F811
    """As many voxels in crops of 4^3 as in crops of 16^3: up to five times the time (a
    tile holds 64% of useful voxels at the finest level and 20% and 6% at the coarser ones
    of crops of 4^3; with a tile to each plane of each crop it was nine times)."""
    best = {}
    with P.WarmStartNet(0) as net:
        net.set_params(bf16_params(35))
        for side in (4, 16):
            v = torch.rand(((1 << 20) // side ** 3, side, side, side)).cuda()
            net.forward(v)
            times = []
            for _ in range(7):
                t0 = time.perf_counter()
                net.forward(v)
                times.append(time.perf_counter() - t0)
            best[side] = min(times)
    assert best[4] <= 5.0 * best[16], best
