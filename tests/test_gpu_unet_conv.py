"""GPU parity of the network's tcgen05 convolutions at the edges of their work
units (columns of 8 voxels along W by 16 or 32 along H, chunks of planes along
D): ragged and single-tile sides against the FP64 oracle, and volumes of several
units per CTA against the same cubes alone.

Tolerances: those of tests/test_gpu_unet.py (BF16 storage of every activation
and activation gradient: 3e-2 for the output, 5e-2 for a parameter array's
gradient); batch against single is exact, every voxel sums the same products in
the same order whatever unit it falls into.
"""
import numpy as np
import pytest

from oracle import unet as OU
from test_gpu_unet import GRAD_TOL, H_TOL, P, bf16_params, inputs, rel  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# (B, D, H, W): H past one and past two 16-voxel tiles with W past 8; one plane at the
# coarsest level; a long D (several chunks of planes); W one tile, H one voxel over a tile
EDGES = [(1, 8, 36, 12), (1, 4, 20, 20), (1, 44, 8, 8), (2, 12, 68, 4)]


@pytest.mark.parametrize("shape", EDGES)
def test_edges_match_oracle(P, shape):  # noqa: F811
    theta = bf16_params(11)
    v, tgt = inputs(shape, 12)
    with P.WarmStartNet(0) as net:
        net.set_params(torch.from_numpy(theta).cuda())
        vd = torch.from_numpy(v).cuda()
        u, s, t = (x.cpu().numpy() for x in net.forward(vd))
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


@pytest.mark.parametrize("shape,batch", [((20, 36, 28), 24), ((64, 36, 44), 12)])
def test_batch_equals_single(P, shape, batch):  # noqa: F811
    theta = torch.from_numpy(bf16_params(13)).cuda()
    v = torch.rand((batch,) + shape, generator=torch.Generator().manual_seed(3)).cuda()
    with P.WarmStartNet(0) as net:
        net.set_params(theta)
        together = net.forward(v)
        for i in (0, 1, batch // 2, batch - 1):
            for a, b in zip(together, net.forward(v[i].contiguous())):
                assert torch.equal(a[i], b), i
