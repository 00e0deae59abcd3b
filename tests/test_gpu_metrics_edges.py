"""GPU parity of s3ttv_quality at the edges of its kernels' tiles: one output
row, columns past a tile of 8, bands past a warp of 32, several row chunks, and
images of enough pixels that a warp takes several spectra.  Tolerances as in
tests/test_gpu_metrics.py (FP64 sums of the same FP32 inputs: 1e-9)."""
import numpy as np
import pytest

import oracle as O
from test_gpu_metrics import solver  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,trim", [((11, 27, 70), 3), ((150, 19, 33), 0), ((60, 41, 39), 3), ((11, 11, 1), 0)])
def test_quality_tile_edges(solver, shape, trim):  # noqa: F811
    r = np.random.default_rng(sum(shape))
    ref = r.uniform(0.0, 1.0, shape).astype(np.float32)
    u = np.clip(ref + 0.1 * r.standard_normal(shape), 0, 1).astype(np.float32)
    u[-1, -1, :] = 0.0
    q = solver.quality(torch.from_numpy(u).cuda(), torch.from_numpy(ref).cuda(), trim=trim, sam_map=True)
    u64, r64 = u.astype(np.float64), ref.astype(np.float64)
    assert q["mpsnr"] == pytest.approx(O.mpsnr(u64, r64, trim), rel=1e-9)
    assert q["mssim"] == pytest.approx(O.mssim(u64, r64, trim), rel=1e-9)
    m = O.sam_map(u64, r64)
    assert q["sam"] == pytest.approx(m.mean(), rel=1e-9)
    np.testing.assert_allclose(q["sam_map"].cpu().numpy(), m, atol=2e-7)
