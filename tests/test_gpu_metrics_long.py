"""GPU parity of s3ttv_quality on long, narrow images: more tiles of output columns
than a grid's second dimension holds (65535 of 8), more row chunks than 64, and
tiles with a single output column.  Tolerance as in tests/test_gpu_metrics.py
(FP64 sums of the same FP32 inputs: 1e-9)."""
import numpy as np
import pytest

import oracle as O
from test_gpu_metrics import solver  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(11, 524291, 1), (12, 524299, 2), (5003, 13, 3), (3001, 11, 40), (70001, 19, 1)])
def test_long_images(solver, shape):  # noqa: F811
    r = np.random.default_rng(sum(shape))
    ref = r.uniform(0.0, 1.0, shape).astype(np.float32)
    u = np.clip(ref + 0.1 * r.standard_normal(shape), 0, 1).astype(np.float32)
    q = solver.quality(torch.from_numpy(u).cuda(), torch.from_numpy(ref).cuda(), trim=0)
    u64, r64 = u.astype(np.float64), ref.astype(np.float64)
    assert q["mssim"] == pytest.approx(O.mssim(u64, r64, 0), rel=1e-9)
    assert q["mpsnr"] == pytest.approx(O.mpsnr(u64, r64, 0), rel=1e-9)
    assert q["sam"] == pytest.approx(O.sam_map(u64, r64).mean(), rel=1e-9)
