"""GPU parity of the per-warp block dual where its column chunks (32 columns) change
form: only a ragged chunk, one whole chunk, whole chunks and a ragged one, whole
chunks only, at every block size of that form.  Tolerance: the per-operator bound of
the parity tests, 1e-5."""
import math

import numpy as np
import pytest

import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N3", [3, 4, 16, 20, 32, 50])
@pytest.mark.parametrize("k", [1, 2, 3, 4, 5])
def test_block_dual_column_chunks(k, N3):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2404_03313_gb300 as P
    shape = (7, 9, N3)
    rng = np.random.default_rng(100 * k + N3)
    scale = rng.uniform(0.02, 3.0, size=(63, 1, 1)) / math.sqrt(k * k + 2 * N3)
    Y = (rng.standard_normal((63, k * k, 2 * N3)) * scale).astype(np.float32)
    ubar = rng.uniform(-0.5, 1.5, size=shape).astype(np.float32)
    s = P.Solver(0)
    try:
        s.set_option(P.OPT_TENSOR_CORES, 2)
        Yd = torch.from_numpy(Y).cuda()
        Zv, Zh, info = s.block_dual(Yd, torch.from_numpy(ubar).cuda(), k)
    finally:
        s.close()
    assert info["jacobi_nonconverged"] == 0
    ref = O.block_dual_update(Y.astype(np.float64), O.structure_tensors(ubar.astype(np.float64), k), 0.25)
    for got, want in zip((Yd, Zv, Zh), (ref, *O.structure_tensors_adjoint(ref, k, shape))):
        assert np.linalg.norm(got.cpu().numpy() - want) <= 1e-5 * np.linalg.norm(want)
