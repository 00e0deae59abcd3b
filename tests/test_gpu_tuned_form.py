"""GPU: s3ttv_tuned_form reports the CTAs per SM that the chosen block-dual form is
compiled for.  The streaming form's count depends on the block side; the others run
4 (tensor cores) or 4 and 5 (CUDA cores)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CTAS = {0: lambda k: (4, 5), 1: lambda k: (4,), 2: lambda k: (4 if k == 5 else 5 if k == 3 else 6,)}


@pytest.fixture(scope="module")
def P():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2404_03313_gb300 as P
    P.library()
    return P


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5])
def test_tuned_form_reports_the_compiled_ctas(P, k):
    v = np.random.default_rng(k).uniform(0, 1, (40, 40, 24)).astype(np.float32)
    with P.Solver(0) as s:
        s.set_option(P.OPT_AUTOTUNE, 1)
        _, _, _, info = s.solve(v, 0.05 * v.size ** 0.5, 0.02 * v.size, 0.02 * v.size, k, max_iter=40, tol=0.0)
        tc, ctas = s.tuned_form()
    assert info["iters"] == 40
    assert tc in CTAS and ctas in CTAS[tc](k), (tc, ctas)
