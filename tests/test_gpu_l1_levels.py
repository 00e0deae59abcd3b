"""GPU parity of the l1-ball threshold search where its histogram passes change
form: lengths around the float4 pieces and the CTA size, buffers that start off a
16-byte boundary, values all alike or spread over the whole exponent range, and
repeated calls on one context (the counters of the last-CTA scans return to
zero).  Tolerance: the per-operator bound of the parity tests, 1e-5."""
import numpy as np
import pytest

import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def solver():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2404_03313_gb300 as P
    s = P.Solver(0)
    yield s
    s.close()


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 255, 256, 1023, 1024, 1025, 40000, 400003])
@pytest.mark.parametrize("offset", [0, 1, 2])
def test_l1_ball_lengths_and_alignment(solver, n, offset):
    r = np.random.default_rng(n + offset)
    x = (r.standard_normal(n) * 10.0 ** r.uniform(-6, 3, n)).astype(np.float32)
    base = torch.zeros(n + offset, device="cuda")
    view = base[offset:]
    view.copy_(torch.from_numpy(x))
    for share in (0.3, 0.999, 1.5):
        radius = share * float(np.abs(x.astype(np.float64)).sum())
        out, _ = solver.l1_ball(view, radius)
        ref = O.proj_l1_ball(x.astype(np.float64), radius)
        err = np.linalg.norm(out.cpu().numpy() - ref) / max(np.linalg.norm(ref), 1e-30)
        assert err <= 1e-5, (n, offset, share, err)


def test_l1_ball_equal_values_and_zeros(solver):
    for n in (7, 4096):
        x = np.full(n, 0.25, np.float32)
        x[::3] = 0.0
        radius = 0.1 * float(np.abs(x).sum())
        out, _ = solver.l1_ball(torch.from_numpy(x).cuda(), radius)
        ref = O.proj_l1_ball(x.astype(np.float64), radius)
        assert np.linalg.norm(out.cpu().numpy() - ref) <= 1e-5 * np.linalg.norm(ref)


def test_l1_ball_largest(solver):
    """Every element in one bin of every level, its low bits all ones: the bin sums of
    1.4e9 elements pass 2^32 per CTA unless the grid grows with n.  The projection of a
    constant c to radius n r is the constant r."""
    n = 1_400_000_000
    if torch.cuda.mem_get_info()[0] < 12e9:
        pytest.skip("needs 12 GB")
    x = torch.full((n,), float(np.nextafter(np.float32(2.0), np.float32(0.0))), device="cuda")
    out, tau = solver.l1_ball(x, float(n), out=x)
    assert abs(tau - (2.0 - 2.0 ** -23 - 1.0)) <= 1e-5
    lo, hi = torch.aminmax(out)
    assert abs(float(lo) - 1.0) <= 1e-5 and abs(float(hi) - 1.0) <= 1e-5
