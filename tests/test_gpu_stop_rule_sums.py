"""GPU: the norms of the stop rule, ||u+ - u|| / ||u||, over many voxels per thread
against FP64.

Tolerance, with u = 2^-24: a thread's chunk of four squares is one FP32 chain (4 u
of its sum, all terms positive), the chunks' rounding errors are kept, the thread's
result rounds once (u), the rest is FP64: 5 u on each sum, half of it on each norm,
plus u for the difference u+ - u itself: 6 u = 3.6e-7.  A plain FP32 chain over a
thread's 431 chunks of equal values is 1.8e-6 off."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 6 * 2.0 ** -24


@pytest.mark.parametrize("kind", ["equal", "random"])
@pytest.mark.parametrize("shape", [(512, 512, 256), (40, 33, 17)])
def test_relative_change_against_fp64(kind, shape):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2404_03313_gb300 as P
    gen = torch.Generator(device="cuda").manual_seed(3)
    v = torch.rand(shape, device="cuda", generator=gen)
    u0 = torch.full(shape, 0.3, device="cuda") if kind == "equal" else torch.rand(shape, device="cuda", generator=gen)
    with P.Solver(0) as s:
        s.set_option(P.OPT_REGULARIZER, P.REG_SSTV)
        s.setup(v, 0.5 * v.numel() ** 0.5, 0.01 * v.numel(), 0.01 * v.numel(), 1)
        s.set_state("u", u0)
        s.set_state("y3", torch.full(shape, 0.01, device="cuda"))
        info = s.iterate(1)
        u1 = s.get_state("u", like=v)
    ref = ((u1.double() - u0.double()).norm() / u0.double().norm()).item()
    assert ref > 1e-4
    assert abs(info["rel_change"] / ref - 1) <= TOL, (info["rel_change"], ref)
