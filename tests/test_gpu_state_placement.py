"""GPU: the block duals come out the same wherever the destination lies: the pairs of
the paper layout go out as 8-byte stores only where the destination allows them."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("reg,layout,shape", [("REG_S3TTV", 0, (9, 10, 7)), ("REG_S3TTV", 1, (9, 10, 7)),
                                              ("REG_SSST", 0, (9, 10, 7)), ("REG_STV", 0, (40, 33, 17))])
def test_block_duals_into_any_destination(reg, layout, shape):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2404_03313_gb300 as P
    r = np.random.default_rng(1)
    v = r.uniform(0, 1, shape).astype(np.float32)
    with P.Solver(0) as s:
        s.set_option(P.OPT_REGULARIZER, getattr(P, reg))
        s.set_option(P.OPT_LAYOUT, layout)
        s.setup(v, 3.0, 20.0, 10.0, 2)
        size = int(np.prod(s._state_size("Y")))
        Y = r.standard_normal(size).astype(np.float32).reshape(s._state_size("Y"))
        s.set_state("Y", Y)
        np.testing.assert_array_equal(s.get_state("Y"), Y)
        for offset in (0, 1, 2, 3):  # in floats: 16-, 4-, 8- and 4-byte boundaries
            buf = torch.full((size + 8,), 7.0, device="cuda")
            dst = buf[offset:offset + size].view(Y.shape)
            rc = P.library().s3ttv_get_state(s._h, P.STATE["Y"], dst.data_ptr())
            assert rc == P.OK
            assert torch.equal(dst.cpu(), torch.from_numpy(Y)), offset
            assert (buf[:offset] == 7.0).all() and (buf[offset + size:] == 7.0).all()
